// What the stand-in runtime (fake_cudart.cpp) has seen.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <map>
#include <string>

namespace fake {
extern int races;               // frees of memory while another stream of its device had work in flight
extern int wrong_device;        // frees ordered after a stream of another device than the memory's
extern int fail_set_attribute;  // calls of cudaMemPoolSetAttribute still to fail
extern std::map<std::string, unsigned> last_grid;  // blocks of each kernel's last launch
size_t used();                // of a device's bytes
size_t reserved();            // bytes the pools hold: in use, freed and kept, freed and not yet seen to be
uint64_t lowest_threshold();  // of the pools there are
bool from_pool(const void* p);
int blocks();                 // allocations there are
extern size_t capacity;       // bytes of a device
}  // namespace fake
