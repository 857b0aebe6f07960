// Host program for tests/test_point_places.py: reads "first_chunk at part", one
// a line, and prints where nn_place puts that part, in floats.
#include <stdio.h>

#include "gp_nn_device.cuh"

int main() {
  long long first, at;
  int k;
  while (scanf("%lld %lld %d", &first, &at, &k) == 3) printf("%lld\n", (long long)nn_place(first, (uint32_t)at, k));
  return 0;
}
