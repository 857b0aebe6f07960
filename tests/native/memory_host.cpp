// Host program for tests/test_device_memory.py: runs the library's calls on the
// stand-in runtime and prints what it saw, one "name value" a line.
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "fake_cudart.h"
#include "gridpull.h"

static gp_band* make_band(gp_ctx* ctx, int64_t J) {
  void* pts = nullptr;
  cudaMalloc(&pts, 3 * J * sizeof(float));
  gp_grid_desc d = {16, 1, 1, 4, 0, 0};
  gp_band* b = nullptr;
  if (gp_build_band(ctx, (const float*)pts, J, &d, &b)) printf("error %s\n", gp_last_error(ctx));
  cudaFree(pts);
  return b;
}

static gp_multi* make_multi(gp_ctx* ctx, gp_band* b, int64_t B) {
  gp_multi* m = nullptr;
  if (gp_multi_create(ctx, &b, 1, &B, &B, 1, GP_SAMPLE_SPATIAL, &m)) printf("error %s\n", gp_last_error(ctx));
  return m;
}

static void step(gp_multi* m) {
  const gp_loss_w w = {1.f, 1.f, 0.005f};
  const gp_adam hp = {1e-3f, 0.9f, 0.999f, 1e-8f};
  static float loss[8];
  if (gp_multi_step(m, &w, &hp, 1.f, 0, loss)) printf("error step\n");
}

static void report() {
  int dev = -1;
  cudaGetDevice(&dev);
  printf("device %d\nraces %d\nwrong_device %d\n", dev, fake::races, fake::wrong_device);
}

int main(int argc, char** argv) {
  const char* what = argc > 1 ? argv[1] : "";
  const cudaStream_t s1 = (cudaStream_t)0x10, s2 = (cudaStream_t)0x20;
  if (!strcmp(what, "other_device")) {
    // A step of a multi of device 1 is in flight; it is destroyed while device 0 is current.
    gp_ctx* ctx = nullptr;
    gp_create(&ctx, 1, s1);
    gp_band* b = make_band(ctx, 100);
    gp_multi* m = make_multi(ctx, b, 1000);
    step(m);
    cudaSetDevice(0);
    gp_multi_destroy(m);
    report();
  } else if (!strcmp(what, "tiles")) {
    // A step is in flight on one stream when the multi is tuned on another.
    gp_ctx* ctx = nullptr;
    gp_create(&ctx, 0, s1);
    gp_multi* m = make_multi(ctx, make_band(ctx, 100), 1000);
    step(m);
    gp_set_stream(ctx, s2);
    const gp_loss_w w = {1.f, 1.f, 0.005f};
    if (gp_multi_autotune(m, &w)) printf("error autotune\n");
    report();
  } else if (!strcmp(what, "given_back")) {
    // A band beyond what the pool keeps, then the last context of the device.
    gp_ctx *ctx = nullptr, *other = nullptr;
    gp_create(&ctx, 0, s1);
    gp_create(&other, 0, s2);
    const size_t keep = fake::lowest_threshold();
    gp_band* b = make_band(ctx, (int64_t)keep / 12 + 1);
    printf("above_while_alive %d\n", fake::reserved() > keep);
    gp_band_destroy(b);
    printf("above_after_the_band %d\n", fake::reserved() > keep);
    gp_destroy(other);
    b = make_band(ctx, 100);
    gp_multi* m = make_multi(ctx, b, 1000);
    step(m);
    gp_multi_destroy(m);
    gp_destroy(ctx);
    gp_band_destroy(b);
    printf("after_the_last_context %d\n", (int)fake::reserved());
  } else if (!strcmp(what, "no_threshold")) {
    // The pool's threshold cannot be set at the first context, then it can.
    gp_ctx* ctx = nullptr;
    fake::fail_set_attribute = 1;
    const gp_status first = gp_create(&ctx, 0, s1);
    const gp_status second = gp_create(&ctx, 0, s1);
    printf("first %d\nsecond %d\nkeeps %d\n", first, second, fake::lowest_threshold() > 0);
  } else if (!strcmp(what, "shown")) {
    // Where the pointers that callers receive lie.
    gp_ctx* ctx = nullptr;
    gp_create(&ctx, 0, s1);
    gp_band* b = make_band(ctx, 100);
    gp_multi* m = make_multi(ctx, b, 1000);
    float *d = nullptr, *am = nullptr, *av = nullptr, *rec = nullptr, *grad = nullptr;
    int32_t* src = nullptr;
    gp_band_values(b, &d, &am, &av);
    gp_multi_buffers(m, 0, &rec, &src, &grad);
    printf("values %d\nmoments %d\n", fake::from_pool(d), fake::from_pool(am) + fake::from_pool(av));
    printf("multi %d\n", fake::from_pool(rec) + fake::from_pool(src) + fake::from_pool(grad));
    gp_multi_destroy(m);
    gp_band_destroy(b);
    b = make_band(ctx, 100);
    float* again = nullptr;
    gp_band_values(b, &again, nullptr, nullptr);
    printf("kept %d\n", again == d || again == grad);
    m = make_multi(ctx, b, 1000);
    gp_band_destroy(b);
    gp_destroy(ctx);
    gp_multi_destroy(m);  // last, as a collector may have it
    printf("left %d\n", (int)fake::reserved() + fake::blocks());
  } else if (!strcmp(what, "tuned")) {
    // Blocks of the search's launch against gp_multi_info, before and after the
    // autotuner (which here finds the longest tiles the fastest).
    gp_ctx* ctx = nullptr;
    gp_create(&ctx, 0, s1);
    gp_multi* m = make_multi(ctx, make_band(ctx, 100), 100000);
    gp_multi_info i;
    const gp_loss_w w = {1.f, 1.f, 0.005f};
    step(m);
    gp_multi_get_info(m, &i);
    printf("default %d\n", (int)fake::last_grid["k_m_nn"] - 8 * i.blocks_per_sm_nn);
    if (gp_multi_autotune(m, &w)) printf("error autotune\n");
    step(m);
    gp_multi_get_info(m, &i);
    printf("records_per_tile %d\ntuned %d\n", i.records_per_tile,
           (int)fake::last_grid["k_m_nn"] - 8 * i.blocks_per_sm_nn);
  } else if (!strcmp(what, "full")) {
    // Allocations that fit only once kept memory is given up: a band's from the
    // pool with blocks kept, then a multi's blocks with the pool's memory kept.
    gp_ctx* ctx = nullptr;
    gp_create(&ctx, 0, s1);
    gp_band* b = make_band(ctx, 100);
    gp_multi* m = make_multi(ctx, b, 4000000);
    gp_multi_destroy(m);
    gp_band_destroy(b);
    fake::capacity = fake::used() + (size_t(60) << 20);
    b = make_band(ctx, 2000000);
    printf("band %d\n", b != nullptr);
    gp_band_destroy(b);
    b = make_band(ctx, 100);
    fake::capacity = fake::used() + (size_t(20) << 20);
    m = make_multi(ctx, b, 2000000);
    printf("multi %d\n", m != nullptr);
  }
  return 0;
}
