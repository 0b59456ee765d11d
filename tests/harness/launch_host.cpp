// Host harness of the kernels' launches: the library's own objects over the
// stand-in for the CUDA runtime of fake_cuda.cpp, which records each launch.
// Prints, for handles without and with a particle, stepped alone and as a batch
// of two storage types, a line "RUN kernel early" per launch.
#include <cstdio>

#include "../../include/vlb.h"
#include "fake_cuda.h"

static vlb_handle* make(int precision, int np) {
  vlb_params p;
  vlb_params_default(&p);
  p.precision = precision;
  vlb_handle* h = nullptr;
  const double xy[2] = {30.0, 30.0}, r = 5.0, T0 = 0.0;
  if (vlb_create(&p, &h) != VLB_OK || (np && vlb_add_particles(h, 1, xy, &r, &T0, nullptr, nullptr, nullptr) != VLB_OK))
    std::printf("setup failed\n");
  vlb_step(h, 0);
  return h;
}
static void report(const char* run, int np) {
  for (const auto& l : fake::launches) std::printf("%s%d %s %d\n", run, np, l.kernel.c_str(), l.early);
  fake::launches.clear();
}

int main() {
  for (int np = 0; np < 2; ++np) {
    vlb_handle* h[3] = {make(VLB_FP32, np), make(VLB_FP64, np), make(VLB_FP16_STORE, np)};
    fake::launches.clear();
    vlb_step(h[0], 3);
    vlb_step(h[1], 3);
    report("alone", np);
    int failed = 0;
    if (vlb_step_batch(h, 3, 3, &failed) != VLB_OK) std::printf("batch failed\n");
    report("batch", np);
    for (vlb_handle* q : h) vlb_destroy(q);
  }
  return 0;
}
