// Host harness of the kernels' launches: the library's own objects over the
// stand-in for the CUDA runtime of fake_cuda.cpp, which records each launch.
// Prints, for handles without and with a particle, stepped alone and as a batch
// of two storage types, and for crowded ones ("alone2", "batch2"), a line "RUN
// kernel early" per launch.
#include <cstdio>
#include <vector>

#include "../../include/vlb.h"
#include "fake_cuda.h"

static vlb_handle* make(int precision, int np, int per_row = 1, double pitch = 30.0) {
  vlb_params p;
  vlb_params_default(&p);
  p.precision = precision;
  p.nx = p.ny = per_row > 1 ? (int)(per_row * pitch) + 4 : 64;
  vlb_handle* h = nullptr;
  std::vector<double> xy, r, T0;
  for (int k = 0; k < np * per_row * per_row; ++k) {
    xy.push_back(pitch * (k % per_row + 0.5) + 2.0);
    xy.push_back(pitch * (k / per_row + 0.5) + 2.0);
    r.push_back(1.5);
    T0.push_back(0.0);
  }
  if (vlb_create(&p, &h) != VLB_OK ||
      vlb_add_particles(h, (int)r.size(), xy.data(), r.data(), T0.data(), nullptr, nullptr, nullptr) != VLB_OK)
    std::printf("setup failed\n");
  vlb_step(h, 0);
  return h;
}
static void report(const char* run, int number) {
  for (const auto& l : fake::launches) std::printf("%s%d %s %d\n", run, number, l.kernel.c_str(), l.early);
  fake::launches.clear();
}

int main() {
  for (int run = 0; run < 3; ++run) {
    const int np = run > 0 ? 1 : 0, per_row = run == 2 ? 20 : 1;
    const double pitch = run == 2 ? 6.0 : 30.0;
    vlb_handle* h[3] = {make(VLB_FP32, np, per_row, pitch), make(VLB_FP64, np, per_row, pitch),
                        make(VLB_FP16_STORE, np, per_row, pitch)};
    fake::launches.clear();
    vlb_step(h[0], 3);
    vlb_step(h[1], 3);
    report("alone", run);
    int failed = 0;
    if (vlb_step_batch(h, 3, 3, &failed) != VLB_OK) std::printf("batch failed\n");
    report("batch", run);
    for (vlb_handle* q : h) vlb_destroy(q);
  }
  return 0;
}
