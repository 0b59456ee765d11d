// Host harness of the C ABI's host code (vlb_capi.cu) over the stand-in for the
// CUDA runtime of fake_cuda.cpp, where kernels do nothing but split and join
// population planes.
//
// Usage: capi_host CHECK, one of
//   roundtrip   loads an image of random bytes into handles of each storage type
//               and saves it again: the two must be equal
//   full        the same with no device memory left, fields read in between, at
//               step 0 and later: no device allocation, the populations of the
//               level unchanged
//   helpers     reads a field with helper threads that get no buffer: the calling
//               thread takes their pieces
//   footprint   device bytes of a handle with ellipses and one without, after
//               the first step: what vlb_device_bytes says
// Prints "ok", or what differs and exits with 1.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <thread>
#include <string>
#include <vector>

#include "../../include/vlb.h"
#include "fake_cuda.h"

// (no-throw array allocations of other threads fail on request)
static bool g_fail_helpers = false;
static const std::thread::id g_main = std::this_thread::get_id();
void* operator new[](size_t n, const std::nothrow_t&) noexcept {
  return g_fail_helpers && std::this_thread::get_id() != g_main ? nullptr : std::malloc(n);
}
void operator delete[](void* p) noexcept { std::free(p); }
void operator delete[](void* p, size_t) noexcept { std::free(p); }

static int bad(const char* what, int precision) {
  std::printf("%s (precision %d)\n", what, precision);
  return 1;
}
// A handle of three particles, two of them ellipses unless `disks`, at its
// initial state.
static vlb_handle* make(int precision, bool disks = false, uint64_t* bytes = nullptr) {
  vlb_params p;
  vlb_params_default(&p);
  p.nx = 61;
  p.ny = 43;
  p.precision = precision;
  p.max_particles = 5;
  vlb_handle* h = nullptr;
  const double disk[2] = {12.5, 30.25}, two[4] = {20.0, 12.0, 45.0, 25.0}, a[2] = {6.0, 7.0}, b[2] = {3.0, 4.0};
  const double theta[2] = {0.3, -0.4}, T0[2] = {0.0, 0.0}, r = 5.0, radius[3] = {5.0, 6.0, 7.0};
  if (bytes) vlb_device_bytes(&p, 3, radius, bytes);
  if (vlb_create(&p, &h) != VLB_OK || vlb_add_particles(h, 1, disk, &r, T0, nullptr, nullptr, nullptr) != VLB_OK ||
      vlb_add_ellipses(h, 2, two, a, disks ? a : b, theta, T0, nullptr, nullptr, nullptr) != VLB_OK || vlb_step(h, 0) != VLB_OK) {
    std::printf("setup: %s\n", vlb_last_error(h));
    std::exit(1);
  }
  return h;
}
// An image of the handle's shape with random bytes in place of its state.
static std::vector<char> random_image(vlb_handle* h) {
  uint64_t n = 0;
  if (vlb_state_size(h, &n) != VLB_OK) std::exit(bad("state size", -1));
  std::vector<char> image(n);
  if (vlb_save_state(h, image.data(), n) != VLB_OK) std::exit(bad("save", -1));
  uint32_t header = 0, s = 12345;
  std::memcpy(&header, image.data() + 12, sizeof(header));  // (magic, version, the header's bytes)
  // (the populations and S; what follows says which particles are ellipses)
  uint64_t sizes[2];
  std::memcpy(sizes, image.data() + 72, sizeof(sizes));
  const size_t end = header + 2 * (sizes[0] + sizes[1]);
  for (size_t i = header; i < end; ++i) image[i] = (char)((s = s * 1664525u + 1013904223u) >> 24);
  return image;
}
static int roundtrip() {
  for (int precision : {VLB_FP64, VLB_FP32, VLB_FP16_STORE, VLB_BF16_STORE}) {
    vlb_handle* h = make(precision);
    const std::vector<char> image = random_image(h);
    std::vector<char> again(image.size());
    if (vlb_load_state(h, image.data(), image.size()) != VLB_OK) return bad(vlb_last_error(h), precision);
    if (vlb_save_state(h, again.data(), again.size()) != VLB_OK) return bad(vlb_last_error(h), precision);
    if (again != image) return bad("the saved image differs from the loaded one", precision);
    vlb_destroy(h);
  }
  return 0;
}

static int full() {
  for (int precision : {VLB_FP64, VLB_FP32, VLB_FP16_STORE, VLB_BF16_STORE}) {
    vlb_handle* h = make(precision);
    std::vector<char> image = random_image(h), again(image.size());
    const long allocs = fake::allocs;
    if (vlb_load_state(h, image.data(), image.size()) != VLB_OK ||
        vlb_save_state(h, again.data(), again.size()) != VLB_OK || fake::allocs != allocs)
      return bad("an image allocated device memory", precision);
    fake::full = true;
    std::vector<double> T(61 * 43);
    for (int step : {0, 7}) {
      const int64_t at = step;
      std::memcpy(image.data() + 64, &at, sizeof(at));
      if (vlb_load_state(h, image.data(), image.size()) != VLB_OK) return bad(vlb_last_error(h), precision);
      for (int times = 0; times < 3; ++times) {
        // (a read-back leaves valid macroscopic planes; at step 0 the other
        // population buffer then has no content)
        if (vlb_get_fields(h, VLB_FIELD_T, nullptr, nullptr, nullptr, T.data(), nullptr) != VLB_OK)
          return bad(vlb_last_error(h), precision);
        if (vlb_save_state(h, again.data(), again.size()) != VLB_OK) return bad(vlb_last_error(h), precision);
        uint32_t header = 0;
        uint64_t pop = 0;
        std::memcpy(&header, image.data() + 12, sizeof(header));
        std::memcpy(&pop, image.data() + 72, sizeof(pop));
        if (std::memcmp(again.data() + header, image.data() + header, pop) != 0) return bad("populations changed", precision);
        if (step > 0 && again != image) return bad("the saved image differs", precision);
      }
    }
    fake::full = false;
    vlb_destroy(h);
  }
  return 0;
}
static int helpers() {
  vlb_params p;
  vlb_params_default(&p);
  p.nx = p.ny = 1500;
  p.precision = VLB_FP32;
  p.max_particles = 0;
  vlb_handle* h = nullptr;
  if (vlb_create(&p, &h) != VLB_OK || vlb_step(h, 0) != VLB_OK) return bad("setup", p.precision);
  std::vector<double> ux(1500 * 1500, 1.0), T(1500 * 1500, 1.0);
  g_fail_helpers = true;
  const vlb_status s = vlb_get_fields(h, VLB_FIELD_UX | VLB_FIELD_T, nullptr, ux.data(), nullptr, T.data(), nullptr);
  g_fail_helpers = false;
  if (s != VLB_OK) return bad(vlb_last_error(h), p.precision);
  float a5;  // (device memory as the stand-in hands it out)
  std::memset(&a5, 0xA5, sizeof(a5));
  for (size_t c = 0; c < T.size(); ++c)
    if (ux[c] != a5 || T[c] != a5) return bad("values missing", p.precision);
  vlb_destroy(h);
  return 0;
}
static int footprint() {
  for (int precision : {VLB_FP64, VLB_FP32, VLB_FP16_STORE, VLB_BF16_STORE}) {
    for (bool disks : {true, false}) {
      uint64_t bytes = 0;
      const size_t before = fake::live;
      vlb_handle* h = make(precision, disks, &bytes);
      if (vlb_step(h, 2) != VLB_OK) return bad(vlb_last_error(h), precision);
      if (fake::live - before != bytes) return bad(disks ? "disks: other bytes" : "ellipses: other bytes", precision);
      vlb_destroy(h);
      if (fake::live != before) return bad("bytes left behind", precision);
    }
  }
  return 0;
}

int main(int argc, char** argv) {
  const std::map<std::string, int (*)()> checks = {{"roundtrip", roundtrip}, {"full", full}, {"helpers", helpers}, {"footprint", footprint}};
  const auto it = argc > 1 ? checks.find(argv[1]) : checks.end();
  if (it == checks.end() || it->second() != 0) return 1;
  std::printf("ok\n");
  return 0;
}
