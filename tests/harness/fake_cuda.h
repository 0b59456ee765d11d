// State of the stand-in for the CUDA runtime (fake_cuda.cpp).
#pragma once
#include <cstddef>
#include <string>
#include <vector>

namespace fake {
extern size_t live;   // bytes of the live device buffers
extern long allocs;   // device allocations so far
extern bool full;     // no device memory is left
struct Launch {
  std::string kernel;  // (mangled)
  bool early;          // programmatic: may come in while the one before runs
};
extern std::vector<Launch> launches;
void legacy_wait();   // what the legacy stream still has to write is written
}  // namespace fake
