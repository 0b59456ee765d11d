// State of the stand-in for the CUDA runtime (fake_cuda.cpp).
#pragma once
#include <cstddef>

namespace fake {
extern size_t live;   // bytes of the live device buffers
extern long allocs;   // device allocations so far
extern bool full;     // no device memory is left
void legacy_wait();   // what the legacy stream still has to write is written
}  // namespace fake
