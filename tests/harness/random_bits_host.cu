// Host harness of the random bits of stochastic rounding (vlb_lattice_body.cuh):
// for the keys on standard input, the bits of the nine pairs.
#include <cstdio>

#include "vlb_lattice_body.cuh"

int main() {
  unsigned key;
  while (std::scanf("%u", &key) == 1) {
    for (int i = 0; i < 9; ++i) std::printf("%u ", vlb::sr_bits(key, i));
    std::printf("\n");
  }
  return 0;
}
