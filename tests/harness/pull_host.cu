// Host harness of the lattice kernel's wall rules (vlb_lattice_body.cuh).
// Reads lines "nx ny per_x per_y open0 open1 open2 open3 x y i" and prints
// whether direction i of cell (x, y) bounces back, whether off a y side, and
// the cell index it comes from (rows of nx + 3 entries).
#include <cstdio>

#include "vlb_lattice_body.cuh"

int main() {
  vlb::LatticeConst<float> K{};
  int x, y, i;
  while (std::scanf("%d %d %d %d %d %d %d %d %d %d %d", &K.nx, &K.ny, &K.per_x, &K.per_y, &K.outflow[0],
                    &K.outflow[1], &K.outflow[2], &K.outflow[3], &x, &y, &i) == 11) {
    K.pitch = K.nx + 3;
    const vlb::PullFrom f = vlb::pull_from(vlb::crossing(K, x, y), i);
    const int here = y * K.pitch + x;
    std::printf("%d %d %d\n", f.bounce, f.y_wall,
                f.bounce ? here : here - vlb::ex(i) - vlb::ey(i) * K.pitch + f.shift);
  }
  return 0;
}
