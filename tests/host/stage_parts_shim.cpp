// C shim over csrc/stage_parts.hpp for the host tests.
#include "stage_parts.hpp"

extern "C" {
int hp_part_begin(int zp, int nz, int BS) { return acm::part_begin(zp, nz, BS); }
int hp_upper_in_prologue(int z0, int M) { return acm::upper_in_prologue(z0, M); }
int hp_upper_in_loop(int z, int z0, int z1, int M) { return acm::upper_in_loop(z, z0, z1, M); }
int hp_z_parts(long long n, int NS, int BS, long long slots, long long start) {
  return acm::z_parts_rule(n, NS, BS, slots, start);
}
}
