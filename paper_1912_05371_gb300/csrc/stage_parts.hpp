// Parts of a block along z in the fused stage kernel (stage.cu): the plain arithmetic of the split, kept
// apart from the CUDA code so that the CPU can check every part of every count.
#pragma once

#include <cstdint>

namespace acm {

// Part zp of nz of a block of BS planes holds the planes part_begin(zp) .. part_begin(zp + 1) - 1.
constexpr int part_begin(int zp, int nz, int BS) { return zp * BS / nz; }

// Planes M + 1 .. M + 3 beyond the block's upper z face come to shared memory by cp.async and are first
// read in iteration M - 2.  A copy may be read after a wait that leaves only newer groups pending; the
// loop's wait leaves one group pending, the one committed in the same iteration, and the last iteration
// has none.  So the request has to be committed at least one iteration before M - 2: in iteration
// z0 + 1, where it hides behind the first planes' work, only if that is M - 3 or earlier; else before
// the loop, in the group of the first plane's halos, which the first wait completes.
constexpr bool upper_in_prologue(int z0, int M) { return z0 >= M - 3; }
constexpr bool upper_in_loop(int z, int z0, int z1, int M) {
  return z == z0 + 1 && !upper_in_prologue(z0, M) && z1 > M - 2;
}

// The number of parts whose waves of CTAs over the chip cost least: n blocks of NS CTAs each run side by
// side on `slots` resident CTAs, and a CTA costs `start` planes' time plus its planes.
constexpr int z_parts_rule(int64_t n, int NS, int BS, int64_t slots, int64_t start) {
  int best = 1;
  int64_t cost = -1;
  for (int nz = 1; nz <= BS / 2; ++nz) {
    const int64_t c = (n * NS * nz + slots - 1) / slots * (start + (BS + nz - 1) / nz);
    if (cost < 0 || c < cost) {
      cost = c;
      best = nz;
    }
  }
  return best;
}

// Every part of every count up to BS / 2 has at least two planes (the loop's first wait needs a second
// one) and requests the upper planes early enough (see upper_in_loop): checked at compile time.
constexpr bool parts_are_sound(int BS) {
  const int M = BS - 1;
  for (int nz = 1; nz <= BS / 2; ++nz)
    for (int zp = 0; zp < nz; ++zp) {
      const int z0 = part_begin(zp, nz, BS), z1 = part_begin(zp + 1, nz, BS);
      if (z1 - z0 < 2) return false;
      if (z1 <= M - 2 || upper_in_prologue(z0, M)) continue;
      // requested in iteration z0 + 1, complete after the wait of iteration z0 + 2, which must not be
      // the last one nor come after the first read
      if (z0 + 2 > M - 2 || z0 + 3 >= z1) return false;
    }
  return true;
}

}  // namespace acm
