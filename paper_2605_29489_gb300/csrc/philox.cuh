// Philox4x32-10 counter-based generator (Salmon, Moraes, Dror and Shaw, "Parallel random
// numbers: as easy as 1, 2, 3", SC 2011), written from the published round function:
// each round multiplies counter words 0 and 2 by 0xD2511F53 and 0xCD9E8D57 (32x32->64),
// mixes the high halves with words 1 and 3 and the round key, and the key (k0, k1) is
// bumped by the Weyl constants 0x9E3779B9 and 0xBB67AE85 between rounds.
//
// The counters of a DARE mask are (g low, g high, i, tag) for 8-element group g of expert i.
// Round 1 multiplies only g low (the same for every expert) and i (the same for every group),
// and of round 2's two products one still depends on g alone and the other on (g high, i) alone.
// So the first two rounds are done once per group and once per expert, and a (group, expert)
// pair starts at round 3 with two XORs: 8 rounds instead of 10.  (The compiler hoisted the
// group's share out of a loop over experts by itself; the expert's share it made anew for every
// vector.)  A product is one widening multiply, 64 lanes per clock and SM; the high half alone
// runs at 32.
#pragma once

#include <stdint.h>

namespace mp {

struct Philox4 {
  uint32_t w[4];
};

constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

__device__ __forceinline__ void philox_mul(uint32_t m, uint32_t x, uint32_t& lo, uint32_t& hi) {
  asm("{\n .reg .b64 t;\n mul.wide.u32 t, %2, %3;\n mov.b64 {%0, %1}, t;\n}" : "=r"(lo), "=r"(hi) : "r"(m), "r"(x));
}

// what counter word 0 (g low) and word 3 (the tag) put into the state after two rounds
struct PhiloxGroup {
  uint32_t x0, x1, x2;
};
// what counter words 1 and 2 (g high, expert) put into it
struct PhiloxExpert {
  uint32_t x0, x2, x3;
};

// rk[r] = (k0 + r*0x9E3779B9, k1 + r*0xBB67AE85) for r = 0..9, the round keys: they do not
// depend on the counter, so a kernel takes them precomputed from its launch parameters
__device__ __forceinline__ PhiloxGroup philox_group(uint32_t g_lo, uint32_t tag, const uint32_t (&rk)[10][2]) {
  uint32_t lo0, hi0;
  philox_mul(kPhiloxM0, g_lo, lo0, hi0);
  PhiloxGroup a;
  philox_mul(kPhiloxM1, hi0 ^ tag ^ rk[0][1], a.x1, a.x0);
  a.x0 ^= rk[1][0];
  a.x2 = lo0 ^ rk[1][1];
  return a;
}

__device__ __forceinline__ PhiloxExpert philox_expert(uint32_t g_hi, uint32_t i, const uint32_t (&rk)[10][2]) {
  uint32_t hi1;
  PhiloxExpert e;
  philox_mul(kPhiloxM1, i, e.x0, hi1);
  philox_mul(kPhiloxM0, hi1 ^ g_hi ^ rk[0][0], e.x3, e.x2);
  return e;
}

// the generator's output for the counter (g low, g high, i, tag): rounds 3 to 10
__device__ __forceinline__ Philox4 philox_finish(const PhiloxGroup a, const PhiloxExpert e,
                                                 const uint32_t (&rk)[10][2]) {
  uint32_t c0 = a.x0 ^ e.x0, c1 = a.x1, c2 = a.x2 ^ e.x2, c3 = e.x3;
#pragma unroll
  for (int r = 2; r < 10; ++r) {
    uint32_t lo0, hi0, lo1, hi1;
    philox_mul(kPhiloxM0, c0, lo0, hi0);
    philox_mul(kPhiloxM1, c2, lo1, hi1);
    c0 = hi1 ^ c1 ^ rk[r][0];
    c1 = lo1;
    c2 = hi0 ^ c3 ^ rk[r][1];
    c3 = lo0;
  }
  return Philox4{{c0, c1, c2, c3}};
}

}  // namespace mp
