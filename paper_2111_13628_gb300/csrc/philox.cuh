// Philox4x32-10 counter-based generator (Salmon, Moraes, Dror, Shaw, "Parallel random
// numbers: as easy as 1, 2, 3", SC'11), written from the published definition: ten rounds;
// a round multiplies counter words 0 and 2 by 0xD2511F53 and 0xCD9E8D57, and the new counter
// is (hi(M1*c2) ^ c1 ^ k0, lo(M1*c2), hi(M0*c0) ^ c3 ^ k1, lo(M0*c0)); the key is bumped by
// the Weyl constants 0x9E3779B9 and 0xBB67AE85 between rounds.
#pragma once
#include <stdint.h>

namespace nmc {

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    if (round > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c.x;
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

// The blocks of a sweep's attempts, counters (v, t, g, tag) for many v and few (t, g), from the
// point where the two meet. Round 1 multiplies v and g apart and round 2 multiplies one word that
// depends on (t, g) only and one that depends on v only, so a PhiloxRow per (t, g) and a PhiloxCol
// per v hold everything up to there and a block starts at round 3: eight rounds instead of ten
// and, for the eight blocks of an attempt, 40 of 320 products and 40 of 240 logic operations less.
struct PhiloxRow {
  uint32_t u, v, w;
};
struct PhiloxCol {
  uint32_t a, y, w;
};

__device__ __forceinline__ PhiloxRow philox_row(uint32_t t, uint32_t g, uint32_t k0, uint32_t k1) {
  const uint32_t x = __umulhi(0xCD9E8D57u, g) ^ t ^ k0;  // round 1, word 0
  PhiloxRow r;
  r.u = 0xCD9E8D57u * g ^ (k0 + 0x9E3779B9u);
  r.v = __umulhi(0xD2511F53u, x) ^ (k1 + 0xBB67AE85u);
  r.w = 0xD2511F53u * x;
  return r;
}

__device__ __forceinline__ PhiloxCol philox_col(uint32_t v, uint32_t tag, uint32_t k1) {
  const uint32_t z = __umulhi(0xD2511F53u, v) ^ tag ^ k1;  // round 1, word 2
  PhiloxCol c;
  c.a = __umulhi(0xCD9E8D57u, z);
  c.y = 0xCD9E8D57u * z;
  c.w = 0xD2511F53u * v;
  return c;
}

// Rounds 3..10 of the block of (row, col): equal to philox4x32_10(make_uint4(v, t, g, tag), k0, k1).
__device__ __forceinline__ uint4 philox4x32_meet(const PhiloxRow &r, const PhiloxCol &c, uint32_t k0,
                                                 uint32_t k1) {
  uint4 s = make_uint4(c.a ^ r.u, c.y, r.v ^ c.w, r.w);
  k0 += 0x9E3779B9u;
  k1 += 0xBB67AE85u;
#pragma unroll
  for (int round = 2; round < 10; ++round) {
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
    const uint32_t lo0 = 0xD2511F53u * s.x;
    const uint32_t hi0 = __umulhi(0xD2511F53u, s.x);
    const uint32_t lo1 = 0xCD9E8D57u * s.z;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, s.z);
    s = make_uint4(hi1 ^ s.y ^ k0, lo1, hi0 ^ s.w ^ k1, lo0);
  }
  return s;
}

__device__ __forceinline__ uint32_t uint4_word(const uint4 &u, int j) {
  return j == 0 ? u.x : (j == 1 ? u.y : (j == 2 ? u.z : u.w));
}

}  // namespace nmc
