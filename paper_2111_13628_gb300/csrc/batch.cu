// Batched k-SAT sweep: one persistent launch runs many replica sets of uneven instances
// (sampling stage of Algorithm 1 for many problems at once).
//
// Work item = (replica set, word w of 32 replicas, sweep range). A cluster of CS CTAs takes
// items from a device counter; each CTA loads the item's word vector x[0..n) into its shared
// memory, runs the sweeps with the variables of one colour class spread over the cluster's
// threads (one thread per variable, or a team of 4 or 8 lanes where a class has few variables on a
// CTA, for the 32 replicas of the word), stores every new word into all CS copies, and meets the
// other CTAs between classes. Words are independent chains, so no grid-wide synchronisation is
// needed and uneven instances fill the GPU. The dynamics are identical to the single-instance
// kernels. Occurrence lists are read in a warp-interleaved layout (one coalesced load per
// occurrence for 32 variables); a thread of the one-thread kernel keeps its share of the sweep's
// energy change as 16 bit-sliced planes and converts them to per-replica sums once per sweep.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdlib>
#include <map>
#include <mutex>

#include "nmc.h"
#include "nmc_internal.h"
#include "bits.cuh"
#include "philox.cuh"

namespace cg = cooperative_groups;

namespace nmc {

namespace {

// One-thread kernel for k <= 4: 16 warps, up to 128 registers (no spills; a DSatur colour class
// of the 50,000-variable bench instance puts at most ~490 variables on each CTA of a 4-CTA
// cluster, one round of 512 threads; 640 threads with 96 registers spill 200 bytes: 44.5 ms per 200
// sweeps against 36.4). For k <= 8 (two int4 list entries per occurrence, twice the
// prefetched registers) 12 warps with up to 168 registers, so that nothing spills.
template <int KQ>
__host__ __device__ constexpr int one_thread_threads() {
  return KQ == 1 ? 512 : 384;
}
constexpr int kTeamThreads = 384;   // team kernel with teams of 4: 12 warps, up to 168 registers
constexpr int kTeam8Threads = 512;  // team kernel with teams of 8, k <= 4: up to 128 registers

// Threads of the sweep kernel with TL lanes per variable: 384 for teams of 4, which hold four to
// eight of their list entries per lane, and for teams of 8 with two int4 per occurrence (512 threads
// spilled 400 bytes); 512 for teams of 8 with k <= 4; single threads as one_thread_threads.
template <int KQ, int TL>
__host__ __device__ constexpr int sweep_threads() {
  return (TL == 4 || (TL == 8 && KQ == 2)) ? kTeamThreads
                                           : (TL == 8 ? kTeam8Threads : one_thread_threads<KQ>());
}

template <int NB>
__device__ __forceinline__ void csa4(uint32_t (&c)[NB], uint32_t a0, uint32_t a1, uint32_t a2,
                                     uint32_t a3) {
  const uint32_t s1 = c[0] ^ a0 ^ a1;
  const uint32_t y1 = maj3b(c[0], a0, a1);
  const uint32_t s2 = s1 ^ a2 ^ a3;
  const uint32_t y2 = maj3b(s1, a2, a3);
  c[0] = s2;
  const uint32_t s3 = c[1] ^ y1 ^ y2;
  uint32_t carry = maj3b(c[1], y1, y2);
  c[1] = s3;
#pragma unroll
  for (int j = 2; j < NB; ++j) {
    const uint32_t t = c[j] & carry;
    c[j] ^= carry;
    carry = t;
  }
}

// Adds a0..a3 into the weight-1 and weight-2 planes c[0], c[1] of a bit-sliced counter and
// returns the weight-4 carry, which the caller adds from plane 2 up.
template <int NB>
__device__ __forceinline__ uint32_t csa4_low(uint32_t (&c)[NB], uint32_t a0, uint32_t a1,
                                             uint32_t a2, uint32_t a3) {
  const uint32_t s1 = c[0] ^ a0 ^ a1;
  const uint32_t y1 = maj3b(c[0], a0, a1);
  c[0] = s1 ^ a2 ^ a3;
  const uint32_t y2 = maj3b(s1, a2, a3);
  const uint32_t s3 = c[1] ^ y1 ^ y2;
  const uint32_t f = maj3b(c[1], y1, y2);
  c[1] = s3;
  return f;
}

// c += f * 4 (f one bit per replica), carries rippled up to the top plane.
template <int NB>
__device__ __forceinline__ void add_carry(uint32_t (&c)[NB], uint32_t f) {
#pragma unroll
  for (int j = 2; j < NB; ++j) {
    const uint32_t t = c[j] & f;
    c[j] ^= f;
    f = t;
  }
}

// c += (f + g) * 4: a full adder at plane 2, then one ripple from plane 3.
template <int NB>
__device__ __forceinline__ void add_carry_pair(uint32_t (&c)[NB], uint32_t f, uint32_t g) {
  const uint32_t s = c[2] ^ f ^ g;
  uint32_t carry = maj3b(c[2], f, g);
  c[2] = s;
#pragma unroll
  for (int j = 3; j < NB; ++j) {
    const uint32_t t = c[j] & carry;
    c[j] ^= carry;
    carry = t;
  }
}

constexpr int kAccPlanes = 16;  // per-thread energy accumulator: 16-bit two's complement

// k <= 4 entries of the interleaved lists: literal words by byte offset into the word vector
// (which starts at the beginning of dynamic shared memory); sign i is bit 7 of byte i of the
// first field, turned into an all-zeros / all-ones mask.
__device__ __forceinline__ uint32_t xs_at(const uint32_t *xs, int byte_off) {
  return *reinterpret_cast<const uint32_t *>(reinterpret_cast<const char *>(xs) + byte_off);
}

// prmt with the top bit of every selector nibble set replicates the sign (bit 7) of byte I of
// sg into all four result bytes: one instruction per mask.
template <int I>
__device__ __forceinline__ uint32_t sign_mask(uint32_t sg) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(sg), "r"(0u), "n"(0x8888 + 0x1111 * I));
  return r;
}

// Byte b (0..3) of x, zero-extended.
__device__ __forceinline__ uint32_t byte_of(uint32_t x, int b) {
  return __byte_perm(x, 0u, 0x4440u + (uint32_t)b);
}

// Table index of an uphill move: (b dE) >> 8 clamped to tab_len, whose entry is 0. With b at most
// tab_len << 8 (a larger inverse temperature rejects every uphill move all the same) the product of
// b and a byte stays below 2^32: one product, one shift, one minimum. For dE <= 0 (bytes 0 and
// 128..255) the index is in range and meaningless: those replicas accept whatever the table says.
__device__ __forceinline__ uint32_t table_index(uint32_t b, uint32_t de, int tab_len) {
  return min((b * de) >> 8, (uint32_t)tab_len);
}

// Inverse temperature of a replica with multiplier m: min(2^32 - 1, (m bq) >> 16), clamped for
// table_index.
__device__ __forceinline__ uint32_t pt_beta(uint32_t m, uint32_t bq, int tab_len) {
  const uint32_t lo = m * bq, hi = __umulhi(m, bq);
  const uint32_t cap = (uint32_t)tab_len << 8;
  return hi >> 16 ? cap : min(__funnelshift_r(lo, hi, 16), cap);
}

// The sweep's Philox rows (one per group of 4 replicas of the word), in shared memory.
struct SweepRows {
  uint2 vw[8];
  uint32_t u[8];
  __device__ __forceinline__ PhiloxRow at(int g) const {
    const uint2 x = vw[g];
    return PhiloxRow{u[g], x.x, x.y};
  }
  // written by threads 0..7 for sweep t; a barrier lies between this and the readers on both sides
  __device__ __forceinline__ void fill(const BatchItem &B, int t) {
    if (threadIdx.x < 8) {
      const PhiloxRow r = philox_row((uint32_t)t, (uint32_t)(8 * B.w) + threadIdx.x, B.k0, B.k1);
      vw[threadIdx.x] = make_uint2(r.v, r.w);
      u[threadIdx.x] = r.u;
    }
  }
};

// ORs over the other literals of N slots' clauses of their truth values (32 replicas), from the slots'
// entries: {sign bits, byte offsets of literals 1..3}; for k > 4 also {byte offsets of literals
// 4..7}, whose signs sit in bit 6 of bytes 0..3 of the sign word (shifted up to bit 7 here). few: no
// clause of the formula has more than six literals, so literals 6 and 7 are always false.
template <int KQ, int N>
__device__ __forceinline__ void others_or(const uint32_t *xs, const int4 (&q)[N * KQ], bool few,
                                          uint32_t (&o)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int4 &a = q[j * KQ];
    const uint32_t sg = (uint32_t)a.x;
    o[j] = (xs_at(xs, a.y) ^ sign_mask<1>(sg)) | (xs_at(xs, a.z) ^ sign_mask<2>(sg)) |
           (xs_at(xs, a.w) ^ sign_mask<3>(sg));
    if (KQ == 2) {
      const int4 &b = q[j * KQ + KQ - 1];
      o[j] |= (xs_at(xs, b.x) ^ sign_mask<0>(sg << 1)) | (xs_at(xs, b.y) ^ sign_mask<1>(sg << 1));
    }
  }
  if (KQ == 2 && !few) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int4 &b = q[j * KQ + KQ - 1];
      const uint32_t s6 = (uint32_t)q[j * KQ].x << 1;
      o[j] |= (xs_at(xs, b.z) ^ sign_mask<2>(s6)) | (xs_at(xs, b.w) ^ sign_mask<3>(s6));
    }
  }
}

// The loads of one attempt that do not depend on the replicas' states: the variable's Q16
// inverse temperature, its list length and its first group of occurrence entries. A thread
// requests them for its next variable before it waits at the barrier that ends the current
// colour class, so their L2 / HBM latency overlaps the barrier.
template <int KQ>
struct AttemptPrep {
  int4 q[4 * KQ];
  const int4 *ent;
  int len;
  int regions;  // of the variable's group: region_pre, region_few
  uint32_t bq;
  uint32_t vo;  // original id
};

// What is kept of a group beside its list: slots from `pre` on may hold literals of the previous
// colour class, those below do not.
__device__ __forceinline__ int region_pre(int r) { return r & 0xFFFF; }
// k > 4: no clause of the formula has more than six literals
__device__ __forceinline__ bool region_few(int r) { return (r >> 30) & 1; }

// v = c0 + off is a variable of colour class c (starting at new id c0; cg: the class's first
// group of 32 variables), attempted at sweep t.
template <int KQ>
__device__ __forceinline__ void prep_attempt(const BatchItem &B, int cg, int c0, int v, int t,
                                             AttemptPrep<KQ> &p) {
  p.bq = __ldg(B.bq + (size_t)t * B.n + v);
  p.vo = (uint32_t)__ldg(B.orig + v);
  const int off = v - c0;
  const int g = cg + (off >> 5), ln = off & 31;
  const int gb = __ldg(B.grp_base + g);
  p.len = (__ldg(B.grp_base + g + 1) - gb) / (32 * KQ);
  p.ent = B.occ_t + gb + ln;
  p.regions = __ldg(B.grp_base + B.n_groups + 1 + g);
  if (p.len > 0) {
#pragma unroll
    for (int j = 0; j < 4 * KQ; ++j) p.q[j] = __ldg(p.ent + (size_t)j * 32);
  }
}

// Bit-sliced counters of one attempt.
// One counter. With z = "every other literal of the clause false", a replica's energy change
// is x ? Zp - Zn : Zn - Zp, Zp / Zn counting z over the occurrences whose own literal is positive /
// negated. Counting z over the first and not z over the second gives Zp - Zn + K, K the lane's
// number of slots counted as negated, so a counter that starts at -K ends at Zp - Zn (8 planes, two's
// complement). K sits in free bits of the lane's first sign word: the low 7 bits (k <= 4), or the low
// 6 bits of byte 1 and bit 16 (k > 4).
template <int KQ>
__device__ __forceinline__ uint32_t marked_slots(uint32_t sg) {  // K, from the first sign word
  return KQ == 1 ? sg & 0x7Fu : ((sg >> 8) & 0x3Fu) | ((sg >> 10) & 0x40u);
}
template <int KQ>
struct Counts {
  uint32_t c[8];
  __device__ __forceinline__ void start(const AttemptPrep<KQ> &P) {
    const uint32_t k = P.len > 0 ? 0u - marked_slots<KQ>((uint32_t)P.q[0].x) : 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j) c[j] = (uint32_t)((int)(k << (31 - j)) >> 31);
  }
  // planes of dE for the variable's word x
  __device__ __forceinline__ void change(uint32_t x, uint32_t (&d)[8]) const {
    uint32_t carry = ~x;  // negated where x = 0
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      d[j] = (c[j] ^ ~x) ^ carry;
      carry = (c[j] ^ ~x) & carry;
    }
  }
};

// Requests the entries of slots e .. e + 3 of the list.
template <int KQ>
__device__ __forceinline__ void load_slots(const int4 *ent, int e, int4 (&q)[4 * KQ]) {
#pragma unroll
  for (int j = 0; j < 4 * KQ; ++j) q[j] = __ldg(ent + (size_t)(e * KQ + j) * 32);
}

// What N slots add to the counter: z, complemented where the own literal is negated.
template <int KQ, int N>
__device__ __forceinline__ void slot_masks(const uint32_t *xs, const int4 (&q)[N * KQ], bool few,
                                           uint32_t (&z)[N]) {
  others_or<KQ, N>(xs, q, few, z);
#pragma unroll
  for (int j = 0; j < N; ++j) z[j] = ~z[j] ^ sign_mask<0>((uint32_t)q[j * KQ].x);
}

// Adds slots [e0, e1) (multiples of 4) of the variable's list to the counters; P.q holds the
// entries of slot e0's group on entry and those of slot e1's on return (while there are any).
// Two groups of 4 a trip, without a branch between them: each group's weight-4 carry is kept aside and
// the pair's carries enter the planes from weight 4 up together, and the entries of a group are
// requested into the other of two buffers while the group before it is evaluated, so the L2 latency of
// the list overlaps the shared-memory gathers and counting and no entry is copied. (Counting slots
// whose own signs agree in all lanes without the sign mask saves one instruction in such a slot, and
// its three-way branch per group costs more: 36.4 -> 35.9 ms without it, 4-SAT, 50,000 variables, 1,024
// replicas, 200 sweeps; 24 uneven 3-/4-SAT sets 12.1 -> 11.8.)
template <int KQ>
__device__ __forceinline__ void count_slots(const uint32_t *xs, AttemptPrep<KQ> &P, int e0, int e1,
                                            Counts<KQ> &C) {
  const int len = P.len;
  const int4 *ent = P.ent;
  int4 qb[4 * KQ];
  const bool few = region_few(P.regions);
  const auto count4 = [&](const int4 (&q)[4 * KQ]) {
    uint32_t z[4];
    slot_masks<KQ, 4>(xs, q, few, z);
    return csa4_low<8>(C.c, z[0], z[1], z[2], z[3]);
  };
#pragma unroll 1
  for (int e = e0; e < e1; e += 8) {
    if (e + 4 < len) load_slots<KQ>(ent, e + 4, qb);
    const uint32_t f = count4(P.q);
    if (e + 4 < e1) {
      if (e + 8 < len) load_slots<KQ>(ent, e + 8, P.q);
      add_carry_pair<8>(C.c, f, count4(qb));
    } else {
      add_carry<8>(C.c, f);
#pragma unroll
      for (int j = 0; j < 4 * KQ; ++j) P.q[j] = qb[j];
    }
  }
}

// Acceptance of the variable with original id vo at the sweep of `rows` for the 32 replicas of the
// word, from the counters of its whole list; returns its new word. The table index from one product,
// the eight-word transpose and the Philox blocks from their third round on took 200 sweeps of the
// 50,000-variable bench instance with 1,024 replicas from 43.94 to 41.90 ms, 24 uneven 3-/4-SAT sets
// from 16.96 to 15.75 per 100 (37.9 and 12.0 with all later steps). With PT, replica j of the word moves at min(2^32-1,
// (mult_s[j] * bq) >> 16) instead of bq.
template <int KQ, bool PT>
__device__ __forceinline__ uint32_t accept_batch(const BatchItem &B, const uint32_t *tab_s,
                                                 int tab_len, const uint32_t *mult_s,
                                                 const SweepRows &rows, uint32_t vo, uint32_t x,
                                                 uint32_t bqv, const Counts<KQ> &C,
                                                 uint32_t (&acc)[kAccPlanes]) {
  uint32_t s8[8];
  C.change(x, s8);
  const PhiloxCol col = philox_col(vo, kTagKsatSweep, B.k1);
  const uint32_t bqc = min(bqv, (uint32_t)tab_len << 8);
  // replicas whose dE <= 0 (sign plane set, or every plane zero) accept without a draw
  uint32_t flip = s8[7] | ~(s8[0] | s8[1] | s8[2] | s8[3] | s8[4] | s8[5] | s8[6]);
  uint32_t de[8];  // byte q of de[j]: the dE of replica 8q + j
#pragma unroll
  for (int j = 0; j < 8; ++j) de[j] = s8[j];
  transpose8x32(de);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    // replicas 8q .. 8q+7: Philox groups 2q and 2q+1, drawn together and always (a draw that
    // cannot change an acceptance changes nothing; a branch on whether any lane needs one rarely
    // skips the work for the whole warp and keeps the four pairs from overlapping: 236.5 -> 225.7
    // us per sweep on the 50,000-variable bench instance)
    uint32_t th[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t b = PT ? pt_beta(mult_s[8 * q + j], bqv, tab_len) : bqc;
      th[j] = tab_s[table_index(b, byte_of(de[j], q), tab_len)];
    }
    const uint4 u0 = philox4x32_meet(rows.at(2 * q), col, B.k0, B.k1);
    const uint4 u1 = philox4x32_meet(rows.at(2 * q + 1), col, B.k0, B.k1);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t u = j < 4 ? uint4_word(u0, j) : uint4_word(u1, j - 4);
      flip |= (uint32_t)(u < th[j]) << (8 * q + j);
    }
  }
  // energy bookkeeping: acc += D on the flipped replicas (bit-sliced, sign-extended add)
  {
    uint32_t carry = 0u;
#pragma unroll
    for (int j = 0; j < kAccPlanes; ++j) {
      const uint32_t b = s8[j < 8 ? j : 7] & flip;
      const uint32_t a = acc[j];
      acc[j] = a ^ b ^ carry;
      carry = maj3b(a, b, carry);
    }
  }
  return x ^ flip;
}

// A colour class [c0, c1) is shared out among the CS CTAs of a cluster by 32-variable groups,
// round-robin: CTA `rank` takes groups rank, rank + CS, ... Variables are degree-descending
// inside a class, so each CTA gets a like mix of long and short occurrence lists (contiguous
// shares would give rank 0 all the longest lists and make every class wait for it).
template <int CS>
__device__ __forceinline__ int share_count(int c0, int c1, int rank) {
  const int ng = (c1 - c0 + 31) >> 5;
  const int mine = ng > rank ? (ng - rank + CS - 1) / CS : 0;
  int cnt = mine * 32;
  if (mine > 0 && rank + (mine - 1) * CS == ng - 1) cnt -= ng * 32 - (c1 - c0);  // last, partial
  return cnt;
}

// Local index li (0 <= li < share_count) -> variable.
template <int CS>
__device__ __forceinline__ int share_var(int c0, int rank, int li) {
  return c0 + 32 * (rank + CS * (li >> 5)) + (li & 31);
}

// Synchronises the CS CTAs of a cluster (or the CTA when CS = 1); cluster barriers are
// hardware barriers with release/acquire semantics for distributed shared memory.
template <int CS>
__device__ __forceinline__ void group_sync() {
  if (CS == 1) {
    __syncthreads();
  } else {
    cg::this_cluster().sync();
  }
}

// The cluster barrier in two halves: arrive (releasing this thread's earlier shared-memory
// stores to the cluster) and wait (acquiring everyone's). Work between the two halves overlaps
// the barrier; it must not touch shared memory that other CTAs read before the wait.
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t shared_at(uint32_t saddr, int rank) {  // the same word of a CTA
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(saddr), "r"(rank));
  return ra;
}

template <int CS, typename T>
__device__ __forceinline__ T *rank_ptr(T *p, int r) {
  if (CS == 1) return p;
  return cg::this_cluster().map_shared_rank(p, r);
}

// ---- what both sweep kernels share --------------------------------------------------------------

// Static shared memory of a sweep kernel.
struct SweepShared {
  BatchItem item;   // the current item, read from here where needed
  int ep[2][32];    // energy changes of the even and odd sweeps, per replica
  uint32_t mult[32];  // temperature multipliers (replica exchange)
  SweepRows rows;
  uint32_t improved;  // replicas that improved in the last sweep
  int next;           // index of the current item
  unsigned long long full[2];  // CS > 1: barriers of the even and odd class steps (ClassBarrier)
};

// Energies of the word's replicas, kept by warp 0 of every CTA (its lane's replica), and the
// replicas that improved during the item.
struct EnergyTrack {
  int e, best;
  long long s1, s2;  // sums of E and E^2 of the sampled sweeps
  uint32_t m_item;
};

// The barrier between colour classes in two halves: a thread arrives once its own words of the class
// are stored, and waits only before its first read of that class.
//
// One CTA: its stores need ordering among its threads only, so it fences at CTA scope and arrives
// relaxed at the hardware barrier (512 threads, a round: 120 cycles; 505 with the cluster release,
// 85 for __syncthreads, which cannot be split).
//
// Several CTAs: a release at cluster scope waits for all remote stores, 300 cycles at the least and
// 1,000 - 1,700 in a sweep. Instead every new word is an asynchronous store that counts its bytes at
// the receiving CTA's mbarrier (st.async), for the class step's parity. A step of a CTA completes
// when all words of the class have arrived there, all its own warps have (none can miss a step), and
// one warp of every CTA has (so that no CTA, also one without a variable in the class, is passed by
// more than a step and a barrier never counts two steps at once). Words overwritten by a CTA that is
// a step ahead are words nobody reads any more: every warp with a variable in the class has stored it,
// hence finished reading, and warps counting ahead read neither their own class nor the one before.
// The last class of a sweep meets at the hardware cluster barrier, which also publishes the CTAs'
// energy changes.
//
// A wait gives up after about a second. Its warp is `dead` from then on: it marks the set at hand and
// that of every later item of the launch (kStepTimeout at the end of best_energy), runs through
// without waiting, and leaves the mbarriers alone, whose phases it no longer follows: its words are
// plain stores, and the warps that wait for it give up as well.
constexpr long long kStepLimitCycles = 1ll << 31;
constexpr long long kDrainCycles = 1ll << 21;  // a millisecond: hundreds of times what a store takes

template <int CS, int WARPS>
struct ClassBarrier {
  uint32_t bar;                 // shared address of full[0]
  uint32_t arrived, waited;     // steps at the mbarriers so far
  bool dead;                    // of the warp: a wait has given up
  long long limit;

  // by all threads, before a barrier of the CTAs
  __device__ __forceinline__ void init(SweepShared &sh, long long limit_cycles = kStepLimitCycles) {
    bar = (uint32_t)__cvta_generic_to_shared(&sh.full[0]);
    arrived = waited = 0;
    dead = false;
    limit = limit_cycles;
    if (CS > 1 && threadIdx.x == 0) {
      for (int i = 0; i < 2; ++i)
        asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(bar + 8 * i), "r"(WARPS + CS) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  __device__ __forceinline__ static void mark(const BatchItem &B) { B.best_energy[32 * B.W] = kStepTimeout; }
  // Before the first class of an item.
  __device__ __forceinline__ void begin(const BatchItem &B) const {
    if (CS > 1 && dead) mark(B);
  }
  // After the barrier of the CTAs that ends an item; the CTAs meet again before any of them exits.
  // A dead warp holds them until the cluster's asynchronous stores, which nobody waits for any more,
  // have arrived in shared memory that is still there.
  __device__ __forceinline__ void drain() const {
    if (CS > 1 && dead) {
      const long long t0 = clock64();
      while (clock64() - t0 < kDrainCycles) {
      }
    }
  }
  // Stores v at word `saddr` of CTA `rank`, as part of the step being worked on.
  __device__ __forceinline__ void store(uint32_t saddr, int rank, uint32_t v, bool last) const {
    if (last || dead)
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(shared_at(saddr, rank)), "r"(v) : "memory");
    else
      asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(
                       shared_at(saddr, rank)),
                   "r"(v), "r"(shared_at(bar + 8 * (arrived & 1), rank))
                   : "memory");
  }
  // The warp has stored its words of the class (n_words in all CTAs together).
  __device__ __forceinline__ void arrive(int n_words, bool last) {
    __syncwarp();
    if (CS == 1) {
      __threadfence_block();
      asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    } else if (last) {
      cluster_arrive();
    } else {
      const int lane = threadIdx.x & 31;
      const uint32_t b = bar + 8 * (arrived & 1);
      ++arrived;
      if (dead) return;
      if (threadIdx.x < CS)
        asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                         shared_at(b, threadIdx.x))
                     : "memory");
      if (threadIdx.x == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(4 * n_words)
                     : "memory");
      else if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(b) : "memory");
    }
  }
  // Waits for the class before the one at hand (last: the sweep's last one).
  __device__ __forceinline__ void wait(const BatchItem &B, bool last) {
    __syncwarp();
    if (CS == 1 || last) {
      cluster_wait();
      return;
    }
    const uint32_t b = bar + 8 * (waited & 1), parity = (waited >> 1) & 1;
    ++waited;
    if (dead) return;
    uint32_t done = 0;
    long long t0 = 0;
    while (true) {
      asm volatile(
          "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
          "selp.u32 %0, 1, 0, p;\n}"
          : "=r"(done)
          : "r"(b), "r"(parity)
          : "memory");
      if (done) break;
      if (t0 == 0) t0 = clock64();
      if (clock64() - t0 > limit) {
        dead = true;
        mark(B);
        break;
      }
    }
    dead = __any_sync(0xFFFFFFFFu, dead);
  }
};

// Takes the next item from the counter into sh.item; false when there is none left.
template <int CS>
__device__ __forceinline__ bool next_batch_item(const BatchItem *items, int n_items, int *next_item,
                                                int rank, SweepShared &sh) {
  if (rank == 0 && threadIdx.x == 0) sh.next = atomicAdd(next_item, 1);
  group_sync<CS>();
  const int it = *rank_ptr<CS>(&sh.next, 0);
  if (it < n_items && threadIdx.x == 0) sh.item = items[it];
  group_sync<CS>();  // every rank has read the item id before any rank moves on or exits
  return it < n_items;
}

// The item's word vector, energies and multipliers into shared memory and registers, and the Philox
// rows of its first sweep. A barrier of the CTAs must follow.
template <int CS, bool PT>
__device__ __forceinline__ void load_item(const BatchItem &B, int rank, uint32_t *xs, SweepShared &sh,
                                          EnergyTrack &k) {
  const int n = B.n, W = B.W, w = B.w;
  for (int v = threadIdx.x; v < n; v += blockDim.x) xs[v] = B.S[(size_t)(2 * v) * W + w];
  if (threadIdx.x == 0) xs[n] = 0u;
  k = EnergyTrack{};
  if (threadIdx.x < 32) {
    sh.ep[0][threadIdx.x] = sh.ep[1][threadIdx.x] = 0;
    if (PT) sh.mult[threadIdx.x] = B.mult[32 * w + threadIdx.x];
    k.e = B.energy[32 * w + threadIdx.x];
    k.best = B.best_energy[32 * w + threadIdx.x];
  }
  sh.rows.fill(B, B.t0);
}

// After the last class of sweep t is published (and with it every CTA's energy changes): energies,
// best energies and, where a replica improved, its state. Every CTA sums the changes itself, so the
// CTAs only meet again when there is a state to copy.
// Best states go to a word-major staging row (the second half of the best buffer) at each improving
// sweep end, and into the [var][word] layout once, at the end of the item: a merge into that layout
// touches one 32-byte sector per variable, which at every improving sweep cost about 30 us per sweep
// on the 50,000-variable bench instance.
template <int CS, bool PT>
__device__ __forceinline__ void end_sweep(const BatchItem &B, int rank, int t, uint32_t *xs,
                                          SweepShared &sh, EnergyTrack &k) {
  const int n = B.n;
  if (threadIdx.x < 32) {
    int sum = k.e;
#pragma unroll
    for (int r = 0; r < CS; ++r) sum += rank_ptr<CS>(&sh.ep[t & 1][0], r)[threadIdx.x];
    k.e = sum;
    if (PT && B.stats && t >= B.stats_t0) {
      k.s1 += sum;
      k.s2 += (long long)sum * sum;
    }
    const bool better = sum < k.best;
    if (better) k.best = sum;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, better);
    if (threadIdx.x == 0) sh.improved = m;
    sh.ep[~t & 1][threadIdx.x] = 0;  // last read before this sweep's class barriers
  }
  sh.rows.fill(B, t + 1);
  __syncthreads();
  const uint32_t m = sh.improved;
  if (m) {
    uint32_t *best_t = B.best + (size_t)n * B.W + (size_t)B.w * n;
    const int share = (n + CS - 1) / CS, b0 = rank * share, b1 = min(n, b0 + share);
    for (int v = b0 + threadIdx.x; v < b1; v += blockDim.x)
      best_t[v] = (best_t[v] & ~m) | (xs[v] & m);
    k.m_item |= m;
    group_sync<CS>();
  }
}

// States, best states and energies of the item back to memory.
template <int CS, bool PT>
__device__ __forceinline__ void store_item(const BatchItem &B, int rank, const uint32_t *xs,
                                           const EnergyTrack &k) {
  const int n = B.n, W = B.W, w = B.w;
  const uint32_t *best_t = B.best + (size_t)n * W + (size_t)w * n;
  const int share = (n + CS - 1) / CS, b0 = rank * share, b1 = min(n, b0 + share);
  for (int v = b0 + threadIdx.x; v < b1; v += blockDim.x) {
    B.S[(size_t)(2 * v) * W + w] = xs[v];
    B.S[(size_t)(2 * v + 1) * W + w] = ~xs[v];
    if (k.m_item) {  // replicas improved during the item: their last best state from staging
      const size_t bi = (size_t)v * W + w;
      B.best[bi] = (B.best[bi] & ~k.m_item) | (best_t[v] & k.m_item);
    }
  }
  if (rank == 0 && threadIdx.x < 32) {
    B.energy[32 * w + threadIdx.x] = k.e;
    B.best_energy[32 * w + threadIdx.x] = k.best;
    if (PT && B.stats) {  // one item per word in a launch: plain read-modify-write
      B.stats[32 * w + threadIdx.x] += k.s1;
      B.stats[32 * (B.W + w) + threadIdx.x] += k.s2;
    }
  }
}

// CS = CTAs per item. With CS > 1 every CTA of the cluster keeps a full copy of the item's
// word vector; each CTA updates its share of every colour class and stores the new words
// into all CS copies (distributed shared memory), then the cluster barrier publishes them.
// PT: every item carries per-replica temperature multipliers and, optionally, accumulates the
// end-of-sweep energies of sweeps t >= stats_t0 (sums of E and E^2 per replica).
template <int KQ, int CS, bool PT>
__global__ void __launch_bounds__(one_thread_threads<KQ>(), 1)
    ksat_batch_kernel(const BatchItem *__restrict__ items, int n_items, int *next_item,
                      const uint32_t *tab, int tab_len, int xs_words, int) {
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t *xs = smem;                               // word vector first (byte offsets in lists)
  uint32_t *tab_s = smem + ((xs_words + 31) & ~31);  // then the acceptance table
  __shared__ SweepShared sh;
  const int rank = CS == 1 ? 0 : (int)cg::this_cluster().block_rank();
  for (int i = threadIdx.x; i <= tab_len; i += blockDim.x) tab_s[i] = i < tab_len ? tab[i] : 0u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ClassBarrier<CS, one_thread_threads<KQ>() / 32> step;
  step.init(sh);
  while (true) {
    if (!next_batch_item<CS>(items, n_items, next_item, rank, sh)) break;
    const BatchItem &B = sh.item;
    EnergyTrack track;
    load_item<CS, PT>(B, rank, xs, sh, track);
    step.begin(B);
    group_sync<CS>();
    for (int t = B.t0; t < B.t1; ++t) {
      uint32_t acc[kAccPlanes];
#pragma unroll
      for (int j = 0; j < kAccPlanes; ++j) acc[j] = 0u;
      // class bounds and first group: those of class c + 1 are requested during class c and
      // arrive behind its barrier
      int c0 = __ldg(B.col_ptr), c1 = __ldg(B.col_ptr + 1), cg = __ldg(B.cgrp);
      constexpr int kThreads = one_thread_threads<KQ>();
      // the state-independent loads of this thread's first variable of each class: requested
      // for class c + 1 between the two halves of the barrier that ends class c
      // (every thread loads, those without a variable in the class for variable c0, so that
      // P is written before every class)
      AttemptPrep<KQ> P;
      // the warp's group of the class's share (its first round): dealt on from class to class,
      // so that the warps left without a group, and those with the longest lists, change
      constexpr int kWarps = kThreads / 32;
      int mygrp = warp;
      {
        const int cnt0 = share_count<CS>(c0, c1, rank);
        const bool mine = (int)threadIdx.x < cnt0;
        prep_attempt<KQ>(B, cg, c0, mine ? share_var<CS>(c0, rank, threadIdx.x) : c0, t, P);
      }
      for (int c = 0; c < B.n_colours; ++c) {
        int c2 = 0, cgn = 0;
        if (c + 1 < B.n_colours) {
          c2 = __ldg(B.col_ptr + c + 2);
          cgn = __ldg(B.cgrp + c + 1);
        }
        // the class's 32-variable groups are dealt round-robin to the cluster's CTAs, and the
        // CTA's share of them to its warps
        const int cnt = share_count<CS>(c0, c1, rank);
        const int ngr = (cnt + 31) >> 5;
        const bool last_class = c + 1 == B.n_colours;
        {
          auto store = [&](int v, uint32_t xn) {
            if (CS == 1) {
              xs[v] = xn;
            } else {
              const uint32_t sa = (uint32_t)__cvta_generic_to_shared(xs + v);
#pragma unroll
              for (int r = 0; r < CS; ++r) step.store(sa, r, xn, last_class);
            }
          };
          // first round: the slots before `pre` are counted before the wait for the previous
          // class, the rest after it; further rounds (more variables than threads) follow it.
          // Warps that are done early, or had no group, so fill the time that the class's slower
          // warps and the barrier take (4-SAT, 50,000 variables, 1,024 replicas, 200 sweeps:
          // 47.05 -> 43.94 ms; 24 uneven 3-/4-SAT sets: 18.06 -> 16.96 ms).
          for (int base = 32 * mygrp, first = 1;; base += kThreads, first = 0) {
            const int li = base + lane;
            int v = li < cnt ? share_var<CS>(c0, rank, li) : c0;
            if (!first) prep_attempt<KQ>(B, cg, c0, v, t, P);
            const bool go = li < cnt && P.bq != kFrozenQ16;  // a held variable takes no attempt
            const uint32_t x = xs[v];
            Counts<KQ> C;
            C.start(P);
#pragma unroll 1
            for (int part = 0; part < 2; ++part) {
              const int pre = region_pre(P.regions);
              if (part == 1 && first && c > 0) step.wait(B, false);
              if (go) count_slots<KQ>(xs, P, part ? pre : 0, part ? P.len : pre, C);
            }
            uint32_t xn = x;
            if (go)
              xn = accept_batch<KQ, PT>(B, tab_s, tab_len, sh.mult, sh.rows, P.vo, x, P.bq, C, acc);
            // every word counts at the receiving barriers, also one that did not change
            if (CS > 1 ? li < cnt : go) store(v, xn);
            if (base + kThreads >= cnt) break;
          }
        }
        if (last_class) {
          // the sweep's energy changes, published with its last class: planes -> 16-bit values (one
          // byte transpose for each half of the planes), then a warp reduction per replica
          uint32_t lo[8], hi[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            lo[j] = acc[j];
            hi[j] = acc[8 + j];
          }
          transpose8x32(lo);
          transpose8x32(hi);
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              // bytes q of lo and hi as one signed 16-bit value, sign-extended
              uint32_t val;
              asm("prmt.b32 %0, %1, %2, %3;"
                  : "=r"(val)
                  : "r"(lo[j]), "r"(hi[j]), "r"(0xCC40u + 0x1111u * (uint32_t)q));
              const int sum = __reduce_add_sync(0xFFFFFFFFu, (int)val);
              if (lane == 0 && sum != 0) atomicAdd(&sh.ep[t & 1][8 * q + j], sum);
            }
        }
        // this CTA's words of the class are published; the next class's loads are requested and
        // its slots before `pre` counted (none holds a literal of this class) before the wait
        step.arrive(c1 - c0, last_class);
        mygrp -= ngr;
        while (mygrp < 0) mygrp += kWarps;
        if (c + 1 < B.n_colours) {
          const int cntn = share_count<CS>(c1, c2, rank), ln = 32 * mygrp + lane;
          prep_attempt<KQ>(B, cgn, c1,
                           ln < cntn ? share_var<CS>(c1, rank, ln) : c1, t, P);
        }
        c0 = c1;
        c1 = c2;
        cg = cgn;
      }
      step.wait(B, true);
      end_sweep<CS, PT>(B, rank, t, xs, sh, track);
    }
    store_item<CS, PT>(B, rank, xs, track);
    group_sync<CS>();
    step.drain();
  }
}

// ---- team kernel: every class with TL lanes per variable ---------------------------------------
//
// For instances whose classes put few variables on a CTA the sweep is a chain of class latencies,
// so whatever does not depend on the previous class is taken off that chain. A warp handles 32 / TL
// variables, and the warps of a CTA are dealt out over consecutive classes. A warp looks up to two
// classes ahead for its next unit and requests that unit's list entries at once (class bounds and
// list positions come from shared memory, so nothing waits); between its arrival at the class before
// and its wait it draws the Philox words of its replicas and counts the slots that hold no literal
// of the class still being updated, summed over the team. After the wait remain the last slots of
// each lane, their sum over the team, the table lookups and the new word.
//
// Lane tl of a team resolves the replicas r = tl + TL k: their dE come out of the bit planes by one
// shift and one masked merge per plane, and one ballot per k gives TL bits of each team's flips.
// The Philox block of replicas 4g .. 4g + 3 is drawn by lane g TL / 8, its words handed round the
// team by shuffles ahead of the wait.

// What it measured (the kernel before it, with every load and draw after the barrier, in brackets):
// N = 200, 64 replicas, one CTA a word, 8 lanes: 24.0 us a sweep (34.5); N = 5,000, 1,024 replicas,
// 4 CTAs, 4 lanes: 61.4 (95.9); 6-SAT N = 8,678, 226 replicas, 8 CTAs, 4 lanes: 185 (334). Clock
// reads at N = 5,000 put 1,000 - 1,700 of a class's 4,400 cycles in the release of the cluster
// barrier, 350 - 500 in the late slots and 350 - 900 in the acceptance.

// Slots per lane behind `pre` that are loaded ahead of the wait; lists with more (few classes) take
// all their slots after it.
template <int TL>
__host__ __device__ constexpr int post_slots() { return 16 / TL; }

// Words of shared memory for the class bounds and list positions of an instance (read from global
// memory where an instance has more).
constexpr int kMetaWords = 4096;

constexpr int kLookAhead = 2;  // classes a warp looks ahead for its next unit

// A warp's next unit and its state-independent loads.
template <int KQ, int TL>
struct TeamPrep {
  int c, t;                   // class and sweep of the unit, or of the class to look on from
  bool work;                  // a unit
  int v0, c0, c1, cg, units;  // the CTA's share of that class
  const int4 *ent;  // the lane's column of its group's interleaved list
  int len, pre, regions;
  bool late;
  uint32_t bq, vo, first;  // first: the first slot's sign word
  // k <= 4: the lane's first slots before and behind `pre` (two entries per slot would not fit)
  int4 q[KQ == 1 ? 4 : 1], qp[KQ == 1 ? post_slots<TL>() : 1];
};

// Adds the other lanes' counters of the team (A planes) in a butterfly: one plane more per stage,
// at most 8 (two's complement).
template <int TL, int A, int S = 1>
__device__ __forceinline__ void team_sum(uint32_t (&c)[8]) {
  if constexpr (S < TL) {
    constexpr int N = A < 8 ? A + 1 : 8;
    uint32_t p[A];
#pragma unroll
    for (int j = 0; j < A; ++j) p[j] = __shfl_xor_sync(0xFFFFFFFFu, c[j], S);
    uint32_t carry = 0u;
#pragma unroll
    for (int j = 0; j < A; ++j) {
      const uint32_t a = c[j];
      c[j] = a ^ p[j] ^ carry;
      carry = maj3b(a, p[j], carry);
    }
    if constexpr (A < 8) c[A] = carry;
    team_sum<TL, N, 2 * S>(c);
  }
}

template <int KQ, int CS, int TL, bool PT>
__global__ void __launch_bounds__(sweep_threads<KQ, TL>(), 1)
    ksat_team_kernel(const BatchItem *__restrict__ items, int n_items, int *next_item,
                     const uint32_t *tab, int tab_len, int xs_words, int meta_words) {
  constexpr int kThreads = sweep_threads<KQ, TL>(), kWarps = kThreads / 32;
  constexpr int VPW = 32 / TL;        // variables of a warp
  constexpr int RPL = 32 / TL;        // replicas of a lane
  constexpr int POST = post_slots<TL>();
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t *xs = smem;                               // word vector first (byte offsets in lists)
  uint32_t *tab_s = smem + ((xs_words + 31) & ~31);  // then the acceptance table
  int *meta = reinterpret_cast<int *>(tab_s + tab_len + 1);  // then class bounds, list positions
  __shared__ SweepShared sh;
  const int rank = CS == 1 ? 0 : (int)cg::this_cluster().block_rank();
  for (int i = threadIdx.x; i <= tab_len; i += blockDim.x) tab_s[i] = i < tab_len ? tab[i] : 0u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tl = lane % TL, team = lane / TL;
  ClassBarrier<CS, kWarps> step;
  step.init(sh);
  while (true) {
    if (!next_batch_item<CS>(items, n_items, next_item, rank, sh)) break;
    const BatchItem &B = sh.item;
    const int n = B.n, W = B.W, w = B.w;
    const int32_t inert_off = n * 4;
    EnergyTrack track;
    load_item<CS, PT>(B, rank, xs, sh, track);
    step.begin(B);
    uint32_t pm[PT ? RPL : 1];  // the lane's replicas' temperature multipliers
    if (PT) {
#pragma unroll
      for (int k = 0; k < RPL; ++k) pm[k] = B.mult[32 * w + tl + TL * k];
    }
    // [v0, v0 + n_units * VPW) of class [c0, c1): the CTA's contiguous share, in warp-sized units
    auto share_of = [&](int c0, int c1, int &v0) {
      const int part = ((c1 - c0 + CS - 1) / CS + VPW - 1) / VPW * VPW;
      v0 = c0 + rank * part;
      return max(0, (min(c1, v0 + part) - v0 + VPW - 1) / VPW);
    };
    const int nc = B.n_colours, G = B.n_groups;
    const int32_t *col_ptr = B.col_ptr, *cgrp = B.cgrp, *grp = B.grp_base;
    const bool staged = 2 * (nc + 1) + 2 * G + 1 <= meta_words;
    if (staged) {
      for (int i = threadIdx.x; i <= nc; i += blockDim.x) {
        meta[i] = col_ptr[i];
        meta[nc + 1 + i] = cgrp[i];
      }
      for (int i = threadIdx.x; i <= 2 * G; i += blockDim.x) meta[2 * (nc + 1) + i] = grp[i];
      col_ptr = meta;
      cgrp = meta + nc + 1;
      grp = meta + 2 * (nc + 1);
    }
    __syncthreads();
    TeamPrep<KQ, TL> P{};
    auto load_slot = [&](int j, int end, int4 &q, int4 &q2) {
      if (j < end) {
        q = __ldg(P.ent + (size_t)(j * KQ) * 32);
        if (KQ == 2) q2 = __ldg(P.ent + (size_t)(j * KQ + 1) * 32);
      } else {  // inert: literal 1 always true
        q = make_int4(1 << 15, inert_off, inert_off, inert_off);
        if (KQ == 2) q2 = make_int4(inert_off, inert_off, inert_off, inert_off);
      }
    };
    // requests the loads of unit `unit` of P's class
    auto request = [&](int unit) {
      const int v = P.v0 + unit * VPW + team;
      P.len = 0;
      P.bq = kFrozenQ16;
      if (v < P.c1) {
        const int off = v - P.c0, g = P.cg + (off >> 5);
        const int gb = grp[g], ge = grp[g + 1];
        P.bq = __ldg(B.bq + (size_t)P.t * n + v);
        P.vo = (uint32_t)__ldg(B.orig + v);
        P.regions = grp[G + 1 + g];
        P.ent = B.occ_t + gb + (off & 31);
        P.len = (ge - gb) / (32 * KQ);
        if (P.len > 0) P.first = (uint32_t)__ldg(&P.ent->x);
      }
      // lists with more late slots than are kept in registers: everything after the wait
      P.late = P.len - region_pre(P.regions) > POST * TL;
      P.pre = P.len > 0 ? (P.late ? P.len : region_pre(P.regions)) : 0;
      if (KQ == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) load_slot(tl + i * TL, P.pre, P.q[i], P.q[i]);
#pragma unroll
        for (int i = 0; i < POST; ++i) load_slot(P.pre + tl + i * TL, P.len, P.qp[i], P.qp[i]);
      }
    };
    // finds the warp's next unit from class c of sweep t on: `mine` counts down over the units of
    // the classes passed, and is the unit's number in the class found
    int mine = warp;
    auto seek = [&](int c, int t) {
#pragma unroll 1
      for (int left = kLookAhead;; --left) {
        if (c == nc) {
          c = 0;
          ++t;
        }
        P.c = c;
        P.t = t;
        P.work = false;
        if (t >= B.t1 || left == 0) return;
        P.c0 = col_ptr[c];
        P.c1 = col_ptr[c + 1];
        P.cg = cgrp[c];
        P.units = share_of(P.c0, P.c1, P.v0);
        if (mine < P.units) break;
        mine -= P.units;
        ++c;
      }
      P.work = true;
      request(mine);
    };
    seek(0, B.t0);
    group_sync<CS>();
    for (int t = B.t0; t < B.t1; ++t) {
      int acc[RPL];  // energy change of the lane's replicas
#pragma unroll
      for (int k = 0; k < RPL; ++k) acc[k] = 0;
      for (int c = 0; c < nc; ++c) {
        const int c0 = col_ptr[c], c1 = col_ptr[c + 1];
        const bool last_class = c + 1 == nc;
        bool waited = c == 0;  // a sweep starts with every word published
        auto wait = [&]() {
          if (!waited) step.wait(B, false);
          waited = true;
        };
        if (P.c == c && P.t == t && !P.work) seek(c, t);
        const bool here = P.c == c && P.t == t;
        for (int unit = mine; here && unit < P.units; unit += kWarps) {
          if (unit != mine) request(unit);
          const int v = P.v0 + unit * VPW + team;
          const bool go = v < P.c1;
          const int len = P.len, pre = P.pre;
          if (__any_sync(0xFFFFFFFFu, P.late)) wait();
          // the lane's next four slots, which arrive behind the Philox blocks
          const bool few = region_few(P.regions);
          int4 r[4 * KQ];
#pragma unroll
          for (int i = 0; i < 4; ++i) load_slot((4 + i) * TL + tl, pre, r[i * KQ], r[i * KQ + KQ - 1]);
          // Philox words of the replicas tl + TL k
          uint32_t u[RPL];
          {
            const PhiloxCol col = philox_col(P.vo, kTagKsatSweep, B.k1);
            constexpr int GPL = 8 / TL;  // groups this lane draws
            uint4 own[GPL];
#pragma unroll
            for (int i = 0; i < GPL; ++i)
              own[i] = philox4x32_meet(sh.rows.at(tl * GPL + i), col, B.k0, B.k1);
#pragma unroll
            for (int k = 0; k < RPL; ++k) {
              // group (tl + TL k) / 4, word tl % 4 (TL is a multiple of 4)
              const int src = TL == 8 ? 2 * k + (tl >> 2) : k >> 1;
              const uint4 &o = own[TL == 8 ? 0 : k & 1];
              const uint32_t a = __shfl_sync(0xFFFFFFFFu, o.x, src, TL),
                             b = __shfl_sync(0xFFFFFFFFu, o.y, src, TL),
                             d = __shfl_sync(0xFFFFFFFFu, o.z, src, TL),
                             e = __shfl_sync(0xFFFFFFFFu, o.w, src, TL);
              u[k] = (tl & 2) ? ((tl & 1) ? e : d) : ((tl & 1) ? b : a);
            }
          }
          const uint32_t x = go ? xs[v] : 0u;
          // the slots before `pre`, from -K on, summed over the team
          uint32_t cnt[8];
          {
            const uint32_t k = tl == 0 && len > 0 ? 0u - marked_slots<KQ>(P.first) : 0u;
#pragma unroll
            for (int j = 0; j < 8; ++j) cnt[j] = (uint32_t)((int)(k << (31 - j)) >> 31);
            const int top = __reduce_max_sync(0xFFFFFFFFu, pre);
            int4 q[4 * KQ];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (KQ == 1) q[i] = P.q[i];
              else load_slot(tl + i * TL, pre, q[i * KQ], q[i * KQ + KQ - 1]);
            }
#pragma unroll 1
            for (int j = 0; j < top; j += 4 * TL) {
              uint32_t z[4];
              slot_masks<KQ, 4>(xs, q, few, z);
              csa4<8>(cnt, z[0], z[1], z[2], z[3]);
#pragma unroll
              for (int i = 0; i < 4 * KQ; ++i) q[i] = r[i];
              if (j + 8 * TL < top) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                  load_slot(j + (8 + i) * TL + tl, pre, r[i * KQ], r[i * KQ + KQ - 1]);
              }
            }
            team_sum<TL, 8>(cnt);
          }
          int4 qp[POST * KQ];
#pragma unroll
          for (int i = 0; i < POST; ++i) {
            if (KQ == 1) qp[i] = P.qp[i];
            else load_slot(pre + tl + i * TL, len, qp[i * KQ], qp[i * KQ + KQ - 1]);
          }
          const uint32_t bq = P.bq;
          const bool free_ = go && bq != kFrozenQ16;  // a held variable takes no attempt
          uint32_t beta[PT ? RPL : 1];
          beta[0] = min(bq, (uint32_t)tab_len << 8);
          if (PT) {
#pragma unroll
            for (int k = 0; k < RPL; ++k) beta[k] = pt_beta(pm[k], bq, tab_len);
          }
          wait();
          // the remaining slots: at most POST per lane
          {
            uint32_t z[POST], p[8];
            slot_masks<KQ, POST>(xs, qp, few, z);
            if constexpr (POST == 2) {
              p[0] = z[0] ^ z[1];
              p[1] = z[0] & z[1];
              team_sum<TL, 2>(p);
            } else {
              const uint32_t s = z[0] ^ z[1] ^ z[2], m = maj3b(z[0], z[1], z[2]), g = s & z[3];
              p[0] = s ^ z[3];
              p[1] = m ^ g;
              p[2] = m & g;
              team_sum<TL, 3>(p);
            }
            uint32_t carry = 0u;  // at most 16 slots: 5 planes
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t a = cnt[j], b = j < 5 ? p[j] : 0u;
              cnt[j] = a ^ b ^ carry;
              carry = maj3b(a, b, carry);
            }
          }
          // dE planes, negated where x = 0; byte i of de[h]: replica tl + h TL + 8 i
          uint32_t de[8 / TL] = {};
          {
            uint32_t carry = ~x;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t y = cnt[j] ^ ~x, d = y ^ carry;
              carry = y & carry;
#pragma unroll
              for (int h = 0; h < 8 / TL; ++h)
                de[h] |= ((d >> (tl + h * TL)) << j) & (0x01010101u << j);
            }
          }
          // every lookup before the first test: none depends on another, and none is skipped
          uint32_t th[RPL];
          int val[RPL];
#pragma unroll
          for (int k = 0; k < RPL; ++k) {
            const uint32_t b8 = byte_of(de[TL == 8 ? 0 : k & 1], TL == 8 ? k : k >> 1);
            val[k] = (int)(signed char)b8;
            th[k] = tab_s[table_index(beta[PT ? k : 0], b8, tab_len)];
          }
          uint32_t flip = 0u;
#pragma unroll
          for (int k = 0; k < RPL; ++k) {
            const bool ok = free_ & ((val[k] <= 0) | (u[k] < th[k]));
            const uint32_t votes = __ballot_sync(0xFFFFFFFFu, ok);
            flip |= ((votes >> (team * TL)) & ((1u << TL) - 1u)) << (TL * k);
            acc[k] += ok ? val[k] : 0;
          }
          if (CS == 1) {
            if (flip && tl == 0) xs[v] = x ^ flip;
          } else if (go && tl < CS) {
            // every word counts at the receiving barriers, also one that did not change
            const uint32_t sa = (uint32_t)__cvta_generic_to_shared(xs + v);
            step.store(sa, tl, x ^ flip, last_class);
            if (CS > TL) step.store(sa, tl + TL, x ^ flip, last_class);
          }
        }
        wait();
        if (last_class) {  // the sweep's energy changes, published with its last class
#pragma unroll
          for (int k = 0; k < RPL; ++k) {
            int s = acc[k];
#pragma unroll
            for (int o = TL; o < 32; o <<= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            if (team == 0 && s != 0) atomicAdd(&sh.ep[t & 1][tl + TL * k], s);
          }
        }
        step.arrive(c1 - c0, last_class);
        if (here) {
          mine -= P.units;
          while (mine < 0) mine += kWarps;
          seek(c + 1, t);
        }
      }
      step.wait(B, true);
      end_sweep<CS, PT>(B, rank, t, xs, sh, track);
    }
    store_item<CS, PT>(B, rank, xs, track);
    group_sync<CS>();
    step.drain();
  }
}

// The class barrier between two CTAs of which one never arrives at the first step, over n items of two
// classes each (items[i].W == 1): the other's wait runs out at the first item, and every item has to
// be marked. Both keep meeting at the cluster barrier.
constexpr int kSelftestThreads = 64;
__global__ void __cluster_dims__(2, 1, 1) step_selftest_kernel(const BatchItem *items, int n, long long limit) {
  __shared__ SweepShared sh;
  const bool absent = cg::this_cluster().block_rank() == 1;
  ClassBarrier<2, kSelftestThreads / 32> step;
  step.init(sh, limit);
  group_sync<2>();
  for (int i = 0; i < n; ++i) {
    const BatchItem &B = items[i];
    step.begin(B);
    if (!absent) {
      step.arrive(0, false);
      step.wait(B, false);
    }
    step.arrive(0, true);
    step.wait(B, true);
    step.drain();
  }
  group_sync<2>();
}

// The launch shape of each kernel instance is queried once per (device, shared-memory size):
// occupancy and cluster queries are slow host calls.
template <int KQ, int CS, int TL, bool PT = false>
cudaError_t launch_batch(const BatchItem *items, int n_items, int *next_item,
                         const uint32_t *tab, int tab_len, int max_n, int device,
                         cudaStream_t st) {
  const int xs_words = max_n + 1;
  size_t words = ((size_t)xs_words + 31) / 32 * 32 + (size_t)tab_len + 1;
  int meta_words = 0;
  if (TL > 1) {  // what room there is beside the vector and the table, up to kMetaWords
    const long long room = (long long)batch_max_vars(tab_len, device) - max_n;
    meta_words = (int)std::max(0LL, std::min((long long)kMetaWords, room));
    words += meta_words;
  }
  const size_t smem = sizeof(uint32_t) * words;
  auto kern = TL == 1 ? ksat_batch_kernel<KQ, CS, PT> : ksat_team_kernel<KQ, CS, (TL > 1 ? TL : 4), PT>;
  constexpr int threads = sweep_threads<KQ, TL>();
  static std::mutex mu;
  static std::map<std::pair<int, size_t>, int> shapes;  // (device, smem) -> resident clusters
  static std::map<int, size_t> smem_set;                // device -> largest smem attribute set
  int clusters = 0;
  {
    std::lock_guard<std::mutex> g(mu);
    cudaError_t err;
    size_t &cur = smem_set[device];
    if (smem > cur) {
      err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (err != cudaSuccess) return err;
      cur = smem;
    }
    auto it = shapes.find({device, smem});
    if (it != shapes.end()) {
      clusters = it->second;
    } else {
      int sms = 0;
      err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
      if (err != cudaSuccess) return err;
      if (CS == 1) {
        int per_sm = 0;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (err != cudaSuccess) return err;
        clusters = sms * per_sm;
      } else {
        cudaLaunchConfig_t q = {};
        q.blockDim = dim3(threads);
        q.dynamicSmemBytes = smem;
        q.gridDim = dim3(CS * sms);
        cudaLaunchAttribute qa[1];
        qa[0].id = cudaLaunchAttributeClusterDimension;
        qa[0].val.clusterDim.x = CS;
        qa[0].val.clusterDim.y = 1;
        qa[0].val.clusterDim.z = 1;
        q.attrs = qa;
        q.numAttrs = 1;
        err = cudaOccupancyMaxActiveClusters(&clusters, kern, &q);
        if (err != cudaSuccess) return err;
      }
      shapes[{device, smem}] = clusters;
    }
  }
  if (clusters < 1) return cudaErrorInvalidConfiguration;
  if (clusters > n_items) clusters = n_items;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(clusters * CS);
  return cudaLaunchKernelEx(&cfg, kern, items, n_items, next_item, tab, tab_len, xs_words,
                            meta_words);
}

// Lanes per variable of the batched kernel: 1 (one thread per variable) or a team of 4 or 8.
int batch_lanes(int cs, int max_n, int want) {
  if (const char *env = getenv("NMC_BATCH_LANES")) {
    const int l = atoi(env);
    if (l == 1 || l == 4 || l == 8) return l;
  }
  if (want == 1 || want == 4 || want == 8) return want;  // a tuned shape
  return choose_lanes(cs, max_n / 32);  // taking ~32 classes
}

// Stands in for the sweep kernels when the number of resident clusters is asked for.
template <int CS>
__global__ void cluster_probe_kernel() {}

template <int KQ, int CS>
cudaError_t dispatch_lanes(const BatchItem *items, int n_items, int *next_item, const uint32_t *tab,
                           int tab_len, int max_n, int device, cudaStream_t st, bool pt, int lanes) {
  if (pt) {
    switch (batch_lanes(CS, max_n, lanes)) {
      case 4: return launch_batch<KQ, CS, 4, true>(items, n_items, next_item, tab, tab_len, max_n, device, st);
      case 8: return launch_batch<KQ, CS, 8, true>(items, n_items, next_item, tab, tab_len, max_n, device, st);
      default: return launch_batch<KQ, CS, 1, true>(items, n_items, next_item, tab, tab_len, max_n, device, st);
    }
  }
  switch (batch_lanes(CS, max_n, lanes)) {
    case 4: return launch_batch<KQ, CS, 4>(items, n_items, next_item, tab, tab_len, max_n, device, st);
    case 8: return launch_batch<KQ, CS, 8>(items, n_items, next_item, tab, tab_len, max_n, device, st);
    default: return launch_batch<KQ, CS, 1>(items, n_items, next_item, tab, tab_len, max_n, device, st);
  }
}

template <int KQ>
cudaError_t dispatch_batch(int cs, const BatchItem *items, int n_items, int *next_item,
                           const uint32_t *tab, int tab_len, int max_n, int device, cudaStream_t st,
                           bool pt, int lanes) {
  switch (cs) {
    case 8: return dispatch_lanes<KQ, 8>(items, n_items, next_item, tab, tab_len, max_n, device, st, pt, lanes);
    case 4: return dispatch_lanes<KQ, 4>(items, n_items, next_item, tab, tab_len, max_n, device, st, pt, lanes);
    case 2: return dispatch_lanes<KQ, 2>(items, n_items, next_item, tab, tab_len, max_n, device, st, pt, lanes);
    default: return dispatch_lanes<KQ, 1>(items, n_items, next_item, tab, tab_len, max_n, device, st, pt, lanes);
  }
}

}  // namespace

// Clusters of cs CTAs that run at once, one CTA per SM: clusters do not span a GPC, so this is less
// than SMs / cs (152 SMs: 76, 36 and 15 clusters of 2, 4 and 8).
// Asked of `device`, whichever is current; an answer is kept, a failed query (0: no clusters) is not.
int batch_clusters(int cs, int device) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, int> known;
  std::lock_guard<std::mutex> g(mu);
  const auto it = known.find({cs, device});
  if (it != known.end()) return it->second;
  int n = 0, prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
  if (prev != device && cudaSetDevice(device) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const size_t smem = 128 * 1024;  // more than half of an SM's
  cudaLaunchConfig_t q = {};
  q.blockDim = dim3(kTeamThreads);
  q.dynamicSmemBytes = smem;
  q.gridDim = dim3(cs * 256);
  cudaLaunchAttribute a[1];
  a[0].id = cudaLaunchAttributeClusterDimension;
  a[0].val.clusterDim.x = cs;
  a[0].val.clusterDim.y = 1;
  a[0].val.clusterDim.z = 1;
  q.attrs = a;
  q.numAttrs = 1;
  const auto query = [&](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) ==
               cudaSuccess &&
           cudaOccupancyMaxActiveClusters(&n, kern, &q) == cudaSuccess;
  };
  const bool ok = cs == 2 ? query(cluster_probe_kernel<2>)
                          : (cs == 4 ? query(cluster_probe_kernel<4>) : query(cluster_probe_kernel<8>));
  if (!ok) cudaGetLastError();
  if (prev >= 0 && prev != device) cudaSetDevice(prev);
  if (!ok) return 0;
  known[{cs, device}] = n;
  return n;
}

// ---- batched sweep without any allocation ----------------------------------------------------
//
// Work list and counters live in one fixed device array of this file instead of memory the
// context allocates on demand. kNoAllocBytes bounds one call: two counters, then up to
// kNoAllocItems work items (one item = one 32-replica word of one replica set).
constexpr size_t kNoAllocBytes = 1u << 20;  // 1 MiB on every GPU that loads the library
constexpr size_t kNoAllocHeader = 256;      // two int counters, padded to the item alignment
constexpr size_t kNoAllocItems = (kNoAllocBytes - kNoAllocHeader) / sizeof(BatchItem);
static_assert(sizeof(BatchItem) == 136 && kNoAllocItems == 7708, "limit stated in nmc.h");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

namespace {

// Device address of g_noalloc_scratch, looked up once per device (with that device current)
// and kept for the rest of the process: a device reset after the first call is not supported.
// In host code the array's name is only a host-side stand-in, never a device address.
std::mutex g_noalloc_mu;
void *g_noalloc_addr[64] = {};

int noalloc_scratch(int device, void **out) {
  if (device < 0 || device >= 64) return NMC_EINVAL;
  std::lock_guard<std::mutex> g(g_noalloc_mu);
  if (!g_noalloc_addr[device]) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      return NMC_ECUDA;
    }
    g_noalloc_addr[device] = p;
  }
  *out = g_noalloc_addr[device];
  return NMC_OK;
}

}  // namespace

}  // namespace nmc

extern "C" int nmc_batch_run_noalloc(nmc_ctx *ctx, int32_t n_sets, const int32_t *rs,
                                     const int32_t *t0, const int32_t *t1) {
  using namespace nmc;
  if (!ctx) return NMC_EINVAL;
  BatchPlan plan;
  int rc = batch_plan(ctx, n_sets, rs, t0, t1, &plan);
  if (rc != NMC_OK) return rc;
  if (plan.items.empty()) return NMC_OK;
  if (plan.items.size() > kNoAllocItems)
    return set_ctx_error(ctx, NMC_EINVAL,
                         "nmc_batch_run_noalloc: more work items (32-replica words) than the "
                         "fixed scratch array holds; split the batch or use nmc_batch_run");
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
  if (cudaSetDevice(plan.device) != cudaSuccess) {
    cudaGetLastError();
    return set_ctx_error(ctx, NMC_ECUDA, "nmc_batch_run_noalloc: cannot select the device");
  }
  void *base = nullptr;
  rc = noalloc_scratch(plan.device, &base);
  cudaError_t e = cudaSuccess;
  if (rc == NMC_OK) {
    int *counters = static_cast<int *>(base);
    BatchItem *items = reinterpret_cast<BatchItem *>(static_cast<char *>(base) + kNoAllocHeader);
    e = cudaMemcpyAsync(items, plan.items.data(), sizeof(BatchItem) * plan.items.size(),
                        cudaMemcpyHostToDevice, plan.stream);
    for (int q = 0; q < 2 && e == cudaSuccess; ++q)
      if (plan.cnt[q] > 0)  // the launcher clears counters[q] on the stream before the kernel
        e = ksat_batch(items + plan.off[q], plan.cnt[q], q + 1, plan.cs[q], plan.max_n[q],
                       counters + q, plan.tab, plan.tab_len, plan.device, plan.stream, false,
                       plan.lanes[q]);
  }
  if (prev >= 0) cudaSetDevice(prev);
  if (rc != NMC_OK)
    return set_ctx_error(ctx, rc, "nmc_batch_run_noalloc: cudaGetSymbolAddress failed");
  if (e != cudaSuccess) {
    cudaGetLastError();
    return set_ctx_error(ctx, NMC_ECUDA, cudaGetErrorString(e));
  }
  return NMC_OK;
}

namespace nmc {

size_t batch_max_vars(int tab_len, int device) {
  int optin = 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess)
    return 0;
  // dynamic shared memory: table + n+1 words; the static part is under 192 words
  const long long words = (long long)optin / 4 - tab_len - 1 - 32 - 1 - 192;
  return words > 0 ? (size_t)words : 0;
}

cudaError_t step_selftest(const BatchItem *items_dev, int n, long long limit_cycles, cudaStream_t st) {
  step_selftest_kernel<<<2, kSelftestThreads, 0, st>>>(items_dev, n, limit_cycles);
  return cudaGetLastError();
}

cudaError_t ksat_batch(const BatchItem *items_dev, int n_items, int kq, int cs, int max_n,
                       int *next_item, const uint32_t *tab, int tab_len, int device,
                       cudaStream_t st, bool pt, int lanes, bool cleared) {
  if (n_items <= 0) return cudaSuccess;
  if (!cleared) {
    const cudaError_t err = cudaMemsetAsync(next_item, 0, sizeof(int), st);
    if (err != cudaSuccess) return err;
  }
  if (kq == 1) return dispatch_batch<1>(cs, items_dev, n_items, next_item, tab, tab_len, max_n, device, st, pt, lanes);
  return dispatch_batch<2>(cs, items_dev, n_items, next_item, tab, tab_len, max_n, device, st, pt, lanes);
}

}  // namespace nmc
