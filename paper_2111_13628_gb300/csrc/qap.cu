// QAP kernels: Metropolis over permutations with pairwise swap moves (Koopmans-Beckmann cost,
// Sec. "Quadratic Assignment Problems"; per-facility inverse temperature as in the sampling
// stage of Algorithm 1).
//
// A CTA runs 32 replicas. Each replica has LPR lanes: LPR = 16 (two replicas per warp, one per
// half) for n <= 128, where the per-attempt broadcasts, reductions and branches are the larger
// part of the work and then serve two replicas at once, and LPR = 32 (one per warp) beyond.
// With NPL = ceil(n / LPR), lane l of a replica owns the locations p[k] of the facilities
// k = NPL l + i (i < NPL) in registers. F and D (entries 0..255, stored as bytes) of the CTA's
// instance sit in shared memory, shared by its replicas; each F row is stored as LPR lane
// chunks of CHB = 4, 8 or 16 bytes (a lane's facilities, zero padded), so a lane reads its part
// of a row with one aligned load. The swap change
//   dC(r,s) = 2 sum_{k != r,s} (F_rk - F_sk)(D_{p(s)p(k)} - D_{p(r)p(k)})
// is an O(n) dot product split over the replica's lanes. Entries up to 127 (the narrow form): the
// lanes first write the row difference D_{p(s).} - D_{p(r).} as signed bytes to a row of the
// replica's own, then each gathers its facilities' bytes from it, packs them four to a word and
// sums their products with F_r - F_s by dp4a. Larger entries (their differences need nine bits):
// both D rows are gathered and the four byte products F_r D_s + F_s D_r - F_r D_r - F_s D_s are
// summed. The narrow form has half the random byte loads, which the shared-memory pipe was 75 %
// busy with, half the packing and a quarter of the dp4a. Then the sums over the lanes. The Philox blocks of LPR consecutive attempts of each replica are drawn
// in parallel, one per lane, and broadcast in turn.
#include <algorithm>
#include <climits>
#include <cmath>

#include "nmc_internal.h"
#include "philox.cuh"

namespace nmc {

namespace {

// Launch shapes: shape q < 8 runs n <= 16 (q + 1) with LPR = 16; shape 8 + q runs
// n <= 32 (q + 5) with LPR = 32.
template <int LPR>
constexpr int qap_threads() { return 32 * LPR; }  // at most 32 replicas per CTA

template <int NPL>
__device__ __forceinline__ void put(int (&p)[NPL], int i, int v) {
#pragma unroll
  for (int q = 0; q < NPL; ++q)
    if (q == i) p[q] = v;
}

// Shared-memory layout of F: row r at r * LDF, as LPR lane chunks of CHB bytes; facility k
// sits in chunk k / NPL at byte k % NPL (padding bytes zero).
template <int NPL, int LPR>
struct FLayout {
  static constexpr int CHB = NPL <= 4 ? 4 : (NPL <= 8 ? 8 : 16);  // bytes of one lane chunk
  static constexpr int LDF = LPR * CHB;                            // row stride in bytes
  __device__ __forceinline__ static int at(int r, int k) { return r * LDF + CHB * (k / NPL) + k % NPL; }
};

// Four zero-extended bytes (b0 lowest) packed into one word.
__device__ __forceinline__ uint32_t pack4(uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3) {
  return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
}

// Differences a - b of four bytes, each at most 127, as signed bytes.
__device__ __forceinline__ uint32_t sub4(uint32_t a, uint32_t b) {
  return ((a | 0x80808080u) - b) ^ 0x80808080u;
}

// N words from a 4 N-byte aligned address of shared memory.
template <int N>
__device__ __forceinline__ void load_words(const uint8_t *p, uint32_t (&w)[N]) {
  if constexpr (N == 4) {
    const uint4 v = *reinterpret_cast<const uint4 *>(p);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
  } else if constexpr (N == 2) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    w[0] = v.x; w[1] = v.y;
  } else {
    w[0] = *reinterpret_cast<const uint32_t *>(p);
  }
}

// Cost of the permutation ps with the whole warp: sum_i sum_j F_ij D_{p(i)p(j)}. The warp's
// 32 / LPR lane groups take rows i in turn; lane l of a group reads its chunk of F row i and the
// bytes D_{p(i)p(k)} of its facilities k = NPL l + q, four to a word, and sums the products with
// dp4a (a row's partial sum stays below 2^22).
template <int NPL, int LPR>
__device__ long long warp_cost(const uint8_t *Fs, const uint8_t *Ds, int ldd, const uint8_t *ps,
                               int n, int lane) {
  constexpr int CHB = FLayout<NPL, LPR>::CHB, LDF = FLayout<NPL, LPR>::LDF, RPW = 32 / LPR;
  const int hl = lane % LPR;
  int pk[NPL];
#pragma unroll
  for (int q = 0; q < NPL; ++q) {
    const int k = NPL * hl + q;
    pk[q] = k < n ? ps[k] : 0;  // padding facilities: F entries zero
  }
  long long acc = 0;
  for (int i = lane / LPR; i < n; i += RPW) {
    const uint8_t *Drow = Ds + ps[i] * ldd;
    const uint32_t *Fw = reinterpret_cast<const uint32_t *>(Fs + i * LDF + CHB * hl);
    uint32_t row = 0u;
#pragma unroll
    for (int w4 = 0; w4 < CHB / 4; ++w4) {
      uint32_t b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = 4 * w4 + q;
        b[q] = j < NPL ? (uint32_t)Drow[pk[j < NPL ? j : 0]] : 0u;
      }
      row = __dp4a(Fw[w4], pack4(b[0], b[1], b[2], b[3]), row);
    }
    acc += row;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
  return acc;
}

// Initial permutation of replica r into its shared-memory row ps (Fisher-Yates from the
// identity, position q = n-1..1 exchanged with (u (q+1)) >> 32, or a copy of the given state),
// then its cost and the global copies. Whole warp.
template <int NPL, int LPR>
__device__ void qap_init_one(const QapArgs &a, const uint8_t *Fs, const uint8_t *Ds, int ldd,
                             uint8_t *ps, int r, int lane) {
  const int n = a.n;
  int16_t *gp = a.perm + (size_t)r * n;
  if (a.init_mode == 1) {
    for (int k = lane; k < n; k += 32) ps[k] = (uint8_t)k;
    __syncwarp();
    for (int q0 = n - 1; q0 >= 1; q0 -= 32) {
      const int q = q0 - lane;
      uint32_t u = 0u;
      if (q >= 1)
        u = philox4x32_10(make_uint4((uint32_t)q, 0u, (uint32_t)r, kTagQapInit), a.k0, a.k1).x;
      const int cnt = q0 >= 32 ? 32 : q0;
      for (int j = 0; j < cnt; ++j) {
        const uint32_t uj = __shfl_sync(0xFFFFFFFFu, u, j);
        const int qq = q0 - j;
        const int kk = (int)(((unsigned long long)uj * (unsigned)(qq + 1)) >> 32);
        if (lane == 0) {
          const uint8_t tmp = ps[qq];
          ps[qq] = ps[kk];
          ps[kk] = tmp;
        }
        __syncwarp();
      }
    }
  } else {
    for (int k = lane; k < n; k += 32) ps[k] = (uint8_t)gp[k];
    __syncwarp();
  }
  const long long c = warp_cost<NPL, LPR>(Fs, Ds, ldd, ps, n, lane);
  const bool set_best = a.init_mode != 3;
  for (int k = lane; k < n; k += 32) {
    gp[k] = (int16_t)ps[k];
    if (set_best) a.best_perm[(size_t)r * n + k] = (int16_t)ps[k];
  }
  if (lane == 0) {
    a.energy[r] = c;
    if (set_best) a.best_energy[r] = c;
  }
  __syncwarp();
}

// A byte of shared memory by its 32-bit address.
__device__ __forceinline__ uint32_t shared_byte(uint32_t addr) {
  return *static_cast<const uint8_t *>(__cvta_shared_to_generic(addr));
}

// Largest uphill change an attempt with draw u accepts at inverse temperature b (Q16). The table does
// not increase, so with c entries above u the test u < tab[(b d) >> 8] is (b d) >> 8 < c, that is
// d <= (256 c - 1) / b. Found once by the lane that draws the attempt: the attempt itself, which all
// lanes of a replica go through one after the other, is left with one comparison. c comes from the
// logarithm the table was built from and is then set right by the table itself.
__device__ __forceinline__ int largest_uphill(const uint32_t *tab_s, int tab_len, uint32_t u,
                                              uint32_t b) {
  int c = min(max((int)(256.0f * (22.18071f - __logf((float)u))), 0), tab_len);
  while (c < tab_len && tab_s[c] > u) ++c;
  while (c > 0 && tab_s[c - 1] <= u) --c;
  if (c == 0) return 0;
  return b == 0u ? INT_MAX : (int)min(((uint32_t)c * 256u - 1u) / b, (uint32_t)INT_MAX);
}

// A CTA runs the a.rpb (at most 32) replicas of one block: lane group h = lane / LPR of warp w runs
// replica rpb block + RPW w + h, its lane l = lane % LPR owning facilities NPL l + i.
template <int NPL, int LPR, bool NARROW>
__device__ __forceinline__ void qap_body(const QapArgs &a, int block) {
  constexpr int RPW = 32 / LPR;  // replicas per warp
  extern __shared__ __align__(16) uint32_t smem[];
  const int n = a.n;
  constexpr int CHB = FLayout<NPL, LPR>::CHB, LDF = FLayout<NPL, LPR>::LDF;
  uint32_t *tab_s = smem;
  uint8_t *Fs = (uint8_t *)(smem + ((a.tab_len + 31) & ~31));
  uint8_t *Ds = Fs + ((n * LDF + 15) & ~15);
  const int ldd = NARROW ? LDF : n;  // the narrow form reads D rows in lane chunks
  uint8_t *pw_all = Ds + ((n * ldd + 15) & ~15);  // one n-byte row per replica (permutation copy)
  const int pstride = (n + 15) & ~15;
  uint8_t *diff_all = pw_all + 32 * pstride;  // NARROW: one LDF-byte row per replica
  for (int i = threadIdx.x; i < a.tab_len; i += blockDim.x) tab_s[i] = a.tab[i];
  for (int i = threadIdx.x; i < n * LDF; i += blockDim.x) {
    const int row = i / LDF, col = i % LDF, j = col % CHB, k = NPL * (col / CHB) + j;
    Fs[i] = (j < NPL && k < n) ? a.F[row * n + k] : (uint8_t)0;
  }
  if (NARROW) {
    for (int i = threadIdx.x; i < n * LDF; i += blockDim.x) {
      const int row = i / LDF, col = i % LDF;
      Ds[i] = col < n ? a.D[row * n + col] : (uint8_t)0;
    }
  } else {
    for (int i = threadIdx.x; i < n * n; i += blockDim.x) Ds[i] = a.D[i];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r0 = block * a.rpb + RPW * warp;  // the warp's first replica
  if (r0 >= a.R) return;                      // the whole warp
  if (a.init_mode != 0) {
    for (int h = 0; h < RPW && r0 + h < a.R; ++h)
      qap_init_one<NPL, LPR>(a, Fs, Ds, ldd, pw_all + (RPW * warp + h) * pstride, r0 + h, lane);
    return;
  }
  const int half = lane / LPR, hl = lane % LPR;
  const int r = r0 + half;
  const bool live = r < a.R;  // the second half of the last warp may have no replica
  uint8_t *pw = pw_all + (RPW * warp + half) * pstride;
  uint8_t *diff = diff_all + (RPW * warp + half) * LDF;
  const int16_t *gp = a.perm + (size_t)(live ? r : r0) * n;
  for (int k = hl; k < n; k += LPR) pw[k] = live ? (uint8_t)gp[k] : (uint8_t)0;
  __syncwarp();
  // Locations of the lane's facilities; padding facilities (k >= n) sit at location 0, their F
  // entries are zero. NARROW: as shared addresses of their bytes in the difference row.
  const int off = NARROW ? (int)(uint32_t)__cvta_generic_to_shared(diff) : 0;
  int p[NPL];
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    const int k = NPL * hl + i;
    p[i] = off + (k < n ? pw[k] : 0);
  }
  long long e = live ? a.energy[r] : 0;
  long long be = live ? a.best_energy[r] : 0;
  const int nm1 = n - 1;
  const unsigned long long mr = (a.mult && live) ? a.mult[r] : 0ull;  // replica exchange multiplier
  // energy statistics: running double sums of the costs after steps t >= stats_t0 (and of their
  // squares), continued from the stored values so that split runs add in step order
  double s1 = 0.0, s2 = 0.0;
  if (a.stats && live) {
    s1 = a.stats[r];
    s2 = a.stats[(size_t)a.R + r];
  }
  for (int t = a.t0; t < a.t1; ++t) {
    if (n >= 2) {
      const uint32_t *bqt = a.bq + (size_t)t * n;
      for (int a0 = 0; a0 < n; a0 += LPR) {
        // lane l of each replica draws its attempt a0 + l
        const int at = a0 + hl;
        int fr = 0, fs = 0, frs = 0, frz = live ? 0 : 1;  // no replica: every attempt rejected
        int dm = INT_MIN;  // the largest change the attempt accepts
        if (at < n && live) {
          const uint4 u =
              philox4x32_10(make_uint4((uint32_t)at, (uint32_t)t, (uint32_t)r, kTagQapStep), a.k0, a.k1);
          fr = (int)(((unsigned long long)u.x * (unsigned)n) >> 32);
          fs = (int)(((unsigned long long)u.y * (unsigned)nm1) >> 32);
          fs += fs >= fr;
          const uint32_t br = __ldg(bqt + fr), bs = __ldg(bqt + fs);
          frz = (br == kFrozenQ16 || bs == kFrozenQ16) ? 1 : 0;  // a held facility: reject
          uint32_t bj = (uint32_t)(((unsigned long long)br + bs) >> 1);
          if (a.mult) {  // min(2^32 - 1, (mult * bq) >> 16)
            const unsigned long long be2 = (mr * bj) >> 16;
            bj = be2 > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)be2;
          }
          if (!frz) dm = largest_uphill(tab_s, a.tab_len, u.z, bj);
          frs = Fs[FLayout<NPL, LPR>::at(fr, fs)];
        }
        const int cnt = (n - a0) < LPR ? (n - a0) : LPR;
        // r, s and F_rs (a byte each) and the held flag of every lane's attempt in one word: one
        // broadcast per attempt within each replica's lanes
        const int packed = fr | (fs << 8) | (frs << 16) | (frz << 24);
        const bool any_held = __any_sync(0xFFFFFFFFu, frz);
        // the next attempt's broadcasts are under way while the current one is evaluated
        int pnext = __shfl_sync(0xFFFFFFFFu, packed, 0, LPR), dnext = __shfl_sync(0xFFFFFFFFu, dm, 0, LPR);
        for (int j = 0; j < cnt; ++j) {
          const int pj = pnext, dj = dnext;
          pnext = __shfl_sync(0xFFFFFFFFu, packed, j + 1, LPR);
          dnext = __shfl_sync(0xFFFFFFFFu, dm, j + 1, LPR);
          // every replica of the warp held
          if (any_held && __all_sync(0xFFFFFFFFu, (pj >> 24) != 0)) continue;
          const int rr = pj & 255, ss = (pj >> 8) & 255;
          const int pr = pw[rr], ps = pw[ss];
          const uint8_t *Dr = Ds + pr * ldd, *Dsr = Ds + ps * ldd;
          // this lane's chunks of rows r and s of F
          uint32_t fr4[CHB / 4], fs4[CHB / 4];
          load_words<CHB / 4>(Fs + rr * LDF + CHB * hl, fr4);
          load_words<CHB / 4>(Fs + ss * LDF + CHB * hl, fs4);
          // sum over every k (padding bytes of F are zero); the k = r and k = s terms sum to
          // -2 F_rs D_{p(r)p(s)} by symmetry and are added back below
          int acc = 0;
          if constexpr (NARROW) {
            uint32_t dr4[CHB / 4], ds4[CHB / 4];
            load_words<CHB / 4>(Dr + CHB * hl, dr4);
            load_words<CHB / 4>(Dsr + CHB * hl, ds4);
#pragma unroll
            for (int w4 = 0; w4 < CHB / 4; ++w4) dr4[w4] = sub4(ds4[w4], dr4[w4]);
            if constexpr (CHB == 16)
              *reinterpret_cast<uint4 *>(diff + 16 * hl) = make_uint4(dr4[0], dr4[1], dr4[2], dr4[3]);
            else if constexpr (CHB == 8)
              *reinterpret_cast<uint2 *>(diff + 8 * hl) = make_uint2(dr4[0], dr4[1]);
            else
              *reinterpret_cast<uint32_t *>(diff + 4 * hl) = dr4[0];
            __syncwarp();  // the row is complete; the end of the attempt orders its next writes
#pragma unroll
            for (int w4 = 0; w4 < CHB / 4; ++w4) {
              uint32_t g[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int i = 4 * w4 + q;
                g[q] = i < NPL ? shared_byte((uint32_t)p[i < NPL ? i : 0]) : 0u;
              }
              acc = __dp4a((int)sub4(fr4[w4], fs4[w4]), (int)pack4(g[0], g[1], g[2], g[3]), acc);
            }
          } else {
            // positive and negative products are summed apart (unsigned, below 2^22)
            uint32_t accp = 0u, accn = 0u;
#pragma unroll
            for (int w4 = 0; w4 < CHB / 4; ++w4) {
              uint32_t dr[4], dsb[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int i = 4 * w4 + q;
                dr[q] = i < NPL ? (uint32_t)Dr[p[i < NPL ? i : 0]] : 0u;
                dsb[q] = i < NPL ? (uint32_t)Dsr[p[i < NPL ? i : 0]] : 0u;
              }
              const uint32_t wr = pack4(dr[0], dr[1], dr[2], dr[3]);
              const uint32_t wsv = pack4(dsb[0], dsb[1], dsb[2], dsb[3]);
              accp = __dp4a(fr4[w4], wsv, accp);
              accp = __dp4a(fs4[w4], wr, accp);
              accn = __dp4a(fr4[w4], wr, accn);
              accn = __dp4a(fs4[w4], wsv, accn);
            }
            acc = (int)(accp - accn);
          }
          if constexpr (LPR == 32) {
            acc = __reduce_add_sync(0xFFFFFFFFu, acc);
          } else {
            // the two replicas' sums as two whole-warp reductions side by side
            const int lo = __reduce_add_sync(0xFFFFFFFFu, half == 0 ? acc : 0);
            const int hi = __reduce_add_sync(0xFFFFFFFFu, half == 0 ? 0 : acc);
            acc = half == 0 ? lo : hi;
          }
          acc += 2 * ((pj >> 16) & 255) * (int)Dr[ps];
          const int d = 2 * acc;  // |acc| < 2^25
          if (d <= dj) {
            if (hl == rr / NPL) put<NPL>(p, rr % NPL, off + ps);
            if (hl == ss / NPL) put<NPL>(p, ss % NPL, off + pr);
            if (hl == 0) {
              pw[rr] = (uint8_t)ps;
              pw[ss] = (uint8_t)pr;
            }
            e += d;
          }
          __syncwarp();  // the row updates are seen by the next attempt
        }
      }
    }
    if (live && e < be) {
      be = e;
#pragma unroll
      for (int i = 0; i < NPL; ++i) {
        const int k = NPL * hl + i;
        if (k < n) a.best_perm[(size_t)r * n + k] = (int16_t)(p[i] - off);
      }
    }
    if (a.stats && live && t >= a.stats_t0) {
      const double ed = (double)e;
      s1 = __dadd_rn(s1, ed);
      s2 = __dadd_rn(s2, __dmul_rn(ed, ed));
    }
  }
  if (!live) return;
  int16_t *gq = a.perm + (size_t)r * n;
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    const int k = NPL * hl + i;
    if (k < n) gq[k] = (int16_t)(p[i] - off);
  }
  if (hl == 0) {
    a.energy[r] = e;
    a.best_energy[r] = be;
    if (a.stats) {
      a.stats[r] = s1;
      a.stats[(size_t)a.R + r] = s2;
    }
  }
}

// Facilities per lane from which the narrow form is used: its row exchange costs more than it
// saves for one or two gathers a lane (4 sets of 4,096 replicas, wide -> narrow: n = 16 677 -> 736
// us per 40 steps, n = 64 1,460 -> 1,467 per 20, n = 96 2,705 -> 2,445, n = 128 4,129 -> 3,300,
// n = 192 4,979 -> 4,331 per 10, n = 256 7,435 -> 6,033).
constexpr int kNarrowNpl = 3;

template <int NPL, int LPR>
__global__ void __launch_bounds__(qap_threads<LPR>(), LPR == 16 ? 2 : 1) qap_kernel(QapArgs a) {
  if (NPL >= kNarrowNpl && a.narrow) qap_body<NPL, LPR, NPL >= kNarrowNpl>(a, blockIdx.x);
  else qap_body<NPL, LPR, false>(a, blockIdx.x);
}

// Batched QAP: CTA b runs replica block items[b].block of the replica set items[b] describes.
template <int NPL, int LPR>
__global__ void __launch_bounds__(qap_threads<LPR>(), LPR == 16 ? 2 : 1) qap_batch_kernel(const QapArgs *items) {
  const QapArgs a = items[blockIdx.x];
  if (NPL >= kNarrowNpl && a.narrow) qap_body<NPL, LPR, NPL >= kNarrowNpl>(a, a.block);
  else qap_body<NPL, LPR, false>(a, a.block);
}

// Shape parameters: NPL and LPR of shape q.
__host__ __device__ constexpr int shape_npl(int q) { return q < 8 ? q + 1 : q - 3; }
__host__ __device__ constexpr int shape_lpr(int q) { return q < 8 ? 16 : 32; }

size_t qap_smem_shape(int n, int q, int tab_len) {
  const int npl = shape_npl(q);
  const int ldf = shape_lpr(q) * (npl <= 4 ? 4 : (npl <= 8 ? 8 : 16));  // FLayout::LDF
  // the narrow form's layout, the larger one (ldf >= n, and its difference rows)
  return sizeof(uint32_t) * ((tab_len + 31) & ~31) + 2 * (size_t)((n * ldf + 15) & ~15) +
         (size_t)32 * ((n + 15) & ~15) + (size_t)32 * ldf;
}

template <int Q>
cudaError_t launch_qap(const QapArgs &a, cudaStream_t st) {
  constexpr int NPL = shape_npl(Q), LPR = shape_lpr(Q);
  const size_t smem = qap_smem_shape(a.n, Q, a.tab_len);
  auto kern = qap_kernel<NPL, LPR>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  const int blocks = (a.R + a.rpb - 1) / a.rpb;
  kern<<<blocks, a.rpb * LPR, smem, st>>>(a);
  return cudaGetLastError();
}

#define NMC_QAP_CASES(CALL) \
  CALL(0) CALL(1) CALL(2) CALL(3) CALL(4) CALL(5) CALL(6) CALL(7) CALL(8) CALL(9) CALL(10) CALL(11)

cudaError_t dispatch_qap(QapArgs a, cudaStream_t st) {
  int device = 0;
  const cudaError_t err = cudaGetDevice(&device);
  if (err != cudaSuccess) return err;
  a.rpb = qap_replicas_per_block(qap_load(a.n, a.R), qap_lanes(qap_shape(a.n)), device);
  switch (qap_shape(a.n)) {
#define NMC_CASE(k) case k: return launch_qap<k>(a, st);
    NMC_QAP_CASES(NMC_CASE)
#undef NMC_CASE
    default: return cudaErrorInvalidValue;
  }
}

__global__ void qap_unpack_kernel(const int16_t *perm, const int16_t *best_perm,
                                  const long long *energy, const long long *best_energy,
                                  int32_t n, int32_t R, int16_t *p_out, int16_t *bp_out,
                                  int64_t *e_out, int64_t *be_out) {
  const long long total = (long long)R * n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    if (p_out) p_out[i] = perm[i];
    if (bp_out) bp_out[i] = best_perm[i];
    if (i < R) {
      if (e_out) e_out[i] = energy[i];
      if (be_out) be_out[i] = best_energy[i];
    }
  }
}

QapArgs make_args(const QapDevice &I, QapReplicas &Rp, uint64_t seed) {
  QapArgs a;
  a.F = (const uint8_t *)I.F;
  a.D = (const uint8_t *)I.D;
  a.perm = Rp.perm;
  a.best_perm = Rp.best_perm;
  a.energy = (long long *)Rp.energy;
  a.best_energy = (long long *)Rp.best_energy;
  a.bq = nullptr;
  a.tab = nullptr;
  a.tab_len = 0;
  a.n = I.n;
  a.R = Rp.R;
  a.t0 = a.t1 = 0;
  a.k0 = (uint32_t)seed;
  a.k1 = (uint32_t)(seed >> 32);
  a.init_mode = 0;
  a.block = -1;
  a.narrow = I.narrow ? 1 : 0;
  a.rpb = 32;
  a.mult = nullptr;
  a.stats = nullptr;
  a.stats_t0 = 0;
  return a;
}

template <int Q>
cudaError_t launch_qap_batch(const QapArgs *items_dev, int n_blocks, int rpb, int max_n, int tab_len,
                             cudaStream_t st) {
  constexpr int NPL = shape_npl(Q), LPR = shape_lpr(Q);
  const size_t smem = qap_smem_shape(max_n, Q, tab_len);
  auto kern = qap_batch_kernel<NPL, LPR>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  kern<<<n_blocks, rpb * LPR, smem, st>>>(items_dev);
  return cudaGetLastError();
}

}  // namespace

QapArgs qap_block_args(const QapDevice &I, QapReplicas &Rp, const uint32_t *bq, const uint32_t *tab,
                       int32_t tab_len, int32_t t0, int32_t t1, uint64_t seed, int rpb,
                       int block) {
  QapArgs a = make_args(I, Rp, seed);
  a.rpb = rpb;
  a.bq = bq;
  a.tab = tab;
  a.tab_len = tab_len;
  a.t0 = t0;
  a.t1 = t1;
  a.block = block;
  return a;
}

int qap_lanes(int shape) { return shape_lpr(shape); }

int qap_shape(int n) { return n <= 128 ? (n + 15) / 16 - 1 : 8 + (n + 31) / 32 - 5; }

// A CTA of 32 replicas with 32 lanes each fills an SM, one with 16 lanes each half of one. The blocks
// of a call take as many rounds of the SMs as full CTAs would, in equal parts: of 27 replicas where
// 4 x 128 full CTAs would leave the last of four rounds two fifths empty (4 sets of 4,096 replicas,
// n = 256), of few where full CTAs would leave SMs without any (256 replicas, n = 33: 8 CTAs of 32,
// 60 % of their issue slots busy: 1.18 -> 0.95 ms per 100 steps). At least four warps, which also load the CTA's copies of F, D and
// the table.
int qap_replicas_per_block(double load, int lanes, int device) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1) {
    cudaGetLastError();
    return 32;
  }
  const double share = load / (sms * std::max(1.0, std::ceil(load / sms)));
  const int rpw = 32 / lanes;  // whole warps
  const int rpb = (static_cast<int>(std::ceil(32.0 * share)) + rpw - 1) / rpw * rpw;
  return std::min(32, std::max(rpb, 4 * rpw));
}

double qap_load(int32_t n, int32_t R) { return ((R + 31) / 32) * (n <= 128 ? 0.5 : 1.0); }

cudaError_t qap_batch(const QapArgs *items_dev, int n_blocks, int shape, int rpb, int max_n, int tab_len,
                      cudaStream_t st) {
  if (n_blocks <= 0) return cudaSuccess;
  switch (shape) {
#define NMC_CASE(k) case k: return launch_qap_batch<k>(items_dev, n_blocks, rpb, max_n, tab_len, st);
    NMC_QAP_CASES(NMC_CASE)
#undef NMC_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t qap_init_states(const QapDevice &I, QapReplicas &Rp, uint64_t seed,
                            const int16_t *init_dev, cudaStream_t st, bool set_best) {
  QapArgs a = make_args(I, Rp, seed);
  if (init_dev) {
    cudaError_t err = cudaMemcpyAsync(Rp.perm, init_dev, sizeof(int16_t) * (size_t)Rp.R * I.n,
                                      cudaMemcpyDeviceToDevice, st);
    if (err != cudaSuccess) return err;
    a.init_mode = set_best ? 2 : 3;
  } else {
    a.init_mode = 1;
  }
  return dispatch_qap(a, st);
}

cudaError_t qap_steps(const QapDevice &I, QapReplicas &Rp, const uint32_t *bq,
                      const uint32_t *tab, int32_t tab_len, int32_t t0, int32_t t1,
                      uint64_t seed, cudaStream_t st) {
  if (t1 <= t0) return cudaSuccess;
  QapArgs a = make_args(I, Rp, seed);
  a.bq = bq;
  a.tab = tab;
  a.tab_len = tab_len;
  a.t0 = t0;
  a.t1 = t1;
  return dispatch_qap(a, st);
}

cudaError_t qap_unpack(const QapDevice &I, const QapReplicas &Rp, int16_t *perms,
                       int16_t *best_perms, int64_t *energies, int64_t *best_energies,
                       cudaStream_t st) {
  const long long total = (long long)Rp.R * I.n;
  long long blocks = (total + 255) / 256;
  if (blocks > 65535) blocks = 65535;
  if (blocks < 1) blocks = 1;
  qap_unpack_kernel<<<(int)blocks, 256, 0, st>>>(Rp.perm, Rp.best_perm,
                                                 (const long long *)Rp.energy,
                                                 (const long long *)Rp.best_energy, I.n, Rp.R,
                                                 perms, best_perms, energies, best_energies);
  return cudaGetLastError();
}

}  // namespace nmc
