// tile.cu — persistent tile kernels: one CTA works on one (instance, 32-replica
// group) tile at a time, pulled from a work queue largest first, with the
// instance's spins bit-packed in shared memory (bit r of word i = replica r of
// spin i is +1).  CTAs of 256 threads (four per SM, two for the lattice mode), or
// of 512 and 1024 where the tiles are few.  Without a sweep budget a tile's
// descents are independent, so where the tiles leave CTAs idle each is cut into
// segments of consecutive descents, and the last segment to end keeps the best.
//
// Method (García & Markov, Sec. IV): single-spin moves taken when their gain
// -2 s_i f_i is positive, whole sweeps repeated until no move is taken (a 1-flip
// local minimum), independent random starts, the best result kept.  Colour
// classes are independent sets, so all spins of a class decide at once.
//
// Four evaluators share the sweep/restart machinery:
//   MODE 0  integer couplings, exact int32 fields recomputed from the neighbours'
//           bits at each visit, four lanes per spin with 8 replicas each where a
//           warp has several pending spins, else a warp per spin, lane = replica;
//   MODE 1  FP32 couplings, four lanes per spin with 8 replicas each, FP32 fields
//           kept per (spin, replica) and updated at each visit from the neighbours
//           that flipped since the previous visit (the paper's incremental gain
//           update), with a from-scratch refresh at descent sweeps
//           d % refresh == 0 (always d == 0): the FP64 sum rounded to FP32,
//           formed exactly in fixed point when that is exact (runit >= 0; else, and
//           for one or two pending spins of a warp, a warp per spin, lane = replica);
//           fields of instances that fit stay in shared memory;
//   MODE 2  multi-spin coding for J in {-1,+1}, h in {-1,0,+1}: one thread per
//           spin evaluates all 32 replicas with bitwise logic (unsatisfied-bond
//           masks counted in a bit-sliced adder, compared with the per-field
//           thresholds);
//   MODE 3  the same on periodic 2-d/3-d lattices, with neighbours computed
//           from the lattice geometry and the field folded into the count.
// In the index order the lane modes give a tile's spins to one warp, one after
// another, multi-spin coding to one thread a step.
// Replicas of a tile run their descents in lockstep rounds: descent k of every
// lane starts together; a lane whose descent ended waits (masked) until the
// round ends.  Each replica's own sequence of states is exactly the one its
// C-ABI semantics define.
#include <cfloat>

#include <algorithm>
#include <type_traits>

#include "device_common.cuh"

namespace isg {

namespace {

// Energies of all 32 replica lanes of the tile at once (Eq. 1 + Eq. 6): one
// warp per spin, lane = replica.  Integer couplings sum exactly in int64;
// FP32 couplings sum exactly in 64-bit fixed point when the instance allows it
// (InstDesc::ebase >= 0; one final rounding to FP64), else in FP64 with warps
// added in ascending order.  Each pair is counted at its smaller index, each
// hyper-edge once.  Every path is deterministic; the result goes to E[32].
template <bool FLOAT>
__device__ void tile_energy_lanes(const DevGraph &G, const InstDesc &I, const uint32_t *sw, double *red,
                                  double *E) {
  const int n = I.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int ub = I.ebase;
  const bool fx = FLOAT && ub >= 0;
  double accd = 0.0;
  long long acci = 0;
  unsigned long long accl = 0;
  // the warp's spins i = warp + k nw, 32 at a time: lane k reads spin k's row
  // bounds and field in one pass, then the spins are taken in order
  for (int ib = warp; ib < n; ib += 32 * nw) {
    const int il = ib + lane * nw;
    uint32_t k0l = 0, k1l = 0, hvl = 0;
    if (il < n) {
      const int64_t g = I.spin_off + il;
      k0l = __ldg(G.row + g);
      k1l = __ldg(G.row + g + 1);
      hvl = FLOAT ? __float_as_uint(__ldg(reinterpret_cast<const float *>(G.h) + g))
                  : (uint32_t)(int32_t)__ldg(reinterpret_cast<const int8_t *>(G.h) + g);
    }
    const int cnt = min(32, (n - ib + nw - 1) / nw);
    for (int src = 0; src < cnt; ++src) {
      const int i = ib + src * nw;
      const uint32_t bi = (sw[i] >> lane) & 1u;
      const uint32_t k0 = __shfl_sync(0xffffffffu, k0l, src), k1 = __shfl_sync(0xffffffffu, k1l, src);
      const uint32_t hraw = __shfl_sync(0xffffffffu, hvl, src);
      if (FLOAT) {
        const float *Jf = reinterpret_cast<const float *>(G.J);
        const float hv = __uint_as_float(hraw);
        if (fx) {
          const int64_t th = xr_term(hv, ub);
          xe_add(acci, accl, bi ? -th : th);
          for (uint32_t k = k0; k < k1; ++k) {
            const int j = __ldg(G.col + k);
            if (j > i) {
              const int64_t t = xr_term(__ldg(Jf + k), ub);
              xe_add(acci, accl, (((sw[j] >> lane) & 1u) ^ bi) ? t : -t);
            }
          }
        } else {
          double e = bi ? (double)hv : -(double)hv;
          for (uint32_t k = k0; k < k1; ++k) {
            const int j = __ldg(G.col + k);
            if (j > i) {
              const double w = (double)__ldg(Jf + k);
              e += (((sw[j] >> lane) & 1u) ^ bi) ? -w : w;
            }
          }
          accd -= e;
        }
      } else {
        const int8_t *Ji = reinterpret_cast<const int8_t *>(G.J);
        const int hv = (int)hraw;
        int e = bi ? hv : -hv;
        for (uint32_t k = k0; k < k1; ++k) {
          const int j = __ldg(G.col + k);
          if (j > i) {
            const int w = __ldg(Ji + k);
            e += (((sw[j] >> lane) & 1u) ^ bi) ? -w : w;
          }
        }
        acci -= e;
      }
    }
  }
  for (int e = warp; e < I.n_hyper; e += nw) {
    const int64_t ge = I.hyper_off + e;
    uint32_t neg = 0;
    for (uint32_t q = __ldg(G.hptr + ge), qe = __ldg(G.hptr + ge + 1); q < qe; ++q)
      neg ^= ~(sw[__ldg(G.hmem + q)] >> lane) & 1u;
    if (FLOAT) {
      const float w = __ldg(reinterpret_cast<const float *>(G.hJ) + ge);
      if (fx) {
        const int64_t t = xr_term(w, ub);
        xe_add(acci, accl, neg ? t : -t);
      } else {
        accd -= neg ? -(double)w : (double)w;
      }
    } else {
      const int w = __ldg(reinterpret_cast<const int8_t *>(G.hJ) + ge);
      acci -= neg ? -w : w;
    }
  }
  long long *ri = reinterpret_cast<long long *>(red);
  __syncthreads();
  if (FLOAT && !fx) red[warp * 32 + lane] = accd;
  else ri[warp * 32 + lane] = acci;
  __syncthreads();
  long long hi = 0;
  if (warp == 0) {
    if (FLOAT && !fx) {
      double a = red[lane];
      for (int w = 1; w < nw; ++w) a += red[w * 32 + lane];
      E[lane] = a;
    } else {
      for (int w = 0; w < nw; ++w) hi += ri[w * 32 + lane];
      if (!FLOAT) E[lane] = (double)hi;
    }
  }
  if (fx) {
    __syncthreads();
    reinterpret_cast<unsigned long long *>(red)[warp * 32 + lane] = accl;
    __syncthreads();
    if (warp == 0) {
      unsigned long long lo = 0;
      for (int w = 0; w < nw; ++w) lo += reinterpret_cast<unsigned long long *>(red)[w * 32 + lane];
      E[lane] = xe_value(hi, lo, ub);
    }
  }
  __syncthreads();
}

// The same in integers with a lane per spin (and per hyper-edge): with p the parity
// word of a term's spins (bit r: their product in replica r is -1), the term is
// -t + 2 t p_r, so a predicated add per replica for 32 spins at once, where the form
// above spends that and the term's decoding on every spin for itself (bound by
// issue).  FP32: 64-bit fixed point, NV = 8 replicas at a time, the rows read again
// from L1 for each (1,024 cell grids of 128 to 2,048 spins: 1,754 us a call with
// the form above, 1,623 / 1,577 / 1,699 with 4 / 8 / 16); integers: all 32 (a graph of
// 1,000 spins, 1,024 replicas, 20 descents: 1,112 -> 1,036 us).  Instances of up to
// kFewSpins leave most lanes without a spin and take the form above (5,000 of 40 spins,
// 10 descents: 6.04 against 5.31 ms).  False, and nothing done, when FP32
// terms are not integers of one unit, or so wide or so many that a lane's sum could
// leave its 62 bits (integers: a warp's its 31); the same for the whole CTA.
template <bool FLOAT, int THREADS>
__device__ bool tile_energy_sites(const DevGraph &G, const InstDesc &I, const uint32_t *sw, double *red, double *E) {
  using T = std::conditional_t<FLOAT, long long, int>;
  constexpr int NV = FLOAT ? 8 : 32;
  const int n = I.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ub = I.ebase;
  // (a lane's terms; 64-bit: the degree is not bounded by the tile's size)
  const int64_t terms = (int64_t)((n + THREADS - 1) / THREADS) * (I.max_deg + 1) + (I.n_hyper + THREADS - 1) / THREADS;
  if (FLOAT ? ub < 0 || I.ebits + (64 - __clzll(terms)) + 1 > 62 : terms > 1 << 19) return false;
  long long hi = 0;  // lane r: replica r's warp total
  unsigned long long lo = 0;
#pragma unroll 1
  for (int r0 = 0; r0 < 32; r0 += NV) {
    T acc[NV], csum = 0;
#pragma unroll
    for (int r = 0; r < NV; ++r) acc[r] = 0;
    auto value = [&](const void *arr, int64_t at) -> T {
      if constexpr (FLOAT) return (T)xr_term(__ldg(reinterpret_cast<const float *>(arr) + at), ub);
      else return (T)__ldg(reinterpret_cast<const int8_t *>(arr) + at);
    };
    auto add = [&](T t, uint32_t p) {
      csum += t;
      p >>= r0;
#pragma unroll
      for (int r = 0; r < NV; ++r)
        if ((p >> r) & 1u) acc[r] += t;
    };
    for (int i = tid; i < n; i += THREADS) {
      const int64_t gi = I.spin_off + i;
      const uint32_t w = sw[i];
      add(value(G.h, gi), ~w);
      for (uint32_t k = __ldg(G.row + gi), k1 = __ldg(G.row + gi + 1); k < k1; ++k) {
        const int j = __ldg(G.col + k);
        if (j > i) add(value(G.J, k), w ^ sw[j]);
      }
    }
    for (int e = tid; e < I.n_hyper; e += THREADS) {
      const int64_t ge = I.hyper_off + e;
      uint32_t p = 0u;
      for (uint32_t q = __ldg(G.hptr + ge), qe = __ldg(G.hptr + ge + 1); q < qe; ++q) p ^= ~sw[__ldg(G.hmem + q)];
      add(value(G.hJ, ge), p);
    }
#pragma unroll
    for (int r = 0; r < NV; ++r) {
      const T v = 2 * acc[r] - csum;
      if constexpr (FLOAT) {  // (20-bit pieces: 32 of them add up in 32 bits)
        const int p0 = __reduce_add_sync(0xffffffffu, (int)(v & 0xfffff));
        const int p1 = __reduce_add_sync(0xffffffffu, (int)((v >> 20) & 0xfffff));
        const int p2 = __reduce_add_sync(0xffffffffu, (int)(v >> 40));
        if (lane == r0 + r) {
          hi = (long long)p2 << 8;
          lo = ((unsigned long long)(unsigned)p1 << 20) + (unsigned)p0;
        }
      } else {
        const int t = __reduce_add_sync(0xffffffffu, v);
        if (lane == r) hi = t;
      }
    }
  }
  long long *ri = reinterpret_cast<long long *>(red);
  __syncthreads();
  ri[warp * 32 + lane] = hi;
  __syncthreads();
  hi = 0;
  if (warp == 0)
    for (int w = 0; w < THREADS / 32; ++w) hi += ri[w * 32 + lane];
  if (FLOAT) {
    __syncthreads();
    reinterpret_cast<unsigned long long *>(red)[warp * 32 + lane] = lo;
    __syncthreads();
    lo = 0;
    if (warp == 0)
      for (int w = 0; w < THREADS / 32; ++w) lo += reinterpret_cast<unsigned long long *>(red)[w * 32 + lane];
  }
  if (warp == 0) E[lane] = FLOAT ? xe_value(hi, lo, ub) : (double)hi;
  __syncthreads();
  return true;
}

// Energies of all 32 lanes for a +/-1 periodic lattice with |h| <= 1 (the
// multi-spin coded lattice path): E = 2 U - (n d + #{h != 0}), U = the lane's
// number of unsatisfied bonds and fields.  Each thread adds, per site, the
// unsatisfied masks of its forward bonds (+x, +y, +z) and of its field into a
// bit-sliced per-lane counter; a butterfly of bit-sliced adds totals the
// counters over the warp, and warps are added in shared memory.  Exact integers.
__device__ void tile_energy_lattice(const DevGraph &G, const InstDesc &I, const uint32_t *sw, int *cnt,
                                    double *E) {
  constexpr int Q = 14;  // counter depth: up to 2^14 - 1 per lane and thread
  const int n = I.n, L = I.lat_L, D = I.lat_d, lane = threadIdx.x & 31;
  const int stride[3] = {1, L, L * L};
  uint32_t acc[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) acc[q] = 0u;
  int nz = 0;
  if (threadIdx.x < 32) cnt[threadIdx.x] = 0;
  if (threadIdx.x == 32) cnt[32] = 0;
  __syncthreads();
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    const int j = __ldg(G.order + I.spin_off + v);
    const uint32_t info = __ldg(G.latinfo + I.spin_off + v);
    const int hv = __ldg(reinterpret_cast<const int8_t *>(G.h) + I.spin_off + j);
    const uint32_t wj = sw[j];
    uint32_t f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      f[a] = 0u;
      if (a < D) {
        const int d = 2 * a;  // forward direction along axis a
        const int nb = j + stride[a] - (((info >> d) & 1u) ? L * stride[a] : 0);
        f[a] = wj ^ sw[nb] ^ (((info >> (8 + d)) & 1u) ? 0xffffffffu : 0u);
      }
    }
    const uint32_t uf = hv == 0 ? 0u : (hv > 0 ? ~wj : wj);
    nz += hv != 0;
    // compress the four masks into weights 1, 2, 4 and add them to the counter
    const uint32_t s1 = f[0] ^ f[1] ^ f[2], c1 = (f[0] & f[1]) | (f[0] & f[2]) | (f[1] & f[2]);
    const uint32_t s2 = s1 ^ uf, c2 = s1 & uf;
    const uint32_t t1 = c1 ^ c2, t2 = c1 & c2;
    uint32_t cy = acc[0] & s2;
    acc[0] ^= s2;
    const uint32_t x1 = acc[1] ^ t1 ^ cy;
    cy = (acc[1] & t1) | (acc[1] & cy) | (t1 & cy);
    acc[1] = x1;
    const uint32_t x2 = acc[2] ^ t2 ^ cy;
    cy = (acc[2] & t2) | (acc[2] & cy) | (t2 & cy);
    acc[2] = x2;
#pragma unroll
    for (int q = 3; q < Q; ++q) {
      const uint32_t c = acc[q] & cy;
      acc[q] ^= cy;
      cy = c;
    }
  }
  const long long mine = warp_sliced_total<Q>(acc, lane);  // lane r: replica r's warp total
  nz = warp_sum(nz);
  atomicAdd(&cnt[lane], (int)mine);
  if (lane == 0) atomicAdd(&cnt[32], nz);
  __syncthreads();
  if (threadIdx.x < 32) E[threadIdx.x] = 2.0 * (double)cnt[threadIdx.x] - (double)n * D - (double)cnt[32];
  __syncthreads();
}

// u >= t for a bit-sliced 4-bit count (c0 least significant), t a per-thread value.
__device__ __forceinline__ uint32_t sliced_ge(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                              int t) {
  if (t <= 0) return 0xffffffffu;
  if (t > 15) return 0u;
  uint32_t gt = 0, eq = 0xffffffffu;
  const uint32_t c[4] = {c0, c1, c2, c3};
#pragma unroll
  for (int p = 3; p >= 0; --p) {
    const uint32_t tb = ((t >> p) & 1) ? 0xffffffffu : 0u;
    gt |= eq & c[p] & ~tb;
    eq &= ~(c[p] ^ tb);
  }
  return gt | eq;
}

// FP32 visits: four lanes share a pending spin, 8 replicas each from r0, and a warp
// takes 8 spins at a time.  A visit by the whole warp, a lane per replica, spent the
// row, the neighbours' words and each term's decoding on one spin (some 380
// instructions) and was bound by issue; here a term is a predicated add per replica
// for 8 spins at once, and 8 pending spins of a class fill a warp.  1,024 cell grids
// of 128 to 2,048 spins: 1,577 -> 965 us (one lane for all 32 replicas of a spin:
// 1,127, and slower than a whole warp on small classes); 4,096 of them: 5,983 ->
// 3,265; one graph of 6,000 spins: 1,718 -> 964.  Both forms return the replicas in
// which the spin is against its field and leave the fields in F.

// The parities of the other members' spins (flips) of incident hyper-edge q of j.
__device__ __forceinline__ uint32_t own_parity(const DevGraph &G, const uint32_t *words, uint32_t inv, int j, uint32_t q) {
  const int2 oth = __ldg(G.inc_oth + q);
  if (oth.x >= 0) return words[oth.x] ^ words[oth.y];
  const int e = __ldg(G.inc_edge + q);
  uint32_t p = 0u;
  for (uint32_t m = __ldg(G.hptr + e), me = __ldg(G.hptr + e + 1); m < me; ++m) {
    const int mm = __ldg(G.hmem + m);
    if (mm != j) p ^= words[mm] ^ inv;
  }
  return p;
}

// Replica r's place in spin j's row of fields: quads of replicas are turned by the
// spin, so that lanes reading the same quad of several spins spread over the banks
// of shared memory (cell grids' classes visit every 16th spin).
__device__ __forceinline__ int field_at(int j, int r) { return r ^ (((j ^ (j >> 4)) & 7) << 2); }

// The fields are stored; those against the spins (word w) are returned, in place.
__device__ __forceinline__ uint32_t own_store(float *F, int j, int r0, const float *f, uint32_t w) {
  F += (size_t)j * 32;
  *reinterpret_cast<float4 *>(F + field_at(j, r0)) = make_float4(f[0], f[1], f[2], f[3]);
  *reinterpret_cast<float4 *>(F + field_at(j, r0 + 4)) = make_float4(f[4], f[5], f[6], f[7]);
  uint32_t m = 0u;
  w >>= r0;
#pragma unroll
  for (int r = 0; r < 8; ++r)
    if ((w >> r) & 1u ? f[r] < 0.0f : f[r] > 0.0f) m |= 1u << r;
  return m << r0;
}

// From scratch: the exact sum in fixed point (the spin's unit), rounded to FP32.
__device__ __forceinline__ uint32_t own_refresh(const DevGraph &G, const InstDesc &I, const uint32_t *sw, float *F, int j,
                                                int r0, uint32_t k0, uint32_t k1, uint32_t e0, uint32_t e1, int unit) {
  const float *Jf = reinterpret_cast<const float *>(G.J), *hJ = reinterpret_cast<const float *>(G.hJ);
  int64_t sum = xr_term(__ldg(reinterpret_cast<const float *>(G.h) + I.spin_off + j), unit), acc[8] = {};
  auto add = [&](int64_t t, uint32_t minus) {
    sum += t;
    minus >>= r0;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if ((minus >> r) & 1u) acc[r] += t;
  };
  for (uint32_t k = k0; k < k1; ++k) add(xr_term(__ldg(Jf + k), unit), ~sw[__ldg(G.col + k)]);
  for (uint32_t q = e0; q < e1; ++q)
    add(xr_term(__ldg(hJ + __ldg(G.inc_edge + q)), unit), own_parity(G, sw, 0xffffffffu, j, q));
  float f[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) f[r] = xr_round(sum - 2 * acc[r], unit);
  return own_store(F, j, r0, f, sw[j]);
}

// Fewer than this many pending spins of a warp's 32 positions are visited by the
// whole warp, a lane per replica: its terms cost one add where four lanes take
// eight predicated ones each, and its marks take fewer steps.  Integers: 6,000 spins
// of degree 5, 20 replicas, 2 descents 889 -> 623 us (all by four lanes 639), 300
// spins 110 -> 114 (144); 1,000 spins, 1,024 replicas, 20 descents 982 -> 792 (3 / 6
// spins: 802 / 806).  FP32, where the fields are read and written besides: one or two,
// as in dense rows, small classes and the last sweeps (32 replicas, all by four lanes /
// from 2 / 3 / 4 / 5 spins: 200 spins of degree 40 1,096 / 561 / 543 / 535 / 545 us,
// 1,000 of degree 100 10.0 / 9.2 / 8.3 / 8.6 / 8.6 ms, 4,096 cell grids 3.26 / 3.22 /
// 3.24 / 3.28 / 3.33), up to three in instances of few spins (5,000 of 40 spins 748 /
// 654 / 527 / 516 / 520 us, 3,000 of 64 spins 515 / 498 / 465 / 432 / 433).
constexpr int kFewSpins = 80;  // ten a warp of the smallest CTA
template <int MODE>
__device__ __forceinline__ int own_least(int n) {
  return MODE == 0 || n <= kFewSpins ? 4 : 3;
}

// Integer couplings: the exact field from scratch, not kept.
__device__ __forceinline__ uint32_t own_int(const DevGraph &G, const InstDesc &I, const uint32_t *sw, int j, int r0,
                                            uint32_t k0, uint32_t k1, uint32_t e0, uint32_t e1) {
  const int8_t *Ji = reinterpret_cast<const int8_t *>(G.J), *hJ = reinterpret_cast<const int8_t *>(G.hJ);
  int sum = __ldg(reinterpret_cast<const int8_t *>(G.h) + I.spin_off + j), acc[8] = {};
  auto add = [&](int t, uint32_t minus) {
    sum += t;
    minus >>= r0;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if ((minus >> r) & 1u) acc[r] += t;
  };
  for (uint32_t k = k0; k < k1; ++k) add(__ldg(Ji + k), ~sw[__ldg(G.col + k)]);
  for (uint32_t q = e0; q < e1; ++q)
    add(__ldg(hJ + __ldg(G.inc_edge + q)), own_parity(G, sw, 0xffffffffu, j, q));
  const uint32_t w = sw[j] >> r0;
  uint32_t m = 0u;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int f = sum - 2 * acc[r];
    if ((w >> r) & 1u ? f < 0 : f > 0) m |= 1u << r;
  }
  return m << r0;
}

// By the neighbours' flips since the previous visit (their words in fm), in CSR order
// and then by hyper-edge; a replica with none keeps its field and its spin.
__device__ __forceinline__ uint32_t own_visit(const DevGraph &G, const uint32_t *sw, const uint32_t *fm, float *F, int j,
                                              int r0, uint32_t k0, uint32_t k1, uint32_t e0, uint32_t e1) {
  const float *Jf = reinterpret_cast<const float *>(G.J), *hJ = reinterpret_cast<const float *>(G.hJ);
  constexpr int kPre = 6;  // row entries fetched together
  const int dg = (int)(k1 - k0);
  uint32_t pf[kPre], ps[kPre], dirty = 0u;
  float pw[kPre];
#pragma unroll
  for (int q = 0; q < kPre; ++q) {
    pf[q] = 0u;
    if (q < dg) {
      const int i = __ldg(G.col + k0 + q);
      pw[q] = 2.0f * __ldg(Jf + k0 + q);
      pf[q] = fm[i];
      ps[q] = ~sw[i];
      dirty |= pf[q];
    }
  }
  const bool more = dg > kPre || e1 > e0;
  if (!more && !((dirty >> r0) & 0xffu)) return 0u;
  const float4 a = *reinterpret_cast<const float4 *>(F + (size_t)j * 32 + field_at(j, r0));
  const float4 b = *reinterpret_cast<const float4 *>(F + (size_t)j * 32 + field_at(j, r0 + 4));
  float f[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  auto pull = [&](float w2, uint32_t flipped, uint32_t minus) {
    flipped >>= r0;
    minus >>= r0;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if ((flipped >> r) & 1u)
        f[r] = __fadd_rn(f[r], __uint_as_float(__float_as_uint(w2) ^ ((minus << (31 - r)) & 0x80000000u)));
  };
#pragma unroll
  for (int q = 0; q < kPre; ++q) pull(pw[q], pf[q], ps[q]);
  if (more) {
    for (uint32_t k = k0 + kPre; k < k1; ++k) {
      const int i = __ldg(G.col + k);
      dirty |= fm[i];
      pull(2.0f * __ldg(Jf + k), fm[i], ~sw[i]);
    }
    for (uint32_t q = e0; q < e1; ++q) {
      const uint32_t p = own_parity(G, fm, 0u, j, q);
      dirty |= p;
      pull(2.0f * __ldg(hJ + __ldg(G.inc_edge + q)), p, own_parity(G, sw, 0xffffffffu, j, q));
    }
  }
  return own_store(F, j, r0, f, sw[j]) & dirty;
}

}  // namespace

// SEG: tiles in segments of descents.  (A separate instantiation: the segments'
// few values in the whole-tile kernel spill at 64 registers and cost full batches
// 8 %.)  SEQ: the index order, at 256 threads and with segments (one where there are
// none); its tests in the colour order's loops cost small instances 4 %.
template <int MODE, int THREADS, bool SEG, bool SEQ = false>
__global__ void __launch_bounds__(THREADS, (MODE == 3 ? 512 : 1024) / THREADS < 1 ? 1 : (MODE == 3 ? 512 : 1024) / THREADS)
tile_kernel(const __grid_constant__ TileArgs A) {
  // (a parameter, so that its pointers stay in constant memory: read through a pointer
  // they took registers, and the 64 spilled)
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ int s_tile, s_last, s_segs;
  __shared__ bool s_merge;
  __shared__ uint32_t s_any, s_active, s_convround, s_upd;
  __shared__ int32_t s_total[32], s_minima[32];
  __shared__ double s_best[32], s_E[32];
  __shared__ double s_red[THREADS];
  __shared__ uint8_t s_slot[MODE <= 1 ? THREADS : 32];
  __shared__ int s_cnt[33];

  const DevGraph &G = A.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = THREADS / 32;
  const int nmax = A.nmax;
  uint32_t *sw = smem;
  uint32_t *fm = smem + nmax;
  // pending bits: spin i's bit is set when a neighbour flipped (in any lane)
  // since i's last visit; a spin without it keeps its field and stays stable
  uint32_t *pb = smem + (MODE >= 2 ? 1 : 2) * nmax;
  uint32_t *bw = A.bw + (size_t)blockIdx.x * nmax;
  float *F = A.F ? A.F + (size_t)blockIdx.x * nmax * 32 : nullptr;
  // FP32 fields of instances up to A.fsm_cap spins stay in shared memory
  float *Fs = reinterpret_cast<float *>(smem + (((MODE >= 2 ? 1 : 2) * nmax + (nmax + 31) / 32 + 3) & ~3));
  // Work counters: thread 0's sweep-level counts go straight to shared memory;
  // every thread counts its flips and evaluated pairs of the current sweep in
  // 32 bits and adds the warp's total at the end of each sweep.
  //   s_work: 0 flip_evals, 1 flips, 2 minima, 3 descents, 4 sweeps, 5 evaluated
  __shared__ unsigned long long s_work[6];
  if (tid < 6) s_work[tid] = 0;
  if (SEG && tid == 0) s_segs = A.segs;  // (read where it is needed: registers are short)
  uint32_t my_flips = 0, my_eval = 0;

  for (;;) {
    if (tid == 0) s_tile = atomicAdd(A.queue, 1);
    __syncthreads();
    const int t = s_tile;
    if (t >= (SEG ? A.n_tiles * s_segs : A.n_tiles)) break;
    const int b = A.tiles[SEG ? t / s_segs : t].x, g = A.tiles[SEG ? t / s_segs : t].y;
    if (SEG && tid == 0) s_last = (int)((int64_t)A.restarts * (t % s_segs + 1) / s_segs);  // end of its descents
    const InstDesc I = G.inst[b];
    const int n = I.n;
    const int rem = A.R - 32 * g;
    const uint32_t lane_valid = rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u);
    const uint64_t seed = A.seeds[b];
    // On lanes, warp 0 takes the spins of the index order one after another and the
    // others wait for the sweep's end; multi-spin coded, a thread takes one and the
    // CTA waits for it.
    constexpr bool seq = MODE <= 1 && SEQ;
    const int ncls = seq ? 1 : (SEQ ? n : I.ncls);
    float *Fc = (MODE == 1 && n <= A.fsm_cap) ? Fs : F;
    if (tid < 32) {
      s_total[tid] = 0;
      s_minima[tid] = 0;
      s_best[tid] = DBL_MAX;
    }
    __syncthreads();

    for (int k = SEG ? (int)((int64_t)A.restarts * (t % s_segs) / s_segs) : 0;; ++k) {
      if (tid == 0) {
        uint32_t start = 0;
        if (k < (SEG ? s_last : A.restarts))
          for (int r = 0; r < 32; ++r)
            if (((lane_valid >> r) & 1u) && (A.budget <= 0 || s_total[r] < A.budget)) start |= 1u << r;
        s_active = start;
        s_convround = 0;
        s_work[3] += __popc(start);
      }
      __syncthreads();
      uint32_t active = s_active;
      if (!active) break;

      // Random starts for the lanes beginning descent k (Sec. IV); a warp
      // transposes 32 replicas x 128 spins with shuffle exchanges.
      for (int w = warp; w * 128 < n; w += nwarps) {
        const uint4 x = start_bits(seed, (uint32_t)w, (uint32_t)(32 * g + lane), (uint32_t)k, (uint32_t)b);
        for (int q = 0; q < 4; ++q) {
          const uint32_t xw = word_of(x, q);
          const uint32_t mine = warp_transpose32(xw, lane);  // lane u: site u's word
          const int i = w * 128 + q * 32 + lane;
          if (i < n) {
            sw[i] = (sw[i] & ~active) | (mine & active);
            if (MODE == 1) fm[i] &= ~active;
          }
        }
      }
      __syncthreads();

      for (int d = 0; active; ++d) {
        const bool refresh = (d == 0) || (A.refresh > 0 && d % A.refresh == 0);
        const bool fresh = MODE == 1 ? refresh : d == 0;  // every spin is evaluated
        auto pending = [&](int j) -> bool { return fresh || ((pb[j >> 5] >> (j & 31)) & 1u); };
        auto clear_pending = [&](int j) {
          if ((pb[j >> 5] >> (j & 31)) & 1u) atomicAnd(&pb[j >> 5], ~(1u << (j & 31)));
        };
        auto mark = [&](int i) { atomicOr(&pb[i >> 5], 1u << (i & 31)); };
        if (tid == 0) s_any = 0;
        uint32_t anyf = 0;
        for (int c = 0; c < ncls; ++c) {
          int c0, c1;
          if (SEQ) {
            c0 = c;
            c1 = seq ? n : c + 1;
          } else {
            c0 = __ldg(G.cls + I.cls_off + c);
            c1 = __ldg(G.cls + I.cls_off + c + 1);
          }
          if (MODE == 3) {
            // +/-1 periodic lattice, |h| <= 1: the field counts as one more
            // bond, so every site flips when at least deg/2 + 1 of its bonds and
            // field are unsatisfied (3-d: majority of three carries; 2-d: >= 3).
            const int L = I.lat_L, D = I.lat_d;
            const int stride[3] = {1, L, L * L};
            for (int v = c0 + tid; v < c1; v += THREADS) {
              const int j = __ldg(G.order + I.spin_off + v);
              if (!pending(j)) continue;
              clear_pending(j);
              my_eval += __popc(active);
              const uint32_t info = __ldg(G.latinfo + I.spin_off + v);
              const int hv = __ldg(reinterpret_cast<const int8_t *>(G.h) + I.spin_off + j);
              const uint32_t wj = sw[j];
              uint32_t x[6];
#pragma unroll
              for (int d = 0; d < 6; ++d) {
                x[d] = 0u;
                if (d < 2 * D) {
                  const int a = d >> 1, st = stride[a];
                  int nb = (d & 1) ? j - st : j + st;
                  if ((info >> d) & 1u) nb += (d & 1) ? L * st : -L * st;
                  x[d] = wj ^ sw[nb] ^ (((info >> (8 + d)) & 1u) ? 0xffffffffu : 0u);
                }
              }
              const uint32_t uf = hv == 0 ? 0u : (hv > 0 ? ~wj : wj);
              uint32_t flip;
              const uint32_t s1 = x[0] ^ x[1] ^ x[2], c1 = (x[0] & x[1]) | (x[0] & x[2]) | (x[1] & x[2]);
              if (D == 3) {
                const uint32_t s2 = x[3] ^ x[4] ^ x[5], c2 = (x[3] & x[4]) | (x[3] & x[5]) | (x[4] & x[5]);
                const uint32_t c3 = (s1 & s2) | (s1 & uf) | (s2 & uf);
                flip = (c1 & c2) | (c1 & c3) | (c2 & c3);  // count >= 4
              } else {
                const uint32_t s2 = x[3] ^ uf ^ s1, c2 = (x[3] & uf) | (x[3] & s1) | (uf & s1);
                flip = (c1 & c2) | ((c1 | c2) & s2);  // count >= 3
              }
              flip &= active;
              if (flip)
                for (int d = 0; d < 2 * D; ++d) {
                  const int a = d >> 1, st = stride[a];
                  int nb = (d & 1) ? j - st : j + st;
                  if ((info >> d) & 1u) nb += (d & 1) ? L * st : -L * st;
                  mark(nb);
                }
              sw[j] = wj ^ flip;
              anyf |= flip;
              my_flips += __popc(flip);
            }
          } else if (MODE == 2) {
            const int8_t *Ji = reinterpret_cast<const int8_t *>(G.J);
            const int8_t *hi = reinterpret_cast<const int8_t *>(G.h);
            for (int v = c0 + tid; v < c1; v += THREADS) {
              const int j = SEQ ? v : __ldg(G.order + I.spin_off + v);
              if (!pending(j)) continue;
              clear_pending(j);
              my_eval += __popc(active);
              const int64_t gj = I.spin_off + j;
              const uint32_t wj = sw[j];
              uint32_t c0b = 0, c1b = 0, c2b = 0, c3b = 0;
              const uint32_t k0 = __ldg(G.row + gj), k1 = __ldg(G.row + gj + 1);
              for (uint32_t kk = k0; kk < k1; ++kk) {
                const int i = __ldg(G.col + kk);
                const uint32_t neg = __ldg(Ji + kk) < 0 ? 0xffffffffu : 0u;
                uint32_t x = wj ^ sw[i] ^ neg;  // unsatisfied bond
                uint32_t cy = c0b & x;
                c0b ^= x;
                x = cy;
                cy = c1b & x;
                c1b ^= x;
                x = cy;
                cy = c2b & x;
                c2b ^= x;
                c3b ^= cy;
              }
              const int deg = (int)(k1 - k0);
              const int hv = __ldg(hi + gj);
              // flip iff 2u > deg + h s  (dE = 2 s f < 0 with |J| = 1)
              uint32_t flip;
              if (hv == 0) {
                flip = sliced_ge(c0b, c1b, c2b, c3b, deg / 2 + 1);
              } else {
                const uint32_t plus = hv > 0 ? wj : ~wj;  // lanes with h s = +1
                const int tp = (deg + 1) / 2 + 1;
                const int tm = deg >= 1 ? (deg - 1) / 2 + 1 : 0;
                flip = (sliced_ge(c0b, c1b, c2b, c3b, tp) & plus) |
                       (sliced_ge(c0b, c1b, c2b, c3b, tm) & ~plus);
              }
              flip &= active;
              if (flip)
                for (uint32_t kk = k0; kk < k1; ++kk) mark(__ldg(G.col + kk));
              sw[j] = wj ^ flip;
              anyf |= flip;
              my_flips += __popc(flip);
            }
          } else {
            // The warp's positions v = c0 + warp + k nwarps, 32 at a time: lane k
            // reads position k's spin and pending bit (one round trip for the 32),
            // a position with nothing pending is settled at once (its visit flips
            // nothing), and the others are visited in order.
            // (In index order warp 0's next 32 spins; each one's pending bit is read
            // when its turn comes.)
            const int vstep = seq ? 1 : nwarps;
            for (int vb = seq && warp ? c1 : c0 + warp; vb < c1; vb += 32 * vstep) {
              const int vl = vb + lane * vstep;
              const bool inr = vl < c1;
              const int jl = inr ? (seq ? vl : __ldg(G.order + I.spin_off + vl)) : 0;
              const bool pl = inr && (seq || pending(jl));
              if (MODE == 1 && inr && !pl && fm[jl]) fm[jl] = 0u;
              // a pending position's row and hyper-edge bounds, read with the batch
              uint32_t k0l = 0, k1l = 0, e0l = 0, e1l = 0;
              if (pl) {
                const int64_t g = I.spin_off + jl;
                k0l = __ldg(G.row + g);
                k1l = __ldg(G.row + g + 1);
                e0l = __ldg(G.inc_ptr + g);
                e1l = __ldg(G.inc_ptr + g + 1);
              }
              uint32_t todo = __ballot_sync(0xffffffffu, pl);
              if (!seq) {
                const int ul = MODE == 1 && refresh && pl ? __ldg(G.runit + I.spin_off + jl) : 0;
                uint32_t own = __ballot_sync(0xffffffffu, pl && ul >= 0);
                if (__popc(own) < own_least<MODE>(n)) own = 0u;
                if (own) {
                  if ((own >> lane) & 1u) s_slot[(tid & ~31) + __popc(own & ((1u << lane) - 1u))] = (uint8_t)lane;
                  __syncwarp();
                  const int cnt = __popc(own), r0 = 8 * (lane & 3);
                  for (int p = lane >> 2; p - (lane >> 2) < cnt; p += 8) {
                    const bool on = p < cnt;
                    const int src = on ? s_slot[(tid & ~31) + p] : 0;
                    const int j = __shfl_sync(0xffffffffu, jl, src);
                    const uint32_t k0 = __shfl_sync(0xffffffffu, k0l, src), k1 = __shfl_sync(0xffffffffu, k1l, src);
                    const uint32_t e0 = __shfl_sync(0xffffffffu, e0l, src), e1 = __shfl_sync(0xffffffffu, e1l, src);
                    const int u = __shfl_sync(0xffffffffu, ul, src);
                    uint32_t m = 0u;
                    if (MODE == 0) {
                      if (on) m = active & own_int(G, I, sw, j, r0, k0, k1, e0, e1);
                    } else if (on)
                      m = active & (refresh ? own_refresh(G, I, sw, Fc, j, r0, k0, k1, e0, e1, u)
                                            : own_visit(G, sw, fm, Fc, j, r0, k0, k1, e0, e1));
                    m |= __shfl_xor_sync(0xffffffffu, m, 1);
                    m |= __shfl_xor_sync(0xffffffffu, m, 2);
                    if (!on) continue;
                    if (r0 == 0) {
                      my_eval += __popc(active);
                      my_flips += __popc(m);
                      clear_pending(j);
                      sw[j] ^= m;
                      if (MODE == 1) fm[j] = m;
                      anyf |= m;
                    }
                    if (m) {
                      for (uint32_t kk = k0 + (lane & 3); kk < k1; kk += 4) mark(__ldg(G.col + kk));
                      for (uint32_t q = e0; q < e1; ++q) {
                        const int2 oth = __ldg(G.inc_oth + q);
                        if (oth.x >= 0) {
                          if ((lane & 3) < 2) mark((lane & 3) == 0 ? oth.x : oth.y);
                          continue;
                        }
                        const int e = __ldg(G.inc_edge + q);
                        for (uint32_t mm = __ldg(G.hptr + e) + (lane & 3), me = __ldg(G.hptr + e + 1); mm < me; mm += 4) {
                          const int o = __ldg(G.hmem + mm);
                          if (o != j) mark(o);
                        }
                      }
                    }
                  }
                  todo &= ~own;
                  __syncwarp();
                }
              }
              while (todo) {
              const int src = __ffs(todo) - 1;
              todo &= todo - 1u;
              const int j = __shfl_sync(0xffffffffu, jl, src);
              if (seq) {
                __syncwarp();  // the flips and marks of the spins before
                if (!pending(j)) {
                  if (MODE == 1 && lane == 0) fm[j] = 0u;
                  continue;
                }
              }
              const int64_t gj = I.spin_off + j;
              const uint32_t wj = sw[j];
              const bool up = (wj >> lane) & 1u;
              const uint32_t k0 = __shfl_sync(0xffffffffu, k0l, src), k1 = __shfl_sync(0xffffffffu, k1l, src);
              const uint32_t e0 = __shfl_sync(0xffffffffu, e0l, src), e1 = __shfl_sync(0xffffffffu, e1l, src);
              bool flip;
              if (MODE == 0) {
                const int8_t *Ji = reinterpret_cast<const int8_t *>(G.J);
                const int8_t *hJ = reinterpret_cast<const int8_t *>(G.hJ);
                int f = __ldg(reinterpret_cast<const int8_t *>(G.h) + gj);
                for (uint32_t kk = k0; kk < k1; ++kk) {
                  const int i = __ldg(G.col + kk);
                  const int w = __ldg(Ji + kk);
                  f += ((sw[i] >> lane) & 1u) ? w : -w;
                }
                for (uint32_t q = e0; q < e1; ++q) {
                  const int e = __ldg(G.inc_edge + q);
                  const int2 oth = __ldg(G.inc_oth + q);
                  uint32_t neg = 0;
                  if (oth.x >= 0) {
                    neg = (~(sw[oth.x] >> lane) & 1u) ^ (~(sw[oth.y] >> lane) & 1u);
                  } else {
                    for (uint32_t m = __ldg(G.hptr + e), me = __ldg(G.hptr + e + 1); m < me; ++m) {
                      const int mm = __ldg(G.hmem + m);
                      if (mm != j) neg ^= ~(sw[mm] >> lane) & 1u;
                    }
                  }
                  const int w = __ldg(hJ + e);
                  f += neg ? -w : w;
                }
                flip = up ? (f < 0) : (f > 0);
              } else {
                const float *Jf = reinterpret_cast<const float *>(G.J);
                const float *hJ = reinterpret_cast<const float *>(G.hJ);
                const uint32_t bit = 1u << lane;
                // +1 products of an incidence's other spins
                auto product = [&](uint32_t q) -> uint32_t { return ~own_parity(G, sw, 0xffffffffu, j, q); };
                float f;
                bool dirty = true;
                if (refresh) {
                  const float hj = __ldg(reinterpret_cast<const float *>(G.h) + gj);
                  const int u = __ldg(G.runit + gj);
                  if (u >= 0) {
                    int64_t acc = xr_term(hj, u);
                    for (uint32_t kk = k0; kk < k1; ++kk) {
                      const int64_t t = xr_term(__ldg(Jf + kk), u);
                      acc += sw[__ldg(G.col + kk)] & bit ? t : -t;
                    }
                    for (uint32_t q = e0; q < e1; ++q) {
                      const int64_t t = xr_term(__ldg(hJ + __ldg(G.inc_edge + q)), u);
                      acc += product(q) & bit ? t : -t;
                    }
                    f = xr_round(acc, u);
                  } else {  // no exact unit: the FP64 sum in order, rounded
                    double acc = (double)hj;
                    for (uint32_t kk = k0; kk < k1; ++kk) {
                      const double w = (double)__ldg(Jf + kk);
                      acc = __dadd_rn(acc, sw[__ldg(G.col + kk)] & bit ? w : -w);
                    }
                    for (uint32_t q = e0; q < e1; ++q) {
                      const double w = (double)__ldg(hJ + __ldg(G.inc_edge + q));
                      acc = __dadd_rn(acc, product(q) & bit ? w : -w);
                    }
                    f = __double2float_rn(acc);
                  }
                } else {
                  // the flips of the neighbours since the previous visit, in order; the
                  // words are the warp's, so every lane takes each term or leaves it
                  // without a branch
                  f = Fc[(size_t)j * 32 + field_at(j, lane)];
                  uint32_t dirtyw = 0u;  // replicas whose field changes
                  auto pull = [&](float w2, uint32_t flipped, uint32_t plus) {
                    const float g = __fadd_rn(f, plus & bit ? w2 : -w2);
                    f = flipped & bit ? g : f;
                    dirtyw |= flipped;
                  };
#pragma unroll 4
                  for (uint32_t kk = k0; kk < k1; ++kk) {
                    const int i = __ldg(G.col + kk);
                    pull(2.0f * __ldg(Jf + kk), fm[i], sw[i]);
                  }
                  for (uint32_t q = e0; q < e1; ++q)
                    pull(2.0f * __ldg(hJ + __ldg(G.inc_edge + q)), own_parity(G, fm, 0u, j, q), product(q));
                  dirty = dirtyw & bit;
                }
                if (dirty) Fc[(size_t)j * 32 + field_at(j, lane)] = f;
                flip = dirty && (up ? f < 0.0f : f > 0.0f);
              }
              flip = flip && ((active >> lane) & 1u);
              const uint32_t m = __ballot_sync(0xffffffffu, flip);
              if (lane == 0) {
                my_eval += __popc(active);
                clear_pending(j);
                sw[j] = wj ^ m;
                if (MODE == 1) fm[j] = m;
              }
              if (m) {
                // the neighbours' pending marks, one lane per row entry / member
                for (uint32_t kk = k0 + lane; kk < k1; kk += 32) mark(__ldg(G.col + kk));
                for (uint32_t q = e0; q < e1; ++q) {
                  const int2 oth = __ldg(G.inc_oth + q);
                  if (oth.x >= 0) {
                    if (lane < 2) mark(lane == 0 ? oth.x : oth.y);
                    continue;
                  }
                  const int e = __ldg(G.inc_edge + q);
                  for (uint32_t mm = __ldg(G.hptr + e) + lane, me = __ldg(G.hptr + e + 1); mm < me; mm += 32) {
                    const int o = __ldg(G.hmem + mm);
                    if (o != j) mark(o);
                  }
                }
              }
              anyf |= m;
              my_flips += flip ? 1 : 0;
              }
            }
          }
          __syncthreads();
        }
        // end of sweep: which lanes flipped at all?
        anyf = __reduce_or_sync(0xffffffffu, anyf);
        if (lane == 0 && anyf) atomicOr(&s_any, anyf);
        {
          const uint32_t wf = __reduce_add_sync(0xffffffffu, my_flips);
          const uint32_t we = __reduce_add_sync(0xffffffffu, my_eval);
          if (lane == 0 && wf) atomicAdd(&s_work[1], (unsigned long long)wf);
          if (lane == 0 && we) atomicAdd(&s_work[5], (unsigned long long)we);
          my_flips = my_eval = 0;
        }
        __syncthreads();
        if (tid == 0) {
          const uint32_t any = s_any;
          uint32_t ended = 0;
          for (int r = 0; r < 32; ++r)
            if ((active >> r) & 1u) s_total[r] += 1;
          const uint32_t conv = active & ~any;
          ended |= conv;
          if (d + 1 >= A.max_sweeps) ended |= active;
          if (A.budget > 0)
            for (int r = 0; r < 32; ++r)
              if (((active >> r) & 1u) && s_total[r] >= A.budget) ended |= 1u << r;
          s_work[4] += __popc(active);
          s_work[0] += (unsigned long long)__popc(active) * (unsigned long long)n;
          s_work[2] += __popc(conv);
          s_convround |= conv;
          s_active = active & ~ended;
        }
        __syncthreads();
        active = s_active;
        if (!active) {
          // Round over: converged lanes have been frozen since their last sweep,
          // so all of them are scored in one lane-parallel pass.
          const uint32_t cr = s_convround;
          if (cr) {
            if (MODE == 3) tile_energy_lattice(G, I, sw, s_cnt, s_E);
            else if (n <= kFewSpins || !tile_energy_sites<MODE == 1, THREADS>(G, I, sw, s_red, s_E))
              tile_energy_lanes<MODE == 1>(G, I, sw, s_red, s_E);
            if (tid == 0) {
              uint32_t upd = 0;
              for (int r = 0; r < 32; ++r)
                if ((cr >> r) & 1u) {
                  s_minima[r] += 1;
                  if (s_E[r] < s_best[r]) {
                    s_best[r] = s_E[r];
                    upd |= 1u << r;
                  }
                }
              s_upd = upd;
            }
            __syncthreads();
            const uint32_t upd = s_upd;
            if (upd)
              for (int i = tid; i < n; i += THREADS) bw[i] = (bw[i] & ~upd) | (sw[i] & upd);
          }
        }
        __syncthreads();
      }
    }

    // Result per lane: best converged state, else the final state of its last descent.
    const int unit = SEG ? s_tile : 0, segs = SEG ? s_segs : 1, tile = unit / segs;
    uint32_t has_best = 0;
    for (int r = 0; r < 32; ++r)
      if (s_minima[r] > 0) has_best |= 1u << r;
    if ((lane_valid & ~has_best) && (!SEG || unit % segs == segs - 1)) {
      if (MODE == 3) tile_energy_lattice(G, I, sw, s_cnt, s_E);
      else if (n <= kFewSpins || !tile_energy_sites<MODE == 1, THREADS>(G, I, sw, s_red, s_E))
        tile_energy_lanes<MODE == 1>(G, I, sw, s_red, s_E);
      if (tid < 32 && !((has_best >> tid) & 1u)) s_best[tid] = s_E[tid];
    }
    __syncthreads();
    const uint32_t *from = nullptr;  // the words of the tile's segments
    if (SEG && segs > 1) {
      // this segment's words, energies and minima; the last CTA of the tile
      // chooses per lane among the segments (strictly lower energy, ties keep the
      // earlier; without a converged descent the last segment)
      uint32_t *words = A.seg_words + (size_t)unit * nmax;
      for (int i = tid; i < n; i += THREADS) words[i] = (bw[i] & has_best) | (sw[i] & ~has_best);
      if (tid < 32) {
        A.seg_best[(size_t)unit * 32 + tid] = s_best[tid];
        A.seg_minima[(size_t)unit * 32 + tid] = s_minima[tid];
      }
      __threadfence();
      __syncthreads();
      if (tid == 0) s_merge = atomicAdd(A.queue + 4 + tile, 1) == segs - 1;
      __syncthreads();
      if (!s_merge) continue;
      __threadfence();
      from = A.seg_words + (size_t)tile * segs * nmax;
      if (tid < 32) {
        double e = DBL_MAX;
        int m = 0, best = segs - 1;
        for (int q = 0; q < segs; ++q) {
          const size_t o = ((size_t)tile * segs + q) * 32 + tid;
          const int mq = __ldcg(A.seg_minima + o);
          const double eq = __ldcg(A.seg_best + o);
          m += mq;
          if (mq > 0 && eq < e) {
            e = eq;
            best = q;
          }
        }
        if (m == 0) e = __ldcg(A.seg_best + ((size_t)tile * segs + best) * 32 + tid);
        s_best[tid] = e;
        s_minima[tid] = m;
        s_total[tid] = best;
      }
      __syncthreads();
    }
    const int64_t out_base = (int64_t)A.R * I.spin_off + (int64_t)(32 * g) * n;
    // whole words of spins at 16-byte addresses: a transpose hands lane r replica r's
    // 32 spins of the warp, 32 bytes of its row (1,024 cell grids: 965 -> 941 us); else byte by byte
    const bool wide = (n & 31) == 0 && ((uintptr_t)(A.spins + out_base) & 15) == 0;
    for (int i = tid; i < n; i += THREADS) {
      uint32_t wv = 0;
      if (SEG && from) {
        for (int r = 0; r < 32; ++r) wv |= __ldcg(from + (size_t)s_total[r] * nmax + i) & (1u << r);
      } else {
        wv = (bw[i] & has_best) | (sw[i] & ~has_best);
      }
      if (wide) {
        const uint32_t mine = warp_transpose32(wv, lane);
        if ((lane_valid >> lane) & 1u) store_spins32(A.spins + out_base + (int64_t)lane * n + (i - lane), mine);
        continue;
      }
      for (int r = 0; r < 32; ++r)
        if ((lane_valid >> r) & 1u) A.spins[out_base + (int64_t)r * n + i] = ((wv >> r) & 1u) ? 1 : -1;
    }
    if (tid < 32 && ((lane_valid >> tid) & 1u)) {
      const int64_t o = (int64_t)b * A.R + 32 * g + tid;
      A.energy[o] = s_best[tid];
      if (A.energy_i32) A.energy_i32[o] = (int32_t)s_best[tid];
      if (A.minima) A.minima[o] = s_minima[tid];
    }
    __syncthreads();
  }

  // work counters
  __syncthreads();
  if (tid < 6 && s_work[tid]) atomicAdd(A.stats + tid, s_work[tid]);
}

size_t tile_smem_bytes(int mode, int nmax) {
  return (size_t)(mode >= 2 ? 1 : 2) * (size_t)nmax * sizeof(uint32_t) + (size_t)((nmax + 31) / 32) * sizeof(uint32_t);
}

size_t tile_smem_limit() { return 200 * 1024; }

// Spins whose FP32 fields (32 lanes) fit in shared memory next to the tile's
// words, within `budget` bytes of dynamic shared memory.
int tile_fsm_cap(int nmax, size_t budget) {
  const size_t base = (tile_smem_bytes(1, nmax) + 15) / 16 * 16;
  if (budget <= base) return 0;
  const size_t cap = (budget - base) / (32 * sizeof(float));
  return (int)std::min<size_t>(cap, (size_t)nmax);
}

namespace {
using TileKernel = void (*)(const TileArgs);
template <int MODE, bool SEG>
TileKernel tile_kernel_of(int threads) {
  return threads == 256 ? tile_kernel<MODE, 256, SEG> : (threads == 512 ? tile_kernel<MODE, 512, SEG> : tile_kernel<MODE, 1024, SEG>);
}
template <int MODE>
TileKernel tile_kernel_of(int threads, bool seg) {
  return seg ? tile_kernel_of<MODE, true>(threads) : tile_kernel_of<MODE, false>(threads);
}
TileKernel tile_kernel_for(int mode, int threads, bool seg, bool seq) {
  if (seq) return mode == 0 ? tile_kernel<0, 256, true, true> : (mode == 1 ? tile_kernel<1, 256, true, true> : tile_kernel<2, 256, true, true>);
  return mode == 0 ? tile_kernel_of<0>(threads, seg)
                   : (mode == 1 ? tile_kernel_of<1>(threads, seg)
                                : (mode == 2 ? tile_kernel_of<2>(threads, seg) : tile_kernel_of<3>(threads, seg)));
}
}  // namespace

int tile_max_ctas_per_sm(int mode, int threads, size_t smem, bool seq) {
  int blocks = 0, least = 0;
  for (int seg = 0; seg < 2; ++seg) {
    const TileKernel k = tile_kernel_for(mode, threads, seg != 0, seq);
    // (the same limit for every size: the attribute is the process's, and another
    // thread's handle may launch the same kernel at a larger size)
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem_limit());
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k, threads, smem);
    if (e != cudaSuccess) return 0;
    least = seg ? std::min(least, blocks) : blocks;
  }
  return least;
}

// Launch only: the shared-memory attribute was set by tile_max_ctas_per_sm.
cudaError_t launch_tile(const TileArgs &a, int mode, int threads, bool seg, int grid, size_t smem, cudaStream_t s) {
  tile_kernel_for(mode, threads, seg, a.sequential != 0)<<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace isg
