// energy.cu — energies of caller-supplied configurations (Eq. 1 extended by
// Eq. 6), int8 spins [instance][replica][spin].
//
// Integer couplings, and FP32 couplings whose terms are multiples of one unit
// (InstDesc::ebase): the spins are packed into words (bit r = replica r of a
// 32-replica group is -1), and every term is read once per group and added to
// the replicas whose bits select it, in integers (FP32: 64-bit fixed point, one
// rounding at the end).  With p_r the parity of a term's spins in replica r,
// -t prod s = -t + 2 t p_r, so E_r = -sum t + 2 sum_{p_r = 1} t.
// Otherwise (wider exponent ranges): two passes with a fixed summation order in
// FP64, chunks of kChunk spins (and a proportional share of the hyper-edges)
// and then their partial sums in order.  FP64 couplings: one thread per
// configuration takes the compensated sequential sum the C ABI defines.
#include <algorithm>
#include <type_traits>

#include "device_common.cuh"

namespace isg {

namespace {
constexpr int kChunk = 4096;
constexpr int kThreads = 256;


// ---- replica words ---------------------------------------------------------
// Instances of up to kTileSpins spins stay in one CTA's shared memory (pack, sum
// and write, one launch) when there are enough of them, or when they are so
// small that a second launch costs more than it spreads; others are packed into
// global words first and summed by CTAs of a part each.  A CTA pays about 5 us
// of dependent reads and reductions whatever its size, so the parts are as
// large as still fill the chip once (two CTAs per SM), within kPartMin and
// kPartMax: 10^6 sites and 16 replicas take 35 us in parts of 3,328 sites and 38 us
// in parts of 1,024 (a thread per configuration and spin with FP64 sums: 629 us);
// 60,000 spins of degree 5 and 32 replicas 23 us (256 us).
constexpr int kTileSpins = 2048;
constexpr int kTileAlways = 1024;
constexpr int kPartMin = 256;
constexpr int kPartMax = 4096;
constexpr int kWarps = kThreads / 32;
constexpr int kHalf = 16;  // replicas exchanged at a time in the warp totals

// words[i - i0] for sites i0 <= i < i1 of `cnt` replicas at s (replica stride n)
__device__ __forceinline__ void pack_sites(const int8_t *__restrict__ s, int n, int cnt, int i0, int i1,
                                           uint32_t *words) {
  if (!(n & 3) && !((uintptr_t)(s + i0) & 3)) {  // four sites per 4-byte load
    const int q4 = (i1 - i0) >> 2;
    for (int q = threadIdx.x; q < q4; q += blockDim.x) {
      const uint32_t *src = reinterpret_cast<const uint32_t *>(s + i0) + q;
      const int64_t st = n >> 2;
      uint32_t w0 = 0, w1 = 0, w2 = 0, w3 = 0;
#pragma unroll 8
      for (int r = 0; r < cnt; ++r) {
        const uint32_t v = __ldg(src + (int64_t)r * st);
        w0 |= ((v >> 7) & 1u) << r;
        w1 |= ((v >> 15) & 1u) << r;
        w2 |= ((v >> 23) & 1u) << r;
        w3 |= (v >> 31) << r;
      }
      uint32_t *dst = words + 4 * q;
      dst[0] = w0;
      dst[1] = w1;
      dst[2] = w2;
      dst[3] = w3;
    }
    for (int i = i0 + 4 * q4 + threadIdx.x; i < i1; i += blockDim.x) {
      uint32_t w = 0;
      for (int r = 0; r < cnt; ++r) w |= (uint32_t)(__ldg(s + (int64_t)r * n + i) < 0) << r;
      words[i - i0] = w;
    }
    return;
  }
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    uint32_t w = 0;
#pragma unroll 8
    for (int r = 0; r < cnt; ++r) w |= (uint32_t)(__ldg(s + (int64_t)r * n + i) < 0) << r;
    words[i - i0] = w;
  }
}

// Sum over the sites [i0, i1) (each pair at its smaller index, or at the site it
// leaves in the + direction on periodic lattices) and hyper-edges [ea, eb) of
// one replica group whose words are at sw (by local site index).  A lane adds
// its terms to NV per-replica registers; the warp totals go through shared
// memory, split into high and low 32-bit halves so that no cross-lane sum can
// overflow.  Returns in threads r < NV the CTA's (hi, lo) of replica r.
// Bound by latency: 100^3, 16 replicas, 33 us of 14 warps an SM at 105 registers, issue
// active 36 %, long_scoreboard the top stall (4.5 per issue); the predicated adds (three
// instructions per term and replica) keep the ALU pipe at 54 %.
template <bool FLOAT, int NV>
__device__ __forceinline__ void unit_energy(const DevGraph &G, const InstDesc &I, const uint32_t *sw, int i0, int i1,
                                            int ea, int eb, long long &hi, unsigned long long &lo) {
  using T = std::conditional_t<FLOAT, long long, int>;
  __shared__ T s_x[kWarps][kHalf][33];
  __shared__ long long s_hi[kWarps][NV];
  __shared__ unsigned long long s_lo[kWarps][NV];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ub = I.ebase;
  const int64_t so = I.spin_off;
  T acc[NV], csum = 0;
#pragma unroll
  for (int r = 0; r < NV; ++r) acc[r] = 0;
  auto value = [&](const void *arr, int64_t at) -> T {
    if constexpr (FLOAT) return (T)xr_term(__ldg(reinterpret_cast<const float *>(arr) + at), ub);
    else return (T)__ldg(reinterpret_cast<const int8_t *>(arr) + at);
  };
  auto add = [&](T t, uint32_t p) {
    csum += t;
#pragma unroll
    for (int r = 0; r < NV; ++r)
      if ((p >> r) & 1u) acc[r] += t;
  };
  if (I.lat_d > 0) {
    const int L = I.lat_L, n = I.n;
    // j / L for j < 2^24 by a reciprocal and one correction, else by division
    const float inv = 1.0f / (float)L;
    const bool small = n <= (1 << 24);
    auto div_L = [&](int j) -> int {
      if (!small) return j / L;
      int q = (int)((float)j * inv);
      const int rem = j - q * L;
      q += rem >= L ? 1 : (rem < 0 ? -1 : 0);
      return q;
    };
    // four sites at a time, their reads in one round trip
    constexpr int U = 4;
    const bool d3 = I.lat_d == 3;
    for (int jb = i0 + tid; jb < i1; jb += U * kThreads) {
      uint32_t w[U], p[U][3];
      T t[U][4];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = jb + u * kThreads;
        w[u] = 0u;
#pragma unroll
        for (int a = 0; a < 4; ++a) t[u][a] = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) p[u][a] = 0u;
        if (j < i1) {
          const int q1 = div_L(j), q2 = div_L(q1);
          const int x = j - q1 * L, y = q1 - q2 * L;  // (in two dimensions y = q1, q2 = 0)
          w[u] = sw[j];
          p[u][0] = sw[x == L - 1 ? j - (L - 1) : j + 1];
          p[u][1] = sw[y == L - 1 ? j - (L - 1) * L : j + L];
          t[u][0] = value(G.Jfwd, so + j);
          t[u][1] = value(G.Jfwd, G.nsp + so + j);
          if (d3) {
            p[u][2] = sw[q2 == L - 1 ? j - (L - 1) * L * L : j + L * L];
            t[u][2] = value(G.Jfwd, 2 * G.nsp + so + j);
          }
          t[u][3] = value(G.h, so + j);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        add(t[u][0], w[u] ^ p[u][0]);
        add(t[u][1], w[u] ^ p[u][1]);
        if (d3) add(t[u][2], w[u] ^ p[u][2]);
        if (t[u][3] != 0) add(t[u][3], w[u]);
      }
    }
  } else {
    // rows of 48 entries or more: a warp per row, lane per entry
    const bool by_row = I.max_deg >= 48;
    const int step = by_row ? kWarps : kThreads;
    for (int i = i0 + (by_row ? warp : tid); i < i1; i += step) {
      const uint32_t w = sw[i];
      const uint32_t k0 = __ldg(G.row + so + i), k1 = __ldg(G.row + so + i + 1);
      // four entries at a time: their columns and values, then their words
      const uint32_t st = by_row ? 32 : 1;
      for (uint32_t k = k0 + (by_row ? lane : 0); k < k1; k += 4 * st) {
        int j[4];
        T t[4];
        uint32_t p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = k + u * st < k1;
          j[u] = in ? __ldg(G.col + k + u * st) : -1;
          t[u] = in ? value(G.J, k + u * st) : (T)0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) p[u] = j[u] > i ? w ^ sw[j[u]] : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j[u] > i) add(t[u], p[u]);
      }
      if (!by_row || lane == 0) {
        const T th = value(G.h, so + i);
        if (th != 0) add(th, w);
      }
    }
    for (int e = ea + tid; e < eb; e += kThreads) {
      const int64_t ge = I.hyper_off + e;
      uint32_t p = 0;
      for (uint32_t q = __ldg(G.hptr + ge), qe = __ldg(G.hptr + ge + 1); q < qe; ++q) p ^= sw[__ldg(G.hmem + q)];
      add(value(G.hJ, ge), p);
    }
  }
#pragma unroll
  for (int r0 = 0; r0 < NV; r0 += kHalf) {
    constexpr int W = NV < kHalf ? NV : kHalf;  // replicas of this exchange
#pragma unroll
    for (int r = 0; r < W; ++r) s_x[warp][r][lane] = 2 * acc[r0 + r] - csum;
    __syncwarp();
    // 32 / W lanes per replica, W values each
    const int r = lane % W, part = lane / W;
    long long h = 0, l = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) {
      const long long v = (long long)s_x[warp][r][part * W + k];
      h += v >> 32;
      l += (long long)(uint32_t)v;
    }
#pragma unroll
    for (int o = W; o < 32; o <<= 1) {
      h += __shfl_xor_sync(0xffffffffu, h, o);
      l += __shfl_xor_sync(0xffffffffu, l, o);
    }
    if (lane < W) {
      s_hi[warp][r0 + lane] = h;
      s_lo[warp][r0 + lane] = (unsigned long long)l;
    }
    __syncwarp();
  }
  __syncthreads();
  hi = 0;
  lo = 0;
  if (tid < NV)
    for (int w = 0; w < kWarps; ++w) {
      hi += s_hi[w][tid];
      lo += s_lo[w][tid];
    }
}

// the total (hi, lo) of one (instance, replica) as its outputs
template <bool FLOAT>
__device__ __forceinline__ void write_energy(const InstDesc &I, long long hi, unsigned long long lo, int64_t o,
                                             double *E, int32_t *E32) {
  if (FLOAT) {
    E[o] = xe_value(hi, lo, I.ebase);
  } else {
    const long long v = hi * 4294967296ll + (long long)lo;
    E[o] = (double)v;
    if (E32) E32[o] = (int32_t)v;
  }
}

// One CTA per (instance, replica group), instances of at most kTileSpins spins.
template <bool FLOAT, int NV>
__global__ void __launch_bounds__(kThreads, 2) energy_tile_kernel(DevGraph G, const int8_t *__restrict__ spins,
                                                                  int32_t R, int32_t groups, double *E, int32_t *E32) {
  __shared__ uint32_t sw[kTileSpins];
  const int b = blockIdx.x / groups, g = blockIdx.x % groups;
  const InstDesc I = G.inst[b];
  const int cnt = min(32, R - 32 * g);
  pack_sites(spins + (int64_t)R * I.spin_off + (int64_t)(32 * g) * I.n, I.n, cnt, 0, I.n, sw);
  __syncthreads();
  long long hi;
  unsigned long long lo;
  unit_energy<FLOAT, NV>(G, I, sw, 0, I.n, 0, I.n_hyper, hi, lo);
  if (threadIdx.x < cnt) write_energy<FLOAT>(I, hi, lo, (int64_t)b * R + 32 * g + threadIdx.x, E, E32);
}

// Larger instances: words of every part, then the parts' sums.
__global__ void __launch_bounds__(kThreads) energy_pack_kernel(DevGraph G, const int8_t *__restrict__ spins, int32_t R,
                                                               int32_t groups, int32_t part,
                                                               const int4 *__restrict__ work, uint32_t *words) {
  const int4 wk = work[blockIdx.x];  // (instance, group, part, parts)
  const InstDesc I = G.inst[wk.x];
  const int i0 = wk.z * part, i1 = min(I.n, i0 + part);
  pack_sites(spins + (int64_t)R * I.spin_off + (int64_t)(32 * wk.y) * I.n, I.n, min(32, R - 32 * wk.y), i0, i1,
             words + (int64_t)groups * I.spin_off + (int64_t)wk.y * I.n + i0);
}

// acc[(b * groups + g)][32][2]: 64-bit sums over the parts (integers: the order
// does not matter), done[...]: parts finished.  The last part's CTA writes the
// energies and leaves both zero for the next call.
template <bool FLOAT, int NV>
__global__ void __launch_bounds__(kThreads, 2)
energy_part_kernel(DevGraph G, int32_t R, int32_t groups, int32_t part, const int4 *__restrict__ work,
                   const uint32_t *words, unsigned long long *acc, unsigned int *done, double *E, int32_t *E32) {
  __shared__ bool s_last;
  const int4 wk = work[blockIdx.x];
  const InstDesc I = G.inst[wk.x];
  const int i0 = wk.z * part, i1 = min(I.n, i0 + part);
  const int e_per = (I.n_hyper + wk.w - 1) / wk.w;
  const int ea = min(I.n_hyper, wk.z * e_per), eb = min(I.n_hyper, ea + e_per);
  long long hi;
  unsigned long long lo;
  unit_energy<FLOAT, NV>(G, I, words + (int64_t)groups * I.spin_off + (int64_t)wk.y * I.n, i0, i1, ea, eb, hi, lo);
  const int64_t slot = (int64_t)wk.x * groups + wk.y;
  const int t = threadIdx.x;
  if (t < NV) {
    atomicAdd(acc + (slot * 32 + t) * 2, (unsigned long long)hi);
    atomicAdd(acc + (slot * 32 + t) * 2 + 1, lo);
    __threadfence();
  }
  __syncthreads();
  if (t == 0) s_last = atomicAdd(done + slot, 1u) + 1u == (unsigned int)wk.w;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (t < NV) {
    hi = (long long)atomicExch(acc + (slot * 32 + t) * 2, 0ull);
    lo = atomicExch(acc + (slot * 32 + t) * 2 + 1, 0ull);
    if (t < min(32, R - 32 * wk.y)) write_energy<FLOAT>(I, hi, lo, (int64_t)wk.x * R + 32 * wk.y + t, E, E32);
  }
  if (t == 0) done[slot] = 0u;
}

template <bool FLOAT>
__global__ void __launch_bounds__(kThreads) energy_partial_kernel(DevGraph G, const int8_t *__restrict__ spins,
                                                                  int32_t R, const int4 *__restrict__ work,
                                                                  double *partd, long long *parti) {
  __shared__ double redd[kThreads / 32];
  __shared__ long long redi[kThreads / 32];
  const int4 wk = work[blockIdx.x];  // (b, r, chunk, nchunks)
  const InstDesc I = G.inst[wk.x];
  const int8_t *s = spins + (int64_t)R * I.spin_off + (int64_t)wk.y * I.n;
  const int i0 = wk.z * kChunk, i1 = min(I.n, i0 + kChunk);
  const int e_per = (I.n_hyper + wk.w - 1) / wk.w;
  const int ea = wk.z * e_per, eb = min(I.n_hyper, ea + e_per);
  if (FLOAT) {
    const float *Jf = reinterpret_cast<const float *>(G.J);
    const float *hf = reinterpret_cast<const float *>(G.h);
    const float *hJ = reinterpret_cast<const float *>(G.hJ);
    double acc = 0.0;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      const int64_t gi = I.spin_off + i;
      const double si = (double)s[i];
      double e = (double)__ldg(hf + gi) * si;
      for (uint32_t k = __ldg(G.row + gi), ke = __ldg(G.row + gi + 1); k < ke; ++k) {
        const int j = __ldg(G.col + k);
        if (j > i) e += (double)__ldg(Jf + k) * si * (double)s[j];
      }
      acc -= e;
    }
    for (int e = ea + threadIdx.x; e < eb; e += blockDim.x) {
      const int64_t ge = I.hyper_off + e;
      double p = 1.0;
      for (uint32_t q = __ldg(G.hptr + ge), qe = __ldg(G.hptr + ge + 1); q < qe; ++q)
        p *= (double)s[__ldg(G.hmem + q)];
      acc -= (double)__ldg(hJ + ge) * p;
    }
    acc = block_sum(acc, redd);
    if (threadIdx.x == 0) partd[blockIdx.x] = acc;
  } else {
    const int8_t *Ji = reinterpret_cast<const int8_t *>(G.J);
    const int8_t *hi = reinterpret_cast<const int8_t *>(G.h);
    const int8_t *hJ = reinterpret_cast<const int8_t *>(G.hJ);
    long long acc = 0;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      const int64_t gi = I.spin_off + i;
      const int si = s[i];
      int e = (int)__ldg(hi + gi) * si;
      for (uint32_t k = __ldg(G.row + gi), ke = __ldg(G.row + gi + 1); k < ke; ++k) {
        const int j = __ldg(G.col + k);
        if (j > i) e += (int)__ldg(Ji + k) * si * (int)s[j];
      }
      acc -= e;
    }
    for (int e = ea + threadIdx.x; e < eb; e += blockDim.x) {
      const int64_t ge = I.hyper_off + e;
      int p = 1;
      for (uint32_t q = __ldg(G.hptr + ge), qe = __ldg(G.hptr + ge + 1); q < qe; ++q)
        p *= (int)s[__ldg(G.hmem + q)];
      acc -= (long long)__ldg(hJ + ge) * p;
    }
    acc = block_sum(acc, redi);
    if (threadIdx.x == 0) parti[blockIdx.x] = acc;
  }
}

__global__ void energy_finish_kernel(const int4 *__restrict__ work, int32_t nwork, const int32_t *__restrict__ first,
                                     int32_t nout, int32_t R, const double *partd, const long long *parti,
                                     bool is_float, double *E, int32_t *E32) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;  // o = b * R + r
  if (o >= nout) return;
  const int w0 = first[o];
  const int nch = work[w0].w;
  if (is_float) {
    double acc = 0.0;
    for (int c = 0; c < nch; ++c) acc += partd[w0 + c];
    E[o] = acc;
  } else {
    long long acc = 0;
    for (int c = 0; c < nch; ++c) acc += parti[w0 + c];
    E[o] = (double)acc;
    if (E32) E32[o] = (int32_t)acc;
  }
  (void)nwork;
  (void)R;
}
// FP64 instances: the defined sequential compensated sum, one thread per
// (instance, replica)
__global__ void energy_f64_kernel(DevGraph G, int32_t n_inst, const int8_t *__restrict__ spins, int32_t R,
                                  double *E) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)n_inst * R) return;
  const int b = (int)(t / R), r = (int)(t % R);
  const InstDesc I = G.inst[b];
  E[t] = energy_f64_seq(G, I, spins + (int64_t)R * I.spin_off + (int64_t)r * I.n);
}

}  // namespace

void energy_plan_free(ising_handle *h) {
  void *ptrs[] = {h->d_en_work, h->d_en_first, h->d_en_partd, h->d_en_parti, h->d_en_words, h->d_en_acc};
  for (void *p : ptrs) cudaFree(p);
  h->d_en_work = nullptr;
  h->d_en_first = nullptr;
  h->d_en_partd = nullptr;
  h->d_en_parti = nullptr;
  h->d_en_words = nullptr;
  h->d_en_acc = nullptr;
  h->en_R = -1;
  h->en_nwork = 0;
}

namespace {

// Whether every instance's terms can be summed in integers: FP32 couplings with a
// unit whose terms, as many as one lane adds, fit 62 bits (doubled and offset by the
// constant: two more bits, within the 64); int8 ones whose sums fit 30 bits of 32 (not
// with some 2^27 couplings in the rows of a few spins).
bool integer_sums(const ising_handle *h) {
  const bool fl = h->dtype == ISING_F32;
  for (const InstDesc &I : h->inst) {
    if (fl && I.ebase < 0) return false;
    const bool by_row = I.max_deg >= 48;
    const int64_t sites = std::min<int64_t>(I.n, kPartMax);  // (a tile holds fewer)
    const int64_t parts = (I.n + sites - 1) / sites;
    const int64_t lane_sites = by_row ? (sites + kWarps - 1) / kWarps : (sites + kThreads - 1) / kThreads;
    // entries: the longest row at every site, or every row of the handle
    int64_t entries = lane_sites * (by_row ? (I.max_deg + 31) / 32 : I.max_deg);
    if (by_row) entries = std::min(entries, lane_sites + h->total_nnz / 32);
    const int64_t edges = ((I.n_hyper + parts - 1) / parts + kThreads - 1) / kThreads;
    const int64_t terms = lane_sites + entries + edges;
    int lg = 0;
    while (((int64_t)1 << lg) < terms) ++lg;
    if (I.ebits + lg > (fl ? 62 : 30) - 1) return false;
  }
  return true;
}

template <typename T>
cudaError_t put(T **dst, const std::vector<T> &src, cudaStream_t setup) {
  const cudaError_t e = cudaMalloc((void **)dst, src.size() * sizeof(T));
  return e != cudaSuccess ? e : cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, setup);
}

// Work list, words and accumulators of the packed form.  On failure nothing
// stays allocated.
cudaError_t plan_parts(ising_handle *h, int32_t R, int32_t groups) {
  (void)R;
  const int64_t fill = ((int64_t)groups * h->total_spins + 2 * h->sm_count - 1) / (2 * h->sm_count);
  h->en_part = (int32_t)std::min<int64_t>(kPartMax, std::max<int64_t>(kPartMin, (fill + 255) / 256 * 256));
  const int part = h->en_part;
  std::vector<int4> work;
  for (int b = 0; b < h->n_inst; ++b) {
    const int parts = (h->inst[b].n + part - 1) / part;
    for (int g = 0; g < groups; ++g)
      for (int c = 0; c < parts; ++c) work.push_back(make_int4(b, g, c, parts));
  }
  if (work.size() > 0x7fffffffu) return cudaErrorInvalidValue;
  const size_t slots = (size_t)h->n_inst * groups;
  const size_t acc_bytes = slots * 32 * 2 * sizeof(unsigned long long);
  cudaStream_t setup = nullptr;
  cudaError_t e = setup_stream(h, &setup);
  if (e == cudaSuccess) e = put(&h->d_en_work, work, setup);
  if (e == cudaSuccess) e = cudaMalloc((void **)&h->d_en_words, (size_t)groups * h->total_spins * sizeof(uint32_t));
  if (e == cudaSuccess) e = cudaMalloc((void **)&h->d_en_acc, acc_bytes + slots * sizeof(unsigned int));
  if (e == cudaSuccess) e = cudaMemsetAsync(h->d_en_acc, 0, acc_bytes + slots * sizeof(unsigned int), setup);
  if (e == cudaSuccess) e = cudaStreamSynchronize(setup);  // (before the caller's stream reads them)
  if (e != cudaSuccess) {
    energy_plan_free(h);
    return e;
  }
  h->en_nwork = (int32_t)work.size();
  return cudaSuccess;
}

// Work list and partial sums of the FP64 (or fallback) two-pass form.
cudaError_t plan_partials(ising_handle *h, int32_t R) {
  std::vector<int4> work;
  std::vector<int32_t> first;
  for (int b = 0; b < h->n_inst; ++b) {
    const int nch = (int)((h->inst[b].n + kChunk - 1) / kChunk);
    for (int r = 0; r < R; ++r) {
      first.push_back((int32_t)work.size());
      for (int c = 0; c < nch; ++c) work.push_back(make_int4(b, r, c, nch));
    }
  }
  cudaStream_t setup = nullptr;
  cudaError_t e = setup_stream(h, &setup);
  if (e == cudaSuccess) e = put(&h->d_en_work, work, setup);
  if (e == cudaSuccess) e = put(&h->d_en_first, first, setup);
  if (e == cudaSuccess) e = cudaStreamSynchronize(setup);
  if (e == cudaSuccess) e = cudaMalloc(&h->d_en_partd, work.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&h->d_en_parti, work.size() * sizeof(long long));
  if (e != cudaSuccess) {
    energy_plan_free(h);
    return e;
  }
  h->en_nwork = (int32_t)work.size();
  return cudaSuccess;
}

enum { kFormTile = 0, kFormParts = 1, kFormPartials = 2 };

template <bool FLOAT, int NV>
void run_packed(ising_handle *h, const int8_t *spins, int32_t R, int32_t groups, double *E, int32_t *E32,
                cudaStream_t s) {
  const DevGraph G = h->graph();
  if (h->en_form == kFormTile) {
    energy_tile_kernel<FLOAT, NV><<<(unsigned)((int64_t)h->n_inst * groups), kThreads, 0, s>>>(G, spins, R, groups, E, E32);
    return;
  }
  unsigned int *done = reinterpret_cast<unsigned int *>(h->d_en_acc + (size_t)h->n_inst * groups * 64);
  energy_pack_kernel<<<h->en_nwork, kThreads, 0, s>>>(G, spins, R, groups, h->en_part, h->d_en_work, h->d_en_words);
  energy_part_kernel<FLOAT, NV><<<h->en_nwork, kThreads, 0, s>>>(G, R, groups, h->en_part, h->d_en_work, h->d_en_words,
                                                                 h->d_en_acc, done, E, E32);
}

}  // namespace

// Host launcher: chooses the form and builds its work list once per replica
// count, then runs it on stream s.  Work lists, words and sums live in the handle.
cudaError_t launch_energy(ising_handle *h, const int8_t *spins, int32_t R, double *E, int32_t *E32,
                          cudaStream_t s) {
  cudaError_t e;
  if (h->dtype == ISING_F64) {
    const int64_t nout = (int64_t)h->n_inst * R;
    energy_f64_kernel<<<(int)((nout + 127) / 128), 128, 0, s>>>(h->graph(), h->n_inst, spins, R, E);
    return cudaGetLastError();
  }
  const int32_t groups = (R + 31) / 32;
  if (h->en_R != R) {
    energy_plan_free(h);
    h->en_form = kFormPartials;
    if (integer_sums(h) && (int64_t)h->n_inst * groups <= 0x7fffffff) {
      const bool many = (int64_t)h->n_inst * groups >= h->sm_count;
      if (h->nmax <= (many ? kTileSpins : kTileAlways)) h->en_form = kFormTile;
      else if (plan_parts(h, R, groups) == cudaSuccess) h->en_form = kFormParts;
      else cudaGetLastError();  // no room for the words: the two-pass form needs less
    }
    if (h->en_form == kFormPartials && (e = plan_partials(h, R)) != cudaSuccess) return e;
    h->en_R = R;
  }
  const bool fl = h->dtype == ISING_F32;
  if (h->en_form != kFormPartials) {
    if (R <= 4) fl ? run_packed<true, 4>(h, spins, R, groups, E, E32, s) : run_packed<false, 4>(h, spins, R, groups, E, E32, s);
    else if (R <= 16) fl ? run_packed<true, 16>(h, spins, R, groups, E, E32, s) : run_packed<false, 16>(h, spins, R, groups, E, E32, s);
    else fl ? run_packed<true, 32>(h, spins, R, groups, E, E32, s) : run_packed<false, 32>(h, spins, R, groups, E, E32, s);
    return cudaGetLastError();
  }
  const DevGraph G = h->graph();
  if (fl)
    energy_partial_kernel<true><<<h->en_nwork, kThreads, 0, s>>>(G, spins, R, h->d_en_work, h->d_en_partd, h->d_en_parti);
  else
    energy_partial_kernel<false><<<h->en_nwork, kThreads, 0, s>>>(G, spins, R, h->d_en_work, h->d_en_partd, h->d_en_parti);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int nout = h->n_inst * R;
  energy_finish_kernel<<<(nout + 255) / 256, 256, 0, s>>>(h->d_en_work, h->en_nwork, h->d_en_first, nout, R, h->d_en_partd,
                                                          h->d_en_parti, fl, E, E32);
  return cudaGetLastError();
}

}  // namespace isg
