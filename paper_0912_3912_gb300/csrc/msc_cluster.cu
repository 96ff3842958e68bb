// msc_cluster.cu — multi-spin-coded descent on periodic lattices with one
// thread-block cluster per (instance, 32-replica group).
//
// Same method and semantics as the multi-spin-coded tile kernel (García &
// Markov, Sec. IV: improving single-spin moves by colour class, a sweep without
// flips ends a descent, Philox restarts, best state kept), but the lattice is
// split over the P CTAs of a cluster: CTA q holds the spin words of sites
// [q n/P, (q+1) n/P) (whole z-slabs, or y-slabs in 2D) in its shared memory and
// reads the neighbour words owned by other CTAs through distributed shared
// memory.  The two checkerboard classes are separated by cluster barriers, so
// one lattice uses P SMs instead of one.
//
// Work layout: words lie by colour class, the site o of a CTA at place o >> 1 of
// its class's half (each row holds equally many sites of both parities).  A
// warp visits a chunk of 64 consecutive sites per step, lane t taking place t of
// the current class in the chunk; its neighbours are then the places t and t + 1
// or t - 1 of the row in the other class and the same places of the rows above and
// below, so the warp reads consecutive words (by site index they would lie two
// apart, two words to a bank) and the slab axis's remote reads are uniform.
// Coupling signs and the field of every site are one byte in shared memory.
// Pending flags per (class, chunk) say whether some site of the class in the chunk
// has a neighbour that flipped since its last visit; a chunk without one is
// stable and skipped (only the first sweep of a descent visits everything).  All
// per-lane bookkeeping (sweep counts, convergence, best energies) is replicated
// identically in every CTA of the cluster, so the cluster's control flow stays
// uniform and every barrier is matched.
//
// A visit is bound by its logic instructions (64 lanes a cycle and SM): on the 128 SMs
// that hold a CTA the ALU pipe is 74 % busy and 69 % of the issue slots are, the top
// stalls are not_selected 1.4, math pipe 1.2 and wait 1.1 per issue.  The class layout, sign planes, one pending target per lane and two chunks at a time took
// 32^3 with fields, 1,024 replicas, 10 descents from 719 to 535 us a call with four
// CTAs a cluster; two CTAs and two segments of descents each: 504, and 482 with the
// arguments as a parameter (their pointers in constant memory).  With 32 replicas,
// ten segments of eight CTAs: 467 -> 84 us.
#include <cfloat>
#include <type_traits>

#include "device_common.cuh"
#include "tc.cuh"

namespace isg {

namespace {

// CTAs of 512 threads, one per SM (two per SM at 64 registers, in clusters of
// 8, measured slower on the 32^3 lattice; 768 threads 640, 1,024 740 against 602 us)
constexpr int kCT = 512;

// MASKS: the signs and fields as bytes of 0 or -1, one plane per direction and two
// for the field, which the loads extend to whole words; else packed in one byte
// per site (large slabs, for shared memory's sake).
template <int D, bool MASKS>
__global__ void __launch_bounds__(kCT, 1) msc_cluster_kernel(const __grid_constant__ TileArgs A, int P) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ uint32_t s_any[2], s_active, s_convround, s_upd;
  __shared__ int32_t s_total[32], s_minima[32];
  __shared__ double s_best[32], s_E[32];
  __shared__ int32_t s_cnt[33];
  __shared__ int32_t s_rng[2][2];

  const DevGraph &G = A.g;
  const uint32_t rank = tc::cluster_rank();
  // one cluster per tile and segment of its descents (see the tile kernels)
  const int unit = blockIdx.x / P, segs = A.segs, tile = unit / segs;
  const int k0 = (int)((int64_t)A.restarts * (unit % segs) / segs), k1 = (int)((int64_t)A.restarts * (unit % segs + 1) / segs);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int b = A.tiles[tile].x, g = A.tiles[tile].y;
  const InstDesc I = G.inst[b];
  const int n = I.n, L = I.lat_L, lgL = 31 - __clz(L);
  const int csz = n / P;  // sites per CTA: a power of two, a multiple of 64 and of L^(D-1)
  const int lgc = 31 - __clz(csz);
  const int nch = csz >> 6;  // 64-site chunks per CTA
  const int lo = (int)rank * csz;
  const int half = csz >> 1, hl = L >> 1, lghl = lgL - 1;       // places per class, per row
  uint32_t *sw = smem;                                          // [2][half] words of sites lo .. lo + csz - 1
  uint32_t *pend = smem + csz;                                  // [2][nch] pending flags
  uint32_t *bw = smem + csz + 2 * nch;                          // [2][half]: best words of my sites
  // [2][half]: coupling signs (0 the x neighbour at the same place, 1 the other one,
  // 2, 3 +y, -y, 4, 5 +z, -z), h != 0, h > 0: bits of a byte, or eight planes
  uint8_t *tab = reinterpret_cast<uint8_t *>(smem + 2 * csz + 2 * nch);
  const int rem = A.R - 32 * g;
  const uint32_t lane_valid = rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u);
  const uint64_t seed = A.seeds[b];
  const int64_t so = I.spin_off;
  unsigned long long my_evals = 0, my_sweeps = 0, my_minima = 0, my_desc = 0;
  uint32_t my_flips = 0;  // of the current sweep
  unsigned long long all_flips = 0;
  unsigned long long my_eval = 0;  // (site, replica) pairs of the chunks visited (skipped chunks excluded)

  // class of global site j; place of a site of mine: cls * half + ((j - lo) >> 1)
  auto cls_of = [&](int j) -> int { return (j + (j >> lgL) + (D == 3 ? j >> (2 * lgL) : 0)) & 1; };
  auto place = [&](int j) -> int { return cls_of(j) * half + ((j - lo) >> 1); };
  // The neighbour words of place q of class c: x[0], x[1] in the row (the same place
  // of the other class, and the one beside it), then +y, -y (and +z, -z).  Only
  // neighbours along the slab axis (z in 3D, y in 2D) can lie in another CTA: those of
  // the slab's first and last step along it (`edge`; a chunk has one such coordinate).
  const int sstep = D == 3 ? hl << lgL : hl;  // places per step along the slab axis
  auto nwords = [&](auto edge, int c, int q, uint32_t (&x)[6]) {
    const uint32_t *oth = sw + (c ^ 1) * half;
    const int row = q >> lghl;  // local row
    const int s = ((lo >> lgL) + row + (D == 3 ? (lo >> (2 * lgL)) + (row >> lgL) : 0) + c) & 1;
    x[0] = oth[q];
    x[1] = oth[(q & ~(hl - 1)) | ((q + (s ? 1 : -1)) & (hl - 1))];  // (s: the site's x is odd)
    if (D == 3) {
      const int ym = (L - 1) << lghl;
      x[2] = oth[(q & ~ym) | ((q + hl) & ym)];
      x[3] = oth[(q & ~ym) | ((q - hl) & ym)];
    }
#pragma unroll
    for (int dn = 0; dn < 2; ++dn) {
      const int t = dn ? q - sstep : q + sstep;
      uint32_t w;
      if (!decltype(edge)::value || (t >= 0 && t < half))
        w = oth[t];
      else
        w = tc::ld_cluster_u32(tc::map_shared(oth + (t & (half - 1)), (rank + (dn ? P - 1 : 1)) & (P - 1)));
      x[2 * D - 2 + dn] = w;
    }
  };
  // Chunks holding the neighbours of a chunk's flipped sites (lanes: one target
  // each): the chunk itself, those of the rows above and below, of the planes above
  // and below and, in rows longer than a chunk, the next ones in the row; a lane's
  // target is due when one of the flipping lanes in its mask m_from flipped.
  //   target = (ch & ~m_wrap) | ((ch + m_step) & m_wrap), in the CTA m_rank once it
  //   leaves the slab
  const int cpr = L > 64 ? L >> 6 : 1, cpp = (L * L) >> 6;  // chunks per row, per plane
  const int m_edge = D == 3 ? cpp : cpr;  // chunks of the slab's first (last) step
  const uint32_t m_inner = __ballot_sync(0xffffffffu, warp + lane * nwarps >= m_edge && warp + lane * nwarps < nch - m_edge);
  uint32_t m_from = 0u;
  int m_step = 0, m_wrap = 0, m_rank = (int)rank;
  {
    const int dir = lane & 1 ? 1 : -1, kind = lane == 0 ? 0 : (lane + 1) >> 1;  // lanes 1, 2: y; 3, 4: z; 5, 6: x
    const uint32_t lastrow = hl >= 32 ? 0xffffffffu : ~0u << (32 - hl), firstrow = hl >= 32 ? 0xffffffffu : (1u << hl) - 1u;
    const bool slab = kind == D - 1;
    if (lane == 0) {
      m_from = 0xffffffffu;
    } else if (lane < 2 * D - 1 || (kind == 3 && L > 64)) {
      m_step = dir * (kind == 3 ? 1 : (kind == 2 ? cpp : cpr));
      m_wrap = slab ? nch - 1 : (kind == 3 ? cpr - 1 : cpp - 1);
      m_from = kind == 3 ? (dir > 0 ? 0x80000000u : 1u) : (slab ? 0xffffffffu : (dir > 0 ? lastrow : firstrow));
      if (slab) m_rank = (int)((rank + (dir > 0 ? 1 : P - 1)) & (P - 1));
    }
  }
  // sign (or field) mask d of place o: all ones or zeros in every replica
  auto mask = [&](int o, uint32_t t, int d) -> uint32_t {
    if (MASKS) return (uint32_t)(int32_t)reinterpret_cast<const int8_t *>(tab)[d * csz + o];
    return (t >> d) & 1u ? 0xffffffffu : 0u;
  };
  // my part of each colour class (positions whose site lies in [lo, lo + csz))
  if (tid < 2) {
    const int c = tid;
    int a = __ldg(G.cls + I.cls_off + c), e = __ldg(G.cls + I.cls_off + c + 1);
    int l1 = a, h1 = e;
    while (l1 < h1) {
      const int mid = (l1 + h1) >> 1;
      if (__ldg(G.order + so + mid) < lo) l1 = mid + 1;
      else h1 = mid;
    }
    int l2 = l1, h2 = e;
    while (l2 < h2) {
      const int mid = (l2 + h2) >> 1;
      if (__ldg(G.order + so + mid) < lo + csz) l2 = mid + 1;
      else h2 = mid;
    }
    s_rng[c][0] = l1;
    s_rng[c][1] = l2;
  }
  if (tid < 32) {
    s_total[tid] = 0;
    s_minima[tid] = 0;
    s_best[tid] = DBL_MAX;
  }
  if (tid < 2) s_any[tid] = 0u;
  for (int q = tid; q < 2 * nch; q += blockDim.x) pend[q] = 0u;
  __syncthreads();
  // per-site byte: coupling signs by direction and the field
  for (int c = 0; c < 2; ++c)
    for (int v = s_rng[c][0] + tid; v < s_rng[c][1]; v += blockDim.x) {
      const int j = __ldg(G.order + so + v);
      const uint32_t info = __ldg(G.latinfo + so + v);
      const int hv = __ldg(reinterpret_cast<const int8_t *>(G.h) + so + j);
      uint32_t neg = (info >> 8) & 63u;  // by direction: +x, -x, +y, -y, +z, -z
      if (j & 1) neg = (neg & ~3u) | ((neg >> 1) & 1u) | ((neg & 1u) << 1);  // (odd x: -x lies at the same place)
      neg |= (hv != 0 ? 64u : 0u) | (hv > 0 ? 128u : 0u);
      if (MASKS) {
        for (int d = 0; d < 8; ++d) tab[d * csz + place(j)] = (neg >> d) & 1u ? 0xffu : 0u;
      } else {
        tab[place(j)] = (uint8_t)neg;
      }
    }
  __syncthreads();

  // lane-parallel energies of the cluster's lattice: every CTA counts its own
  // sites (one site per thread, the forward bonds +x, +y, +z and the field),
  // the counts are summed over the cluster in rank order
  auto energies = [&]() {
    constexpr int Q = 8;  // per-thread counts stay below 2^8: at most 32 sites of D + 1 terms (csz <= 16384)
    uint32_t acc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = 0u;
    int nz = 0;
    if (tid < 33) s_cnt[tid] = 0;
    __syncthreads();
    for (int o = tid; o < csz; o += blockDim.x) {
      const int c = o >= half, q = o - c * half;
      const uint32_t wj = sw[o], t = MASKS ? 0u : tab[o];
      const uint32_t *oth = sw + (c ^ 1) * half;
      // +x is the neighbour at the same place for even x, else the one beside it
      const int row = q >> lghl;
      const int odd = ((lo >> lgL) + row + (D == 3 ? (lo >> (2 * lgL)) + (row >> lgL) : 0) + c) & 1;
      uint32_t f[3] = {0u, 0u, 0u};
      f[0] = wj ^ oth[(q & ~(hl - 1)) | ((q + odd) & (hl - 1))] ^ mask(o, t, odd);
      if (D == 3) {
        const int ym = (L - 1) << lghl;
        f[1] = wj ^ oth[(q & ~ym) | ((q + hl) & ym)] ^ mask(o, t, 2);
      }
      const int up = q + sstep;
      f[D - 1] = wj ^ mask(o, t, 2 * D - 2) ^
                 (up < half ? oth[up] : tc::ld_cluster_u32(tc::map_shared(oth + (up - half), (rank + 1) & (P - 1))));
      const uint32_t field = mask(o, t, 6), uf = (wj ^ mask(o, t, 7)) & field;
      nz += field & 1u;
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
    // lane r: replica r's warp total (a plane's transpose counts its bits: a third
    // of the exchanges of adding the planes across the lanes)
    int mine = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) mine += __popc(warp_transpose32(acc[q], lane)) << q;
    nz = warp_sum(nz);
    atomicAdd(&s_cnt[lane], mine);
    if (lane == 0) atomicAdd(&s_cnt[32], nz);
    __syncthreads();
    tc::cluster_sync();
    if (tid < 32) {
      long long u = 0, z = 0;
#pragma unroll 4
      for (int c = 0; c < P; ++c) {
        u += (int)tc::ld_cluster_u32(tc::map_shared(&s_cnt[tid], (uint32_t)c));
        z += (int)tc::ld_cluster_u32(tc::map_shared(&s_cnt[32], (uint32_t)c));
      }
      s_E[tid] = 2.0 * (double)u - (double)n * D - (double)z;
    }
    tc::cluster_sync();  // counts read everywhere before they are reset
  };

  uint32_t sc = 0;  // sweeps so far (all descents): picks the convergence buffer
  for (int k = k0;; ++k) {
    if (warp == 0) {
      const uint32_t start = __ballot_sync(
          0xffffffffu, k < k1 && ((lane_valid >> lane) & 1u) && (A.budget <= 0 || s_total[lane] < A.budget));
      if (lane == 0) {
        s_active = start;
        s_convround = 0;
        if (rank == 0) my_desc += __popc(start);
      }
    }
    __syncthreads();
    uint32_t active = s_active;
    if (!active) break;  // identical in every CTA of the cluster
    // random starts of my sites (Philox, counter layout of the C ABI)
    for (int w = (lo >> 7) + warp; w < ((lo + csz) >> 7); w += nwarps) {
      const uint4 x = start_bits(seed, (uint32_t)w, (uint32_t)(32 * g + lane), (uint32_t)k, (uint32_t)b);
      for (int q = 0; q < 4; ++q) {
        const uint32_t xw = word_of(x, q);
        const uint32_t mine = warp_transpose32(xw, lane);  // lane u: site u's word
        const int o = place(w * 128 + q * 32 + lane);
        sw[o] = active == lane_valid ? mine : (sw[o] & ~active) | (mine & active);
      }
    }
    tc::cluster_sync();

    for (int d = 0; active; ++d, ++sc) {
      const bool fresh = d == 0;
      const int pb = sc & 1;
      uint32_t anyf = 0;
      for (int c = 0; c < 2; ++c) {
        // the warp's chunks ch = warp + k nwarps: lane k reads chunk k's flag
        const int mych = warp + lane * nwarps;
        const bool pending = mych < nch && (fresh || pend[c * nch + mych]);
        if (pending) pend[c * nch + mych] = 0u;  // marks made in this phase go to the other class
        uint32_t todo = __ballot_sync(0xffffffffu, pending);
        if (lane == 0) my_eval += 32ull * (unsigned long long)(__popc(active) * __popc(todo));
        // one chunk: its words, then its decisions and the pending flags of the chunks
        // holding the flipped sites' neighbours (few branches: they cost more than what
        // they skip)
        auto load = [&](auto edge, int ch, uint32_t &wj, uint32_t &uf, uint32_t (&x)[6]) {
          const int q = ch * 32 + lane, o = c * half + q;
          wj = sw[o];
          const uint32_t t = MASKS ? 0u : tab[o];
          nwords(edge, c, q, x);
          uf = (wj ^ mask(o, t, 7)) & mask(o, t, 6);
#pragma unroll
          for (int dd = 0; dd < 2 * D; ++dd) x[dd] ^= wj ^ mask(o, t, dd);
        };
        auto decide = [&](auto edge, int ch, uint32_t wj, uint32_t uf, uint32_t (&x)[6]) {
          const int q = ch * 32 + lane;
          const uint32_t s1 = x[0] ^ x[1] ^ x[2], c1 = (x[0] & x[1]) | (x[0] & x[2]) | (x[1] & x[2]);
          uint32_t flip;
          if (D == 3) {
            const uint32_t s2 = x[3] ^ x[4] ^ x[5], c2 = (x[3] & x[4]) | (x[3] & x[5]) | (x[4] & x[5]);
            const uint32_t c3 = (s1 & s2) | (s1 & uf) | (s2 & uf);
            flip = (c1 & c2) | (c1 & c3) | (c2 & c3);
          } else {
            const uint32_t s2 = x[3] ^ uf ^ s1, c2 = (x[3] & uf) | (x[3] & s1) | (uf & s1);
            flip = (c1 & c2) | ((c1 | c2) & s2);
          }
          flip &= active;
          sw[c * half + q] = wj ^ flip;
          anyf |= flip;
          my_flips += __popc(flip);
          const uint32_t fb = __ballot_sync(0xffffffffu, flip != 0u);
          const int t0 = ch + m_step;
          uint32_t *f = pend + (c ^ 1) * nch + ((ch & ~m_wrap) | (t0 & m_wrap));
          const bool due = fb & m_from, far = decltype(edge)::value && m_rank != (int)rank && (t0 < 0 || t0 >= nch);
          if (due && !far) *f = 1u;
          if (due && far) tc::st_cluster_u32(tc::map_shared(f, (uint32_t)m_rank), 1u);
        };
        // the slab's inner chunks two at a time (a class's sites do not read each other)
        uint32_t inner = todo & m_inner, outer = todo & ~m_inner;
        while (inner) {
          const int a = warp + (__ffs(inner) - 1) * nwarps;
          inner &= inner - 1u;
          const bool two = inner != 0u;
          const int b2 = two ? warp + (__ffs(inner) - 1) * nwarps : a;
          inner &= inner - 1u;
          uint32_t wa, ta, xa[6], wb, tb, xb[6];
          load(std::false_type(), a, wa, ta, xa);
          load(std::false_type(), b2, wb, tb, xb);
          decide(std::false_type(), a, wa, ta, xa);
          if (two) decide(std::false_type(), b2, wb, tb, xb);
        }
        while (outer) {
          const int ch = warp + (__ffs(outer) - 1) * nwarps;
          outer &= outer - 1u;
          uint32_t wj, t, x[6];
          load(std::true_type(), ch, wj, t, x);
          decide(std::true_type(), ch, wj, t, x);
        }
        if (c == 1) {
          // this warp's flipped replicas to every CTA of the cluster
          anyf = __reduce_or_sync(0xffffffffu, anyf);
          if (lane < P && anyf)
            asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(
                             tc::map_shared(&s_any[pb], (uint32_t)lane)),
                         "r"(anyf)
                         : "memory");
        }
        tc::cluster_sync();  // class done in every CTA: its flips, marks and flags visible
        // (the other buffer was read after the last sweep; peers add to it after the next barrier)
        if (c == 0 && tid == 0) s_any[pb ^ 1] = 0u;
      }
      if (warp == 0) {
        const uint32_t any = s_any[pb];  // lane = replica
        const bool act = (active >> lane) & 1u;
        int tot = s_total[lane];
        if (act) s_total[lane] = ++tot;
        const uint32_t conv = active & ~any;
        uint32_t ended = conv | __ballot_sync(0xffffffffu, act && A.budget > 0 && tot >= A.budget);
        if (d + 1 >= A.max_sweeps) ended |= active;
        if (lane == 0) {
          if (rank == 0) {
            my_sweeps += __popc(active);
            my_evals += (unsigned long long)__popc(active) * (unsigned long long)n;
            my_minima += __popc(conv);
          }
          s_convround |= conv;
          s_active = active & ~ended;
        }
      }
      all_flips += my_flips;
      my_flips = 0;
      __syncthreads();
      active = s_active;
      if (!active) {
        const uint32_t cr = s_convround;
        if (cr) {
          energies();
          if (warp == 0) {
            bool better = false;
            if ((cr >> lane) & 1u) {
              s_minima[lane] += 1;
              better = s_E[lane] < s_best[lane];
              if (better) s_best[lane] = s_E[lane];
            }
            const uint32_t upd = __ballot_sync(0xffffffffu, better);
            if (lane == 0) s_upd = upd;
          }
          __syncthreads();
          const uint32_t upd = s_upd;
          if (upd)
            for (int o = tid; o < csz; o += blockDim.x) bw[o] = (bw[o] & ~upd) | (sw[o] & upd);
        }
        // stale pending flags are harmless: the next descent's first sweep
        // visits every chunk and resets them
      }
      __syncthreads();
    }
  }

  // results: best converged state per lane, else the final state of its last descent
  uint32_t has_best = 0;
  for (int r = 0; r < 32; ++r)
    if (s_minima[r] > 0) has_best |= 1u << r;
  if ((lane_valid & ~has_best) && unit % segs == segs - 1) {
    energies();
    if (tid < 32 && !((has_best >> tid) & 1u)) s_best[tid] = s_E[tid];
  }
  __syncthreads();
  bool write = true;  // this cluster writes the tile's results (the same in every CTA of it)
  if (segs > 1) {
    // this segment's words (by place), energies and minima; the last cluster of the
    // tile chooses per lane among the segments (strictly lower energy, ties keep the
    // earlier; without a converged descent the last segment)
    uint32_t *words = A.seg_words + (size_t)unit * A.nmax + lo;
    for (int o = tid; o < csz; o += blockDim.x) words[o] = (bw[o] & has_best) | (sw[o] & ~has_best);
    if (rank == 0 && tid < 32) {
      A.seg_best[(size_t)unit * 32 + tid] = s_best[tid];
      A.seg_minima[(size_t)unit * 32 + tid] = s_minima[tid];
    }
    __threadfence();
    __syncthreads();
    tc::cluster_sync();
    if (rank == 0 && tid == 0) s_upd = atomicAdd(A.queue + 4 + tile, 1) == segs - 1;
    __syncthreads();
    tc::cluster_sync();
    write = rank == 0 ? s_upd : tc::ld_cluster_u32(tc::map_shared(&s_upd, 0u));
    tc::cluster_sync();  // read before that CTA goes on
    if (write) {
      __threadfence();
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
      // the chosen words in place of the best ones
      const uint32_t *from = A.seg_words + (size_t)tile * segs * A.nmax + lo;
      for (int o = tid; o < csz; o += blockDim.x) {
        uint32_t wv = 0u;
        for (int r = 0; r < 32; ++r) wv |= __ldcg(from + (size_t)s_total[r] * A.nmax + o) & (1u << r);
        bw[o] = wv;
      }
      has_best = 0xffffffffu;
      __syncthreads();
    }
  }
  const int64_t out_base = (int64_t)A.R * I.spin_off + (int64_t)(32 * g) * n;
  if (write && ((uintptr_t)(A.spins + out_base) & 15) == 0) {
    // (n is a multiple of 32 here) 32 sites a warp step: the transpose hands lane r
    // replica r's spins, 32 bytes of its row
    for (int o = 32 * warp; o < csz; o += blockDim.x) {
      const int pl = place(lo + o + lane);
      const uint32_t mine = warp_transpose32((bw[pl] & has_best) | (sw[pl] & ~has_best), lane);
      if ((lane_valid >> lane) & 1u) store_spins32(A.spins + out_base + (int64_t)lane * n + lo + o, mine);
    }
  } else if (write) {
    for (int o = tid; o < csz; o += blockDim.x) {
      const int pl = place(lo + o);
      const uint32_t wv = (bw[pl] & has_best) | (sw[pl] & ~has_best);
      for (int r = 0; r < 32; ++r)
        if ((lane_valid >> r) & 1u) A.spins[out_base + (int64_t)r * n + lo + o] = ((wv >> r) & 1u) ? 1 : -1;
    }
  }
  if (write && rank == 0 && tid < 32 && ((lane_valid >> tid) & 1u)) {
    const int64_t o = (int64_t)b * A.R + 32 * g + tid;
    A.energy[o] = s_best[tid];
    if (A.energy_i32) A.energy_i32[o] = (int32_t)s_best[tid];
    if (A.minima) A.minima[o] = s_minima[tid];
  }
  __syncthreads();
  if (tid == 0) {
    atomicAdd(A.stats + 0, my_evals);
    atomicAdd(A.stats + 2, my_minima);
    atomicAdd(A.stats + 3, my_desc);
    atomicAdd(A.stats + 4, my_sweeps);
  }
  __shared__ unsigned long long s_fl[kCT / 32];
  all_flips = block_sum(all_flips, s_fl);
  if (tid == 0) atomicAdd(A.stats + 1, all_flips);
  my_eval = block_sum(my_eval, s_fl);
  if (tid == 0) atomicAdd(A.stats + 5, my_eval);
  tc::cluster_sync();  // no CTA leaves while peers may still read its shared memory
}

}  // namespace

// words, pending flags, best words, per-site signs (in planes while those fit)
static bool cluster_masks(int csz) { return csz <= 8192; }
// dynamic shared memory of a CTA at most (232,448 bytes less the static part)
size_t msc_cluster_smem_limit() { return 232448 - 4096; }
size_t msc_cluster_smem(int csz) {
  return (size_t)csz * 4 + (size_t)(csz / 64) * 2 * 4 + (size_t)csz * 4 + (size_t)csz * (cluster_masks(csz) ? 8 : 1);
}

template <int D, bool MASKS>
cudaError_t launch_cfg(cudaLaunchConfig_t &cfg, const TileArgs &args, int P, int *max_active) {
  auto kern = msc_cluster_kernel<D, MASKS>;
  // (the same limit for every size: the attribute is the process's, and another
  // thread's handle may launch the same kernel at a larger size)
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)msc_cluster_smem_limit());
  if (e != cudaSuccess) return e;
  if (max_active) return cudaOccupancyMaxActiveClusters(max_active, kern, &cfg);
  return cudaLaunchKernelEx(&cfg, kern, args, P);
}

// Launch (max_active == nullptr) or report how many clusters can be resident at once.
static cudaError_t msc_cluster_launch_or_query(const TileArgs &args, int n_tiles, int P, int csz_max, int D, cudaStream_t s,
                                        int *max_active) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_tiles * P);
  cfg.blockDim = dim3(kCT);
  cfg.dynamicSmemBytes = msc_cluster_smem(csz_max);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = P;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cluster_masks(csz_max))
    return D == 3 ? launch_cfg<3, true>(cfg, args, P, max_active) : launch_cfg<2, true>(cfg, args, P, max_active);
  return D == 3 ? launch_cfg<3, false>(cfg, args, P, max_active) : launch_cfg<2, false>(cfg, args, P, max_active);
}

cudaError_t launch_msc_cluster(const TileArgs &args, int units, int P, int csz_max, int D, cudaStream_t s) {
  return msc_cluster_launch_or_query(args, units, P, csz_max, D, s, nullptr);
}

int msc_cluster_max_active(int n_tiles, int P, int csz_max, int D) {
  int m = 0;
  if (msc_cluster_launch_or_query(TileArgs(), n_tiles, P, csz_max, D, nullptr, &m) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return m;
}

}  // namespace isg
