// api.cu — the C ABI (include/ising.h): instance validation and upload,
// colouring, planning, dispatch to the kernel families, status strings.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "internal.h"

namespace isg {
cudaError_t launch_plain(ising_handle *h, const ising_search_params *p, int32_t R, int8_t *spins, double *E,
                         int32_t *E32, int32_t *minima, const uint64_t *seeds_host, cudaStream_t s);
cudaError_t launch_sweep(ising_handle *h, const ising_search_params *p, int32_t R, int8_t *spins, double *E,
                         int32_t *E32, int32_t *minima, bool detached, cudaStream_t s);
cudaError_t launch_dense(ising_handle *h, const ising_search_params *p, int32_t R, int8_t *spins, double *E,
                         int32_t *E32, int32_t *minima, const uint64_t *seeds_host, cudaStream_t s);
bool dense_supported(const ising_handle *h, int32_t R);
void sweep_free(ising_handle *h);
void dense_free(ising_handle *h);
void plain_free(ising_handle *h);
}  // namespace isg

using namespace isg;

#define CUDA_OK(x)                          \
  do {                                      \
    if ((x) != cudaSuccess) return ISING_ERR_CUDA; \
  } while (0)

DevGraph ising_handle::graph() const {
  DevGraph g;
  g.inst = d_inst;
  g.row = d_row;
  g.col = d_col;
  g.J = d_J;
  g.h = d_h;
  g.inc_ptr = d_inc_ptr;
  g.inc_edge = d_inc_edge;
  g.inc_oth = d_inc_oth;
  g.hptr = d_hptr;
  g.hmem = d_hmem;
  g.hJ = d_hJ;
  g.order = d_order;
  g.cls = d_cls;
  g.meta = d_meta;
  g.Jpos = d_Jpos;
  g.latinfo = d_latinfo;
  g.Jfwd = d_Jfwd;
  g.runit = d_runit;
  g.nsp = total_spins;
  g.dtype = dtype;
  g.hyper = has_hyper ? 1 : 0;
  return g;
}

namespace {

// ---------------------------------------------------------------- validation
struct HostInst {
  int32_t n = 0;
  std::vector<int64_t> row;  // n + 1
  std::vector<int32_t> col;
  std::vector<float> Jf;
  std::vector<int8_t> Ji;
  std::vector<double> Jd;  // ISING_F64
  std::vector<float> hf;
  std::vector<int8_t> hi;
  std::vector<double> hd;
  std::vector<int64_t> hptr;
  std::vector<int32_t> hmem;
  std::vector<float> hJf;
  std::vector<int8_t> hJi;
  std::vector<double> hJd;
  std::vector<int32_t> colour;
  int32_t ncls = 0;
  int32_t max_deg = 0;
  int32_t lat_L = 0, lat_d = 0;
};

// Unit (biased exponent) for exact fixed-point energies of an FP32 instance.
// Every nonzero coupling and field is then an integer multiple M << (e - ebase)
// of 2^(ebase - 150) with a 24-bit M; with a spread of at most 38 every term
// fits below 2^62, and the high halves of up to 2^22 terms stay below 2^53 so
// the final conversion to FP64 rounds once.  Returns -1 when that does not hold
// (subnormal values, a wider spread or more terms).
int32_t energy_base_exponent(const HostInst &I, int32_t *emax_out = nullptr) {
  int emin = 256, emax = -1;
  bool sub = false;
  auto see = [&](float v) {
    uint32_t b;
    std::memcpy(&b, &v, 4);
    b &= 0x7fffffffu;
    if (!b) return;
    const int e = (int)(b >> 23);
    if (e == 0 || e == 255) sub = true;
    emin = std::min(emin, e);
    emax = std::max(emax, e);
  };
  for (float v : I.Jf) see(v);
  for (float v : I.hf) see(v);
  for (float v : I.hJf) see(v);
  if (emax_out) *emax_out = emax;
  if (sub) return -1;
  if (emax < 0) return 1;  // all zero
  const int64_t terms = (int64_t)I.col.size() / 2 + I.n + (int64_t)I.hJf.size();
  if (emax - emin > 38 || terms >= (int64_t)1 << 22) return -1;
  return emin;
}

// InstDesc::fx53: with unit u (2^(ebase - 150), or 1 for int8), A = the sum
// of |term| / u over the energy's terms (each pair once, fields, hyper-edge
// couplings) bounds every energy, every field and every partial sum of either
// (each is a signed sum of a subset of those terms); below 2^53 all of them
// are exact in FP64, and the gains, twice a field, are too.
int32_t fp64_exact(const HostInst &I, bool fl, int32_t ebase) {
  if (!fl) return 1;  // |terms| <= 127 and far fewer than 2^45 of them
  if (ebase < 0) return 0;
  auto units = [&](float v) -> unsigned __int128 {
    uint32_t b;
    std::memcpy(&b, &v, 4);
    b &= 0x7fffffffu;
    if (!b) return 0;
    const int e = (int)(b >> 23);
    return (unsigned __int128)((b & 0x7fffffu) | 0x800000u) << (e - ebase);
  };
  unsigned __int128 pairs2 = 0, rest = 0;  // pairs2: both CSR directions, twice the pair sum
  for (float v : I.Jf) pairs2 += units(v);
  for (float v : I.hf) rest += units(v);
  for (float v : I.hJf) rest += units(v);
  return pairs2 / 2 + rest < ((unsigned __int128)1 << 53) ? 1 : 0;
}

// InstDesc::fm_ent, fbits and funit (see there); inc: hyper-edges per spin.
// Returns the most entries of one spin with the same target.
int32_t fm_entries(const HostInst &I, const std::vector<std::vector<int32_t>> &inc, bool fl, InstDesc &D) {
  D.fm_ent = D.fbits = D.funit = -1;
  if (I.n > fm_max_spins()) return 1;
  const int32_t n_hyper = (int32_t)I.hptr.size() - 1;
  for (int32_t e = 0; e < n_hyper; ++e)
    if (I.hptr[e + 1] - I.hptr[e] > 3) return 1;
  int64_t most = 0;
  int32_t rounds = 1, t[32];
  for (int32_t i = 0; i < I.n; ++i) {
    int64_t ent = I.row[i + 1] - I.row[i];
    for (int32_t e : inc[i]) ent += I.hptr[e + 1] - I.hptr[e] - 1;
    most = std::max(most, ent);
    if (most > 31) return 1;
    if (inc[i].empty()) continue;  // the row's columns are distinct
    int32_t k = 0;
    for (int64_t q = I.row[i]; q < I.row[i + 1]; ++q) t[k++] = I.col[q];
    for (int32_t e : inc[i])
      for (int64_t q = I.hptr[e]; q < I.hptr[e + 1]; ++q)
        if (I.hmem[q] != i) {
          int32_t same = 1;
          for (int32_t a = 0; a < k; ++a) same += t[a] == I.hmem[q];
          rounds = std::max(rounds, same);
          t[k++] = I.hmem[q];
        }
    if (rounds > 15) return 1;
  }
  D.fm_ent = (int32_t)most;
  if (fl && D.ebase < 0) return rounds;
  // (the FP64 sums of at most 32 magnitudes round up by far less than the factor)
  double top = 0.0;
  int32_t unit = 256;
  auto see = [&](float v) -> double {
    uint32_t b;
    std::memcpy(&b, &v, 4);
    b &= 0x7fffffffu;
    if (b) unit = std::min(unit, (int32_t)(b >> 23) + __builtin_ctz((b & 0x7fffffu) | 0x800000u));
    return std::fabs((double)v);
  };
  for (int32_t i = 0; i < I.n; ++i) {
    double a = fl ? see(I.hf[i]) : std::abs((int)I.hi[i]);
    for (int64_t k = I.row[i]; k < I.row[i + 1]; ++k) a += fl ? see(I.Jf[k]) : std::abs((int)I.Ji[k]);
    for (int32_t e : inc[i]) a += fl ? see(I.hJf[e]) : std::abs((int)I.hJi[e]);
    top = std::max(top, a);
  }
  D.funit = fl ? (unit < 256 ? unit : D.ebase) : -1;
  D.fbits = 0;
  if (top > 0.0) {
    int ex = 0;
    std::frexp(top * (1.0 + 1e-12), &ex);  // top < 2^ex
    D.fbits = std::max(0, ex - (fl ? D.funit - 150 : 0));
  }
  return rounds;
}

// Recognise a periodic hypercubic lattice (side L >= 3, d = 2 or 3, spin index
// x0 + L*x1 + L^2*x2) from the CSR structure alone.
void detect_lattice(HostInst &I) {
  const int32_t n = I.n;
  for (int d = 3; d >= 2; --d) {
    const int32_t L = (int32_t)std::llround(std::pow((double)n, 1.0 / d));
    int64_t p = 1;
    for (int a = 0; a < d; ++a) p *= L;
    if (L < 3 || p != n || I.max_deg != 2 * d) continue;
    bool ok = true;
    for (int32_t i = 0; i < n && ok; ++i) {
      if (I.row[i + 1] - I.row[i] != 2 * d) { ok = false; break; }
      for (int64_t k = I.row[i]; k < I.row[i + 1] && ok; ++k) {
        const int32_t j = I.col[k];
        bool found = false;
        int64_t stride = 1;
        for (int a = 0; a < d && !found; ++a, stride *= L) {
          const int32_t c = (int32_t)((i / stride) % L);
          const int64_t up = i + (((c + 1) % L) - c) * stride, dn = i + (((c + L - 1) % L) - c) * stride;
          found = (j == up) || (j == dn);
        }
        ok = found;
      }
    }
    if (ok) {
      I.lat_L = L;
      I.lat_d = d;
      return;
    }
  }
}

double jval(const HostInst &I, int64_t k, ising_dtype dt) {
  return dt == ISING_F64 ? I.Jd[k] : (dt == ISING_F32 ? (double)I.Jf[k] : (double)I.Ji[k]);
}

ising_status load_desc(const ising_instance_desc &d, ising_dtype dtype, HostInst &I) {
  const bool fl = dtype == ISING_F32, f64 = dtype == ISING_F64;
  if (d.n < 1 || d.n > (1 << 30)) return ISING_ERR_INVALID_ARG;
  if (d.dtype != dtype) return ISING_ERR_INVALID_ARG;
  const int32_t n = d.n;
  I.n = n;
  if (d.J_dense) {
    if (!fl || d.row_ptr || d.col || d.J) return ISING_ERR_INVALID_ARG;
    if ((int64_t)n * (n - 1) > 0x7fffffffLL) return ISING_ERR_UNSUPPORTED;
    I.row.assign(n + 1, 0);
    for (int32_t i = 0; i < n; ++i) {
      if (d.J_dense[(int64_t)i * n + i] != 0.0f) return ISING_ERR_SELF_LOOP;
      for (int32_t j = 0; j < n; ++j) {
        const float w = d.J_dense[(int64_t)i * n + j];
        if (!std::isfinite(w)) return ISING_ERR_INVALID_ARG;
        if (w != d.J_dense[(int64_t)j * n + i]) return ISING_ERR_ASYMMETRIC;
        if (j == i) continue;
        I.col.push_back(j);
        I.Jf.push_back(w);
      }
      I.row[i + 1] = (int64_t)I.col.size();
    }
  } else {
    if (!d.row_ptr) return ISING_ERR_INVALID_ARG;
    if (d.row_ptr[0] != 0) return ISING_ERR_INVALID_ARG;
    for (int32_t i = 0; i < n; ++i)
      if (d.row_ptr[i + 1] < d.row_ptr[i]) return ISING_ERR_INVALID_ARG;
    const int64_t nnz = d.row_ptr[n];
    if (nnz > 0 && (!d.col || !d.J)) return ISING_ERR_INVALID_ARG;
    if (nnz > 0x7fffffffLL) return ISING_ERR_UNSUPPORTED;
    I.row.assign(d.row_ptr, d.row_ptr + n + 1);
    I.col.assign(d.col, d.col + nnz);
    if (fl) {
      I.Jf.assign((const float *)d.J, (const float *)d.J + nnz);
      for (float w : I.Jf)
        if (!std::isfinite(w)) return ISING_ERR_INVALID_ARG;
    } else if (f64) {
      I.Jd.assign((const double *)d.J, (const double *)d.J + nnz);
      for (double w : I.Jd)
        if (!std::isfinite(w)) return ISING_ERR_INVALID_ARG;
    } else {
      I.Ji.assign((const int8_t *)d.J, (const int8_t *)d.J + nnz);
    }
    // structure: range, self loops, repeats; then symmetry of structure and values
    std::vector<std::pair<int32_t, double>> sorted(nnz);
    for (int32_t i = 0; i < n; ++i) {
      for (int64_t k = I.row[i]; k < I.row[i + 1]; ++k) {
        const int32_t j = I.col[k];
        if (j < 0 || j >= n) return ISING_ERR_INVALID_ARG;
        if (j == i) return ISING_ERR_SELF_LOOP;
        sorted[k] = {j, jval(I, k, dtype)};
      }
      std::sort(sorted.begin() + I.row[i], sorted.begin() + I.row[i + 1]);
      for (int64_t k = I.row[i] + 1; k < I.row[i + 1]; ++k)
        if (sorted[k].first == sorted[k - 1].first) return ISING_ERR_INVALID_ARG;
    }
    for (int32_t i = 0; i < n; ++i)
      for (int64_t k = I.row[i]; k < I.row[i + 1]; ++k) {
        const int32_t j = sorted[k].first;
        auto lo = sorted.begin() + I.row[j], hi = sorted.begin() + I.row[j + 1];
        auto it = std::lower_bound(lo, hi, std::make_pair(i, -(double)INFINITY));
        if (it == hi || it->first != i || it->second != sorted[k].second) return ISING_ERR_ASYMMETRIC;
      }
  }
  for (int32_t i = 0; i < n; ++i) I.max_deg = std::max<int32_t>(I.max_deg, (int32_t)(I.row[i + 1] - I.row[i]));
  if (fl) {
    I.hf.assign(n, 0.0f);
    if (d.h) {
      std::memcpy(I.hf.data(), d.h, n * sizeof(float));
      for (float v : I.hf)
        if (!std::isfinite(v)) return ISING_ERR_INVALID_ARG;
    }
  } else if (f64) {
    I.hd.assign(n, 0.0);
    if (d.h) {
      std::memcpy(I.hd.data(), d.h, n * sizeof(double));
      for (double v : I.hd)
        if (!std::isfinite(v)) return ISING_ERR_INVALID_ARG;
    }
  } else {
    I.hi.assign(n, 0);
    if (d.h) std::memcpy(I.hi.data(), d.h, n);
  }
  // hyper-edges
  if (d.n_hyper < 0) return ISING_ERR_INVALID_ARG;
  I.hptr.assign(1, 0);
  if (d.n_hyper > 0) {
    if (!d.hyper_ptr || !d.hyper_members || !d.hyper_J) return ISING_ERR_INVALID_ARG;
    if (d.hyper_ptr[0] != 0) return ISING_ERR_BAD_HYPEREDGE;
    std::vector<int32_t> seen(n, -1);
    for (int32_t e = 0; e < d.n_hyper; ++e) {
      const int64_t a = d.hyper_ptr[e], b = d.hyper_ptr[e + 1];
      if (b - a < 2) return ISING_ERR_BAD_HYPEREDGE;
      for (int64_t q = a; q < b; ++q) {
        const int32_t m = d.hyper_members[q];
        if (m < 0 || m >= n || seen[m] == e) return ISING_ERR_BAD_HYPEREDGE;
        seen[m] = e;
        I.hmem.push_back(m);
      }
      I.hptr.push_back((int64_t)I.hmem.size());
    }
    if (fl) {
      I.hJf.assign((const float *)d.hyper_J, (const float *)d.hyper_J + d.n_hyper);
      for (float v : I.hJf)
        if (!std::isfinite(v)) return ISING_ERR_INVALID_ARG;
    } else if (f64) {
      I.hJd.assign((const double *)d.hyper_J, (const double *)d.hyper_J + d.n_hyper);
      for (double v : I.hJd)
        if (!std::isfinite(v)) return ISING_ERR_INVALID_ARG;
    } else {
      I.hJi.assign((const int8_t *)d.hyper_J, (const int8_t *)d.hyper_J + d.n_hyper);
    }
  }
  // colouring of the conflict graph (CSR edges + pairs inside hyper-edges)
  std::vector<std::vector<int32_t>> inc(n);
  for (int32_t e = 0; e + 1 < (int32_t)I.hptr.size(); ++e)
    for (int64_t q = I.hptr[e]; q < I.hptr[e + 1]; ++q) inc[I.hmem[q]].push_back(e);
  I.colour.assign(n, -1);
  if (d.colour) {
    for (int32_t i = 0; i < n; ++i) {
      if (d.colour[i] < 0 || d.colour[i] >= n) return ISING_ERR_BAD_COLOURING;
      I.colour[i] = d.colour[i];
    }
    for (int32_t i = 0; i < n; ++i) {
      for (int64_t k = I.row[i]; k < I.row[i + 1]; ++k)
        if (I.colour[I.col[k]] == I.colour[i]) return ISING_ERR_BAD_COLOURING;
      for (int32_t e : inc[i])
        for (int64_t q = I.hptr[e]; q < I.hptr[e + 1]; ++q)
          if (I.hmem[q] != i && I.colour[I.hmem[q]] == I.colour[i]) return ISING_ERR_BAD_COLOURING;
    }
  } else {
    // greedy in index order: smallest colour not held by an earlier conflicting spin
    std::vector<int32_t> stamp(n + 1, -1);
    for (int32_t i = 0; i < n; ++i) {
      for (int64_t k = I.row[i]; k < I.row[i + 1]; ++k) {
        const int32_t c = I.colour[I.col[k]];
        if (c >= 0) stamp[c] = i;
      }
      for (int32_t e : inc[i])
        for (int64_t q = I.hptr[e]; q < I.hptr[e + 1]; ++q) {
          const int32_t c = I.colour[I.hmem[q]];
          if (c >= 0) stamp[c] = i;
        }
      int32_t c = 0;
      while (stamp[c] == i) ++c;
      I.colour[i] = c;
    }
  }
  I.ncls = 0;
  for (int32_t c : I.colour) I.ncls = std::max(I.ncls, c + 1);
  if (I.hptr.size() == 1 && !f64) detect_lattice(I);  // (FP64 instances take no lattice path)
  return ISING_OK;
}

// Host-side fault injection for tests (ISING_FAULT): "alloc:k" makes the k-th
// device upload of ising_create fail ("alloc" = the first); "launch" makes
// ising_local_search fail as a failed launch would; "scratch:k" makes scratch
// requests of more than k bytes fail; "device_timeout" (read by the dense
// tensor-core path) makes one CTA's bounded wait run out.
bool fault_is(const char *what) {
  const char *f = std::getenv("ISING_FAULT");
  return f && std::strncmp(f, what, std::strlen(what)) == 0;
}
int g_alloc_countdown = 0;  // allocations left before the injected failure (0: none)

// Enqueued on the handle's own stream: uploads_done() before src goes and before
// any stream reads *dst.
template <class T>
cudaError_t upload(ising_handle *h, T **dst, const std::vector<T> &src) {
  if (g_alloc_countdown > 0 && --g_alloc_countdown == 0) return cudaErrorMemoryAllocation;
  cudaStream_t setup = nullptr;
  cudaError_t e = setup_stream(h, &setup);
  if (e == cudaSuccess) e = cudaMalloc((void **)dst, std::max<size_t>(1, src.size()) * sizeof(T));
  if (e != cudaSuccess || src.empty()) return e;
  return cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, setup);
}
bool uploads_done(ising_handle *h) { return !h->setup || cudaStreamSynchronize(h->setup) == cudaSuccess; }

void free_handle(ising_handle *h) {
  if (!h) return;
  int cur = 0;
  cudaGetDevice(&cur);
  cudaSetDevice(h->device);
  for (auto &t : h->ktimers) {
    cudaEventDestroy(t.a);
    cudaEventDestroy(t.b);
  }
  energy_plan_free(h);
  sweep_free(h);
  fm_free(h);
  dense_free(h);
  plain_free(h);
  void *ptrs[] = {h->d_inst, h->d_row, h->d_col, h->d_J, h->d_h, h->d_inc_ptr, h->d_inc_edge, h->d_inc_oth, h->d_hptr,
                  h->d_hmem, h->d_hJ, h->d_order, h->d_cls, h->d_Jdense, h->d_meta, h->d_Jpos, h->d_Jfwd, h->d_latinfo, h->d_runit,
                  h->d_scratch, h->d_seeds, h->d_stats, h->d_queue, h->d_tiles};
  for (void *p : ptrs)
    if (p) cudaFree(p);
  if (h->h_stats_pinned) cudaFreeHost(h->h_stats_pinned);
  if (h->setup) cudaStreamDestroy(h->setup);
  cudaSetDevice(cur);
  delete h;
}

ising_status ensure_scratch(ising_handle *h, size_t bytes) {
  if (fault_is("scratch:") && bytes > (size_t)std::atoll(std::getenv("ISING_FAULT") + 8)) return ISING_ERR_OOM;
  if (bytes <= h->scratch_bytes) return ISING_OK;
  if (h->d_scratch) cudaFree(h->d_scratch);
  h->d_scratch = nullptr;
  h->scratch_bytes = 0;
  if (cudaMalloc(&h->d_scratch, bytes) != cudaSuccess) {
    cudaGetLastError();  // (the caller may do with less)
    return ISING_ERR_OOM;
  }
  h->scratch_bytes = bytes;
  return ISING_OK;
}

ising_status validate_params(const ising_search_params *p) {
  if (!p) return ISING_ERR_INVALID_ARG;
  if (p->max_sweeps < 1 || p->restarts < 1 || p->sweep_budget < 0 || p->refresh_every < 0)
    return ISING_ERR_INVALID_ARG;
  if (p->schedule != ISING_SCHED_COLOUR && p->schedule != ISING_SCHED_SEQUENTIAL) return ISING_ERR_INVALID_ARG;
  if (p->kernel < ISING_KERNEL_AUTO || p->kernel > ISING_KERNEL_PLAIN) return ISING_ERR_INVALID_ARG;
  if (p->dense_variant != ISING_DENSE_OWN && p->dense_variant != ISING_DENSE_LIBRARY) return ISING_ERR_INVALID_ARG;
  if (p->cluster_ctas < 0 || p->cluster_ctas > 8 || (p->cluster_ctas & (p->cluster_ctas - 1)))
    return ISING_ERR_INVALID_ARG;
  return ISING_OK;
}

bool tile_fits(const ising_handle *h, int mode) {
  return tile_smem_bytes(mode, h->nmax) <= tile_smem_limit();
}

// Few large instances on lanes (no multi-spin coding): whether a launch per
// colour class over the whole GPU beats one CTA per tile and segment, by their
// times per sweep.  A tile is put at 10 ns per spin (1024 threads) and wave of
// its units; the sweep family takes its instances and descents one after another,
// 3.1 us per class launch, 0.35 ns per spin and replica group, and once for a new
// handle the capture of its graph (about 16 us a sweep over a search's 25).
// Measured (tile / sweep, us a call): degree-5 graphs, 20 replicas, 2 descents: 3,000
// spins 670 / 1380, 6,000 1045 / 1422, 9,000 1465 / 1326, 12,000 1902 / 1531, 20,000
// 3037 / 1786; Gaussian squares, 32 replicas, 4 descents: 64 x 64 348 / 551, 96 x 96
// 668 / 592, 128 x 128 1113 / 739 and with 256 replicas 1112 / 1439.
// A tile launch returns at once, and a program that drives several handles or streams
// from one thread counts on that: without counters to wait for, the sweep family runs
// such a search detached (launch_sweep) instead of following it on the host.
bool sweep_is_faster(const ising_handle *h, int32_t R, const ising_search_params *p) {
  const int32_t groups = (R + 31) / 32;
  if (groups > 32 || p->schedule == ISING_SCHED_SEQUENTIAL) return false;
  for (const InstDesc &I : h->inst)
    if (I.ncls > 120) return false;  // (a detached search's loop holds 4 sweeps of 512 launches at most)
  const double descents = p->sweep_budget > 0 ? 1 : p->restarts;
  const double waves = std::max(1.0, std::ceil((double)h->n_inst * groups * descents / h->sm_count));
  const double tile = waves * 10e-9 * h->nmax;
  double sweep = 16e-6;
  for (const InstDesc &I : h->inst) sweep += descents * ((I.ncls + 1.5) * 3.1e-6 + 0.35e-9 * I.n * groups);
  return sweep < tile;
}

// Kernel family for these arguments (ISING_KERNEL_AUTO resolved), or negative status.
// *by_time is set where the sweep family was taken though a tile could run the call.
int32_t resolve_kernel(ising_handle *h, int32_t R, const ising_search_params *p, bool *by_time = nullptr) {
  int32_t k = p->kernel;
  if (h->dtype == ISING_F64)  // FP64 couplings: the plain family only
    return (k == ISING_KERNEL_AUTO || k == ISING_KERNEL_PLAIN) ? ISING_KERNEL_PLAIN : -(int32_t)ISING_ERR_UNSUPPORTED;
  if (k == ISING_KERNEL_AUTO) {
    auto it = h->tuned.find(R);
    if (it != h->tuned.end()) return it->second;
    if (h->dense && dense_supported(h, R)) return ISING_KERNEL_DENSE_TC;
    if (h->msc_ok && tile_fits(h, 2)) return ISING_KERNEL_MSC;
    if (!tile_fits(h, h->dtype == ISING_F32 ? 1 : 0)) return ISING_KERNEL_SWEEP;
    if (!sweep_is_faster(h, R, p)) return ISING_KERNEL_TILE;
    if (by_time) *by_time = true;
    return ISING_KERNEL_SWEEP;
  }
  switch (k) {
    case ISING_KERNEL_TILE:
      return tile_fits(h, h->dtype == ISING_F32 ? 1 : 0) ? k : -(int32_t)ISING_ERR_UNSUPPORTED;
    case ISING_KERNEL_MSC:
      return (h->msc_ok && tile_fits(h, 2)) ? k : -(int32_t)ISING_ERR_UNSUPPORTED;
    case ISING_KERNEL_DENSE_TC:
      return (h->dense && dense_supported(h, R)) ? k : -(int32_t)ISING_ERR_UNSUPPORTED;
    default:
      return k;
  }
}

// Cluster split of the multi-spin-coded lattice path.  Every instance must split
// into P power-of-two slabs of at least 1024 sites (whole Philox blocks).  A
// cluster of P CTAs runs a descent about P^0.8 times as fast as one CTA (a barrier
// per class and the exchange of flags stay); tiles whose descents are independent
// run as many segments at once as clusters are resident.  Taken is the P whose
// clusters get through the call's descents soonest, in whole waves (ties: the
// smaller), so long as the tiles alone would leave most SMs idle.
const ClusterPlan &cluster_plan(ising_handle *h, int32_t R, const ising_search_params *p) {
  ClusterPlan &T = h->cluster_plan_cache;
  const int32_t parallel = p->sweep_budget > 0 ? 1 : p->restarts;
  if (T.R == R && T.parallel == parallel && T.only == p->cluster_ctas) return T;
  T = ClusterPlan();
  T.R = R;
  T.parallel = parallel;
  T.only = p->cluster_ctas;
  if (!h->msc_ok || !h->all_lattice || !h->lat_parity || p->cluster_ctas == 1) return T;
  const int64_t tiles = (int64_t)h->n_inst * ((R + 31) / 32);
  double best = 0.0;
  for (int P : {8, 4, 2}) {
    if (p->cluster_ctas > 1 && p->cluster_ctas != P) continue;  // restricted to one size
    if (tiles * P > 2 * (int64_t)h->sm_count) continue;
    bool ok = true;
    int d = -1;
    for (const auto &I : h->inst) {
      const int csz = I.n / P;
      if (I.n % P || csz < 1024 || (csz & (csz - 1)) || csz % 128) ok = false;
      if (msc_cluster_smem(csz) > msc_cluster_smem_limit()) ok = false;
      if (d >= 0 && I.lat_d != d) ok = false;
      d = I.lat_d;
    }
    if (!ok) continue;
    const int64_t active = std::max(1, msc_cluster_max_active((int)std::min<int64_t>(tiles * parallel, 4096), P, h->nmax / P, d));
    // Clusters of 8 only when every CTA gets an SM of its own and all clusters of
    // one segment are resident at once.
    if (P == 8 && (tiles * P > (int64_t)h->sm_count || active < tiles)) continue;
    const int64_t segs = std::max<int64_t>(1, std::min<int64_t>(parallel, active / tiles));
    const double waves = std::max(1.0, std::ceil((double)(tiles * segs) / (double)active));
    const double time = waves * std::ceil((double)parallel / (double)segs) / std::pow((double)P, 0.8);
    if (T.P == 0 || time <= best) {
      best = time;
      T.P = P;
      T.segs = (int32_t)segs;
    }
  }
  return T;
}

// CTA size and segments of the tile kernels for these arguments, null when no
// CTA fits.  A descent's time in one CTA goes like a constant (barriers, round
// trips) plus the steps the largest class takes: a warp's spins in the lane modes
// (constant 6 steps; 10, or 15 with 1024 threads, in the FP32 visits, eight spins a
// warp), a thread per spin in the multi-spin-coded ones (30).  The tiles' descents
// (without a budget each descent is a unit of its own) run in waves over the CTA
// slots; uneven instances fill the waves, a last wave of equal ones does not.
// Measured, us a call at 256 / 512 / 1024 threads (FP32): cell grids of up to 2,048
// spins, 64 tiles 603 / 370 / 338, 512 tiles 816 / 501 / 742, 1,024 tiles 971 / 950 /
// 1395, 4,096 tiles 3197 / 3555 / 5318, of 128 spins each, 700 tiles 210 / 319 / 577;
// 6,000 spins of degree 5, 20 replicas, 2 descents 2579 / 1340 / 979; 45 x 45, 10
// descents of 64 replicas 323 / 230 / 218, of 1,024 447 / 561 / 553.  +/-J: 31^3, 1,024
// replicas, 10 descents 2499 / 1572 / 1279; 16 x 16, 64 replicas, 10 descents 52 / 42 /
// 44 (125 in one segment).
// The index order, a spin at a time in any CTA, runs at 256 threads only: multi-spin
// coded, its barrier per spin takes longer the more warps wait at it (64 x 64, 64
// replicas 6.4 ms; in a kernel for both orders 9.1 / 9.3 / 10.1).
const TilePlan *tile_plan(ising_handle *h, int mode, int32_t R, const ising_search_params *p) {
  TilePlan &T = h->tile_plan_cache;
  const int32_t parallel = p->sweep_budget > 0 ? 1 : p->restarts;
  const bool sequential = p->schedule == ISING_SCHED_SEQUENTIAL;
  if (T.mode == mode && T.R == R && T.parallel == parallel && T.sequential == sequential) return T.slots > 0 ? &T : nullptr;
  T = TilePlan();
  T.mode = mode;
  T.sequential = sequential;
  T.R = R;
  T.parallel = parallel;
  const int64_t tiles = (int64_t)h->n_inst * ((R + 31) / 32);
  double weight = 0.0;  // of all units, in units of the largest instance
  int32_t ncls = 1, nmin = h->nmax;
  for (const InstDesc &I : h->inst) {
    weight += (double)I.n / h->nmax;
    nmin = std::min(nmin, I.n);
    if (I.n == h->nmax) ncls = std::max(ncls, I.ncls);
  }
  weight *= (double)((R + 31) / 32) * parallel;
  double best = 0.0;
  for (int threads : {256, 512, 1024}) {
    if (sequential && threads != 256) break;
    // FP32 lanes: fields in shared memory for every instance that fits, within a
    // budget that lets four CTAs share an SM (one CTA of 1024 threads with four
    // times as much, and so less L1, was 5 % slower)
    int fsm_cap = mode == 1 ? tile_fsm_cap(h->nmax, (size_t)48 * 1024) : 0;
    if (nmin > fsm_cap) fsm_cap = 0;
    size_t smem = tile_smem_bytes(mode, h->nmax);
    if (fsm_cap > 0) smem = (smem + 15) / 16 * 16 + (size_t)fsm_cap * 128;
    const int64_t slots = (int64_t)tile_max_ctas_per_sm(mode, threads, smem, sequential) * h->sm_count;
    if (slots < 1) continue;
    const double per_step = mode >= 2 ? 2.0 * threads : (double)ncls * threads / 32;
    const double fixed = mode >= 2 ? 30.0 : (mode == 0 ? 6.0 : (threads == 1024 ? 15.0 : 10.0));
    const double unit = fixed + std::ceil(h->nmax / per_step);
    double waves = weight / (double)slots;
    if (mode != 1) {
      waves = std::max(1.0, waves);
      if (nmin == h->nmax && waves < 2.0) waves = std::ceil(waves);
    } else if (waves < 1.0) {
      waves = 0.6 + 0.4 * waves;  // (SMs with fewer CTAs than they hold run them faster)
    } else if (nmin == h->nmax && waves < 2.0) {
      waves = 0.5 * (waves + std::ceil(waves));
    }
    if (T.slots == 0 || unit * waves <= best) {  // (ties: the larger CTA)
      best = unit * waves;
      T.threads = threads;
      T.slots = slots;
      T.fsm_cap = fsm_cap;
      T.smem = smem;
    }
  }
  if (T.slots == 0) return nullptr;
  T.segs = (int32_t)std::max<int64_t>(1, std::min<int64_t>(parallel, T.slots / tiles));
  return &T;
}

ising_status run_tile(ising_handle *h, int mode, int32_t R, const ising_search_params *p, int8_t *spins,
                      double *E, int32_t *E32, int32_t *minima, cudaStream_t s) {
  // tiles: (instance, 32-replica group), largest instances first
  const int32_t groups = (R + 31) / 32;
  if (h->tiles_R != R) {
    std::vector<int32_t> ord(h->n_inst);
    std::iota(ord.begin(), ord.end(), 0);
    std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return h->inst[a].n > h->inst[b].n; });
    std::vector<int2> tiles;
    tiles.reserve((size_t)h->n_inst * groups);
    for (int32_t b : ord)
      for (int32_t g = 0; g < groups; ++g) tiles.push_back(make_int2(b, g));
    if (h->d_tiles) cudaFree(h->d_tiles);
    h->d_tiles = nullptr;
    h->tiles_R = -1;
    const cudaError_t e = upload(h, &h->d_tiles, tiles);
    if (!uploads_done(h) || e != cudaSuccess) return ISING_ERR_CUDA;
    h->n_tiles = (int32_t)tiles.size();
    h->tiles_R = R;
  }
  auto up256 = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
  // counters of the segments ended, per tile, behind the work queue's
  auto ensure_counters = [&](int32_t counters) -> ising_status {
    if (counters <= h->queue_tiles) return ISING_OK;
    int32_t *q = nullptr;
    if (cudaMalloc(&q, sizeof(int32_t) * (4 + (size_t)counters)) != cudaSuccess) {
      cudaGetLastError();
      return ISING_ERR_OOM;
    }
    cudaFree(h->d_queue);
    h->d_queue = q;
    h->queue_tiles = counters;
    return ISING_OK;
  };
  TileArgs a = {};
  a.g = h->graph();
  a.tiles = h->d_tiles;
  a.n_tiles = h->n_tiles;
  a.R = R;
  a.max_sweeps = p->max_sweeps;
  a.restarts = p->restarts;
  a.budget = p->sweep_budget;
  a.refresh = p->refresh_every;
  a.sequential = p->schedule == ISING_SCHED_SEQUENTIAL ? 1 : 0;
  a.seeds = h->d_seeds;
  a.nmax = h->nmax;
  a.spins = spins;
  a.energy = E;
  a.energy_i32 = E32;
  a.minima = minima;
  a.stats = h->d_stats;
  if (mode == 3) {
    const ClusterPlan &C = cluster_plan(h, R, p);
    if (C.P > 0) {
      const size_t seg_bytes = up256((size_t)h->n_tiles * C.segs * h->nmax * sizeof(uint32_t));
      const size_t lane_bytes = up256((size_t)h->n_tiles * C.segs * 32 * sizeof(double));
      // without room for the segments' results the tiles run whole, which needs none
      const int segs = C.segs > 1 && ensure_scratch(h, seg_bytes + 2 * lane_bytes + 256) == ISING_OK &&
                               ensure_counters(h->n_tiles) == ISING_OK
                           ? C.segs
                           : 1;
      const int units = h->n_tiles * segs;
      a.queue = h->d_queue;
      a.segs = segs;
      a.seg_words = (uint32_t *)h->d_scratch;
      a.seg_best = (double *)((char *)h->d_scratch + seg_bytes);
      a.seg_minima = (int32_t *)((char *)h->d_scratch + seg_bytes + lane_bytes);
      if (segs > 1) CUDA_OK(cudaMemsetAsync(h->d_queue, 0, sizeof(int32_t) * (4 + (size_t)h->n_tiles), s));
      kt_begin(h, "msc_cluster_kernel", s);
      CUDA_OK(launch_msc_cluster(a, units, C.P, h->nmax / C.P, h->inst[0].lat_d, s));
      kt_end(h, s);
      h->launches += 1;
      return ISING_OK;
    }
  }
  const TilePlan *plan = tile_plan(h, mode, R, p);
  if (!plan) return ISING_ERR_UNSUPPORTED;
  const int threads = plan->threads, fsm_cap = plan->fsm_cap;
  const size_t smem = plan->smem;
  int segs = plan->segs, grid;
  size_t f_bytes, bw_bytes, seg_bytes, lane_bytes;
  for (;; segs = 1) {  // without room for the segments' results and CTAs the tiles run whole
    const int64_t work = (int64_t)h->n_tiles * segs;
    grid = (int)std::min<int64_t>(work, plan->slots);
    f_bytes = mode == 1 ? up256((size_t)grid * h->nmax * 32 * sizeof(float)) : 0;
    bw_bytes = up256((size_t)grid * h->nmax * sizeof(uint32_t));
    seg_bytes = segs > 1 ? up256((size_t)work * h->nmax * sizeof(uint32_t)) : 0;
    lane_bytes = segs > 1 ? up256((size_t)work * 32 * sizeof(double)) : 0;
    ising_status st = ensure_scratch(h, f_bytes + bw_bytes + seg_bytes + 2 * lane_bytes + 256);
    if (st == ISING_OK && segs > 1) st = ensure_counters(h->n_tiles);
    if (st == ISING_OK) break;
    if (segs == 1) return st;
  }
  const int32_t counters = segs > 1 ? h->n_tiles : 0;
  a.queue = h->d_queue;
  a.F = mode == 1 ? (float *)h->d_scratch : nullptr;
  a.fsm_cap = fsm_cap;
  char *scratch = (char *)h->d_scratch + f_bytes;
  a.bw = (uint32_t *)scratch;
  a.segs = segs;
  a.seg_words = (uint32_t *)(scratch + bw_bytes);
  a.seg_best = (double *)(scratch + bw_bytes + seg_bytes);
  a.seg_minima = (int32_t *)(scratch + bw_bytes + seg_bytes + lane_bytes);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  CUDA_OK(cudaStreamIsCapturing(s, &cap));
  if (cap != cudaStreamCaptureStatusNone) return ISING_ERR_CUDA;  // (scratch and work queue are the handle's)
  CUDA_OK(cudaMemsetAsync(h->d_queue, 0, sizeof(int32_t) * (4 + (size_t)counters), s));
  kt_begin(h, "tile_kernel", s);
  CUDA_OK(launch_tile(a, mode, threads, segs > 1, grid, smem, s));
  kt_end(h, s);
  h->launches += 1;
  return ISING_OK;
}

// ---------------------------------------------------------------- tuning cache
// Decisions are keyed by the GPU name and an instance class (dtype, instance
// count, largest instance, lattice / multi-spin eligibility, replicas,
// schedule).  With ISING_TUNE_CACHE=<file> they persist across processes as
// lines of a small JSON object: {"key": family, ...}.
std::string tune_key(const ising_handle *h, int32_t R, const ising_search_params *p) {
  cudaDeviceProp prop;
  cudaGetDeviceProperties(&prop, h->device);
  char buf[512];
  snprintf(buf, sizeof buf, "%s|dt%d|b%d|n%d|lat%d|msc%d|dense%d|R%d|sched%d|refresh%d", prop.name, h->dtype,
           h->n_inst, h->nmax, h->all_lattice ? 1 : 0, h->msc_ok ? 1 : 0, h->dense ? 1 : 0, R, (int)p->schedule,
           p->refresh_every);
  return buf;
}

std::map<std::string, int32_t> read_tune_file(const char *path) {
  std::map<std::string, int32_t> m;
  FILE *f = path ? fopen(path, "r") : nullptr;
  if (!f) return m;
  char line[1024];
  while (fgets(line, sizeof line, f)) {
    char *a = strchr(line, '"');
    if (!a) continue;
    char *b = strchr(a + 1, '"');
    if (!b) continue;
    char *c = strchr(b, ':');
    if (!c) continue;
    m[std::string(a + 1, b)] = (int32_t)strtol(c + 1, nullptr, 10);
  }
  fclose(f);
  return m;
}

int32_t tune_cache_lookup(const std::string &key) {
  const char *path = getenv("ISING_TUNE_CACHE");
  if (!path) return -1;
  auto m = read_tune_file(path);
  auto it = m.find(key);
  return it == m.end() ? -1 : it->second;
}

void tune_cache_store(const std::string &key, int32_t fam) {
  const char *path = getenv("ISING_TUNE_CACHE");
  if (!path) return;
  auto m = read_tune_file(path);
  m[key] = fam;
  FILE *f = fopen(path, "w");
  if (!f) return;
  fprintf(f, "{\n");
  size_t i = 0;
  for (auto &kv : m) fprintf(f, "  \"%s\": %d%s\n", kv.first.c_str(), kv.second, ++i < m.size() ? "," : "");
  fprintf(f, "}\n");
  fclose(f);
}

}  // namespace

namespace isg {

// An NVTX range for the duration of a C-ABI call (visible to profilers that
// record NVTX; a no-op otherwise).
struct NvtxRange {
  explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange &) = delete;
  NvtxRange &operator=(const NvtxRange &) = delete;
};

cudaError_t setup_stream(ising_handle *h, cudaStream_t *s) {
  cudaError_t e = cudaSuccess;
  if (!h->setup) e = cudaStreamCreateWithFlags(&h->setup, cudaStreamNonBlocking);
  *s = h->setup;
  return e;
}

void kt_begin(ising_handle *h, const char *name, cudaStream_t s) {
  if (!h->timing) return;
  if (h->kt_used == h->ktimers.size()) {
    ising_handle::KTimer t{name, nullptr, nullptr};
    if (cudaEventCreate(&t.a) != cudaSuccess) return;
    if (cudaEventCreate(&t.b) != cudaSuccess) {
      cudaEventDestroy(t.a);
      return;
    }
    h->ktimers.push_back(t);
  }
  h->ktimers[h->kt_used].name = name;
  cudaEventRecord(h->ktimers[h->kt_used].a, s);
}

void kt_end(ising_handle *h, cudaStream_t s) {
  if (!h->timing || h->kt_used == h->ktimers.size()) return;  // (begin could not create its events)
  cudaEventRecord(h->ktimers[h->kt_used].b, s);
  ++h->kt_used;
}

}  // namespace isg

extern "C" {

ising_status ising_create(const ising_instance_desc *descs, int32_t n_instances, ising_handle **out) {
  const NvtxRange nvtx_range("ising_create");
  g_alloc_countdown = 0;
  if (fault_is("alloc")) {
    const char *f = std::getenv("ISING_FAULT");
    g_alloc_countdown = f[5] == ':' ? std::max(1, std::atoi(f + 6)) : 1;
  }
  if (!out) return ISING_ERR_INVALID_ARG;
  *out = nullptr;
  if (!descs || n_instances < 1) return ISING_ERR_INVALID_ARG;
  const ising_dtype dtype = descs[0].dtype;
  if (dtype != ISING_I8 && dtype != ISING_F32 && dtype != ISING_F64) return ISING_ERR_INVALID_ARG;
  const bool fl = dtype == ISING_F32, f64 = dtype == ISING_F64;
  std::vector<HostInst> hin(n_instances);
  bool dense = true, msc = dtype == ISING_I8, hyper = false;
  int64_t absb = 0;
  for (int32_t b = 0; b < n_instances; ++b) {
    ising_status st = load_desc(descs[b], dtype, hin[b]);
    if (st != ISING_OK) return st;
    const HostInst &I = hin[b];
    dense = dense && descs[b].J_dense != nullptr;
    hyper = hyper || I.hptr.size() > 1;
    if (dtype == ISING_I8) {
      for (int8_t w : I.Ji) {
        if (w != 1 && w != -1) msc = false;
        absb += std::abs((int)w);
      }
      absb /= 1;  // each pair appears twice; bound kept conservative
      for (int8_t v : I.hi) {
        if (v < -1 || v > 1) msc = false;
        absb += std::abs((int)v);
      }
      for (int8_t v : I.hJi) absb += std::abs((int)v);
      if (I.hptr.size() > 1 || I.max_deg > 15) msc = false;
    }
  }
  ising_handle *h = new ising_handle();
  cudaGetDevice(&h->device);
  cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device);
  h->n_inst = n_instances;
  h->dtype = dtype;
  h->dense = dense && !hyper;  // hyper-edges on a dense instance: the CSR paths take it
  h->msc_ok = msc;
  h->has_hyper = hyper;
  h->abs_energy_bound = absb;

  // concatenate
  std::vector<InstDesc> inst(n_instances);
  std::vector<uint32_t> row;
  std::vector<int32_t> col, order, cls;
  std::vector<int8_t> Ji, hi, hJi;
  std::vector<float> Jf, hf, hJf;
  std::vector<double> Jd, hd, hJd;
  std::vector<uint32_t> inc_ptr, hptr;
  std::vector<int32_t> inc_edge, hmem;
  std::vector<int2> inc_oth;  // per incidence: the other two members of a 3-member edge
  std::vector<std::pair<int32_t, std::vector<int32_t>>> lat_sites;
  int64_t spin_off = 0, nnz_off = 0, edge_off = 0, mem_off = 0, cls_off = 0;
  for (int32_t b = 0; b < n_instances; ++b) {
    const HostInst &I = hin[b];
    InstDesc &D = inst[b];
    D.n = I.n;
    D.ncls = I.ncls;
    D.spin_off = spin_off;
    D.cls_off = cls_off;
    D.hyper_off = edge_off;
    D.n_hyper = (int32_t)I.hptr.size() - 1;
    D.max_deg = I.max_deg;
    D.lat_L = I.lat_L;
    D.lat_d = I.lat_d;
    int32_t emax = -1;
    D.ebase = fl ? energy_base_exponent(I, &emax) : -1;
    D.fx53 = f64 ? 0 : fp64_exact(I, fl, D.ebase);  // FP64 instances: the FP64 forms only
    D.ebits = f64 ? -1 : (!fl ? 7 : (D.ebase >= 0 ? 24 + std::max(0, emax - D.ebase) : -1));
    h->any_lattice = h->any_lattice || I.lat_d > 0;
    h->all_lattice = (b == 0 ? true : h->all_lattice) && I.lat_d > 0;
    h->nmax = std::max(h->nmax, I.n);
    for (int32_t i = 0; i < I.n; ++i) row.push_back((uint32_t)(nnz_off + I.row[i]));
    col.insert(col.end(), I.col.begin(), I.col.end());
    if (fl) {
      Jf.insert(Jf.end(), I.Jf.begin(), I.Jf.end());
      hf.insert(hf.end(), I.hf.begin(), I.hf.end());
      hJf.insert(hJf.end(), I.hJf.begin(), I.hJf.end());
    } else if (f64) {
      Jd.insert(Jd.end(), I.Jd.begin(), I.Jd.end());
      hd.insert(hd.end(), I.hd.begin(), I.hd.end());
      hJd.insert(hJd.end(), I.hJd.begin(), I.hJd.end());
    } else {
      Ji.insert(Ji.end(), I.Ji.begin(), I.Ji.end());
      hi.insert(hi.end(), I.hi.begin(), I.hi.end());
      hJi.insert(hJi.end(), I.hJi.begin(), I.hJi.end());
    }
    // incidence of hyper-edges per spin, ascending edge id
    std::vector<std::vector<int32_t>> inc(I.n);
    for (int32_t e = 0; e < D.n_hyper; ++e)
      for (int64_t q = I.hptr[e]; q < I.hptr[e + 1]; ++q) inc[I.hmem[q]].push_back(e);
    for (int32_t i = 0; i < I.n; ++i) {
      inc_ptr.push_back((uint32_t)inc_edge.size());
      for (int32_t e : inc[i]) {
        inc_edge.push_back((int32_t)(edge_off + e));
        int2 o = make_int2(-1, -1);
        if (I.hptr[e + 1] - I.hptr[e] == 3) {
          int32_t m[2], k = 0;
          for (int64_t q = I.hptr[e]; q < I.hptr[e + 1]; ++q)
            if (I.hmem[q] != i && k < 2) m[k++] = I.hmem[q];
          if (k == 2) o = make_int2(m[0], m[1]);
        }
        inc_oth.push_back(o);
      }
    }
    D.has_h = 0;
    for (float v : I.hf) D.has_h |= v != 0.0f;
    for (int8_t v : I.hi) D.has_h |= v != 0;
    for (double v : I.hd) D.has_h |= v != 0.0;
    D.fm_ent = D.fbits = D.funit = -1;
    if (!f64) h->fm_rounds = std::max(h->fm_rounds, fm_entries(I, inc, fl, D));
    for (int32_t e = 0; e < D.n_hyper; ++e) hptr.push_back((uint32_t)(mem_off + I.hptr[e]));
    hmem.insert(hmem.end(), I.hmem.begin(), I.hmem.end());
    // colour classes: spins sorted by (colour, index)
    std::vector<int32_t> cnt(I.ncls + 1, 0);
    for (int32_t c : I.colour) cnt[c + 1]++;
    for (int32_t c = 0; c < I.ncls; ++c) cnt[c + 1] += cnt[c];
    cls.insert(cls.end(), cnt.begin(), cnt.end());
    std::vector<int32_t> fill(cnt.begin(), cnt.end() - 1), ord(I.n);
    for (int32_t i = 0; i < I.n; ++i) ord[fill[I.colour[i]]++] = i;
    order.insert(order.end(), ord.begin(), ord.end());
    if (I.lat_d > 0) lat_sites.push_back({b, ord});
    spin_off += I.n;
    nnz_off += I.row[I.n];
    edge_off += D.n_hyper;
    mem_off += (int64_t)I.hmem.size();
    cls_off += I.ncls + 1;
  }
  if (nnz_off >= 0xffffffffLL || mem_off >= 0xffffffffLL || (int64_t)inc_edge.size() >= 0xffffffffLL) {
    delete h;
    return ISING_ERR_UNSUPPORTED;
  }
  row.push_back((uint32_t)nnz_off);
  inc_ptr.push_back((uint32_t)inc_edge.size());
  hptr.push_back((uint32_t)mem_off);
  std::vector<int16_t> runit;
  if (fl) {
    // per-spin refresh unit: the same test as the kernels' xr_exact, once here
    runit.assign(spin_off, 0);
    for (int64_t gi = 0; gi < spin_off; ++gi) {
      int emin = 256, emax = -1, k = 0;
      auto see = [&](float v) {
        uint32_t bits;
        std::memcpy(&bits, &v, 4);
        bits &= 0x7fffffffu;
        ++k;
        if (bits) {
          const int e = (int)(bits >> 23);
          emin = std::min(emin, e);
          emax = std::max(emax, e);
        }
      };
      see(hf.empty() ? 0.0f : hf[gi]);
      for (uint32_t kk = row[gi]; kk < row[gi + 1]; ++kk) see(Jf[kk]);
      for (uint32_t q = inc_ptr[gi]; q < inc_ptr[gi + 1]; ++q) see(hJf[inc_edge[q]]);
      int lg = 0;
      while (lg < 31 && (1u << lg) <= (uint32_t)k) ++lg;  // 2^lg > k
      const bool ex = emax < 0 || (emin >= 24 && emax <= 200 && (emax - emin) + 24 + lg <= 53);
      runit[gi] = (int16_t)(emax < 0 ? 24 : (ex ? emin : -1));
    }
    // InstDesc::fx53 = 2: fields exact in FP64 spin by spin (every spin has a
    // refresh unit), though not the energy as one integer sum
    for (int32_t b = 0; b < n_instances; ++b) {
      InstDesc &D = inst[b];
      if (D.fx53) continue;
      bool all = true;
      for (int64_t gi = D.spin_off; gi < D.spin_off + D.n && all; ++gi) all = runit[gi] >= 0;
      if (all) D.fx53 = 2;
    }
  }
  h->inst = inst;
  h->h_cls = cls;
  h->total_spins = spin_off;
  h->total_nnz = nnz_off;
  h->total_edges = edge_off;
  h->total_members = mem_off;

  bool ok = upload(h, &h->d_inst, inst) == cudaSuccess && upload(h, &h->d_row, row) == cudaSuccess &&
            upload(h, &h->d_col, col) == cudaSuccess && upload(h, &h->d_inc_ptr, inc_ptr) == cudaSuccess &&
            upload(h, &h->d_inc_edge, inc_edge) == cudaSuccess && upload(h, &h->d_inc_oth, inc_oth) == cudaSuccess &&
            upload(h, &h->d_hptr, hptr) == cudaSuccess &&
            upload(h, &h->d_hmem, hmem) == cudaSuccess && upload(h, &h->d_order, order) == cudaSuccess &&
            upload(h, &h->d_cls, cls) == cudaSuccess;
  if (ok) {
    if (fl) {
      ok = upload(h, (float **)&h->d_J, Jf) == cudaSuccess && upload(h, (float **)&h->d_h, hf) == cudaSuccess &&
           upload(h, (float **)&h->d_hJ, hJf) == cudaSuccess;
      ok = ok && upload(h, &h->d_runit, runit) == cudaSuccess;
    } else if (f64) {
      ok = upload(h, (double **)&h->d_J, Jd) == cudaSuccess && upload(h, (double **)&h->d_h, hd) == cudaSuccess &&
           upload(h, (double **)&h->d_hJ, hJd) == cudaSuccess;
    } else {
      ok = upload(h, (int8_t **)&h->d_J, Ji) == cudaSuccess && upload(h, (int8_t **)&h->d_h, hi) == cudaSuccess &&
           upload(h, (int8_t **)&h->d_hJ, hJi) == cudaSuccess;
    }
  }
  if (ok && h->any_lattice) {
    // lattice metadata in colour order (see DevGraph::meta)
    const int64_t nsp = spin_off;
    std::vector<uint32_t> meta(nsp, 0);
    std::vector<uint16_t> latinfo(nsp, 0);
    std::vector<float> Jpf(fl ? 6 * nsp : 0, 0.0f);
    std::vector<int8_t> Jpi(fl ? 0 : 6 * nsp, 0);
    std::vector<float> Jff(fl ? 3 * nsp : 0, 0.0f);
    std::vector<int8_t> Jfi(fl ? 0 : 3 * nsp, 0);
    h->lat_parity = h->all_lattice;
    for (auto &ls : lat_sites) {
      const HostInst &I = hin[ls.first];
      const InstDesc &D = inst[ls.first];
      if (I.lat_d == 0) continue;
      const int32_t L = I.lat_L;
      if (D.ncls != 2) h->lat_parity = false;
      for (int32_t v = 0; v < I.n; ++v) {
        const int32_t j = ls.second[v];
        if (h->lat_parity) {
          int par = 0;
          for (int32_t a = 0, r = j; a < I.lat_d; ++a, r /= L) par += r % L;
          const int c = v < h->h_cls[D.cls_off + 1] - h->h_cls[D.cls_off] ? 0 : 1;
          if ((par & 1) != c) h->lat_parity = false;
        }
        uint32_t m = 0;
        int kk = 0;
        for (int64_t k = I.row[j]; k < I.row[j + 1]; ++k, ++kk) {
          const int32_t t = I.col[k];
          int64_t stride = 1;
          int dir = -1, wrap = 0;
          for (int a = 0; a < I.lat_d; ++a, stride *= L) {
            const int32_t c = (int32_t)((j / stride) % L);
            if (t == j + (((c + 1) % L) - c) * stride) { dir = 2 * a; wrap = (c == L - 1); break; }
            if (t == j + (((c + L - 1) % L) - c) * stride) { dir = 2 * a + 1; wrap = (c == 0); break; }
          }
          m |= (uint32_t)wrap << kk;
          m |= (uint32_t)dir << (8 + 3 * kk);
          const double w = fl ? (double)I.Jf[k] : (double)I.Ji[k];
          if (w < 0) m |= 1u << (26 + kk);
          latinfo[D.spin_off + v] |= (uint16_t)((wrap << dir) | ((w < 0 ? 1 : 0) << (8 + dir)));
          if (fl) Jpf[(int64_t)kk * nsp + D.spin_off + v] = I.Jf[k];
          else Jpi[(int64_t)kk * nsp + D.spin_off + v] = I.Ji[k];
          if (!(dir & 1)) {  // the bond to the +a neighbour, by site
            if (fl) Jff[(int64_t)(dir >> 1) * nsp + D.spin_off + j] = I.Jf[k];
            else Jfi[(int64_t)(dir >> 1) * nsp + D.spin_off + j] = I.Ji[k];
          }
        }
        meta[D.spin_off + v] = m;
      }
    }
    ok = upload(h, &h->d_meta, meta) == cudaSuccess && upload(h, &h->d_latinfo, latinfo) == cudaSuccess &&
         (fl ? upload(h, (float **)&h->d_Jpos, Jpf) : upload(h, (int8_t **)&h->d_Jpos, Jpi)) == cudaSuccess &&
         (fl ? upload(h, (float **)&h->d_Jfwd, Jff) : upload(h, (int8_t **)&h->d_Jfwd, Jfi)) == cudaSuccess;
    ok = uploads_done(h) && ok;
  }
  if (ok && dense) {
    std::vector<float> Jd;
    for (int32_t b = 0; b < n_instances; ++b)
      Jd.insert(Jd.end(), descs[b].J_dense, descs[b].J_dense + (int64_t)descs[b].n * descs[b].n);
    ok = upload(h, &h->d_Jdense, Jd) == cudaSuccess;
    ok = uploads_done(h) && ok;
  }
  ok = ok && cudaMalloc(&h->d_seeds, sizeof(uint64_t) * n_instances) == cudaSuccess &&
       cudaMalloc(&h->d_stats, sizeof(unsigned long long) * 8) == cudaSuccess &&
       cudaMalloc(&h->d_queue, sizeof(int32_t) * 4) == cudaSuccess &&
       cudaMallocHost(&h->h_stats_pinned, sizeof(unsigned long long) * 8) == cudaSuccess;
  ok = uploads_done(h) && ok;
  if (!ok) {
    cudaGetLastError();
    free_handle(h);
    return ISING_ERR_OOM;
  }
  *out = h;
  return ISING_OK;
}

ising_status ising_energy(ising_handle *h, const int8_t *spins_dev, int32_t replicas, double *energy_dev,
                          int32_t *energy_i32_dev, cudaStream_t stream) {
  const NvtxRange nvtx_range("ising_energy");
  if (!h || !spins_dev || !energy_dev || replicas < 1) return ISING_ERR_INVALID_ARG;
  if (h->latched != ISING_OK) {
    ising_status l = h->latched;
    h->latched = ISING_OK;
    return l;
  }
  if (energy_i32_dev && (h->dtype != ISING_I8 || h->abs_energy_bound > 0x7fffffffLL))
    return ISING_ERR_UNSUPPORTED;
  int cur = 0;
  cudaGetDevice(&cur);
  if (cur != h->device) cudaSetDevice(h->device);
  cudaError_t e = launch_energy(h, spins_dev, replicas, energy_dev, energy_i32_dev, stream);
  if (cur != h->device) cudaSetDevice(cur);
  return e == cudaSuccess ? ISING_OK : ISING_ERR_CUDA;
}

int32_t ising_plan_kernel(ising_handle *h, int32_t replicas, const ising_search_params *p) {
  if (!h || replicas < 1) return -(int32_t)ISING_ERR_INVALID_ARG;
  ising_status st = validate_params(p);
  if (st != ISING_OK) return -(int32_t)st;
  return resolve_kernel(h, replicas, p);
}

ising_status ising_local_search(ising_handle *h, const uint64_t *seeds, int32_t replicas,
                                const ising_search_params *p, int8_t *spins_dev, double *energy_dev,
                                int32_t *energy_i32_dev, int32_t *minima_dev, ising_stats *stats,
                                cudaStream_t stream) {
  const NvtxRange nvtx_range("ising_local_search");
  if (!h || !seeds || replicas < 1 || !spins_dev || !energy_dev) return ISING_ERR_INVALID_ARG;
  ising_status st = validate_params(p);
  if (st != ISING_OK) return st;
  if (h->latched != ISING_OK) {
    ising_status l = h->latched;
    h->latched = ISING_OK;
    return l;
  }
  if (energy_i32_dev && (h->dtype != ISING_I8 || h->abs_energy_bound > 0x7fffffffLL))
    return ISING_ERR_UNSUPPORTED;
  if ((int64_t)replicas * h->total_spins > (int64_t)1 << 40) return ISING_ERR_UNSUPPORTED;
  bool by_time = false;
  const int32_t kernel = resolve_kernel(h, replicas, p, &by_time);
  if (kernel < 0) return (ising_status)(-kernel);
  int cur = 0;
  cudaGetDevice(&cur);
  if (cur != h->device) cudaSetDevice(h->device);
  st = ISING_OK;
  h->launches = 0;
  do {
    if (cudaMemcpyAsync(h->d_seeds, seeds, sizeof(uint64_t) * h->n_inst, cudaMemcpyHostToDevice, stream) !=
            cudaSuccess ||
        cudaMemsetAsync(h->d_stats, 0, sizeof(unsigned long long) * 8, stream) != cudaSuccess) {
      st = ISING_ERR_CUDA;
      break;
    }
    if (fault_is("launch")) {  // injected: as if the family's launch had failed
      st = ISING_ERR_CUDA;
      break;
    }
    switch (kernel) {
      case ISING_KERNEL_TILE:
        st = run_tile(h, h->dtype == ISING_F32 ? 1 : 0, replicas, p, spins_dev, energy_dev, energy_i32_dev,
                      minima_dev, stream);
        break;
      case ISING_KERNEL_MSC:
        st = run_tile(h, (h->all_lattice && p->schedule == ISING_SCHED_COLOUR) ? 3 : 2, replicas, p, spins_dev,
                      energy_dev, energy_i32_dev, minima_dev, stream);
        break;
      case ISING_KERNEL_SWEEP:
        if (launch_sweep(h, p, replicas, spins_dev, energy_dev, energy_i32_dev, minima_dev, by_time && !stats, stream) !=
            cudaSuccess)
          st = ISING_ERR_CUDA;
        break;
      case ISING_KERNEL_DENSE_TC: {
        const cudaError_t e = launch_dense(h, p, replicas, spins_dev, energy_dev, energy_i32_dev, minima_dev, seeds,
                                           stream);
        if (e == cudaErrorLaunchTimeout) st = ISING_ERR_TIMEOUT;  // a bounded device wait gave up
        else if (e != cudaSuccess) st = ISING_ERR_CUDA;
        break;
      }
      case ISING_KERNEL_PLAIN:
        kt_begin(h, "plain_path", stream);
        if (launch_plain(h, p, replicas, spins_dev, energy_dev, energy_i32_dev, minima_dev, seeds, stream) !=
            cudaSuccess)
          st = ISING_ERR_CUDA;
        kt_end(h, stream);
        break;
      default:
        st = ISING_ERR_UNSUPPORTED;
        break;
    }
  } while (0);
  if (st == ISING_OK && stats) {
    if (cudaMemcpyAsync(h->h_stats_pinned, h->d_stats, sizeof(unsigned long long) * 6, cudaMemcpyDeviceToHost,
                        stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess) {
      st = ISING_ERR_CUDA;
    } else {
      stats->flip_evals = h->h_stats_pinned[0];
      stats->flips = h->h_stats_pinned[1];
      stats->minima = h->h_stats_pinned[2];
      stats->descents = h->h_stats_pinned[3];
      stats->sweeps = h->h_stats_pinned[4];
      stats->launches = h->launches;
      // the families that skip visits count the evaluated ones; the others
      // compute every gain they visit
      const bool skips = kernel == ISING_KERNEL_TILE || kernel == ISING_KERNEL_MSC || kernel == ISING_KERNEL_SWEEP;
      stats->evaluated = skips ? h->h_stats_pinned[5] : h->h_stats_pinned[0];
    }
  }
  if (cur != h->device) cudaSetDevice(cur);
  return st;
}

ising_status ising_autotune(ising_handle *h, int32_t replicas, const ising_search_params *p, int32_t *chosen,
                            cudaStream_t stream) {
  const NvtxRange nvtx_range("ising_autotune");
  if (!h || !p || replicas < 1) return ISING_ERR_INVALID_ARG;
  ising_status st = validate_params(p);
  if (st != ISING_OK) return st;
  const std::string key = tune_key(h, replicas, p);
  // a cached decision for this GPU and instance class?
  int32_t cached = tune_cache_lookup(key);
  if (cached > 0) {
    ising_search_params q = *p;
    q.kernel = (ising_kernel)cached;
    if (resolve_kernel(h, replicas, &q) == cached) {
      h->tuned[replicas] = cached;
      if (chosen) *chosen = cached;
      return ISING_OK;
    }
  }
  // time every eligible family on this handle with these parameters
  const int32_t families[] = {ISING_KERNEL_MSC, ISING_KERNEL_TILE, ISING_KERNEL_SWEEP, ISING_KERNEL_DENSE_TC};
  int8_t *spins = nullptr;
  double *E = nullptr;
  int32_t *mins = nullptr;
  if (cudaMalloc(&spins, (size_t)replicas * h->total_spins) != cudaSuccess ||
      cudaMalloc(&E, sizeof(double) * replicas * h->n_inst) != cudaSuccess ||
      cudaMalloc(&mins, sizeof(int32_t) * replicas * h->n_inst) != cudaSuccess) {
    cudaFree(spins);
    cudaFree(E);
    cudaFree(mins);
    return ISING_ERR_OOM;
  }
  std::vector<uint64_t> seeds(h->n_inst);
  for (int32_t b = 0; b < h->n_inst; ++b) seeds[b] = 0x9E3779B97F4A7C15ull * (uint64_t)(b + 1);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  int32_t best_k = -1;
  float best_ms = 0.0f;
  h->tuned.erase(replicas);
  for (int32_t fam : families) {
    ising_search_params q = *p;
    q.kernel = (ising_kernel)fam;
    if (resolve_kernel(h, replicas, &q) != fam) continue;
    ising_stats s1;
    if (ising_local_search(h, seeds.data(), replicas, &q, spins, E, nullptr, mins, &s1, stream) != ISING_OK) continue;
    cudaEventRecord(e0, stream);
    ising_status r = ising_local_search(h, seeds.data(), replicas, &q, spins, E, nullptr, mins, nullptr, stream);
    cudaEventRecord(e1, stream);
    if (r != ISING_OK || cudaEventSynchronize(e1) != cudaSuccess) continue;
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (best_k < 0 || ms < best_ms) {
      best_k = fam;
      best_ms = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(spins);
  cudaFree(E);
  cudaFree(mins);
  if (best_k < 0) return ISING_ERR_UNSUPPORTED;
  h->tuned[replicas] = best_k;
  tune_cache_store(key, best_k);
  if (chosen) *chosen = best_k;
  return ISING_OK;
}

ising_status ising_destroy(ising_handle *h) {
  free_handle(h);
  return ISING_OK;
}

ising_status ising_fm_search(ising_handle *h, const uint64_t *seeds, int32_t replicas, const ising_fm_params *p,
                             int8_t *spins_dev, double *energy_dev, int32_t *passes_dev, ising_stats *stats,
                             cudaStream_t stream) {
  const NvtxRange nvtx_range("ising_fm_search");
  if (!h || !seeds || !p || replicas < 1 || p->restarts < 1 || p->max_passes < 0 || p->starts < 0 ||
      p->starts > 2 || p->reg_kernel < -1 || p->reg_kernel > 1 || !spins_dev || !energy_dev)
    return ISING_ERR_INVALID_ARG;
  if (h->latched != ISING_OK) {
    ising_status l = h->latched;
    h->latched = ISING_OK;
    return l;
  }
  if (h->nmax > fm_max_spins()) return ISING_ERR_UNSUPPORTED;
  if ((int64_t)replicas * h->n_inst > 0x7fffffffLL) return ISING_ERR_UNSUPPORTED;
  int cur = 0;
  cudaGetDevice(&cur);
  if (cur != h->device) cudaSetDevice(h->device);
  ising_status st = ISING_OK;
  h->launches = 0;
  if (fault_is("launch")) {
    st = ISING_ERR_CUDA;
  } else if (cudaMemcpyAsync(h->d_seeds, seeds, sizeof(uint64_t) * h->n_inst, cudaMemcpyHostToDevice, stream) !=
                 cudaSuccess ||
             cudaMemsetAsync(h->d_stats, 0, sizeof(unsigned long long) * 8, stream) != cudaSuccess) {
    st = ISING_ERR_CUDA;
  } else {
    kt_begin(h, "fm_kernel", stream);
    if (launch_fm(h, replicas, p, spins_dev, energy_dev, passes_dev, stream) != cudaSuccess)
      st = ISING_ERR_CUDA;
    kt_end(h, stream);
  }
  if (st == ISING_OK && stats) {
    if (cudaMemcpyAsync(h->h_stats_pinned, h->d_stats, sizeof(unsigned long long) * 5, cudaMemcpyDeviceToHost,
                        stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess) {
      st = ISING_ERR_CUDA;
    } else {
      stats->flip_evals = h->h_stats_pinned[0];
      stats->flips = h->h_stats_pinned[1];
      stats->minima = h->h_stats_pinned[2];
      stats->descents = h->h_stats_pinned[3];
      stats->sweeps = h->h_stats_pinned[4];
      stats->launches = h->launches;
      stats->evaluated = h->h_stats_pinned[0];
    }
  }
  if (cur != h->device) cudaSetDevice(cur);
  return st;
}

ising_status ising_set_timing(ising_handle *h, int32_t enable) {
  if (!h) return ISING_ERR_INVALID_ARG;
  if (enable && h->kt_used && cudaEventSynchronize(h->ktimers[h->kt_used - 1].b) != cudaSuccess)
    return ISING_ERR_CUDA;
  h->timing = enable != 0;
  if (enable) h->kt_used = 0;
  return ISING_OK;
}

int32_t ising_kernel_times(ising_handle *h, ising_kernel_time *out, int32_t cap) {
  if (!h || cap < 0 || (cap > 0 && !out)) return -(int32_t)ISING_ERR_INVALID_ARG;
  std::vector<ising_kernel_time> acc;
  for (size_t i = 0; i < h->kt_used; ++i) {
    const auto &t = h->ktimers[i];
    float ms = 0.0f;
    if (cudaEventSynchronize(t.b) != cudaSuccess || cudaEventElapsedTime(&ms, t.a, t.b) != cudaSuccess)
      return -(int32_t)ISING_ERR_CUDA;
    size_t k = 0;
    while (k < acc.size() && std::strcmp(acc[k].name, t.name) != 0) ++k;
    if (k == acc.size()) acc.push_back(ising_kernel_time{t.name, 0.0, 0});
    acc[k].ms += (double)ms;
    acc[k].launches += 1;
  }
  for (size_t k = 0; k < acc.size() && (int32_t)k < cap; ++k) out[k] = acc[k];
  return (int32_t)acc.size();
}

const char *ising_status_string(ising_status s) {
  switch (s) {
    case ISING_OK: return "ok";
    case ISING_ERR_INVALID_ARG: return "invalid argument";
    case ISING_ERR_ASYMMETRIC: return "coupling matrix is not symmetric";
    case ISING_ERR_SELF_LOOP: return "coupling matrix has a self loop";
    case ISING_ERR_BAD_HYPEREDGE: return "malformed hyper-edge";
    case ISING_ERR_BAD_COLOURING: return "colouring is not proper for the conflict graph";
    case ISING_ERR_UNSUPPORTED: return "unsupported instance/kernel combination";
    case ISING_ERR_OOM: return "out of memory";
    case ISING_ERR_CUDA: return "CUDA runtime error";
    case ISING_ERR_TIMEOUT: return "device-side wait timed out";
    case ISING_ERR_DEVICE: return "device-side check failed";
  }
  return "unknown status";
}

}  // extern "C"
