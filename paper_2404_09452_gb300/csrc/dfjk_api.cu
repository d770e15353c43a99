// C ABI of the DF-J/K build: handle lifetime, setup (integrals, metric,
// Cholesky, whitening) and build (X, K, rho, J, energies) orchestration, diagnostic accessors and error plumbing.
// Paper: Introduction, contribution 1 (density fitting: 3-centre integrals,
// then tensor contractions) and Sec. "Dataset and Performance" (intermediates
// of small and medium molecules kept resident in GPU memory).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <initializer_list>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "boys.cuh"
#include "common.cuh"
#include "grad.cuh"
#include "integrals.cuh"
#include "ksplit.cuh"
#include "linalg.cuh"
#include "ozaki.cuh"
#include "pool.cuh"
#include "stream_scope.cuh"

namespace dfjk {

static thread_local std::string g_last_error;
void set_error(const std::string &msg) { g_last_error = msg; }
std::atomic<uint64_t> &launch_counter() {
  static std::atomic<uint64_t> c{0};
  return c;
}

// ---- phase timing ----------------------------------------------------------------

struct PhaseRec {
  int phase;
  cudaEvent_t a, b;
};
static std::mutex g_timing_mu;
static bool g_timing = false;
static std::vector<PhaseRec> g_phase_recs;
static std::vector<cudaEvent_t> g_event_pool;

static cudaEvent_t take_event() {
  if (!g_event_pool.empty()) {
    cudaEvent_t e = g_event_pool.back();
    g_event_pool.pop_back();
    return e;
  }
  cudaEvent_t e;
  DFJK_CUDA_CHECK(cudaEventCreate(&e));
  return e;
}

PhaseScope::PhaseScope(int ph, cudaStream_t s) : phase(ph), st(s) {
  std::lock_guard<std::mutex> lk(g_timing_mu);
  if (!g_timing) return;
  cudaEvent_t e = take_event();
  DFJK_CUDA_CHECK(cudaEventRecord(e, st));
  ev0 = (void *)e;
}

PhaseScope::~PhaseScope() {
  if (!ev0) return;
  std::lock_guard<std::mutex> lk(g_timing_mu);
  cudaEvent_t e1;
  if (!g_event_pool.empty()) {
    e1 = g_event_pool.back();
    g_event_pool.pop_back();
  } else if (cudaEventCreate(&e1) != cudaSuccess) {
    return;
  }
  if (cudaEventRecord(e1, st) != cudaSuccess) return;
  g_phase_recs.push_back(PhaseRec{phase, (cudaEvent_t)ev0, e1});
}

// ---- device buffers -------------------------------------------------------------

template <class T>
struct DBuf {
  T *p = nullptr;
  size_t n = 0;
  void alloc(size_t count) {
    release();
    if (count == 0) return;
    p = (T *)pool_alloc(count * sizeof(T));
    n = count;
  }
  void upload(const std::vector<T> &v, cudaStream_t st) {
    alloc(v.size());
    if (!v.empty()) DFJK_CUDA_CHECK(cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, st));
  }
  void release() {
    if (p) pool_free(p, n * sizeof(T));
    p = nullptr;
    n = 0;
  }
  size_t bytes() const { return n * sizeof(T); }
  ~DBuf() { release(); }
};

// B: device memory from the cache, or pinned host memory mapped into the device
// address space, read and written by the kernels in place (NVLink-C2C on a
// Grace-Blackwell node) so that molecules whose B does not fit next to the
// build's work buffers still run.
struct BStore {
  double *p = nullptr;   // device-usable address
  void *hp = nullptr;    // host allocation (host-resident only)
  size_t n = 0;
  bool host = false;
  void alloc(size_t count, bool on_host) {
    release();
    if (on_host) {
      if (cudaHostAlloc(&hp, std::max<size_t>(count, 1) * sizeof(double), cudaHostAllocMapped) != cudaSuccess) {
        cudaGetLastError();
        hp = nullptr;
        throw Error{DFJK_ERR_OOM, "pinned host memory for B (" + std::to_string(count * 8) + " bytes)"};
      }
      void *d = nullptr;
      DFJK_CUDA_CHECK(cudaHostGetDevicePointer(&d, hp, 0));
      p = (double *)d;
    } else {
      p = (double *)pool_alloc(std::max<size_t>(count, 1) * sizeof(double));
    }
    host = on_host;
    n = count;
  }
  void release() {
    if (host && hp) cudaFreeHost(hp);
    if (!host && p) pool_free(p, std::max<size_t>(n, 1) * sizeof(double));
    p = nullptr;
    hp = nullptr;
    n = 0;
  }
  size_t bytes() const { return n * sizeof(double); }
  size_t device_bytes() const { return host ? 0 : bytes(); }
  ~BStore() { release(); }
};

// A double as a double-single pair.
static float2 df_pair(double v) {
  const float hi = (float)v;
  return make_float2(hi, (float)(v - (double)hi));
}

// ---- Boys table per device ---------------------------------------------------------

const double *boys_table_device() {
  static std::mutex mu;
  static std::map<int, double *> tabs;
  int dev = 0;
  DFJK_CUDA_CHECK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  auto it = tabs.find(dev);
  if (it != tabs.end()) return it->second;
  std::vector<double> h((size_t)BOYS_NPT * (BOYS_NCOL + 1));
  boys_table_host(h.data());
  double *d = nullptr;
  DFJK_CUDA_CHECK(cudaMalloc(&d, h.size() * sizeof(double)));
  DFJK_CUDA_CHECK(cudaMemcpy(d, h.data(), h.size() * sizeof(double), cudaMemcpyHostToDevice));
  tabs[dev] = d;
  return d;
}

const float2 *boys_table_device_df() {
  static std::mutex mu;
  static std::map<int, float2 *> tabs;
  int dev = 0;
  DFJK_CUDA_CHECK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  auto it = tabs.find(dev);
  if (it != tabs.end()) return it->second;
  std::vector<double> h((size_t)BOYS_NPT * (BOYS_NCOL + 1));
  boys_table_host(h.data());
  std::vector<float2> f(h.size());
  for (size_t i = 0; i < h.size(); ++i) f[i] = df_pair(h[i]);
  float2 *d = nullptr;
  DFJK_CUDA_CHECK(cudaMalloc(&d, f.size() * sizeof(float2)));
  DFJK_CUDA_CHECK(cudaMemcpy(d, f.data(), f.size() * sizeof(float2), cudaMemcpyHostToDevice));
  tabs[dev] = d;
  return d;
}

const float *boys_table_device_f32() {
  static std::mutex mu;
  static std::map<int, float *> tabs;
  int dev = 0;
  DFJK_CUDA_CHECK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  auto it = tabs.find(dev);
  if (it != tabs.end()) return it->second;
  std::vector<double> h((size_t)BOYS_NPT * (BOYS_NCOL + 1));
  boys_table_host(h.data());
  std::vector<float> f(h.begin(), h.end());
  float *d = nullptr;
  DFJK_CUDA_CHECK(cudaMalloc(&d, f.size() * sizeof(float)));
  DFJK_CUDA_CHECK(cudaMemcpy(d, f.data(), f.size() * sizeof(float), cudaMemcpyHostToDevice));
  tabs[dev] = d;
  return d;
}

// ---- host-side basis ---------------------------------------------------------------

struct HostBasis {
  int nshell = 0, nfunc = 0;
  std::vector<int> l, nprim, prim_off, func_off, atom;
  std::vector<double> exps, coefs_raw, coefs, center;  // coefs: normalised radial
};

static void read_basis(const dfjk_basis *b, int natom, const double *coords, HostBasis &hb,
                       const char *what) {
  if (!b || b->nshell < 0 || (b->nshell > 0 && !b->shells))
    throw Error{DFJK_ERR_ARG, std::string(what) + ": null basis"};
  hb = HostBasis();
  hb.nshell = b->nshell;
  for (int s = 0; s < b->nshell; ++s) {
    const dfjk_shell &sh = b->shells[s];
    if (sh.l < 0 || sh.l > 2) throw Error{DFJK_ERR_UNSUPPORTED, std::string(what) + ": l must be 0..2"};
    if (sh.nprim < 1 || sh.nprim > 8)
      throw Error{DFJK_ERR_UNSUPPORTED, std::string(what) + ": nprim must be 1..8"};
    if (sh.atom < 0 || sh.atom >= natom) throw Error{DFJK_ERR_ARG, std::string(what) + ": atom index"};
    if (!sh.exps || !sh.coefs) throw Error{DFJK_ERR_ARG, std::string(what) + ": null exps/coefs"};
    hb.l.push_back(sh.l);
    hb.atom.push_back(sh.atom);
    hb.nprim.push_back(sh.nprim);
    hb.prim_off.push_back((int)hb.exps.size());
    hb.func_off.push_back(hb.nfunc);
    hb.nfunc += ncart(sh.l);
    for (int d = 0; d < 3; ++d) {
      const double x = coords[3 * sh.atom + d];
      if (!std::isfinite(x)) throw Error{DFJK_ERR_ARG, "non-finite coordinate"};
      hb.center.push_back(x);
    }
    // <chi|chi> with per-component normalised primitives:
    // sum_kl d_k d_l (2 sqrt(a_k a_l)/(a_k + a_l))^(l + 3/2)
    double ss = 0.0;
    for (int k = 0; k < sh.nprim; ++k) {
      if (!(sh.exps[k] > 0.0) || !std::isfinite(sh.exps[k]) || !std::isfinite(sh.coefs[k]))
        throw Error{DFJK_ERR_ARG, std::string(what) + ": exponents must be positive and finite"};
      for (int q = 0; q < sh.nprim; ++q) {
        const double a = sh.exps[k], c = sh.exps[q];
        ss += sh.coefs[k] * sh.coefs[q] * std::pow(2.0 * std::sqrt(a * c) / (a + c), sh.l + 1.5);
      }
    }
    if (!(ss > 0.0)) throw Error{DFJK_ERR_ARG, std::string(what) + ": contraction has zero norm"};
    const double scale = 1.0 / std::sqrt(ss);
    for (int k = 0; k < sh.nprim; ++k) {
      const double a = sh.exps[k];
      hb.exps.push_back(a);
      hb.coefs_raw.push_back(sh.coefs[k]);
      hb.coefs.push_back(sh.coefs[k] * scale * std::pow(2.0 * a / M_PI, 0.75) * std::pow(4.0 * a, 0.5 * sh.l));
    }
  }
}

// Work buffers of the X GEMM over kept pairs: the slices of B for a chunk of rows
// P, and of C for the groups of AOs.  C's are taken for ranges of groups that fit
// C_SLICE_CAP (one range up to about 110 atoms; more than one re-slices C in
// every chunk).
struct XWork {
  DBuf<__nv_bfloat16> bsl, cdat;
  DBuf<int> cexp;
  std::vector<int> range;  // group boundaries
  bool b_ready = false;    // bsl holds the slices of all of B (build_one)
  void release() {
    b_ready = false;
    bsl.release();
    cdat.release();
    cexp.release();
    range.clear();
  }
};
constexpr size_t C_SLICE_CAP = (size_t)1 << 30;

// Buffers of the K GEMM over sliced operands, sized once for the longest reduction
// range (alloc_kwork): graphs and queued builds keep their addresses.
struct KWork {
  DBuf<double> part;  // partial sums of the splits
  DBuf<int> seq;      // split counters of the ordered kernel
  void release() {
    part.release();
    seq.release();
  }
};

// Launch-shape choices that do not change what is computed, only how fast:
// rows per block of the slicing kernels, the K GEMM's split-K range and the
// mixed build's work-buffer cap (which sets the aux-row chunk).  0 = the
// built-in default (or the corresponding environment variable).
struct Tuning {
  int slice_rows = 0;   // DFJK_SLICE_ROWS: 8, 16, 32
  int pslice_rows = 0;  // DFJK_PSLICE_ROWS: warps per block of B's slicing, 4, 8, 16 (default 8)
  int k_range_mb = 0;   // DFJK_K_RANGE_MB
  int build_ws_mb = 0;  // DFJK_BUILD_WS_MB
};

// A tuning table: text lines "nao_lo nao_hi slice_rows pslice_rows k_range_mb
// build_ws_mb [anything]" ('#' starts a comment); the first line with
// nao_lo <= nao < nao_hi applies.  Tables are parsed once per path.
static bool lookup_tuning(const char *path, int nao, Tuning &t) {
  if (!path || !*path) return false;
  static std::mutex mu;
  static std::map<std::string, std::vector<std::vector<long>>> tables;
  std::lock_guard<std::mutex> lk(mu);
  auto it = tables.find(path);
  if (it == tables.end()) {
    std::vector<std::vector<long>> rows;
    FILE *f = std::fopen(path, "r");
    if (!f) throw Error{DFJK_ERR_ARG, std::string("tuning table not readable: ") + path};
    char line[512];
    while (std::fgets(line, sizeof line, f)) {
      if (char *c = std::strchr(line, '#')) *c = 0;
      long v[6];
      if (std::sscanf(line, "%ld %ld %ld %ld %ld %ld", &v[0], &v[1], &v[2], &v[3], &v[4], &v[5]) == 6)
        rows.push_back(std::vector<long>(v, v + 6));
    }
    std::fclose(f);
    it = tables.emplace(path, rows).first;
  }
  for (const auto &r : it->second)
    if (r[0] <= nao && nao < r[1]) {
      t.slice_rows = (int)r[2];
      t.pslice_rows = (int)r[3];
      t.k_range_mb = (int)r[4];
      t.build_ws_mb = (int)r[5];
      return true;
    }
  return false;
}

}  // namespace dfjk

using namespace dfjk;

struct dfjk_ctx {
  int device = 0;
  dfjk_options opt{};
  int natom = 0;
  std::vector<double> coords;
  HostBasis orb, aux;
  int nao = 0, naux = 0, naux_pad = 0;
  bool resident = false;

  // device: bases
  DBuf<double> o_center, o_exps, o_coefs, a_center, a_exps, a_cdiv, a_g1;
  DBuf<float2> a_df;   // aux centres (from c0), exponents, cdiv, g1 as double-single pairs
  double c0[3] = {0.0, 0.0, 0.0};  // centroid
  bool df_range = false;  // a mixed handle whose exponents and coordinates suit FP32 pairs (df_range_ok)
  bool use_df = false;  // its integrals in double-single, unless fp32_pair_thresh = 0 asks for FP64
  DBuf<int> o_prim_off, o_nprim, o_func_off, a_prim_off, a_nprim, a_func_off;
  DBuf<int> aux_cls[3];
  std::vector<int> aux_cls_n = std::vector<int>(3, 0);
  // shell pairs (global ids in class order)
  std::vector<int> cls_begin;  // 7 entries: ss ps pp ds dp dd
  std::vector<int> pa_h, pb_h, npp_h;
  DBuf<int> pair_a, pair_b, pair_npp, pair_keep, kept;
  DBuf<long long> pair_rec_off, pair_col;
  DBuf<double> rec, q, scal;
  DBuf<float2> recd;   // double-single records (use_df, or FP32 pairs)
  std::vector<int> kept_h;
  std::vector<long long> pair_col_h;
  std::vector<int> kept_cls_begin;  // 7 entries into kept list
  long long ncol = 0;
  int npair_kept = 0;
  std::vector<int> kept32_begin;  // per class: first kept index evaluated in FP32
  long long prim_pairs64[6] = {0, 0, 0, 0, 0, 0}, prim_pairs32[6] = {0, 0, 0, 0, 0, 0};
  int npair_fp32 = 0;
  double fp32_thresh = 0.0;
  int nslab = 0;  // T column slabs of the last setup (one whitening launch each)
  DBuf<int> colmu, colnu;
  // metric
  DBuf<double> V, L, Linv, Dinv;
  DBuf<int> status;
  DBuf<int> tctr;  // tile counter of the tensor-core GEMM launches (stream-ordered)
  // whitened tensor B, P contiguous: DFJK_FP64 keeps both triangles,
  // B[(mu nao + nu) ldb + P]; DFJK_MIXED keeps one row per kept column m (the
  // whitening's output order), B[m ldb + P], found through rowmap, and slices
  // it per build, chunk by chunk of rows P, just before X = B C of that chunk
  BStore B;
  long long ldb = 0;
  bool lean = false;    // B of the kept pairs only (the mixed path)
  // dense products on the tensor cores: always for DFJK_MIXED, for DFJK_FP64 above
  // OZ_F64_MIN_WORK (use_slices); slice formats of the whitening and of the build
  bool sliced = false;
  int wfmt = OZ_48, bfmt = OZ_36;
  PairLists pl;         // kept partners of every AO (sliced products)
  DBuf<int> pl_buf, pl_krow;
  std::vector<int> pl_h;  // list, gstep, zstep and zgroup, in this order
  std::vector<int> gstep_h, gfirst_h;  // host copies: K steps before a group, its first AO
  XWork xw;
  DBuf<double> b_stage;  // B in host memory: the columns of B of a build's chunk on the device
  int chunk_rows = 0;   // rows P per build chunk (sliced products)
  DBuf<int> Bexpo;      // slice exponents of B's slices, [mu][expo_rows][pl.nkb]
  int expo_rows = 0;    // rows P of Bexpo (naux_pad rounded up to 128)
  Tuning tune;          // launch-shape choices (tuning table entry or defaults)
  // build workspace
  int ws_nocc = -1;
  DBuf<double> D, rho, rho_work, X, Kpart, en_work, e;
  DBuf<int> rowmap;  // DFJK_MIXED: row of B for AO pair (mu, nu), -1 if screened
  int ksplit = 1;
  SlicedOp Xsl;  // slices of X, the K GEMM's operand
  KWork kw;
  DBuf<double> uks_D, uks_J;  // spin-unrestricted build: D_a + D_b and J[D_b]
  cudaStream_t side = nullptr;  // setup: Cholesky + inverse beside the integrals
  cudaStream_t side2 = nullptr;  // the Cholesky's bulk trailing updates (look-ahead)
  cudaStream_t side3 = nullptr;  // the triangular inverse, behind the Cholesky
  cudaEvent_t ev_done = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_panel = nullptr, ev_bulk = nullptr;
  cudaEvent_t ev_int = nullptr;  // integral streams: fork, then join, in turn
  ~dfjk_ctx() {
    oz_free(Xsl);
    for (cudaStream_t s : {side, side2, side3})
      if (s) {
        cudaStreamSynchronize(s);
        cudaStreamDestroy(s);
      }
    for (cudaEvent_t e : {ev_fork, ev_join, ev_panel, ev_bulk, ev_int, ev_done})
      if (e) cudaEventDestroy(e);
  }
};

namespace {

cudaStream_t S(void *s) { return (cudaStream_t)s; }

int fail(const Error &e) {
  set_error(e.msg);
  return e.code;
}

// Orbital shell pairs (l_a >= l_b; equal l: a >= b), grouped by class.
void enumerate_pairs(dfjk_ctx *h) {
  static const int cls[6][2] = {{0, 0}, {1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
  h->cls_begin.assign(7, 0);
  h->pa_h.clear();
  h->pb_h.clear();
  h->npp_h.clear();
  std::vector<int> by_l[3];  // orbital shells of each l, ascending
  for (int a = 0; a < h->orb.nshell; ++a) by_l[h->orb.l[a]].push_back(a);
  for (int c = 0; c < 6; ++c) {
    h->cls_begin[c] = (int)h->pa_h.size();
    for (int a : by_l[cls[c][0]])
      for (int b : by_l[cls[c][1]]) {
        if (cls[c][0] == cls[c][1] && b > a) break;
        h->pa_h.push_back(a);
        h->pb_h.push_back(b);
        h->npp_h.push_back(h->orb.nprim[a] * h->orb.nprim[b]);
      }
  }
  h->cls_begin[6] = (int)h->pa_h.size();
}

// DFJK_FP64 takes its dense products (whitening, X, K and the gradient's and the
// density build's GEMMs) as exact products of 56-bit slices (OZ_F64) on the tensor
// cores, some 40 TFLOP/s of FP64-grade work against the FP64 pipe's 1.06, once
// nao^2 naux reaches this (one build at 4 atoms, 6.9e5: 345 us on the FP64 pipe,
// 216 us here; at 20 atoms 12.8 and 1.0 ms, whitening 14.2 and 0.96); the water
// input (2e4) takes 183 us on the FP64 pipe and 186 us here.  Errors against 64-bit
// references, geometric means of the largest relative ones: 24 molecules of 5 to 23 atoms
// J 3.7e-12 and K 4.4e-13 (FP64 pipe and an earlier Cholesky: 3.4e-12 and 4.6e-13); 32 of 5
// to 10 atoms, gradient of E_J - E_K/2, 2.63e-12 here and on the FP64 pipe (2.87e-12
// before).  V, T and L^-1 set them; one molecule alone goes either way by a factor of two.
constexpr double OZ_F64_MIN_WORK = 3e5;
bool use_slices(int precision, int nao, int np) {
  return precision == DFJK_MIXED || (double)nao * nao * np >= OZ_F64_MIN_WORK;
}

// Device bytes of a handle's resident data: B (none when B is in host
// memory) and the metric, its Cholesky factor and inverse.  Before screening:
// the mixed path's B holds one row per kept AO pair, at most the
// nao (nao + 1) / 2 of the triangle (the bound used here); the FP64 path's
// holds both triangles of every pair.
size_t resident_estimate(const dfjk_ctx *h) {
  const size_t np2 = (size_t)h->naux_pad * h->naux_pad;
  const bool mixed = h->opt.precision == DFJK_MIXED;
  const size_t rows = mixed ? (size_t)h->nao * (h->nao + 1) / 2 : (size_t)h->nao * h->nao;
  const size_t b = h->opt.b_on_host ? 0 : rows * h->naux_pad * sizeof(double);
  return b + 3 * np2 * sizeof(double);
}

void upload_bases(dfjk_ctx *h, cudaStream_t st) {
  h->o_center.upload(h->orb.center, st);
  h->o_exps.upload(h->orb.exps, st);
  h->o_coefs.upload(h->orb.coefs, st);
  h->o_prim_off.upload(h->orb.prim_off, st);
  h->o_nprim.upload(h->orb.nprim, st);
  h->o_func_off.upload(h->orb.func_off, st);
  std::vector<double> cdiv(h->aux.exps.size()), g1(h->aux.exps.size());
  for (size_t k = 0; k < h->aux.exps.size(); ++k) {
    cdiv[k] = h->aux.coefs[k] / h->aux.exps[k];
    g1[k] = 0.5 / h->aux.exps[k];
  }
  h->a_center.upload(h->aux.center, st);
  h->a_exps.upload(h->aux.exps, st);
  h->a_cdiv.upload(cdiv, st);
  h->a_g1.upload(g1, st);
  {
    const size_t ns = h->aux.nshell, npr = h->aux.exps.size();
    std::vector<float2> d;
    d.reserve(3 * ns + 3 * npr);
    for (size_t i = 0; i < 3 * ns; ++i) d.push_back(df_pair(h->aux.center[i] - h->c0[i % 3]));
    for (const std::vector<double> *v : {(const std::vector<double> *)&h->aux.exps, (const std::vector<double> *)&cdiv,
                                         (const std::vector<double> *)&g1})
      for (double x : *v) d.push_back(df_pair(x));
    h->a_df.upload(d, st);
  }
  h->a_prim_off.upload(h->aux.prim_off, st);
  h->a_nprim.upload(h->aux.nprim, st);
  h->a_func_off.upload(h->aux.func_off, st);
  for (int c = 0; c < 3; ++c) {
    std::vector<int> lst;
    for (int s = 0; s < h->aux.nshell; ++s)
      if (h->aux.l[s] == c) lst.push_back(s);
    h->aux_cls_n[c] = (int)lst.size();
    h->aux_cls[c].upload(lst, st);
  }
}

OrbArgs orb_args(dfjk_ctx *h) {
  return OrbArgs{h->o_center.p, h->o_prim_off.p, h->o_nprim.p, h->o_exps.p, h->o_coefs.p, h->o_func_off.p};
}
AuxArgs aux_args(dfjk_ctx *h) {
  const size_t ns = h->aux.nshell, npr = h->aux.exps.size();
  const float2 *d = h->a_df.p;
  return AuxArgs{h->a_center.p, h->a_prim_off.p, h->a_nprim.p, h->a_exps.p, h->a_cdiv.p, h->a_g1.p,
                 h->a_func_off.p, d, d + 3 * ns, d + 3 * ns + npr, d + 3 * ns + 2 * npr};
}

__global__ void pad_identity_kernel(double *V, int n, int npad, int ld) {
  const int i = n + blockIdx.x * blockDim.x + threadIdx.x;
  if (i < npad) V[(long long)i * ld + i] = 1.0;
}

__global__ void zero_upper_kernel(double *A, int n, int ld) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n * n) return;
  const int i = (int)(e / n), j = (int)(e % n);
  if (j > i) A[(long long)i * ld + j] = 0.0;
}

// Whether double-single integrals keep their 48 bits: exponents whose powers stay
// inside the FP32 range ((2 alpha)^6 and (2p)^-4; (2 alpha)^8 of the FP32 Schwarz diagonal,
// which a handle beyond the range takes in FP64 as well), and coordinates (relative to the
// centroid) whose 48 bits resolve 5e-13 bohr.
bool df_range_ok(const dfjk_ctx *h) {
  for (const std::vector<double> *e : {&h->orb.exps, &h->aux.exps})
    for (double x : *e)
      if (x < 1e-4 || x > 1e4) return false;
  for (size_t i = 0; i < h->coords.size(); ++i)
    if (std::fabs(h->coords[i] - h->c0[i % 3]) > 256.0) return false;
  return true;
}

// Metric (P|Q) into V (naux_pad^2, identity on the padding).
void compute_metric(dfjk_ctx *h, const double *tab, cudaStream_t st) {
  const int np = h->naux_pad;
  h->V.alloc((size_t)np * np);
  DFJK_CUDA_CHECK(cudaMemsetAsync(h->V.p, 0, h->V.bytes(), st));
  if (np > h->naux) {
    pad_identity_kernel<<<ceil_div(np - h->naux, 64), 64, 0, st>>>(h->V.p, h->naux, np, np);
    DFJK_LAUNCHED();
  }
  static const int cls[6][2] = {{0, 0}, {1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
  for (int c = 0; c < 6; ++c) {
    const int lp = cls[c][0], lq = cls[c][1];
    const long long n = h->aux_cls_n[lp], m = h->aux_cls_n[lq];
    const MetricArgs a{lp == lq ? n * (n + 1) / 2 : n * m, std::max((int)m, 1), h->aux_cls[lp].p, h->aux_cls[lq].p, h->V.p, np};
    launch_metric(lp, lq, a, aux_args(h), tab, st);
  }
}

// Streams the classes of the 3-centre integrals are spread over (36 launches per
// slab, most of them small for a small molecule; the FP32 pairs run beside the
// others).  Four per device, shared by all handles: work of several handles on them
// is only ordered, never lost, and each call joins them to its own stream by events.
constexpr int INT_STREAMS = 4;
const cudaStream_t *integral_streams() {
  static std::mutex mu;
  static std::map<int, std::vector<cudaStream_t>> all;
  int dev = 0;
  DFJK_CUDA_CHECK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  std::vector<cudaStream_t> &v = all[dev];
  while ((int)v.size() < INT_STREAMS) {
    cudaStream_t s;
    DFJK_CUDA_CHECK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    v.reserve(INT_STREAMS);
    v.push_back(s);
  }
  return v.data();
}

// `st` forked to the integral streams for the scope's lifetime and joined at its end, also
// when a launch throws (what the kernels use is then not released under them).
struct IntegralFork {
  const cudaStream_t *is = integral_streams();
  const cudaStream_t st;
  const cudaEvent_t ev;
  IntegralFork(cudaStream_t st, cudaEvent_t ev) : st(st), ev(ev) {
    DFJK_CUDA_CHECK(cudaEventRecord(ev, st));
    for (int k = 0; k < INT_STREAMS; ++k) DFJK_CUDA_CHECK(cudaStreamWaitEvent(is[k], ev, 0));
  }
  ~IntegralFork() {
    for (int k = 0; k < INT_STREAMS; ++k) {
      cudaEventRecord(ev, is[k]);
      cudaStreamWaitEvent(st, ev, 0);
    }
  }
};

// Boys tables of the three arithmetics.
struct IntegralTables {
  const double *f64 = boys_table_device();
  const float *f32 = boys_table_device_f32();
  const float2 *dfs = boys_table_device_df();
};

// The integrals of one class (c, lc) for `n` pairs into a slab.
void launch_integrals(dfjk_ctx *h, int c, int lc, const int *pairs, int n, bool fp32, void *T, long long col0,
                      const IntegralTables &tab, cudaStream_t st) {
  static const int cls[6][2] = {{0, 0}, {1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
  const Eri3cArgs a{pairs, n, h->pair_rec_off.p, h->pair_npp.p, h->pair_col.p, h->rec.p, h->recd.p, h->aux_cls[lc].p,
                    h->aux_cls_n[lc], T, col0, h->naux_pad, h->use_df ? 1 : 0};
  if (fp32) launch_eri3c32(cls[c][0], cls[c][1], lc, a, aux_args(h), tab.f32, st);
  else if (h->use_df) launch_eri3cdf(cls[c][0], cls[c][1], lc, a, aux_args(h), tab.dfs, st);
  else launch_eri3c(cls[c][0], cls[c][1], lc, a, aux_args(h), tab.f64, st);
}

// The kept partners of every AO (PairLists): for each shell, the functions of the
// shells it has a kept pair with.
void make_pair_lists(dfjk_ctx *h) {
  const int ns = h->orb.nshell;
  std::vector<std::vector<int>> part(ns);
  for (int i : h->kept_h) {
    const int a = h->pa_h[i], b = h->pb_h[i];
    part[a].push_back(b);
    if (a != b) part[b].push_back(a);
  }
  std::vector<int> &list = h->pl_h, zstep, zgroup;
  std::vector<int> &gstep = h->gstep_h, &gfirst = h->gfirst_h;
  list.clear();
  gstep.assign(1, 0);
  gfirst.clear();
  int zs = 0, longest = 1;
  for (int a = 0; a < ns; ++a) {
    std::sort(part[a].begin(), part[a].end());
    const size_t at = list.size();
    for (int b : part[a])
      for (int c = 0; c < ncart(h->orb.l[b]); ++c) list.push_back(h->orb.func_off[b] + c);
    const int n = std::max<int>(1, ceil_div((long long)(list.size() - at), OZ_BK));
    list.resize(at + (size_t)n * OZ_BK, -1);
    longest = std::max(longest, n);
    gfirst.push_back(h->orb.func_off[a]);
    gstep.push_back(gstep.back() + n);
    for (int c = 0; c < ncart(h->orb.l[a]); ++c) {
      zstep.push_back(zs);
      zgroup.push_back(a);
      zs += n;
    }
  }
  zstep.push_back(zs);
  gfirst.push_back(h->nao);
  for (const std::vector<int> *v : {&gstep, &zstep, &zgroup}) list.insert(list.end(), v->begin(), v->end());
  h->pl.ngroup = ns;
  h->pl.fmt = h->bfmt;
  h->pl.longest = longest * OZ_BK;
  h->pl.nkb = ceil_div(h->pl.longest, oz_kblock(h->bfmt));
  h->pl.steps = zs;
  h->pl.gsteps = gstep.back();
}

void upload_pair_lists(dfjk_ctx *h, cudaStream_t st) {
  PairLists &pl = h->pl;
  h->pl_buf.upload(h->pl_h, st);
  h->pl_krow.alloc((size_t)pl.steps * OZ_BK);
  pl.list = h->pl_buf.p;
  pl.gstep = pl.list + pl.gsteps * OZ_BK;
  pl.zstep = pl.gstep + pl.ngroup + 1;
  pl.zgroup = pl.zstep + h->nao + 1;
  pl.krow = h->pl_krow.p;
  oz_krow(pl, h->lean ? h->rowmap.p : nullptr, h->nao, h->pl_krow.p, st);
}

// Doubles of `pc` columns of B, for every row.
size_t stage_size(const dfjk_ctx *h, int pc) {
  return std::max<size_t>(1, h->lean ? (size_t)h->ncol : (size_t)h->nao * h->nao) * pc;
}
// Columns [p0, p0 + pc) of a host-resident B, for every row, on the device (rows
// of pc doubles): the kernels that slice B read each pair twice.  `buf` has been
// sized by its owner: a buffer that moved here would leave a captured or queued
// build behind with the old one.
const double *stage_columns(dfjk_ctx *h, const DBuf<double> &buf, int p0, int pc, cudaStream_t st) {
  const size_t rows = h->lean ? (size_t)h->ncol : (size_t)h->nao * h->nao;
  if (buf.n < stage_size(h, pc)) throw Error{DFJK_ERR_STATE, "staging buffer of B"};
  if (rows)
    DFJK_CUDA_CHECK(cudaMemcpy2DAsync(buf.p, (size_t)pc * sizeof(double), h->B.p + p0,
                                      (size_t)h->ldb * sizeof(double), (size_t)pc * sizeof(double), rows,
                                      cudaMemcpyDefault, st));
  return buf.p;
}

// rho and J over the kept columns of B, stored as rows m (lean) or mu nao + nu.
void rho_kept(dfjk_ctx *h, const double *b, long long ldb, const double *D, int pc, double *rho, double *work,
              cudaStream_t st) {
  rho_kept_f64(b, ldb, h->ncol, h->colmu.p, h->colnu.p, h->nao, !h->lean, D, pc, rho, work, st);
}
void j_kept(dfjk_ctx *h, const double *rho, double *J, cudaStream_t st) {
  j_kept_f64(h->B.p, h->ldb, h->ncol, h->colmu.p, h->colnu.p, h->nao, !h->lean, h->naux_pad, rho, J, st);
}

// The setup on the device: shell pairs and screening, metric, Cholesky and
// inverse, 3-centre integrals, whitening.
void make_resident(dfjk_ctx *h, cudaStream_t st) {
  const IntegralTables tables;
  const double *tab = tables.f64;
  const float *tab32 = tables.f32;
  const int np = h->naux_pad;
  if (h->opt.hbm_budget_bytes > 0 && resident_estimate(h) > h->opt.hbm_budget_bytes)
    throw Error{DFJK_ERR_BUDGET, "resident data (" + std::to_string(resident_estimate(h)) +
                                     " bytes) exceeds hbm_budget_bytes"};
  PhaseScope span(12, st);
  upload_bases(h, st);
  h->status.alloc(1);
  if (!h->tctr.p) h->tctr.alloc(1);
  DFJK_CUDA_CHECK(cudaMemsetAsync(h->status.p, 0, sizeof(int), st));

  PhaseScope *ph0 = new PhaseScope(0, st);
  // a2: metric
  compute_metric(h, tab, st);

  // a3: Cholesky and inverse of the metric, on a side stream: they depend on
  // the metric alone, so they run beside the shell-pair kernels, the host's
  // pair bookkeeping and the 3-centre integrals; the first whitening waits
  // for them
  const bool mixed = h->opt.precision == DFJK_MIXED;
  if (!h->side) {
    // highest priority: the Cholesky chain is a sequence of small launches on
    // the critical path, its blocks go first whenever the integrals free an SM
    int lo = 0, hi = 0;
    DFJK_CUDA_CHECK(cudaDeviceGetStreamPriorityRange(&lo, &hi));
    DFJK_CUDA_CHECK(cudaStreamCreateWithPriority(&h->side, cudaStreamNonBlocking, hi));
    DFJK_CUDA_CHECK(cudaStreamCreateWithPriority(&h->side2, cudaStreamNonBlocking, hi));
    DFJK_CUDA_CHECK(cudaStreamCreateWithPriority(&h->side3, cudaStreamNonBlocking, std::min(lo, hi + 1)));
    DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&h->ev_done, cudaEventDisableTiming));
    DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
    DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming));
    DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&h->ev_panel, cudaEventDisableTiming));
    DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&h->ev_bulk, cudaEventDisableTiming));
    DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&h->ev_int, cudaEventDisableTiming));
  }
  const cudaStream_t s2 = h->side;
  DFJK_CUDA_CHECK(cudaEventRecord(h->ev_fork, st));
  DFJK_CUDA_CHECK(cudaStreamWaitEvent(s2, h->ev_fork, 0));
  struct OzLocal {  // slice buffers that live only during setup
    SlicedOp op;
    ~OzLocal() { oz_free(op); }
  } linv8_, t8_;
  SlicedOp &Linv8 = linv8_.op, &T8 = t8_.op;
  DBuf<double> inv_work, stage;
  DBuf<double> T;  // doubles, or double-single pairs (use_df)
  StreamDrain drain{st}, drain_side{s2}, drain_side2{h->side2}, drain_side3{h->side3};  // destroyed before the buffers above
  {
    PhaseScope ph1(1, s2);
    h->L.alloc((size_t)np * np);
    DFJK_CUDA_CHECK(cudaMemcpyAsync(h->L.p, h->V.p, h->V.bytes(), cudaMemcpyDeviceToDevice, s2));
    h->Dinv.alloc((size_t)(np / CHOL_NB) * CHOL_NB * CHOL_NB);
    h->Linv.alloc((size_t)np * np);
    inv_work.alloc((size_t)np * np);
    cholesky_inverse_f64(h->L.p, np, np, h->Dinv.p, h->Linv.p, inv_work.p, h->status.p,
                         CholStreams{s2, h->side2, h->side3, h->ev_panel, h->ev_bulk, h->ev_done});
    zero_upper_kernel<<<(unsigned)(((long long)np * np + 255) / 256), 256, 0, s2>>>(h->L.p, np, np);
    DFJK_LAUNCHED();
  }
  if (h->sliced) {  // L^-1 as the B operand of the whitening (rows P, K Q), 8 slices
    PhaseScope ph3(3, s2);
    oz_alloc(Linv8, 1, h->wfmt, np, np, OZ_BN);
    oz_slice_f64(h->Linv.p, 0, np, 1, Linv8, s2);
  }
  DFJK_CUDA_CHECK(cudaEventRecord(h->ev_join, s2));


  // a0: shell pairs, primitive-pair records, Schwarz factors
  enumerate_pairs(h);
  const int npair = h->cls_begin[6];
  std::vector<long long> rec_off(npair);
  long long tot = 0, rec_cls[7];
  static const int cls[6][2] = {{0, 0}, {1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
  for (int c = 0; c < 6; ++c) {
    rec_cls[c] = tot;
    for (int i = h->cls_begin[c]; i < h->cls_begin[c + 1]; ++i) {
      rec_off[i] = tot;
      tot += (long long)h->npp_h[i] * pair_record_len(cls[c][0], cls[c][1]);
    }
  }
  rec_cls[6] = tot;
  h->pair_a.upload(h->pa_h, st);
  h->pair_b.upload(h->pb_h, st);
  h->pair_npp.upload(h->npp_h, st);
  h->pair_rec_off.upload(rec_off, st);
  h->rec.alloc((size_t)std::max<long long>(tot, 1));
  h->q.alloc(std::max(npair, 1));
  for (int c = 0; c < 6; ++c) {
    const int b0 = h->cls_begin[c], n = h->cls_begin[c + 1] - b0;
    PairClassArgs a{n, h->pair_a.p + b0, h->pair_b.p + b0, h->pair_rec_off.p + b0, h->rec.p, h->q.p + b0,
                    h->pair_npp.p + b0};
    launch_pair_kernel(cls[c][0], cls[c][1], a, orb_args(h), tab, st);
    launch_schwarz(cls[c][0], cls[c][1], a, tab, tab32, h->df_range, st);
  }
  h->scal.alloc(1);
  max_sqrt_diag(h->V.p, h->naux, np, h->scal.p, st);
  h->pair_keep.alloc(std::max(npair, 1));
  screen_pairs(h->q.p, npair, h->scal.p, h->opt.schwarz_thresh, h->pair_keep.p, st);
  delete ph0;
  std::vector<int> keep(npair);
  std::vector<double> qh(npair);
  double scal = 0.0;
  if (npair) {
    DFJK_CUDA_CHECK(cudaMemcpyAsync(keep.data(), h->pair_keep.p, npair * sizeof(int), cudaMemcpyDeviceToHost, st));
    DFJK_CUDA_CHECK(cudaMemcpyAsync(qh.data(), h->q.p, npair * sizeof(double), cudaMemcpyDeviceToHost, st));
  }
  DFJK_CUDA_CHECK(cudaMemcpyAsync(&scal, h->scal.p, sizeof(double), cudaMemcpyDeviceToHost, st));
  DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
  // Schwarz-guided precision: kept pairs with bound below thr32 go to the FP32
  // kernels; within each class the FP64 pairs come first
  const double thr32 = h->opt.fp32_pair_thresh >= 0.0 ? h->opt.fp32_pair_thresh
                       : (h->opt.precision == DFJK_MIXED ? 1e-5 : 0.0);
  h->fp32_thresh = thr32;

  // kept list, columns, column -> (mu, nu) map (host bookkeeping)
  h->kept_h.clear();
  h->kept_cls_begin.assign(7, 0);
  h->pair_col_h.assign(npair, -1);
  std::vector<int> cmu, cnu;
  long long col = 0;
  h->kept32_begin.assign(6, 0);
  h->npair_fp32 = 0;
  for (int c = 0; c < 6; ++c) {
    h->kept_cls_begin[c] = (int)h->kept_h.size();
    const int na = ncart(cls[c][0]), nb = ncart(cls[c][1]);
    std::vector<int> order;
    for (int i = h->cls_begin[c]; i < h->cls_begin[c + 1]; ++i)
      if (keep[i] && !(qh[i] * scal < thr32)) order.push_back(i);
    h->kept32_begin[c] = h->kept_cls_begin[c] + (int)order.size();
    for (int i = h->cls_begin[c]; i < h->cls_begin[c + 1]; ++i)
      if (keep[i] && qh[i] * scal < thr32) order.push_back(i);
    h->npair_fp32 += h->kept_cls_begin[c] + (int)order.size() - h->kept32_begin[c];
    for (int i : order) {
      h->kept_h.push_back(i);
      h->pair_col_h[i] = col;
      const int sa = h->pa_h[i], sb = h->pb_h[i];
      for (int ca = 0; ca < na; ++ca)
        for (int cb = 0; cb < nb; ++cb) {
          const bool dup = (sa == sb) && (ca < cb);
          cmu.push_back(dup ? -1 : h->orb.func_off[sa] + ca);
          cnu.push_back(dup ? -1 : h->orb.func_off[sb] + cb);
        }
      col += na * nb;
    }
  }
  h->kept_cls_begin[6] = (int)h->kept_h.size();
  for (int c = 0; c < 6; ++c) {  // primitive pairs per class and precision
    h->prim_pairs64[c] = h->prim_pairs32[c] = 0;
    for (int i = h->kept_cls_begin[c]; i < h->kept_cls_begin[c + 1]; ++i)
      (i < h->kept32_begin[c] ? h->prim_pairs64 : h->prim_pairs32)[c] += h->npp_h[h->kept_h[i]];
  }
  h->npair_kept = (int)h->kept_h.size();
  h->ncol = col;
  h->kept.upload(h->kept_h, st);
  h->pair_col.upload(h->pair_col_h, st);
  h->colmu.upload(cmu, st);
  h->colnu.upload(cnu, st);
  if (mixed) {
    h->rowmap.alloc((size_t)h->nao * h->nao);
    build_rowmap(h->colmu.p, h->colnu.p, h->ncol, h->nao, h->rowmap.p, st);
  }

  bool joined = false;

  // a4 + a5: 3-centre integrals in column slabs, whitened into B
  // mixed: one row per kept column (the whitening writes every row); FP64:
  // both triangles of every AO pair, zero for the screened ones
  h->ldb = np;
  h->lean = mixed;
  h->B.alloc((h->lean ? (size_t)std::max<long long>(h->ncol, 1) : (size_t)h->nao * h->nao) * np,
             h->opt.b_on_host != 0);
  if (!h->lean) DFJK_CUDA_CHECK(cudaMemsetAsync(h->B.p, 0, h->B.bytes(), st));
  // bytes of one T slab: 4 GiB, or 2 GiB with sliced products, whose slab also
  // has an 8-slice copy (twice the bytes) during the whitening
  const long long slab_budget = h->sliced ? (2LL << 30) : (4LL << 30);
  long long slab_cols = std::max<long long>(36, slab_budget / ((long long)np * 8));
  slab_cols = std::min<long long>(slab_cols, std::max<long long>(h->ncol, 1));
  T.alloc((size_t)slab_cols * np);
  DFJK_CUDA_CHECK(cudaMemsetAsync(T.p, 0, T.bytes(), st));
  if (h->use_df || h->npair_fp32 > 0) {
    h->recd.alloc((size_t)std::max<long long>(tot, 1));
    convert_records(h->rec.p, rec_cls, h->c0, h->recd.p, st);
  }
  int r0 = 0;
  h->nslab = 0;
  while (r0 < h->npair_kept) {
    ++h->nslab;
    const long long c0 = h->pair_col_h[h->kept_h[r0]];
    int r1 = r0;
    while (r1 < h->npair_kept) {
      const int g = h->kept_h[r1];
      const int c = [&] { int k = 0; while (g >= h->cls_begin[k + 1]) ++k; return k; }();
      const long long cend = h->pair_col_h[g] + ncart(cls[c][0]) * ncart(cls[c][1]);
      if (cend - c0 > slab_cols) break;
      ++r1;
    }
    const long long c1 = (r1 < h->npair_kept) ? h->pair_col_h[h->kept_h[r1]] : h->ncol;
    // the FP32 pairs of every class on one stream, the others spread over three
    // (phase timers 11 and 2)
    {
      PhaseScope ph2(2, st);
      const IntegralFork fork(st, h->ev_int);
      const cudaStream_t *is = fork.is;
      PhaseScope ph11(11, is[INT_STREAMS - 1]);
      for (int prec32 = 0; prec32 < 2; ++prec32)
        for (int c = 5; c >= 0; --c) {  // the largest classes first
          const int lo = std::max(r0, h->kept_cls_begin[c]), hi = std::min(r1, h->kept_cls_begin[c + 1]);
          if (hi <= lo) continue;
          const int mid = std::min(std::max(lo, h->kept32_begin[c]), hi);  // [lo, mid) FP64, [mid, hi) FP32
          for (int lc = 2; lc >= 0; --lc)
            launch_integrals(h, c, lc, h->kept.p + (prec32 ? mid : lo), prec32 ? hi - mid : mid - lo, prec32 != 0, T.p, c0,
                             tables, is[prec32 ? INT_STREAMS - 1 : (c + lc) % (INT_STREAMS - 1)]);
        }
    }
    if (h->sliced && r0 == 0) make_pair_lists(h);  // on the host, while the device works on the integrals
    PhaseScope ph3(3, st);
    const int ncols = (int)(c1 - c0);
    if (h->sliced) {  // slices of T need only T: taken before waiting for L^-1
      if (!T8.data) oz_alloc(T8, 1, h->wfmt, (int)slab_cols, np, OZ_BM);
      SlicedOp t8 = oz_view(T8, ncols, np);
      if (h->use_df) oz_slice_df((const float2 *)T.p, np, t8, st, h->tune.slice_rows);
      else oz_slice_f64(T.p, 0, np, 1, t8, st, h->tune.slice_rows);
    }
    if (!joined) {  // L^-1 (and its slices) ready
      DFJK_CUDA_CHECK(cudaStreamWaitEvent(st, h->ev_join, 0));
      joined = true;
    }
    if (!h->sliced) {
      GemmArgs g;  // B[(mu,nu)][P] = sum_Q T[col][Q] Linv[P][Q]
      g.M = (int)(c1 - c0); g.N = np; g.K = np;
      g.A = T.p; g.sAm = np; g.sAk = 1;
      g.B = h->Linv.p; g.sBn = np; g.sBk = 1;
      g.k_upto_n = 1;
      g.colmu = h->colmu.p + c0; g.colnu = h->colnu.p + c0;
      g.nao = h->nao; g.ldo = h->ldb; g.out = h->B.p;
      gemm_f64(g, st);
    } else {  // the same product on the tensor cores, 8 slices per operand
      OzGemmArgs g;  // lean: B row c0 + m = whitened column c0 + m
      g.M = ncols; g.N = np; g.K = np; g.k_upto_n = 1;
      g.ldo = h->ldb;
      if (h->lean) {
        g.mode = 0; g.out = h->B.p + c0 * h->ldb;
      } else {  // both triangles of every pair
        g.mode = 1; g.out = h->B.p; g.colmu = h->colmu.p + c0; g.colnu = h->colnu.p + c0; g.nao = h->nao;
      }
      g.status = h->status.p; g.timeout = h->opt.timeout_iters;
      g.tile_ctr = h->tctr.p;
      g.phase = 8;
      oz_gemm(oz_view(T8, ncols, np), Linv8, g, st);
    }
    r0 = r1;
  }
  if (!joined) DFJK_CUDA_CHECK(cudaStreamWaitEvent(st, h->ev_join, 0));
  if (h->sliced) {
    // the partner lists, and the slice exponents of B (per mu, P and K block of
    // mu's list), which do not change between builds
    if (h->npair_kept == 0) make_pair_lists(h);
    upload_pair_lists(h, st);
    PhaseScope ph(3, st);
    const int nkb = h->pl.nkb;
    h->expo_rows = (np + OZ_BM - 1) / OZ_BM * OZ_BM;
    h->Bexpo.alloc((size_t)h->nao * h->expo_rows * nkb);
    if (!h->B.host) {
      oz_expo_pairs(h->B.p, h->ldb, np, h->pl, h->nao, h->expo_rows, 0, h->expo_rows, h->Bexpo.p, st);
    } else {  // in chunks of columns, each copied to the device once
      stage.alloc(stage_size(h, std::min(512, np)));
      for (int p0 = 0; p0 < h->expo_rows; p0 += 512) {
        const int pc = std::min(512, h->expo_rows - p0), live = std::max(0, std::min(pc, np - p0));
        if (live > 0) stage_columns(h, stage, p0, live, st);
        oz_expo_pairs(stage.p, live, live, h->pl, h->nao, pc, p0, h->expo_rows, h->Bexpo.p, st);
      }
    }
    DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    oz_free(T8);
    oz_free(Linv8);
  }
  int status = 0;
  DFJK_CUDA_CHECK(cudaMemcpyAsync(&status, h->status.p, sizeof(int), cudaMemcpyDeviceToHost, st));
  DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
  if (status & STATUS_NOT_PD)
    throw Error{DFJK_ERR_NOT_PD, "(P|Q) metric is not positive definite (non-positive Cholesky pivot)"};
  if (status & STATUS_TIMEOUT) throw Error{DFJK_ERR_TIMEOUT, "a bounded device wait expired during setup"};
  h->resident = true;
}

void release_device(dfjk_ctx *h) {
  h->B.release();
  h->Bexpo.release();
  h->rowmap.release();
  h->pl = PairLists();
  h->pl_buf.release();
  h->pl_krow.release();
  h->xw.release();
  h->b_stage.release();
  h->V.release();
  h->L.release();
  h->Linv.release();
  h->Dinv.release();
  h->rec.release();
  h->recd.release();
  h->q.release();
  h->colmu.release();
  h->colnu.release();
  h->D.release();
  h->rho.release();
  h->rho_work.release();
  h->X.release();
  h->Kpart.release();
  h->kw.release();
  h->en_work.release();
  h->e.release();
  oz_free(h->Xsl);
  h->chunk_rows = 0;
  h->uks_D.release();
  h->uks_J.release();
  h->ws_nocc = -1;
  h->resident = false;
}

// The cap on a build's work buffers.
size_t build_ws_bytes(int ws_mb) {
  static const size_t cap_env = [] {
    const char *e = std::getenv("DFJK_BUILD_WS_MB");
    const long v = e ? std::atol(e) : 0;
    return (size_t)(v > 0 ? v : 8192) << 20;
  }();
  return ws_mb > 0 ? (size_t)ws_mb << 20 : cap_env;
}
// Bytes that a row P of a chunk takes: X in FP64 and its slices, the slices of B's
// kept pairs (`steps` K steps of 16 over all AOs).
size_t chunk_row_bytes(int nao, int nocc, int fmt, long long steps) {
  const size_t rp = ((size_t)nao + OZ_BM - 1) / OZ_BM * OZ_BM;
  const size_t el = 2 * (size_t)oz_slices(fmt);  // bytes of an element's slices
  return (size_t)nao * nocc * 8 + rp * nocc * el + (size_t)steps * OZ_BK * el;
}
// Rows P per chunk of the build: the largest multiple of 128 whose work buffers stay
// within DFJK_BUILD_WS_MB megabytes (default 8192), at least 128, at most the whole
// (padded) aux range.
int build_chunk_rows(int nao, int np, int nocc, int fmt, long long steps, int ws_mb = 0) {
  size_t rows = std::max<size_t>(128, build_ws_bytes(ws_mb) / chunk_row_bytes(nao, nocc, fmt, steps) / 128 * 128);
  return (int)std::min<size_t>(rows, (size_t)np);
}

// Bytes of one K step of C's slices (rows padded to whole tiles).
size_t c_step_bytes(int fmt, int nocc) {
  return (size_t)ceil_div(nocc, OZ_BN) * OZ_BN * oz_slices(fmt) * OZ_BK * sizeof(__nv_bfloat16);
}

void alloc_xwork(dfjk_ctx *h, const PairLists &pl, XWork &w, int pc, int nocc) {
  const size_t step = c_step_bytes(pl.fmt, nocc);
  w.b_ready = false;
  w.bsl.alloc(oz_pairs_bytes(pl.fmt, pl.steps, pc) / sizeof(__nv_bfloat16));
  w.range.assign(1, 0);
  size_t most = 0, most_g = 0;
  for (int g = 0; g < pl.ngroup;) {
    int e = g + 1;
    while (e < pl.ngroup && (h->gstep_h[e + 1] - h->gstep_h[g]) * step <= C_SLICE_CAP) ++e;
    most = std::max(most, (h->gstep_h[e] - h->gstep_h[g]) * step);
    most_g = std::max<size_t>(most_g, e - g);
    w.range.push_back(e);
    g = e;
  }
  w.cdat.alloc(most / sizeof(__nv_bfloat16));
  w.cexp.alloc(most_g * ceil_div(nocc, OZ_BN) * OZ_BN * pl.nkb);
}

// X[mu][p][i] = sum_nu B[(mu, nu)][p0 + p] C[nu][i] for p < pc over the kept pairs, on
// the tensor cores: out[mu obs + p ldo + i], or out[mu obs + i ldo + p] (mode 3).
// `b`, `ldb`: B's columns from p0 on; `expo`: their exponents (all rows P).
// `first`: C has not been sliced yet for this build.
struct XArgs {
  const double *b;
  long long ldb;
  const double *C;  // C[nu][i] = C[nu ldc + i ldi]
  long long ldc, ldi;
  int nocc, p0, pc;
  double *out;
  long long ldo, obs;
  int mode;
  bool first;
  bool keep_b = false;  // B's slices of these rows are in place already
  int *status = nullptr;  // status word of the call (null: the handle's)
};
void x_gemm_sliced(dfjk_ctx *h, const PairLists &pl, const int *expo, XWork &w, const XArgs &a, cudaStream_t st) {
  const int nao = h->nao;
  SlicedOp A, c;
  A.data = w.bsl.p;
  A.expo = const_cast<int *>(expo) + (long long)a.p0 * pl.nkb;
  A.row_tile = OZ_BM;
  A.rows = a.pc;
  A.rows_pad = h->expo_rows;
  A.batch = nao;
  c.data = w.cdat.p;
  c.expo = w.cexp.p;
  c.row_tile = OZ_BN;
  c.rows = a.nocc;
  c.rows_pad = ceil_div(a.nocc, OZ_BN) * OZ_BN;
  for (SlicedOp *o : {&A, &c}) {
    o->fmt = pl.fmt;
    o->S = oz_slices(pl.fmt);
    o->nkb = pl.nkb;
  }
  if (!a.keep_b) oz_slice_pairs(a.b, a.ldb, a.pc, pl, nao, A.expo, h->expo_rows, w.bsl.p, st, h->tune.pslice_rows);
  const int nr = (int)w.range.size() - 1;
  for (int r = 0; r < nr; ++r) {
    const int g0 = w.range[r], g1 = w.range[r + 1];
    if (a.first || nr > 1) oz_slice_c(a.C, a.ldc, a.ldi, a.nocc, pl, g0, g1, c, st);
    OzGemmArgs x;
    x.M = a.pc; x.N = a.nocc;
    x.z0 = h->gfirst_h[g0]; x.nz = h->gfirst_h[g1] - x.z0; x.g0 = g0;
    x.zstep = pl.zstep; x.zgroup = pl.zgroup; x.gstep = pl.gstep;
    x.mode = a.mode; x.out = a.out; x.ldo = a.ldo; x.out_bs = a.obs;
    x.status = a.status ? a.status : h->status.p; x.timeout = h->opt.timeout_iters;
    x.tile_ctr = h->tctr.p;
    x.phase = 9;
    oz_gemm(A, c, x, st);
  }
}

size_t k_range_bytes(int range_mb) {
  static const size_t env = [] {
    const char *e = std::getenv("DFJK_K_RANGE_MB");
    const long v = e ? std::atol(e) : 0;
    return (size_t)(v > 0 ? v : 64) << 20;
  }();
  return range_mb > 0 ? (size_t)range_mb << 20 : env;
}

// The K GEMM of operands with nao rows in format fmt.
KShape k_shape(int nao, int fmt, int range_mb) {
  KShape s;
  s.nao = nao;
  s.tiles = k_tiles(nao, OZ_BM, OZ_BN);
  s.block_bytes = (size_t)ceil_div(nao, OZ_BM) * OZ_BM * oz_slices(fmt) * 2 * oz_kblock(fmt);
  s.range_bytes = k_range_bytes(range_mb);
  s.ordered = !oz_simple_mode();
  return s;
}

void alloc_kwork(KWork &w, const KShape &s, int fmt, long long kt) {
  w.part.alloc(k_part_doubles(s, ceil_div(kt, oz_kblock(fmt))));
  w.seq.alloc(oz_tile_seq_count(s.nao, s.nao));
}

// Build buffers, sized on the first build at a given nocc and reused after.
void ensure_workspace(dfjk_ctx *h, int nocc, int nset) {
  const size_t nao2 = (size_t)h->nao * h->nao;
  if (h->ws_nocc < nocc || !h->D.p) {
    h->D.alloc(nao2);
    h->rho.alloc(h->naux_pad);
    if (h->sliced) {
      const int pc = build_chunk_rows(h->nao, h->naux_pad, nocc, h->bfmt, h->pl.steps, h->tune.build_ws_mb);
      h->chunk_rows = pc;
      h->X.alloc((size_t)h->nao * pc * nocc);
      h->rho_work.alloc((size_t)RHO_PARTS * h->naux_pad);
      oz_alloc(h->Xsl, 1, h->bfmt, h->nao, pc * nocc, OZ_BM);
      alloc_xwork(h, h->pl, h->xw, pc, nocc);
      if (h->B.host) h->b_stage.alloc(stage_size(h, pc));
      alloc_kwork(h->kw, k_shape(h->nao, h->bfmt, h->tune.k_range_mb), h->bfmt, (long long)pc * nocc);
    } else {
      h->rho_work.alloc(std::max((size_t)128 * ceil_div(h->naux_pad, 256) * 256, (size_t)h->nao * h->naux_pad));
      h->X.alloc((size_t)h->nao * h->naux_pad * nocc);
      const int t = ceil_div(h->nao, 64);
      const int tiles = t * (t + 1) / 2;
      h->ksplit = std::max(1, std::min(64, ceil_div(4 * 152, tiles)));
      h->Kpart.alloc(nao2 * h->ksplit);
    }
    h->en_work.alloc(2 * 256);
    h->ws_nocc = nocc;
  }
  if (!h->e.p || h->e.n < (size_t)(2 * nset)) h->e.alloc(2 * nset);
}

// After the stream of a call has been synchronised: an expired bounded wait left part of
// its results unwritten.  The status bit is cleared, so that the next call starts afresh.
void throw_on_timeout(dfjk_ctx *h, int status, const char *what) {
  if (status & STATUS_TIMEOUT) {
    DFJK_CUDA_CHECK(cudaMemset(h->status.p, 0, sizeof(int)));
    throw Error{DFJK_ERR_TIMEOUT, std::string("a bounded device wait expired during the ") + what};
  }
}

void throw_on_timeout(dfjk_ctx *h, const char *what) {
  int status = 0;
  DFJK_CUDA_CHECK(cudaMemcpy(&status, h->status.p, sizeof(int), cudaMemcpyDeviceToHost));
  throw_on_timeout(h, status, what);
}

__global__ void split_energies_kernel(const double *e, int nset, double *EJ, double *EK) {
  const int s = threadIdx.x + blockIdx.x * blockDim.x;
  if (s < nset) {
    EJ[s] = e[2 * s];
    EK[s] = e[2 * s + 1];
  }
}

// y += x over n doubles (the sum of the two spin densities and of their J).
__global__ void add_inplace_kernel(double *__restrict__ y, const double *__restrict__ x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] += x[i];
}

void add_inplace(double *y, const double *x, long long n, cudaStream_t st) {
  add_inplace_kernel<<<(unsigned)std::min<long long>(ceil_div(n, 256), 152 * 8), 256, 0, st>>>(y, x, n);
  DFJK_LAUNCHED();
}

// K (lower triangle) += Xs Ys^T for one chunk of the reduction range (K
// dimension kt = rows P of the chunk x nocc; Ys = Xs but for the density build),
// on the tensor cores.  Split-K
// ranges of about 64 MB of operand slices (all rows): the tiles in flight
// (work is handed out split-major, a few ranges at a time) then reuse their
// operands from L2.  The splits of a tile are summed in split order either way
// (`add`: after the previous chunks' sum): the persistent kernel adds them into K
// one after the other, each waiting for the one before, without partial buffers;
// while the partials of all splits take at most K_PART_BYTES they are written out
// and reduced by a second kernel, because a small K has few tiles, hence many
// splits per tile, and the chain of adds (about 3 us each) was longer than the
// products (an FP64 density build at 8 atoms 3.95 -> 0.77 ms, a build at 5 atoms 331
// -> 226 us).  The one-tile-per-CTA kernel always writes partials.
// `w`: from alloc_kwork for at least this range.
void k_gemm_sliced(dfjk_ctx *h, KWork &w, const SlicedOp &xs, const SlicedOp &ys, int nao, long long kt, double *Kout,
                   bool add, int *status, cudaStream_t st) {
  const KShape s = k_shape(nao, xs.fmt, h->tune.k_range_mb);
  const KSplit p = k_split(s, xs.nkb);
  if (p.partials ? w.part.n < (size_t)p.n * nao * nao : w.seq.n < oz_tile_seq_count(nao, nao))
    throw Error{DFJK_ERR_STATE, "K work buffers"};
  OzGemmArgs k;
  k.M = nao; k.N = nao; k.K = (int)kt; k.nz = p.n; k.kb_per_split = p.per; k.lower_only = 1;
  k.status = status; k.timeout = h->opt.timeout_iters;
  k.tile_ctr = h->tctr.p;
  k.phase = 10;
  if (!p.partials) {
    k.mode = 2; k.out = Kout; k.ldo = nao; k.tile_seq = w.seq.p; k.accumulate = add ? 1 : 0;
    oz_gemm(xs, ys, k, st);
  } else {
    k.mode = 0; k.out = w.part.p; k.ldo = nao; k.out_bs = (long long)nao * nao;
    oz_gemm(xs, ys, k, st);
    reduce_sym_f64(w.part.p, p.n, nao, Kout, st, add ? 1 : 0);
  }
}

// The build for one occupied set.  X = B C and K run on the tensor cores as exact
// sliced products (DFJK_MIXED: 36 bits, DFJK_FP64: 56 bits), or, for the small
// molecules of DFJK_FP64, on the FP64 pipe; D, rho, J and the energies are FP64.
void build_one(dfjk_ctx *h, int nocc, const double *C, double *J, double *Kout, double *e,
               cudaStream_t st) {
  const int nao = h->nao, np = h->naux_pad;
  // D, rho and J beside the tensor-core GEMMs, on the handle's side stream: they need
  // C and B only (rho = B vec D over the kept rows of B)
  const cudaStream_t sj = h->sliced && h->side ? h->side : st;
  SideScope side(st, sj, h->ev_fork, h->ev_join);
  side.fork();
  GemmArgs d;  // D = C C^T
  d.M = nao; d.N = nao; d.K = nocc;
  d.A = C; d.sAm = nocc; d.sAk = 1;
  d.B = C; d.sBn = nocc; d.sBk = 1;
  d.C = h->D.p; d.sCm = nao; d.sCn = 1;
  d.tile = 32;  // latency-bound: a 64 x 64 tile's K loop took 195 us at 272 functions
  {
    PhaseScope ph(6, sj);
    gemm_f64(d, sj);
  }
  const long long kt = (long long)np * nocc;
  if (!h->sliced) {
    GemmArgs x;  // X[mu][P][i] = sum_nu B[(mu,nu)][P] C[nu][i]
    x.M = np; x.N = nocc; x.K = nao; x.batch = nao;
    x.A = h->B.p; x.sAm = 1; x.sAk = h->ldb; x.sAb = (long long)nao * h->ldb;
    x.B = C; x.sBn = 1; x.sBk = nocc; x.sBb = 0;
    x.C = h->X.p; x.sCm = nocc; x.sCn = 1; x.sCb = (long long)np * nocc;
    {
      PhaseScope ph(4, st);
      gemm_f64(x, st);
    }
    {  // rho from X (5x smaller than B), then J over B
      PhaseScope ph(6, st);
      rho_from_x_f64(h->X.p, C, nao, np, nocc, h->rho.p, h->rho_work.p, st);
      j_gemv_f64(h->B.p, h->ldb, nao, np, h->rho.p, J, st);
    }
    GemmArgs k;  // K[mu][nu] = sum_(P,i) X[mu][(P,i)] X[nu][(P,i)]
    k.M = nao; k.N = nao; k.K = (int)kt;
    k.A = h->X.p; k.sAm = kt; k.sAk = 1;
    k.B = h->X.p; k.sBn = kt; k.sBk = 1;
    k.C = h->Kpart.p; k.sCm = nao; k.sCn = 1; k.sCb = (long long)nao * nao;
    k.k_split = (int)((kt + h->ksplit - 1) / h->ksplit);
    k.k_split = ((k.k_split + 15) / 16) * 16;
    k.lower_only = 1;
    PhaseScope ph(5, st);
    gemm_f64(k, st);
    reduce_sym_f64(h->Kpart.p, ceil_div(kt, k.k_split), nao, Kout, st);
  } else {
    // Works through the aux index in chunks of rows P: per chunk, the slices of B's kept pairs,
    // X_P = B_P C for P in the chunk, the slices of X and its contribution to K
    // (added in chunk order).  One chunk holds the whole aux range unless the
    // build's work buffers would exceed the workspace cap.
    const auto rho_of = [&](const double *b, long long ldb, int p0, int pc, cudaStream_t s) {
      PhaseScope ph(6, s);
      rho_kept(h, b, ldb, h->D.p, pc, h->rho.p + p0, h->rho_work.p, s);
    };
    const auto j_of = [&](cudaStream_t s) {
      PhaseScope ph(6, s);
      j_kept(h, h->rho.p, J, s);
    };
    if (!h->B.host) {
      rho_of(h->B.p, h->ldb, 0, np, sj);
      j_of(sj);
    }
    if (h->B.host) side.join();  // D ready
    const int pc_max = h->chunk_rows;
    const int nchunk = ceil_div(np, pc_max);
    // B does not change after setup: with one chunk its slices stay in the work
    // buffer from build to build (the second spin of an unrestricted build included).
    // A captured build slices B itself, so that a replay stands alone.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    DFJK_CUDA_CHECK(cudaStreamIsCapturing(st, &cap));
    const bool keep = nchunk == 1 && !h->B.host && cap == cudaStreamCaptureStatusNone;
    const bool keep_b = keep && h->xw.b_ready;
    h->xw.b_ready = false;
    for (int c = 0; c < nchunk; ++c) {
      const int p0 = c * pc_max, pc = std::min(pc_max, np - p0);
      const long long kt = (long long)pc * nocc;  // K of the K GEMM: (P, i) of the chunk, P-major
      double *Xc = h->X.p;                        // X[mu][p][i] of this chunk
      const double *b = h->B.p + p0;
      long long ldb = h->ldb;
      if (h->B.host) {  // one copy of the chunk's columns; rho of the chunk from it
        b = stage_columns(h, h->b_stage, p0, pc, st);
        ldb = pc;
        rho_of(b, ldb, p0, pc, st);
      }
      {
        PhaseScope ph(4, st);
        x_gemm_sliced(h, h->pl, h->Bexpo.p, h->xw, XArgs{b, ldb, C, nocc, 1, nocc, p0, pc, Xc, nocc, kt, 0, c == 0, keep_b}, st);
      }
      h->xw.b_ready = keep;
      if (h->B.host && c == nchunk - 1) {  // J beside the last K GEMM
        side.fork();
        j_of(sj);
      }
      PhaseScope ph(5, st);
      SlicedOp xs = oz_view(h->Xsl, nao, (int)kt);  // rows mu, K (p, i)
      oz_slice_f64(Xc, 0, kt, 1, xs, st, h->tune.slice_rows);
      k_gemm_sliced(h, h->kw, xs, xs, nao, kt, Kout, c > 0, h->status.p, st);
    }
    mirror_lower_f64(Kout, nao, st);
    side.join();  // D and J ready
  }
  PhaseScope ph(7, st);
  energies_f64(h->D.p, J, Kout, nao, e, h->en_work.p, st);
}

// Buffers of the density build, for the duration of a call.
struct DensityWork {
  bool sliced = false;
  const double *Bf = nullptr;  // B with both triangles of every pair
  DBuf<double> Bfull, W, Kpart, stage, e;
  int ksplit = 1;
  // sliced: X for a range of sigma, the slices of X and B, the lists and exponents
  PairLists pl;
  DBuf<int> expo_own;
  const int *expo = nullptr;
  XWork xw;
  KWork kw;
  SlicedOp xs, bs;
  int ns = 0, pc = 0;  // sigma and rows P per chunk
  int *status = nullptr;  // the call's own status word, behind the energies
  ~DensityWork() {
    oz_free(xs);
    oz_free(bs);
  }
};

void density_work(dfjk_ctx *h, DensityWork &w, cudaStream_t st) {
  const int nao = h->nao, np = h->naux_pad;
  const size_t nao2 = (size_t)nao * nao;
  // a B of kept rows only is expanded into a temporary copy
  w.Bf = h->B.p;
  if (h->lean) {
    w.Bfull.alloc(nao2 * h->ldb);
    unpack_rows_f64(h->B.p, h->ldb, nao, h->rowmap.p, w.Bfull.p, st);
    w.Bf = w.Bfull.p;
  }
  w.sliced = use_slices(DFJK_FP64, nao, np);
  if (!w.sliced) {
    const int t = ceil_div(nao, 64);
    w.ksplit = std::max(1, std::min(64, ceil_div(4 * 152, t * (t + 1) / 2)));
    w.Kpart.alloc(nao2 * w.ksplit);
    w.W.alloc(nao2 * h->ldb);  // W[mu][sigma][P] = sum_lambda D[sigma][lambda] B[mu][lambda][P]
    return;
  }
  w.pl = h->pl;
  w.expo = h->Bexpo.p;
  if (w.pl.fmt != OZ_F64) {  // a mixed handle's exponents belong to its own K blocks
    w.pl.fmt = OZ_F64;
    w.pl.nkb = ceil_div(w.pl.longest, oz_kblock(OZ_F64));
    w.expo_own.alloc((size_t)nao * h->expo_rows * w.pl.nkb);
    w.expo = w.expo_own.p;
    oz_expo_pairs(h->B.p, h->ldb, np, w.pl, nao, h->expo_rows, 0, h->expo_rows, w.expo_own.p, st);
  }
  // ranges of sigma whose X and slices of X and B stay near the build's cap
  const size_t rp = (size_t)ceil_div(nao, OZ_BM) * OZ_BM, cap = (size_t)8 << 30;
  const size_t per = np * ((size_t)nao * 8 + 2 * rp * 16);
  w.ns = (int)std::min<size_t>(nao, std::max<size_t>(64, cap / per / 64 * 64));
  w.pc = build_chunk_rows(nao, np, 1, OZ_F64, w.pl.steps);
  w.W.alloc((size_t)nao * w.ns * np);
  oz_alloc(w.xs, 1, OZ_F64, nao, w.ns * np, OZ_BM);
  oz_alloc(w.bs, 1, OZ_F64, nao, w.ns * np, OZ_BM);
  alloc_xwork(h, w.pl, w.xw, w.pc, w.ns);
  if (h->B.host) w.stage.alloc(stage_size(h, w.pc));
  alloc_kwork(w.kw, k_shape(nao, OZ_F64, h->tune.k_range_mb), OZ_F64, (long long)w.ns * np);
}

// K = sum_P B_P D B_P on the tensor cores, for ranges of sigma: W[mu][sigma][P] =
// sum_nu B[(mu, nu)][P] D[sigma][nu] over the kept pairs, then K += W B^T over
// (sigma, P).
// `again`: not the first density of the call, whose slices of B still serve when one
// range holds them.
void density_k_sliced(dfjk_ctx *h, DensityWork &w, const double *D, double *Kout, bool again, cudaStream_t st) {
  const int nao = h->nao, np = h->naux_pad;
  const bool keep_a = again && w.pc >= np, keep_b = again && w.ns >= nao;
  for (int s0 = 0; s0 < nao; s0 += w.ns) {
    const int ns = std::min(w.ns, nao - s0);
    const long long kt = (long long)ns * np;
    {
      PhaseScope ph(4, st);
      for (int p0 = 0; p0 < np; p0 += w.pc) {
        const int pc = std::min(w.pc, np - p0);
        const double *b = h->B.p + p0;
        if (h->B.host && !keep_a) b = stage_columns(h, w.stage, p0, pc, st);
        x_gemm_sliced(h, w.pl, w.expo, w.xw,
                      XArgs{b, h->B.host ? pc : h->ldb, D + (long long)s0 * nao, 1, nao, ns, p0, pc, w.W.p + p0, np, kt, 3,
                            p0 == 0, keep_a || (w.pc >= np && s0 > 0), w.status},
                      st);
      }
    }
    PhaseScope ph(5, st);
    SlicedOp xs = oz_view(w.xs, nao, (int)kt), bs = oz_view(w.bs, nao, (int)kt);
    oz_slice_f64(w.W.p, 0, kt, 1, xs, st, h->tune.slice_rows);
    if (!keep_b)
      oz_slice_f64(w.Bf + (long long)s0 * h->ldb, 0, (long long)nao * h->ldb, 1, bs, st, h->tune.slice_rows);
    k_gemm_sliced(h, w.kw, xs, bs, nao, kt, Kout, s0 > 0, w.status, st);
  }
  mirror_lower_f64(Kout, nao, st);
}

// The same on the FP64 pipe (small molecules).
void density_k_f64(dfjk_ctx *h, DensityWork &dw, const double *D, double *Kout, cudaStream_t st) {
  const int nao = h->nao, np = h->naux_pad;
  const long long kt = (long long)nao * h->ldb;
  {
    PhaseScope ph(4, st);
    GemmArgs w;  // batch mu: W_mu (sigma x P) = D (sigma x lambda) B_mu (lambda x P)
    w.M = nao; w.N = np; w.K = nao; w.batch = nao;
    w.A = D; w.sAm = nao; w.sAk = 1; w.sAb = 0;
    w.B = dw.Bf; w.sBn = 1; w.sBk = h->ldb; w.sBb = (long long)nao * h->ldb;
    w.C = dw.W.p; w.sCm = h->ldb; w.sCn = 1; w.sCb = (long long)nao * h->ldb;
    gemm_f64(w, st);
  }
  PhaseScope ph(5, st);
  GemmArgs k;  // K[mu][nu] = sum_(sigma,P) W[mu][(sigma,P)] B[nu][(sigma,P)]
  k.M = nao; k.N = nao; k.K = (int)kt;
  k.A = dw.W.p; k.sAm = kt; k.sAk = 1;
  k.B = dw.Bf; k.sBn = kt; k.sBk = 1;
  k.C = dw.Kpart.p; k.sCm = nao; k.sCn = 1; k.sCb = (long long)nao * nao;
  k.k_split = (int)((kt + dw.ksplit - 1) / dw.ksplit);
  k.k_split = ((k.k_split + 15) / 16) * 16;
  k.lower_only = 1;
  gemm_f64(k, st);
  reduce_sym_f64(dw.Kpart.p, ceil_div(kt, k.k_split), nao, Kout, st);
}

}  // namespace

extern "C" {

void dfjk_default_options(dfjk_options *opt) {
  if (!opt) return;
  opt->precision = DFJK_FP64;
  opt->schwarz_thresh = 1e-12;
  opt->hbm_budget_bytes = 0;
  opt->timeout_iters = 1LL << 26;
  opt->energies_on_host = 1;
  opt->fp32_pair_thresh = -1.0;
  opt->b_on_host = 0;
  opt->tune_table = nullptr;
}

const char *dfjk_status_string(int code) {
  switch (code) {
    case DFJK_OK: return "ok";
    case DFJK_ERR_ARG: return "invalid argument";
    case DFJK_ERR_UNSUPPORTED: return "unsupported input";
    case DFJK_ERR_NOT_PD: return "metric not positive definite";
    case DFJK_ERR_OOM: return "out of device memory";
    case DFJK_ERR_BUDGET: return "HBM budget exceeded";
    case DFJK_ERR_TIMEOUT: return "bounded device wait expired";
    case DFJK_ERR_CUDA: return "CUDA error";
    case DFJK_ERR_STATE: return "invalid handle state";
    default: return "unknown status";
  }
}

const char *dfjk_last_error(void) { return g_last_error.c_str(); }

uint64_t dfjk_launch_count(void) { return launch_counter().load(); }

int dfjk_set_timing(int32_t enable) {
  std::lock_guard<std::mutex> lk(g_timing_mu);
  g_timing = enable != 0;
  return DFJK_OK;
}

int dfjk_phase_times(double *ms, int32_t n) {
  if (!ms || n < 0) return fail(Error{DFJK_ERR_ARG, "phase_times arguments"});
  std::lock_guard<std::mutex> lk(g_timing_mu);
  for (int i = 0; i < n; ++i) ms[i] = 0.0;
  int rc = DFJK_OK;
  for (auto &r : g_phase_recs) {
    float t = 0.f;
    if (cudaEventSynchronize(r.b) == cudaSuccess && cudaEventElapsedTime(&t, r.a, r.b) == cudaSuccess) {
      if (r.phase >= 0 && r.phase < n) ms[r.phase] += t;
    } else {
      rc = DFJK_ERR_CUDA;
    }
    g_event_pool.push_back(r.a);
    g_event_pool.push_back(r.b);
  }
  g_phase_recs.clear();
  if (rc) set_error("event timing failed");
  return rc;
}

int dfjk_setup(const dfjk_basis *orb, const dfjk_basis *aux, int32_t natom, const double *coords,
               const dfjk_options *opt, void *stream, dfjk_handle *out) {
  if (!out) return fail(Error{DFJK_ERR_ARG, "out is null"});
  *out = nullptr;
  dfjk_ctx *h = nullptr;
  try {
    if (natom <= 0 || !coords) throw Error{DFJK_ERR_ARG, "natom/coords"};
    h = new dfjk_ctx();
    DFJK_CUDA_CHECK(cudaGetDevice(&h->device));
    if (opt) h->opt = *opt;
    else dfjk_default_options(&h->opt);
    if (h->opt.precision != DFJK_FP64 && h->opt.precision != DFJK_MIXED)
      throw Error{DFJK_ERR_UNSUPPORTED, "precision"};
    if (!(h->opt.schwarz_thresh >= 0.0)) throw Error{DFJK_ERR_ARG, "schwarz_thresh"};
    h->natom = natom;
    h->coords.assign(coords, coords + 3 * (size_t)natom);
    read_basis(orb, natom, coords, h->orb, "orbital basis");
    read_basis(aux, natom, coords, h->aux, "aux basis");
    h->nao = h->orb.nfunc;
    h->naux = h->aux.nfunc;
    if (h->nao == 0 || h->naux == 0) throw Error{DFJK_ERR_ARG, "empty basis"};
    h->naux_pad = ((h->naux + 63) / 64) * 64;
    const char *tab = h->opt.tune_table ? h->opt.tune_table : std::getenv("DFJK_TUNE_TABLE");
    lookup_tuning(tab, h->nao, h->tune);
    h->sliced = use_slices(h->opt.precision, h->nao, h->naux_pad);
    if (h->opt.precision == DFJK_FP64) h->wfmt = h->bfmt = OZ_F64;
    for (int d = 0; d < 3; ++d) {
      h->c0[d] = 0.0;
      for (int a = 0; a < natom; ++a) h->c0[d] += h->coords[3 * (size_t)a + d] / natom;
    }
    h->df_range = h->opt.precision == DFJK_MIXED && df_range_ok(h);
    h->use_df = h->df_range && h->opt.fp32_pair_thresh != 0.0;
    h->opt.tune_table = nullptr;  // the caller's string is not kept
    make_resident(h, S(stream));
    *out = h;
    return DFJK_OK;
  } catch (const Error &e) {
    delete h;
    return fail(e);
  } catch (const std::exception &e) {
    delete h;
    return fail(Error{DFJK_ERR_CUDA, e.what()});
  }
}

int dfjk_query(dfjk_handle h, int32_t *nao, int32_t *naux, int32_t *npair_kept, size_t *bytes) {
  if (!h) return fail(Error{DFJK_ERR_ARG, "null handle"});
  if (nao) *nao = h->nao;
  if (naux) *naux = h->naux;
  if (npair_kept) *npair_kept = h->npair_kept;
  if (bytes) *bytes = h->B.device_bytes() + h->Bexpo.bytes() + h->rowmap.bytes() + h->pl_buf.bytes() + h->pl_krow.bytes() +
                      h->V.bytes() + h->L.bytes() + h->Linv.bytes() + h->rec.bytes() + h->recd.bytes();
  return DFJK_OK;
}

int dfjk_query_precision(dfjk_handle h, int32_t *npair_fp32, double *fp32_thresh) {
  if (!h) return fail(Error{DFJK_ERR_ARG, "null handle"});
  if (npair_fp32) *npair_fp32 = h->npair_fp32;
  if (fp32_thresh) *fp32_thresh = h->fp32_thresh;
  return DFJK_OK;
}

int dfjk_estimate_bytes(int32_t nao, int32_t naux, int32_t nocc, int32_t precision, size_t *resident,
                        size_t *build_ws, size_t *setup_ws) {
  if (nao < 1 || naux < 1 || nocc < 1 || nocc > nao || (precision != DFJK_FP64 && precision != DFJK_MIXED))
    return fail(Error{DFJK_ERR_ARG, "estimate_bytes arguments"});
  const size_t np = ((size_t)naux + 63) / 64 * 64, n = (size_t)nao, no = (size_t)nocc;
  const bool mixed = precision == DFJK_MIXED;
  const size_t npack = n * (n + 1) / 2;
  const size_t b = (mixed ? npack : n * n) * np * 8;
  auto rup = [](size_t x, size_t m) { return (x + m - 1) / m * m; };
  const size_t steps = n * (rup(n, OZ_BK) / OZ_BK);  // K steps of the pair lists, every pair kept
  const bool sl = use_slices(precision, nao, (int)np);
  const int fmt = mixed ? OZ_36 : OZ_F64;
  const size_t kb = oz_kblock(fmt);
  const size_t r = b + 3 * np * np * 8 +
                   (sl ? n * rup(np, OZ_BM) * ((n + kb - 1) / kb) * 4 + 2 * steps * OZ_BK * 4 : 0);
  size_t ws = n * n * 8 + np * 8 * 2;  // D, rho
  if (sl) {
    // X, its slices and the slices of B for a chunk: fewer kept pairs make the chunk
    // longer, so the cap is the bound unless the whole aux range fits (or 128 rows do not)
    const size_t row = chunk_row_bytes(nao, nocc, fmt, (long long)steps);
    const size_t nkb = (np * no + kb - 1) / kb;
    ws += std::min(row * rup(np, OZ_BM), std::max(build_ws_bytes(0), row * OZ_BM)) + RHO_PARTS * np * 8;
    ws += rup(n, OZ_BM) * (2 * oz_slices(fmt) * OZ_BK + nkb * 4);         // X slices' padding, exponents
    const size_t cs = c_step_bytes(fmt, nocc);                            // C slices
    ws += std::min(std::max(C_SLICE_CAP, rup(n, OZ_BK) / OZ_BK * cs), steps * cs);
    ws += k_part_doubles(k_shape(nao, fmt, 0), (int)nkb) * 8 + oz_tile_seq_count(nao, nao) * 4;  // K partials
  } else {
    const size_t t = (n + 63) / 64, ksplit = std::max<size_t>(1, std::min<size_t>(64, (4 * 152 + t * (t + 1) / 2 - 1) / (t * (t + 1) / 2)));
    ws += n * np * no * 8 + n * n * ksplit * 8 + n * np * 8;  // X, K partials, rho partials
  }
  // setup: one T slab of at most 4 GiB (2 GiB plus its 8 slices with sliced products),
  // L^-1 and a work copy (plus L^-1's 8 slices)
  const size_t slab = std::min<size_t>((size_t)(sl ? 2 : 4) << 30, npack * np * 8);
  size_t sw = slab * (sl ? 3 : 1) + 2 * np * np * 8 + (sl ? np * np * 16 : 0);
  if (resident) *resident = r;
  if (build_ws) *build_ws = ws;
  if (setup_ws) *setup_ws = sw;
  return DFJK_OK;
}

int dfjk_query_pair_classes(dfjk_handle h, int64_t *prim_pairs_fp64, int64_t *prim_pairs_fp32) {
  if (!h) return fail(Error{DFJK_ERR_ARG, "null handle"});
  for (int c = 0; c < 6; ++c) {
    if (prim_pairs_fp64) prim_pairs_fp64[c] = h->prim_pairs64[c];
    if (prim_pairs_fp32) prim_pairs_fp32[c] = h->prim_pairs32[c];
  }
  return DFJK_OK;
}

int dfjk_query_tuning(dfjk_handle h, int32_t *vals) {
  if (!h || !vals) return fail(Error{DFJK_ERR_ARG, "null argument"});
  vals[0] = h->tune.slice_rows;
  vals[1] = h->tune.pslice_rows;
  vals[2] = h->tune.k_range_mb;
  vals[3] = h->tune.build_ws_mb;
  return DFJK_OK;
}

int dfjk_query_setup(dfjk_handle h, int32_t *nslab, int32_t *lean) {
  if (!h) return fail(Error{DFJK_ERR_ARG, "null handle"});
  if (nslab) *nslab = h->nslab;
  if (lean) *lean = h->lean ? 1 : 0;
  return DFJK_OK;
}

int dfjk_query_build(dfjk_handle h, int32_t *chunk_rows, int32_t *nchunk) {
  if (!h) return fail(Error{DFJK_ERR_ARG, "null handle"});
  const bool mixed = h->opt.precision == DFJK_MIXED && h->chunk_rows > 0;
  if (chunk_rows) *chunk_rows = mixed ? h->chunk_rows : 0;
  if (nchunk) *nchunk = mixed ? ceil_div(h->naux_pad, h->chunk_rows) : 0;
  return DFJK_OK;
}

int dfjk_build(dfjk_handle h, int32_t nset, int32_t nocc, const double *C, double *J, double *K,
               double *EJ, double *EK, void *stream) {
  try {
    if (!h) throw Error{DFJK_ERR_ARG, "null handle"};
    if (nset < 1 || nocc < 1 || !C || !J || !K || !EJ || !EK) throw Error{DFJK_ERR_ARG, "build arguments"};
    cudaStream_t st = S(stream);
    DFJK_CUDA_CHECK(cudaSetDevice(h->device));
    if (!h->resident) make_resident(h, st);
    ensure_workspace(h, nocc, nset);
    const size_t nao2 = (size_t)h->nao * h->nao;
    {
      PhaseScope span(13, st);
      for (int s = 0; s < nset; ++s) {
        const double *Cs = C + (size_t)s * h->nao * nocc;
        build_one(h, nocc, Cs, J + s * nao2, K + s * nao2, h->e.p + 2 * s, st);
      }
    }
    // energies go to host or device memory as the pointers are (detected per call)
    cudaPointerAttributes pa{}, pb{};
    DFJK_CUDA_CHECK(cudaPointerGetAttributes(&pa, EJ));
    DFJK_CUDA_CHECK(cudaPointerGetAttributes(&pb, EK));
    const bool dev_j = pa.type == cudaMemoryTypeDevice || pa.type == cudaMemoryTypeManaged;
    const bool dev_k = pb.type == cudaMemoryTypeDevice || pb.type == cudaMemoryTypeManaged;
    if (dev_j != dev_k) throw Error{DFJK_ERR_ARG, "E_J and E_K must both be host or both device memory"};
    if (!dev_j) {
      std::vector<double> e(2 * nset);
      DFJK_CUDA_CHECK(cudaMemcpyAsync(e.data(), h->e.p, e.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
      DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
      for (int s = 0; s < nset; ++s) {
        EJ[s] = e[2 * s];
        EK[s] = e[2 * s + 1];
      }
      throw_on_timeout(h, "build");
    } else {
      split_energies_kernel<<<ceil_div(nset, 64), 64, 0, st>>>(h->e.p, nset, EJ, EK);
      DFJK_LAUNCHED();
    }
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_build_uks(dfjk_handle h, int32_t nocc_a, const double *C_a, int32_t nocc_b, const double *C_b,
                   double *J, double *K_a, double *K_b, double *E, void *stream) {
  try {
    if (!h) throw Error{DFJK_ERR_ARG, "null handle"};
    if (nocc_a < 1 || nocc_b < 0 || nocc_b > nocc_a || !C_a || (nocc_b > 0 && !C_b) || !J || !K_a || !K_b || !E)
      throw Error{DFJK_ERR_ARG, "build_uks arguments"};
    cudaStream_t st = S(stream);
    DFJK_CUDA_CHECK(cudaSetDevice(h->device));
    if (!h->resident) make_resident(h, st);
    ensure_workspace(h, nocc_a, 3);
    const size_t nao2 = (size_t)h->nao * h->nao;
    if (!h->uks_D.p) h->uks_D.alloc(nao2);
    if (!h->uks_J.p) h->uks_J.alloc(nao2);
    double *e = h->e.p;  // [E_J a, E_K a, E_J b, E_K b, E_J total, -]
    build_one(h, nocc_a, C_a, J, K_a, e, st);
    DFJK_CUDA_CHECK(cudaMemcpyAsync(h->uks_D.p, h->D.p, nao2 * sizeof(double), cudaMemcpyDeviceToDevice, st));
    if (nocc_b > 0) {
      build_one(h, nocc_b, C_b, h->uks_J.p, K_b, e + 2, st);
      add_inplace(h->uks_D.p, h->D.p, (long long)nao2, st);
      add_inplace(J, h->uks_J.p, (long long)nao2, st);
    } else {
      DFJK_CUDA_CHECK(cudaMemsetAsync(K_b, 0, nao2 * sizeof(double), st));
      DFJK_CUDA_CHECK(cudaMemsetAsync(e + 2, 0, 2 * sizeof(double), st));
    }
    {
      PhaseScope ph(7, st);
      energies_f64(h->uks_D.p, J, K_a, h->nao, e + 4, h->en_work.p, st);
    }
    // E = {E_J of the total density, E_K alpha, E_K beta}
    cudaPointerAttributes pa{};
    DFJK_CUDA_CHECK(cudaPointerGetAttributes(&pa, E));
    const bool dev = pa.type == cudaMemoryTypeDevice || pa.type == cudaMemoryTypeManaged;
    if (dev) {  // E[0] = e[4], E[1] = e[1], E[2] = e[3], stream-ordered
      DFJK_CUDA_CHECK(cudaMemcpyAsync(E, e + 4, sizeof(double), cudaMemcpyDeviceToDevice, st));
      DFJK_CUDA_CHECK(cudaMemcpyAsync(E + 1, e + 1, sizeof(double), cudaMemcpyDeviceToDevice, st));
      DFJK_CUDA_CHECK(cudaMemcpyAsync(E + 2, e + 3, sizeof(double), cudaMemcpyDeviceToDevice, st));
    } else {
      double host[6];
      DFJK_CUDA_CHECK(cudaMemcpyAsync(host, e, sizeof(host), cudaMemcpyDeviceToHost, st));
      DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
      E[0] = host[4];
      E[1] = host[1];
      E[2] = host[3];
      throw_on_timeout(h, "build");
    }
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_build_density(dfjk_handle h, int32_t nset, const double *D, double *J, double *K, double *EJ,
                       double *EK, void *stream) {
  try {
    if (!h) throw Error{DFJK_ERR_ARG, "null handle"};
    if (nset < 1 || !D || !J || !K || !EJ || !EK) throw Error{DFJK_ERR_ARG, "build_density arguments"};
    cudaStream_t st = S(stream);
    DFJK_CUDA_CHECK(cudaSetDevice(h->device));
    if (!h->resident) make_resident(h, st);
    const int nao = h->nao, np = h->naux_pad;
    const size_t nao2 = (size_t)nao * nao;
    DBuf<double> rho, work, en;
    rho.alloc(np);
    work.alloc((size_t)RHO_PARTS * np);
    en.alloc(2 * 256);
    DensityWork dw;
    const StreamDrain drain{st};
    DBuf<double> &e = dw.e;  // energies, then the status word: one read-back for both
    e.alloc(2 * nset + 1);
    dw.status = reinterpret_cast<int *>(e.p + 2 * nset);
    DFJK_CUDA_CHECK(cudaMemsetAsync(dw.status, 0, sizeof(double), st));
    density_work(h, dw, st);
    for (int s = 0; s < nset; ++s) {
      const double *Ds = D + s * nao2;
      double *Js = J + s * nao2, *Ks = K + s * nao2;
      {  // J = B^T (B vec D)
        PhaseScope ph(6, st);
        rho_kept(h, h->B.p, h->ldb, Ds, np, rho.p, work.p, st);
        j_kept(h, rho.p, Js, st);
      }
      if (dw.sliced) density_k_sliced(h, dw, Ds, Ks, s > 0, st);
      else density_k_f64(h, dw, Ds, Ks, st);
      PhaseScope pe(7, st);
      energies_f64(Ds, Js, Ks, nao, e.p + 2 * s, en.p, st);
    }
    cudaPointerAttributes pa{}, pb{};
    DFJK_CUDA_CHECK(cudaPointerGetAttributes(&pa, EJ));
    DFJK_CUDA_CHECK(cudaPointerGetAttributes(&pb, EK));
    const bool dev_j = pa.type == cudaMemoryTypeDevice || pa.type == cudaMemoryTypeManaged;
    const bool dev_k = pb.type == cudaMemoryTypeDevice || pb.type == cudaMemoryTypeManaged;
    if (dev_j != dev_k) throw Error{DFJK_ERR_ARG, "E_J and E_K must both be host or both device memory"};
    if (dev_j) {
      split_energies_kernel<<<ceil_div(nset, 64), 64, 0, st>>>(e.p, nset, EJ, EK);
      DFJK_LAUNCHED();
    }
    std::vector<double> back(2 * nset + 1);
    DFJK_CUDA_CHECK(cudaMemcpyAsync(back.data(), e.p, e.bytes(), cudaMemcpyDeviceToHost, st));
    DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    if (!dev_j)
      for (int s = 0; s < nset; ++s) {
        EJ[s] = back[2 * s];
        EK[s] = back[2 * s + 1];
      }
    int status;
    std::memcpy(&status, &back[2 * nset], sizeof(int));
    if (status & STATUS_TIMEOUT) throw Error{DFJK_ERR_TIMEOUT, "a bounded device wait expired during the density build"};
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

// Intermediates of a gradient's finished stage up to this size stay to the end of its
// dense part: giving them back takes a wait of some 20 us.
constexpr size_t GRAD_HELD_BYTES = (size_t)4 << 30;

// Buffers of a gradient call.
struct GradWork {
  DBuf<double> D, rho, work, d, X, Xt, Z, stage, W, gam;
  DBuf<double> rec, gm;  // pair records and weights: doubles or double-single pairs
  DBuf<long long> goff;
  DBuf<int> orb_atom, aux_atom, aux_l;
  DBuf<unsigned> top;  // high words of the largest |D|, |d|, |C|, |Z|, and the status word
  XWork xw;
  std::deque<SlicedOp> ops;  // slices of the tensor-core GEMMs
  void free_ops() {
    for (SlicedOp &o : ops) oz_free(o);
    ops.clear();
  }
  ~GradWork() { free_ops(); }
};

// Whether weights of this size keep the double-single derivative kernels inside the FP32
// range: they multiply Hermite integrals of up to 1e28 (exponents of 1e4) on the way
// up and lose the low parts near 1e-38 on the way down.  Densities far from 1 (scaled
// or difference densities) take the FP64 kernels.
static bool df_weight_ok(double w, double lo, double hi) { return w == 0.0 || (w >= lo && w <= hi); }

// d(cj E_J + ck E_K)/dR at fixed D = C C^T (or the given D when ck = 0).
// E = sum_PQ (V^-1)_PQ M_PQ / 2 for both energies, M_PQ = u_P u_Q (J) or
// Tr(D T_P D T_Q) (K), so dE/dR = sum_P Tr(Gam_P dT_P/dR) - Tr(Wt dV/dR) / 2
// with Gam_P = (V^-1 M-side)_P: d_P D for J and D (L^-T B)_P D = C Z_P C^T for
// K, Z_P = sum_Q (L^-1)_QP C^T B_Q C; Wt = d d^T for J and Z Z^T for K.
static void jk_gradient(dfjk_ctx *h, const double *Din, int nocc, const double *C, double cj, double ck,
                 double *grad, cudaStream_t st) {
  DFJK_CUDA_CHECK(cudaSetDevice(h->device));
  if (!h->resident) make_resident(h, st);
  const int nao = h->nao, np = h->naux_pad;
  const double *tab = boys_table_device();
  GradWork wk;
  const StreamDrain drain{st};
  const double *D = Din;
  if (!D) {  // D = C C^T
    wk.D.alloc((size_t)nao * nao);
    GemmArgs dd;
    dd.M = nao; dd.N = nao; dd.K = nocc;
    dd.A = C; dd.sAm = nocc; dd.sAk = 1;
    dd.B = C; dd.sBn = nocc; dd.sBk = 1;
    dd.C = wk.D.p; dd.sCm = nao; dd.sCn = 1;
    gemm_f64(dd, st);
    D = wk.D.p;
  }
  // rho = B vec D (= L^-1 u), then the fitted coefficients d = L^-T rho = V^-1 u
  DBuf<double> &rho = wk.rho, &work = wk.work, &d = wk.d;
  rho.alloc(np);
  work.alloc(std::max<size_t>((size_t)128 * ceil_div(np, 256) * 256, (size_t)16 * np));
  d.alloc(np);
  DFJK_CUDA_CHECK(cudaMemsetAsync(d.p, 0, d.bytes(), st));
  rho_kept(h, h->B.p, h->ldb, D, np, rho.p, work.p, st);
  fitted_coefficients(h->Linv.p, h->naux, np, rho.p, work.p, d.p, st);
  DBuf<double> &gam = wk.gam, &W = wk.W;
  // view x(z, r, k) = p[z sz + r sr + k sk] in sliced form
  auto slice = [&](const double *p, long long sz, long long sr, long long sk, int batch, int rows, int K,
                   int tile) -> SlicedOp & {
    wk.ops.emplace_back();
    SlicedOp &o = wk.ops.back();
    oz_alloc(o, batch, h->bfmt, rows, K, tile);
    oz_slice_f64(p, sz, sr, sk, o, st);
    return o;
  };
  // out[z][m][n] = sum_k A(z, m, k) B(n, k) on the tensor cores (A batched when nz > 1)
  auto tc_gemm = [&](const SlicedOp &A, const SlicedOp &Bo, int M, int N, int K, int nz, double *out,
                     long long ldo, long long obs, int lower) {
    OzGemmArgs o;
    o.M = M; o.N = N; o.K = K; o.nz = nz; o.a_batched = nz > 1 ? 1 : 0;
    o.lower_only = lower; o.mode = 0; o.out = out; o.ldo = ldo; o.out_bs = obs;
    o.status = h->status.p; o.timeout = h->opt.timeout_iters; o.tile_ctr = h->tctr.p;
    oz_gemm(A, Bo, o, st);
  };
  // out[P][m][n] = sum_k x(P, m, k) B(n, k) for all P, x(P, r, k) = p[P sz + r sr + k sk]: the
  // slices are cut for ranges of P within a quarter of the build's work-buffer cap
  auto tc_gemm_per_aux = [&](const double *p, long long sz, long long sr, long long sk, int rows, int K, const SlicedOp &Bo,
                             int N, double *out, long long ldo, long long obs) {
    const size_t per = oz_bytes(h->bfmt, rows, K, OZ_BM);
    const int nb = (int)std::min<size_t>(np, std::max<size_t>(1, build_ws_bytes(h->tune.build_ws_mb) / 4 / per));
    wk.ops.emplace_back();
    SlicedOp &o = wk.ops.back();
    oz_alloc(o, nb, h->bfmt, rows, K, OZ_BM);
    for (int p0 = 0; p0 < np; p0 += nb) {
      SlicedOp v = o;
      v.batch = std::min(nb, np - p0);
      oz_slice_f64(p + p0 * sz, sz, sr, sk, v, st);
      tc_gemm(v, Bo, rows, N, K, v.batch, out + p0 * obs, ldo, obs, 0);
    }
  };
  // What a finished stage held goes back once it amounts to something: FP64 slices are
  // twice their operand's size, and G alone is naux_pad nao^2 doubles.
  auto stage_done = [&](std::initializer_list<DBuf<double> *> bufs) {
    size_t held = wk.xw.bsl.bytes() + wk.xw.cdat.bytes();
    for (const SlicedOp &o : wk.ops) held += o.data_bytes();
    for (DBuf<double> *b : bufs) held += b->bytes();
    if (held < GRAD_HELD_BYTES) return;
    DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    for (DBuf<double> *b : bufs) b->release();
    wk.xw.release();
    wk.free_ops();
  };
  const bool exch = ck != 0.0;
  AbsMax am{};
  am.x[0] = D; am.n[0] = (long long)nao * nao;
  am.x[1] = d.p; am.n[1] = h->naux;
  wk.top.alloc(5);
  if (exch) {
    // the build's slices on the tensor cores, or FP64 CUDA-core GEMMs for the small
    // molecules of DFJK_FP64
    const bool tc = h->sliced;
    const long long no2 = (long long)nocc * nocc;
    DBuf<double> &X = wk.X, &Xt = wk.Xt, &Z = wk.Z, &stage = wk.stage;
    XWork &xw = wk.xw;
    X.alloc((size_t)nao * np * nocc);
    Xt.alloc((size_t)np * no2);
    Z.alloc((size_t)np * no2);
    W.alloc((size_t)np * np);
    if (tc) {
      const SlicedOp &csl = slice(C, 0, 1, nocc, 1, nocc, nao, OZ_BN);  // rows i, K nu
      // X[mu][P][i] = sum_nu B[(mu,nu)][P] C[nu][i], chunk by chunk of rows P
      // as the build does
      const int pcm = build_chunk_rows(nao, np, nocc, h->bfmt, h->pl.steps, h->tune.build_ws_mb);
      alloc_xwork(h, h->pl, xw, pcm, nocc);
      if (h->B.host) stage.alloc(stage_size(h, pcm));
      for (int p0 = 0; p0 < np; p0 += pcm) {
        const int pc = std::min(pcm, np - p0);
        const double *b = h->B.p + p0;
        if (h->B.host) b = stage_columns(h, stage, p0, pc, st);
        x_gemm_sliced(h, h->pl, h->Bexpo.p, xw,
                      XArgs{b, h->B.host ? pc : h->ldb, C, nocc, 1, nocc, p0, pc, X.p + (size_t)p0 * nocc, nocc,
                            (long long)np * nocc, 0, p0 == 0}, st);
      }
      // Xt[P][j][i] = sum_mu X[mu][P][j] C[mu][i]  (symmetric in i, j)
      tc_gemm_per_aux(X.p, nocc, 1, (long long)np * nocc, nocc, nao, csl, nocc, Xt.p, nocc, no2);
      stage_done({&stage});
      // Z[P][ij] = sum_Q Linv[Q][P] Xt[Q][ij]
      const SlicedOp &lt = slice(h->Linv.p, 0, 1, np, 1, np, np, OZ_BM);
      const SlicedOp &xts = slice(Xt.p, 0, 1, no2, 1, (int)no2, np, OZ_BN);
      tc_gemm(lt, xts, np, (int)no2, np, 1, Z.p, no2, 0, 0);
      // W = Z Z^T, lower triangle, then mirrored
      const SlicedOp &zs = slice(Z.p, 0, no2, 1, 1, np, (int)no2, OZ_BM);
      tc_gemm(zs, zs, np, np, (int)no2, 1, W.p, np, 0, 1);
      mirror_lower_f64(W.p, np, st);
      // Yt[P][j][mu] = sum_i Z[P][i][j] C[mu][i]   (Yt reuses X)
      stage_done({&Xt});
      const SlicedOp &cn = slice(C, 0, nocc, 1, 1, nao, nocc, OZ_BN);  // rows mu, K i
      tc_gemm_per_aux(Z.p, no2, 1, nocc, nocc, nocc, cn, nao, X.p, nao, (long long)nao * nocc);
      // Gam[P][mu][nu] = sum_j Yt[P][j][mu] C[nu][j]
      gam.alloc((size_t)np * nao * nao);
      tc_gemm_per_aux(X.p, (long long)nao * nocc, 1, nao, nao, nocc, cn, nao, gam.p, nao, (long long)nao * nao);
    } else {
      gam.alloc((size_t)np * nao * nao);
      GemmArgs x;  // X[mu][P][i] = sum_nu B[(mu,nu)][P] C[nu][i]
      x.M = np; x.N = nocc; x.K = nao; x.batch = nao;
      x.A = h->B.p; x.sAm = 1; x.sAk = h->ldb; x.sAb = (long long)nao * h->ldb;
      x.B = C; x.sBn = 1; x.sBk = nocc; x.sBb = 0;
      x.C = X.p; x.sCm = nocc; x.sCn = 1; x.sCb = (long long)np * nocc;
      gemm_f64(x, st);
      GemmArgs t;  // Xt[P][i][j] = sum_mu C[mu][i] X[mu][P][j]
      t.M = nocc; t.N = nocc; t.K = nao; t.batch = np;
      t.A = C; t.sAm = 1; t.sAk = nocc; t.sAb = 0;
      t.B = X.p; t.sBn = 1; t.sBk = (long long)np * nocc; t.sBb = nocc;
      t.C = Xt.p; t.sCm = nocc; t.sCn = 1; t.sCb = no2;
      gemm_f64(t, st);
      GemmArgs z;  // Z[P][ij] = sum_{Q >= P} Linv[Q][P] Xt[Q][ij]
      z.M = np; z.N = (int)no2; z.K = np;
      z.A = h->Linv.p; z.sAm = 1; z.sAk = np; z.k_from_m = 1;
      z.B = Xt.p; z.sBn = 1; z.sBk = no2;
      z.C = Z.p; z.sCm = no2; z.sCn = 1;
      gemm_f64(z, st);
      GemmArgs w;  // W = Z Z^T, lower triangle, then mirrored
      w.M = np; w.N = np; w.K = (int)no2;
      w.A = Z.p; w.sAm = no2; w.sAk = 1;
      w.B = Z.p; w.sBn = no2; w.sBk = 1;
      w.C = W.p; w.sCm = np; w.sCn = 1;
      w.lower_only = 1;
      gemm_f64(w, st);
      mirror_lower_f64(W.p, np, st);
      GemmArgs y;  // Y[P][mu][j] = sum_i C[mu][i] Z[P][i][j]   (Y reuses X)
      y.M = nao; y.N = nocc; y.K = nocc; y.batch = np;
      y.A = C; y.sAm = nocc; y.sAk = 1; y.sAb = 0;
      y.B = Z.p; y.sBn = 1; y.sBk = nocc; y.sBb = no2;
      y.C = X.p; y.sCm = nocc; y.sCn = 1; y.sCb = (long long)nao * nocc;
      gemm_f64(y, st);
      GemmArgs gm;  // Gam[P][mu][nu] = sum_j Y[P][mu][j] C[nu][j]
      gm.M = nao; gm.N = nao; gm.K = nocc; gm.batch = np;
      gm.A = X.p; gm.sAm = nocc; gm.sAk = 1; gm.sAb = (long long)nao * nocc;
      gm.B = C; gm.sBn = nocc; gm.sBk = 1; gm.sBb = 0;
      gm.C = gam.p; gm.sCm = nao; gm.sCn = 1; gm.sCb = (long long)nao * nao;
      gemm_f64(gm, st);
    }
    am.x[2] = C; am.n[2] = (long long)nao * nocc;
    am.x[3] = Z.p; am.n[3] = np * no2;
  }
  if (h->use_df) abs_max(am, wk.top.p, st);
  if (exch) {
    DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    for (DBuf<double> *b : {&wk.X, &wk.Xt, &wk.Z, &wk.stage}) b->release();
    wk.xw.release();
    wk.free_ops();
  }
  DBuf<int> &oat = wk.orb_atom, &aat = wk.aux_atom, &al = wk.aux_l;
  oat.upload(h->orb.atom, st);
  aat.upload(h->aux.atom, st);
  al.upload(h->aux.l, st);
  GradArgs g{};
  g.pair_a = h->pair_a.p;
  g.pair_b = h->pair_b.p;
  g.npp = h->pair_npp.p;
  g.pair_col = h->pair_col.p;
  g.ldg = np;
  g.d = d.p;
  g.D = D;
  g.nao = nao;
  g.cj = cj;
  g.gam = gam.p;
  g.W = W.p;
  g.ldw = np;
  g.ck = ck;
  g.orb_atom = oat.p;
  g.aux_atom = aat.p;
  g.grad = grad;
  static const int cls[6][2] = {{0, 0}, {1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
  const GradBoysTabs tabs{tab, boys_table_device_f32(), boys_table_device_df()};
  std::vector<long long> off(h->npair_kept + 1, 0);
  for (int c = 0; c < 6; ++c)
    for (int i = h->kept_cls_begin[c]; i < h->kept_cls_begin[c + 1]; ++i)
      off[i + 1] = off[i] + (long long)h->npp_h[h->kept_h[i]] * grad_record_len(cls[c][0], cls[c][1], exch);
  DBuf<long long> &goff = wk.goff;
  goff.upload(off, st);
  DBuf<double> &rec = wk.rec, &gm = wk.gm;
  rec.alloc(std::max<size_t>(1, (size_t)off.back()));
  if (exch) gm.alloc((size_t)std::max<long long>(h->ncol, 1) * np);
  const auto run = [&](bool dfs) {
    DFJK_CUDA_CHECK(cudaMemsetAsync(grad, 0, sizeof(double) * 3 * (size_t)h->natom, st));
    // Coulomb-only gradients of a mixed handle take the build's precision split: the
    // kept pairs it evaluates in FP32 (Schwarz bound below fp32_pair_thresh) get FP32
    // derivative weights, the others double-single (FP64 beyond its range)
    const bool split32 = !exch && dfs;
    for (int q = 0; q < 3; ++q) g.c0[q] = dfs ? h->c0[q] : 0.0;
    for (int c = 0; c < 6; ++c) {
      g.pairs = h->kept.p + h->kept_cls_begin[c];
      g.npairs = h->kept_cls_begin[c + 1] - h->kept_cls_begin[c];
      g.rec_off = goff.p + h->kept_cls_begin[c];
      launch_grad_tables(cls[c][0], cls[c][1], exch, dfs, g, orb_args(h), rec.p, st);
      if (exch) launch_grad_gamma(cls[c][0], cls[c][1], dfs, g, orb_args(h), h->naux, gm.p, st);
    }
    g.rec = rec.p;
    g.gamma = gm.p;
    // The classes run on the integral streams, the largest first: one after the other each
    // left the GPU to its own last wave: 45 atoms (Coulomb) 11.3 -> 9.7 ms,
    // 30 atoms (Coulomb and exchange) 19.2 -> 16.1.
    {
      const IntegralFork fork(st, h->ev_int);
      launch_grad2c(g, aux_args(h), al.p, h->aux.nshell, tab, fork.is[INT_STREAMS - 1]);
      for (int c = 5; c >= 0; --c) {
        const int lo = h->kept_cls_begin[c], hi = h->kept_cls_begin[c + 1];
        if (hi <= lo) continue;
        const int mid = split32 ? std::min(std::max(lo, h->kept32_begin[c]), hi) : hi;
        for (int lc = 2; lc >= 0; --lc) {
          g.aux_shells = h->aux_cls[lc].p;
          g.naux_shells = h->aux_cls_n[lc];
          g.pairs = h->kept.p + lo;
          g.rec_off = goff.p + lo;
          g.npairs = mid - lo;
          launch_grad3c(cls[c][0], cls[c][1], lc, dfs ? GRAD_DF : GRAD_F64, g, aux_args(h), tabs,
                        fork.is[(c + lc) % (INT_STREAMS - 1)]);
          g.pairs = h->kept.p + mid;
          g.rec_off = goff.p + mid;
          g.npairs = hi - mid;
          launch_grad3c(cls[c][0], cls[c][1], lc, GRAD_F32, g, aux_args(h), tabs, fork.is[INT_STREAMS - 1]);
        }
      }
    }
  };
  run(h->use_df);
  unsigned top[5];
  DFJK_CUDA_CHECK(cudaMemcpyAsync(wk.top.p + 4, h->status.p, sizeof(int), cudaMemcpyDeviceToDevice, st));
  DFJK_CUDA_CHECK(cudaMemcpyAsync(top, wk.top.p, sizeof(top), cudaMemcpyDeviceToHost, st));
  DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
  if (h->use_df) {
    const double Dm = abs_max_value(top[0]), dm = std::fabs(cj) * abs_max_value(top[1]), Cm = abs_max_value(top[2]);
    const double gamma = std::fabs(ck) * Cm * Cm * abs_max_value(top[3]);  // Gam = C Z C^T
    const bool ok = exch ? df_weight_ok(std::max(dm * Dm, gamma * nocc * nocc), 0x1p-50, 0x1p60)
                         : df_weight_ok(Dm, 0x1p-40, 0x1p30) && df_weight_ok(dm, 0x1p-40, 0x1p30);
    if (!ok) {  // once more, in FP64: the rare case pays, not every call with a wait for the sizes
      run(false);
      DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    }
  }
  throw_on_timeout(h, (int)top[4], "gradient");
}

int dfjk_coulomb_gradient(dfjk_handle h, const double *D, double *grad, void *stream) {
  try {
    if (!h || !D || !grad) throw Error{DFJK_ERR_ARG, "coulomb_gradient arguments"};
    jk_gradient(h, D, 0, nullptr, 1.0, 0.0, grad, S(stream));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_jk_gradient(dfjk_handle h, int32_t nocc, const double *C_occ, double c_j, double c_k, double *grad,
                     void *stream) {
  try {
    if (!h || !C_occ || !grad || nocc < 1 || nocc > h->nao || !std::isfinite(c_j) || !std::isfinite(c_k))
      throw Error{DFJK_ERR_ARG, "jk_gradient arguments"};
    jk_gradient(h, nullptr, nocc, C_occ, c_j, c_k, grad, S(stream));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_build_batch(int32_t nmol, const dfjk_handle *hs, const int32_t *nocc, const double *const *C,
                     double *const *J, double *const *K, double *EJ, double *EK, int32_t nstreams,
                     void *stream) {
  try {
    if (nmol < 0 || (nmol > 0 && (!hs || !nocc || !C || !J || !K || !EJ || !EK)))
      throw Error{DFJK_ERR_ARG, "build_batch arguments"};
    if (nmol == 0) return DFJK_OK;
    nstreams = std::max(1, std::min(nstreams, 32));
    cudaStream_t st = S(stream);
    for (int i = 0; i < nmol; ++i) {
      if (!hs[i] || nocc[i] < 1 || !C[i] || !J[i] || !K[i]) throw Error{DFJK_ERR_ARG, "build_batch entry"};
      if (!hs[i]->resident) throw Error{DFJK_ERR_STATE, "build_batch: handle evicted"};
      for (int j = 0; j < i; ++j)
        if (hs[j] == hs[i]) throw Error{DFJK_ERR_ARG, "build_batch: a handle appears twice"};
    }
    // internal streams and events, created once per device
    struct Fork {
      std::vector<cudaStream_t> streams;
      std::vector<cudaEvent_t> done;
      cudaEvent_t start;
    };
    static std::mutex mu;
    static std::map<int, Fork> forks;
    int dev = 0;
    DFJK_CUDA_CHECK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    Fork &f = forks[dev];
    if (f.streams.empty()) DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&f.start, cudaEventDisableTiming));
    while ((int)f.streams.size() < nstreams) {
      cudaStream_t s2;
      cudaEvent_t e2;
      DFJK_CUDA_CHECK(cudaStreamCreateWithFlags(&s2, cudaStreamNonBlocking));
      DFJK_CUDA_CHECK(cudaEventCreateWithFlags(&e2, cudaEventDisableTiming));
      f.streams.push_back(s2);
      f.done.push_back(e2);
    }
    DFJK_CUDA_CHECK(cudaEventRecord(f.start, st));
    for (int k = 0; k < nstreams; ++k) DFJK_CUDA_CHECK(cudaStreamWaitEvent(f.streams[k], f.start, 0));
    for (int i = 0; i < nmol; ++i) {
      dfjk_ctx *h = hs[i];
      cudaStream_t s2 = f.streams[i % nstreams];
      ensure_workspace(h, nocc[i], 1);
      build_one(h, nocc[i], C[i], J[i], K[i], h->e.p, s2);
      split_energies_kernel<<<1, 64, 0, s2>>>(h->e.p, 1, EJ + i, EK + i);
      DFJK_LAUNCHED();
    }
    for (int k = 0; k < nstreams; ++k) {
      DFJK_CUDA_CHECK(cudaEventRecord(f.done[k], f.streams[k]));
      DFJK_CUDA_CHECK(cudaStreamWaitEvent(st, f.done[k], 0));
    }
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_overlap(dfjk_handle h, double *Sout, void *stream) {
  try {
    if (!h || !Sout) throw Error{DFJK_ERR_ARG, "overlap arguments"};
    cudaStream_t st = S(stream);
    if (!h->o_center.p) upload_bases(h, st);
    static const int cls[6][2] = {{0, 0}, {1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
    for (int c = 0; c < 6; ++c) {
      std::vector<int> sa, sb;
      for (int a = 0; a < h->orb.nshell; ++a)
        for (int b = 0; b < h->orb.nshell; ++b)
          if (h->orb.l[a] == cls[c][0] && h->orb.l[b] == cls[c][1] && (cls[c][0] != cls[c][1] || b <= a)) {
            sa.push_back(a);
            sb.push_back(b);
          }
      if (sa.empty()) continue;
      DBuf<int> da, db;
      da.upload(sa, st);
      db.upload(sb, st);
      OverlapArgs a{(int)sa.size(), da.p, db.p, Sout, h->nao};
      launch_overlap(cls[c][0], cls[c][1], a, orb_args(h), st);
      DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    }
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_overlap_matrix(const dfjk_basis *orb, int32_t natom, const double *coords, double *Sout,
                        void *stream) {
  dfjk_ctx *h = nullptr;
  try {
    if (natom <= 0 || !coords || !Sout) throw Error{DFJK_ERR_ARG, "overlap_matrix arguments"};
    h = new dfjk_ctx();
    DFJK_CUDA_CHECK(cudaGetDevice(&h->device));
    h->natom = natom;
    read_basis(orb, natom, coords, h->orb, "orbital basis");
    h->nao = h->orb.nfunc;
    const int rc = dfjk_overlap(h, Sout, stream);
    delete h;
    return rc;
  } catch (const Error &e) {
    delete h;
    return fail(e);
  }
}

int dfjk_evict(dfjk_handle h) {
  if (!h) return fail(Error{DFJK_ERR_ARG, "null handle"});
  try {
    DFJK_CUDA_CHECK(cudaSetDevice(h->device));
    DFJK_CUDA_CHECK(cudaDeviceSynchronize());
    release_device(h);
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_destroy(dfjk_handle h) {
  if (!h) return DFJK_OK;
  cudaSetDevice(h->device);
  cudaDeviceSynchronize();
  delete h;
  return DFJK_OK;
}

int dfjk_boys(int32_t mmax, int32_t n, const double *T, double *F, void *stream) {
  try {
    if (n < 0 || (n > 0 && (!T || !F))) throw Error{DFJK_ERR_ARG, "boys arguments"};
    launch_boys(mmax, n, T, F, boys_table_device(), S(stream));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_get_metric(dfjk_handle h, double *Vout, void *stream) {
  try {
    if (!h || !Vout) throw Error{DFJK_ERR_ARG, "null argument"};
    if (!h->resident) throw Error{DFJK_ERR_STATE, "handle evicted"};
    DFJK_CUDA_CHECK(cudaMemcpy2DAsync(Vout, h->naux * 8, h->V.p, h->naux_pad * 8, h->naux * 8, h->naux,
                                      cudaMemcpyDeviceToDevice, S(stream)));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_get_cholesky(dfjk_handle h, double *Lout, void *stream) {
  try {
    if (!h || !Lout) throw Error{DFJK_ERR_ARG, "null argument"};
    if (!h->resident) throw Error{DFJK_ERR_STATE, "handle evicted"};
    DFJK_CUDA_CHECK(cudaMemcpy2DAsync(Lout, h->naux * 8, h->L.p, h->naux_pad * 8, h->naux * 8, h->naux,
                                      cudaMemcpyDeviceToDevice, S(stream)));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_get_B(dfjk_handle h, double *Bout, void *stream) {
  try {
    if (!h || !Bout) throw Error{DFJK_ERR_ARG, "null argument"};
    if (!h->resident) throw Error{DFJK_ERR_STATE, "handle evicted"};
    cudaStream_t st = S(stream);
    std::vector<int> ident(h->naux);
    for (int i = 0; i < h->naux; ++i) ident[i] = i;
    DBuf<int> perm;
    perm.upload(ident, st);
    gather_B_f64(h->B.p, h->ldb, h->nao, perm.p, h->naux, Bout, h->lean ? h->rowmap.p : nullptr, st);
    DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_get_B_columns(dfjk_handle h, int32_t ncol, const int32_t *mu, const int32_t *nu, double *out,
                       void *stream) {
  try {
    if (!h || ncol < 0 || (ncol > 0 && (!mu || !nu || !out))) throw Error{DFJK_ERR_ARG, "null argument"};
    if (!h->resident) throw Error{DFJK_ERR_STATE, "handle evicted"};
    if (ncol == 0) return DFJK_OK;
    cudaStream_t st = S(stream);
    std::vector<int> rows(ncol), ident(h->naux), map;
    if (h->lean) {  // rows of the kept pairs (-1: screened, zero)
      map.resize((size_t)h->nao * h->nao);
      DFJK_CUDA_CHECK(cudaMemcpyAsync(map.data(), h->rowmap.p, map.size() * sizeof(int), cudaMemcpyDeviceToHost, st));
      DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    }
    for (int c = 0; c < ncol; ++c) {
      if (mu[c] < 0 || mu[c] >= h->nao || nu[c] < 0 || nu[c] >= h->nao) throw Error{DFJK_ERR_ARG, "AO index"};
      const long long e = (long long)mu[c] * h->nao + nu[c];
      rows[c] = h->lean ? map[e] : (int)e;
    }
    for (int i = 0; i < h->naux; ++i) ident[i] = i;
    DBuf<int> r, p;
    r.upload(rows, st);
    p.upload(ident, st);
    gather2d_f64(h->B.p, h->ldb, r.p, p.p, ncol, h->naux, out, h->naux, st);
    DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

int dfjk_get_pair_mask(dfjk_handle h, int32_t *keep, void *stream) {
  try {
    if (!h || !keep) throw Error{DFJK_ERR_ARG, "null argument"};
    const int ns = h->orb.nshell;
    std::vector<int> m((size_t)ns * ns, 0);
    for (int i = 0; i < (int)h->pa_h.size(); ++i)
      if (h->pair_col_h[i] >= 0) {
        m[(size_t)h->pa_h[i] * ns + h->pb_h[i]] = 1;
        m[(size_t)h->pb_h[i] * ns + h->pa_h[i]] = 1;
      }
    DFJK_CUDA_CHECK(cudaMemcpyAsync(keep, m.data(), m.size() * sizeof(int), cudaMemcpyHostToDevice, S(stream)));
    DFJK_CUDA_CHECK(cudaStreamSynchronize(S(stream)));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}

}  // extern "C"

namespace {
__global__ void scatter_T_kernel(const void *T, int dfT, int ldT, long long ncol, int naux, const int *colmu,
                                 const int *colnu, int nao, double *out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ncol * naux) return;
  const long long c = e / naux;
  const int P = (int)(e % naux);
  const int mu = colmu[c], nu = colnu[c];
  if (mu < 0) return;
  double v;
  if (dfT) {
    const float2 p = static_cast<const float2 *>(T)[c * ldT + P];
    v = (double)p.x + (double)p.y;
  } else {
    v = static_cast<const double *>(T)[c * ldT + P];
  }
  const long long n2 = (long long)nao * nao;
  out[P * n2 + (long long)mu * nao + nu] = v;
  out[P * n2 + (long long)nu * nao + mu] = v;
}
}  // namespace

extern "C" int dfjk_get_three_center(dfjk_handle h, double *Tout, void *stream) {
  try {
    if (!h || !Tout) throw Error{DFJK_ERR_ARG, "null argument"};
    if (!h->resident) throw Error{DFJK_ERR_STATE, "handle evicted"};
    cudaStream_t st = S(stream);
    const int np = h->naux_pad;
    const double *tab = boys_table_device();
    DBuf<double> T;
    T.alloc((size_t)std::max<long long>(h->ncol, 1) * np);
    DFJK_CUDA_CHECK(cudaMemsetAsync(T.p, 0, T.bytes(), st));
    DFJK_CUDA_CHECK(cudaMemsetAsync(Tout, 0, sizeof(double) * (size_t)h->naux * h->nao * h->nao, st));
    const IntegralTables tables;
    for (int c = 0; c < 6; ++c) {  // the same split of the pairs as the setup
      const int lo = h->kept_cls_begin[c], hi = h->kept_cls_begin[c + 1];
      if (hi <= lo) continue;
      const int mid = std::min(std::max(lo, h->kept32_begin[c]), hi);
      for (int lc = 0; lc < 3; ++lc) {
        launch_integrals(h, c, lc, h->kept.p + lo, mid - lo, false, T.p, 0, tables, st);
        launch_integrals(h, c, lc, h->kept.p + mid, hi - mid, true, T.p, 0, tables, st);
      }
    }
    const long long n = h->ncol * h->naux;
    if (n > 0) {
      scatter_T_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(T.p, h->use_df ? 1 : 0, np, h->ncol, h->naux, h->colmu.p,
                                                                     h->colnu.p, h->nao, Tout);
      DFJK_LAUNCHED();
    }
    DFJK_CUDA_CHECK(cudaStreamSynchronize(st));
    return DFJK_OK;
  } catch (const Error &e) {
    return fail(e);
  }
}
