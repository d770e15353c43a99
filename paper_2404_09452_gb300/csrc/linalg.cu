// FP64 dense kernels of the DF-J/K build: a generic strided GEMM (64x64x16
// tiles, 4x4 outputs per thread), blocked Cholesky and triangular inverse of
// the metric, the two streaming GEMVs of J (rho = B vec(D), J = B^T rho) and
// deterministic reductions.
//
// Paper: Introduction, contribution 1 (after the 3-centre integrals, density
// fitting is tensor operations) and the accuracy passage of the PySCF
// compatibility section (the fitting solve).  On this GPU FP64 runs at about
// 1.2 TFLOP/s, 1/62 of FP32, so these SIMT kernels are bound by the FP64 pipe
// at any reasonable tiling; they are the plain-FP64 reference path.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "linalg.cuh"

namespace dfjk {

constexpr int GBK = 16;

// TILE x TILE output tile per 256-thread CTA, (TILE/16)^2 outputs per thread;
// TILE = 32 gives four times more CTAs for the small, latency-bound GEMMs of
// the Cholesky factorisation and the triangular inverse.
template <int TILE, bool A_KC, bool B_KC, bool SCATTER>
__global__ void __launch_bounds__(256) gemm_f64_kernel(GemmArgs g) {
  constexpr int GBM = TILE, GBN = TILE, TT = TILE / 16;
  __shared__ double As[GBK][GBM + 1];
  __shared__ double Bs[GBK][GBN + 1];
  const int m0 = blockIdx.y * GBM, n0 = blockIdx.x * GBN;
  if (g.lower_only && n0 > m0 + GBM - 1) return;
  const int z = blockIdx.z;
  const double *A = g.A, *B = g.B;
  double *C = g.C;
  long long kbeg = 0, kend = g.K;
  if (g.k_split > 0) {
    kbeg = (long long)z * g.k_split;
    kend = min((long long)g.K, kbeg + g.k_split);
    C += z * g.sCb;
  } else {
    A += z * g.sAb;
    B += z * g.sBb;
    C += z * g.sCb;
  }
  if (g.k_upto_n) kend = min(kend, (long long)(n0 + GBN));
  if (g.k_upto_m) kend = min(kend, (long long)(m0 + GBM));
  if (g.k_from_n) kbeg = max(kbeg, (long long)n0);
  if (g.k_from_m) kbeg = max(kbeg, (long long)m0);
  const int Mz = g.M;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double acc[TT][TT];
#pragma unroll
  for (int i = 0; i < TT; ++i)
#pragma unroll
    for (int j = 0; j < TT; ++j) acc[i][j] = 0.0;

  for (long long k0 = kbeg; k0 < kend; k0 += GBK) {
#pragma unroll
    for (int i = 0; i < TT; ++i) {
      const int e = tid + i * 256;
      const int mm = A_KC ? (e >> 4) : (e % GBM);
      const int kk = A_KC ? (e & 15) : (e / GBM);
      const long long gm = m0 + mm, gk = k0 + kk;
      As[kk][mm] = (gm < Mz && gk < kend) ? A[gm * g.sAm + gk * g.sAk] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < TT; ++i) {
      const int e = tid + i * 256;
      const int nn = B_KC ? (e >> 4) : (e % GBN);
      const int kk = B_KC ? (e & 15) : (e / GBN);
      const long long gn = n0 + nn, gk = k0 + kk;
      Bs[kk][nn] = (gn < g.N && gk < kend) ? B[gn * g.sBn + gk * g.sBk] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GBK; ++kk) {
      double a[TT], b[TT];
#pragma unroll
      for (int i = 0; i < TT; ++i) a[i] = As[kk][ty * TT + i];
#pragma unroll
      for (int j = 0; j < TT; ++j) b[j] = Bs[kk][tx * TT + j];
#pragma unroll
      for (int i = 0; i < TT; ++i)
#pragma unroll
        for (int j = 0; j < TT; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < TT; ++i) {
    const int m = m0 + ty * TT + i;
    if (m >= Mz) continue;
    if (SCATTER) {
      const int mu = g.colmu[m], nu = g.colnu[m];
      if (mu < 0) continue;
      double *o1 = g.out + ((long long)mu * g.nao + nu) * g.ldo;
      double *o2 = g.out + ((long long)nu * g.nao + mu) * g.ldo;
#pragma unroll
      for (int j = 0; j < TT; ++j) {
        const int n = n0 + tx * TT + j;
        if (n < g.N) {
          o1[n] = acc[i][j];
          if (mu != nu) o2[n] = acc[i][j];
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < TT; ++j) {
        const int n = n0 + tx * TT + j;
        if (n >= g.N) continue;
        double *c = C + m * g.sCm + n * g.sCn;
        *c = (g.beta != 0.0) ? fma(g.alpha, acc[i][j], g.beta * *c) : g.alpha * acc[i][j];
      }
    }
  }
}

template <int TILE>
static void gemm_f64_launch(const GemmArgs &g, cudaStream_t st) {
  const int nz = g.k_split > 0 ? ceil_div(g.K, g.k_split) : g.batch;
  if (nz <= 0) return;
  dim3 grid(ceil_div(g.N, TILE), ceil_div(g.M, TILE), nz);
  if (grid.y > 65535 || grid.z > 65535) throw Error{DFJK_ERR_ARG, "gemm grid too large"};
  const bool akc = g.sAk == 1, bkc = g.sBk == 1, sc = g.out != nullptr;
  if (sc) {
    if (akc && bkc) gemm_f64_kernel<TILE, true, true, true><<<grid, 256, 0, st>>>(g);
    else throw Error{DFJK_ERR_ARG, "scatter gemm needs K-contiguous operands"};
  } else if (akc && bkc) {
    gemm_f64_kernel<TILE, true, true, false><<<grid, 256, 0, st>>>(g);
  } else if (akc && !bkc) {
    gemm_f64_kernel<TILE, true, false, false><<<grid, 256, 0, st>>>(g);
  } else if (!akc && bkc) {
    gemm_f64_kernel<TILE, false, true, false><<<grid, 256, 0, st>>>(g);
  } else {
    gemm_f64_kernel<TILE, false, false, false><<<grid, 256, 0, st>>>(g);
  }
  DFJK_LAUNCHED();
}

void gemm_f64(const GemmArgs &g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return;
  if (g.tile == 32) gemm_f64_launch<32>(g, st);
  else gemm_f64_launch<64>(g, st);
}

// ---- Cholesky -------------------------------------------------------------------

constexpr int NB = CHOL_NB;

// 1 / sqrt(d) for a positive normal d: FP32 estimate, one third-order step (2^-23 ->
// below 2^-60), no division.
__device__ __forceinline__ double rsqrt_chain(double d) {
  // the estimate of the mantissa in [1, 4), the even part of the exponent apart
  const int hi = __double2hiint(d), ex = ((hi >> 20) - 1023) >> 1;  // floor(exponent / 2)
  const double m = __hiloint2double(hi - (ex << 21), __double2loint(d));
  const double y = (double)rsqrtf((float)m);
  const double e = fma(-m * y, y, 1.0);
  const double r = fma(y * e, fma(e, 0.375, 0.5), y);
  return __hiloint2double(__double2hiint(r) - (ex << 20), __double2loint(r));
}

// Factors the 32 x 32 lower block at A in place (upper part zeroed) and writes its
// inverse (lower triangular) to Dinv and to Linv (row pitch ldi).  A non-positive or
// non-finite pivot (or one below the normal range) sets STATUS_NOT_PD and continues
// with pivot 1 so no NaN spreads.  Warps 0-3 factor: thread (row = lane, warp w) holds columns w, w + 4, .. in
// registers; the warp of column j + 1 updates that column first, takes its pivot and
// publishes the column while the others finish step j.  Warps 4-7 form the inverse
// one step behind (thread: column = lane, rows w, w + 4, ..) from the same published
// columns.  An FP64 instruction of one warp takes 64 cycles here (1/4 of the SM's two
// lanes per cycle), so the chain is the pivot's eight dependent ones per column: one
// barrier per column, all four schedulers busy.  256 threads with three barriers per
// column, a square root and a division took 46 us, one warp alone 54 us, this 29 us
// (the chain's eight instructions and the other warps' 500 cycles per column share the
// FP64 lanes).
__global__ void __launch_bounds__(256) potrf_diag_kernel(double *A, int lda, double *Dinv, double *Linv, int ldi,
                                                         int *status) {
  __shared__ double sm[NB][NB + 1];
  __shared__ double col[4][NB], row[4][NB], rdiag[NB];
  const int tid = threadIdx.x, lane = tid & 31, w = (tid >> 5) & 3;
  const bool fac = tid < 128;
  for (int i = tid >> 5; i < NB; i += 8) sm[i][lane] = lane <= i ? A[(long long)i * lda + lane] : 0.0;
  __syncthreads();
  double r[8];  // factor: columns 4 q + w of row `lane`; inverse: rows 4 q + w of column `lane`
#pragma unroll
  for (int q = 0; q < 8; ++q) r[q] = fac ? sm[lane][4 * q + w] : (4 * q + w == lane ? 1.0 : 0.0);
  const auto pivot = [&](int j, double &x) {  // x: column j of this row, up to date
    double d = __shfl_sync(0xffffffffu, x, j);
    if (!(d >= 2.2250738585072014e-308) || !isfinite(d)) {
      if (lane == 0) atomicOr(status, STATUS_NOT_PD);
      d = 1.0;
    }
    const double y = rsqrt_chain(d);
    double v = x * y;
    if (lane == j) {
      const double l = d * y;
      v = fma(fma(-l, l, d), 0.5 * y, l);
      rdiag[j] = y;
    }
    x = lane >= j ? v : 0.0;
    col[j & 3][lane] = x;
  };
  if (fac && w == 0) pivot(0, r[0]);
  __syncthreads();
#pragma unroll
  for (int j = 0; j < NB; ++j) {  // column j is published in col[j & 3]
    if (fac) {
      const double v = col[j & 3][lane];
      const bool next = j + 1 < NB && w == ((j + 1) & 3);
      if (next) {
        r[(j + 1) >> 2 & 7] = fma(-v, col[j & 3][(j + 1) & 31], r[(j + 1) >> 2 & 7]);
        pivot(j + 1, r[(j + 1) >> 2 & 7]);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int c = 4 * q + w;
        if (c > j + (next ? 1 : 0)) r[q] = fma(-v, col[j & 3][c], r[q]);
      }
    } else {
      // row j - 1 of the inverse is published in row[(j - 1) & 3]: update the later
      // rows, then publish row j
      if (j > 0) {
        const double x = row[(j - 1) & 3][lane];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int i = 4 * q + w;
          if (i >= j) r[q] = fma(-col[(j - 1) & 3][i], x, r[q]);
        }
      }
      if (w == (j & 3)) {
        r[j >> 2] *= rdiag[j];
        row[j & 3][lane] = r[j >> 2];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = 4 * q + w;
    if (fac) {
      sm[lane][k] = k <= lane ? r[q] : 0.0;
    } else {
      Dinv[k * NB + lane] = r[q];
      Linv[(long long)k * ldi + lane] = r[q];
    }
  }
  __syncthreads();
  for (int i = tid >> 5; i < NB; i += 8) A[(long long)i * lda + lane] = sm[i][lane];
}

// C = A B^T (sub = 0, in place when C = A) or C -= A B^T for `rows` rows of 32 columns and
// K = 32: the panel L_ik = A_ik Dinv_k^T and the next block column's update, both
// on the critical path.  A block takes 8 rows, so a panel of 2000 rows covers the
// GPU and a block's 8192 multiply-adds take 4k cycles (32-row tiles: 16k).
__global__ void __launch_bounds__(256) chol_skinny_kernel(const double *A, long long lda, const double *__restrict__ B,
                                                          long long ldb, double *C, long long ldc, int rows, int sub) {
  __shared__ double As[8][NB + 1], Bs[NB][NB + 1];
  const int c = threadIdx.x & 31, q = threadIdx.x >> 5, row = blockIdx.x * 8 + q;
  if (row < rows) As[q][c] = A[row * lda + c];
#pragma unroll
  for (int i = 0; i < NB; i += 8) Bs[i + q][c] = B[(i + q) * ldb + c];
  const double old = sub && row < rows ? C[row * ldc + c] : 0.0;
  __syncthreads();
  double s0 = 0.0, s1 = 0.0;
#pragma unroll
  for (int k = 0; k < NB; k += 2) {
    s0 = fma(As[q][k], Bs[c][k], s0);
    s1 = fma(As[q][k + 1], Bs[c][k + 1], s1);
  }
  if (row < rows) C[row * ldc + c] = sub ? old - (s0 + s1) : s0 + s1;
}

static void chol_skinny(const double *A, long long lda, const double *B, long long ldb, double *C, long long ldc,
                        int rows, int sub, cudaStream_t st) {
  chol_skinny_kernel<<<ceil_div(rows, 8), 256, 0, st>>>(A, lda, B, ldb, C, ldc, rows, sub);
  DFJK_LAUNCHED();
}

// Merges two neighbouring inverted diagonal blocks, rows [at, at + s) and [at + s, at + s +
// valid): the lower-left block of the merged inverse is -Linv22 (L21 Linv11).
static void merge_inverse(const double *L, int ld, double *Linv, int at, int s, int valid, double *work,
                          cudaStream_t st) {
  const double *L21 = L + (long long)(at + s) * ld + at;
  double *I11 = Linv + (long long)at * ld + at, *I21 = Linv + (long long)(at + s) * ld + at;
  const double *I22 = Linv + (long long)(at + s) * (ld + 1);
  GemmArgs a;  // work = L21 Linv11
  a.M = valid; a.N = s; a.K = s;
  a.A = L21; a.sAm = ld; a.sAk = 1;
  a.B = I11; a.sBn = 1; a.sBk = ld;
  a.C = work; a.sCm = s; a.sCn = 1;
  a.k_from_n = 1;  // Linv11 lower triangular: B(n, k) = Linv11[k][n] = 0 for k < n
  a.tile = 32;
  gemm_f64(a, st);
  GemmArgs b;  // Linv21 = -Linv22 work
  b.M = valid; b.N = s; b.K = valid;
  b.A = I22; b.sAm = ld; b.sAk = 1;
  b.B = work; b.sBn = 1; b.sBk = s;
  b.C = I21; b.sCm = ld; b.sCn = 1;
  b.alpha = -1.0;
  b.k_upto_m = 1;  // Linv22 lower triangular: A(m, k) = 0 for k > m
  b.tile = 32;
  gemm_f64(b, st);
}

void cholesky_inverse_f64(double *A, int n, int lda, double *Dinv, double *Linv, double *work, int *status,
                          const CholStreams &cs) {
  const cudaStream_t st = cs.chain, st2 = cs.bulk, st3 = cs.inverse;
  DFJK_CUDA_CHECK(cudaMemsetAsync(Linv, 0, sizeof(double) * (size_t)n * lda, st));
  const int nb = n / NB;
  bool bulk_pending = false;
  for (int k = 0; k < nb; ++k) {
    double *Akk = A + (long long)k * NB * lda + k * NB;
    double *Dk = Dinv + (long long)k * NB * NB;
    potrf_diag_kernel<<<1, 256, 0, st>>>(Akk, lda, Dk, Linv + (long long)k * NB * (lda + 1), lda, status);
    DFJK_LAUNCHED();
    const int rows = n - (k + 1) * NB;
    double *panel = Akk + (long long)NB * lda;
    if (rows > 0) chol_skinny(panel, lda, Dk, NB, panel, lda, rows, 0, st);  // L_ik = A_ik Dinv_k^T
    // the inverse blocks that are complete with this diagonal block and panel
    const int done = (k + 1) * NB;
    if (k > 0) {
      DFJK_CUDA_CHECK(cudaEventRecord(cs.ev_done, st));
      DFJK_CUDA_CHECK(cudaStreamWaitEvent(st3, cs.ev_done, 0));
      for (int s = NB; s < n; s *= 2) {
        if (done % (2 * s) == 0) {
          merge_inverse(A, lda, Linv, done - 2 * s, s, s, work, st3);
        } else if (done == n) {  // the ragged last pair of this level
          const int at = n / (2 * s) * (2 * s);
          if (at + s < n) merge_inverse(A, lda, Linv, at, s, n - at - s, work, st3);
        }
      }
    }
    if (rows <= 0) break;
    // look-ahead: the next block column (k + 1) is updated on the critical stream, so
    // the next diagonal block can start, while the rest of the trailing matrix
    // (block columns >= k + 2) is updated on the second stream; block column k + 1
    // also receives the second stream's earlier updates, which must have landed first
    DFJK_CUDA_CHECK(cudaEventRecord(cs.ev_panel, st));
    if (bulk_pending) DFJK_CUDA_CHECK(cudaStreamWaitEvent(st, cs.ev_bulk, 0));
    chol_skinny(panel, lda, panel, lda, A + (long long)(k + 1) * NB * (lda + 1), lda, rows, 1, st);
    const int rest = rows - NB;
    if (rest > 0) {
      DFJK_CUDA_CHECK(cudaStreamWaitEvent(st2, cs.ev_panel, 0));
      GemmArgs t;  // A_ij -= L_ik L_jk^T for block rows and columns >= k + 2
      t.M = rest; t.N = rest; t.K = NB;
      t.A = panel + (long long)NB * lda; t.sAm = lda; t.sAk = 1;
      t.B = panel + (long long)NB * lda; t.sBn = lda; t.sBk = 1;
      t.C = A + (long long)(k + 2) * NB * (lda + 1); t.sCm = lda; t.sCn = 1;
      t.alpha = -1.0; t.beta = 1.0; t.lower_only = 1;
      t.tile = 32;
      gemm_f64(t, st2);
      DFJK_CUDA_CHECK(cudaEventRecord(cs.ev_bulk, st2));
      bulk_pending = true;
    }
  }
  DFJK_CUDA_CHECK(cudaEventRecord(cs.ev_done, st3));
  DFJK_CUDA_CHECK(cudaStreamWaitEvent(st, cs.ev_done, 0));
}

// ---- J: rho = B vec(D), J = B^T rho ------------------------------------------------

__device__ __forceinline__ void tri_row(long long r, int &mu, int &nu) {
  int m = (int)((sqrt(8.0 * (double)r + 1.0) - 1.0) * 0.5);
  while ((long long)m * (m + 1) / 2 > r) --m;
  while ((long long)(m + 1) * (m + 2) / 2 <= r) ++m;
  mu = m;
  nu = (int)(r - (long long)m * (m + 1) / 2);
}

__global__ void column_sum_kernel(const double *__restrict__ work, int ldw, int nrow, int n,
                                  double *__restrict__ out) {
  const int P = blockIdx.x * blockDim.x + threadIdx.x;
  if (P >= n) return;
  double s = 0.0;
  for (int r = 0; r < nrow; ++r) s += work[(long long)r * ldw + P];
  out[P] = s;
}

// part[mu][P] = sum_i C[mu][i] X[mu][P][i]: one warp per (mu, P), lanes along i.
__global__ void __launch_bounds__(256) rho_from_x_kernel(const double *__restrict__ X,
                                                         const double *__restrict__ C, int nao, int np,
                                                         int nocc, double *__restrict__ part) {
  const long long w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= (long long)nao * np) return;
  const int mu = (int)(w / np);
  const double *x = X + w * nocc;
  const double *c = C + (long long)mu * nocc;
  double s = 0.0;
  for (int i = lane; i < nocc; i += 32) s = fma(__ldg(c + i), x[i], s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) part[w] = s;
}

void rho_from_x_f64(const double *X, const double *C, int nao, int np, int nocc, double *rho,
                    double *part, cudaStream_t st) {
  const long long n = (long long)nao * np;
  rho_from_x_kernel<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(X, C, nao, np, nocc, part);
  DFJK_LAUNCHED();
  column_sum_kernel<<<ceil_div(np, 256), 256, 0, st>>>(part, np, nao, np, rho);
  DFJK_LAUNCHED();
}

// J[mu][nu] = J[nu][mu] = B_row . rho, one warp per pair: the mu >= nu pairs
// (colmu null) or the kept columns (J of the other pairs is 0, set before), stored
// as row mu nao + nu (full) or as row r.
__global__ void __launch_bounds__(256) j_gemv_kernel(const double *__restrict__ B, long long ldb, long long nrows,
                                                     int nao, int naux, const double *__restrict__ rho,
                                                     double *__restrict__ J, const int *__restrict__ colmu,
                                                     const int *__restrict__ colnu, int full) {
  const long long r = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= nrows) return;
  int mu, nu;
  if (colmu) {
    mu = colmu[r];
    nu = colnu[r];
    if (mu < 0) return;
  } else {
    tri_row(r, mu, nu);
  }
  const double *row = B + (full ? (long long)mu * nao + nu : r) * ldb;
  double s = 0.0;
  if ((naux & 1) == 0 && (ldb & 1) == 0) {  // 16-byte loads, two partial sums, 4 loads in flight
    const double2 *row2 = reinterpret_cast<const double2 *>(row);
    const double2 *rho2 = reinterpret_cast<const double2 *>(rho);
    double s1 = 0.0;
#pragma unroll 4
    for (int q = lane; q < naux / 2; q += 32) {
      const double2 b = row2[q], x = __ldg(rho2 + q);
      s = fma(b.x, x.x, s);
      s1 = fma(b.y, x.y, s1);
    }
    s += s1;
  } else {
    for (int P = lane; P < naux; P += 32) s = fma(row[P], __ldg(rho + P), s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    J[(long long)mu * nao + nu] = s;
    J[(long long)nu * nao + mu] = s;
  }
}

void j_gemv_f64(const double *B, long long ldb, int nao, int naux, const double *rho, double *J, cudaStream_t st) {
  const long long nrows = (long long)nao * (nao + 1) / 2;
  j_gemv_kernel<<<(unsigned)((nrows + 7) / 8), 256, 0, st>>>(B, ldb, nrows, nao, naux, rho, J, nullptr, nullptr, 1);
  DFJK_LAUNCHED();
}

void j_kept_f64(const double *B, long long ldb, long long ncol, const int *colmu, const int *colnu, int nao,
                bool full, int naux, const double *rho, double *J, cudaStream_t st) {
  DFJK_CUDA_CHECK(cudaMemsetAsync(J, 0, sizeof(double) * (size_t)nao * nao, st));
  if (ncol == 0) return;
  j_gemv_kernel<<<(unsigned)((ncol + 7) / 8), 256, 0, st>>>(B, ldb, ncol, nao, naux, rho, J, colmu, colnu, full ? 1 : 0);
  DFJK_LAUNCHED();
}

// Partial sums of rho = B vec D over the stored columns: part y of the columns, 128
// P per block, the weights of 128 columns at a time in shared memory.
__global__ void __launch_bounds__(128) rho_kept_kernel(const double *__restrict__ B, long long ldb, long long ncol,
                                                       const int *__restrict__ colmu, const int *__restrict__ colnu,
                                                       int nao, int full, const double *__restrict__ D, int np,
                                                       long long per, double *__restrict__ work) {
  __shared__ double w[128];
  __shared__ long long row[128];
  const int P = blockIdx.x * 128 + threadIdx.x;
  const long long m0 = blockIdx.y * per, m1 = min(ncol, m0 + per);
  double s = 0.0;
  for (long long m = m0; m < m1; m += 128) {
    const long long q = m + threadIdx.x;
    double x = 0.0;
    long long at = full ? 0 : q;
    if (q < m1) {
      const int mu = colmu[q], nu = colnu[q];
      if (mu >= 0) {
        const long long e = (long long)mu * nao + nu;
        x = D[e] * (mu == nu ? 1.0 : 2.0);
        if (full) at = e;
      }
    }
    __syncthreads();
    w[threadIdx.x] = x;
    row[threadIdx.x] = at * ldb;
    __syncthreads();
    const int n = (int)min(m1 - m, 128LL);
    if (P < np) {
      const double *b = B + P;
#pragma unroll 8
      for (int k = 0; k < n; ++k) s = fma(w[k], b[row[k]], s);
    }
  }
  if (P < np) work[(long long)blockIdx.y * np + P] = s;
}

void rho_kept_f64(const double *B, long long ldb, long long ncol, const int *colmu, const int *colnu, int nao,
                  bool full, const double *D, int np, double *rho, double *work, cudaStream_t st) {
  // the split of the columns depends on their number alone, so that a part of
  // the rows P (a chunk of a host-resident B) sums in the same order
  const int parts = (int)std::max<long long>(1, std::min<long long>(RHO_PARTS, ncol / 64));
  const long long per = std::max<long long>(1, (ncol + parts - 1) / parts);
  rho_kept_kernel<<<dim3(ceil_div(np, 128), parts), 128, 0, st>>>(B, ldb, ncol, colmu, colnu, nao, full ? 1 : 0, D, np, per, work);
  DFJK_LAUNCHED();
  column_sum_kernel<<<ceil_div(np, 256), 256, 0, st>>>(work, np, parts, np, rho);
  DFJK_LAUNCHED();
}

// Bfull[(mu nao + nu) ldb + P] = Bc[rowmap[mu nao + nu] ldb + P] (0 where the
// map is -1): one block per (mu, nu) pair, threads along P (coalesced).
__global__ void __launch_bounds__(256) unpack_rows_kernel(const double *__restrict__ Bc, long long ldb, int nao,
                                                          const int *__restrict__ rowmap, double *__restrict__ Bf) {
  const long long e = blockIdx.x;  // mu nao + nu
  const int row = rowmap[e];
  double *dst = Bf + e * ldb;
  if (row < 0) {
    for (long long P = threadIdx.x; P < ldb; P += 256) dst[P] = 0.0;
    return;
  }
  const double *src = Bc + (long long)row * ldb;
  for (long long P = threadIdx.x; P < ldb; P += 256) dst[P] = src[P];
}

void unpack_rows_f64(const double *Bc, long long ldb, int nao, const int *rowmap, double *Bfull, cudaStream_t st) {
  const long long n2 = (long long)nao * nao;
  if (n2 == 0) return;
  unpack_rows_kernel<<<(unsigned)n2, 256, 0, st>>>(Bc, ldb, nao, rowmap, Bfull);
  DFJK_LAUNCHED();
}

// rowmap[mu nao + nu] = rowmap[nu nao + mu] = m for every column m with
// colmu[m] >= 0 (the map is -1 elsewhere).
__global__ void build_rowmap_kernel(const int *__restrict__ colmu, const int *__restrict__ colnu, long long ncol,
                                    int nao, int *__restrict__ rowmap) {
  const long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= ncol) return;
  const int mu = colmu[m], nu = colnu[m];
  if (mu < 0) return;
  rowmap[(long long)mu * nao + nu] = (int)m;
  rowmap[(long long)nu * nao + mu] = (int)m;
}

void build_rowmap(const int *colmu, const int *colnu, long long ncol, int nao, int *rowmap, cudaStream_t st) {
  DFJK_CUDA_CHECK(cudaMemsetAsync(rowmap, 0xFF, (size_t)nao * nao * sizeof(int), st));
  if (ncol == 0) return;
  build_rowmap_kernel<<<(unsigned)((ncol + 255) / 256), 256, 0, st>>>(colmu, colnu, ncol, nao, rowmap);
  DFJK_LAUNCHED();
}

// ---- reductions -----------------------------------------------------------------------

__global__ void reduce_sym_kernel(const double *__restrict__ part, int nsplit, int n,
                                  double *__restrict__ out, int add) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n * n) return;
  const int mu = (int)(e / n), nu = (int)(e % n);
  if (nu > mu) return;
  double s = add ? out[e] : 0.0;
  for (int k = 0; k < nsplit; ++k) s += part[(long long)k * n * n + e];
  out[e] = s;
  out[(long long)nu * n + mu] = s;
}

void reduce_sym_f64(const double *part, int nsplit, int n, double *out, cudaStream_t st, int add) {
  const long long n2 = (long long)n * n;
  reduce_sym_kernel<<<(unsigned)((n2 + 255) / 256), 256, 0, st>>>(part, nsplit, n, out, add);
  DFJK_LAUNCHED();
}

__global__ void mirror_lower_kernel(double *__restrict__ K, int n) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n * n) return;
  const int mu = (int)(e / n), nu = (int)(e % n);
  if (nu > mu) K[e] = K[(long long)nu * n + mu];
}

void mirror_lower_f64(double *K, int n, cudaStream_t st) {
  const long long n2 = (long long)n * n;
  mirror_lower_kernel<<<(unsigned)((n2 + 255) / 256), 256, 0, st>>>(K, n);
  DFJK_LAUNCHED();
}

constexpr int EN_BLOCKS = 256;

__global__ void __launch_bounds__(256) energy_partial_kernel(const double *__restrict__ D,
                                                             const double *__restrict__ J,
                                                             const double *__restrict__ K,
                                                             long long n2, double *work) {
  __shared__ double sj[256], sk[256];
  double aj = 0.0, ak = 0.0;
  for (long long e = (long long)blockIdx.x * 256 + threadIdx.x; e < n2; e += (long long)EN_BLOCKS * 256) {
    aj = fma(D[e], J[e], aj);
    ak = fma(D[e], K[e], ak);
  }
  sj[threadIdx.x] = aj;
  sk[threadIdx.x] = ak;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      sj[threadIdx.x] += sj[threadIdx.x + s];
      sk[threadIdx.x] += sk[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    work[2 * blockIdx.x] = sj[0];
    work[2 * blockIdx.x + 1] = sk[0];
  }
}

__global__ void energy_final_kernel(const double *__restrict__ work, double *e) {
  __shared__ double sj[EN_BLOCKS], sk[EN_BLOCKS];
  sj[threadIdx.x] = work[2 * threadIdx.x];
  sk[threadIdx.x] = work[2 * threadIdx.x + 1];
  __syncthreads();
  for (int s = EN_BLOCKS / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      sj[threadIdx.x] += sj[threadIdx.x + s];
      sk[threadIdx.x] += sk[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    e[0] = 0.5 * sj[0];
    e[1] = 0.5 * sk[0];
  }
}

void energies_f64(const double *D, const double *J, const double *K, int n, double *e,
                  double *work, cudaStream_t st) {
  energy_partial_kernel<<<EN_BLOCKS, 256, 0, st>>>(D, J, K, (long long)n * n, work);
  DFJK_LAUNCHED();
  energy_final_kernel<<<1, EN_BLOCKS, 0, st>>>(work, e);
  DFJK_LAUNCHED();
}

__global__ void max_sqrt_diag_kernel(const double *V, int n, int ld, double *out) {
  __shared__ double s[256];
  double m = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) m = fmax(m, sqrt(fmax(V[(long long)i * ld + i], 0.0)));
  s[threadIdx.x] = m;
  __syncthreads();
  for (int k = 128; k > 0; k >>= 1) {
    if (threadIdx.x < k) s[threadIdx.x] = fmax(s[threadIdx.x], s[threadIdx.x + k]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = s[0];
}

void max_sqrt_diag(const double *V, int n, int ld, double *out, cudaStream_t st) {
  max_sqrt_diag_kernel<<<1, 256, 0, st>>>(V, n, ld, out);
  DFJK_LAUNCHED();
}

__global__ void screen_kernel(const double *q, int n, const double *maxdiag, double thresh,
                              int *keep) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) keep[i] = (q[i] * (*maxdiag) >= thresh) ? 1 : 0;
}

void screen_pairs(const double *q, int n, const double *maxdiag, double thresh, int *keep,
                  cudaStream_t st) {
  if (n == 0) return;
  screen_kernel<<<ceil_div(n, 256), 256, 0, st>>>(q, n, maxdiag, thresh, keep);
  DFJK_LAUNCHED();
}

// Non-negative doubles order like their bits, so the maxima are of 32-bit integers (the
// FP64 pipe is the scarce one); bound by reading the arrays.
__global__ void __launch_bounds__(256) abs_max_kernel(AbsMax a, unsigned *out) {
  const double *x = a.x[blockIdx.y];
  const long long n = a.n[blockIdx.y];
  unsigned m = 0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256)
    m = max(m, (unsigned)__double2hiint(x[i]) & 0x7FFFFFFFu);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(out + blockIdx.y, m);
}

void abs_max(const AbsMax &a, unsigned *out, cudaStream_t st) {
  long long most = 1;
  for (long long n : a.n) most = std::max(most, n);
  DFJK_CUDA_CHECK(cudaMemsetAsync(out, 0, 4 * sizeof(unsigned), st));
  abs_max_kernel<<<dim3((unsigned)std::min<long long>((most + 255) / 256, 152 * 8), 4), 256, 0, st>>>(a, out);
  DFJK_LAUNCHED();
}

double abs_max_value(unsigned hi) {
  const uint64_t u = (uint64_t)hi << 32;
  double v;
  std::memcpy(&v, &u, sizeof(v));
  return v;
}

__global__ void gather2d_kernel(const double *in, long long ldi, const int *pr, const int *pc,
                                int nr, int nc, double *out, long long ldo) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)nr * nc) return;
  const int i = (int)(e / nc), j = (int)(e % nc);
  out[i * ldo + j] = pr[i] < 0 ? 0.0 : in[(long long)pr[i] * ldi + pc[j]];
}

void gather2d_f64(const double *in, long long ldi, const int *perm_r, const int *perm_c, int nr,
                  int nc, double *out, long long ldo, cudaStream_t st) {
  const long long n = (long long)nr * nc;
  if (n == 0) return;
  gather2d_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, ldi, perm_r, perm_c, nr, nc, out, ldo);
  DFJK_LAUNCHED();
}

__global__ void gather_B_kernel(const double *Bint, long long ldb, int nao, const int *perm,
                                int naux, double *out, const int *rowmap) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n2 = (long long)nao * nao;
  if (e >= n2 * naux) return;
  const int P = (int)(e / n2);
  const long long mn = e % n2;
  const long long row = rowmap ? rowmap[mn] : mn;
  out[e] = row < 0 ? 0.0 : Bint[row * ldb + perm[P]];
}

void gather_B_f64(const double *Bint, long long ldb, int nao, const int *perm, int naux,
                  double *out, const int *rowmap, cudaStream_t st) {
  const long long n = (long long)nao * nao * naux;
  if (n == 0) return;
  gather_B_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(Bint, ldb, nao, perm, naux, out, rowmap);
  DFJK_LAUNCHED();
}

}  // namespace dfjk
