// Derivative 3-centre kernels of the DF Coulomb/exchange gradient, shared by the
// per-aux-class translation units grad3c_l{0,1,2}.cu (split so that they
// compile in parallel).  The scheme is described in grad.cu.
//
// With the pair's primitives expanded as sum_tuv E_tuv Lambda_tuv(P) and an aux
// function's as shifts of the Hermite index (W below), the derivatives of one
// primitive triple are
//   d/dC_q = -sum E_tuv W_{tuv + 1_q},
//   d/dA_q = (a/p) sum E_tuv W_{tuv + 1_q} + sum E'_{q,tuv} W_tuv,
// E'_q the derivative of E with respect to (A - B)_q at fixed P.  Everything that
// belongs to the pair alone is prepared once per primitive pair and read by every
// aux shell (grad_tables_kernel); the earlier kernels rebuilt it in every block.
//  * Coulomb alone: the weights c_j d_P D_mu nu factor, so the tables hold sums
//    over the component pairs, six numbers per Hermite index
//    (sum D dE/dA_q and sum D E shifted by 1_q), and the aux components are summed
//    into one W.
//  * exchange: the weights Gamma[mu nu][P] differ per aux function; the tables hold
//    E and E'_q per term, and a thread takes one aux function.
// The threads of an aux shell (one per component, adjacent lanes) share its R,
// built in shared memory.  Loops over terms are rolled and read their indices from
// small tables: the unrolled kernels before spilled their outputs (FP64 pipe 25 to
// 39 % busy in the dd classes) and their code did not fit the instruction caches.
// The arithmetic is FP64 for DFJK_FP64 handles, double-single for mixed ones (some
// 48 bits, five times the rate), and FP32 for the Coulomb weights of the pairs
// whose integrals the build takes in FP32.  Measured: E_J gradient
// at 45 atoms 33.5 -> 12.4 ms (FP64 and FP32 before; 9.7 with the classes on
// streams), E_J - E_K/2 at 30 atoms 60 -> 20.6 ms (16.1), FP64 handle at 12 atoms
// 23.3 -> 6.7 ms.  Errors of E_J gradients of mixed handles against 64-bit references (32
// molecules of 6 to 24 atoms, geometric mean of the largest relative ones): 6.8e-12; 6.7e-12
// with these kernels in FP64, 6.6e-12 with the integrals of the setup in FP64 as
// well, 7.5e-12 for the kernels before (the metric sets them); E_J - E_K/2 1.0e-9 as before.
#pragma once

#include "grad.cuh"
#include "md.cuh"

namespace dfjk {

// (t, u, v) of a dense Hermite index (the inverse of tuv_idx).
__device__ __forceinline__ void tuv_decode(int idx, int &t, int &u, int &v) {
  int N = 0;
  while (ntuv(N) <= idx) ++N;
  int r = idx - (N > 0 ? ntuv(N - 1) : 0), sl = 0;
  while ((sl + 1) * (sl + 2) / 2 <= r) ++sl;
  v = r - sl * (sl + 1) / 2;
  u = sl - v;
  t = N - sl;
}

// What a kernel reads (EriIn) and sums in.
template <typename Real>
struct GradIn : EriIn<Real> {
  using Acc = df;
  static __device__ __forceinline__ df acc(Real v) { return df(v); }
};
template <>
struct GradIn<df> : EriIn<df> {
  using Acc = df;
  static __device__ __forceinline__ df acc(df v) { return v; }
};
template <>
struct GradIn<double> : EriIn<double> {
  using Acc = double;
  static __device__ __forceinline__ double acc(double v) { return v; }
};
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ df shfl_xor(df v, int o) {
  return df(__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o));
}

// The terms (component pair, t, u, v) of a class in record order, packed as
// t | u << 3 | v << 6 | ca << 9 | cb << 12, and the first term of each component pair.
template <int LA, int LB>
struct GradTerms {
  int e[nterms(LA, LB)];
  int start[ncart(LA) * ncart(LB) + 1];
  constexpr GradTerms() : e(), start() {
    int k = 0;
    for (int ca = 0; ca < ncart(LA); ++ca)
      for (int cb = 0; cb < ncart(LB); ++cb) {
        start[ca * ncart(LB) + cb] = k;
        for (int t = 0; t <= cart_x(LA, ca) + cart_x(LB, cb); ++t)
          for (int u = 0; u <= cart_y(LA, ca) + cart_y(LB, cb); ++u)
            for (int v = 0; v <= cart_z(LA, ca) + cart_z(LB, cb); ++v) e[k++] = t | (u << 3) | (v << 6) | (ca << 9) | (cb << 12);
      }
    start[ncart(LA) * ncart(LB)] = k;
  }
};
template <int LA, int LB>
static __device__ const GradTerms<LA, LB> d_grad_terms{};

constexpr int GRAD_HDR = 6;  // p, Px, Py, Pz, c_a c_b K_ab 2 pi^(5/2)/p, a/p
// Values of a primitive pair's record.
__host__ __device__ constexpr int grad_rec_len(int la, int lb, bool exch) {
  return GRAD_HDR + (exch ? 4 * nterms(la, lb) : 6 * ntuv(la + lb + 1));
}

__device__ __forceinline__ void put_raw(double *o, double v) { *o = v; }
__device__ __forceinline__ void put_raw(float2 *o, double v) {
  const df r(v);
  *o = make_float2(r.h, r.l);
}

// The records of one kept pair per block, FP64 throughout, stored as doubles or as
// double-single pairs (centres relative to c0 then).
template <int LA, int LB, bool EXCH, typename Raw>
__global__ void __launch_bounds__(128) grad_tables_kernel(GradArgs g, OrbArgs orb, Raw *__restrict__ out) {
  constexpr int NCA = ncart(LA), NCB = ncart(LB), LAB = LA + LB;
  constexpr int EI = LA + 2, EJ = LB + 1, ET = LAB + 2;  // E[i <= LA+1][j <= LB][t <= LAB+1]
  constexpr int NT1 = ntuv(LAB + 1), NT0 = ntuv(LAB), NT = nterms(LA, LB);
  constexpr int LEN = grad_rec_len(LA, LB, EXCH);
  constexpr int KK = 4;  // primitive pairs at a time
  __shared__ double sE[KK][3][EI][EJ][ET];
  __shared__ double sR1[KK][3][LA + 1][EJ][ET];  // 2 alpha E^{i+1, j} - i E^{i-1, j}
  __shared__ double sHdr[KK][GRAD_HDR];
  __shared__ double sD[NCA * NCB], sH0[KK][NT0];
  const int tid = threadIdx.x;
  const int pair = g.pairs[blockIdx.x];
  const int sa = g.pair_a[pair], sb = g.pair_b[pair];
  const int mu0 = orb.func_off[sa], nu0 = orb.func_off[sb];
  if (!EXCH && tid < NCA * NCB) {
    const int ca = tid / NCB, cb = tid % NCB;
    sD[tid] = g.D[(long long)(mu0 + ca) * g.nao + nu0 + cb] * (sa == sb ? 1.0 : 2.0) *
              (comp_factor(LA, ca) * comp_factor(LB, cb));
  }
  const double A3[3] = {orb.center[3 * sa], orb.center[3 * sa + 1], orb.center[3 * sa + 2]};
  const double B3[3] = {orb.center[3 * sb], orb.center[3 * sb + 1], orb.center[3 * sb + 2]};
  double AB2 = 0.0;
  for (int q = 0; q < 3; ++q) AB2 += (A3[q] - B3[q]) * (A3[q] - B3[q]);
  const int pa0 = orb.prim_off[sa], na = orb.nprim[sa], pb0 = orb.prim_off[sb], nb = orb.nprim[sb];
  Raw *o0 = out + g.rec_off[blockIdx.x];
#pragma unroll 1
  for (int k0 = 0; k0 < na * nb; k0 += KK) {
    const int cnt = min(KK, na * nb - k0);
    __syncthreads();
    if (tid < 3 * cnt) {  // one thread per (primitive pair, direction) builds its tables
      const int k = tid / 3, dir = tid % 3, kk = k0 + k;
      const int ka = kk / nb, kb = kk % nb;
      const double a = orb.exps[pa0 + ka], b = orb.exps[pb0 + kb], p = a + b, ip_ = 1.0 / p;
      const double A = dir == 0 ? A3[0] : dir == 1 ? A3[1] : A3[2], Bc = dir == 0 ? B3[0] : dir == 1 ? B3[1] : B3[2];
      const double P = (a * A + b * Bc) * ip_;
      double E[EI][EJ][ET];
      hermite_E<LA + 1, LB>(0.5 * ip_, P - A, P - Bc, E);
#pragma unroll
      for (int i = 0; i < EI; ++i)
#pragma unroll
        for (int j = 0; j < EJ; ++j)
#pragma unroll
          for (int t = 0; t < ET; ++t) {
            sE[k][dir][i][j][t] = E[i][j][t];
            if (i <= LA) sR1[k][dir][i][j][t] = 2.0 * a * E[i + 1][j][t] - (i > 0 ? i * E[i - 1][j][t] : 0.0);
          }
      sHdr[k][1 + dir] = P - (dir == 0 ? g.c0[0] : dir == 1 ? g.c0[1] : g.c0[2]);
      if (dir == 0) {
        sHdr[k][0] = p;
        sHdr[k][4] = orb.coefs[pa0 + ka] * orb.coefs[pb0 + kb] * exp(-a * b * ip_ * AB2) *
                     (2.0 * 17.493418327624862846 * ip_);  // c_a c_b K_ab 2 pi^(5/2) / p
        sHdr[k][5] = a * ip_;
      }
    }
    __syncthreads();
    for (int e = tid; e < cnt * GRAD_HDR; e += blockDim.x)
      put_raw(o0 + (long long)(k0 + e / GRAD_HDR) * LEN + e % GRAD_HDR, sHdr[e / GRAD_HDR][e % GRAD_HDR]);
    if constexpr (EXCH) {
      for (int e = tid; e < cnt * NT; e += blockDim.x) {
        const int k = e / NT, w = d_grad_terms<LA, LB>.e[e % NT];
        const int t[3] = {w & 7, (w >> 3) & 7, (w >> 6) & 7}, ca = (w >> 9) & 7, cb = (w >> 12) & 7;
        const int ax[3] = {cart_x(LA, ca), cart_y(LA, ca), cart_z(LA, ca)};
        const int bx[3] = {cart_x(LB, cb), cart_y(LB, cb), cart_z(LB, cb)};
        const double f = comp_factor(LA, ca) * comp_factor(LB, cb), aop = sHdr[k][5];
        double e0[3], e1[3];
        for (int r = 0; r < 3; ++r) {
          e0[r] = sE[k][r][ax[r]][bx[r]][t[r]];
          e1[r] = sR1[k][r][ax[r]][bx[r]][t[r]] - (t[r] > 0 ? aop * sE[k][r][ax[r]][bx[r]][t[r] - 1] : 0.0);
        }
        Raw *o = o0 + (long long)(k0 + k) * LEN + GRAD_HDR + 4 * (e % NT);
        put_raw(o, f * e0[0] * e0[1] * e0[2]);
        put_raw(o + 1, f * e1[0] * e0[1] * e0[2]);
        put_raw(o + 2, f * e0[0] * e1[1] * e0[2]);
        put_raw(o + 3, f * e0[0] * e0[1] * e1[2]);
      }
    } else {
      // sums over the component pairs: q < 3 sum D dE/dA_q [tuv], q = 3 sum D E [tuv]
      constexpr int NH = 3 * NT1 + NT0;
      for (int ek = tid; ek < cnt * NH; ek += blockDim.x) {
        const int k = ek / NH, e = ek % NH, q = e < 3 * NT1 ? e / NT1 : 3;
        int tt[3];
        tuv_decode(q < 3 ? e - q * NT1 : e - 3 * NT1, tt[0], tt[1], tt[2]);
        double h = 0.0;
#pragma unroll 1
        for (int ca = 0; ca < NCA; ++ca)
#pragma unroll 1
          for (int cb = 0; cb < NCB; ++cb) {
            const int ax[3] = {cart_x(LA, ca), cart_y(LA, ca), cart_z(LA, ca)};
            const int bx[3] = {cart_x(LB, cb), cart_y(LB, cb), cart_z(LB, cb)};
            double f = sD[ca * NCB + cb];
            for (int r = 0; r < 3; ++r)
              f *= (r == q) ? sR1[k][r][ax[r]][bx[r]][tt[r]] : sE[k][r][ax[r]][bx[r]][tt[r]];
            h += f;
          }
        if (q < 3) put_raw(o0 + (long long)(k0 + k) * LEN + GRAD_HDR + 6 * (e - q * NT1) + q, h);
        else sH0[k][e - 3 * NT1] = h;
      }
      __syncthreads();
      for (int ek = tid; ek < cnt * 3 * NT1; ek += blockDim.x) {  // sum D E at tuv - 1_q
        const int k = ek / (3 * NT1), e = (ek / 3) % NT1, q = ek % 3;
        int t[3];
        tuv_decode(e, t[0], t[1], t[2]);
        --t[q];
        put_raw(o0 + (long long)(k0 + k) * LEN + GRAD_HDR + 6 * e + 3 + q,
                t[q] < 0 ? 0.0 : sH0[k][tuv_idx(t[0], t[1], t[2])]);
      }
    }
  }
}

// Gamma[(column of (a, b)) ld + P] = c (c_k G_P + c_j d_P D)[mu nu], c = 2 for a pair of
// different shells: one block per kept pair and 256 aux functions.
template <typename Raw>
__global__ void __launch_bounds__(256) grad_gamma_kernel(GradArgs g, OrbArgs orb, const long long *__restrict__ pair_col,
                                                         int nca, int ncb, int naux, Raw *__restrict__ out,
                                                         long long ld) {
  const int P = blockIdx.y * 256 + threadIdx.x;
  if (P >= naux) return;
  const int pair = g.pairs[blockIdx.x], sa = g.pair_a[pair], sb = g.pair_b[pair];
  const int mu0 = orb.func_off[sa], nu0 = orb.func_off[sb];
  const double c = sa == sb ? 1.0 : 2.0, dP = g.cj * g.d[P];
  const double *gp = g.gam + (long long)P * g.nao * g.nao;
  const long long col = pair_col[pair];
  for (int ca = 0; ca < nca; ++ca)
    for (int cb = 0; cb < ncb; ++cb) {
      const long long mn = (long long)(mu0 + ca) * g.nao + nu0 + cb;
      put_raw(out + (col + ca * ncb + cb) * ld + P, c * fma(dP, g.D[mn], g.ck * gp[mn]));
    }
}

// Shapes of the two kernels: NW warps of SPW aux shells, the odd pitches of the rows
// in shared memory (no bank conflicts between lanes) and its size.
template <int LAB, int LC, bool EXCH, typename Real, int NREC>
struct GradShape {
  static constexpr int L1 = LAB + LC + 1;
  // low orders of the Coulomb kernel: one thread per aux shell, R in registers
  static constexpr bool REGS = !EXCH && L1 <= 4;
  static constexpr int G = REGS ? 1 : ncart(LC), SPW = 32 / G;
  static constexpr int NR = ntuv(L1), NT1 = ntuv(LAB + 1);
  static constexpr int RP = NR | 1, WP = NT1 | 1;
  static constexpr int warp_bytes() {
    return ((REGS ? 0 : 2 * SPW * RP) + (EXCH && LC > 0 ? 32 * WP : 0)) * (int)sizeof(Real);
  }
  // up to 4 warps per block, at most about 100 KB (two blocks per SM)
  static constexpr int nw() {
    int n = 4;
    while (n > 1 && n * warp_bytes() + NREC * (int)sizeof(Real) > 100 * 1024) --n;
    return n;
  }
  static constexpr int NW = nw();
  static constexpr int NS = NW * SPW, THREADS = 32 * NW;
  static constexpr int SMEM = NW * warp_bytes() + NREC * (int)sizeof(Real);
};

// Adds a pair's block sums to the atoms of its shells (B = -(A + C)).
template <int NW, typename Acc>
__device__ __forceinline__ void add_pair(const GradArgs &g, int sa, int sb, const Acc *gA, const Acc *gCp,
                                         double (*sRed)[6]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Acc red[6];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    red[q] = gA[q];
    red[3 + q] = gCp[q];
  }
#pragma unroll
  for (int q = 0; q < 6; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) red[q] = red[q] + shfl_xor(red[q], o);
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < 6; ++q) sRed[warp][q] = (double)red[q];
  __syncthreads();
  if (threadIdx.x < 6) {
    const int q = threadIdx.x % 3;
    double a = 0.0, c = 0.0;
    for (int w = 0; w < NW; ++w) {
      a += sRed[w][q];
      c += sRed[w][3 + q];
    }
    atomicAdd(&g.grad[3 * (threadIdx.x < 3 ? g.orb_atom[sa] : g.orb_atom[sb]) + q], threadIdx.x < 3 ? a : -(a + c));
  }
}

// Coulomb weights alone: g.pair_chunk kept pairs per block (blockIdx.x), the aux
// shells of blockIdx.y.
template <int LAB, int LC, typename Real>
__global__ void __launch_bounds__(128) grad3c_j_kernel(GradArgs g, AuxArgs aux,
                                                       const typename EriIn<Real>::Tab *__restrict__ boys_tab) {
  using In = GradIn<Real>;
  using Acc = typename In::Acc;
  constexpr int NREC = GRAD_HDR + 6 * ntuv(LAB + 1);
  using Sh = GradShape<LAB, LC, false, Real, NREC>;
  constexpr int G = Sh::G, SPW = Sh::SPW, NT1 = Sh::NT1, NR = Sh::NR, NCC = ncart(LC), NSH = LC == 0 ? 1 : NCC + 1;
  extern __shared__ __align__(16) uint8_t gsm[];
  Real *Rb = reinterpret_cast<Real *>(gsm);
  Real *srec = Rb + (Sh::REGS ? 0 : Sh::NW * 2 * SPW * Sh::RP);
  __shared__ typename In::Pos sP[3];
  __shared__ int srt[NR];
  __shared__ uint8_t sidx[NT1 * NSH];  // Hermite index of e shifted by each term of the aux expansion
  __shared__ double sRed[Sh::NW][6];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < NR; i += blockDim.x) srt[i] = c_rec.e[i];
  for (int i = tid; i < NT1 * NSH; i += blockDim.x) {
    int t, u, v;
    tuv_decode(i / NSH, t, u, v);
    const int s = i % NSH;  // 0: none, s > 0: component s - 1's powers
    sidx[i] = (uint8_t)(s == 0 ? tuv_idx(t, u, v)
                               : tuv_idx(t + cart_x(LC, s - 1), u + cart_y(LC, s - 1), v + cart_z(LC, s - 1)));
  }
  const int gr = lane / G, cc = lane - gr * G;
  const bool used = lane < SPW * G;
  const int slot = warp * SPW + (used ? gr : 0), as = blockIdx.y * Sh::NS + slot;
  const bool active = used && as < g.naux_shells;
  const int sc = active ? g.aux_shells[as] : 0;
  const typename In::Raw *cen = In::center(aux) + 3 * sc;
  const typename In::Pos Cx = In::pos(cen[0]), Cy = In::pos(cen[1]), Cz = In::pos(cen[2]);
  const int pc0 = aux.prim_off[sc], nc = active ? aux.nprim[sc] : 0;
  int ncmax = nc;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ncmax = max(ncmax, __shfl_xor_sync(0xffffffffu, ncmax, o));
  Real dP[NCC];
#pragma unroll
  for (int k = 0; k < NCC; ++k) dP[k] = Real(active ? g.cj * g.d[aux.func_off[sc] + k] * comp_factor(LC, k) : 0.0);
  Acc gC[3] = {Acc(0), Acc(0), Acc(0)};
  Real *R0 = Rb + slot * 2 * Sh::RP, *R1 = R0 + Sh::RP;
  const int p0 = blockIdx.x * g.pair_chunk, p1 = min(g.npairs, p0 + g.pair_chunk);
#pragma unroll 1
  for (int ip = p0; ip < p1; ++ip) {
    const int pair = g.pairs[ip], npp = g.npp[pair];
    const typename In::Raw *rec0 = static_cast<const typename In::Raw *>(g.rec) + g.rec_off[ip];
    Acc gA[3] = {Acc(0), Acc(0), Acc(0)}, gCp[3] = {Acc(0), Acc(0), Acc(0)};
#pragma unroll 1
    for (int ipp = 0; ipp < npp; ++ipp) {
      __syncthreads();
      for (int i = tid; i < NREC; i += blockDim.x) {
        const typename In::Raw v = rec0[(long long)ipp * NREC + i];
        srec[i] = In::real(v);
        if (i >= 1 && i <= 3) sP[i - 1] = In::pos(v);
      }
      __syncthreads();
      const Real X = In::diff(sP[0], Cx), Y = In::diff(sP[1], Cy), Z = In::diff(sP[2], Cz), p = srec[0];
#pragma unroll 1
      for (int kc = 0; kc < ncmax; ++kc) {
        const bool live = kc < nc;
        const Real gm = live ? In::real(In::exps(aux)[pc0 + kc]) : Real(1);
        const Real g1 = live ? In::real(In::g1(aux)[pc0 + kc]) : Real(0);
        const Real s = real_rsqrt(p + gm);
        const Real al = p * gm * (s * s);
        Real F[Sh::L1 + 1];
        boys_eval<Sh::L1>(al * (X * X + Y * Y + Z * Z), boys_tab, F);
        // coefficients of the aux function sum: x: -1/(2g); xx: 1/(2g) and 1/(4g^2) with
        // shift 2; xy: 1/(4g^2)
        Real a[NSH];
        if (LC == 0) {
          a[0] = dP[0];
        } else if (LC == 1) {
          a[0] = Real(0);
#pragma unroll
          for (int k = 0; k < NCC; ++k) a[1 < NSH ? k + 1 : 0] = -(g1 * dP[k]);
        } else {
          Real sum = Real(0);
#pragma unroll
          for (int k = 0; k < NCC; ++k) {
            if (cart_x(LC, k) == 2 || cart_y(LC, k) == 2 || cart_z(LC, k) == 2) sum = sum + dP[k];
            a[1 < NSH ? k + 1 : 0] = g1 * (g1 * dP[k]);
          }
          a[0] = g1 * sum;
        }
        Real h[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) h[q] = Real(0);
        const Real *R = nullptr;
        if constexpr (Sh::REGS) {
          Real r[NR];
          hermite_R<Sh::L1, Real>(F, al, X, Y, Z, r);
#pragma unroll
          for (int N = 0; N <= LAB + 1; ++N)
#pragma unroll
            for (int t = N; t >= 0; --t)
#pragma unroll
              for (int u = N - t; u >= 0; --u) {
                const int v = N - t - u, e = tuv_idx(t, u, v);
                Real w = LC == 1 ? Real(0) : a[0] * r[e];
                if (LC > 0)
#pragma unroll
                  for (int k = 0; k < NCC; ++k)
                    w = acc_fma(a[1 < NSH ? k + 1 : 0], r[tuv_idx(t + cart_x(LC, k), u + cart_y(LC, k), v + cart_z(LC, k))], w);
                w = acc_done(w);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                  h[q] = acc_fma(srec[GRAD_HDR + 6 * e + q], w, h[q]);
                  if ((q == 0 ? t : q == 1 ? u : v) > 0) h[3 + q] = acc_fma(srec[GRAD_HDR + 6 * e + 3 + q], w, h[3 + q]);
                }
              }
        } else {
          R = build_R<Sh::L1, G, Real>(R0, R1, cc, used, srt, F, al, X, Y, Z);
        }
        if (live) {
          if constexpr (!Sh::REGS) {
#pragma unroll 1
            for (int e = cc; e < NT1; e += G) {
              Real w = Real(0);
#pragma unroll
              for (int k = (LC == 1 ? 1 : 0); k < NSH; ++k) w = acc_fma(a[k], R[sidx[e * NSH + k]], w);
              w = acc_done(w);
#pragma unroll
              for (int q = 0; q < 6; ++q) h[q] = acc_fma(srec[GRAD_HDR + 6 * e + q], w, h[q]);
            }
          }
          const Real pt = srec[4] * In::real(In::cdiv(aux)[pc0 + kc]) * s;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            gA[q] = gA[q] + In::acc(pt * acc_done(h[q]));
            gCp[q] = gCp[q] + In::acc(-(pt * acc_done(h[3 + q])));
          }
        }
        if (!Sh::REGS) __syncwarp();  // R reads done before the next primitive overwrites it
      }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) gC[q] = gC[q] + gCp[q];
    add_pair<Sh::NW>(g, g.pair_a[pair], g.pair_b[pair], gA, gCp, sRed);
  }
  if (active)
#pragma unroll
    for (int q = 0; q < 3; ++q) atomicAdd(&g.grad[3 * g.aux_atom[sc] + q], (double)gC[q]);
}

// Weights Gamma per aux function: a thread takes one component of an aux shell.
template <int LA, int LB, int LC, typename Real>
__global__ void __launch_bounds__(128) grad3c_x_kernel(GradArgs g, AuxArgs aux,
                                                       const typename EriIn<Real>::Tab *__restrict__ boys_tab) {
  using In = GradIn<Real>;
  using Acc = typename In::Acc;
  constexpr int LAB = LA + LB, NT = nterms(LA, LB), NREC = GRAD_HDR + 4 * NT, NAB = ncart(LA) * ncart(LB);
  using Sh = GradShape<LAB, LC, true, Real, NREC>;
  constexpr int G = Sh::G, SPW = Sh::SPW, NT1 = Sh::NT1, NR = Sh::NR;
  extern __shared__ __align__(16) uint8_t gsm[];
  Real *Rb = reinterpret_cast<Real *>(gsm);
  Real *Wb = Rb + Sh::NW * 2 * SPW * Sh::RP;
  Real *srec = Wb + (LC > 0 ? Sh::THREADS * Sh::WP : 0);
  __shared__ typename In::Pos sP[3];
  __shared__ int srt[NR];
  __shared__ int sterm[NT];        // Hermite indices of tuv, tuv + 1_x, + 1_y, + 1_z, one byte each
  __shared__ int sstart[NAB + 1];  // first term of each component pair
  __shared__ int stuv[NT1];        // t | u << 4 | v << 8
  __shared__ double sRed[Sh::NW][6];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < NR; i += blockDim.x) srt[i] = c_rec.e[i];
  for (int i = tid; i < NT; i += blockDim.x) {
    const int w = d_grad_terms<LA, LB>.e[i], t = w & 7, u = (w >> 3) & 7, v = (w >> 6) & 7;
    sterm[i] = tuv_idx(t, u, v) | (tuv_idx(t + 1, u, v) << 8) | (tuv_idx(t, u + 1, v) << 16) | (tuv_idx(t, u, v + 1) << 24);
  }
  for (int i = tid; i <= NAB; i += blockDim.x) sstart[i] = d_grad_terms<LA, LB>.start[i];
  for (int i = tid; i < NT1; i += blockDim.x) {
    int t, u, v;
    tuv_decode(i, t, u, v);
    stuv[i] = t | (u << 4) | (v << 8);
  }
  const int gr = lane / G, cc = lane - gr * G;
  const bool used = lane < SPW * G;
  const int slot = warp * SPW + (used ? gr : 0), as = blockIdx.y * Sh::NS + slot;
  const bool active = used && as < g.naux_shells;
  const int sc = active ? g.aux_shells[as] : 0;
  const typename In::Raw *cen = In::center(aux) + 3 * sc;
  const typename In::Pos Cx = In::pos(cen[0]), Cy = In::pos(cen[1]), Cz = In::pos(cen[2]);
  const int pc0 = aux.prim_off[sc], nc = active ? aux.nprim[sc] : 0;
  int ncmax = nc;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ncmax = max(ncmax, __shfl_xor_sync(0xffffffffu, ncmax, o));
  const int cx = cart_x(LC, cc), cy = cart_y(LC, cc), cz = cart_z(LC, cc);
  const bool two = cx == 2 || cy == 2 || cz == 2;
  const double fc = two ? 0.57735026918962576451 : 1.0;
  const typename In::Raw *gamma = static_cast<const typename In::Raw *>(g.gamma) + (active ? aux.func_off[sc] + cc : 0);
  Acc gC[3] = {Acc(0), Acc(0), Acc(0)};
  Real *R0 = Rb + slot * 2 * Sh::RP, *R1 = R0 + Sh::RP;
  Real *W = Wb + tid * Sh::WP;
  const int p0 = blockIdx.x * g.pair_chunk, p1 = min(g.npairs, p0 + g.pair_chunk);
#pragma unroll 1
  for (int ip = p0; ip < p1; ++ip) {
    const int pair = g.pairs[ip], npp = g.npp[pair];
    const typename In::Raw *rec0 = static_cast<const typename In::Raw *>(g.rec) + g.rec_off[ip];
    const typename In::Raw *gam = gamma + g.pair_col[pair] * g.ldg;
    Acc gA[3] = {Acc(0), Acc(0), Acc(0)}, gCp[3] = {Acc(0), Acc(0), Acc(0)};
#pragma unroll 1
    for (int ipp = 0; ipp < npp; ++ipp) {
      __syncthreads();
      for (int i = tid; i < NREC; i += blockDim.x) {
        const typename In::Raw v = rec0[(long long)ipp * NREC + i];
        srec[i] = In::real(v);
        if (i >= 1 && i <= 3) sP[i - 1] = In::pos(v);
      }
      __syncthreads();
      const Real X = In::diff(sP[0], Cx), Y = In::diff(sP[1], Cy), Z = In::diff(sP[2], Cz), p = srec[0];
#pragma unroll 1
      for (int kc = 0; kc < ncmax; ++kc) {
        const bool live = kc < nc;
        const Real gm = live ? In::real(In::exps(aux)[pc0 + kc]) : Real(1);
        const Real g1 = live ? In::real(In::g1(aux)[pc0 + kc]) : Real(0);
        const Real s = real_rsqrt(p + gm);
        const Real al = p * gm * (s * s);
        Real F[Sh::L1 + 1];
        boys_eval<Sh::L1>(al * (X * X + Y * Y + Z * Z), boys_tab, F);
        const Real *R = build_R<Sh::L1, G, Real>(R0, R1, cc, used, srt, F, al, X, Y, Z);
        if (live) {
          // W of this aux component: x: R shifted (times -1/(2g)); xx: R + R shifted
          // by 2 / (2g) (times 1/(2g)); xy: R shifted (times 1/(4g^2))
          const Real *w = R;
          if (LC > 0) {
#pragma unroll 1
            for (int e = 0; e < NT1; ++e) {
              const int q = stuv[e], t = q & 15, u = (q >> 4) & 15, v = q >> 8;
              const int n1 = t + u + v + LC, s1 = u + v + cy + cz;
              const Real r1 = R[n1 * (n1 + 1) * (n1 + 2) / 6 + s1 * (s1 + 1) / 2 + v + cz];
              W[e] = (LC == 2 && two) ? fma(g1, r1, R[e]) : r1;
            }
            w = W;
          }
          Real S[3], T[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) S[q] = T[q] = Real(0);
#pragma unroll 1
          for (int ab = 0; ab < NAB; ++ab) {
            const Real gv = In::real(gam[ab * g.ldg]);
            Real x[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) x[q] = Real(0);
#pragma unroll 2
            for (int k = sstart[ab]; k < sstart[ab + 1]; ++k) {
              const unsigned i4 = (unsigned)sterm[k];
              const Real *e = srec + GRAD_HDR + 4 * k;
              const Real w0 = w[i4 & 255], e0 = e[0];
              x[0] = acc_fma(e0, w[(i4 >> 8) & 255], x[0]);
              x[1] = acc_fma(e0, w[(i4 >> 16) & 255], x[1]);
              x[2] = acc_fma(e0, w[i4 >> 24], x[2]);
              x[3] = acc_fma(e[1], w0, x[3]);
              x[4] = acc_fma(e[2], w0, x[4]);
              x[5] = acc_fma(e[3], w0, x[5]);
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              S[q] = fma(gv, acc_done(x[q]), S[q]);
              T[q] = fma(gv, acc_done(x[3 + q]), T[q]);
            }
          }
          Real ps = srec[4] * In::real(In::cdiv(aux)[pc0 + kc]) * s * Real(fc);
          if (LC == 1) ps = -(ps * g1);
          if (LC == 2) ps = two ? ps * g1 : ps * (g1 * g1);
          const Real aop = srec[5];
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            gA[q] = gA[q] + In::acc(ps * fma(aop, S[q], T[q]));
            gCp[q] = gCp[q] + In::acc(-(ps * S[q]));
          }
        }
        __syncwarp();
      }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) gC[q] = gC[q] + gCp[q];
    add_pair<Sh::NW>(g, g.pair_a[pair], g.pair_b[pair], gA, gCp, sRed);
  }
  if (active)
#pragma unroll
    for (int q = 0; q < 3; ++q) atomicAdd(&g.grad[3 * g.aux_atom[sc] + q], (double)gC[q]);
}

// Pairs per block: enough blocks for the GPU (about 12 per SM), at most 16 pairs,
// whose C sums then take one atomic per thread.
inline int grad_chunk(int npairs, int aux_blocks) {
  return std::max(1, std::min<int>(16, (int)((long long)npairs * aux_blocks / (152 * 12))));
}

template <int LAB, int LC, typename Real>
void launch_grad3c_j(GradArgs a, const AuxArgs &x, const typename EriIn<Real>::Tab *tab, cudaStream_t st) {
  using Sh = GradShape<LAB, LC, false, Real, GRAD_HDR + 6 * ntuv(LAB + 1)>;
  static OncePerDevice once;
  allow_smem(once, grad3c_j_kernel<LAB, LC, Real>, Sh::SMEM);
  const int ny = ceil_div(a.naux_shells, Sh::NS);
  a.pair_chunk = grad_chunk(a.npairs, ny);
  grad3c_j_kernel<LAB, LC, Real><<<dim3(ceil_div(a.npairs, a.pair_chunk), ny), Sh::THREADS, Sh::SMEM, st>>>(a, x, tab);
}

template <int LA, int LB, int LC, typename Real>
void launch_grad3c_x(GradArgs a, const AuxArgs &x, const typename EriIn<Real>::Tab *tab, cudaStream_t st) {
  using Sh = GradShape<LA + LB, LC, true, Real, GRAD_HDR + 4 * nterms(LA, LB)>;
  static OncePerDevice once;
  allow_smem(once, grad3c_x_kernel<LA, LB, LC, Real>, Sh::SMEM);
  const int ny = ceil_div(a.naux_shells, Sh::NS);
  a.pair_chunk = grad_chunk(a.npairs, ny);
  grad3c_x_kernel<LA, LB, LC, Real><<<dim3(ceil_div(a.npairs, a.pair_chunk), ny), Sh::THREADS, Sh::SMEM, st>>>(a, x, tab);
}

template <int LC>
void launch_grad3c_lc(int la, int lb, int arith, const GradArgs &a, const AuxArgs &x, const GradBoysTabs &t,
                      cudaStream_t st) {
  if (a.gamma) {
    DISPATCH_LALB(la, lb, ({
      if (arith == GRAD_DF) launch_grad3c_x<A_, B_, LC, df>(a, x, t.dfs, st);
      else launch_grad3c_x<A_, B_, LC, double>(a, x, t.f64, st);
    }));
  } else {
    DISPATCH_LALB(la, lb, ({
      if (arith == GRAD_F32) launch_grad3c_j<A_ + B_, LC, float>(a, x, t.f32, st);
      else if (arith == GRAD_DF) launch_grad3c_j<A_ + B_, LC, df>(a, x, t.dfs, st);
      else launch_grad3c_j<A_ + B_, LC, double>(a, x, t.f64, st);
    }));
  }
}

}  // namespace dfjk
