// Local operator in FP64-level accuracy by sum factorisation (Sec. 4.1 cell
// matrices applied without forming them):
//
//   Y += alpha * sum_e Q_e^T (cK K^e + cV V^e + c_j M^e) Q_e X
//
// For affine cubic cells with tensor-product Gauss rules the cell matrices
// factor into 1D matrices:
//   K^e = (1/2)(h/2) [D (x) M (x) M + M (x) D (x) M + M (x) M (x) D]   ((p+1)-point Gauss)
//   M^e = (h/2)^3 M (x) M (x) M
//   V^e = (h/2)^3 Psi diag(V_q) Phi,  Phi = phi (x) phi (x) phi, Psi likewise of psi = phi^T diag(w)
//                                                                     ((p+2)-point Gauss, 1D weights w)
// with M, D the 1D reference mass and stiffness matrices and phi the Lagrange
// basis at the 1D Gauss points.  Each application is a chain of 1D
// contractions of the (p+1)^3 nodal tensor instead of dense products with H^e
// and M^e.  X and Y are FP64; the contractions run in 59-bit fixed point on the
// integer pipes (fx64.cuh), because GB300 issues only 2 FP64 FMAs per clock and
// SM.  All FP64 paths (Y = H X - S X Lambda, the FP64 filter form, Rayleigh-Ritz
// products, residuals) use this form.
#include <algorithm>
#include <memory>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "fx64.cuh"

namespace pawfe {

namespace {

// Even/odd halves of a centro-symmetric 1D matrix A (m x n, A[m-1-i][n-1-j] = A[i][j]):
//   Ae[i][j] = (A[i][j] + A[i][n-1-j]) / 2   (j < n/2),  Ae[i][n/2] = A[i][n/2] / 2 for odd n,
//   Ao[i][j] = (A[i][j] - A[i][n-1-j]) / 2   (i < m/2, j < n/2),
// so that with e[j] = x[j] + x[n-1-j] (e[n/2] = 2 x[n/2]) and o[j] = x[j] - x[n-1-j]:
//   y[i] = E[i] + O[i],  y[m-1-i] = E[i] - O[i],  E = Ae e,  O = Ao o   (y[m/2] = E[m/2] for odd m).
// The GLL nodes and Gauss points are symmetric about the cell centre, so the 1D mass and
// stiffness matrices and the Lagrange values at the Gauss points are all of this form.
// The skew matrix C of the Bloch term is centro-antisymmetric: its even part maps the odd
// half of a line to E and its odd part the even half to O.
constexpr int EOMAX = 5;   // ceil(10 / 2): up to 10 points per direction
struct EoMat {
  double e[EOMAX * EOMAX];   // [i < ceil(m/2)][j < ceil(n/2)]
  double o[EOMAX * EOMAX];   // [i < m/2][j < n/2]
};
struct FxEo {
  fx2 e[EOMAX * EOMAX], o[EOMAX * EOMAX];
};

// one line of a tensor as limbs of its even and odd halves
template <int N>
struct Halves {
  static constexpr int NE = (N + 1) / 2, NO = N / 2;
  int eh[NE], el[NE], oh[NO], ol[NO];
  __device__ __forceinline__ void set_e(int j, long long x) {
    eh[j] = fx_hi(x);
    el[j] = fx_lo(x);
  }
  __device__ __forceinline__ void set_o(int j, long long x) {
    oh[j] = fx_hi(x);
    ol[j] = fx_lo(x);
  }
  // x[0], x[s], ..., x[(N-1) s]
  __device__ __forceinline__ void load(const long long *x, int s) {
#pragma unroll
    for (int j = 0; j < N / 2; ++j) {
      const long long a = x[j * s], b = x[(N - 1 - j) * s];
      set_e(j, a + b);
      set_o(j, a - b);
    }
    if (N & 1) set_e(N / 2, 2 * x[(N / 2) * s]);
  }
};

// accumulators of the even and odd halves of a line of M results
template <int M>
struct Acc {
  static constexpr int ME = (M + 1) / 2, MO = M / 2;
  long long eh[ME], em[ME], oh[MO], om[MO];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < ME; ++i) {
      eh[i] = 0;
      em[i] = FX_HALF;
    }
#pragma unroll
    for (int i = 0; i < MO; ++i) {
      oh[i] = 0;
      om[i] = FX_HALF;
    }
  }
  // the sums so far into the high words, times 2^-d (before the next table: see fx64.cuh)
  __device__ __forceinline__ void fold(int d = 0) {
#pragma unroll
    for (int i = 0; i < ME; ++i) {
      eh[i] = E(i) >> d;
      em[i] = FX_HALF;
    }
#pragma unroll
    for (int i = 0; i < MO; ++i) {
      oh[i] = O(i) >> d;
      om[i] = FX_HALF;
    }
  }
  // += A x (A centro-symmetric, from constant memory)
  template <int N>
  __device__ __forceinline__ void mac(const FxEo &A, const Halves<N> &x) {
#pragma unroll
    for (int i = 0; i < ME; ++i)
#pragma unroll
      for (int j = 0; j < (N + 1) / 2; ++j) fx_mac(eh[i], em[i], x.eh[j], x.el[j], A.e[i * ((N + 1) / 2) + j]);
#pragma unroll
    for (int i = 0; i < MO; ++i)
#pragma unroll
      for (int j = 0; j < N / 2; ++j) fx_mac(oh[i], om[i], x.oh[j], x.ol[j], A.o[i * (N / 2) + j]);
  }
  // += A x (A centro-antisymmetric: e-table on the odd half, o-table on the even half)
  template <int N>
  __device__ __forceinline__ void mac_anti(const FxEo &A, const Halves<N> &x) {
#pragma unroll
    for (int i = 0; i < ME; ++i)
#pragma unroll
      for (int j = 0; j < N / 2; ++j) fx_mac(eh[i], em[i], x.oh[j], x.ol[j], A.e[i * (N / 2) + j]);
#pragma unroll
    for (int i = 0; i < MO; ++i)
#pragma unroll
      for (int j = 0; j < (N + 1) / 2; ++j) fx_mac(oh[i], om[i], x.eh[j], x.el[j], A.o[i * ((N + 1) / 2) + j]);
  }
  __device__ __forceinline__ long long E(int i) const { return fx_sum(eh[i], em[i]); }
  __device__ __forceinline__ long long O(int i) const { return fx_sum(oh[i], om[i]); }
  // f(i, result i of the line)
  template <class F>
  __device__ __forceinline__ void each(F f) const {
#pragma unroll
    for (int i = 0; i < MO; ++i) {
      const long long a = E(i), b = O(i);
      f(i, a + b);
      f(M - 1 - i, a - b);
    }
    if (M & 1) f(M / 2, E(M / 2));
  }
  template <class P>
  __device__ __forceinline__ void store(P *y, int s) const {
    each([&](int i, long long r) { y[i * s] = r; });
  }
};

// Row scales: the rows of M, D, C and psi that belong to node i are divided by 2^tau_i, where
// 2^tau_i is the size of row i of M.  The rows of a corner node are a tenth of those in the middle
// of a cell, (1/10)^3 for a corner of the cube, and a result in one common unit would keep that
// many bits fewer there (largest error of one cell of degree 6, relative to the sum of magnitudes
// of the entry: S 1.6e-14, with the row scales 2.4e-16, FP64 sums 4.5e-16).  All values of a line
// carry the factors of the directions already contracted, so that only the exponents of the
// outputs see them: y at the node (a, b, c) is in units of 2^(tau_a + tau_b + tau_c).
//
// Scales, relative to the unit u of the cell's values (|A| the largest row sum of magnitudes
// of a table A with its row scales; all chosen on the host):
//   U after three contractions with phi:            |phi|^3
//   Z = V U, aligned for the last stage:            |phi|^3 2^(zeta + D)
//   P = M x: |M|,  Q = D x: |D|,  S = M P: |M|^2,  R = kD P + kM Q + c S:  rho 2^D
//   y = fD S + fM R + fB B1:                        2^(eta + D), each of the three sums at most 1
// The kinetic part leaves 1/16 of the range of R to the mass part (c); D (>= 0 with a kinetic
// part) makes room, per cell and vector, for a coefficient or a potential that is larger.
struct FxLocal {
  FxEo phi, psi, M, D, kD, kM, fD, fM, fB;
  int tau[9];
  const int *cell_dofs;
  const fx2 *V;         // ncells x NQ^3: V_q in the unit of the cell
  const int *sV;        // ncells: the coefficients are V 2^-(sV + 1) (FX_BAD: not finite)
  const double *X;
  double *Y;
  const double *cMcol;
  double cM, mf;        // c = (cM + cMcol[j]) mf, in the scale of S and R
  int64_t ldx, ldy;
  int ncols, ntile;
  int hasK, hasM, doV, bad;   // bad: a factor is not finite
  int eta, zeta;
};

// VT vectors per block, one line of a contraction per thread: the longest stage ((p+2)^2
// lines) in one pass.  Eight vectors and two blocks per SM at degrees up to 6 (measured per
// 256 vectors of 16^3 cells, before the sums of fx_sum left the IMAD pipe: 9.9 ms at degree 6 and
// 2.9 ms at degree 4, with four vectors and three to five blocks 10.1 and 3.4 ms: fewer idle lanes in the stages of (p+1)^2 lines);
// four for blocks of at most four vectors, and at degrees 7 and 8, whose lines need more
// registers.
constexpr int FX_VT = 8, FX_VT_SMALL = 4;
template <int NP, int VT>
constexpr int fx_threads() { return ((NP + 1) * (NP + 1) * VT + 31) / 32 * 32; }
// odd row pitches: lines along x of four or eight vectors then start in different banks
template <int NP>
constexpr int fx_row() { return (NP + 1) | 1; }
template <int NP>
constexpr int fx_rown() { return NP | 1; }
template <int NP, int VT>
constexpr size_t fx_smem() {
  return sizeof(long long) * VT * ((NP + 1) * (NP + 1) * fx_row<NP>() + 2 * NP * NP * fx_rown<NP>());
}
template <int NP, int VT>
constexpr int fx_blocks() { return NP > 7 ? 1 : VT == FX_VT ? 2 : 4; }

// gather of the cell's values of four vectors into fixed point; returns the largest exponent
// field of this thread's vector over the cell (0x7ff: a non-finite value)
template <int NP, int VT, typename T>
__device__ __forceinline__ int fx_gather(const int *cell_dofs, const T *X, int64_t ldx, int ncols, int v0,
                                         int *sdof, int *sred, long long *sx) {
  constexpr int NT = fx_threads<NP, VT>(), N3 = NP * NP * NP, NPER = (N3 + NT / VT - 1) / (NT / VT), RN = fx_rown<NP>();
  const int tid = threadIdx.x, v = tid & (VT - 1), r0 = tid / VT;
  T xv[NPER];
  const bool on = v0 + v < ncols;
#pragma unroll
  for (int k = 0; k < NPER; ++k) {
    const int r = r0 + k * (NT / VT);
    const int dof = r < N3 ? cell_dofs[r] : 0;
    xv[k] = (on && r < N3) ? X[dof * ldx + v0 + v] : T(0);
    if (v == 0 && r < N3) sdof[r] = dof;
  }
  int E = 1;
#pragma unroll
  for (int k = 0; k < NPER; ++k) E = max(E, fx_field(xv[k]));
#pragma unroll
  for (int o = VT; o < 32; o <<= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  if ((tid & 31) < VT) sred[(tid >> 5) * VT + v] = E;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) E = max(E, sred[w * VT + v]);
#pragma unroll
  for (int k = 0; k < NPER; ++k) {
    const int r = r0 + k * (NT / VT);
    if (r < N3) sx[((RN == NP) ? r : (r / NP) * RN + r % NP) * VT + v] = fx_from(xv[k], E);
  }
  return E;
}

// What bounds it: the IMAD pipe, three IMAD.WIDE per product at 32 per clock and SM (measured;
// some 40% of all instructions at p = 6): 6.8 ms of the 9.7 ms per 256 vectors of 16^3 cells at
// p = 6 (9.5 ms without the row scales; 9.9 ms with the sums of the accumulator pairs on that pipe
// too), the rest barriers and dependent issue.  The same contractions
// with FP64 FMAs took 53.2 ms there (FP64 pipe 88% busy); p = 4: 2.9 ms.
// The tables are kernel parameters, read by the IMADs as constant operands.  The nodal tensor
// of the potential part grows in place to the (p+2)^3 Gauss points and back (W); the kinetic
// part works in place in two (p+1)^3 tensors (X, Q).  Stages of the two parts that do not
// depend on one another share a barrier interval.
template <int NP, int VT>
__global__ void __launch_bounds__(fx_threads<NP, VT>(), fx_blocks<NP, VT>()) k_local_fx(const __grid_constant__ FxLocal A) {
  constexpr int NQ = NP + 1, NT = fx_threads<NP, VT>(), N3 = NP * NP * NP;
  constexpr int RS = fx_row<NP>(), RN = fx_rown<NP>();
  extern __shared__ long long sm[];
  long long *W = sm;                                   // [c or k][b or j][i]: NQ, RS pitches
  long long *SX = W + NQ * NQ * RS * VT;            // x, then P, then S   [c][b][a]
  long long *SQ = SX + NP * NP * RN * VT;           // Q, then R
  __shared__ int sdof[N3], sred[NT / 32 * VT];
  __shared__ int sD[VT], sZ[VT], sbad[VT];
  __shared__ fx2 scm[VT];
  const int e = blockIdx.x / A.ntile, v0 = (blockIdx.x - e * A.ntile) * VT;
  const int tid = threadIdx.x, v = tid & (VT - 1), ln = tid / VT;
  const bool doV = A.doV != 0;
  if (tid < VT) {
    double cm = A.cM;
    if (A.cMcol && v0 + v < A.ncols) cm += A.cMcol[v0 + v];
    cm *= A.mf;
    // |c| < 2^sc.  The kinetic part takes 15/16 2^-D of the range of R: c has 1/16 where D is 0
    // and 1/2 (the largest coefficient) from there on
    const int f = fx_field(cm), sc = cm == 0.0 ? FX_NONE : fx_field_coef(cm) - 1022;
    const int sv = doV ? A.sV[e] : FX_NONE;
    int D = A.hasK ? (sc <= -4 ? 0 : max(sc + 1, 1)) : max(sc + 1, -4000);
    if (doV) D = max(D, sv - A.zeta);
    const bool bad = A.bad || f == 0x7ff || sv == FX_BAD;
    sbad[v] = bad;
    if (bad) D = 0;
    sD[v] = D;
    sZ[v] = doV && !bad ? min(A.zeta + D - sv, 63) : 0;
    const long long C = (bad || cm == 0.0) ? 0 : fx_from<63>(cm, D + 1021);
    scm[v].h = fx_hi(C);
    scm[v].l = fx_lo(C);
  }
  const int Emax = fx_gather<NP, VT>(A.cell_dofs + (size_t)e * N3, A.X, A.ldx, A.ncols, v0, sdof, sred, SX);
  __syncthreads();
  // U1: lines along x, nodes -> Gauss points
  if (doV && ln < NP * NP) {
    Halves<NP> x;
    x.load(SX + ln * RN * VT + v, VT);
    Acc<NQ> U;
    U.init();
    U.mac(A.phi, x);
    U.store(W + ((ln / NP) * NQ + ln % NP) * RS * VT + v, VT);
  }
  __syncthreads();
  // U2: lines along y of W
  if (doV && ln < NQ * NP) {
    long long *w = W + ((ln / NQ) * NQ * RS + ln % NQ) * VT + v;
    Halves<NP> x;
    x.load(w, RS * VT);
    Acc<NQ> U;
    U.init();
    U.mac(A.phi, x);
    U.store(w, RS * VT);
  }
  // P = M x, Q = D x: lines along z
  if (ln < NP * NP) {
    const int o = ((ln / NP) * RN + ln % NP) * VT + v;
    Halves<NP> x;
    x.load(SX + o, NP * RN * VT);
    {
      Acc<NP> P;
      P.init();
      P.mac(A.M, x);
      P.store(SX + o, NP * RN * VT);
    }
    if (A.hasK) {
      Acc<NP> Q;
      Q.init();
      Q.mac(A.D, x);
      Q.store(SQ + o, NP * RN * VT);
    }
  }
  __syncthreads();
  // U3, Z = V U3 and B2 = psi Z: lines along z of W, in registers
  if (doV && ln < NQ * NQ) {
    const int2 *Vq = reinterpret_cast<const int2 *>(A.V) + (size_t)e * (NQ * NQ * NQ) + ln;
    const int zs = sZ[v];
    const long long half = zs > 1 ? 1ll << (zs - 2) : 0;
    long long *w = W + ((ln / NQ) * RS + ln % NQ) * VT + v;
    Halves<NP> x;
    x.load(w, NQ * RS * VT);
    Acc<NQ> U;
    U.init();
    U.mac(A.phi, x);
    Halves<NQ> z;
#pragma unroll
    for (int i = 0; i < (NQ + 1) / 2; ++i) {
      const bool mid = (NQ & 1) && i == NQ / 2;
      long long r[2];
      if (mid) {
        r[0] = U.E(i);
      } else {
        const long long a = U.E(i), b = U.O(i);
        r[0] = a + b;
        r[1] = a - b;
      }
#pragma unroll
      for (int t = 0; t < (mid ? 1 : 2); ++t) {
        const int2 q = __ldg(Vq + (t ? NQ - 1 - i : i) * NQ * NQ);
        long long hh = half, mm = FX_HALF;
        fx_mac(hh, mm, fx_hi(r[t]), fx_lo(r[t]), fx2{q.x, q.y});
        r[t] = 2 * fx_sum(hh, mm) >> zs;   // twice the product: coefficients are below 1/2
      }
      if (mid) {
        z.set_e(i, 2 * r[0]);
      } else {
        z.set_e(i, r[0] + r[1]);
        z.set_o(i, r[0] - r[1]);
      }
    }
    Acc<NP> B;
    B.init();
    B.mac(A.psi, z);
    B.store(w, NQ * RS * VT);
  }
  // S = M P, R = kD P + kM Q + c S: lines along y
  if (ln < NP * NP) {
    const int o = ((ln / NP) * NP * RN + ln % NP) * VT + v;
    const int D = sD[v];
    const fx2 cm = scm[v];
    Halves<NP> p;
    p.load(SX + o, RN * VT);
    Acc<NP> T;
    T.init();
    if (A.hasK) {
      T.mac(A.kD, p);
      T.fold();
      Halves<NP> q;
      q.load(SQ + o, RN * VT);
      T.mac(A.kM, q);
      if (D > 0) T.fold(min(D, 63));
    }
    Acc<NP> S;
    S.init();
    S.mac(A.M, p);
    S.store(SX + o, RN * VT);
    if (A.hasM) {
#pragma unroll
      for (int i = 0; i < (NP + 1) / 2; ++i) {
        const long long a = S.E(i);
        fx_mac(T.eh[i], T.em[i], fx_hi(a), fx_lo(a), cm);
      }
#pragma unroll
      for (int i = 0; i < NP / 2; ++i) {
        const long long b = S.O(i);
        fx_mac(T.oh[i], T.om[i], fx_hi(b), fx_lo(b), cm);
      }
    }
    T.store(SQ + o, RN * VT);
  }
  __syncthreads();
  // B1: lines along y of W, Gauss points -> nodes
  if (doV && ln < NQ * NP) {
    long long *w = W + ((ln / NQ) * NQ * RS + ln % NQ) * VT + v;
    Halves<NQ> x;
    x.load(w, RS * VT);
    Acc<NP> B;
    B.init();
    B.mac(A.psi, x);
    B.store(w, RS * VT);
  }
  __syncthreads();
  // y = fD S + fM R + fB B1: lines along x, added into Y from the registers
  if (ln < NP * NP) {
    const int D = sD[v];
    Acc<NP> y;
    y.init();
    if (A.hasK) {
      Halves<NP> s;
      s.load(SX + ln * RN * VT + v, VT);
      y.mac(A.fD, s);
      y.fold(min(D, 63));
    }
    {
      Halves<NP> r;
      r.load(SQ + ln * RN * VT + v, VT);
      y.mac(A.fM, r);
    }
    if (doV) {
      y.fold();
      Halves<NQ> b;
      b.load(W + ((ln / NP) * NQ + ln % NP) * RS * VT + v, VT);
      y.mac(A.fB, b);
    }
    if (v0 + v < A.ncols) {
      const int ex = Emax - FX_BIAS + A.eta + D + A.tau[ln % NP] + A.tau[ln / NP];
      const bool bad = Emax == 0x7ff || sbad[v];
      double *Yv = A.Y + v0 + v;
      y.each([&](int a, long long r) {
        atomicAdd(Yv + sdof[ln * NP + a] * A.ldy,
                  bad ? __longlong_as_double(0x7ff8000000000000ll) : fx_to(r, ex + A.tau[a]));
      });
    }
  }
}

// Bloch term at a wavevector k: y = (h/2)^2 [k_x C (x) M (x) M + k_y M (x) C (x) M
// + k_z M (x) M (x) C] x per cell (C = the skew 1D matrix (C1 - C1^T)/2,
// C1[a][b] = int l_a l_b' dxi; M the 1D reference mass), accumulated into
// Y with factor alpha.  The chain of the kinetic part of k_local_fx (z, then y, then x) with
// C in the place of D; the factors k_x, k_y, k_z, (h/2)^2 and alpha are folded into the tables.
struct FxBloch {
  FxEo M, C, kyC, kzM, fC, fM;   // z: M, C;  y: M, k_y C, k_z M;  x: alpha (h/2)^2 (k_x C, M)
  int tau[9];                    // as FxLocal
  const int *cell_dofs;
  const double *X;
  double *Y;
  int64_t ldx, ldy;
  int ncols, ntile, eta;
};

template <int NP, int VT>
__global__ void __launch_bounds__(fx_threads<NP, VT>(), fx_blocks<NP, VT>()) k_bloch_fx(const __grid_constant__ FxBloch A) {
  constexpr int NT = fx_threads<NP, VT>(), N3 = NP * NP * NP, RN = fx_rown<NP>();
  extern __shared__ long long sm[];
  long long *SX = sm, *SQ = SX + NP * NP * RN * VT;
  __shared__ int sdof[N3], sred[NT / 32 * VT];
  const int e = blockIdx.x / A.ntile, v0 = (blockIdx.x - e * A.ntile) * VT;
  const int tid = threadIdx.x, v = tid & (VT - 1), ln = tid / VT;
  const int Emax = fx_gather<NP, VT>(A.cell_dofs + (size_t)e * N3, A.X, A.ldx, A.ncols, v0, sdof, sred, SX);
  __syncthreads();
  // z lines: P = M x, Q = C x
  if (ln < NP * NP) {
    const int o = ((ln / NP) * RN + ln % NP) * VT + v;
    Halves<NP> x;
    x.load(SX + o, NP * RN * VT);
    {
      Acc<NP> P;
      P.init();
      P.mac(A.M, x);
      P.store(SX + o, NP * RN * VT);
    }
    Acc<NP> Q;
    Q.init();
    Q.mac_anti(A.C, x);
    Q.store(SQ + o, NP * RN * VT);
  }
  __syncthreads();
  // y lines: S = M P, T = k_y C P + k_z M Q
  if (ln < NP * NP) {
    const int o = ((ln / NP) * NP * RN + ln % NP) * VT + v;
    Halves<NP> p;
    p.load(SX + o, RN * VT);
    {
      Acc<NP> T;
      T.init();
      T.mac_anti(A.kyC, p);
      T.fold();
      Halves<NP> q;
      q.load(SQ + o, RN * VT);
      T.mac(A.kzM, q);
      T.store(SQ + o, RN * VT);
    }
    Acc<NP> S;
    S.init();
    S.mac(A.M, p);
    S.store(SX + o, RN * VT);
  }
  __syncthreads();
  // x lines: y = fC S + fM T
  if (ln < NP * NP) {
    Acc<NP> y;
    y.init();
    {
      Halves<NP> s;
      s.load(SX + ln * RN * VT + v, VT);
      y.mac_anti(A.fC, s);
      y.fold();
    }
    Halves<NP> t;
    t.load(SQ + ln * RN * VT + v, VT);
    y.mac(A.fM, t);
    if (v0 + v < A.ncols) {
      const int ex = Emax - FX_BIAS + A.eta + A.tau[ln % NP] + A.tau[ln / NP];
      double *Yv = A.Y + v0 + v;
      y.each([&](int a, long long r) {
        atomicAdd(Yv + sdof[ln * NP + a] * A.ldy,
                  Emax == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : fx_to(r, ex + A.tau[a]));
      });
    }
  }
}

// out[e][q] = wq[q] sum_v f[v] u_v(x_q)^2, u_v = phi X_v at the (p+2)^3 Gauss points (wq, f NULL: 1):
// the interpolation of k_local_fx for tiles of VT vectors, the squares summed in FP64 (one or
// two FP64 operations per point and vector) by the thread of each line and vector, and over the
// vectors of a tile at the end.  One block per cell.  16^3 cells of degree 4, 16 FP32 vectors:
// 0.14 ms, where dense FP64 products with the 216 x 125 basis values took 6.1 ms.
struct FxDensity {
  FxEo phi;
  const int *cell_dofs;
  const double *wq, *f;
  double *out;
  int64_t ldx;
  int ncols;
  double unit;   // |phi|^3: scale of the interpolated values
};

template <int NP, int VT, typename T>
__global__ void __launch_bounds__(fx_threads<NP, VT>(), fx_blocks<NP, VT>())
    k_density_fx(const __grid_constant__ FxDensity A, const T *__restrict__ X) {
  constexpr int NQ = NP + 1, NT = fx_threads<NP, VT>(), N3 = NP * NP * NP;
  constexpr int RS = fx_row<NP>(), RN = fx_rown<NP>();
  extern __shared__ long long sm[];
  long long *W = sm, *SX = W + NQ * NQ * RS * VT;
  __shared__ int sdof[N3], sred[NT / 32 * VT];
  const size_t e = blockIdx.x;
  const int tid = threadIdx.x, v = tid % VT, ln = tid / VT;
  double s[NQ];
#pragma unroll
  for (int k = 0; k < NQ; ++k) s[k] = 0.0;
  for (int v0 = 0; v0 < A.ncols; v0 += VT) {
    if (v0) __syncthreads();
    const int Emax = fx_gather<NP, VT>(A.cell_dofs + e * N3, X, A.ldx, A.ncols, v0, sdof, sred, SX);
    __syncthreads();
    if (ln < NP * NP) {
      Halves<NP> x;
      x.load(SX + ln * RN * VT + v, VT);
      Acc<NQ> U;
      U.init();
      U.mac(A.phi, x);
      U.store(W + ((ln / NP) * NQ + ln % NP) * RS * VT + v, VT);
    }
    __syncthreads();
    if (ln < NQ * NP) {
      long long *w = W + ((ln / NQ) * NQ * RS + ln % NQ) * VT + v;
      Halves<NP> x;
      x.load(w, RS * VT);
      Acc<NQ> U;
      U.init();
      U.mac(A.phi, x);
      U.store(w, RS * VT);
    }
    __syncthreads();
    if (ln < NQ * NQ && v0 + v < A.ncols) {
      Halves<NP> x;
      x.load(W + ((ln / NQ) * RS + ln % NQ) * VT + v, NQ * RS * VT);
      Acc<NQ> U;
      U.init();
      U.mac(A.phi, x);
      const bool bad = Emax == 0x7ff;
      const double fv = A.f ? A.f[v0 + v] : 1.0;
      U.each([&](int k, long long r) {
        const double u = bad ? __longlong_as_double(0x7ff8000000000000ll) : fx_to_small(r, Emax - FX_BIAS);
        s[k] = fma(A.f ? fv * u : u, u, s[k]);
      });
    }
  }
#pragma unroll
  for (int k = 0; k < NQ; ++k)
#pragma unroll
    for (int o = VT / 2; o; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
  if (ln < NQ * NQ && v == 0) {
    const double g = A.unit * A.unit;
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
      const int q = k * NQ * NQ + ln;
      A.out[e * (NQ * NQ * NQ) + q] = (A.wq ? A.wq[q] * g : g) * s[k];
    }
  }
}

// V_q of one cell per block in the cell's own unit
__global__ void __launch_bounds__(128) k_V_fx(int nq, const double *__restrict__ Vq, fx2 *__restrict__ out,
                                              int *__restrict__ sV) {
  __shared__ int sred[4];
  const size_t e = blockIdx.x;
  int E = 1, any = 0, bad = 0;
  for (int i = threadIdx.x; i < nq; i += 128) {
    const double x = Vq[e * nq + i];
    E = max(E, fx_field_coef(x));
    any |= x != 0.0;
    bad |= fx_field(x) == 0x7ff;
  }
  any = __syncthreads_or(any);
  bad = __syncthreads_or(bad);
#pragma unroll
  for (int o = 16; o; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = E;
  __syncthreads();
  E = max(max(sred[0], sred[1]), max(sred[2], sred[3]));
  for (int i = threadIdx.x; i < nq; i += 128) {
    const long long C = bad ? 0 : fx_from<63>(Vq[e * nq + i], E);
    out[e * nq + i] = {fx_hi(C), fx_lo(C)};
  }
  if (threadIdx.x == 0) sV[e] = bad ? FX_BAD : any ? E - 1022 : FX_NONE / 2;
}

// even/odd halves of a row-major m x n matrix (see EoMat); the matrix is
// centro-symmetric up to rounding, and the halves use its symmetrised form
void eo_halves(const double *A, int m, int n, EoMat &out) {
  const int ne = (n + 1) / 2, no = n / 2;
  for (int i = 0; i < (m + 1) / 2; ++i) {
    for (int j = 0; j < no; ++j)
      out.e[i * ne + j] = 0.5 * (A[(size_t)i * n + j] + A[(size_t)i * n + (n - 1 - j)]);
    if (n & 1) out.e[i * ne + no] = 0.5 * A[(size_t)i * n + no];
  }
  for (int i = 0; i < m / 2; ++i)
    for (int j = 0; j < no; ++j)
      out.o[i * no + j] = 0.5 * (A[(size_t)i * n + j] - A[(size_t)i * n + (n - 1 - j)]);
}

// even/odd halves of a centro-antisymmetric m x n matrix A (A[m-1-i][n-1-j] = -A[i][j]),
// in the layout of Acc::mac_anti:
//   e[i][j] = (A[i][j] - A[i][n-1-j]) / 2      (i < ceil(m/2), j < n/2; pairs with o-lines),
//   o[i][j] = (A[i][j] + A[i][n-1-j]) / 2      (i < m/2, j < n/2),  o[i][n/2] = A[i][n/2] / 2 for odd n.
void eo_halves_anti(const double *A, int m, int n, EoMat &out) {
  const int ne = (n + 1) / 2, no = n / 2;
  for (int i = 0; i < (m + 1) / 2; ++i)
    for (int j = 0; j < no; ++j)
      out.e[i * no + j] = 0.5 * (A[(size_t)i * n + j] - A[(size_t)i * n + (n - 1 - j)]);
  for (int i = 0; i < m / 2; ++i) {
    for (int j = 0; j < no; ++j)
      out.o[i * ne + j] = 0.5 * (A[(size_t)i * n + j] + A[(size_t)i * n + (n - 1 - j)]);
    if (n & 1) out.o[i * ne + no] = 0.5 * A[(size_t)i * n + no];
  }
}

std::vector<double> row_sums(const std::vector<double> &A, int m, int n) {
  std::vector<double> r(m, 0.0);
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < n; ++j) r[i] += std::fabs(A[(size_t)i * n + j]);
  return r;
}

// powers of two of the row sums of M relative to the largest, rounded up (a row 1/16 of a power of
// two above one still counts with it, which doubles no other: degree 8, second node)
std::vector<int> row_scales(const std::vector<double> &M, int n) {
  const std::vector<double> r = row_sums(M, n, n);
  const double top = *std::max_element(r.begin(), r.end());
  std::vector<int> t(n);
  for (int i = 0; i < n; ++i) t[i] = (int)std::ceil(std::log2(std::min(r[i], r[n - 1 - i]) / top) - 1.0 / 16);   // 0 .. -3 up to degree 8
  return t;
}

// a 1D matrix with its row scales (tau NULL: none), its halves, and its row sums of magnitudes
struct Tab1 {
  EoMat eo{};
  std::vector<double> row;
  double norm = 0.0;
  Tab1(std::vector<double> A, int m, int n, const int *tau, bool anti = false) {
    for (int i = 0; tau && i < m; ++i)
      for (int j = 0; j < n; ++j) A[(size_t)i * n + j] = std::ldexp(A[(size_t)i * n + j], -tau[i]);
    if (anti)
      eo_halves_anti(A.data(), m, n, eo);
    else
      eo_halves(A.data(), m, n, eo);
    row = row_sums(A, m, n);
    for (double &r : row) norm = std::max(norm, r *= 1.0 + 1e-6);   // the limbs of A / |A| stay below their limit
  }
  // limbs of f A (|f| |A| <= 1)
  void put(FxEo &t, long double f) const {
    for (int i = 0; i < EOMAX * EOMAX; ++i) {
      t.e[i] = fx_coef(f * eo.e[i]);
      t.o[i] = fx_coef(f * eo.o[i]);
    }
  }
};

template <int NP, int VT>
void launch_local(paw_context *c, FxLocal &t, cudaStream_t s) {
  const size_t shm = fx_smem<NP, VT>();
  PAW_CUDA(cudaFuncSetAttribute(k_local_fx<NP, VT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  t.ntile = (t.ncols + VT - 1) / VT;
  k_local_fx<NP, VT><<<(unsigned)((int64_t)c->ncells * t.ntile), fx_threads<NP, VT>(), shm, s>>>(t);
  PAW_LAUNCH_CHECK("k_local_fx");
}

template <int NP, int VT>
void launch_bloch(paw_context *c, FxBloch &t, cudaStream_t s) {
  const size_t shm = sizeof(long long) * VT * 2 * NP * NP * fx_rown<NP>();
  PAW_CUDA(cudaFuncSetAttribute(k_bloch_fx<NP, VT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  t.ntile = (t.ncols + VT - 1) / VT;
  k_bloch_fx<NP, VT><<<(unsigned)((int64_t)c->ncells * t.ntile), fx_threads<NP, VT>(), shm, s>>>(t);
  PAW_LAUNCH_CHECK("k_bloch_fx");
}

template <int NP, int VT, typename T>
void launch_density(paw_context *c, const FxDensity &t, const T *X, cudaStream_t s) {
  const size_t shm = sizeof(long long) * VT * ((NP + 1) * (NP + 1) * fx_row<NP>() + NP * NP * fx_rown<NP>());
  PAW_CUDA(cudaFuncSetAttribute(k_density_fx<NP, VT, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  k_density_fx<NP, VT, T><<<(unsigned)c->ncells, fx_threads<NP, VT>(), shm, s>>>(t, X);
  PAW_LAUNCH_CHECK("k_density_fx");
}

// f(points per direction, vectors per block) for the degree of the handle
template <class F>
void with_sizes(const paw_context *c, int ncols, const char *what, F f) {
  const bool few = ncols <= FX_VT_SMALL;
  auto by = [&](auto np) {
    constexpr int NP = decltype(np)::value;
    if (NP > 7 || few)
      f(np, std::integral_constant<int, FX_VT_SMALL>{});
    else
      f(np, std::integral_constant<int, (NP > 7 ? FX_VT_SMALL : FX_VT)>{});
  };
  switch (c->np1) {
    case 2: by(std::integral_constant<int, 2>{}); break;
    case 3: by(std::integral_constant<int, 3>{}); break;
    case 4: by(std::integral_constant<int, 4>{}); break;
    case 5: by(std::integral_constant<int, 5>{}); break;
    case 6: by(std::integral_constant<int, 6>{}); break;
    case 7: by(std::integral_constant<int, 7>{}); break;
    case 8: by(std::integral_constant<int, 8>{}); break;
    case 9: by(std::integral_constant<int, 9>{}); break;
    default: throw Error{PAW_ERR_UNSUPPORTED, what};
  }
}

}  // namespace

// Tables of a handle in fixed point, kept between calls (they depend on the mesh and on the
// factors of the call, not on its vectors): making them takes the host longer than a small
// application takes the GPU.  A bounded number, the oldest is replaced.
struct SfPlans {
  static constexpr size_t MAX = 4;
  std::vector<int> tau;
  Tab1 M, D, C, phi, psi;
  struct Local {
    double alpha, cK, cV, cM;
    FxLocal t;
  };
  struct Bloch {
    double alpha;
    FxBloch t;
  };
  std::vector<Local> local;
  std::vector<Bloch> bloch;
  size_t next_local = 0, next_bloch = 0;
  FxDensity density{};

  // psi[a][i] = phi_a(g_i) w_i
  static std::vector<double> weighted(const paw_context *c) {
    std::vector<double> t((size_t)c->np1 * c->nq1);
    for (int i = 0; i < c->nq1; ++i)
      for (int a = 0; a < c->np1; ++a) t[(size_t)a * c->nq1 + i] = c->phiq[(size_t)i * c->np1 + a] * c->wq1[i];
    return t;
  }
  // largest |a| (A_b B_c) + |b| (B_b A_c) over two rows b, c: bound of a A (x) B + b B (x) A
  static double pair_bound(double a, double b, const Tab1 &A, const Tab1 &B) {
    double m = 0.0;
    for (size_t i = 0; i < A.row.size(); ++i)
      for (size_t j = 0; j < A.row.size(); ++j)
        m = std::max(m, std::fabs(a) * A.row[i] * B.row[j] + std::fabs(b) * B.row[i] * A.row[j]);
    return m;
  }
  explicit SfPlans(const paw_context *c)
      : tau(row_scales(c->M1, c->np1)),
        M(c->M1, c->np1, c->np1, tau.data()),
        D(c->D1, c->np1, c->np1, tau.data()),
        C(c->C1s.empty() ? c->M1 : c->C1s, c->np1, c->np1, tau.data(), true),
        phi(c->phiq, c->nq1, c->np1, nullptr),
        psi(weighted(c), c->np1, c->nq1, tau.data()) {
    const long double nP = phi.norm;
    phi.put(density.phi, 1 / nP);
    density.unit = (double)(nP * nP * nP);
  }

  // the entry to write next: a new one, or the oldest
  template <class E>
  static E &slot(std::vector<E> &v, size_t &next) {
    if (v.size() < MAX) {
      v.emplace_back();
      return v.back();
    }
    E &e = v[next];
    next = (next + 1) % MAX;
    return e;
  }

  const FxBloch &bloch_tables(const paw_context *c, double alpha) {
    for (const Bloch &e : bloch)
      if (e.alpha == alpha) return e.t;
    FxBloch t{};
    const double f = alpha * (c->h / 2.0) * (c->h / 2.0);
    const double kx = c->kvec[0], ky = c->kvec[1], kz = c->kvec[2];
    // T: k_y C P + k_z M Q in the scale rho, then y = fC S + fM T in the scale 2^eta
    const long double nM = M.norm, nC = C.norm, tiny = 1e-300;
    const long double rho = std::max((long double)pair_bound(ky, kz, C, M), tiny);
    const int eta = fx_scale((double)std::max(std::fabs(f) * std::max(std::fabs(kx) * nC * nM * nM, nM * rho), tiny));
    M.put(t.M, 1 / nM);
    C.put(t.C, 1 / nC);
    C.put(t.kyC, ky * nM / rho);
    M.put(t.kzM, kz * nC / rho);
    C.put(t.fC, std::ldexp(f * (kx * nM * nM), -eta));
    M.put(t.fM, std::ldexp(f * rho, -eta));
    t.eta = eta;
    std::copy(tau.begin(), tau.end(), t.tau);
    Bloch &e = slot(bloch, next_bloch);
    e.alpha = alpha;
    e.t = t;
    return e.t;
  }

  const FxLocal &local_tables(const paw_context *c, double alpha_in, double cK, double cV, double cM) {
    for (const Local &e : local)
      if (e.alpha == alpha_in && e.cK == cK && e.cV == cV && e.cM == cM) return e.t;
    FxLocal t{};
    const double hh = c->h / 2.0, kf = cK * 0.5 * hh, mf = hh * hh * hh;
    const long double tiny = 1e-300;
    t.hasK = kf != 0.0;
    t.doV = cV != 0.0;
    t.bad = !std::isfinite(alpha_in) || !std::isfinite(kf) || !std::isfinite(cV);
    const double alpha = t.bad ? 1.0 : alpha_in;
    // scales (see FxLocal); without a kinetic part c is cM / 2 in the scale of cM
    const long double nM = M.norm, nD = D.norm, nP = phi.norm, nS = psi.norm, p3 = nP * nP * nP, akf = std::fabs(kf);
    t.mf = (double)(mf * nM * nM / (t.hasK ? (long double)pair_bound(kf, kf, D, M) * 16 / 15
                                           : mf * nM * nM * 2 * std::max(std::fabs(cM) * (1 + 1e-6L), 1e-270L)));
    const long double rho = mf * nM * nM / t.mf;   // c = cM t.mf has no other rounding
    t.eta = fx_scale((double)std::max(std::fabs(alpha) * std::max(akf * nD * nM * nM, nM * rho), tiny));
    const long double fV = alpha * cV * mf * p3 * nS * nS;   // (h/2)^3: detJ
    t.zeta = fx_scale((double)(std::ldexp((long double)1, t.eta) / std::max(std::fabs(fV) * nS, tiny))) - 1;
    t.cM = cM;
    const Local *near = nullptr;   // tables of another alpha: only the last stage differs
    for (const Local &e : local)
      if (e.cK == cK && e.cV == cV && e.cM == cM && !e.t.bad) near = &e;
    if (near) {
      t.phi = near->t.phi;
      t.psi = near->t.psi;
      t.M = near->t.M;
      t.D = near->t.D;
      t.kD = near->t.kD;
      t.kM = near->t.kM;
    } else {
      phi.put(t.phi, 1 / nP);
      psi.put(t.psi, 1 / nS);
      M.put(t.M, 1 / nM);
      D.put(t.D, 1 / nD);
      D.put(t.kD, kf * nM / rho);
      M.put(t.kM, kf * nD / rho);
    }
    D.put(t.fD, std::ldexp(alpha * (kf * nM * nM), -t.eta));
    M.put(t.fM, std::ldexp(alpha * rho, -t.eta));
    psi.put(t.fB, t.doV ? std::ldexp(fV, t.zeta - t.eta) : 0);
    std::copy(tau.begin(), tau.end(), t.tau);
    Local &e = slot(local, next_local);
    e.alpha = alpha_in;
    e.cK = cK;
    e.cV = cV;
    e.cM = cM;
    e.t = t;
    return e.t;
  }
};

static SfPlans &plans(paw_context *c) {
  if (!c->sf_plans) c->sf_plans = std::make_shared<SfPlans>(c);
  return *c->sf_plans;
}

void bloch_sf(paw_context *c, const double *X, int ldx, double *Y, int ldy, int ncols, double alpha,
              cudaStream_t s) {
  if (ncols <= 0 || !c->kc) return;
  FxBloch t = plans(c).bloch_tables(c, alpha);
  t.cell_dofs = c->cell_dofs.as<int>();
  t.X = X;
  t.Y = Y;
  t.ldx = ldx;
  t.ldy = ldy;
  t.ncols = ncols;
  with_sizes(c, ncols, "degree out of range for the Bloch kernel",
             [&](auto np, auto vt) { launch_bloch<decltype(np)::value, decltype(vt)::value>(c, t, s); });
}

template <typename T>
void density_sf(paw_context *c, const T *X, int ldx, int ncols, const double *wq, const double *f, double *out,
                cudaStream_t s) {
  FxDensity t = plans(c).density;
  t.cell_dofs = c->cell_dofs.as<int>();
  t.wq = wq;
  t.f = f;
  t.out = out;
  t.ldx = ldx;
  t.ncols = ncols;
  with_sizes(c, ncols, "degree out of range for the density kernel",
             [&](auto np, auto vt) { launch_density<decltype(np)::value, decltype(vt)::value>(c, t, X, s); });
}
template void density_sf<double>(paw_context *, const double *, int, int, const double *, const double *, double *,
                                 cudaStream_t);
template void density_sf<float>(paw_context *, const float *, int, int, const double *, const double *, double *,
                                cudaStream_t);

void local_prepare(paw_context *c, cudaStream_t s) {
  if (c->Vfx_valid) return;
  c->Vfx.ensure(sizeof(fx2) * (size_t)c->ncells * c->nq, &c->dev_bytes);
  c->Vfx_exp.ensure(sizeof(int) * (size_t)c->ncells, &c->dev_bytes);
  k_V_fx<<<(unsigned)c->ncells, 128, 0, s>>>(c->nq, c->Vq.as<double>(), c->Vfx.as<fx2>(), c->Vfx_exp.as<int>());
  PAW_LAUNCH_CHECK("k_V_fx");
  c->Vfx_valid = 1;
}

void local_sf(paw_context *c, const double *X, int ldx, double *Y, int ldy, int ncols, double alpha, double cK,
              double cV, double cM, const double *cMcol, cudaStream_t s) {
  if (ncols <= 0) return;
  FxLocal t = plans(c).local_tables(c, alpha, cK, cV, cM);
  local_prepare(c, s);
  t.cell_dofs = c->cell_dofs.as<int>();
  t.V = c->Vfx.as<fx2>();
  t.sV = c->Vfx_exp.as<int>();
  t.X = X;
  t.Y = Y;
  t.cMcol = cMcol;
  t.hasM = cMcol || t.cM != 0.0;
  t.ldx = ldx;
  t.ldy = ldy;
  t.ncols = ncols;
  with_sizes(c, ncols, "degree out of range for the sum-factorised kernel",
             [&](auto np, auto vt) { launch_local<decltype(np)::value, decltype(vt)::value>(c, t, s); });
}

}  // namespace pawfe
