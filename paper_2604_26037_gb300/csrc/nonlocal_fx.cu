// FP64 projector contractions on the tensor cores by exact digit products.
//
//   projection  U[k][al][v] = sum_o P[k][o][al] s(o) X[o][v]          per owner pair k
//   expansion   S[o][v]     = sum_k sum_al P[k][o][al] W[a_k][al][v]  with the output stage of its mode
//
// GB300 retires 2 FP64 FMAs per clock and SM and 1024 products of an FP16 mma.sync.  Rows first: a
// projector falls by 1e-8 to its cut-off, so row o of P is divided by 2^r(o), the size of its
// largest entry over the pairs of the cell, X(o) is multiplied by it, and the sums of the
// expansion take it back; an X that grows where P falls then keeps its bits where the
// products are large.  Each operand is then scaled by a power of two per column (P: per pair and projector;
// X: per vector over the owned nodes of the cell; W: per vector over the coefficients that reach the cell), rounded
// to an integer of at most 2^54 and written in seven balanced digits of radix 256, each exact in
// FP16 (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with
// fixed digits).  Products of digits i and j (0 = lowest) with i + j >= 5 are summed by i + j in FP32
// accumulators: at most seven products of magnitude 2^14 share one and at most 144 terms are
// summed between two flushes, 2^14 * 7 * 144 < 2^24, so every accumulator holds an exact
// integer.  A flush rounds the eight accumulators into one 64-bit sum.  What is left out (i + j
// <= 4) is below 2^-58 of the largest product, the rounding of the operands at most 2^-54 of their
// column's largest entry, and the rounding of a flush 2^-(61 - b) of the product of the two columns' units
// for at most 2^b terms.  Errors relative to the sum of the magnitudes, from a model of these sums: 216
// terms of like size 1.1e-17 (rms; FP64 sums 5.5e-17), 6144 terms 3.3e-17 (5.0e-17); with operands and
// flushes cut off instead of rounded 2.0e-17 and 9.1e-16.  X falling by e^-18 over 216 nodes while P
// grows by as much: 3.2e-17 (FP64 5.1e-17; without the row factors 7.9e-11).
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fx64.cuh"
#include "nonlocal_common.cuh"

namespace pawfe {

namespace {

constexpr int DG = 7;            // digits of an operand
constexpr int DG_BITS = 54;      // |integer| <= 2^54: the top digit stays within +-65
constexpr int DG_SUMS = 8;       // accumulators: digit positions 5 .. 12
constexpr int FLUSH = 9;         // k steps of 16 between two flushes
// coefficients of one batch of the expansion: 8 k steps, or 7 where sums of several batches share
// the shared memory (two blocks per SM at degree 6)
constexpr int EXP_K = 128, EXP_K_MANY = 112;
constexpr int NODE_OFF = -8192;   // row exponent of a node on which every projector of the cell is zero
constexpr int NONFINITE = 1 << 20;   // column exponent that marks an infinity or a NaN
constexpr unsigned long long DG_BIAS = 0x80808080808080ull;

// rows (nodes or coefficients) of VT FP16 digits; the 16-byte pieces of a row are placed so
// that the eight rows of an ldmatrix tile fall into different banks
template <int VT>
__device__ __forceinline__ int piece(int row, int c) {
  constexpr int PER = 128 / (2 * VT);   // rows per 128 bytes
  return row * (VT * 2) + ((c ^ ((row / PER) & (VT / 8 - 1))) << 4);
}

// bytes b0, b1 (a digit + 128 each) of a word as two FP16 digits
__device__ __forceinline__ unsigned digits2(unsigned w, unsigned sel) {
  const unsigned h = __byte_perm(w, 0x64646464u, sel);   // 1024 + byte
  unsigned r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0x64806480u));   // - 1152
  return r;
}

// the digits of two adjacent vectors of one row: plane d at sm + d * plane
__device__ __forceinline__ void store_digits(unsigned char *sm, int plane, int at, long long a, long long b) {
  const unsigned long long ua = (unsigned long long)a + DG_BIAS, ub = (unsigned long long)b + DG_BIAS;
  const unsigned al = (unsigned)ua, ah = (unsigned)(ua >> 32), bl = (unsigned)ub, bh = (unsigned)(ub >> 32);
  const unsigned t[4] = {__byte_perm(al, bl, 0x5140), __byte_perm(al, bl, 0x7362), __byte_perm(ah, bh, 0x5140),
                         __byte_perm(ah, bh, 0x7362)};
#pragma unroll
  for (int d = 0; d < DG; ++d)
    *reinterpret_cast<unsigned *>(sm + d * plane + at) = digits2(t[d / 2], (d & 1) ? 0x4342 : 0x4140);
}

__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm2(unsigned &r0, unsigned &r1, unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void mma16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// accumulators of a 16 x 16 tile (two 8-column mma tiles) and its 64-bit sums
struct Tile {
  float c[2][DG_SUMS][4];
  long long s[2][4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int g = 0; g < DG_SUMS; ++g)
#pragma unroll
        for (int i = 0; i < 4; ++i) c[n][g][i] = 0.f;
  }
  // one k step: A digits from img (one 16 x 16 tile of P, lane order), B digits from the rows
  // row0 .. row0 + 15 of the planes (row_of: this lane's ldmatrix row within them)
  template <int VT>
  __device__ __forceinline__ void step(const uint2 *__restrict__ img, unsigned sm, int plane, int row0, int half) {
    const int lane = threadIdx.x & 31;
    unsigned a[DG][4];
#pragma unroll
    for (int d = 0; d < DG; ++d) {
      const uint2 q = __ldg(img + d * 32 + lane);
      a[d][0] = digits2(q.x, 0x4140);
      a[d][1] = digits2(q.x, 0x4342);
      a[d][2] = digits2(q.y, 0x4140);
      a[d][3] = digits2(q.y, 0x4342);
    }
    // ldmatrix: lanes 0-15 address the 16 rows of one digit, lanes 16-31 those of the next
    const int row = row0 + (lane & 15);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const unsigned at = sm + piece<VT>(row, half * 2 + n) + ((lane >> 4) ? plane : 0);
      unsigned b[DG + 1][2];
#pragma unroll
      for (int d = 0; d < DG - 1; d += 2) {
        unsigned r[4];
        ldsm4(r, at + d * plane);
        b[d][0] = r[0];
        b[d][1] = r[1];
        b[d + 1][0] = r[2];
        b[d + 1][1] = r[3];
      }
      ldsm2(b[DG - 1][0], b[DG - 1][1], sm + piece<VT>(row, half * 2 + n) + (DG - 1) * plane);
#pragma unroll
      for (int i = DG - 1; i >= 0; --i)
#pragma unroll
        for (int j = DG - 1; j >= 0; --j)
          if (i + j >= 5) mma16(c[n][i + j - 5], a[i], b[j][0], b[j][1]);
    }
  }
  // s += the accumulators in units of 2^(72 - sh) (operand units), rounded; accumulators cleared
  __device__ __forceinline__ void flush(int sh) {
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        auto dig = [&](int g) { return __float2int_rz(c[n][g][i]); };
        long long lo = dig(0), hi = dig(4);
        fx_mad(lo, dig(1), 1 << 8);
        fx_mad(lo, dig(2), 1 << 16);
        fx_mad(lo, dig(3), 1 << 24);
        fx_mad(hi, dig(5), 1 << 8);
        fx_mad(hi, dig(6), 1 << 16);
        fx_mad(hi, dig(7), 1 << 24);
        hi += lo >> 32;
        s[n][i] += (long long)((unsigned long long)hi << sh) + ((((unsigned)lo >> (31 - sh)) + 1) >> 1);
      }
    clear();
  }
};

// bits left for the sums: |sum| <= 2^(36 + log2 K) units of 2^72, 2^62 units of 2^(72 - sh)
__host__ __device__ __forceinline__ int sum_shift(int K) {
  int b = 0;
  while ((1 << b) < K) ++b;
  return 26 - b;
}

struct FxNl {
  int n, p, N1, own, kt;          // kt: tiles of 16 owned nodes
  int bp;                         // pairs of one batch of the expansion
  const int *own_off, *own_atom;
  const unsigned char *proj, *exp;   // digit images (operand A of the projection, of the expansion)
  const int *sP;                  // exponent per pair and projector: |P(o) 2^-r(o)| < 2^sP
  const short *r;                 // ncells x own: row exponents (NODE_OFF: P is zero there)
  const unsigned *mask;           // per pair: bit t set when a node of tile t has a nonzero value
};

// pair k, node tile t, projector tile m of an image with MT projector tiles
template <int MT>
__device__ __forceinline__ const uint2 *image(const unsigned char *img, size_t k, int kt, int t, int m) {
  return reinterpret_cast<const uint2 *>(img) + ((k * kt + t) * MT + m) * (DG * 32);
}

// largest common exponent of each of the VT vectors over the threads of the block
template <int VT>
__device__ __forceinline__ void max_of_vectors(int (&E)[2], int *red, int *Em) {
  constexpr int VP = VT / 2;   // thread: vectors 2 (tid % VP) and the next
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int o = VP; o < 32; o <<= 1)
#pragma unroll
    for (int i = 0; i < 2; ++i) E[i] = max(E[i], __shfl_xor_sync(0xffffffffu, E[i], o));
  if (lane < VP) {
    red[warp * VT + 2 * lane] = E[0];
    red[warp * VT + 2 * lane + 1] = E[1];
  }
  __syncthreads();
  if (tid < VT) {
    int m = red[tid];
    for (int w = 1; w < 8; ++w) m = max(m, red[w * VT + tid]);
    Em[tid] = m;
  }
  __syncthreads();
}

// Projection: one cell and VT vectors per block, a warp per (pair, 16 projectors, 16 vectors).
// The digits of the cell's rows are made once and serve all of its pairs; node tiles on which a
// pair is zero are skipped.
// What bounds it: dependent issue of the digit steps (34 digit products per 16 x 8 x 16 tile keep
// the tensor pipe 40% busy; the rest makes and flushes digits).  Projection and expansion of
// 256 vectors of 16^3 cells of degree 6 with 64 atoms take 7.4 ms with the couplings, with FP64
// FMAs on the nonzero entries 24.8 ms (FP64 pipe 80-95% busy).  Loading the next tile's bytes
// ahead of the products was slower (9.5 against 9.2 ms when the step was first made: conversions done twice).
template <int NPAD, int VT, bool SCALED>
__global__ void __launch_bounds__(256, 2) k_fx_project(FxNl A, const double *__restrict__ X, int64_t ldx, int ncols,
                                                       const double *__restrict__ rowscale, double *__restrict__ U) {
  constexpr int MT = NPAD / 16, H = VT / 16, VP = VT / 2, ROWS = 256 / VP;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ int ooff[512];
  __shared__ short rs[512];
  __shared__ int red[8 * VT], Em[VT];
  const int ntile = (ncols + VT - 1) / VT;
  const int e = blockIdx.x / ntile, v0 = (blockIdx.x - e * ntile) * VT;
  const int k0 = A.own_off[e], k1 = A.own_off[e + 1];
  if (k0 == k1) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int own = A.own, plane = A.kt * 16 * VT * 2;
  for (int o = tid; o < own; o += 256) {
    ooff[o] = owned_offset(o, A.p, A.N1);
    rs[o] = A.r[(size_t)e * own + o];
  }
  const int64_t base = owned_base(e, A.n, A.p, A.N1);
  __syncthreads();
  {
    const int vp = tid % VP, r0 = tid / VP, v = v0 + 2 * vp;
    const bool ok0 = v < ncols, ok1 = v + 1 < ncols;
    auto get = [&](int o, double &x, double &y) {
      const int64_t d = base + ooff[o];
      const double *p = X + d * ldx + v;
      x = ok0 ? p[0] : 0.0;
      y = ok1 ? p[1] : 0.0;
      if (SCALED) {
        const double m = rowscale[d];
        x *= m;
        y *= m;
      }
    };
    // exponent that a value counts with; what stands on a node without projectors does not enter
    auto field = [&](double x, int o) {
      const int f = fx_field(x), r = rs[o];
      return f == 0x7ff && r != NODE_OFF ? NONFINITE : f + r;
    };
    // the values of the first NR rows of the thread (all of them up to degree 6) stay in
    // registers between the maxima and the digits
    constexpr int NR = 14;
    double x[NR], y[NR];
    int E[2] = {NODE_OFF / 2, NODE_OFF / 2};
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      x[i] = y[i] = 0.0;
      if (r0 + i * ROWS < own) get(r0 + i * ROWS, x[i], y[i]);
    }
    for (int o = r0 + NR * ROWS; o < own; o += ROWS) {
      double a, b;
      get(o, a, b);
      E[0] = max(E[0], field(a, o));
      E[1] = max(E[1], field(b, o));
    }
#pragma unroll
    for (int i = 0; i < NR; ++i)
      if (r0 + i * ROWS < own) {
        E[0] = max(E[0], field(x[i], r0 + i * ROWS));
        E[1] = max(E[1], field(y[i], r0 + i * ROWS));
      }
    max_of_vectors<VT>(E, red, Em);
    E[0] = Em[2 * vp];
    E[1] = Em[2 * vp + 1];
    auto put = [&](int o, double a, double b) {
      const int r = o < own ? rs[o] : 0;
      store_digits(sm, plane, piece<VT>(o, vp >> 2) + (vp & 3) * 4, a == 0.0 ? 0 : fx_round<DG_BITS>(a, E[0] - r),
                   b == 0.0 ? 0 : fx_round<DG_BITS>(b, E[1] - r));
    };
#pragma unroll
    for (int i = 0; i < NR; ++i)
      if (r0 + i * ROWS < A.kt * 16) put(r0 + i * ROWS, x[i], y[i]);
    for (int o = r0 + NR * ROWS; o < A.kt * 16; o += ROWS) {
      double a = 0.0, b = 0.0;
      if (o < own) get(o, a, b);
      put(o, a, b);
    }
  }
  __syncthreads();
  const unsigned smu = (unsigned)__cvta_generic_to_shared(sm);
  const int sh = sum_shift(A.kt * 16);
  for (int u = warp; u < (k1 - k0) * (MT * H); u += 8) {
    const int half = u % H, mt = (u / H) % MT;
    const size_t k = k0 + u / (MT * H);
    Tile t;
    t.clear();
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) t.s[n][i] = 0;
    int left = FLUSH;
    for (unsigned m = A.mask[k]; m; m &= m - 1) {
      const int kt = __ffs(m) - 1;
      t.step<VT>(image<MT>(A.proj, k, A.kt, kt, mt), smu, plane, kt * 16, half);
      if (--left == 0) {
        t.flush(sh);
        left = FLUSH;
      }
    }
    t.flush(sh);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int al = mt * 16 + r * 8 + (lane >> 2);
      const int ex = 72 - sh - 2 * DG_BITS + A.sP[k * NPAD + al] - 1022;
      double *Uk = U + (k * NPAD + al) * ncols;
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int l = half * 16 + n * 8 + 2 * (lane & 3) + j, v = v0 + l;
          if (v < ncols)
            Uk[v] = Em[l] >= NONFINITE ? __longlong_as_double(0x7ff8000000000000ll)
                                       : fx_to_small(t.s[n][2 * r + j], ex + Em[l]);
        }
    }
  }
}

// Expansion: one cell and VT vectors per block, a warp per (16 owned nodes, 16 vectors).  The
// coefficients W of the cell's pairs, scaled by the pairs' projector exponents, are cut into
// digits in batches of bp pairs; sums of several batches wait in shared memory (digits
// and sums of 32 vectors at degree 6 let two blocks share an SM).  The two coefficient sets of the
// recurrence give one output each: T from W_S, then R_X from W_H.  (With the sums of W_S kept
// beside those of W_H until one emission, one block fits an SM: a step of 128 vectors on 12^3
// cells 13.7 instead of 8.0 ms.)
// What bounds it: dependent issue of the digit steps, as in the projection.
template <int NPAD, int VT, int MODE>
__global__ void __launch_bounds__(256, 2) k_fx_expand(FxNl N, ExpArgs A, const double *__restrict__ W1,
                                                      const double *__restrict__ W2) {
  constexpr int MT = NPAD / 16, H = VT / 16, VP = VT / 2, ROWS = 256 / VP;
  constexpr int NW = (MODE == EXP_RECURRENCE) ? 2 : 1;
  const int BP = N.bp, plane = BP * NPAD * VT * 2;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ int red[8 * VT], Em[NW][VT], ooff[512];
  __shared__ short rs[512];
  const int ncols = A.ncols, ntile = (ncols + VT - 1) / VT;
  const int e = blockIdx.x / ntile, v0 = (blockIdx.x - e * ntile) * VT;
  const int k0 = N.own_off[e], np = N.own_off[e + 1] - k0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, own = N.own;
  for (int o = tid; o < own; o += 256) {   // (synchronised with the maxima)
    ooff[o] = owned_offset(o, N.p, N.N1);
    rs[o] = np ? N.r[(size_t)e * own + o] : NODE_OFF;
  }
  const int vp = tid % VP, r0 = tid / VP;
  const bool ok0 = v0 + 2 * vp < ncols, ok1 = v0 + 2 * vp + 1 < ncols;
  // W of row r (pair r / NPAD of the cell, projector r % NPAD), 0 where there is none
  auto get = [&](const double *W, int r, double &x, double &y) {
    const double *p = W + ((size_t)N.own_atom[k0 + r / NPAD] * NPAD + r % NPAD) * ncols + v0 + 2 * vp;
    x = ok0 ? p[0] : 0.0;
    y = ok1 ? p[1] : 0.0;
  };
  for (int w = 0; w < NW; ++w) {
    const double *W = w ? W2 : W1;
    int E[2] = {-NONFINITE, -NONFINITE};
    for (int r = r0; r < np * NPAD; r += ROWS) {
      double x, y;
      get(W, r, x, y);
      const int s = N.sP[(size_t)k0 * NPAD + r], fx = fx_field(x), fy = fx_field(y);
      if (x != 0.0) E[0] = max(E[0], fx == 0x7ff ? NONFINITE : fx + s);
      if (y != 0.0) E[1] = max(E[1], fy == 0x7ff ? NONFINITE : fy + s);
    }
    max_of_vectors<VT>(E, red, Em[w]);
  }
  const unsigned smu = (unsigned)__cvta_generic_to_shared(sm);
  const int sh = sum_shift(max(np, 1) * NPAD), nbatch = max(1, (np + BP - 1) / BP);
  const int units = N.kt * H;
  long long *S = reinterpret_cast<long long *>(sm + DG * plane);   // [kt * 16][VT]
  const int64_t base = owned_base(e, N.n, N.p, N.N1);
  for (int w = 0; w < NW; ++w) {
    const double *W = w ? W2 : W1;
    for (int b = 0; b < nbatch; ++b) {
      const int pb = min(BP, np - b * BP);                          // pairs of this batch
      if (w || b) __syncthreads();
      for (int r = r0; r < pb * NPAD; r += ROWS) {
        double x, y;
        get(W, b * BP * NPAD + r, x, y);
        const int s = N.sP[((size_t)k0 + b * BP) * NPAD + r];
        store_digits(sm, plane, piece<VT>(r, vp >> 2) + (vp & 3) * 4,
                     x == 0.0 ? 0 : fx_round<DG_BITS>(x, Em[w][2 * vp] - s),
                     y == 0.0 ? 0 : fx_round<DG_BITS>(y, Em[w][2 * vp + 1] - s));
      }
      __syncthreads();
      for (int u = warp; u < units; u += 8) {
        const int half = u % H, kt = u / H;
        Tile t;
        t.clear();
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) t.s[n][i] = 0;
        const size_t kb = k0 + b * BP;
        // the pairs of the batch with a nonzero value on these nodes
        unsigned pm = __ballot_sync(0xffffffffu, lane < pb && (N.mask[kb + min(lane, pb - 1)] >> kt & 1u));
        for (; pm; pm &= pm - 1) {
          const int q = __ffs(pm) - 1;
#pragma unroll
          for (int m = 0; m < MT; ++m)
            t.step<VT>(image<MT>(N.exp, kb + q, N.kt, kt, m), smu, plane, q * NPAD + m * 16, half);
        }
        t.flush(sh);
        const bool last = b + 1 == nbatch;
        const int l0 = half * 16 + 2 * (lane & 3), e0 = 72 - sh - 2 * DG_BITS - 1022;
        auto value = [&](long long y, int E, int r) {
          if (E >= NONFINITE) return r == NODE_OFF ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
          return fx_to_small(y, e0 + E + r);
        };
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int o = kt * 16 + r * 8 + (lane >> 2);
          long long *Sp = S + o * VT + l0;
          if (b > 0)
#pragma unroll
            for (int i = 0; i < 4; ++i) t.s[i >> 1][2 * r + (i & 1)] += Sp[(i >> 1) * 8 + (i & 1)];
          if (!last) {
#pragma unroll
            for (int i = 0; i < 4; ++i) Sp[(i >> 1) * 8 + (i & 1)] = t.s[i >> 1][2 * r + (i & 1)];
            continue;
          }
          if (o >= own) continue;
          const int64_t d = base + ooff[o];
          const int ro = rs[o];
          const double m = MODE == EXP_SET ? 0.0 : static_cast<const double *>(A.mdinv)[d];
          double *Y = static_cast<double *>(A.Y) + d * A.ldy + v0 + l0;
          const double *Xi = MODE == EXP_SET ? nullptr : static_cast<const double *>(A.Xin) + d * A.ldx + v0 + l0;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = (i >> 1) * 8 + (i & 1);
            if (v0 + l0 + c >= ncols) continue;
            const long long s = t.s[i >> 1][2 * r + (i & 1)];
            if (MODE == EXP_SET) {
              Y[c] = value(s, Em[0][l0 + c], ro);
            } else if (MODE == EXP_SINV) {
              Y[c] = m * (Xi[c] - value(s, Em[0][l0 + c], ro));
            } else if (w == 0) {
              Y[c] = m * (Xi[c] - value(s, Em[0][l0 + c], ro));
            } else {
              double *RX = static_cast<double *>(A.RX) + d * A.ldx + v0 + l0 + c;
              const double bracket = -A.beta * Xi[c] - A.gamma * *RX + value(s, Em[NW - 1][l0 + c], ro);
              *RX = fma(A.c64[v0 + l0 + c], static_cast<const double *>(A.Y0)[d * A.ldy0 + v0 + l0 + c], bracket);
            }
          }
        }
      }
    }
  }
}

// Cells of one owned node (degree 1) fill one of the 16 rows of a digit tile: FP64 FMAs over the
// nonzero entries instead, lane = vector.  Bound by the per-pair partials (16 values written and read
// again for one node) and, for few vectors, by the chain over the pairs of a cell, which four warps of the
// expansion share.  On 24^3 cells with 216 atoms, 64 vectors: approximate inverse overlap 0.90
// ms (digits 2.17), H 1.06 (2.26), a filter of 8 steps 11.1 (29.4).  For the eight nodes of degree 2
// the digits are faster (16^3 cells, 64 vectors: H 0.82 ms, FMAs in this form 1.81).
template <int NPAD, bool SCALED>
__global__ void __launch_bounds__(256) k_one_project(FxNl A, const double *__restrict__ P, const double *__restrict__ X,
                                                     int64_t ldx, int ncols, const double *__restrict__ rowscale,
                                                     double *__restrict__ U) {
  const int ntile = (ncols + 31) / 32;
  const int e = blockIdx.x / ntile, v = (blockIdx.x - e * ntile) * 32 + (threadIdx.x & 31);
  const int k0 = A.own_off[e], k1 = A.own_off[e + 1];
  if (k0 == k1 || v >= ncols) return;
  const int64_t d = owned_base(e, A.n, A.p, A.N1);
  double x = X[d * ldx + v];
  if (SCALED) x *= rowscale[d];
  for (int u = threadIdx.x >> 5; u < (k1 - k0) * NPAD; u += 8) {
    const double c = __ldg(P + (size_t)k0 * NPAD + u);
    U[((size_t)k0 * NPAD + u) * ncols + v] = c != 0.0 ? c * x : 0.0;
  }
}

template <int NPAD, int MODE>
__global__ void __launch_bounds__(128) k_one_expand(FxNl N, ExpArgs A, const double *__restrict__ P,
                                                    const double *__restrict__ W1, const double *__restrict__ W2) {
  constexpr int NW = (MODE == EXP_RECURRENCE) ? 2 : 1;
  __shared__ double part[NW][4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ncols = A.ncols, ntile = (ncols + 31) / 32;
  const int e = blockIdx.x / ntile, v = (blockIdx.x - e * ntile) * 32 + lane, vc = min(v, ncols - 1);
  double s[NW] = {};
  for (int k = N.own_off[e] + warp; k < N.own_off[e + 1]; k += 4) {
    const size_t w = (size_t)N.own_atom[k] * NPAD * ncols + vc;
#pragma unroll
    for (int al = 0; al < NPAD; ++al) {
      const double c = __ldg(P + (size_t)k * NPAD + al);
      if (c == 0.0) continue;
#pragma unroll
      for (int i = 0; i < NW; ++i) s[i] = fma(c, __ldg((i ? W2 : W1) + w + (size_t)al * ncols), s[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < NW; ++i) part[i][warp][lane] = s[i];
  __syncthreads();
  if (warp || v >= ncols) return;
#pragma unroll
  for (int i = 0; i < NW; ++i) s[i] = (part[i][0][lane] + part[i][1][lane]) + (part[i][2][lane] + part[i][3][lane]);
  const int64_t d = owned_base(e, N.n, N.p, N.N1);
  double *Y = static_cast<double *>(A.Y) + d * A.ldy + v;
  if (MODE == EXP_SET) {
    *Y = s[0];
    return;
  }
  const double x = static_cast<const double *>(A.Xin)[d * A.ldx + v];
  *Y = static_cast<const double *>(A.mdinv)[d] * (x - s[0]);
  if (MODE == EXP_RECURRENCE) {
    double *RX = static_cast<double *>(A.RX) + d * A.ldx + v;
    *RX = fma(A.c64[v], static_cast<const double *>(A.Y0)[d * A.ldy0 + v], -A.beta * x - A.gamma * *RX + s[NW - 1]);
  }
}

// row exponents of one cell per block: that of the largest entry of the row over the cell's pairs
__global__ void __launch_bounds__(128) k_node_scales(int own, int npad, const int *__restrict__ own_off,
                                                     const double *__restrict__ P, short *__restrict__ r) {
  const int e = blockIdx.x, k0 = own_off[e], k1 = own_off[e + 1];
  for (int o = threadIdx.x; o < own; o += 128) {
    int f = NODE_OFF;
    for (int k = k0; k < k1; ++k)
      for (int al = 0; al < npad; ++al) {
        const double x = P[((size_t)k * own + o) * npad + al];
        if (x != 0.0) f = max(f, fx_field(x) - 1022);
      }
    r[(size_t)e * own + o] = (short)f;
  }
}

// digit images, exponents and node-tile masks of one pair per block
__global__ void __launch_bounds__(128) k_build_digits(int ncells, int own, int kt, int npad,
                                                      const int *__restrict__ own_off, const double *__restrict__ P,
                                                      const short *__restrict__ r, unsigned char *__restrict__ proj,
                                                      unsigned char *__restrict__ exp, int *__restrict__ sP,
                                                      unsigned *__restrict__ mask) {
  __shared__ int E[32];
  __shared__ unsigned ms;
  const size_t k = blockIdx.x;
  int e = 0;   // cell of the pair: own_off[e] <= k < own_off[e + 1]
  for (int n = ncells; n > 1;) {
    const int h = n / 2;
    if (own_off[e + h] <= (int)k) e += h, n -= h;
    else n = h;
  }
  const short *rs = r + (size_t)e * own;
  const int mt = npad / 16;
  const double *Pk = P + k * own * npad;
  if (threadIdx.x < 32) E[threadIdx.x] = NODE_OFF / 2;
  if (threadIdx.x == 0) ms = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < own * npad; i += 128) {
    if (Pk[i] == 0.0) continue;
    atomicMax(&E[i % npad], fx_field(Pk[i]) - rs[i / npad]);
    atomicOr(&ms, 1u << (i / npad / 16));
  }
  __syncthreads();
  if (threadIdx.x < npad) sP[k * npad + threadIdx.x] = E[threadIdx.x] - 1022;
  if (threadIdx.x == 0) mask[k] = ms;
  for (int i = threadIdx.x; i < kt * 16 * npad; i += 128) {
    const int o = i / npad, al = i % npad;
    const double x = o < own ? Pk[(size_t)o * npad + al] : 0.0;
    const long long V = x == 0.0 ? 0 : fx_round<DG_BITS>(x, E[al] + rs[o]);
    const unsigned long long bytes = (unsigned long long)V + DG_BIAS;
    // element (r, c) of a 16 x 16 A tile: lane, byte of its eight
    auto put = [&](unsigned char *img, int r, int c) {
      const size_t tile = ((k * kt + o / 16) * mt + al / 16) * DG;
      const int lane = (r & 7) * 4 + ((c & 7) >> 1), byte = ((r >> 3) + 2 * (c >> 3)) * 2 + (c & 1);
      for (int d = 0; d < DG; ++d) img[((tile + d) * 32 + lane) * 8 + byte] = (unsigned char)(bytes >> (8 * d));
    };
    put(proj, al & 15, o & 15);
    put(exp, o & 15, al & 15);
  }
}

FxNl fx_args(const paw_context *c) {
  FxNl N{};
  N.n = c->n;
  N.p = c->p;
  N.N1 = c->N1;
  N.own = c->own;
  N.kt = (c->own + 15) / 16;
  N.own_off = c->own_off.as<int>();
  N.own_atom = c->own_atom.as<int>();
  N.proj = c->own_proj_dg.as<unsigned char>();
  N.exp = c->own_exp_dg.as<unsigned char>();
  N.sP = c->own_sP.as<int>();
  N.r = c->own_r.as<short>();
  N.mask = c->own_mask.as<unsigned>();
  return N;
}

template <int NPAD, int VT>
void launch_project(paw_context *c, const double *X, int ldx, int ncols, const double *rowscale, double *U,
                    cudaStream_t s) {
  const FxNl N = fx_args(c);
  const size_t shm = (size_t)DG * N.kt * 16 * VT * 2;
  auto kern = rowscale ? k_fx_project<NPAD, VT, true> : k_fx_project<NPAD, VT, false>;
  PAW_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  kern<<<(unsigned)((int64_t)c->ncells * ((ncols + VT - 1) / VT)), 256, shm, s>>>(N, X, ldx, ncols, rowscale, U);
  PAW_LAUNCH_CHECK("k_fx_project");
}

// shared memory of the expansion: the digits of a batch and, for cells of several, the sums
int expand_pairs(const paw_context *c) {
  return (c->max_own_pairs > EXP_K / c->npad ? EXP_K_MANY : EXP_K) / c->npad;
}
size_t expand_smem(const paw_context *c, int vt) {
  const int bp = expand_pairs(c);
  const size_t sums = c->max_own_pairs > bp ? ((c->own + 15) / 16) * 16 * sizeof(long long) : 0;
  return (size_t)vt * (DG * bp * c->npad * 2 + sums);
}

template <int NPAD, int VT, int MODE>
void launch_expand(paw_context *c, const ExpArgs &A, const double *W1, const double *W2, cudaStream_t s) {
  FxNl N = fx_args(c);
  N.bp = expand_pairs(c);
  const size_t shm = expand_smem(c, VT);
  PAW_CUDA(cudaFuncSetAttribute(k_fx_expand<NPAD, VT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  k_fx_expand<NPAD, VT, MODE><<<(unsigned)((int64_t)c->ncells * ((A.ncols + VT - 1) / VT)), 256, shm, s>>>(N, A, W1,
                                                                                                         W2);
  PAW_LAUNCH_CHECK("k_fx_expand");
}

template <int NPAD, int VT>
void expand_mode(paw_context *c, int mode, const ExpArgs &A, const double *W1, const double *W2, cudaStream_t s) {
  if (mode == EXP_SET)
    launch_expand<NPAD, VT, EXP_SET>(c, A, W1, W2, s);
  else if (mode == EXP_SINV)
    launch_expand<NPAD, VT, EXP_SINV>(c, A, W1, W2, s);
  else
    launch_expand<NPAD, VT, EXP_RECURRENCE>(c, A, W1, W2, s);
}

}  // namespace

void nlfx_build(paw_context *c, const double *P) {
  if (c->nown_pairs == 0) return;
  if (c->own == 1) {
    const size_t bytes = sizeof(double) * (size_t)c->nown_pairs * c->npad;
    c->own_P64.ensure(bytes, &c->dev_bytes);
    PAW_CUDA(cudaMemcpy(c->own_P64.ptr, P, bytes, cudaMemcpyDeviceToDevice));
    return;
  }
  const int kt = (c->own + 15) / 16, mt = c->npad / 16;
  const size_t img = (size_t)c->nown_pairs * kt * mt * DG * 256;
  c->own_proj_dg.ensure(img, &c->dev_bytes);
  c->own_exp_dg.ensure(img, &c->dev_bytes);
  c->own_sP.ensure(sizeof(int) * (size_t)c->nown_pairs * c->npad, &c->dev_bytes);
  c->own_mask.ensure(sizeof(unsigned) * (size_t)c->nown_pairs, &c->dev_bytes);
  c->own_r.ensure(sizeof(short) * (size_t)c->ncells * c->own, &c->dev_bytes);
  k_node_scales<<<(unsigned)c->ncells, 128>>>(c->own, c->npad, c->own_off.as<int>(), P, c->own_r.as<short>());
  PAW_LAUNCH_CHECK("k_node_scales");
  k_build_digits<<<(unsigned)c->nown_pairs, 128>>>(c->ncells, c->own, kt, c->npad, c->own_off.as<int>(), P,
                                                   c->own_r.as<short>(), c->own_proj_dg.as<unsigned char>(),
                                                   c->own_exp_dg.as<unsigned char>(), c->own_sP.as<int>(),
                                                   c->own_mask.as<unsigned>());
  PAW_LAUNCH_CHECK("k_build_digits");
}

// Blocks of 32 vectors share the digits and the projector images of a cell between two tiles of
// 16; 16 vectors where there are no more, and where the rows of 32 vectors would not fit into
// shared memory (degree 8).
constexpr size_t FX_SMEM_MAX = 200 * 1024;

void nlfx_project(paw_context *c, const double *X, int ldx, int ncols, const double *rowscale, double *U,
                  cudaStream_t s) {
  PAW_REQUIRE(c->own <= 512 && (c->npad == 16 || c->npad == 32), PAW_ERR_UNSUPPORTED,
              "projection tile exceeds shared memory (degree too high)");
  if (c->own == 1) {
    auto run = [&](auto kern) {
      kern<<<(unsigned)((int64_t)c->ncells * ((ncols + 31) / 32)), 256, 0, s>>>(fx_args(c), c->own_P64.as<double>(), X, ldx,
                                                                                ncols, rowscale, U);
      PAW_LAUNCH_CHECK("k_one_project");
    };
    if (c->npad == 16)
      rowscale ? run(k_one_project<16, true>) : run(k_one_project<16, false>);
    else
      rowscale ? run(k_one_project<32, true>) : run(k_one_project<32, false>);
    return;
  }
  const bool narrow = ncols <= 16 || (size_t)DG * (c->own + 15) * 64 > FX_SMEM_MAX;
  if (c->npad == 16)
    narrow ? launch_project<16, 16>(c, X, ldx, ncols, rowscale, U, s)
           : launch_project<16, 32>(c, X, ldx, ncols, rowscale, U, s);
  else
    narrow ? launch_project<32, 16>(c, X, ldx, ncols, rowscale, U, s)
           : launch_project<32, 32>(c, X, ldx, ncols, rowscale, U, s);
}

void nlfx_expand(paw_context *c, int mode, const ExpArgs &A, const double *W1, const double *W2, cudaStream_t s) {
  PAW_REQUIRE(c->max_own_pairs <= PAIRS_PER_CELL_MAX && c->own <= 512, PAW_ERR_UNSUPPORTED,
              "too many atoms on one cell for the expansion kernel");
  if (c->own == 1) {
    auto run = [&](auto kern) {
      kern<<<(unsigned)((int64_t)c->ncells * ((A.ncols + 31) / 32)), 128, 0, s>>>(fx_args(c), A, c->own_P64.as<double>(), W1,
                                                                                  W2);
      PAW_LAUNCH_CHECK("k_one_expand");
    };
    auto of = [&](auto np) {
      constexpr int NPAD = decltype(np)::value;
      mode == EXP_SET    ? run(k_one_expand<NPAD, EXP_SET>)
      : mode == EXP_SINV ? run(k_one_expand<NPAD, EXP_SINV>)
                         : run(k_one_expand<NPAD, EXP_RECURRENCE>);
    };
    c->npad == 16 ? of(std::integral_constant<int, 16>{}) : of(std::integral_constant<int, 32>{});
    return;
  }
  const bool narrow = A.ncols <= 16 || expand_smem(c, 32) > FX_SMEM_MAX;
  if (c->npad == 16)
    narrow ? expand_mode<16, 16>(c, mode, A, W1, W2, s) : expand_mode<16, 32>(c, mode, A, W1, W2, s);
  else
    narrow ? expand_mode<32, 16>(c, mode, A, W1, W2, s) : expand_mode<32, 32>(c, mode, A, W1, W2, s);
}

}  // namespace pawfe
