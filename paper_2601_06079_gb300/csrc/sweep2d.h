// Row arithmetic of the explicit 2-D step, shared by the kernels that sweep a
// column strip downwards (k_explicit2d.cu: planes in memory; k_onchip2d.cu:
// planes in shared memory), so that all of them give bitwise the same nodes.
//
// A lane holds kP adjacent pairs of columns as packed FP32 (f32x2).  Values
// at the two Gauss points of an interval, g_hi a + g_lo b and g_lo a + g_hi b,
// are carried without their common factor g_hi: a + rho b and rho a + b with
// rho = g_lo / g_hi, one FMA each with no difference to form first.  The
// factors (g_hi^2 for the interpolation, g_hi^2 for the weights back to the
// nodes) are folded into the polynomial's coefficients on the host.  For the
// double well expanded about u = 1/2 the polynomial is odd, p1 v + p3 v^3 =
// p3 (v^2 + p1/p3) v: two operations per point, and p3 multiplies the node's
// sum (kOdd).  Against differences and Horner's rule per point this takes 33
// packed operations per row instead of 41 (Cahn-Hilliard on square cells).
//
// Every sum pairs mirror images before anything else (south with north, west
// with east), so a strip swept over mirrored data gives bitwise mirrored
// results: images beyond a zero-flux boundary need not be stored and re-read.
#pragma once

#include "pf_internal.h"

namespace pf {
namespace sweep {

typedef unsigned long long u64;  // packed FP32 pair: low half = lower column

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ u64 pk(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float plo(u64 v) {
  float l;
  asm("{ .reg .f32 t; mov.b64 {%0, t}, %1; }" : "=f"(l) : "l"(v));
  return l;
}
__device__ __forceinline__ float phi(u64 v) {
  float h;
  asm("{ .reg .f32 t; mov.b64 {t, %0}, %1; }" : "=f"(h) : "l"(v));
  return h;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Packed constants of one mesh (Explicit2DArgs::pair, laid out by
// pack_explicit2d): rho; the odd form's p1/p3 and p3; p0..p3; per stencil
// a = c0 - cd, b = cd, c0, cx, cy, cd.
struct Coef {
  const u64* c;
  __device__ __forceinline__ u64 rho() const { return c[0]; }
  __device__ __forceinline__ u64 r() const { return c[1]; }
  __device__ __forceinline__ u64 s() const { return c[2]; }
  __device__ __forceinline__ u64 p(int i) const { return c[3 + i]; }
  __device__ __forceinline__ u64 k(int stage, int i) const { return c[7 + 6 * stage + i]; }
};

// f' at one Gauss point of both columns, without the factor p3 if kOdd
template <bool kOdd>
__device__ __forceinline__ u64 well(u64 v, const Coef& K) {
  if constexpr (kOdd) return mul2(fma2(v, v, K.r()), v);
  return fma2(fma2(fma2(K.p(3), v, K.p(2)), v, K.p(1)), v, K.p(0));
}

// init + F + K v at the centre row of south / centre / north values and row
// helpers (kIso: 3-sums of the rows, K v = a v + b (9-sum); general: west +
// east sums).  kInit: with init, otherwise without.
template <bool kIso, bool kOdd, bool kInit>
__device__ __forceinline__ u64 node(u64 init, u64 F, u64 s, u64 c, u64 n, u64 as, u64 ac, u64 an,
                                    const Coef& K, int st) {
  const u64 c0 = kIso ? K.k(st, 0) : K.k(st, 2);
  u64 o;
  if constexpr (kOdd)
    o = kInit ? fma2(c0, c, init) : mul2(c0, c);
  else
    o = fma2(c0, c, kInit ? add2(init, F) : F);
  if constexpr (kIso) {
    o = fma2(K.k(st, 1), add2(add2(as, an), ac), o);
  } else {
    o = fma2(K.k(st, 3), ac, o);
    o = fma2(K.k(st, 4), add2(s, n), o);
    o = fma2(K.k(st, 5), add2(as, an), o);
  }
  if constexpr (kOdd) o = fma2(K.s(), F, o);
  return o;
}

// init + K v (the Cahn-Hilliard c stage)
template <bool kIso>
__device__ __forceinline__ u64 stencil(u64 init, u64 s, u64 c, u64 n, u64 as, u64 ac, u64 an,
                                       const Coef& K, int st) {
  if constexpr (kIso) return fma2(K.k(st, 1), add2(add2(as, an), ac), fma2(K.k(st, 0), c, init));
  return fma2(K.k(st, 5), add2(as, an),
              fma2(K.k(st, 4), add2(s, n), fma2(K.k(st, 3), ac, fma2(K.k(st, 2), c, init))));
}

// Row helpers of a row: west + east neighbours' sum (left: the column before
// the lane's first, right: the one after its last), plus the centre if kIso.
template <bool kIso, int kP>
__device__ __forceinline__ void row_aux(const u64 (&P)[kP], float left, float right,
                                        u64 (&x)[kP]) {
#pragma unroll
  for (int j = 0; j < kP; ++j) {
    const float w = j ? phi(P[j ? j - 1 : 0]) : left;
    const float e = j + 1 < kP ? plo(P[j + 1 < kP ? j + 1 : 0]) : right;
    const u64 hs = pk(w + phi(P[j]), plo(P[j]) + e);
    x[j] = kIso ? add2(P[j], hs) : hs;
  }
}

// Sliding window of a lane: rows k-1 and k-2 of the row k consumed next.
template <int kP>
struct Window {
  u64 c1[kP], c2[kP], x1[kP], x2[kP];      // own values and row helpers
  u64 am[kP], ap[kP];                      // x-interpolants of row k-1
  u64 tl[kP], th[kP];                      // element row k-2 -> node row k-1
  u64 mua[kP], mub[kP], mxa[kP], mxb[kP];  // Cahn-Hilliard: mu and helpers, rows k-3, k-2
};

// How far a row takes the window: its own interpolation, the element row
// above it, mu of row k-1 (Cahn-Hilliard), the finished row.
enum Stage { kInterp = 0, kElement = 1, kMu = 2, kOutput = 3 };

// Consumes row k (values P, neighbouring columns cl and cr); at kOutput o is
// the finished row k-1 (Allen-Cahn) or k-2 (Cahn-Hilliard).  The weights back
// in x bring each lane its left neighbour's share by a shuffle; lane 0 takes
// b0 instead if kEdge.
template <bool kCH, bool kIso, bool kOdd, int kP, int kStage, bool kEdge>
__device__ __forceinline__ void row(const u64 (&P)[kP], float cl, float cr, float b0,
                                    Window<kP>& w, const Coef& K, u64 (&o)[kP]) {
  u64 xr[kP], am[kP], ap[kP];
  row_aux<kIso, kP>(P, cl, cr, xr);
#pragma unroll
  for (int j = 0; j < kP; ++j) {
    // scalar FMAs: packed ones would first have to copy the shifted pair
    // together, and take the same time on the FMA pipe
    const float rho = plo(K.rho()), c0 = plo(P[j]), c1 = phi(P[j]);
    const float c2 = j + 1 < kP ? plo(P[j + 1 < kP ? j + 1 : 0]) : cr;
    am[j] = pk(fmaf(rho, c1, c0), fmaf(rho, c2, c1));
    ap[j] = pk(fmaf(rho, c0, c1), fmaf(rho, c1, c2));
  }
  if constexpr (kStage >= kElement) {
    u64 tl[kP], th[kP], F[kP];
    float bl = 0.0f;
    u64 A[kP], B[kP];
#pragma unroll
    for (int j = 0; j < kP; ++j) {  // element row k-1: four Gauss values, weights back in y
      const u64 fll = well<kOdd>(fma2(K.rho(), am[j], w.am[j]), K);
      const u64 flh = well<kOdd>(fma2(K.rho(), w.am[j], am[j]), K);
      const u64 fhl = well<kOdd>(fma2(K.rho(), ap[j], w.ap[j]), K);
      const u64 fhh = well<kOdd>(fma2(K.rho(), w.ap[j], ap[j]), K);
      tl[j] = fma2(K.rho(), fll, flh);  // node row k
      th[j] = fma2(K.rho(), fhl, fhh);
      if constexpr (kStage >= kMu) {  // node row k-1, then the weights back in x
        const u64 sl = add2(fma2(K.rho(), flh, fll), w.tl[j]);
        const u64 sh = add2(fma2(K.rho(), fhh, fhl), w.th[j]);
        A[j] = fma2(K.rho(), sh, sl);
        B[j] = fma2(K.rho(), sl, sh);
      }
    }
    if constexpr (kStage >= kMu) {
      bl = __shfl_up_sync(kFull, phi(B[kP - 1]), 1);
      if constexpr (kEdge) bl = (threadIdx.x & 31) ? bl : b0;
#pragma unroll
      for (int j = 0; j < kP; ++j)
        F[j] = pk(plo(A[j]) + (j ? phi(B[j ? j - 1 : 0]) : bl), phi(A[j]) + plo(B[j]));
      if constexpr (!kCH) {
#pragma unroll
        for (int j = 0; j < kP; ++j)
          o[j] = node<kIso, kOdd, true>(w.c1[j], F[j], w.c2[j], w.c1[j], P[j], w.x2[j], w.x1[j],
                                        xr[j], K, 0);
      } else {
        u64 mu[kP], mx[kP];
#pragma unroll
        for (int j = 0; j < kP; ++j)
          mu[j] = node<kIso, kOdd, false>(0, F[j], w.c2[j], w.c1[j], P[j], w.x2[j], w.x1[j],
                                          xr[j], K, 0);
        const float ml = __shfl_up_sync(kFull, phi(mu[kP - 1]), 1);
        const float mr = __shfl_down_sync(kFull, plo(mu[0]), 1);
        row_aux<kIso, kP>(mu, ml, mr, mx);
#pragma unroll
        for (int j = 0; j < kP; ++j) {
          if constexpr (kStage >= kOutput)
            o[j] = stencil<kIso>(w.c2[j], w.mua[j], w.mub[j], mu[j], w.mxa[j], w.mxb[j], mx[j], K,
                                 1);
          w.mua[j] = w.mub[j];
          w.mxa[j] = w.mxb[j];
          w.mub[j] = mu[j];
          w.mxb[j] = mx[j];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kP; ++j) {
      w.tl[j] = tl[j];
      w.th[j] = th[j];
    }
  }
#pragma unroll
  for (int j = 0; j < kP; ++j) {
    w.c2[j] = w.c1[j];
    w.x2[j] = w.x1[j];
    w.c1[j] = P[j];
    w.x1[j] = xr[j];
    w.am[j] = am[j];
    w.ap[j] = ap[j];
  }
}

// Planes with a mirror frame (k_explicit2d.cu, k_coupled2d.cu): a warp takes 64
// columns, a pair per lane, and writes the 60 of lanes 1..30.
constexpr int kPair = 2;                          // columns per lane
constexpr int kOutCols = 32 * kPair - 2 * kPair;  // 60 output columns per warp
constexpr int kGhost = 2;                         // width of the frame

// Output of one finished pair: real row y, real columns x (lo) and x+1 (hi),
// plus every ghost cell that mirrors it (rows -1, -2 <- 1, 2 and
// ny, ny+1 <- ny-2, ny-3; the same for columns), so the next step reads the
// mirror extension without any index reflection.
__device__ __forceinline__ void store_cols(float* __restrict__ row, int x, int nx, u64 v) {
  const float lo = plo(v), hi = phi(v);
  if (x + 1 < nx) {
    *reinterpret_cast<u64*>(row + x) = v;
  } else {
    row[x] = lo;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int xc = x + h;
    const float val = h ? hi : lo;
    if (xc >= nx) break;
    if (xc == 1 || xc == 2) row[-xc] = val;
    if (xc == nx - 2 || xc == nx - 3) row[2 * (nx - 1) - xc] = val;
  }
}

__device__ __forceinline__ void store_out(float* __restrict__ base0, int64_t pitch, int y, int ny,
                                          int x, int nx, u64 v) {
  store_cols(base0 + (int64_t)y * pitch, x, nx, v);
  if (y == 1 || y == 2) store_cols(base0 - (int64_t)y * pitch, x, nx, v);
  if ((y == ny - 2 || y == ny - 3) && y >= 0)
    store_cols(base0 + (int64_t)(2 * (ny - 1) - y) * pitch, x, nx, v);
}

}  // namespace sweep
}  // namespace pf
