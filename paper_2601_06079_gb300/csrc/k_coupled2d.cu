// Coupled Allen-Cahn / Cahn-Hilliard explicit step on a 2-D mesh (JAX-PF
// Eq. 7 with the phase free energies and interpolation of Supp. 3; the
// conserved composition c in the split form of Eq. 9-10, the order parameter
// eta by Eq. 1; lumped-mass explicit Euler of Eq. 12):
//   f(c, eta) = f_a(c) (1 - h(eta)) + f_b(c) h(eta) + kappa/2 |grad eta|^2
//   mu  = m^-1 sum_q w N_i [f_a'(c) (1 - h) + f_b'(c) h]          (no c gradient term)
//   c'  = c - dt M_c m^-1 K mu
//   eta' = eta - dt M_eta m^-1 (sum_q w N_i (f_b(c) - f_a(c)) h'(eta) + kappa K eta)
//
// A warp sweeps a band of rows down a strip of 64 columns (60 written, a pair
// per lane), both fields in a sliding register window, as k_explicit2d does for
// one field (sweep2d.h: values at Gauss points without their factor g_hi^2, in
// packed FP32); mu never leaves the registers, and neighbouring columns come by
// shuffles.  What binds it is the FP32 pipe: 111 packed and 16 scalar operations
// per row of 64 columns, 84 of them the polynomials at the four points:
//   f_a' (cubic), f_b' - f_a' (cubic), f_b - f_a (quartic) by Horner's rule in
//   c, h = eta^3 (10 - 15 eta + 6 eta^2), h' = 30 (eta - eta^2)^2,
// all expanded on the host in FP64 with the interpolation's factors, h' with
// the weights and -dt M_eta.  Rows that only fill the window leave out what
// later rows do not need (eta's terms above and below the band).
// The working planes carry a mirror frame like k_explicit2d's.
//
// Measured at 2048^2 (us per step, graph replay): 49.3 with 32 x 16 node tiles
// in shared memory, an element pass into corner arrays and gathers from them,
// bound by index arithmetic and shared-memory addressing; 28.0 so, the FMA pipe
// 70 % busy while SMs work (94 registers, 20 warps per SM; held to 80 or 72
// registers the kernel spills: 31 to 34).
#include <string.h>

#include "pf_internal.h"
#include "sweep2d.h"

namespace pf {
namespace {

using namespace sweep;

constexpr int kWarps = 2;   // warps per block, stacked in y
constexpr int kAhead = 3;   // rows of both planes in flight, and the loop's unrolling

struct Window {
  u64 c1, c2, e1, e2, x1, x2;    // rows k-1, k-2; row helpers of eta
  u64 amc, apc, ame, ape;        // x-interpolants of row k-1
  u64 tlc, thc, tle, the;        // element row k-2: its share of node row k-1
  u64 mua, mub, mxa, mxb;        // mu of rows k-3, k-2 and helpers
};

// Packed constants (pack_coupled2d)
struct Coef {
  const u64* c;
  __device__ __forceinline__ u64 rho() const { return c[0]; }
  __device__ __forceinline__ u64 g2() const { return c[1]; }            // -g_hi^2
  __device__ __forceinline__ u64 p(int i) const { return c[2 + i]; }    // f_a'
  __device__ __forceinline__ u64 q(int i) const { return c[6 + i]; }    // f_b' - f_a'
  __device__ __forceinline__ u64 r(int i) const { return c[10 + i]; }   // f_b - f_a
  __device__ __forceinline__ u64 h(int i) const { return c[15 + i]; }   // h / eta^3
  __device__ __forceinline__ u64 k(int stage, int i) const { return c[18 + 6 * stage + i]; }
};

// How far a row goes: its interpolation; c's element row; node row k-1 of c
// and eta's element row; eta's finished row k-1; c's finished row k-2; and
// past eta's band, c alone.
enum Stage { kStart, kElementC, kNodeC, kFirst, kBoth, kOnlyC };

// f_a' + (f_b' - f_a') h, and (f_b - f_a) h' up to constant factors, at one
// Gauss point of both columns
template <bool kEta>
__device__ __forceinline__ void point(u64 d, u64 n, const Coef& K, u64& gc, u64& ge) {
  const u64 n2 = mul2(n, n);
  const u64 h = mul2(mul2(n2, n), fma2(fma2(K.h(2), n, K.h(1)), n, K.h(0)));
  const u64 q = fma2(fma2(fma2(K.q(3), d, K.q(2)), d, K.q(1)), d, K.q(0));
  const u64 p = fma2(fma2(fma2(K.p(3), d, K.p(2)), d, K.p(1)), d, K.p(0));
  gc = fma2(q, h, p);
  if constexpr (kEta) {
    const u64 r = fma2(fma2(fma2(fma2(K.r(4), d, K.r(3)), d, K.r(2)), d, K.r(1)), d, K.r(0));
    const u64 w = fma2(K.g2(), n2, n);  // eta (1 - eta), without one factor
    ge = mul2(r, mul2(w, w));
  }
}

// x-interpolants of a row (scalar FMAs, see sweep2d.h)
__device__ __forceinline__ void interpolate(u64 P, float right, float rho, u64& am, u64& ap) {
  const float v0 = plo(P), v1 = phi(P);
  am = pk(fmaf(rho, v1, v0), fmaf(rho, right, v1));
  ap = pk(fmaf(rho, v0, v1), fmaf(rho, v1, right));
}

// weights back in x: the share of the left neighbour comes from its lane
__device__ __forceinline__ u64 back(u64 sl, u64 sh, const Coef& K) {
  const u64 A = fma2(K.rho(), sh, sl), B = fma2(K.rho(), sl, sh);
  const float bl = __shfl_up_sync(kFull, phi(B), 1);
  return pk(plo(A) + bl, phi(A) + plo(B));
}

template <bool kIso>
__device__ __forceinline__ u64 helper(u64 v, float r) {  // r: the column right of the lane's
  const float l = __shfl_up_sync(kFull, phi(v), 1);
  const u64 hs = pk(l + phi(v), plo(v) + r);
  return kIso ? add2(v, hs) : hs;
}

// init + K v at the centre row
template <bool kIso>
__device__ __forceinline__ u64 apply(u64 init, u64 s, u64 c, u64 n, u64 as, u64 ac, u64 an,
                                     const Coef& K, int st) {
  if constexpr (kIso) return fma2(K.k(st, 1), add2(add2(as, an), ac), fma2(K.k(st, 0), c, init));
  return fma2(K.k(st, 5), add2(as, an),
              fma2(K.k(st, 4), add2(s, n), fma2(K.k(st, 3), ac, fma2(K.k(st, 2), c, init))));
}

// Consumes row k: c and eta in C and E.  oe: eta's finished row k-1 (from
// kFirst on, not kOnlyC); oc: c's finished row k-2 (kBoth, kOnlyC).
template <bool kIso, int kStage>
__device__ __forceinline__ void row(u64 C, u64 E, Window& w, const Coef& K, u64& oc, u64& oe) {
  constexpr bool kEta = kStage >= kNodeC && kStage <= kBoth;   // eta's element row
  constexpr bool kEtaOut = kStage == kFirst || kStage == kBoth;
  const float rho = plo(K.rho());
  u64 amc, apc, ame, ape;
  interpolate(C, __shfl_down_sync(kFull, plo(C), 1), rho, amc, apc);
  const float er = __shfl_down_sync(kFull, plo(E), 1);
  interpolate(E, er, rho, ame, ape);
  u64 xe = 0;
  if constexpr (kStage != kOnlyC) xe = helper<kIso>(E, er);
  if constexpr (kStage >= kElementC) {
    u64 gc[4], ge[4];  // (low x, low y), (low, high), (high, low), (high, high)
    point<kEta>(fma2(K.rho(), amc, w.amc), fma2(K.rho(), ame, w.ame), K, gc[0], ge[0]);
    point<kEta>(fma2(K.rho(), w.amc, amc), fma2(K.rho(), w.ame, ame), K, gc[1], ge[1]);
    point<kEta>(fma2(K.rho(), apc, w.apc), fma2(K.rho(), ape, w.ape), K, gc[2], ge[2]);
    point<kEta>(fma2(K.rho(), w.apc, apc), fma2(K.rho(), w.ape, ape), K, gc[3], ge[3]);
    if constexpr (kStage >= kNodeC) {
      const u64 sl = add2(fma2(K.rho(), gc[1], gc[0]), w.tlc);
      const u64 sh = add2(fma2(K.rho(), gc[3], gc[2]), w.thc);
      const u64 mu = back(sl, sh, K);
      const u64 mx = helper<kIso>(mu, __shfl_down_sync(kFull, plo(mu), 1));
      if constexpr (kStage >= kBoth)
        oc = apply<kIso>(w.c2, w.mua, w.mub, mu, w.mxa, w.mxb, mx, K, 1);
      w.mua = w.mub;
      w.mxa = w.mxb;
      w.mub = mu;
      w.mxb = mx;
    }
    if constexpr (kEtaOut) {
      const u64 sl = add2(fma2(K.rho(), ge[1], ge[0]), w.tle);
      const u64 sh = add2(fma2(K.rho(), ge[3], ge[2]), w.the);
      const u64 F = back(sl, sh, K);
      oe = apply<kIso>(add2(w.e1, F), w.e2, w.e1, E, w.x2, w.x1, xe, K, 0);
    }
    w.tlc = fma2(K.rho(), gc[0], gc[1]);
    w.thc = fma2(K.rho(), gc[2], gc[3]);
    if constexpr (kEta) {
      w.tle = fma2(K.rho(), ge[0], ge[1]);
      w.the = fma2(K.rho(), ge[2], ge[3]);
    }
  }
  w.c2 = w.c1;
  w.c1 = C;
  w.e2 = w.e1;
  w.e1 = E;
  w.x2 = w.x1;
  w.x1 = xe;
  w.amc = amc;
  w.apc = apc;
  w.ame = ame;
  w.ape = ape;
}

// kTY: output rows per band, 1 + a multiple of kAhead
template <bool kIso, int kTY>
__global__ void __launch_bounds__(kWarps * 32) k_coupled2d(const Coupled2DArgs a) {
  static_assert((kTY - 1) % kAhead == 0, "the loop takes kAhead rows at a time");
  const int lane = threadIdx.x & 31;
  const int y0 = (block_row() * kWarps + (threadIdx.x >> 5)) * kTY;
  const int nx = a.nx, ny = a.ny;
  // launched as dependent (launch_coupled2d): the step before this one is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (y0 >= ny) return;
  const Coef K{a.pair};
  const int64_t pitch = a.pitch, plane = a.plane;
  const int x = blockIdx.x * kOutCols - kPair + kPair * lane;  // real column of the low half
  const bool writer = lane >= 1 && lane <= 30 && x < nx;
  const bool plain = writer && x > 2 && x + 1 < nx - 3 && y0 > 2 && y0 + kTY + 3 < ny;
  const float* src = a.in + (int64_t)(y0 - 2 + kGhost) * pitch + kGhost + x;
  float* const out0 = a.out + kGhost * pitch + kGhost;
  u64 nc[kAhead], ne[kAhead];  // rows in flight
  const auto load = [&](int j) {
    nc[j] = __ldg(reinterpret_cast<const u64*>(src));
    ne[j] = __ldg(reinterpret_cast<const u64*>(src + plane));
    src += pitch;
  };
#pragma unroll
  for (int j = 0; j < kAhead; ++j) load(j);
  Window w;
  u64 oc, oe;
  const auto consume = [&](auto stage, int j) {  // j: rows consumed before, modulo kAhead
    const u64 C = nc[j], E = ne[j];
    load(j);  // past the band's last row: not used
    row<kIso, decltype(stage)::value>(C, E, w, K, oc, oe);
  };
  const auto store = [&](float* p, int y, u64 v) {
    if (plain)
      *reinterpret_cast<u64*>(p + (int64_t)y * pitch + x) = v;
    else if (writer && y < ny)
      store_out(p, pitch, y, ny, x, nx, v);
  };
  consume(std::integral_constant<int, kStart>{}, 0);
  consume(std::integral_constant<int, kElementC>{}, 1);
  consume(std::integral_constant<int, kNodeC>{}, 2);
  consume(std::integral_constant<int, kFirst>{}, 0);
  store(out0 + plane, y0, oe);
#pragma unroll 1
  for (int i = 1; i < kTY; i += kAhead) {
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      consume(std::integral_constant<int, kBoth>{}, (1 + j) % kAhead);
      store(out0, y0 + i + j - 1, oc);
      store(out0 + plane, y0 + i + j, oe);
    }
  }
  // the next step may launch; were it let go at this one's start, its waiting
  // blocks would pile up on a part of the SMs (512^2: 7.2 us a step, so 4.3)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  consume(std::integral_constant<int, kOnlyC>{}, 1);
  store(out0, y0 + kTY - 1, oc);
}

}  // namespace

void pack_coupled2d(const CoupledPoly& f, double neg_dt_meta, Coupled2DArgs& a) {
  auto two = [](double v) {
    const float x = (float)v;
    unsigned int b;
    memcpy(&b, &x, 4);
    return (unsigned long long)b | ((unsigned long long)b << 32);
  };
  // a value at a Gauss point is g2 times the one carried, and so is the weight
  // back; the Gauss weight is |cell|/4 over the interior mass |cell|
  const double g2 = kGRho * kGRho, wt = 0.25 * g2;
  double s = 1.0;
  a.pair[0] = two(kRho);
  a.pair[1] = two(-g2);
  for (int i = 0; i < 5; ++i, s *= g2) {
    const double dfa = i < 4 ? (i + 1) * f.fa[i + 1] : 0.0;
    const double dfb = i < 2 ? (i + 1) * f.fb[i + 1] : 0.0;
    const double fb = i < 3 ? f.fb[i] : 0.0;
    if (i < 4) a.pair[2 + i] = two(wt * s * dfa);
    if (i < 4) a.pair[6 + i] = two(wt * s * (dfb - dfa));
    // h' = 30 (eta - eta^2)^2, eta - eta^2 carried without one factor g2
    a.pair[10 + i] = two(neg_dt_meta * 30.0 * g2 * g2 * wt * s * (fb - f.fa[i]));
  }
  const double h[3] = {10.0, -15.0, 6.0};
  s = g2 * g2 * g2;
  for (int i = 0; i < 3; ++i, s *= g2) a.pair[15 + i] = two(h[i] * s);
  const Stencil2D* st[2] = {&a.k1, &a.k2};
  for (int k = 0; k < 2; ++k) {
    const double v[6] = {(double)st[k]->c0 - st[k]->cd, st[k]->cd, st[k]->c0,
                         st[k]->cx, st[k]->cy, st[k]->cd};
    for (int i = 0; i < 6; ++i) a.pair[18 + 6 * k + i] = two(v[i]);
  }
}

namespace {
template <bool kIso, int kTY>
cudaError_t launch(const Coupled2DArgs& a, bool dependent, cudaStream_t s) {
  const dim3 grid = row_grid((a.nx + kOutCols - 1) / kOutCols,
                             (a.ny + kWarps * kTY - 1) / (kWarps * kTY));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kWarps * 32);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_coupled2d<kIso, kTY>, a);
}
}  // namespace

// Bands of 4 rows while 7-row bands would not fill the SMs twice (20 warps of
// them fit), 7 beyond: us per step at 64^2 / 515 x 1031 / 1024^2 / 2048^2 with
// 4 rows 3.8 / 6.9 / 10.4 / 30.6, with 7 rows 5.7 / 8.3 / 11.2 / 28.0, with 13
// rows 9.0 / 11.1 / 12.7 / 28.6.
//
// dependent: for steps launched one by one, whose launch then overlaps the end
// of the step before.  20 steps, us, without / with (node tiles): 64^2 140 / 80
// (125), 64 x 1500 144 / 85 (145), 512^2 140 / 102 (187), 1024^2 270 / 221 (352).
// Steps in a graph, which launches them close behind one another, are not.
cudaError_t launch_coupled2d(const Coupled2DArgs& a, bool dependent, cudaStream_t s) {
  const auto iso = [](const Stencil2D& k) { return k.cx == k.cd && k.cy == k.cd; };
  const bool both = iso(a.k1) && iso(a.k2);
  const int64_t warps = (int64_t)((a.nx + kOutCols - 1) / kOutCols) * ((a.ny + 6) / 7);
  if (warps < 40 * (int64_t)device_sm_count())
    return both ? launch<true, 4>(a, dependent, s) : launch<false, 4>(a, dependent, s);
  return both ? launch<true, 7>(a, dependent, s) : launch<false, 7>(a, dependent, s);
}

}  // namespace pf
