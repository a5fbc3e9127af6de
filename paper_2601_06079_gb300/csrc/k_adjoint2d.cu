// 2-D Cahn-Hilliard with a per-node mobility field: the explicit step and the
// discrete adjoint of that step (JAX-PF Eq. 9-12; sensitivities in the sense
// of Supp. 2, taken through the discrete explicit map).
//
// Forward map (lumped mass m, shifted state d = c - s):
//   mu = m^-1 (F(c) + kappa K c),  c' = c - dt m^-1 K_M mu,
//   (K_M u)_i = sum_e sum_q w|J| M_q grad u_q . grad N_i,  M_q = M sum_a N_a(q) m_a.
// Reverse step for y = m^-1 lambda (lambda = dLoss/dc'):
//   w = m^-1 K_M y,  y_prev = y - dt m^-1 (F'(c) + kappa K) w,
//   dLoss/dM     += -dt / M  sum_i m_i w_i mu_i
//   dLoss/dkappa += -dt sum_i m_i w_i (m^-1 K c)_i
//   dLoss/dW     += -dt / W sum_i m_i w_i (m^-1 F(c))_i
//   dLoss/dm_a   += -dt M sum_e sum_q w|J| N_a(q) grad mu_q . grad y_q
// (F', K, K_M symmetric).  Mirror images beyond the mesh reproduce the
// zero-flux operators divided by the lumped mass; sums that need the real
// (unmirrored) value at a boundary node take the mirrored value times the
// node's mass fraction.  No atomics.
//
// A warp sweeps a band of rows down a strip of 64 columns, a pair per lane, in
// packed FP32 (sweep2d.h: values at Gauss points without their factor g_hi per
// direction).  The planes are plain arrays; images come from reflected load
// addresses.  The mobility's bilinear weights factorise: a flux along x at a y
// Gauss point needs only the sum of M over the two x points, which is the sum
// of M at the two nodes, interpolated in y, and the same the other way round:
//   S(y) = (d u)(y) (m(x) + m(x+1))(y),  K_M u = c_x [S(x-1) - S(x)] + ...,
// 2 products per direction and element instead of 4 points' gradients; so does
// the mobility's gradient (products of differences, projected along one axis).
//
// Constants.  dLoss/dM = (kappa dLoss/dkappa + W dLoss/dW) / M changes sign in
// the course of a trajectory; near there it keeps 1e-8 only if the two parts do,
// and a factor rounded once to FP32 (6e-8) costs each of them more.  So (see
// pack_ch_mob):
//   - g_hi is 1 / (1 + rho) for the rounded rho: interpolated constants stay exact;
//   - the polynomials keep their coefficients, the stiffness stencil is divided by
//     its corner weight (8 and -1 on square cells), and the factors in front of
//     them meet at the node: r = kappa K : F, the fluxes' and the time step's, each
//     an FP32 pair hi + lo that meets an unrounded product;
//   - dLoss/dM's sum is not taken: it follows from the other two.
// dLoss/dM's error against FP64 over 60 meshes of 41 x 70 to 488 x 168 nodes and
// 100 to 1,000 steps, as a share of (|kappa dLoss/dkappa| + |W dLoss/dW|) / M:
// median 5.0e-9, largest 2.7e-8 (the rounding of the states); with g_hi of its own
// and every factor rounded once 3.2e-8 and 1.2e-7; with node tiles, differences and
// dt as the one rounded factor that mattered 1.1e-8 and 3.3e-8.  The pairs cost the
// forward step 1 to 2 % (1,024 steps of 512^2 2,994 and 3,061 us); with the warp's
// running sums asked for at the start and added before the last row, 1,000 steps
// and their reverse take 12.1 ms without them and 12.4 with, on 300 x 400 10.5 and
// 10.1.
//
// Measured at 512^2 (us per step, graph replay): forward 5.7 with 32 x 16 node
// tiles in shared memory (element passes into corner arrays, four barriers), 2.9
// so; reverse 13.6, 7.1 so.  Both are latency-bound there (8 warps per SM); the
// reverse sweep holds 166 registers.
#include "pf_internal.h"
#include "sweep2d.h"

namespace pf {
namespace {

using namespace sweep;

constexpr int kThreads = 256;
constexpr int kWarps = 2;  // warps per block of the sweeps, stacked in y
// Output rows per band, forward and reverse.  Reverse at 100 x 80 / 512^2 /
// 1024^2, us per step: 4 rows 5.9 / 7.1 / 17.1, 2 rows 4.3 / 8.8 / 21.0, 6 rows
// 7.5 / 9.3 / 17.2 (a lone warp's row takes 0.5 us, so short bands suit the
// meshes this calibration runs on); 2 rows in flight 7.5 at 512^2.
constexpr int kTYFwd = 4;
constexpr int kTYRev = 4;
constexpr int kAhead = 3;  // rows in flight

__device__ __forceinline__ u64 bc(float v) { return pk(v, v); }
__device__ __forceinline__ u64 sub2(u64 a, u64 b) { return fma2(b, bc(-1.0f), a); }
__device__ __forceinline__ float from_left(float v) { return __shfl_up_sync(kFull, v, 1); }
__device__ __forceinline__ float from_right(float v) { return __shfl_down_sync(kFull, v, 1); }

// single reflection about the end nodes, then clamped: exact for the stored
// nodes' two-node halo
__device__ __forceinline__ int reflect(int k, int n) {
  k = k < 0 ? -k : k;
  k = k >= n ? 2 * (n - 1) - k : k;
  return k < 0 ? 0 : (k >= n ? n - 1 : k);
}

// a row of one plane in a lane: its two columns and the one right of them
struct Row {
  u64 v;
  float r;
  __device__ __forceinline__ u64 next() const { return pk(phi(v), r); }  // columns x+1, x+2
};
__device__ __forceinline__ Row row_of(u64 v) { return Row{v, from_right(plo(v))}; }

// interpolants along x at the two Gauss points (scalar FMAs, see sweep2d.h)
__device__ __forceinline__ void along_x(const Row& a, float rho, u64& lo, u64& hi) {
  const float v0 = plo(a.v), v1 = phi(a.v);
  lo = pk(fmaf(rho, v1, v0), fmaf(rho, a.r, v1));
  hi = pk(fmaf(rho, v0, v1), fmaf(rho, v1, a.r));
}
// shares of node columns from values at the two x Gauss points
__device__ __forceinline__ u64 back_x(u64 lo, u64 hi, u64 rho) {
  const u64 A = fma2(rho, hi, lo), B = fma2(rho, lo, hi);
  const float bl = from_left(phi(B));
  return pk(plo(A) + bl, phi(A) + plo(B));
}
// west + east neighbours
__device__ __forceinline__ u64 beside(const Row& a) {
  const float l = from_left(phi(a.v));
  return pk(l + phi(a.v), plo(a.v) + a.r);
}

// 9-point stencil from three rows and their west + east sums
struct Stencil {
  u64 c0, cx, cy, cd;
  __device__ __forceinline__ explicit Stencil(const Stencil2D& k)
      : c0(bc(k.c0)), cx(bc(k.cx)), cy(bc(k.cy)), cd(bc(k.cd)) {}
  __device__ __forceinline__ u64 operator()(u64 s, u64 c, u64 n, u64 ws, u64 wc, u64 wn) const {
    return fma2(cd, add2(ws, wn), fma2(cy, add2(s, n), fma2(cx, wc, mul2(c0, c))));
  }
};

// F and K c, row by row, without their factors (ChMobArgs)
struct Potential {
  u64 c1, c2, w1, w2, am, ap, tl, th;  // rows k-1, k-2 of c; their west + east sums
  u64 g[4];                            // Gauss values of the last element row
  __device__ __forceinline__ void start(const Row& c, float rho) {
    c2 = c1;
    w2 = w1;
    c1 = c.v;
    w1 = beside(c);
    along_x(c, rho, am, ap);
  }
  // row k; kNode: F and K c of row k-1
  template <bool kNode>
  __device__ __forceinline__ void take(const Row& c, const ChMobArgs& a, u64 rho, u64& F, u64& Kc) {
    u64 bm, bp;
    along_x(c, plo(rho), bm, bp);
    const u64 wc = beside(c);
    g[0] = fma2(rho, bm, am);
    g[1] = fma2(rho, am, bm);
    g[2] = fma2(rho, bp, ap);
    g[3] = fma2(rho, ap, bp);
    const u64 p0 = bc(a.q[0]), p1 = bc(a.q[1]), p2 = bc(a.q[2]), p3 = bc(a.q[3]);
    u64 f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = fma2(fma2(fma2(p3, g[i], p2), g[i], p1), g[i], p0);
    if constexpr (kNode) {
      F = back_x(add2(fma2(rho, f[1], f[0]), tl), add2(fma2(rho, f[3], f[2]), th), rho);
      Kc = Stencil(a.k)(c2, c1, c.v, w2, w1, wc);
    }
    tl = fma2(rho, f[0], f[1]);
    th = fma2(rho, f[2], f[3]);
    am = bm;
    ap = bp;
    c2 = c1;
    w2 = w1;
    c1 = c.v;
    w1 = wc;
  }
};

// Differences of u along x (per row) and y (per element row) at the Gauss
// points of the other direction
struct Diff {
  Row u;   // row k-1
  u64 dx;  // its differences along x
  __device__ __forceinline__ void start(const Row& r) {
    u = r;
    dx = sub2(r.next(), r.v);
  }
  // row k: x-differences at the element row's two y points, y-differences at
  // its two x points
  __device__ __forceinline__ void take(const Row& r, u64 rho, u64 (&x)[2], u64 (&y)[2]) {
    const u64 d = sub2(r.next(), r.v);
    x[0] = fma2(rho, d, dx);
    x[1] = fma2(rho, dx, d);
    along_x(Row{sub2(r.v, u.v), r.r - u.r}, plo(rho), y[0], y[1]);
    u = r;
    dx = d;
  }
};

// The element row's mobility factors: x sums at the two y points, y sums at the
// two x points
struct Mobility {
  Row m;
  u64 sx;
  __device__ __forceinline__ void start(const Row& r) {
    m = r;
    sx = add2(r.v, r.next());
  }
  __device__ __forceinline__ void take(const Row& r, u64 rho, u64 (&x)[2], u64 (&y)[2]) {
    const u64 s = add2(r.v, r.next());
    x[0] = fma2(rho, s, sx);
    x[1] = fma2(rho, sx, s);
    along_x(Row{add2(r.v, m.v), r.r + m.r}, plo(rho), y[0], y[1]);
    m = r;
    sx = s;
  }
};

// m^-1 K_M u without its factors: the shares of node row k-1 from the fluxes
// along x (ox) and y (oy) of the element rows above and below
struct Flux {
  u64 X, Y;  // carried from the element row above
  template <bool kNode>
  __device__ __forceinline__ void take(const u64 (&dx)[2], const u64 (&dy)[2], const u64 (&mx)[2],
                                       const u64 (&my)[2], u64 rho, u64& ox, u64& oy) {
    const u64 f0 = mul2(dx[0], mx[0]), f1 = mul2(dx[1], mx[1]);
    const u64 T = back_x(mul2(dy[0], my[0]), mul2(dy[1], my[1]), rho);
    if constexpr (kNode) {
      const u64 S = add2(fma2(rho, f1, f0), X);
      const u64 W = pk(from_left(phi(S)), plo(S));  // the element left of each column
      ox = sub2(W, S);
      oy = sub2(Y, T);
    }
    X = fma2(rho, f0, f1);
    Y = T;
  }
};

struct Lane {
  int x, xa, xb;  // first column, load columns of the pair
  bool writer;
  __device__ __forceinline__ explicit Lane(int nx) {
    const int lane = threadIdx.x & 31;
    x = blockIdx.x * kOutCols - kPair + kPair * lane;
    xa = reflect(x, nx);
    xb = reflect(x + 1, nx);
    writer = lane >= 1 && lane <= 30 && x < nx;
  }
  __device__ __forceinline__ u64 load(const float* __restrict__ plane, int64_t row) const {
    return pk(__ldg(plane + row + xa), __ldg(plane + row + xb));
  }
  // 64-bit where the pair is whole and aligned
  __device__ __forceinline__ void store(float* row, int nx, u64 v) const {
    if (x + 1 < nx && (reinterpret_cast<uintptr_t>(row + x) & 7) == 0) {
      *reinterpret_cast<u64*>(row + x) = v;
    } else {
      row[x] = plo(v);
      if (x + 1 < nx) row[x + 1] = phi(v);
    }
  }
};

// u times a factor hi + lo: the low part meets the unrounded product (added to a
// rounded sum it would be lost)
__device__ __forceinline__ u64 times(const float (&f)[2], u64 u) {
  return fma2(bc(f[0]), u, mul2(bc(f[1]), u));
}

// the sum of two such products, the low parts first
__device__ __forceinline__ u64 times(const float (&f)[2], u64 u, const float (&g)[2], u64 v) {
  return fma2(bc(g[0]), v, fma2(bc(f[0]), u, fma2(bc(g[1]), v, mul2(bc(f[1]), u))));
}

__global__ void __launch_bounds__(kWarps * 32) k_ch_mob_step(const ChMobArgs a, float* out) {
  const int nx = a.nx, ny = a.ny;
  const int y0 = (block_row() * kWarps + (threadIdx.x >> 5)) * kTYFwd;
  if (y0 >= ny) return;
  const Lane L(nx);
  const u64 rho = bc(kRho);
  u64 nc[kAhead], nm[kAhead];
  const auto load = [&](int j, int k) {  // row y0 - 2 + k into slot j
    const int64_t row = (int64_t)reflect(y0 - 2 + k, ny) * nx;
    nc[j] = L.load(a.d, row);
    nm[j] = L.load(a.mfield, row);
  };
#pragma unroll
  for (int j = 0; j < kAhead; ++j) load(j, j);
  Potential pot;
  Mobility mob;
  Diff dif;
  Flux flux;
  Row c, m = {0, 0.0f}, m1 = {0, 0.0f};  // rows k; m also of row k-1
  u64 F, Kc, cc[3];
  // the potential and the mobility run one element row apart: mu of row k-1 is
  // known at row k, so its differences and the mobility's rows are k-2 and k-1
  const auto next = [&](int k) {
    m1 = m;
    c = row_of(nc[k % kAhead]);
    m = row_of(nm[k % kAhead]);
    load(k % kAhead, k + kAhead);
    cc[k % 3] = c.v;
  };
  u64 dx[2], dy[2], mx[2], my[2], ox, oy;
  next(0);
  pot.start(c, plo(rho));
  next(1);
  pot.take<false>(c, a, rho, F, Kc);
  next(2);
  pot.take<true>(c, a, rho, F, Kc);  // mu of row y0 - 1
  dif.start(row_of(add2(F, times(a.r, Kc))));
  mob.start(m1);
#pragma unroll
  for (int k = 3; k < kTYFwd + 4; ++k) {
    next(k);
    pot.take<true>(c, a, rho, F, Kc);  // mu of row y0 - 3 + k
    dif.take(row_of(add2(F, times(a.r, Kc))), rho, dx, dy);
    mob.take(m1, rho, mx, my);
    if (k == 3) {
      flux.take<false>(dx, dy, mx, my, rho, ox, oy);
    } else {
      flux.take<true>(dx, dy, mx, my, rho, ox, oy);
      const int y = y0 + k - 4;
      if (L.writer && y < ny) L.store(out + (int64_t)y * nx, nx, add2(cc[(k - 2) % 3], times(a.fx, ox, a.fy, oy)));
    }
  }
}

// hi + lo, a sum with the rounding errors of its additions in lo (Knuth's two-sum)
struct Pair {
  float hi, lo;
  __device__ __forceinline__ void add(float x) {
    const float t = hi + x, bp = t - hi;
    lo += (hi - (t - bp)) + (x - bp);
    hi = t;
  }
};
__device__ __forceinline__ Pair runs(const u64 (&d)[2]) {
  Pair p{plo(d[0]), 0.0f};
  p.add(phi(d[0]));
  p.add(plo(d[1]));
  p.add(phi(d[1]));
  return p;
}

// The reverse step.  acc: per warp two compensated FP32 pairs (hi, lo) of the
// sums for kappa and W over all steps, the factors left to the end.  Two rows'
// products of a column are one FP32 run; runs, lanes and steps add up as pairs.
__global__ void __launch_bounds__(kWarps * 32)
    k_ch_adj_step(const ChMobArgs a, const float* yin, float* yout, float* grad_hi, float* grad_lo,
                  float2* acc) {
  const int nx = a.nx, ny = a.ny;
  const int band = block_row() * kWarps + (threadIdx.x >> 5);
  const int y0 = band * kTYRev;
  if (y0 >= ny) return;
  const Lane L(nx);
  const u64 rho = bc(kRho), gX = bc(a.gX), gY = bc(a.gY);
  const u64 s0 = bc(a.h[0]), s1 = bc(a.h[1]), s2 = bc(a.h[2]);
  // the warp's two pairs so far, asked for before they are needed
  float4* const pairs = reinterpret_cast<float4*>(acc) + ((int64_t)band * gridDim.x + blockIdx.x);
  const float4 kept = (threadIdx.x & 31) == 0 ? *pairs : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  const Stencil K(a.k);
  u64 nc[kAhead], nm[kAhead], nyv[kAhead];
  const auto load = [&](int j, int k) {
    const int64_t row = (int64_t)reflect(y0 - 2 + k, ny) * nx;
    nc[j] = L.load(a.d, row);
    nm[j] = L.load(a.mfield, row);
    nyv[j] = L.load(yin, row);
  };
#pragma unroll
  for (int j = 0; j < kAhead; ++j) load(j, j);
  // mass fractions of this lane's columns; 0 in columns that it does not own
  const auto fx = [&](int x) { return x == 0 || x == nx - 1 ? 0.5f : 1.0f; };
  const float f0 = L.writer ? fx(L.x) : 0.0f;
  const float f1 = L.writer && L.x + 1 < nx ? fx(L.x + 1) : 0.0f;
  const u64 fxp = pk(f0, f1);

  Potential pot;
  Mobility mob;
  Diff dy_, dmu;  // differences of y (rows k-1, k) and mu (rows k-2, k-1)
  Flux flux;
  u64 w1 = 0, w2 = 0, v1 = 0, v2 = 0;  // w of rows k-2, k-3; west + east sums
  u64 wa = 0, wb = 0, hl = 0, hh = 0;  // x-interpolants of w; F' w's carry
  u64 gx = 0, gy = 0;                  // carries of the mobility gradient
  u64 px[2], py[2];                    // y's differences in element row (k-2, k-1)
  u64 dK[2] = {0, 0}, dW[2] = {0, 0};  // rows 0 and 1, rows 2 and 3 of the band
  Row c, m, y;
  u64 yy[3], F, Kc, gq[4];
  const auto next = [&](int k) {
    c = row_of(nc[k % kAhead]);
    m = row_of(nm[k % kAhead]);
    y = row_of(nyv[k % kAhead]);
    load(k % kAhead, k + kAhead);
    yy[k % 3] = y.v;
  };
  u64 ex[2], ey[2], mx[2], my[2], ox, oy;
  next(0);
  pot.start(c, plo(rho));
  dy_.start(y);
  mob.start(m);
  next(1);
  pot.take<false>(c, a, rho, F, Kc);
  dy_.take(y, rho, ex, ey);
  mob.take(m, rho, mx, my);
  flux.take<false>(ex, ey, mx, my, rho, ox, oy);
#pragma unroll
  for (int k = 2; k < kTYRev + 4; ++k) {
    // row k is y0 - 2 + k: mu and w of the row before it
    next(k);
#pragma unroll
    for (int i = 0; i < 4; ++i) gq[i] = pot.g[i];  // c in element row (k-2, k-1)
    px[0] = ex[0];
    px[1] = ex[1];
    py[0] = ey[0];
    py[1] = ey[1];
    pot.take<true>(c, a, rho, F, Kc);
    dy_.take(y, rho, ex, ey);
    mob.take(m, rho, mx, my);
    flux.take<true>(ex, ey, mx, my, rho, ox, oy);
    const u64 w = add2(ox, times(a.ay, oy));  // without cW
    const Row wr = row_of(w);
    const u64 mu = add2(F, times(a.r, Kc)), vw = beside(wr);
    const int yr = y0 - 3 + k;  // the row of mu and w
    if (k >= 3 && k < kTYRev + 3 && yr < ny) {
      const u64 fw = mul2(mul2(fxp, bc(yr == 0 || yr == ny - 1 ? 0.5f : 1.0f)), w);
      const int run = (k - 3) / 2;
      dK[run] = fma2(fw, Kc, dK[run]);
      dW[run] = fma2(fw, F, dW[run]);
    }
    u64 na, nb;
    along_x(wr, plo(rho), na, nb);
    if (k == 2) {
      dmu.start(row_of(mu));
    } else {
      // element row (k-2, k-1): F' w, and grad mu . grad y
      u64 ux[2], uy[2], h[4];
      dmu.take(row_of(mu), rho, ux, uy);
      h[0] = mul2(fma2(fma2(s2, gq[0], s1), gq[0], s0), fma2(rho, na, wa));
      h[1] = mul2(fma2(fma2(s2, gq[1], s1), gq[1], s0), fma2(rho, wa, na));
      h[2] = mul2(fma2(fma2(s2, gq[2], s1), gq[2], s0), fma2(rho, nb, wb));
      h[3] = mul2(fma2(fma2(s2, gq[3], s1), gq[3], s0), fma2(rho, wb, nb));
      const u64 q0 = mul2(ux[0], px[0]), q1 = mul2(ux[1], px[1]);
      const u64 T = back_x(mul2(uy[0], py[0]), mul2(uy[1], py[1]), rho);
      if (k >= 4) {
        const int yo = y0 + k - 4;  // the finished row
        const u64 H = back_x(add2(fma2(rho, h[1], h[0]), hl), add2(fma2(rho, h[3], h[2]), hh), rho);
        const u64 Hw = add2(H, times(a.r, K(w2, w1, w, v2, v1, vw)));
        const u64 S = add2(fma2(rho, q1, q0), gx);
        const u64 both = add2(S, pk(from_left(phi(S)), plo(S)));  // elements right and left
        const u64 G = fma2(gY, add2(gy, T), mul2(gX, both));
        if (L.writer && yo < ny) {
          const int64_t row = (int64_t)yo * nx;
          L.store(yout + row, nx, add2(yy[(k - 2) % 3], times(a.n, Hw)));
          if (grad_hi) {
            const u64 v = mul2(mul2(fxp, bc(yo == 0 || yo == ny - 1 ? 0.5f : 1.0f)), G);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (L.x + i < nx) {
                float* hp = grad_hi + row + L.x + i;
                const float s = i ? phi(v) : plo(v), hi = *hp, t = hi + s, bp = t - hi;
                grad_lo[row + L.x + i] += (hi - (t - bp)) + (s - bp);
                *hp = t;
              }
            }
          }
        }
      }
      hl = fma2(rho, h[0], h[1]);
      hh = fma2(rho, h[2], h[3]);
      gx = fma2(rho, q0, q1);
      gy = T;
    }
    w2 = w1;
    v2 = v1;
    w1 = w;
    v1 = vw;
    wa = na;
    wb = nb;
    if (k == kTYRev + 2) {
      // the warp's sums, into its pairs (FP64 only at the end: an FP64 instruction
      // takes an SM 16 cycles per warp), while the last row is still to do
      static_assert(kTYRev == 4, "two runs of two rows");
      Pair v[2] = {runs(dK), runs(dW)};
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float h = __shfl_down_sync(kFull, v[j].hi, o);
          v[j].lo += __shfl_down_sync(kFull, v[j].lo, o);
          v[j].add(h);
        }
      }
      v[0].lo += kept.y;
      v[0].add(kept.x);
      v[1].lo += kept.w;
      v[1].add(kept.z);
      if ((threadIdx.x & 31) == 0) *pairs = make_float4(v[0].hi, v[0].lo, v[1].hi, v[1].lo);
    }
  }
}

// The gradients of kappa, W and M from the warps' pairs (kappa, W) in acc, one block
__global__ void k_scalar_sums(const float2* __restrict__ acc, int n, ChMobScale sc,
                              double* __restrict__ out) {
  __shared__ double red[2][kThreads / 32];
  double v[2] = {0.0, 0.0};
  for (int i = threadIdx.x; i < n; i += kThreads)
    for (int j = 0; j < 2; ++j) v[j] += (double)acc[2 * (int64_t)i + j].x + (double)acc[2 * (int64_t)i + j].y;
  for (int j = 0; j < 2; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_down_sync(kFull, v[j], o);
    if ((threadIdx.x & 31) == 0) red[j][threadIdx.x >> 5] = v[j];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s[2] = {0.0, 0.0};
    for (int j = 0; j < 2; ++j)
      for (int w = 0; w < kThreads / 32; ++w) s[j] += red[j][w];
    out[0] = sc.kappa * s[0];
    out[1] = sc.W * s[1];
    out[2] = sc.M_kappa * s[0] + sc.M_W * s[1];
  }
}

// out = hi + lo in FP64 (the compensated FP32 pair of the mobility gradient)
__global__ void k_grad_to_double(const float* __restrict__ hi, const float* __restrict__ lo,
                                 double* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (double)hi[i] + (double)lo[i];
}

// loss = 1/2 sum_i wt_i (c_i - t_i)^2 ; y = wt_i (c_i - t_i) / m_i
// (wt = m for the mass-weighted misfit, 1 for the nodal one)
__global__ void k_loss(const float* __restrict__ d, float shift, const float* __restrict__ target,
                       int nx, int ny, double cell, int nodal, float* __restrict__ y,
                       double* __restrict__ partials) {
  __shared__ double red[kThreads / 32];
  const int64_t n = (int64_t)nx * ny;
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kThreads) {
    const int x = (int)(i % nx), yy = (int)(i / nx);
    const double m = cell * ((x == 0 || x == nx - 1) ? 0.5 : 1.0) *
                     ((yy == 0 || yy == ny - 1) ? 0.5 : 1.0);
    const double r = ((double)shift + (double)d[i]) - (double)target[i];
    const double wt = nodal ? 1.0 : m;
    acc += 0.5 * wt * r * r;
    y[i] = (float)(wt * r / m);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) s += red[w];
    partials[blockIdx.x] = s;
  }
}

// fixed-order sums: out[j] = sum_b in[b * stride + j] for j < k
__global__ void k_colsum(const double* __restrict__ in, int nb, int stride, int k,
                         double* __restrict__ out) {
  if (threadIdx.x < k) {
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += in[(int64_t)b * stride + threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// dLoss/dc0 = m_i y_i
__global__ void k_mass_scale(const float* __restrict__ y, int nx, int ny, double cell,
                             float* __restrict__ out) {
  const int64_t n = (int64_t)nx * ny;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % nx), yy = (int)(i / nx);
    const double m = cell * ((x == 0 || x == nx - 1) ? 0.5 : 1.0) *
                     ((yy == 0 || yy == ny - 1) ? 0.5 : 1.0);
    out[i] = (float)(m * (double)y[i]);
  }
}

__global__ void k_add(const float* __restrict__ in, float* __restrict__ out, int64_t n, float add) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = in[i] + add;
}

constexpr int kLossBlocks = 256;

}  // namespace

cudaError_t launch_add(const float* in, float* out, int64_t n, float add, cudaStream_t s) {
  int64_t b = (n + 255) / 256;
  k_add<<<(unsigned)(b < 1216 ? b : 1216), 256, 0, s>>>(in, out, n, add);
  return cudaGetLastError();
}

namespace {
int strips(int nx) { return (nx + kOutCols - 1) / kOutCols; }
dim3 sweep_grid(const ChMobArgs& a, int ty) {
  return row_grid(strips(a.nx), (a.ny + kWarps * ty - 1) / (kWarps * ty));
}
}  // namespace

int ch_mob_warps(int nx, int ny) { return strips(nx) * ((ny + kTYRev - 1) / kTYRev); }

void pack_ch_mob(const ChMobParams& p, ChMobArgs& a, ChMobScale& sc) {
  // a value at a Gauss point is g2 times the one carried, and so is the weight
  // back; the Gauss weight is |cell|/4 over the interior mass |cell|
  const double g = kGRho, g2 = g * g, cF = 0.25 * g2 * g2;
  double s = 1.0 / g2;
  for (int i = 0; i < 4; ++i, s *= g2) {
    a.q[i] = (float)(s * p.f1[i]);
    if (i < 3) a.h[i] = (float)(s * g2 * p.f2[i]);
  }
  const double rx = p.hy / p.hx, ry = p.hx / p.hy, cell = p.hx * p.hy;
  const double cK = (rx + ry) / (6.0 * cell);  // minus the corner weight of m^-1 K
  a.k.c0 = 8.0f;
  a.k.cx = (float)((-4.0 * rx + 2.0 * ry) / (rx + ry));
  a.k.cy = (float)((2.0 * rx - 4.0 * ry) / (rx + ry));
  a.k.cd = -1.0f;
  const auto pair = [](double v, float (&o)[2]) {
    o[0] = (float)v;
    o[1] = (float)(v - (double)o[0]);
  };
  // fluxes: a difference takes g, the other direction's mobility sum and the
  // weight back g each
  const double w = 0.25 * g * g2, ix2 = 1.0 / (p.hx * p.hx), iy2 = 1.0 / (p.hy * p.hy);
  const double cW = p.M * w * ix2;
  pair(p.kappa * cK / cF, a.r);
  pair(-p.dt * cF * cW, a.fx);
  pair(-p.dt * cF * p.M * w * iy2, a.fy);
  pair(iy2 / ix2, a.ay);
  pair(-p.dt * cF * cW, a.n);
  a.gX = (float)(-p.dt * cell * cF * p.M * w * ix2);
  a.gY = (float)(-p.dt * cell * cF * p.M * w * iy2);
  const double f = -p.dt * cell * cW;
  sc.kappa = f * cK;
  sc.W = f * cF / p.W;
  sc.M_kappa = f * cK * p.kappa / p.M;
  sc.M_W = f * cF / p.M;
}

cudaError_t launch_ch_mob_step(const ChMobArgs& a, float* out, cudaStream_t s) {
  k_ch_mob_step<<<sweep_grid(a, kTYFwd), kWarps * 32, 0, s>>>(a, out);
  return cudaGetLastError();
}

cudaError_t launch_ch_adj_step(const ChMobArgs& a, const float* yin, float* yout,
                               float* grad_hi, float* grad_lo, float2* acc, cudaStream_t s) {
  if ((grad_hi == nullptr) != (grad_lo == nullptr)) return cudaErrorInvalidValue;
  k_ch_adj_step<<<sweep_grid(a, kTYRev), kWarps * 32, 0, s>>>(a, yin, yout, grad_hi, grad_lo, acc);
  return cudaGetLastError();
}

cudaError_t launch_scalar_sums(const float2* acc, int n, const ChMobScale& sc, double* out,
                               cudaStream_t s) {
  k_scalar_sums<<<1, kThreads, 0, s>>>(acc, n, sc, out);
  return cudaGetLastError();
}

cudaError_t launch_grad_to_double(const float* hi, const float* lo, double* out, int64_t n,
                                  cudaStream_t s) {
  int64_t blocks = (n + kThreads - 1) / kThreads;
  if (blocks > 8 * (int64_t)device_sm_count()) blocks = 8 * (int64_t)device_sm_count();
  k_grad_to_double<<<(unsigned)blocks, kThreads, 0, s>>>(hi, lo, out, n);
  return cudaGetLastError();
}

cudaError_t launch_loss(const float* d, float shift, const float* target, int nx, int ny,
                        double cell, int nodal, float* y, double* partials, double* out,
                        cudaStream_t s) {
  k_loss<<<kLossBlocks, kThreads, 0, s>>>(d, shift, target, nx, ny, cell, nodal, y, partials);
  k_colsum<<<1, 32, 0, s>>>(partials, kLossBlocks, 1, 1, out);
  return cudaGetLastError();
}

cudaError_t launch_mass_scale(const float* y, int nx, int ny, double cell, float* out,
                              cudaStream_t s) {
  const int64_t n = (int64_t)nx * ny;
  int64_t b = (n + 255) / 256;
  k_mass_scale<<<(unsigned)(b < 1216 ? b : 1216), 256, 0, s>>>(y, nx, ny, cell, out);
  return cudaGetLastError();
}

}  // namespace pf
