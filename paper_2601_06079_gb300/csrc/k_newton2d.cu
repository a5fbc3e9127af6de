// Implicit 2-D steps (JAX-PF Eq. 13-14) of small and medium meshes in one
// cooperative launch: Newton, restarted GMRES with CGS2 and its Givens
// rotations, the same algorithm as the host-driven solver in pf_api.cu.
//
// Why: at 64^2 an Arnoldi step is five launches of a few us and a round trip
// to the host, 58 us in all, for 50 kB of vectors.  Here a block owns node
// tiles for the whole launch; what blocks exchange is the halo of the operator
// and the partial sums of the inner products, and an Arnoldi step is three
// phases that end in a reduction:
//   w = J v on the own tiles, products with the basis;
//   first update and second products;  second update and norm.
// A partial sum travels as a packet of two words under the phase's number
// (packet.h); every block polls all blocks' packets, so a reduction is one
// store and one load through L2, and a barrier where the writer fences first
// and the reader after (needed only before the operator reads a halo).  Every
// block sums the partials in the same order, so all take the same decisions, and thread 0 of each runs the (FP64) Givens
// rotations on its own copy of the Hessenberg matrix.  The basis stays as the
// updates left it; its vectors' scale factors 1/|v| are applied to products,
// updates and the operator's result (which is linear in v), so that no
// further pass and barrier normalise a vector.
// Sums: FP32 products, a compensated FP32 pair per thread and warp (an FP64
// instruction takes an SM 16 cycles per warp, and each of 16 warps would issue
// several per product), FP64 over the blocks.
#include <type_traits>

#include "implicit2d_op.h"
#include "packet.h"
#include "pf_internal.h"

namespace pf {
namespace {

using namespace implicit2d;

constexpr int kThreads = 512;  // one node of a 32 x 16 tile each
constexpr int kWarps = kThreads / 32;
constexpr int kD = 4;     // products whose reductions run together
constexpr int kPoll = 5;  // packets a lane polls together: 160 blocks in one round trip
static_assert(TX * TY == kThreads, "a thread owns one node of a tile");

struct Acc2 {  // Knuth's two-sum, see k_krylov.cu
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float s) {
    const float t = hi + s, bp = t - hi;
    lo += (hi - (t - bp)) + (s - bp);
    hi = t;
  }
};

struct Scalars {
  double H[kMaxBasis][kMaxBasis];  // H[k][j]: column k
  double cs[kMaxBasis], sn[kMaxBasis], gv[kMaxBasis + 1], y[kMaxBasis];
  double sums[kMaxBasis];          // the last reduction's results
  float2 part[kMaxBasis][kWarps];  // the warps' pairs (hi, lo)
  float scale[kMaxBasis];          // 1 / |v_j|
  float coef[kMaxBasis];
  double hk[kMaxBasis], rel;
  int stop, failed;
  unsigned mute;  // 0, or flips the tags of this block's packets (self-test)
};

// Ends a phase: k sums of sc.part over all blocks into sc.sums; a barrier for
// memory too if `ordered`.  Packets alternate between two buffers: a block
// writes phase p + 2 only after it has all of phase p + 1, which the others
// wrote after reading phase p.
__device__ __noinline__ bool end_phase(Scalars& sc, Packet* packets, unsigned tag, int k,
                                       bool ordered, long long limit) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Packet* const p = packets + (size_t)(tag & 1) * kMaxBasis * gridDim.x;
  const int kk = k > 0 ? k : 1;  // without sums: an empty packet
  if (threadIdx.x == 0) sc.failed = 0;
  __syncthreads();
  for (int j = warp; j < kk; j += kWarps) {
    Acc2 v;
    if (k > 0 && lane < kWarps) {
      v.hi = sc.part[j][lane].x;
      v.lo = sc.part[j][lane].y;
    }
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) {
      const float h = __shfl_down_sync(0xffffffffu, v.hi, o);
      const float l = __shfl_down_sync(0xffffffffu, v.lo, o);
      v.add(h);
      v.lo += l;
    }
    if (lane == 0) {
      const unsigned long long w = __double_as_longlong((double)v.hi + (double)v.lo);
      if (ordered) __threadfence();
      publish(p + (size_t)j * gridDim.x + blockIdx.x, (unsigned)w, (unsigned)(w >> 32),
              tag ^ sc.mute);
    }
  }
  for (int j = warp; j < kk; j += kWarps) {
    double v = 0.0;
    // kPoll packets of a lane on the way together
    for (int b0 = lane; b0 < (int)gridDim.x; b0 += 32 * kPoll) {
      Packet q[kPoll];
      long long began = 0;
      for (int spin = 1;; ++spin) {
        bool all = true;
#pragma unroll
        for (int i = 0; i < kPoll; ++i)
          if (b0 + 32 * i < (int)gridDim.x) q[i] = look(p + (size_t)j * gridDim.x + b0 + 32 * i);
#pragma unroll
        for (int i = 0; i < kPoll; ++i)
          if (b0 + 32 * i < (int)gridDim.x) all = all && arrived(q[i], tag);
        if (all) break;
        if (spin % 256 == 0) {
          const long long now = clock64();
          if (!began) began = now;
          if (now - began > limit) {
            sc.failed = 1;
            break;
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kPoll; ++i)
        if (b0 + 32 * i < (int)gridDim.x)
          v += __longlong_as_double(
              (long long)((unsigned long long)value_of(q[i].b) << 32 | value_of(q[i].a)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sc.sums[j] = v;
  }
  if (ordered) __threadfence();
  __syncthreads();
  return !sc.failed;
}

// One block per SM: without that bound the Allen-Cahn form was held to 64 registers
// and spilled (six steps at 64^2 1,610 us, so 1,538; two at 1024^2 2,400 and 2,260).
template <bool kCH>
__global__ void __launch_bounds__(kThreads, 1) k_newton2d(const Newton2DArgs a) {
  __shared__ TileMem<kCH> mem;
  __shared__ Scalars sc;
  const int64_t N = (int64_t)a.op.nx * a.op.ny;
  const int nx = a.op.nx, ny = a.op.ny;
  const int tiles_x = (nx + TX - 1) / TX, tiles = tiles_x * ((ny + TY - 1) / TY);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float cell = a.op.cell;
  float* const u = a.u;
  float* const un = a.un;
  float* const g = a.g;
  float* const d = a.d;
  unsigned phase = 0;
  if (threadIdx.x == 0) sc.mute = (int)blockIdx.x < a.mute ? 0x80000000u : 0u;

  // f(node, x, y) for this thread's nodes, tile by tile; the first tile's node
  // (the only one on small meshes) is worked out once
  const int fx = (int)blockIdx.x % tiles_x * TX + threadIdx.x % TX;
  const int fy = (int)blockIdx.x / tiles_x * TY + threadIdx.x / TX;
  const bool inside = fx < nx && fy < ny;
  const int64_t fo = (int64_t)fy * nx + fx;
  const auto nodes = [&](auto&& f) {
    if (inside) f(fo, fx, fy);
    for (int t = blockIdx.x + gridDim.x; t < tiles; t += gridDim.x) {
      const int x = t % tiles_x * TX + threadIdx.x % TX, y = t / tiles_x * TY + threadIdx.x / TX;
      if (x < nx && y < ny) f((int64_t)y * nx + x, x, y);
    }
  };
  const auto mass = [&](int x, int y) {
    return cell * ((x == 0 || x == nx - 1) ? 0.5f : 1.0f) * ((y == 0 || y == ny - 1) ? 0.5f : 1.0f);
  };
  // the warp's sums of kD accumulators, j of them in use, into sc.part
  const auto warp_parts = [&](Acc2* v, int j0, int k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
      for (int i = 0; i < kD; ++i) {
        const float h = __shfl_down_sync(0xffffffffu, v[i].hi, o);
        const float l = __shfl_down_sync(0xffffffffu, v[i].lo, o);
        v[i].add(h);
        v[i].lo += l;
      }
    }
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < kD; ++i)
        if (j0 + i < k) sc.part[j0 + i][warp] = make_float2(v[i].hi, v[i].lo);
    }
  };
  const auto reduce = [&](int k, bool ordered) {
    return end_phase(sc, static_cast<Packet*>(a.packets), ++phase, k, ordered, a.limit);
  };
  const auto apply = [&](auto jvp, const float* U, const float* W, auto&& put) {
    Implicit2DArgs op = a.op;
    op.U = U;
    op.W = W;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
      __syncthreads();  // the tile's memory is free
      tile_operator<decltype(jvp)::value, kCH, kThreads, true>(op, t, mem, put);
    }
  };
  using Jvp = std::integral_constant<bool, true>;
  using Residual = std::integral_constant<bool, false>;
  const auto basis = [&](int j) { return a.V + (int64_t)j * a.ldv; };
  // products of the first k basis vectors with w over the own nodes, kD at a time
  const auto dots = [&](const float* w, int k) {
    for (int j0 = 0; j0 < k; j0 += kD) {
      Acc2 v[kD];
      nodes([&](int64_t o, int, int) {
        const float w0 = w[o], w1 = kCH ? w[N + o] : 0.0f;
        float p[kD], q[kD];
#pragma unroll
        for (int i = 0; i < kD; ++i) {
          const float* b = basis(j0 + i < k ? j0 + i : j0);
          p[i] = b[o];
          if (kCH) q[i] = b[N + o];
        }
#pragma unroll
        for (int i = 0; i < kD; ++i) {
          float s = p[i] * w0;
          if (kCH) s = fmaf(q[i], w1, s);
          v[i].add(s);
        }
      });
      warp_parts(v, j0, k);
    }
  };
  const auto norm2 = [&](const float* w) {
    Acc2 v[kD];
    nodes([&](int64_t o, int, int) {
      float s = w[o] * w[o];
      if (kCH) s = fmaf(w[N + o], w[N + o], s);
      v[0].add(s);
    });
    warp_parts(v, 0, 1);
  };
  const auto mass_norm = [&](const float* p) {  // own nodes of |M p|^2
    Acc2 v[kD];
    nodes([&](int64_t o, int x, int y) {
      const float m = mass(x, y), s = m * p[o];
      float t = s * s;
      if (kCH) {
        const float s1 = m * p[N + o];
        t = fmaf(s1, s1, t);
      }
      v[0].add(t);
    });
    warp_parts(v, 0, 1);
  };
  // w -= sum_j c_j V_j on the own nodes, c_j = the last reduction's product
  // times the squared scale factor
  const auto update = [&](float* w, int k) {
    for (int j = threadIdx.x; j < k; j += kThreads)
      sc.coef[j] = (float)(sc.sums[j] * sc.scale[j] * sc.scale[j]);
    __syncthreads();
    nodes([&](int64_t o, int, int) {
      float s0 = w[o], s1 = kCH ? w[N + o] : 0.0f;
#pragma unroll 4
      for (int j = 0; j < k; ++j) {
        const float c = -sc.coef[j];
        s0 = fmaf(c, basis(j)[o], s0);
        if (kCH) s1 = fmaf(c, basis(j)[N + o], s1);
      }
      w[o] = s0;
      if (kCH) w[N + o] = s1;
    });
  };

  double initial = 0.0, rn = 0.0, tol = 0.0;
  int newton = 0, gmres = 0, status = 0, step = 0;
  for (; step < a.n_steps; ++step) {
    const float* start = step == 0 && a.guess ? a.guess : a.state;
    nodes([&](int64_t o, int, int) {
      un[o] = a.state[o];
      u[o] = start[o];
      if (kCH) un[N + o] = u[N + o] = 0.0f;
    });
    mass_norm(un);
    if (!reduce(1, true)) return;
    tol = a.newton_rtol * sqrt(sc.sums[0]) * (double)a.inv_dt;
    const double atol = a.atol_factor * tol;
    if (kCH) {  // mu of the starting c: with mu = 0 the mu row of M^-1 R is -M^-1 r(c)
      apply(Residual{}, u, un, [&](int64_t o, int, int, float, float o1) { g[o] = -o1; });
      if (!reduce(0, true)) return;  // every block has read mu = 0
      nodes([&](int64_t o, int, int) { u[N + o] = g[o]; });
      if (!reduce(0, true)) return;
    }
    bool ok = false;
    for (int it = 0;; ++it) {
      apply(Residual{}, u, un, [&](int64_t o, int, int, float o0, float o1) {
        g[o] = o0;
        if (kCH) g[N + o] = o1;
      });
      mass_norm(g);
      if (!reduce(1, true)) return;
      rn = sqrt(sc.sums[0]);
      if (!isfinite(rn)) {
        status = PF_ERR_NONFINITE;
        break;
      }
      if (step == 0 && it == 0) initial = rn;
      if (rn <= tol) {
        ok = true;
        break;
      }
      if (it >= a.max_newton) break;

      // GMRES for (M^-1 J) x = -G at u, x in d
      int total = 0;
      double beta0 = -1.0;
      nodes([&](int64_t o, int, int) {
        d[o] = 0.0f;
        if (kCH) d[N + o] = 0.0f;
      });
      for (;;) {
        float* const v0 = basis(0);
        if (total == 0) {
          nodes([&](int64_t o, int, int) {
            v0[o] = -g[o];
            if (kCH) v0[N + o] = -g[N + o];
          });
        } else {
          if (!reduce(0, true)) return;  // x is complete
          apply(Jvp{}, u, d, [&](int64_t o, int, int, float o0, float o1) {
            v0[o] = -g[o] - o0;
            if (kCH) v0[N + o] = -g[N + o] - o1;
          });
        }
        norm2(v0);
        if (!reduce(1, true)) return;
        const double beta = sqrt(sc.sums[0]);
        if (beta0 < 0.0) beta0 = beta;
        if (beta0 == 0.0) break;
        const double target = fmax(a.gmres_rtol * beta0, atol);
        if (beta <= target || total >= a.maxit) break;
        if (threadIdx.x == 0) {
          sc.scale[0] = (float)(1.0 / beta);
          sc.gv[0] = beta;
          sc.stop = 0;
        }
        __syncthreads();
        int k = 0;
        for (; k < a.restart && total < a.maxit && !sc.stop; ++k) {
          float* const w = basis(k + 1);
          const float sk = sc.scale[k];
          apply(Jvp{}, u, basis(k), [&](int64_t o, int, int, float o0, float o1) {
            w[o] = sk * o0;
            if (kCH) w[N + o] = sk * o1;
          });
          dots(w, k + 1);
          if (!reduce(k + 1, false)) return;
          for (int j = threadIdx.x; j <= k; j += kThreads) sc.hk[j] = sc.sums[j] * sc.scale[j];
          update(w, k + 1);
          dots(w, k + 1);
          if (!reduce(k + 1, false)) return;
          for (int j = threadIdx.x; j <= k; j += kThreads) sc.hk[j] += sc.sums[j] * sc.scale[j];
          update(w, k + 1);
          norm2(w);
          if (!reduce(1, true)) return;
          ++total;
          if (threadIdx.x == 0) {
            double* const h = sc.H[k];
            // reciprocal square roots alone: FP64 roots and divisions take
            // most of a phase's time each
            const double s2 = fmax(sc.sums[0], 0.0), r1 = s2 > 0.0 ? rsqrt(s2) : 0.0;
            const double hk1 = s2 * r1;
            if (k + 1 < kMaxBasis) sc.scale[k + 1] = (float)r1;
            double top = sc.hk[0];
            for (int j = 0; j < k; ++j) {
              const double low = sc.hk[j + 1];
              h[j] = sc.cs[j] * top + sc.sn[j] * low;
              top = -sc.sn[j] * top + sc.cs[j] * low;
            }
            const double d2 = top * top + s2, rd = d2 > 0.0 ? rsqrt(d2) : 0.0;
            sc.cs[k] = d2 > 0.0 ? top * rd : 1.0;
            sc.sn[k] = hk1 * rd;
            h[k] = d2 * rd;
            sc.gv[k + 1] = -sc.sn[k] * sc.gv[k];
            sc.gv[k] = sc.cs[k] * sc.gv[k];
            sc.stop = fabs(sc.gv[k + 1]) <= target || hk1 == 0.0;
          }
          __syncthreads();
        }
        // y = H^-1 g (upper triangular), x += V y
        if (threadIdx.x == 0) {
          for (int i = k - 1; i >= 0; --i) {
            double s = sc.gv[i];
            for (int j = i + 1; j < k; ++j) s -= sc.H[j][i] * sc.y[j];
            sc.y[i] = s / sc.H[i][i];
          }
          for (int j = 0; j < k; ++j) sc.coef[j] = (float)(sc.y[j] * sc.scale[j]);
        }
        __syncthreads();
        nodes([&](int64_t o, int, int) {
          float s0 = d[o], s1 = kCH ? d[N + o] : 0.0f;
          for (int j = 0; j < k; ++j) {
            s0 = fmaf(sc.coef[j], basis(j)[o], s0);
            if (kCH) s1 = fmaf(sc.coef[j], basis(j)[N + o], s1);
          }
          d[o] = s0;
          if (kCH) d[N + o] = s1;
        });
        const bool done = sc.stop || total >= a.maxit;
        __syncthreads();
        if (done) break;
      }
      gmres += total;
      ++newton;
      nodes([&](int64_t o, int, int) {
        u[o] += d[o];
        if (kCH) u[N + o] += d[N + o];
      });
      if (!reduce(0, true)) return;  // u is complete
    }
    if (status == 0 && !ok) status = PF_ERR_NOT_CONVERGED;
    if (status != PF_ERR_NONFINITE) nodes([&](int64_t o, int, int) { a.state[o] = u[o]; });
    if (status != 0) break;
    if (!reduce(0, true)) return;  // the state is complete (the next step's start)
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    double* const r = a.result;
    r[0] = status;
    r[1] = newton;
    r[2] = gmres;
    r[3] = initial;
    r[4] = rn;
    r[5] = tol;
    r[6] = step;
  }
}

}  // namespace

int64_t newton2d_tile_nodes(int nx, int ny) {
  return (int64_t)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY) * (TX * TY);
}

int newton2d_blocks(int nx, int ny) {
  const int64_t tiles = newton2d_tile_nodes(nx, ny) / (TX * TY);
  const int64_t sms = device_sm_count();
  return (int)(tiles < sms ? tiles : sms);
}

size_t newton2d_packet_bytes(int nx, int ny) {
  return sizeof(Packet) * 2 * kMaxBasis * (size_t)newton2d_blocks(nx, ny);
}

cudaError_t launch_newton2d(const Newton2DArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(newton2d_blocks(a.op.nx, a.op.ny));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return a.op.ch ? cudaLaunchKernelEx(&cfg, k_newton2d<true>, a)
                 : cudaLaunchKernelEx(&cfg, k_newton2d<false>, a);
}

}  // namespace pf
