// Fused 2-D explicit step kernels: element gather -> Gauss-point values ->
// f'(u_q) -> node-centric gather of the element contributions -> gradient
// stencil -> lumped-mass Euler update (JAX-PF Eq. 11-12; Cahn-Hilliard via the
// split form of Eq. 9-10).  One pass reads the state once and writes it once.
//
// Work split.  A warp owns 64 consecutive columns (a pair per lane) and
// sweeps down a band of rows with a sliding window in registers; the
// neighbouring columns come from the adjacent lanes by warp shuffle, so there
// is no shared memory and no block barrier, and every element is evaluated
// once per warp.  Lanes 0 and 31 are halo lanes (their outer column lacks a
// neighbour), so warps overlap by 4 columns and each writes the 60 columns of
// lanes 1..30.  All arithmetic is on packed FP32 pairs (one lane's two
// columns) with the f32x2 instructions of sm_100+, which halve the issue slots
// of the FP32 work.
//
// Quadrature is sum-factorised (sweep2d.h): per row, two x-interpolated values
// per segment; per element, the four Gauss values from the segment values of
// its two rows; the weights N_a(q) are applied back the same way (y first into
// per-segment sums, then x into the nodes).  The linear gradient term is the
// exact assembled 9-point Q1 stencil (2x2 Gauss integrates it exactly); on
// square cells it is a v + b (sum of the 3x3 block).
// Zero-flux boundaries are the mirror extension about the boundary nodes,
// which equals the partial element sets divided by the partial lumped masses
// (both double when mirrored), so every node uses the interior formula.  The
// working planes carry that extension explicitly: a frame of 2 ghost rows and
// columns that every step rewrites from the nodes it mirrors, so all warps run
// the same branch-free sweep with no index reflection.
#include <string.h>

#include <cmath>
#include <type_traits>

#include "pf_internal.h"
#include "sweep2d.h"

namespace pf {
namespace {

using namespace sweep;

template <int V>
using Int = std::integral_constant<int, V>;

#ifndef PF_WARPS
#define PF_WARPS 2
#endif
constexpr int kWarps = PF_WARPS;                  // warps per block, stacked in y
#ifndef PF_ROWS_AHEAD
#define PF_ROWS_AHEAD 6
#endif
#ifndef PF_MINB
#define PF_MINB 1  // minimum resident blocks per SM asked of the register allocator
#endif
#ifndef PF_ENS_MINB
#define PF_ENS_MINB 6  // minimum resident ensemble blocks per SM asked of the register allocator
#endif
#ifndef PF_ENS_COEF
#define PF_ENS_COEF 2  // ensemble coefficients: 0 registers, 1 instance table, 2 shared memory
#endif
#ifndef PF_PDL
#define PF_PDL 0  // 1: programmatic dependent launch, dependents released at block end
#endif
constexpr int kAhead = PF_ROWS_AHEAD;  // rows loaded ahead of use (divides the unroll of 6)

__device__ __forceinline__ int reflect_row(int k, int n) {
  k = k < 0 ? -k : k;
  k = k >= n ? 2 * (n - 1) - k : k;
  return k < 0 ? 0 : (k >= n ? n - 1 : k);  // rows this far out are never stored
}

__device__ __forceinline__ int reflect_col(int x, int n) {
  const int p = 2 * (n - 1);
  x %= p;
  if (x < 0) x += p;
  return x < n ? x : p - x;
}

// One warp task: the band of kTY output rows starting at y0, columns of
// warp column bx.
template <bool kCoherent, bool kHint>
__device__ __forceinline__ u64 ld_row(const float* p, u64 pol) {
  // coherent (L2) loads when the planes were written earlier in the same launch;
  // with kHint the load carries the L2 eviction policy `pol`
  if constexpr (kHint) {
    u64 v;
    if constexpr (kCoherent)
      asm volatile("ld.global.cg.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(v) : "l"(p), "l"(pol));
    else
      asm volatile("ld.global.nc.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(v) : "l"(p), "l"(pol));
    return v;
  } else {
    return kCoherent ? __ldcg(reinterpret_cast<const u64*>(p))
                     : __ldg(reinterpret_cast<const u64*>(p));
  }
}

template <bool kHint>
__device__ __forceinline__ void st_row(float* p, u64 v, u64 pol) {
  if constexpr (kHint)
    asm volatile("st.global.L2::cache_hint.b64 [%0], %1, %2;" ::"l"(p), "l"(v), "l"(pol) : "memory");
  else
    *reinterpret_cast<u64*>(p) = v;
}

// L2 eviction policy of an ensemble instance's plane accesses
__device__ __forceinline__ u64 l2_policy(int l2) {
  u64 p;
  if (l2 == kL2Stream)
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  else if (l2 == kL2StreamHalf)
    asm volatile("createpolicy.fractional.L2::evict_first.L2::evict_unchanged.b64 %0, 0.5;"
                 : "=l"(p));
  else
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}

template <bool kCH, bool kIso, bool kOdd, int kTY, bool kCoherent = false, bool kHint = false>
__device__ __forceinline__ void sweep_task(const Explicit2DArgs& a, const float* in, float* out,
                                           const Coef& K, int bx, int y0, u64 pol = 0) {
  constexpr int kLag = kCH ? 2 : 1;
  const int lane = threadIdx.x & 31;
  const int nx = a.nx, ny = a.ny;
  const int64_t pitch = a.pitch;
  const int x = bx * kOutCols - kPair + kPair * lane;  // real column of lo
  const bool writer = lane >= 1 && lane <= 30 && x < nx;
  // plain vector store unless this lane / band also owns mirror-frame cells
  const bool ghost_cols = x <= 2 || x + 1 >= nx - 3;
  const bool ghost_rows = y0 <= 2 || y0 + kTY + 3 >= ny;
  const bool plain = writer && !ghost_cols && !ghost_rows;
  // origin of the real mesh inside the ghost-padded planes
  const float* __restrict__ in0 = in + kGhost * pitch + kGhost;
  float* __restrict__ out0 = out + kGhost * pitch + kGhost;
  const float* src = in0 + (int64_t)(y0 - kLag) * pitch + x;
  Window<1> w;
  u64 ahead[kAhead];  // rows k .. k+kAhead-1 in flight
#pragma unroll
  for (int j = 0; j < kAhead; ++j) {
    ahead[j] = ld_row<kCoherent, kHint>(src, pol);
    src += pitch;
  }
  const auto next = [&]() {
    const u64 P = ahead[0];
#pragma unroll
    for (int j = 0; j + 1 < kAhead; ++j) ahead[j] = ahead[j + 1];
    ahead[kAhead - 1] = ld_row<kCoherent, kHint>(src, pol);
    src += pitch;
    return P;
  };
  u64 o[1];
  const auto consume = [&](auto stage) {
    const u64 P[1] = {next()};
    const float cl = __shfl_up_sync(kFull, phi(P[0]), 1);   // column x-1
    const float cr = __shfl_down_sync(kFull, plo(P[0]), 1);  // column x+2
    row<kCH, kIso, kOdd, 1, decltype(stage)::value, false>(P, cl, cr, 0.0f, w, K, o);
  };
  // fill the window, nothing to store yet: each row goes as far as later rows need
  consume(Int<kInterp>{});
  consume(Int<kElement>{});
  if constexpr (kCH) {
    consume(Int<kMu>{});
    consume(Int<kMu>{});
  }
#pragma unroll 6
  for (int it = 0; it < kTY; ++it) {
    consume(Int<kOutput>{});
    const int y = y0 + it;
    if (plain)
      st_row<kHint>(out0 + (int64_t)y * pitch + x, o[0], pol);
    else if (writer && y < ny)
      store_out(out0, pitch, y, ny, x, nx, o[0]);
  }
}

// One warp per block and one (column, band) task per warp: many small blocks
// spread evenly over the SMs and keep each scheduler fed from several warps.
template <bool kCH, bool kIso, bool kOdd, int kTY>
__global__ void __launch_bounds__(kWarps * 32, PF_MINB) k_explicit2d(const Explicit2DArgs a) {
#if PF_PDL
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the previous step is complete
#endif
  const int warp = threadIdx.x >> 5;
  const int y0 = (block_row() * kWarps + warp) * kTY;
  if (y0 < a.ny) sweep_task<kCH, kIso, kOdd, kTY>(a, a.in, a.out, Coef{a.pair}, blockIdx.x, y0);
#if PF_PDL
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}

// ---------------------------------------------------------------------------
// Batched ensembles of independent 2-D Allen-Cahn instances (different sizes
// and parameters).  Every instance has its own ghost-padded planes A/B and its
// own packed coefficients; the warp tasks of all instances -- (instance,
// column of 60, band of ty rows) -- form one list, so one launch advances the
// whole ensemble.  The persistent form keeps one launch resident for all
// steps, with a bounded grid barrier between steps.

template <bool kIso, bool kOdd, bool kCoherent>
__device__ __forceinline__ void ensemble_task(const EnsTask& t, const Explicit2DArgs* inst,
                                              int parity) {
  const Explicit2DArgs& a = inst[t.inst];
#if PF_ENS_COEF == 0
  unsigned long long pair[19];
#pragma unroll
  for (int i = 0; i < 19; ++i) pair[i] = a.pair[i];
  const Coef K{pair};
#elif PF_ENS_COEF == 1
  const Coef K{a.pair};  // read through the instance table (L1-resident, warp-uniform)
#else
  __shared__ unsigned long long s_pair[kEnsThreads / 32][20];
  unsigned long long* sp = s_pair[threadIdx.x >> 5];
  __syncwarp();
  if ((threadIdx.x & 31) < 19) sp[threadIdx.x & 31] = a.pair[threadIdx.x & 31];
  __syncwarp();
  const Coef K{sp};
#endif
  const float* in = parity ? a.out : a.in;
  float* out = parity ? const_cast<float*>(a.in) : a.out;
  const u64 pol = l2_policy(a.l2);
  switch (t.ty) {
    case 6: sweep_task<false, kIso, kOdd, 6, kCoherent, true>(a, in, out, K, t.bx, t.y0, pol); break;
    case 12: sweep_task<false, kIso, kOdd, 12, kCoherent, true>(a, in, out, K, t.bx, t.y0, pol); break;
    default: sweep_task<false, kIso, kOdd, 24, kCoherent, true>(a, in, out, K, t.bx, t.y0, pol); break;
  }
}

template <bool kIso, bool kOdd>
__global__ void __launch_bounds__(kEnsThreads, PF_ENS_MINB) k_ensemble_step(const EnsTask* __restrict__ tasks,
                                                              int ntasks,
                                                              const Explicit2DArgs* inst,
                                                              int parity) {
  const int warps = kEnsThreads / 32;
  for (int t = blockIdx.x * warps + (threadIdx.x >> 5); t < ntasks; t += gridDim.x * warps)
    ensemble_task<kIso, kOdd, false>(tasks[t], inst, parity);
}

// Grid-wide barrier for a co-resident (cooperative) grid, with a bounded wait.
// bar[0] counts arrivals, bar[1] is the generation, bar[2] the error flag.  A
// block that waits longer than `limit` clock cycles sets the flag and reports
// failure.
__device__ bool grid_barrier(unsigned* bar, long long limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned* vgen = bar + 1;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u);
    if (arrived == gridDim.x - 1) {
      bar[0] = 0;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == gen) {
        if (clock64() - t0 > limit) {
          atomicExch(bar + 2, 1u);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

template <bool kIso, bool kOdd>
__global__ void __launch_bounds__(kEnsThreads, PF_ENS_MINB) k_ensemble_persistent(
    const EnsTask* __restrict__ tasks, int ntasks, const Explicit2DArgs* inst, int n_steps,
    unsigned* bar, long long limit) {
  const int warps = kEnsThreads / 32;
  for (int s = 0; s < n_steps; ++s) {
    for (int t = blockIdx.x * warps + (threadIdx.x >> 5); t < ntasks; t += gridDim.x * warps)
      ensemble_task<kIso, kOdd, true>(tasks[t], inst, s & 1);
    if (!grid_barrier(bar, limit)) return;
  }
}

// Self-test of the bounded barrier: `extra` phantom arrivals are expected that
// never come, so every block's wait must expire and set the error flag.
__global__ void k_barrier_selftest(unsigned* bar, long long limit, int extra) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned* vgen = bar + 1;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u);
    if (arrived == gridDim.x + extra - 1) {
      atomicAdd(bar + 1, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == gen) {
        if (clock64() - t0 > limit) {
          atomicExch(bar + 2, 1u);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
  }
  __syncthreads();
}

// all instances' plain states (packed) <-> their padded working planes
// (grid.y strides over the instances, so any count fits in one launch; blocks
// stride over rows and threads over columns, so no index is divided)
__global__ void k_ens_to_work(const float* __restrict__ packed, const int64_t* __restrict__ off,
                              const Explicit2DArgs* inst, int count, float sub) {
  for (int k = blockIdx.y; k < count; k += gridDim.y) {
    const Explicit2DArgs& a = inst[k];
    const int nx = a.nx, ny = a.ny;
    const int64_t pitch = a.pitch;
    const float* in = packed + off[k];
    for (int v = blockIdx.x; v < a.rows; v += gridDim.x) {
      const int y = v - kGhost;
      const bool row = y >= -kGhost && y < ny + kGhost;
      const int64_t src = (int64_t)reflect_row(y, ny) * nx;
      float* dA = const_cast<float*>(a.in) + v * pitch;
      float* dB = a.out + v * pitch;
      for (int u = threadIdx.x; u < pitch; u += blockDim.x) {
        const int x = u - kGhost;
        float val = 0.0f;
        if (row && x >= -kGhost && x < nx + kGhost) val = in[src + reflect_col(x, nx)] - sub;
        dA[u] = val;
        dB[u] = val;
      }
    }
  }
}

__global__ void k_ens_from_work(float* __restrict__ packed, const int64_t* __restrict__ off,
                                const Explicit2DArgs* inst, int count, int parity, float add) {
  for (int k = blockIdx.y; k < count; k += gridDim.y) {
    const Explicit2DArgs& a = inst[k];
    const int nx = a.nx;
    const float* work = parity ? a.out : a.in;
    float* out = packed + off[k];
    for (int y = blockIdx.x; y < a.ny; y += gridDim.x) {
      const float* src = work + (int64_t)(y + kGhost) * a.pitch + kGhost;
      float* dst = out + (int64_t)y * nx;
      for (int x = threadIdx.x; x < nx; x += blockDim.x) dst[x] = src[x] + add;
    }
  }
}

// Plain <-> padded working layout of grid.y fields one after another.  Working
// cell (u, v) holds real node (reflect(u - kGhost), reflect(v - kGhost)),
// minus/plus the shift for the first field; padding beyond the ghost frame is
// zero.  Both buffers of the ping-pong are filled in one launch (a launch costs
// the host 2 to 6 us, as much as a step of a small mesh).  Blocks stride over
// rows, threads over columns.
__global__ void k_to_work(const float* __restrict__ in, float* __restrict__ a,
                          float* __restrict__ b, int nx, int ny, int64_t pitch, int rows,
                          float sub) {
  in += (int64_t)blockIdx.y * nx * ny;
  a += blockIdx.y * pitch * rows;
  b += blockIdx.y * pitch * rows;
  if (blockIdx.y) sub = 0.0f;
  for (int v = blockIdx.x; v < rows; v += gridDim.x) {
    const int y = v - kGhost;
    const bool row = y >= -kGhost && y < ny + kGhost;
    const int64_t src = (int64_t)reflect_row(y, ny) * nx;
    for (int u = threadIdx.x; u < pitch; u += blockDim.x) {
      const int x = u - kGhost;
      float val = 0.0f;
      if (row && x >= -kGhost && x < nx + kGhost) val = in[src + reflect_col(x, nx)] - sub;
      a[v * pitch + u] = val;
      b[v * pitch + u] = val;
    }
  }
}

__global__ void k_from_work(const float* __restrict__ work, float* __restrict__ out, int nx,
                            int ny, int64_t pitch, int rows, float add) {
  work += blockIdx.y * pitch * rows;
  out += (int64_t)blockIdx.y * nx * ny;
  if (blockIdx.y) add = 0.0f;
  for (int y = blockIdx.x; y < ny; y += gridDim.x) {
    const float* src = work + (int64_t)(y + kGhost) * pitch + kGhost;
    float* dst = out + (int64_t)y * nx;
    for (int x = threadIdx.x; x < nx; x += blockDim.x) dst[x] = src[x] + add;
  }
}

#ifndef PF_TY_CH
#define PF_TY_CH 6
#endif
#ifndef PF_TY_AC
#define PF_TY_AC 6
#endif
// Output rows per warp band (a multiple of the unroll of 6).  Taller bands
// repeat fewer warm-up rows but leave fewer warps and, as a loop, hold the
// coefficients in registers (110 against 70): Allen-Cahn at 12 rows took 59 us
// per step at 4096^2 and 22 at 2700^2, at 6 rows 29 and 13.
constexpr int kTYAc = PF_TY_AC;
constexpr int kTYCh = PF_TY_CH;

template <bool kCH, bool kIso, bool kOdd, int kTY>
cudaError_t launch(const Explicit2DArgs& a, cudaStream_t s) {
  const dim3 grid = row_grid((a.nx + kOutCols - 1) / kOutCols, (a.ny + kWarps * kTY - 1) / (kWarps * kTY));
#if PF_PDL
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kWarps * 32);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_explicit2d<kCH, kIso, kOdd, kTY>, a);
#else
  k_explicit2d<kCH, kIso, kOdd, kTY><<<grid, kWarps * 32, 0, s>>>(a);
  return cudaGetLastError();
#endif
}

bool is_iso(const Stencil2D& k) { return k.cx == k.cd && k.cy == k.cd; }

}  // namespace

cudaError_t launch_ac2d(const Explicit2DArgs& a, cudaStream_t s) {
  switch (sweep_variant(is_iso(a.k1), a.odd)) {
    case 0: return launch<false, true, true, kTYAc>(a, s);
    case 1: return launch<false, false, true, kTYAc>(a, s);
    default: return launch<false, false, false, kTYAc>(a, s);
  }
}

cudaError_t launch_ch2d(const Explicit2DArgs& a, cudaStream_t s) {
  switch (sweep_variant(is_iso(a.k1) && is_iso(a.k2), a.odd)) {
    case 0: return launch<true, true, true, kTYCh>(a, s);
    case 1: return launch<true, false, true, kTYCh>(a, s);
    default: return launch<true, false, false, kTYCh>(a, s);
  }
}

void pack_explicit2d(const double (&f)[4], Explicit2DArgs& a) {
  auto pk_host = [](float v) {
    unsigned int b;
    memcpy(&b, &v, 4);
    return (unsigned long long)b | ((unsigned long long)b << 32);
  };
  a.p0 = (float)f[0];
  a.p1 = (float)f[1];
  a.p2 = (float)f[2];
  a.p3 = (float)f[3];
  // interpolated values lack a factor g_hi^2 and so do the weights back, so
  // p_i carries g_hi^(2 i + 2); the polynomial is odd about the double well's
  // centre (p0 = p2 = 0), and its form p3 (v^2 + p1/p3) v needs p3 != 0.  Every
  // coefficient is rounded once, p1/p3 so that its product with the rounded p3,
  // the slope at the centre, is
  const double g2 = kGRho * kGRho;
  double p[4], s = g2;
  for (int i = 0; i < 4; ++i, s *= g2) p[i] = f[i] * s;
  const float ratio = (float)(p[1] / (double)(float)p[3]);
  a.odd = a.p0 == 0.0f && a.p2 == 0.0f && a.p3 != 0.0f && std::isfinite(ratio);
  a.pair[0] = pk_host(kRho);
  a.pair[1] = pk_host(a.odd ? ratio : 0.0f);
  a.pair[2] = pk_host((float)p[3]);
  for (int i = 0; i < 4; ++i) a.pair[3 + i] = pk_host((float)p[i]);
  const Stencil2D* st[2] = {&a.k1, &a.k2};
  for (int k = 0; k < 2; ++k) {
    a.pair[7 + 6 * k + 0] = pk_host(st[k]->c0 - st[k]->cd);
    a.pair[7 + 6 * k + 1] = pk_host(st[k]->cd);
    a.pair[7 + 6 * k + 2] = pk_host(st[k]->c0);
    a.pair[7 + 6 * k + 3] = pk_host(st[k]->cx);
    a.pair[7 + 6 * k + 4] = pk_host(st[k]->cy);
    a.pair[7 + 6 * k + 5] = pk_host(st[k]->cd);
  }
}

cudaError_t launch_ensemble_step(const EnsTask* tasks, int ntasks, const Explicit2DArgs* inst,
                                 int parity, bool iso, bool odd, int grid, cudaStream_t s) {
  const int v = sweep_variant(iso, odd);
  auto* k = v == 0   ? k_ensemble_step<true, true>
            : v == 1 ? k_ensemble_step<false, true>
                     : k_ensemble_step<false, false>;
  k<<<grid, kEnsThreads, 0, s>>>(tasks, ntasks, inst, parity);
  return cudaGetLastError();
}

namespace {
auto* persistent_kernel(bool iso, bool odd) {
  const int v = sweep_variant(iso, odd);
  return v == 0   ? k_ensemble_persistent<true, true>
         : v == 1 ? k_ensemble_persistent<false, true>
                  : k_ensemble_persistent<false, false>;
}
}  // namespace

int ensemble_persistent_grid(bool iso, bool odd) {
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, persistent_kernel(iso, odd), kEnsThreads,
                                                    0) != cudaSuccess)
    return 0;
  return device_sm_count() * per;
}

cudaError_t launch_ensemble_persistent(const EnsTask* tasks, int ntasks, const Explicit2DArgs* inst,
                                       int n_steps, unsigned* bar, long long limit, bool iso,
                                       bool odd, int grid, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kEnsThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, persistent_kernel(iso, odd), tasks, ntasks, inst, n_steps, bar,
                            limit);
}

cudaError_t launch_ens_to_work(const float* packed, const int64_t* off, const Explicit2DArgs* inst,
                               int count, float shift, cudaStream_t s) {
  const unsigned gy = count < (int)kMaxGridY ? (unsigned)count : kMaxGridY;
  k_ens_to_work<<<dim3(64, gy), 256, 0, s>>>(packed, off, inst, count, shift);
  return cudaGetLastError();
}

cudaError_t launch_ens_from_work(float* packed, const int64_t* off, const Explicit2DArgs* inst,
                                 int count, int parity, float shift, cudaStream_t s) {
  const unsigned gy = count < (int)kMaxGridY ? (unsigned)count : kMaxGridY;
  k_ens_from_work<<<dim3(64, gy), 256, 0, s>>>(packed, off, inst, count, parity, shift);
  return cudaGetLastError();
}

cudaError_t launch_barrier_selftest(unsigned* bar, long long limit, int extra, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(32);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_barrier_selftest, bar, limit, extra);
}

int work_pitch(int nx) {
  const int gx = (nx + kOutCols - 1) / kOutCols;
  const int p = gx * kOutCols + 2 * kGhost + 2 * kPair;
  return (p + 3) / 4 * 4;
}

int work_rows(int ny) {
  // the last band reads up to ty + kLag + kAhead rows past its first row
  int ty = kTYAc > kTYCh ? kTYAc : kTYCh;
  if (ty < kMaxEnsTY) ty = kMaxEnsTY;
  return ny + ty + kAhead + 2 * kGhost + 4;
}

cudaError_t launch_to_work(const float* in, float* a, float* b, int nx, int ny, int fields,
                           float shift, cudaStream_t s) {
  int64_t blocks = work_rows(ny);
  if (blocks > 16 * (int64_t)device_sm_count()) blocks = 16 * (int64_t)device_sm_count();
  k_to_work<<<dim3((unsigned)blocks, fields), 256, 0, s>>>(in, a, b, nx, ny, work_pitch(nx),
                                                           work_rows(ny), shift);
  return cudaGetLastError();
}

cudaError_t launch_from_work(const float* work, float* out, int nx, int ny, int fields,
                             float shift, cudaStream_t s) {
  int64_t blocks = ny;
  if (blocks > 16 * (int64_t)device_sm_count()) blocks = 16 * (int64_t)device_sm_count();
  k_from_work<<<dim3((unsigned)blocks, fields), 256, 0, s>>>(work, out, nx, ny, work_pitch(nx),
                                                             work_rows(ny), shift);
  return cudaGetLastError();
}

}  // namespace pf
