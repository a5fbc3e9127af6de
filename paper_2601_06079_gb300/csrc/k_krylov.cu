// Vector kernels of the Newton-GMRES solver (JAX-PF Eq. 13-14).  The Krylov
// basis is FP32; every inner product and norm keeps about 48 bits per thread
// and finishes in FP64: each thread forms FP32 sums over 8 consecutive
// products (4 in the projections) and adds them into a compensated FP32 pair
// (hi + lo, Knuth's two-sum), warps combine the pairs the same way and blocks add the warps'
// values in FP64, and the last block sums the per-block partials in a fixed
// order, so results are deterministic.  No FP64 arithmetic runs per element: GB300 issues about 2
// FP64 operations per clock per SM, 64 times fewer than FP32.
#include <type_traits>

#include "pf_internal.h"

namespace pf {
namespace {

constexpr int kThreads = 256;
constexpr int kChunk = 8;      // products per FP32 partial sum
constexpr int kMaxFields = 8;  // order parameters of a Newton vector (planes of the mass norm)

// s added to the unevaluated sum hi + lo (Knuth's two-sum: the rounding error
// of hi + s is exact in FP32 and collects in lo)
struct Acc2 {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float s) {
    const float t = hi + s;
    const float bp = t - hi;
    lo += (hi - (t - bp)) + (s - bp);
    hi = t;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// The reductions' last stages.  warp_value: the warp's sum of accumulator j
// into shared memory (no block barrier per vector); then finish_sums: the
// block's sums into partials[j * blocks + b], and the last block to finish adds
// all blocks' partials into out[j], its 8 warps shared out among up to 4 vectors
// (more have a warp each, in turn), in a fixed order (blocks in steps of
// 32 lanes times the vector's warps, a tree, then the warps), so one launch gives
// the final, repeatable values.  count: device counter, 0 before the launch and
// reset to 0 by the last block.  (With two barriers per vector and block, and the
// last block taking the vectors one after another, 8 products of 4,096 values took
// 16.5 us, nearly all of it here; now 4.  A single sum of 456 partials by one warp cost
// 0.9 us more: k_update of 10^6 values 10.3 us, so 9.4.)
constexpr int kWarpsPerBlock = kThreads / 32;

__device__ __forceinline__ void warp_value(Acc2 a, int j, double (*sums)[kWarpsPerBlock]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_down_sync(0xffffffffu, a.hi, o);
    const float l = __shfl_down_sync(0xffffffffu, a.lo, o);
    a.add(h);
    a.lo += l;
  }
  if ((threadIdx.x & 31) == 0) sums[j][threadIdx.x >> 5] = a.value();
}

// a warp's share (part of kShare) of the blocks' partials, in its lane 0
template <int kShare>
__device__ __forceinline__ double partial_sum(const double* p, int blocks, int part, int lane) {
  double v = 0.0;
  for (int b = 32 * part + lane; b < blocks; b += 32 * kShare) v += __ldcg(p + b);
  return warp_sum(v);
}

__device__ void finish_sums(double (*sums)[kWarpsPerBlock], double* partials, int k,
                            double* __restrict__ out, unsigned* count) {
  __shared__ bool last;
  const int blocks = gridDim.x, w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  for (int j = threadIdx.x; j < k; j += kThreads) {
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < kWarpsPerBlock; ++i) v += sums[j][i];
    if (blocks == 1)
      out[j] = v;
    else
      partials[(int64_t)j * blocks + blockIdx.x] = v;
  }
  if (blocks == 1) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(count, 1u) == blocks - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (k > 4) {  // a warp per vector
    for (int j = w; j < k; j += kWarpsPerBlock) {
      const double v = partial_sum<1>(partials + (int64_t)j * blocks, blocks, 0, l);
      if (l == 0) out[j] = v;
    }
  } else {
    const int share = k == 1 ? 8 : (k == 2 ? 4 : 2), j = w / share;
    if (j < k) {
      const double* p = partials + (int64_t)j * blocks;
      const double v = share == 8   ? partial_sum<8>(p, blocks, w % 8, l)
                       : share == 4 ? partial_sum<4>(p, blocks, w % 4, l)
                                    : partial_sum<2>(p, blocks, w % 2, l);
      if (l == 0) sums[j][w % share] = v;
    }
    __syncthreads();
    if (threadIdx.x < k) {
      double v = sums[threadIdx.x][0];
      for (int i = 1; i < share; ++i) v += sums[threadIdx.x][i];
      out[threadIdx.x] = v;
    }
  }
  if (threadIdx.x == 0) *count = 0;
}

// Chunks of kChunk = 8 consecutive values: two 16-byte loads when the vectors
// are 16-byte aligned (kVec) and the chunk is whole, elementwise otherwise
// (values past n read as 0).  Each kernel below is instantiated for a bound
// KMAX on the number of basis vectors (4, 8, 16, 32), so that its accumulators
// (compensated FP32 pairs) take registers only for the vectors a call can have.
template <bool kVec>
__device__ __forceinline__ void load8(const float* __restrict__ p, int64_t i0, int64_t n,
                                      float v[kChunk]) {
  if (kVec && i0 + kChunk <= n) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p + i0));
    const float4 b = __ldg(reinterpret_cast<const float4*>(p + i0 + 4));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int t = 0; t < kChunk; ++t) v[t] = (i0 + t < n) ? p[i0 + t] : 0.0f;
  }
}

template <bool kVec>
__device__ __forceinline__ void load4(const float* p, int64_t i0, int64_t n, float v[4]) {
  if (kVec && i0 + 4 <= n) {
    const float4 a = *reinterpret_cast<const float4*>(p + i0);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = (i0 + t < n) ? p[i0 + t] : 0.0f;
  }
}

template <bool kVec>
__device__ __forceinline__ void store4(float* p, int64_t i0, int64_t n, const float v[4]) {
  if (kVec && i0 + 4 <= n) {
    *reinterpret_cast<float4*>(p + i0) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (i0 + t < n) p[i0 + t] = v[t];
  }
}

template <bool kVec>
__device__ __forceinline__ void store8(float* __restrict__ p, int64_t i0, int64_t n,
                                       const float v[kChunk]) {
  if (kVec && i0 + kChunk <= n) {
    *reinterpret_cast<float4*>(p + i0) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(p + i0 + 4) = make_float4(v[4], v[5], v[6], v[7]);
  } else {
#pragma unroll
    for (int t = 0; t < kChunk; ++t)
      if (i0 + t < n) p[i0 + t] = v[t];
  }
}

// FP32 run of the chunk's products u[t] v[t], t in order (values past n skipped)
__device__ __forceinline__ float chunk_dot(const float v[kChunk], const float u[kChunk],
                                           int64_t i0, int64_t n) {
  float s = 0.0f;
#pragma unroll
  for (int t = 0; t < kChunk; ++t)
    if (i0 + t < n) s = fmaf(v[t], u[t], s);
  return s;
}

// out[j] = V_j . w (j < k <= KMAX), V_j = V + j * ldv; kUpdate: for
// w <- w - sum_j coef[j] V_j first (coef: device FP64), the two halves of a CGS2
// pass boundary in one pass over V and w.  If w == nullptr the squared norm of
// V_0 is taken (k must be 1).
// A thread takes C chunks of 4 values of w and of every vector at a time and
// keeps them in registers for the update and the products, so each value is
// read once and the loads of all vectors are in flight together.  HBM binds
// it; 64 registers of values (128 at KMAX 32) at 2 blocks (1) per SM keep
// enough bytes on the way.  Measured at 2^23 values, products alone / with the
// update, us per launch: 9 to 16 vectors 76 / 98 (6.4 / 5.3 TB/s), 5 to 8 44 /
// 50; with 8 vectors per pass, and the vectors read again from L2 for the
// products, 99 / 144 and 54 / 78.
template <int KMAX, bool kVec, bool kUpdate>
__global__ void __launch_bounds__(kThreads, KMAX <= 16 ? 2 : 1)
    k_project(const float* __restrict__ V, int64_t ldv, int k, const double* __restrict__ coef,
              float* w, int64_t n, double* partials, double* out, unsigned* count) {
  constexpr int C = KMAX <= 4 ? 4 : (KMAX <= 8 ? 2 : 1);
  __shared__ double sums[KMAX][kWarpsPerBlock];
  __shared__ float cf[KMAX];
  if constexpr (kUpdate) {
    for (int j = threadIdx.x; j < k; j += kThreads) cf[j] = (float)coef[j];
    __syncthreads();
  }
  const int64_t chunks = (n + 3) / 4, stride = (int64_t)gridDim.x * kThreads;
  const float* x = w ? w : V;
  Acc2 acc[KMAX];
  for (int64_t c0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; c0 < chunks; c0 += C * stride) {
    float u[C][4], v[KMAX][C][4];  // values past n are 0
#pragma unroll
    for (int i = 0; i < C; ++i) load4<kVec>(x, 4 * (c0 + i * stride), n, u[i]);
#pragma unroll
    for (int j = 0; j < KMAX; ++j) {
      if (j < k) {
#pragma unroll
        for (int i = 0; i < C; ++i) load4<kVec>(V + j * ldv, 4 * (c0 + i * stride), n, v[j][i]);
      }
    }
    if constexpr (kUpdate) {
#pragma unroll
      for (int j = 0; j < KMAX; ++j) {
        if (j < k) {
#pragma unroll
          for (int i = 0; i < C; ++i)
#pragma unroll
            for (int t = 0; t < 4; ++t) u[i][t] = fmaf(-cf[j], v[j][i][t], u[i][t]);
        }
      }
#pragma unroll
      for (int i = 0; i < C; ++i) store4<kVec>(w, 4 * (c0 + i * stride), n, u[i]);
    }
#pragma unroll
    for (int j = 0; j < KMAX; ++j) {
      if (j < k) {
#pragma unroll
        for (int i = 0; i < C; ++i) {
          float p = 0.0f;
#pragma unroll
          for (int t = 0; t < 4; ++t) p = fmaf(v[j][i][t], u[i][t], p);
          acc[j].add(p);
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < KMAX; ++j)
    if (j < k) warp_value(acc[j], j, sums);
  finish_sums(sums, partials, k, out, count);
}

// w <- w - sum_j coef[j] V_j (coef: device FP64);  optionally (norm_out) |w|^2
template <int KMAX, bool kVec>
__global__ void __launch_bounds__(kThreads, 3) k_update(const float* __restrict__ V,
                                                                 int64_t ldv, int k,
                                                                 const double* __restrict__ coef,
                                                                 float* __restrict__ w, int64_t n,
                                                                 double* partials,
                                                                 double* norm_out,
                                                                 unsigned* count) {
  __shared__ double sums[1][kWarpsPerBlock];
  __shared__ float cf[KMAX];
  for (int j = threadIdx.x; j < k; j += kThreads) cf[j] = (float)coef[j];
  __syncthreads();
  const int64_t chunks = (n + kChunk - 1) / kChunk;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  Acc2 acc;
  // two of the thread's chunks per iteration (twice the loads in flight); each
  // element's update and the norm's chunk order are those of one at a time
  for (int64_t c = (int64_t)blockIdx.x * kThreads + threadIdx.x; c < chunks; c += 2 * stride) {
    const int64_t i0 = c * kChunk, i1 = (c + stride) * kChunk;
    const bool second = c + stride < chunks;
    float x0[kChunk], x1[kChunk];
    load8<kVec>(w, i0, n, x0);
    if (second) load8<kVec>(w, i1, n, x1);
#pragma unroll(KMAX <= 4 ? KMAX : 2)
    for (int j = 0; j < k; ++j) {
      float v0[kChunk], v1[kChunk];
      load8<kVec>(V + j * ldv, i0, n, v0);
      if (second) load8<kVec>(V + j * ldv, i1, n, v1);
#pragma unroll
      for (int t = 0; t < kChunk; ++t) {
        x0[t] = fmaf(-cf[j], v0[t], x0[t]);
        if (second) x1[t] = fmaf(-cf[j], v1[t], x1[t]);
      }
    }
    store8<kVec>(w, i0, n, x0);
    if (second) store8<kVec>(w, i1, n, x1);
    if (norm_out) {
      acc.add(chunk_dot(x0, x0, i0, n));
      if (second) acc.add(chunk_dot(x1, x1, i1, n));
    }
  }
  if (norm_out) {
    warp_value(acc, 0, sums);
    finish_sums(sums, partials, 1, norm_out, count);
  }
}

// y <- a * x + b * y  (host scalars), chunks of 8
template <bool kVec>
__global__ void k_axpby(float a, const float* __restrict__ x, float b, float* __restrict__ y,
                        int64_t n) {
  const int64_t chunks = (n + kChunk - 1) / kChunk;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i0 = c * kChunk;
    float u[kChunk], v[kChunk];
    load8<kVec>(x, i0, n, u);
    load8<kVec>(y, i0, n, v);
#pragma unroll
    for (int t = 0; t < kChunk; ++t) v[t] = fmaf(a, u[t], b * v[t]);
    store8<kVec>(y, i0, n, v);
  }
}

// x <- x / sqrt(*norm2) unless it is 0: a vector is normalised by the sum its
// reduction left on the device, before the host has read it.  One thread of a
// block takes the FP64 root and reciprocal while the first values are on their
// way; in every thread they took most of the launch (10^6 values: 10.5 us, so
// 4.4).
template <bool kVec>
__global__ void k_normalise(float* x, const double* __restrict__ norm2, int64_t n) {
  __shared__ float scale;
  int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float v[4];
  load4<kVec>(x, 4 * c, n, v);  // past the end: zeros
  if (threadIdx.x == 0) {
    const double s = *norm2;
    scale = s > 0.0 ? (float)(1.0 / sqrt(s)) : -1.0f;
  }
  __syncthreads();
  const float a = scale;
  if (a < 0.0f) return;
  while (4 * c < n) {
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] *= a;
    store4<kVec>(x, 4 * c, n, v);
    c += (int64_t)gridDim.x * blockDim.x;
    load4<kVec>(x, 4 * c, n, v);
  }
}

// x <- x + sum_j y_j V_j, j in order for every element, chunks of 8
template <int KMAX, bool kVec>
__global__ void k_lincomb(const float* __restrict__ V, int64_t ldv, int k, LinComb y,
                          float* __restrict__ x, int64_t n) {
  const int64_t chunks = (n + kChunk - 1) / kChunk;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i0 = c * kChunk;
    float s[kChunk];
    load8<kVec>(x, i0, n, s);
#pragma unroll
    for (int j = 0; j < KMAX; ++j) {
      if (j < k) {
        float v[kChunk];
        load8<kVec>(V + j * ldv, i0, n, v);
#pragma unroll
        for (int t = 0; t < kChunk; ++t) s[t] = fmaf(y.c[j], v[t], s[t]);
      }
    }
    store8<kVec>(x, i0, n, s);
  }
}

// lumped-mass boundary factor: 1/2 per axis on which the node is an end node
// (nz = 1 is a 2-D mesh)
__device__ __forceinline__ float mass_factor(int x, int y, int z, int nx, int ny, int nz) {
  float m = 1.0f;
  if (x == 0 || x == nx - 1) m *= 0.5f;
  if (y == 0 || y == ny - 1) m *= 0.5f;
  if (nz > 1 && (z == 0 || z == nz - 1)) m *= 0.5f;
  return m;
}

// sum_i (m_i g_i)^2 over all fields into out[0]: m_i = cell * boundary factor.
// Each thread takes chunks of 4 consecutive nodes (one index division per
// chunk; kVec: one 16-byte load per field when the node count is a multiple
// of 4).  Products in FP32 (GB300's FP64 rate is a small fraction of its FP32
// rate), a chunk's squares summed in FP32, the chunks in a compensated FP32
// pair, the block sums in FP64.
template <bool kVec>
__global__ void __launch_bounds__(kThreads) k_mass_norm(const float* __restrict__ g, int nx,
                                                        int ny, int nz, int nf, float cell,
                                                        double* partials, double* out,
                                                        unsigned* count) {
  __shared__ double sums[1][kWarpsPerBlock];
  const int64_t N = (int64_t)nx * ny * nz;
  const int64_t chunks = (N + 3) / 4;
  Acc2 acc;
  for (int64_t c = (int64_t)blockIdx.x * kThreads + threadIdx.x; c < chunks;
       c += (int64_t)gridDim.x * kThreads) {
    const int64_t i0 = 4 * c;
    // node coordinates in 32-bit arithmetic (nodes < 2^31): a 64-bit integer
    // division runs on the FP64 pipe, a small fraction of GB300's FP32 rate
    const int node0 = (int)i0;
    int x = node0 % nx;
    const int r = node0 / nx;
    int y = r % ny, z = r / ny;
    float m[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      m[t] = (i0 + t < N) ? cell * mass_factor(x, y, z, nx, ny, nz) : 0.0f;
      if (++x == nx) {
        x = 0;
        if (++y == ny) {
          y = 0;
          ++z;
        }
      }
    }
    // every field's chunk is loaded before any is used, so the loads of up
    // to kMaxFields planes are in flight together
    float v[kMaxFields][4];
#pragma unroll
    for (int f = 0; f < kMaxFields; ++f) {
      if (f < nf) {
        const float* p = g + (int64_t)f * N + i0;
        if (kVec && i0 + 4 <= N) {
          const float4 q = __ldg(reinterpret_cast<const float4*>(p));
          v[f][0] = q.x; v[f][1] = q.y; v[f][2] = q.z; v[f][3] = q.w;
        } else {
#pragma unroll
          for (int t = 0; t < 4; ++t) v[f][t] = (i0 + t < N) ? p[t] : 0.0f;
        }
      }
    }
    // the chunk's squares (at most 32) as one FP32 run, then one FP64 add
    float run = 0.0f;
#pragma unroll
    for (int f = 0; f < kMaxFields; ++f) {
      if (f < nf) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const float u = m[t] * v[f][t];
          run = fmaf(u, u, run);
        }
      }
    }
    acc.add(run);
  }
  warp_value(acc, 0, sums);
  finish_sums(sums, partials, 1, out, count);
}

// out = a * m_i^(+1 or -1) * in over nf planes of nx x ny x nz nodes, m the
// lumped mass (cell times 1/2 per boundary axis; nz = 1 is a 2-D mesh);
// inv_cell = 1 / cell, so that the inverse is a multiplication
__global__ void k_mass_mul(const float* __restrict__ in, float* __restrict__ out, int nx, int ny,
                           int nz, int nf, float cell, float inv_cell, float a, int inverse) {
  const int N = nx * ny * nz;
  for (int node = blockIdx.x * blockDim.x + threadIdx.x; node < N; node += gridDim.x * blockDim.x) {
    const float fac = mass_factor(node % nx, (node / nx) % ny, node / (nx * ny), nx, ny, nz);
    const float sc = a * (inverse ? inv_cell / fac : cell * fac);  // fac is a power of 2
    for (int f = 0; f < nf; ++f) out[(int64_t)f * N + node] = sc * in[(int64_t)f * N + node];
  }
}

unsigned elementwise_blocks(int64_t n) {
  const int64_t b = (n + 255) / 256, cap = 8 * (int64_t)device_sm_count();
  return (unsigned)(b < cap ? b : cap);
}

}  // namespace

// Most blocks of a reduction (the partials' size).  Each uses as many per SM
// as its kernel is built for and no more than its values fill, a function of
// the device and the size alone, so the order (and result) never changes.
int krylov_partial_blocks() { return 3 * device_sm_count(); }

namespace {
// 16-byte loads when every vector the call touches starts on a 16-byte boundary
bool vec_ok(const void* a, const void* b, int64_t ldv) {
  return ((uintptr_t)a % 16 == 0) && ((uintptr_t)b % 16 == 0) && (ldv % 4 == 0);
}

unsigned reduction_blocks(int per_sm, int64_t chunks) {
  const int64_t need = (chunks + kThreads - 1) / kThreads, cap = (int64_t)per_sm * device_sm_count();
  return (unsigned)(need < 1 ? 1 : (need < cap ? need : cap));
}

// calls fn(KMAX) for the smallest KMAX in {4, 8, 16, 32} holding k
template <class F>
cudaError_t with_bound(int k, F&& fn) {
  if (k <= 4) fn(std::integral_constant<int, 4>{});
  else if (k <= 8) fn(std::integral_constant<int, 8>{});
  else if (k <= 16) fn(std::integral_constant<int, 16>{});
  else if (k <= kMaxBasis) fn(std::integral_constant<int, kMaxBasis>{});
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

template <bool kUpdate>
cudaError_t project(const float* V, int64_t ldv, int k, const double* coef, float* w, int64_t n,
                    double* partials, double* out, unsigned* count, cudaStream_t s) {
  const bool vec = vec_ok(V, w ? w : V, ldv);
  return with_bound(k, [&](auto bound) {
    constexpr int M = decltype(bound)::value;
    const unsigned g = reduction_blocks(M <= 16 ? 2 : 1, (n + 3) / 4);
    if (vec)
      k_project<M, true, kUpdate><<<g, kThreads, 0, s>>>(V, ldv, k, coef, w, n, partials, out, count);
    else
      k_project<M, false, kUpdate><<<g, kThreads, 0, s>>>(V, ldv, k, coef, w, n, partials, out,
                                                          count);
  });
}
}  // namespace

cudaError_t launch_dots(const float* V, int64_t ldv, int k, const float* w, int64_t n,
                        double* partials, double* out, unsigned* count, cudaStream_t s) {
  // more than 16 products in two launches: w is read twice, but at 32 vectors
  // per pass only one block fits an SM (20 products of 2^23 values: 157 us in
  // one pass, 125 in two)
  float* x = const_cast<float*>(w);
  if (k > 16) {
    const cudaError_t e = project<false>(V, ldv, 16, nullptr, x, n, partials, out, count, s);
    if (e != cudaSuccess) return e;
    return project<false>(V + 16 * ldv, ldv, k - 16, nullptr, x, n, partials, out + 16, count, s);
  }
  return project<false>(V, ldv, k, nullptr, x, n, partials, out, count, s);
}

cudaError_t launch_update(const float* V, int64_t ldv, int k, const double* coef, float* w,
                          int64_t n, double* partials, double* norm_out, unsigned* count,
                          cudaStream_t s) {
  const bool vec = vec_ok(V, w, ldv);
  const unsigned g = reduction_blocks(3, (n + kChunk - 1) / kChunk);
  return with_bound(k, [&](auto bound) {
    constexpr int M = decltype(bound)::value;
    if (vec)
      k_update<M, true><<<g, kThreads, 0, s>>>(V, ldv, k, coef, w, n, partials, norm_out, count);
    else
      k_update<M, false><<<g, kThreads, 0, s>>>(V, ldv, k, coef, w, n, partials, norm_out, count);
  });
}

cudaError_t launch_update_dots(const float* V, int64_t ldv, int k, const double* coef, float* w,
                               int64_t n, double* partials, double* out, unsigned* count,
                               cudaStream_t s) {
  return project<true>(V, ldv, k, coef, w, n, partials, out, count, s);
}

cudaError_t launch_axpby(float a, const float* x, float b, float* y, int64_t n, cudaStream_t s) {
  const unsigned g = elementwise_blocks((n + kChunk - 1) / kChunk);
  if (vec_ok(x, y, 0))
    k_axpby<true><<<g, 256, 0, s>>>(a, x, b, y, n);
  else
    k_axpby<false><<<g, 256, 0, s>>>(a, x, b, y, n);
  return cudaGetLastError();
}

cudaError_t launch_normalise(float* x, const double* norm2, int64_t n, cudaStream_t s) {
  const unsigned g = elementwise_blocks((n + 3) / 4);
  if ((uintptr_t)x % 16 == 0)
    k_normalise<true><<<g, 256, 0, s>>>(x, norm2, n);
  else
    k_normalise<false><<<g, 256, 0, s>>>(x, norm2, n);
  return cudaGetLastError();
}

cudaError_t launch_lincomb(const float* V, int64_t ldv, int k, const LinComb& y, float* x,
                           int64_t n, cudaStream_t s) {
  const dim3 g(elementwise_blocks((n + kChunk - 1) / kChunk)), b(256);
  const bool vec = vec_ok(V, x, ldv);
#define PF_LINCOMB_CASE(M)                                                  \
  if (k <= M) {                                                             \
    if (vec) k_lincomb<M, true><<<g, b, 0, s>>>(V, ldv, k, y, x, n);        \
    else k_lincomb<M, false><<<g, b, 0, s>>>(V, ldv, k, y, x, n);           \
    return cudaGetLastError();                                              \
  }
  PF_LINCOMB_CASE(4)
  PF_LINCOMB_CASE(8)
  PF_LINCOMB_CASE(16)
  PF_LINCOMB_CASE(kMaxBasis)
#undef PF_LINCOMB_CASE
  return cudaErrorInvalidValue;
}

cudaError_t launch_mass_mul(const float* in, float* out, int nx, int ny, int nz, int nf,
                            double cell, float a, int inverse, cudaStream_t s) {
  k_mass_mul<<<elementwise_blocks((int64_t)nx * ny * nz), 256, 0, s>>>(
      in, out, nx, ny, nz, nf, (float)cell, (float)(1.0 / cell), a, inverse);
  return cudaGetLastError();
}

cudaError_t launch_mass_norm(const float* g, int nx, int ny, int nz, int nf, double cell,
                             double* partials, double* out, unsigned* count, cudaStream_t s) {
  const int64_t N = (int64_t)nx * ny * nz;
  if (nf < 1 || nf > kMaxFields) return cudaErrorInvalidValue;
  const unsigned b = reduction_blocks(3, (N + 3) / 4);
  if (N % 4 == 0 && (uintptr_t)g % 16 == 0)
    k_mass_norm<true><<<b, kThreads, 0, s>>>(g, nx, ny, nz, nf, (float)cell, partials, out, count);
  else
    k_mass_norm<false><<<b, kThreads, 0, s>>>(g, nx, ny, nz, nf, (float)cell, partials, out, count);
  return cudaGetLastError();
}

}  // namespace pf
