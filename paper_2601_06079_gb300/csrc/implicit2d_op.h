// The 2-D implicit operators on one node tile (k_implicit2d.cu: one block per
// tile; k_newton2d.cu: a resident grid).
#pragma once

#include "pf_internal.h"

namespace pf {
namespace implicit2d {

constexpr int TX = 32, TY = 16;            // output tile
constexpr int SX = TX + 2, SY = TY + 2;    // nodes with a 1-node halo
constexpr int EX = TX + 1, EY = TY + 1;    // elements touching the tile nodes

// Mirror image of node index k on an axis of n nodes (period 2(n-1)).  Halo
// indices lie within one period of the axis, where a reflection at each end
// gives the image without the integer division.
__device__ __forceinline__ int mirror(int k, int n) {
  const int p = 2 * (n - 1);
  if (k >= 1 - n && k <= p) return k < 0 ? -k : (k < n ? k : p - k);
  k %= p;
  if (k < 0) k += p;
  return k < n ? k : p - k;
}

__device__ __forceinline__ float gpt(int i) { return i ? kGHi : kGLo; }

// 9-point stencil s at node (y, x) of a staged plane.  The Q1 stiffness rows
// sum to zero (c0 = -2 cx - 2 cy - 4 cd), so K v is applied to the differences
// v_j - v_i: for smooth fields each difference of neighbouring FP32 values is
// exact, where c0 v_i + sum c_j v_j would cancel to a few significant bits.
template <int W_>
__device__ __forceinline__ float stencil(const float (*V)[W_], int y, int x, const Stencil2D& k) {
  const float c = V[y][x];
  return k.cx * ((V[y][x - 1] - c) + (V[y][x + 1] - c)) +
         k.cy * ((V[y - 1][x] - c) + (V[y + 1][x] - c)) +
         k.cd * (((V[y - 1][x - 1] - c) + (V[y - 1][x + 1] - c)) +
                 ((V[y + 1][x - 1] - c) + (V[y + 1][x + 1] - c)));
}

// Staged planes: U (Allen-Cahn) or c; U^n / v or c^n / v_c; Cahn-Hilliard: mu
// (residual) or v_mu (JVP); the elements' corner contributions.
template <bool kCH>
struct TileMem {
  float U[SY][SX], W[SY][SX], M[kCH ? SY : 1][kCH ? SX : 1];
  float E[4][EY][EX];
};

// kCoherent: U and W are written by other blocks of the same launch and are
// read through L2.  put(node, x, y, o0, o1): the scaled result (M^-1 R, M^-1 J v)
// at a node, o1 for Cahn-Hilliard's second plane.
template <bool kJVP, bool kCH, int kThreads, bool kCoherent, class Put>
__device__ __forceinline__ void tile_operator(const Implicit2DArgs& a, int tile, TileMem<kCH>& m,
                                              Put&& put) {
  const int tiles_x = (a.nx + TX - 1) / TX;
  const int x0 = (tile % tiles_x) * TX, y0 = (tile / tiles_x) * TY;
  const int64_t N = (int64_t)a.nx * a.ny;
  const auto ld = [](const float* p) { return kCoherent ? __ldcg(p) : *p; };

  for (int i = threadIdx.x; i < SX * SY; i += kThreads) {
    const int lx = i % SX, ly = i / SX;
    const int64_t g = (int64_t)mirror(y0 - 1 + ly, a.ny) * a.nx + mirror(x0 - 1 + lx, a.nx);
    m.U[ly][lx] = ld(a.U + g);
    m.W[ly][lx] = ld(a.W + g);
    if (kCH) m.M[ly][lx] = kJVP ? ld(a.W + N + g) : ld(a.U + N + g);
  }
  __syncthreads();

  // element (ey, ex) has lower-left node (ey, ex) in halo coordinates
  for (int i = threadIdx.x; i < EX * EY; i += kThreads) {
    const int ex = i % EX, ey = i / EX;
    const float u[4] = {m.U[ey][ex], m.U[ey][ex + 1], m.U[ey + 1][ex], m.U[ey + 1][ex + 1]};
    const float v[4] = {m.W[ey][ex], m.W[ey][ex + 1], m.W[ey + 1][ex], m.W[ey + 1][ex + 1]};
    float t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float xi = gpt(q & 1), et = gpt(q >> 1);
      const float ub = fmaf(xi, u[1] - u[0], u[0]), ut = fmaf(xi, u[3] - u[2], u[2]);
      const float uq = fmaf(et, ut - ub, ub);
      if (kJVP) {
        const float vb = fmaf(xi, v[1] - v[0], v[0]), vt = fmaf(xi, v[3] - v[2], v[2]);
        const float vq = fmaf(et, vt - vb, vb);
        // f''(u) = 2W (1 - 6u + 6u^2)
        t[q] = a.dw2 * fmaf(6.0f * uq, uq - 1.0f, 1.0f) * vq;
      } else {
        // f'(u) = 2W u (1-u)(1-2u)
        t[q] = a.dw2 * uq * (1.0f - uq) * (1.0f - 2.0f * uq);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float s = 0.0f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float xi = gpt(q & 1), et = gpt(q >> 1);
        s = fmaf(t[q], ((c & 1) ? xi : 1.0f - xi) * ((c >> 1) ? et : 1.0f - et), s);
      }
      m.E[c][ey][ex] = 0.25f * s;  // Gauss weight |cell|/4 over the interior mass |cell|
    }
  }
  __syncthreads();

  for (int i = threadIdx.x; i < TX * TY; i += kThreads) {
    const int lx = i % TX, ly = i / TX;
    const int gx = x0 + lx, gy = y0 + ly;
    if (gx >= a.nx || gy >= a.ny) continue;
    const int x = lx + 1, y = ly + 1;
    const float acc = m.E[0][y][x] + m.E[1][y][x - 1] + m.E[2][y - 1][x] + m.E[3][y - 1][x - 1];
    const float (*V)[SX] = kJVP ? m.W : m.U;  // the stiffness acts on v (JVP) or U (residual)
    const float ks = stencil(V, y, x, a.k);
    const float own = kJVP ? m.W[y][x] : (m.U[y][x] - m.W[y][x]);
    const int64_t o = (int64_t)gy * a.nx + gx;
    if constexpr (kCH)
      // c row: own / dt + M_c m^-1 K (mu or v_mu);  mu row: (mu or v_mu) - m^-1 (r or H v_c)
      put(o, gx, gy, fmaf(own, a.inv_dt, stencil(m.M, y, x, a.km)), m.M[y][x] - (acc + ks));
    else
      put(o, gx, gy, fmaf(own, a.inv_dt, a.mob * (acc + ks)), 0.0f);
  }
}

}  // namespace implicit2d
}  // namespace pf
