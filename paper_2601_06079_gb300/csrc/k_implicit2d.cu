// 2-D implicit-step operators (JAX-PF Eq. 13-14 on a 2-D Q1 mesh) with the
// double well f = W u^2 (1-u)^2, r the gradient and H the Hessian of
// E_h = sum_e sum_q w|J| [f(U_q) + kappa/2 |grad U_q|^2]:
//   Allen-Cahn:  R(U) = M (U - U^n)/dt + L r(U),     J v = M v / dt + L H(U) v
//   split Cahn-Hilliard (Eq. 9-10), unknowns [c; mu]:
//                R = [M (c - c^n)/dt + K_M mu;  M mu - r(c)]
//                J [v_c; v_mu] = [M v_c / dt + K_M v_mu;  M v_mu - H(c) v_c]
// As in 3-D all are evaluated scaled by the lumped mass (M^-1 R, M^-1 J v) on
// a tile with mirror images beyond the mesh, where every node uses the
// interior formula; an optional final multiplication by m_i gives R and J v
// themselves.
//
// One block per 32 x 16 node tile: U and v (or U^n) are staged with a 1-node
// halo; every element touching the tile evaluates f'(u_q) (residual) or
// f''(u_q) v_q (JVP) at its 2x2 Gauss points and projects it to its corners;
// a node-centric gather of the 4 element contributions plus the assembled
// 9-point stiffness stencil gives the output.  No atomics.
#include "implicit2d_op.h"
#include "pf_internal.h"

namespace pf {
namespace {

using namespace implicit2d;

constexpr int kThreads = 256;

template <bool kJVP, bool kCH>
__global__ void __launch_bounds__(kThreads) k_implicit2d(const Implicit2DArgs a) {
  __shared__ TileMem<kCH> m;
  const int64_t N = (int64_t)a.nx * a.ny;
  tile_operator<kJVP, kCH, kThreads, false>(
      a, blockIdx.x, m, [&](int64_t o, int gx, int gy, float o0, float o1) {
        float wm = 1.0f;
        if (a.unscaled) {
          const float wx = (gx == 0 || gx == a.nx - 1) ? 0.5f : 1.0f;
          const float wy = (gy == 0 || gy == a.ny - 1) ? 0.5f : 1.0f;
          wm = a.cell * wx * wy;
        }
        a.out[o] = wm * o0;
        if (kCH) a.out[N + o] = wm * o1;
      });
}

}  // namespace

cudaError_t launch_residual2d(const Implicit2DArgs& a, cudaStream_t s) {
  const int tiles = ((a.nx + TX - 1) / TX) * ((a.ny + TY - 1) / TY);
  if (a.ch)
    k_implicit2d<false, true><<<tiles, kThreads, 0, s>>>(a);
  else
    k_implicit2d<false, false><<<tiles, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_jvp2d(const Implicit2DArgs& a, cudaStream_t s) {
  const int tiles = ((a.nx + TX - 1) / TX) * ((a.ny + TY - 1) / TY);
  if (a.ch)
    k_implicit2d<true, true><<<tiles, kThreads, 0, s>>>(a);
  else
    k_implicit2d<true, false><<<tiles, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace pf
