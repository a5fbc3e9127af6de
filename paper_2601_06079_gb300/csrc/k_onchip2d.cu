// Explicit 2-D trajectories with the state held on chip: one cooperative
// launch advances a mesh (or an ensemble's instances) by all its steps.  Every
// block keeps one tile of the state in shared memory from the first step to
// the last; only the tiles' edges travel between blocks, through L2.
//
// What it is for.  One launch per step costs about 3 us of launch, ramp and
// drain whatever the mesh, re-reads and re-writes every plane, and repeats the
// warm-up rows of 6-row bands (4 rows more for Cahn-Hilliard).  Here a tile is
// one warp strip wide (sweep2d.h: kP pairs of columns per lane) and as tall as
// the mesh and the number of blocks make it; the block's warps split its rows.
// The arithmetic and its order are those of k_explicit2d, so the results are
// bitwise the same.
//
// A step of a block:
//   1. every warp takes the rows around its band that other warps own into
//      its window and a buffer of its own (two above, two below; one each for
//      Allen-Cahn); block barrier;
//   2. the warps sweep their bands and write the finished rows in place (a row
//      is written after the sweep has read the rows that need it); barrier.
// A tile carries a halo of 4 rows and columns (the strip's outermost lanes),
// which lasts kSteps = 2 steps of Cahn-Hilliard or 4 of Allen-Cahn: a step also
// advances the part of the halo that the remaining steps need.  Then
//   3. by tables made once, the threads write the edges that neighbouring tiles
//      need to the exchange buffer and fill the halo: the neighbours' edges,
//      polled, and mirror images beyond the mesh (the arithmetic is mirror
//      symmetric to the last bit, so the images advance like any node).
// The exact form (Allen-Cahn ensembles and small meshes) has no halo lanes: a
// strip is 64 kP columns, all of them output, and the halo of one row and
// column is refreshed after every step; it takes the share that lane 0 needs of
// the elements left of the strip from a column pass before the sweep.
//
// An edge travels as packets of two values (packet.h), the tag being the
// exchange's number: a reader polls the packet itself until both tags match.  Two slots alternate: a
// block writes slot x+2 only after reading its neighbours' exchange x+1, which
// they publish after reading x.  Tags start from a zeroed buffer in every
// launch.  Every wait is bounded; when one runs out the error flag is set,
// and the blocks that wait, or come to, leave and write NaN over their tiles (one
// that has all its packets by then stores what it has: the flag is the report).
#include <algorithm>
#include <functional>
#include <queue>
#include <type_traits>

#include "packet.h"
#include "pf_internal.h"
#include "sweep2d.h"

namespace pf {
namespace {

using namespace sweep;

constexpr int kMaxSmem = 227 * 1024;
constexpr int kBatch = 4;     // packets that a thread polls at a time
constexpr int kMaxBand = 30;  // rows per warp: the edge column of a band fits one warp

// kHalo: columns and rows of the halo (2 or 4), or 1 for the exact form.
template <bool kCH, int kP, int kHalo>
struct Geo {
  static constexpr bool kExact = kHalo == 1;
  static constexpr int kRows = kHalo;                             // halo rows per side
  static constexpr int kEdge = kExact ? 2 : kHalo;                // halo columns per side
  static constexpr int kSteps = kCH ? kHalo / 2 : kHalo;          // steps per exchange
  static constexpr int kOff = kExact ? 4 : kHalo;                 // storage column of column 0
  // storage columns; 4 or 8 more than a multiple of 32, so that the lanes of a
  // column access fall on 8 or 4 groups of banks
  static constexpr int kPitch = 64 * kP + (kExact ? 8 : 4);
  static constexpr int kCols = kExact ? 64 * kP : 64 * kP - 2 * kHalo;  // widest tile
  static constexpr int kPairs = 32 * kP;                          // packets of a tile row
};

// Tile (i, j) of the gx x gy tiles of a mesh: columns in pairs, split evenly.
struct Tile {
  int x0, y0, w, h;
};
__host__ __device__ inline Tile tile_of(const OnchipJob& b, int i, int j) {
  const int64_t np = (b.nx + 1) / 2;
  Tile t;
  t.x0 = (int)(2 * (i * np / b.gx));
  t.w = (i == b.gx - 1 ? b.nx : (int)(2 * ((i + 1) * np / b.gx))) - t.x0;
  t.y0 = (int)((int64_t)j * b.ny / b.gy);
  t.h = (int)((int64_t)(j + 1) * b.ny / b.gy) - t.y0;
  return t;
}
__host__ __device__ inline int tallest(const OnchipJob& b) { return (b.ny + b.gy - 1) / b.gy; }

// Exchange region of a tile, in packets: two slots of
// [top rows | bottom rows | left column pairs | right column pairs].
template <class G>
__host__ __device__ inline int slot_packets(int hmax) {
  return 2 * G::kRows * G::kPairs + G::kEdge * hmax;
}

__device__ __forceinline__ int reflect(int k, int n) {
  const int p = 2 * (n - 1);
  k %= p;
  if (k < 0) k += p;
  return k < n ? k : p - k;
}

// One or two halo cells: where they come from and go to.
enum Kind : unsigned {
  kPair = 0,   // src: a neighbour's packet (of the job's region, slot 0), both halves
  kFirst = 1,  // its first or second half only
  kSecond = 2,
  kImages = 3,  // src: storage indices of two cells of this tile, 16 bits each
  kImage = 4    // of one cell
};
struct Fetch {
  unsigned src, dst;  // dst: storage index, kind << 16
};
// One pair that a neighbour needs: its storage index and its packet in slot 0.
struct Send {
  unsigned cell, packet;
};
// entries of both tables for a w x h tile (the fetch table holds up to two
// entries for a pair of the corners and of an odd width's last column)
template <class G>
__host__ __device__ inline int fetch_entries(int w, int h) {
  return 2 * G::kRows * ((w + 1) / 2 + 2 * G::kEdge + 4) + (G::kEdge + 2) * h;
}
template <class G>
__host__ __device__ inline int send_entries(int w, int h) {
  return 2 * G::kRows * ((w + 1) / 2) + G::kEdge * h;
}

// Source of halo cell (y, x) of tile (ti, tj): an entry without its
// destination, kind in dst; false for a cell of the tile itself.
template <class G>
__device__ bool source(const OnchipJob& b, int ti, int tj, const Tile& t, int hmax, int y, int x,
                       Fetch* f) {
  if (y >= 0 && y < t.h && x >= 0 && x < t.w) return false;
  const int Y = reflect(t.y0 + y, b.ny), X = reflect(t.x0 + x, b.nx);
  const int j = Y < t.y0 ? tj - 1 : (Y >= t.y0 + t.h ? tj + 1 : tj);
  const int i = X < t.x0 ? ti - 1 : (X >= t.x0 + t.w ? ti + 1 : ti);
  if (i == ti && j == tj) {
    f->src = (unsigned)((Y - t.y0 + G::kRows) * G::kPitch + G::kOff + X - t.x0);
    f->dst = kImage;
    return true;
  }
  const Tile n = tile_of(b, i, j);
  const int ry = Y - n.y0, rx = X - n.x0;
  int off;
  if (j < tj)
    off = (G::kRows + ry - (n.h - G::kRows)) * G::kPairs + rx / 2;  // their bottom rows
  else if (j > tj)
    off = ry * G::kPairs + rx / 2;
  else if (i < ti)  // their right columns
    off = 2 * G::kRows * G::kPairs + (G::kEdge / 2 + (rx - (n.w - G::kEdge)) / 2) * hmax + ry;
  else
    off = 2 * G::kRows * G::kPairs + rx / 2 * hmax + ry;
  f->src = (unsigned)(2 * slot_packets<G>(hmax) * (j * b.gx + i) + off);
  f->dst = rx & 1 ? kSecond : kFirst;
  return true;
}

template <bool kCH, bool kIso, bool kOdd, int kP, int kWarps, int kBlocks, int kHalo, bool kEns>
__global__ void __launch_bounds__(32 * kWarps, kBlocks)
    k_onchip2d(const __grid_constant__ OnchipArgs a) {
  using G = Geo<kCH, kP, kHalo>;
  constexpr bool kExact = G::kExact;
  constexpr int H = kCH ? 2 : 1;  // rows that a step reads beyond the one it finishes
  constexpr int HR = G::kRows, kPitch = G::kPitch, kOff = G::kOff, kThreads = 32 * kWarps;
  extern __shared__ __align__(16) float smem[];
  __shared__ int s_abort, s_nfetch, s_nsend;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // this lane's first column (tile-relative; negative in a halo lane)
  const int xl = kExact ? 2 * kP * lane : 2 * kP * lane - kHalo;
  // exact form: the column beyond the strip on this lane's side, from xl
  const int edge = (lane == 31 ? 64 * kP : -1) - xl;
  // the rows below each warp's band (step 1), then the tile
  float* const below = smem + warp * H * kPitch + kOff + xl;
  float* const store = smem + kWarps * H * kPitch;
  float* const mine = store + kOff + xl;

  const int first = kEns ? a.list_first[blockIdx.x] : 0;
  const int last = kEns ? a.list_first[blockIdx.x + 1] : 1;
  for (int item = first; item < last; ++item) {
    const OnchipJob* jp = &a.job;
    int tile = blockIdx.x;
    if constexpr (kEns) {
      jp = a.jobs + a.list[item].job;
      tile = a.list[item].tile;
    }
    const OnchipJob& b = *jp;
    u64 kc[19];
    Coef K{b.pair};
    if constexpr (kEns) {
#pragma unroll
      for (int i = 0; i < 19; ++i) kc[i] = b.pair[i];
      K.c = kc;
    }
    const int ti = tile % b.gx, tj = tile / b.gx;
    const Tile t = tile_of(b, ti, tj);
    const int w = t.w, h = t.h, hmax = tallest(b);
    const float shift = b.shift;
    float* const state = a.state + b.off;
    const int slot = slot_packets<G>(hmax);
    Packet* const region = static_cast<Packet*>(a.xchg) + b.xchg;
    Packet* const own = region + (int64_t)2 * slot * tile;
    Fetch* const fetch = reinterpret_cast<Fetch*>(store + (size_t)(hmax + 2 * HR) * kPitch);
    Send* const send = reinterpret_cast<Send*>(fetch + fetch_entries<G>(w, hmax));

    if (threadIdx.x == 0) s_abort = s_nfetch = s_nsend = 0;
    // the tile and its halo, images beyond the mesh; columns past the halo
    // hold values that nothing stored depends on
    for (int i = threadIdx.x; i < (h + 2 * HR) * kPitch; i += kThreads) {
      const int y = t.y0 + i / kPitch - HR, x = t.x0 + i % kPitch - kOff;
      store[i] = state[(int64_t)reflect(y, b.ny) * b.nx + reflect(x, b.nx)] - shift;
    }
    __syncthreads();
    // the halo's cells, in pairs of columns from -kEdge on
    const int span = (w + 1) / 2 + G::kEdge;
    for (int i = threadIdx.x; i < (h + 2 * HR) * span; i += kThreads) {
      const int y = i / span - HR, x = 2 * (i % span) - G::kEdge;
      Fetch f[2];
      const bool u0 = source<G>(b, ti, tj, t, hmax, y, x, &f[0]);
      const bool u1 = source<G>(b, ti, tj, t, hmax, y, x + 1, &f[1]);
      const unsigned dst = (unsigned)((y + HR) * kPitch + kOff + x);
      if (u0 && u1 && f[0].dst == kFirst && f[1].dst == kSecond && f[0].src == f[1].src) {
        fetch[atomicAdd(&s_nfetch, 1)] = Fetch{f[0].src, dst | kPair << 16};
      } else if (u0 && u1 && f[0].dst == kImage && f[1].dst == kImage) {
        fetch[atomicAdd(&s_nfetch, 1)] = Fetch{f[0].src | f[1].src << 16, dst | kImages << 16};
      } else {
        if (u0) fetch[atomicAdd(&s_nfetch, 1)] = Fetch{f[0].src, dst | f[0].dst << 16};
        if (u1) fetch[atomicAdd(&s_nfetch, 1)] = Fetch{f[1].src, (dst + 1) | f[1].dst << 16};
      }
    }
    // this tile's rows (top, bottom) and columns (left, right) next to others
    const int pw = (w + 1) / 2, srows = 2 * HR * pw;
    for (int i = threadIdx.x; i < srows + G::kEdge * h; i += kThreads) {
      Send q;
      bool wanted;
      if (i < srows) {
        const int side = i / (HR * pw), r = i / pw % HR, p = i % pw;
        q.cell = (unsigned)(((side ? h - HR + r : r) + HR) * kPitch + kOff + 2 * p);
        q.packet = (unsigned)((side * HR + r) * G::kPairs + p);
        wanted = side ? tj < b.gy - 1 : tj > 0;
      } else {
        const int c = (i - srows) / h, r = (i - srows) % h, side = c / (G::kEdge / 2);
        q.cell = (unsigned)((r + HR) * kPitch + kOff + (side ? w - G::kEdge : 0) +
                            2 * (c % (G::kEdge / 2)));
        q.packet = (unsigned)(2 * HR * G::kPairs + c * hmax + r);
        wanted = side ? ti < b.gx - 1 : ti > 0;
      }
      if (wanted) send[atomicAdd(&s_nsend, 1)] = q;
    }
    __syncthreads();
    const int nfetch = s_nfetch, nsend = s_nsend;

    const auto load = [&](const float* p, u64(&P)[kP], float& e) {
      if constexpr (kP == 2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
        P[0] = v.x;
        P[1] = v.y;
      } else {
        P[0] = *reinterpret_cast<const u64*>(p);
      }
      if constexpr (kExact) e = p[edge];
    };
    const auto put = [&](float* p, const u64(&P)[kP]) {
      if constexpr (kP == 2)
        *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(P[0], P[1]);
      else
        *reinterpret_cast<u64*>(p) = P[0];
    };

    unsigned tag = 0;
    for (int s = 0, ext = 0; s < a.n_steps; ++s, ext -= H) {
      // halo rows that this step still has to advance
      if (s % G::kSteps == 0) ext = (min(G::kSteps, a.n_steps - s) - 1) * H;
      const int rows = h + 2 * ext;
      const int r0 = warp * rows / kWarps - ext, r1 = (warp + 1) * rows / kWarps - ext;
      Window<kP> win;
      u64 o[kP];
      float bcol = 0.0f;
      const auto consume = [&](auto stage, const u64(&P)[kP], float e, float b0) {
        float cl = __shfl_up_sync(kFull, phi(P[kP - 1]), 1);
        float cr = __shfl_down_sync(kFull, plo(P[0]), 1);
        if constexpr (kExact) {
          cl = lane == 0 ? e : cl;
          cr = lane == 31 ? e : cr;
        }
        row<kCH, kIso, kOdd, kP, decltype(stage)::value, kExact>(P, cl, cr, b0, win, K, o);
      };
      if (r0 < r1) {
        u64 P[kP];
        float e = 0.0f;
#pragma unroll
        for (int r = 0; r < H; ++r) {
          load(mine + (r1 + r + HR) * kPitch, P, e);
          put(below + r * kPitch, P);
          if constexpr (kExact) {
            if (lane == 0 || lane == 31) below[r * kPitch + edge] = e;
          }
        }
        if constexpr (kExact) {
          // the weights back in x of the elements left of the strip, lane i
          // for node row r0 - 1 + i: their share of column 0
          const float* q = store + (min(r0 - 1 + lane, r1) + HR) * kPitch + kOff;
          const float u = q[-1], v = q[0], rho = plo(K.rho());
          const u64 m = pk(fmaf(rho, v, u), fmaf(rho, u, v));  // (am, ap) of this row
          const u64 mn = pk(__shfl_down_sync(kFull, plo(m), 1), __shfl_down_sync(kFull, phi(m), 1));
          const u64 fl = well<kOdd>(fma2(K.rho(), mn, m), K);  // (fll, fhl): near this row
          const u64 fh = well<kOdd>(fma2(K.rho(), m, mn), K);
          const u64 tn = fma2(K.rho(), fl, fh);  // element row's share of the next node row
          const u64 tp = pk(__shfl_up_sync(kFull, plo(tn), 1), __shfl_up_sync(kFull, phi(tn), 1));
          const u64 sn = add2(fma2(K.rho(), fh, fl), tp);
          bcol = fmaf(rho, plo(sn), phi(sn));
        }
        load(mine + (r0 - H + HR) * kPitch, P, e);
        consume(std::integral_constant<int, kInterp>{}, P, e, 0.0f);
        if constexpr (kCH) {
          load(mine + (r0 - 1 + HR) * kPitch, P, e);
          consume(std::integral_constant<int, kElement>{}, P, e, 0.0f);
        }
      }
      __syncthreads();
      if (r0 < r1) {
        // rows of the band in place, then the ones kept
        const float* src = mine + (r0 + HR) * kPitch;
        int left = r1 - r0;
        const auto get = [&](u64(&P)[kP], float& e) {
          load(src, P, e);
          src = --left == 0 ? below : src + kPitch;
        };
        u64 P[kP], Q[kP];
        float e = 0.0f, eq = 0.0f;
        get(P, e);
        get(Q, eq);
        consume(std::integral_constant<int, kCH ? kMu : kElement>{}, P, e, 0.0f);
        if constexpr (kCH) {
          get(P, e);
          consume(std::integral_constant<int, kMu>{}, Q, eq, 0.0f);
        } else {
#pragma unroll
          for (int j = 0; j < kP; ++j) P[j] = Q[j];
          e = eq;
        }
        float* dst = mine + (r0 + HR) * kPitch;
#pragma unroll 4
        for (int y = r0; y < r1; ++y) {  // consume row y + H: row y is finished
          get(Q, eq);  // past the last row: not used
          const float b0 = kExact ? __shfl_sync(kFull, bcol, y - r0 + 1) : 0.0f;
          consume(std::integral_constant<int, kOutput>{}, P, e, b0);
          put(dst, o);
          dst += kPitch;
#pragma unroll
          for (int j = 0; j < kP; ++j) P[j] = Q[j];
          e = eq;
        }
      }
      __syncthreads();
      if (ext > 0 || s + 1 == a.n_steps) continue;
      ++tag;
      Packet* const out = own + (tag & 1) * slot;
      for (int i = threadIdx.x; i < nsend; i += kThreads) {
        const Send q = send[i];
        const u64 v = *reinterpret_cast<const u64*>(store + q.cell);
        publish(out + q.packet, __float_as_uint(plo(v)), __float_as_uint(phi(v)), tag);
      }
      const Packet* const in = region + (tag & 1) * slot;
      // kBatch polls of a thread are in flight together
      for (int i = threadIdx.x; i < nfetch; i += kBatch * kThreads) {
        Fetch f[kBatch];
        bool wait[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
          wait[k] = i + k * kThreads < nfetch;
          if (!wait[k]) continue;
          f[k] = fetch[i + k * kThreads];
          const unsigned kind = f[k].dst >> 16;
          if (kind >= kImages) {
            float* d = store + (f[k].dst & 0xffffu);
            d[0] = store[f[k].src & 0xffffu];
            if (kind == kImages) d[1] = store[f[k].src >> 16];
            wait[k] = false;
          }
        }
        long long began = 0;
        for (int spin = 1;; ++spin) {
          Packet v[kBatch];
          bool more = false;
#pragma unroll
          for (int k = 0; k < kBatch; ++k)
            if (wait[k]) v[k] = look(in + f[k].src);
#pragma unroll
          for (int k = 0; k < kBatch; ++k) {
            if (!wait[k]) continue;
            if (!arrived(v[k], tag)) {
              more = true;
              continue;
            }
            wait[k] = false;
            float* d = store + (f[k].dst & 0xffffu);
            const unsigned kind = f[k].dst >> 16;
            if (kind == kPair)
              *reinterpret_cast<u64*>(d) =
                  pk(__uint_as_float(value_of(v[k].a)), __uint_as_float(value_of(v[k].b)));
            else
              d[0] = __uint_as_float(value_of(kind == kFirst ? v[k].a : v[k].b));
          }
          if (!more) break;
          if (spin % 256 == 0) {
            const long long now = clock64();
            if (!began) began = now;
            if (now - began > a.limit || *(volatile unsigned*)a.err) {
              atomicExch(a.err, 1u);
              *(volatile int*)&s_abort = 1;
              break;
            }
          }
        }
      }
      __syncthreads();
      if (*(volatile int*)&s_abort) break;
    }
    const bool failed = *(volatile int*)&s_abort != 0;
    for (int i = threadIdx.x; i < w * h; i += kThreads) {
      const int y = i / w, x = i % w;
      state[(int64_t)(t.y0 + y) * b.nx + t.x0 + x] =
          failed ? __int_as_float(0x7fffffff) : store[(y + HR) * kPitch + kOff + x] + shift;
    }
    __syncthreads();
    if (failed) return;
  }
}

// The forms that are built (pairs per lane, warps, blocks per SM, halo).
// Measured, us per step (Cahn-Hilliard 2048^2 / 515 x 1031, Allen-Cahn 64^2):
// one pair, 16 warps, halo 4: 9.0 / 2.6 / 0.95; two pairs, halo 4: 9.2 / 3.7 /
// 1.4, halo 8: 9.4 / 3.7 / 1.9; an exchange every step: 9.8 / 3.4 / 1.6; 24 or
// 32 warps spill (10.2 and 13 at 2048^2).  The step kernel replayed from a
// graph takes 10.0 / 3.7 / 2.7 (12.4 / 4.0 / 5.5 before this arithmetic).
// Cycles of a step (clock64 at the barriers, 1,000 steps): 2048^2 14,400 of
// sweeps, 630 before them and 2,800 of exchange; 515 x 1031 2,770, 630 and 1,500;
// Allen-Cahn 64^2 540, 260 and 770.
// Ensembles: two blocks per SM work on different instances, so one's exchange
// runs under the other's sweeps, and exact strips lose no column at the widths
// of 128: 51 us per step of 256 instances (31.7 M nodes), against 60 to 70 for
// forms with halo lanes, 97 for one launch per step and 109 before.  At other
// widths strips of 128 columns leave lanes idle, and still: 256 square instances,
// us for 200 steps on chip / one launch per step, tuned (the band sweep in one
// launch is within 9 % of that): side 128 1,330 / 4,560, 130 2,840 / 4,560, 150 3,170 /
// 4,980, 190 4,560 / 7,790, 200 4,810 / 8,290, 300 10,820 / 14,540, 350 12,350 /
// 19,910, 500 37,350 / 38,140.  The sweep is level on many tiny instances (5,000
// of 16^2, 120 steps: 3,740 / 3,020, before 3,820) and strips of 8 columns (20 of
// 3000 x 8: 1,870 / 1,800, before 2,140).
struct Form {
  int kp, warps, blocks, halo;
};
constexpr Form kForms[] = {{1, 16, 1, 4}, {2, 8, 2, 1}};
constexpr int kMeshForm = 0, kEnsForm = 1;

template <int I, class F>
auto geo_at(bool ch, F&& fn) {
  constexpr Form f = kForms[I];
  if constexpr (f.halo == 1) {
    return fn(Geo<false, f.kp, 1>{});
  } else {
    if (ch) return fn(Geo<true, f.kp, f.halo>{});
    return fn(Geo<false, f.kp, f.halo>{});
  }
}
template <class F>
auto with_geo(bool ch, int form, F&& fn) {
  return form == kMeshForm ? geo_at<kMeshForm>(ch, fn) : geo_at<kEnsForm>(ch, fn);
}
int cols_of(bool ch, int form) {
  return with_geo(ch, form, [](auto g) { return (int)decltype(g)::kCols; });
}
size_t smem_of(bool ch, int form, const OnchipJob& b) {
  const int h = tallest(b), np = (b.nx + 1) / 2, w = 2 * ((np + b.gx - 1) / b.gx);
  return with_geo(ch, form, [&](auto g) {
    using G = decltype(g);
    return sizeof(float) * (size_t)(h + 2 * G::kRows + kForms[form].warps * (ch ? 2 : 1)) *
               G::kPitch +
           sizeof(Fetch) * fetch_entries<G>(w, h) + sizeof(Send) * send_entries<G>(w, h);
  });
}
size_t smem_cap(int form) { return kMaxSmem / kForms[form].blocks - 1536; }
int blocks_of(int form) { return device_sm_count() * kForms[form].blocks; }

// SM cycles of one step of a tile: 4 warps per scheduler (both blocks of an
// SM), each its band's rows and the rows that fill its window, at the packed
// operations of a row (2 cycles each) or, for few of them, a row's dependent
// latency; barriers; and the exchange's share when there are neighbours, most
// of which the SM's other block covers.
double tile_cycles(bool ch, int form, int h, bool alone) {
  const Form& f = kForms[form];
  const int steps = with_geo(ch, form, [](auto g) { return (int)decltype(g)::kSteps; });
  const double rows = (h + (steps - 1) * (ch ? 2 : 1) + f.warps - 1) / f.warps + (ch ? 2.8 : 1.8);
  const double row = std::max(f.blocks * f.warps / 4.0 * f.kp * (ch ? 72 : 62), 300.0);
  const double exchange = alone ? 300.0 : (f.blocks > 1 ? 2500.0 : 4000.0);
  return rows * row + 500.0 + exchange / steps;
}

template <bool kCH, int I, bool kEns>
cudaError_t launch(const OnchipArgs& a, bool iso, bool odd, int grid, size_t smem,
                   cudaStream_t s) {
  static std::atomic<unsigned long long> done[3];
  constexpr Form f = kForms[I];
  const int v = sweep_variant(iso, odd);
  auto* k = v == 0   ? k_onchip2d<kCH, true, true, f.kp, f.warps, f.blocks, f.halo, kEns>
            : v == 1 ? k_onchip2d<kCH, false, true, f.kp, f.warps, f.blocks, f.halo, kEns>
                     : k_onchip2d<kCH, false, false, f.kp, f.warps, f.blocks, f.halo, kEns>;
  cudaError_t e = raise_smem_limit(k, kMaxSmem - 1024, done[v]);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(32 * f.warps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, a);
}

// the tile grid of a mesh for tiles at most hcap rows tall on `blocks` blocks; false
// if it has none
bool tile_grid(bool ch, int form, int blocks, int hcap, OnchipJob* b) {
  const Form& f = kForms[form];
  const int np = (b->nx + 1) / 2, half = cols_of(ch, form) / 2;
  b->gx = (np + half - 1) / half;
  b->gy = (b->ny + hcap - 1) / hcap;
  if (b->gy > 1 && b->ny / b->gy < f.halo + 1) return false;  // rows that a neighbour needs
  if (b->gx > 1 && np / b->gx < 3) return false;
  return (int64_t)b->gx * b->gy <= blocks &&
         (f.halo > 1 || (tallest(*b) + f.warps - 1) / f.warps <= kMaxBand) &&
         smem_of(ch, form, *b) <= smem_cap(form);
}

size_t exchange_bytes(bool ch, int form, const OnchipJob& b) {
  if (b.gx * b.gy == 1) return 0;
  const int slot =
      with_geo(ch, form, [&](auto g) { return slot_packets<decltype(g)>(tallest(b)); });
  return sizeof(Packet) * 2 * (size_t)slot * b.gx * b.gy;
}

}  // namespace

size_t onchip_exchange_bytes(bool ch, const OnchipJob& b) {
  return exchange_bytes(ch, kMeshForm, b);
}

bool onchip_plan(bool ch, size_t bytes, OnchipJob* job) {
  double best = -1.0;
  OnchipJob pick = *job, b = *job;
  const int half = cols_of(ch, kMeshForm) / 2, gx = ((b.nx + 1) / 2 + half - 1) / half;
  const int blocks = blocks_of(kMeshForm);
  for (int gy = 1; gx * gy <= blocks && gy <= b.ny; ++gy) {
    const int h = (b.ny + gy - 1) / gy;
    if (gy > 1 && b.ny / gy < kForms[kMeshForm].halo + 1) break;  // nor do more
    if ((b.ny + h - 1) / h != gy) continue;  // as fewer tiles of this height
    if (!tile_grid(ch, kMeshForm, blocks, h, &b)) continue;
    if (onchip_exchange_bytes(ch, b) > bytes) continue;
    const double c = tile_cycles(ch, kMeshForm, tallest(b), gx * gy == 1);
    if (best < 0 || c < best) {
      best = c;
      pick = b;
    }
  }
  *job = pick;
  return best >= 0;
}

// us: a step of the band sweep replayed from a graph (fixed, per million nodes) and
// of the on-chip form (fixed, per 100 rows of a tile), by sweep_variant.  A step on
// chip takes what its tile's height does, however many SMs have a tile: 600 x 4300
// makes 77 tiles of 600 rows and takes 10.3 us (Cahn-Hilliard, square cells) where
// the sweep takes 7.1 (8.2 before this form), 1000 x 3000 108 tiles, 8.6 and 7.9,
// 2048^2 148 tiles, 8.9 and 10.4, 300 x 8000 143 tiles, 5.7 and 6.9.  Fitted to 26
// meshes of 64^2 to 3000^2 nodes, each within 0.3 us.
struct Rate {
  double band0, band1, chip0, chip1;
};
constexpr Rate kRates[2][3] = {
    {{2.25, 1.33, 0.75, 1.14}, {2.3, 1.34, 0.75, 1.2}, {2.35, 1.53, 0.8, 1.38}},  // Allen-Cahn
    {{2.45, 1.87, 1.5, 1.45}, {2.4, 1.93, 1.5, 1.56}, {2.5, 2.14, 1.6, 1.74}}};

bool onchip_pays(bool ch, bool iso, bool odd, const OnchipJob& b, int64_t steps, bool graph) {
  const Rate& r = kRates[ch][sweep_variant(iso, odd)];
  const double nodes = 1e-6 * b.nx * b.ny, h = 0.01 * tallest(b);
  // a sweep launched by itself takes up to 2 us more; a call's tiles, tables and
  // conversions
  const double band = r.band0 + r.band1 * nodes + (graph ? 0.0 : 2.0), chip = r.chip0 + r.chip1 * h;
  return 13.0 + 18.0 * h + chip * steps <= 13.5 + 4.0 * nodes + band * steps;
}

cudaError_t launch_onchip(bool ch, const OnchipArgs& a, bool iso, bool odd, int absent,
                          cudaStream_t s) {
  const size_t smem = smem_of(ch, kMeshForm, a.job);
  const int grid = a.job.gx * a.job.gy - absent;
  return ch ? launch<true, kMeshForm, false>(a, iso, odd, grid, smem, s)
            : launch<false, kMeshForm, false>(a, iso, odd, grid, smem, s);
}

// Ensembles: an instance is a job of gx * gy tiles that run together for all
// steps.  Jobs go to the blocks longest first, each to the blocks that are
// free the earliest; every block works through its jobs in that one order, so
// the waits between a job's tiles end.  The tallest tile is the one with the
// shortest schedule by tile_cycles.
bool onchip_plan_ensemble(std::vector<OnchipJob>& jobs, std::vector<int>* first,
                          std::vector<OnchipItem>* list, size_t* exchange, size_t* smem) {
  const int blocks = blocks_of(kEnsForm);
  double best = -1.0;
  std::vector<OnchipJob> best_jobs;
  std::vector<std::pair<int, OnchipItem>> placed, best_placed;  // (block, item) in order
  std::vector<int> heights = {384, 320, 256, 192, 128, 96, 64, 32, 16};
  if (jobs.size() > 4096) heights = {192};  // as many jobs as blocks many times over
  std::vector<OnchipJob> js = jobs;
  std::vector<int> scheduled;
  std::vector<double> cost(js.size());
  std::vector<int> order(js.size());
  for (int hcap : heights) {
    // the next lower cap often gives the grids that were scheduled last
    std::vector<int> rows(js.size());
    bool ok = true;
    for (size_t i = 0; i < js.size() && ok; ++i) {
      ok = tile_grid(false, kEnsForm, blocks, hcap, &js[i]);
      rows[i] = js[i].gy;
    }
    if (!ok || rows == scheduled) continue;
    scheduled.swap(rows);
    for (size_t i = 0; i < js.size(); ++i) {
      cost[i] = tile_cycles(false, kEnsForm, tallest(js[i]), js[i].gx * js[i].gy == 1);
      order[i] = (int)i;
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
      const int gx = js[x].gx * js[x].gy, gy = js[y].gx * js[y].gy;
      return gx != gy ? gx > gy : cost[x] > cost[y];
    });
    typedef std::pair<double, int> Free;  // (time a block is free, block)
    std::vector<Free> idle(blocks);
    for (int b = 0; b < blocks; ++b) idle[b] = Free(0.0, b);
    std::priority_queue<Free, std::vector<Free>, std::greater<Free>> q(std::greater<Free>(),
                                                                       std::move(idle));
    placed.clear();
    double end = 0.0;
    std::vector<int> gang;
    for (int j : order) {
      const int g = js[j].gx * js[j].gy;
      double start = 0.0;
      gang.clear();
      for (int t = 0; t < g; ++t) {
        start = std::max(start, q.top().first);
        gang.push_back(q.top().second);
        q.pop();
      }
      for (int t = 0; t < g; ++t) {
        placed.emplace_back(gang[t], OnchipItem{j, t});
        q.push(Free(start + cost[j], gang[t]));
      }
      end = std::max(end, start + cost[j]);
    }
    if (best < 0 || end < best) {
      best = end;
      best_jobs = js;
      best_placed.swap(placed);
    }
  }
  if (best < 0) return false;
  jobs = best_jobs;
  // the blocks' lists one after another, each in the order of placing
  first->assign(blocks + 1, 0);
  for (const auto& p : best_placed) ++(*first)[p.first + 1];
  for (int b = 0; b < blocks; ++b) (*first)[b + 1] += (*first)[b];
  std::vector<int> next(first->begin(), first->end() - 1);
  list->resize(best_placed.size());
  for (const auto& p : best_placed) (*list)[next[p.first]++] = p.second;
  *exchange = 0;
  *smem = 0;
  for (OnchipJob& b : jobs) {
    b.xchg = (int64_t)(*exchange / sizeof(Packet));
    *exchange += exchange_bytes(false, kEnsForm, b);
    *smem = std::max(*smem, smem_of(false, kEnsForm, b));
  }
  return true;
}

cudaError_t launch_onchip_ensemble(const OnchipArgs& a, size_t smem, bool iso, bool odd,
                                   cudaStream_t s) {
  return launch<false, kEnsForm, true>(a, iso, odd, blocks_of(kEnsForm), smem, s);
}

}  // namespace pf
