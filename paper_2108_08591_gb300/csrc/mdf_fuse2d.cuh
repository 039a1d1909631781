// K updates of a 2D FP32 lattice in one pass over memory.
//
// What bounds the single update is HBM: 120 B per node against ~320
// instructions, which keep the SMs' issue slots less than half busy.  Here
// every population is read once and written once per K updates; the updates
// in between stay in registers.
//
// A warp owns a strip of 64 columns (two x-adjacent nodes per lane, one
// FP32 pair) and marches along y.  In iteration r it pulls row r from memory
// and does update 1 on it, then update 2 on row r - 1, ..., update K on row
// r - K + 1, which it stores.  Update s + 1 of row q pulls, of what update s
// left,
//   - the directions that stay in the row from row q (its x neighbours by
//     warp shuffle), computed one iteration ago and carried,
//   - the direction along +y from row q - 1, carried for two iterations,
//   - the direction along -y from row q + 1, computed just now.
// What is carried sits in shared memory, each lane reading back only what it
// wrote: no barrier, and registers stay for more warps.  The price is redundant
// work at a strip's rim: the outermost column of each side is lost per
// update, so a strip stores 64 - 2 H of its columns (H = K rounded up to
// even: stores stay aligned pairs), and a row segment starts K - 1 rows
// early and ends K - 1 rows late.
//
// The arithmetic per node is the single update's (the same templates on the
// type F2, the same dither draws from the node's global index and the step),
// so the bits are those of K single updates.
//
// Measured (GB300, K = 4, us per update against one update per launch):
// 4096^2 147 / 300, 2048^2 40.3 / 79, 1024^2 13.1 / 22.6;
// 4095^2 149 / (scalar kernel) 330; walls and lid 165 at 4096^2.  K = 4 is
// bound by the FP32 and integer pipes (issue 58 %, the f32x2 operations take
// two slots of theirs): 219 instructions per update and node, of which 1.14
// x is rim.  K = 2 takes 180 us at 4096^2; it serves lattices of fewer than
// 750 000 nodes, where the row updates that fill and drain the pipeline count
// (509 x 515 with walls: 5.6 us per update, 6.6 with K = 4, 10.0 single).
#pragma once

#include "mdf_kernels.cuh"

namespace mdf {

template <int K> constexpr int fuse_halo() { return (K + 1) / 2 * 2; }
template <int K> constexpr int fuse_out() { return 64 - 2 * fuse_halo<K>(); }

enum { FORCE_NONE = 0, FORCE_EQ321 = 1, FORCE_SCHEME2 = 2 };

__device__ __forceinline__ F2 shfl_pair_left(F2 v) {  // values of columns (c0 - 1, c0)
  return F2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
}
__device__ __forceinline__ F2 shfl_pair_right(F2 v) {  // values of columns (c0 + 1, c0 + 2)
  return F2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
}

// One lane's columns and what the walls make of them.
struct FuseCols {
  int xa, xb;          // columns (wrapped into the row)
  bool vec;            // the pair is one aligned 8-byte access
  bool w0a, w0b;       // column 0 behind an x wall (its -x link)
  bool w1a, w1b;       // column nx - 1 before an x wall
  bool wall;           // the strip has a column at an x wall
};

// Row directions of one set: shift along x by one column and bounce back at
// the x walls (the value that leaves through the wall returns negated).
template <class L, bool WALLS>
__device__ __forceinline__ void fuse_shift_row(F2 (&g)[L::Q], const FuseCols &c) {
#pragma unroll
  for (int i = 0; i < L::Q; ++i)
    if (L::c(i, 0) == 1) {
      const int o = L::opp(i);
      const F2 p = g[i], m = g[o];
      F2 fp = shfl_pair_left(p), fm = shfl_pair_right(m);
      if (WALLS && c.wall) {
        fp = F2(c.w0a ? -m.x : fp.x, c.w0b ? -m.y : fp.y);
        fm = F2(c.w1a ? -p.x : fm.x, c.w1b ? -p.y : fm.y);
      }
      g[i] = fp;
      g[o] = fm;
    }
}

__device__ __forceinline__ F2 fuse_load(const float *p, const FuseCols &c) {
  if (c.vec) return F2(__ldg(reinterpret_cast<const float2 *>(p + c.xa)));
  return F2(__ldg(p + c.xa), __ldg(p + c.xb));
}

// Eq. 2-7, 3-15, 2-4 and 3-21 on a pair of nodes: collide_node's operations.
template <class L, int FORCE, class TF>
__device__ __forceinline__ void fuse_collide(F2 (&g)[3][L::Q], const TF (&F)[2], const Rates<F2> &R, uint2 key,
                                             F2 (&u)[2]) {
  F2 Pp, gv[2][L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) { gv[0][i] = g[0][i]; gv[1][i] = g[1][i]; }
  node_moments<L, F2, FORCE == FORCE_SCHEME2>(gv, F, u, Pp);
#pragma unroll
  for (int a = 0; a < 2; ++a) relax_velocity_set<L, F2, true>(g[a], a, u, Pp, R, F[a], key);
  F2 r;
  relax_rho_set<L, F2>(g[2], u, R, r);
}

// Resident blocks per SM the register budget allows for: 128 registers, no
// spills.  Nine (112 registers) ran at 173 us per update at 4096^2 against
// 152, six (168) at 162.
constexpr int kFuseBlocks = 8;

// A 2D lattice as the march sees it.
struct FuseLattice {
  const float *fin;          // populations, node (0, 0)
  float *fout;
  long long plane;           // direction stride
  int nx, ny, px;            // px: row pitch
  bool pairs;                // every row starts on an 8-byte boundary
  bool wx, wy, lid;          // walls, lid on the + y face
  float lid_u[2];            // 2 w u of the lid
  const float *force;        // [2][plane], or null
  float s1, s2;
  uint32_t key0;             // global index of node (0, 0), low word
  int t0;                    // time step of update 1
  float *usave;              // [2][plane]: velocity pulled by update 1 (SAVE)
};

// K updates of rows y0 .. y1 - 1 of a strip by one warp; sb: the lane's
// shared memory, K - 1 x 3 Q slots of 32 lanes.
template <class L, int K, bool WALLS, int FORCE, bool SAVE>
__device__ __forceinline__ void fuse_march(const FuseLattice &A, int strip, int y0, int y1, float2 *const sb) {
  static_assert(L::D == 2 && K >= 2, "2D, at least two updates");
  constexpr int Q = L::Q, H = fuse_halo<K>(), OUT = fuse_out<K>();
  const int lane = threadIdx.x & 31;
  const bool wx = WALLS && A.wx, wy = WALLS && A.wy;

  const int c0 = strip * OUT - H + 2 * lane;
  FuseCols c;
  c.xa = c0 < 0 ? (c0 % A.nx + A.nx) % A.nx : c0 % A.nx;
  c.xb = c.xa + 1 == A.nx ? 0 : c.xa + 1;
  // an odd row is not a whole number of pairs: where the strip leaves it,
  // the wrapped columns are read one by one (behind an x wall they are not
  // used, so any column will do)
  c.vec = A.pairs && ((A.nx & 1) == 0 || wx || (strip * OUT - H >= 0 && strip * OUT - H + 64 <= A.nx));
  if (c.vec && (c.xa & 1)) c.xa = c.xb = 0;  // odd nx behind an x wall
  c.w0a = wx && c0 == 0;
  c.w0b = false;  // c0 is even
  c.wall = wx && (strip * OUT - H <= 0 || strip * OUT - H + 64 >= A.nx);
  c.w1a = wx && c0 == A.nx - 1;
  c.w1b = wx && c0 + 1 == A.nx - 1;
  const bool out_a = lane >= H / 2 && lane < 32 - H / 2 && c0 < A.nx;
  const bool out_b = out_a && c0 + 1 < A.nx;

  const float *__restrict__ fin = A.fin;
  float *__restrict__ fout = A.fout;
  const Rates<F2> R(F2(A.s1, A.s1), F2(A.s2, A.s2));
  const int t0 = A.t0;
  F2 lid[3][Q] = {};
  if (WALLS) {
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (L::c(i, 1) == -1) {
#pragma unroll
        for (int a = 0; a < 2; ++a) lid[a][i] = F2(A.lid_u[a], A.lid_u[a]);
      }
  }

  // what update s + 1 still needs of update s, per lane, in shared memory:
  // the row directions of the row last computed, shifted, and the +y
  // direction of the last two rows (alternating slots)
  constexpr int NROW = Q - 2, SLOTS = 3 * (NROW + 2);
  const int iters = y1 - y0 + 2 * (K - 1);
  for (int it = 0; it < iters; ++it) {
    const int r = y0 - (K - 1) + it;
    F2 g[3][Q];
    {  // update 1 of row r from memory
      const int yr = wy ? min(max(r, 0), A.ny - 1) : wrap(r, A.ny);
      const int ym = yr == 0 ? A.ny - 1 : yr - 1, yp = yr == A.ny - 1 ? 0 : yr + 1;
      const float *p0 = fin + (long long)yr * A.px;
      const float *pm = fin + (long long)ym * A.px, *pp = fin + (long long)yp * A.px;
      const bool lo = wy && r == 0, hi = wy && r == A.ny - 1;
      auto load_row = [&](auto vec) {
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const long long set = (long long)(s < 2 ? s + 1 : 0) * Q;  // velocity sets, then alpha = 0
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            // behind a y wall: the node's own opposite direction
            const bool wall = WALLS && ((L::c(i, 1) == 1 && lo) || (L::c(i, 1) == -1 && hi));
            const float *p = wall ? p0 + (set + L::opp(i)) * A.plane
                                  : (L::c(i, 1) == 1 ? pm : L::c(i, 1) == -1 ? pp : p0) + (set + i) * A.plane;
            if constexpr (vec) g[s][i] = F2(__ldg(reinterpret_cast<const float2 *>(p + c.xa)));
            else g[s][i] = F2(__ldg(p + c.xa), __ldg(p + c.xb));
          }
        }
      };
      if (c.vec) load_row(std::true_type{});
      else load_row(std::false_type{});
      if (WALLS && (lo || hi)) {  // negated, plus the lid
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            if (L::c(i, 1) == 1 && lo) g[s][i] = -g[s][i];
            if (L::c(i, 1) == -1 && hi) {
              g[s][i] = -g[s][i];
              if (s < 2 && A.lid) g[s][i] += lid[s][i];
            }
          }
      }
#pragma unroll
      for (int s = 0; s < 3; ++s) fuse_shift_row<L, WALLS>(g[s], c);
    }
#pragma unroll
    for (int s = 0; s < K; ++s) {  // update s + 1 on row q
      const int q = r - s;
      if (s > 0) {
        // g: update s of row q + 1; assemble the pull of row q, keep the rest
        float2 *const cs = sb + (s - 1) * SLOTS * 32;
        float2 *const cu = cs + (3 * NROW + (it & 1) * 3) * 32;        // +y of row q - 1, then of row q + 1
        float2 *const cv = cs + (3 * NROW + ((it & 1) ^ 1) * 3) * 32;  // +y of row q
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          F2 n[Q];
          int k = 0;
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            if (L::c(i, 1) == 1) {
              n[i] = F2(cu[e * 32]);
            } else if (L::c(i, 1) == -1) {
              n[i] = g[e][i];
              if (WALLS && wy && q == A.ny - 1) {  // row ny - 1 pulls its own +y direction back
                n[i] = -F2(cv[e * 32]);
                if (e < 2 && A.lid) n[i] += lid[e][i];
              }
              if (WALLS && wy && q == -1) cv[e * 32] = (-g[e][i]).f2();  // so does row 0 its -y direction
            } else {
              n[i] = F2(cs[(e * NROW + k++) * 32]);
            }
          }
          fuse_shift_row<L, WALLS>(g[e], c);
          k = 0;
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            if (L::c(i, 1) == 0) cs[(e * NROW + k++) * 32] = g[e][i].f2();
            if (L::c(i, 1) == 1) cu[e * 32] = g[e][i].f2();
            g[e][i] = n[i];
          }
        }
        if (it < 2 * s) break;  // the rows below have not come through yet
      }
      const int yq = wy ? q : wrap(q, A.ny);
      const uint32_t n0 = A.key0 + (uint32_t)(yq * A.nx);
      const uint2 key = make_uint2(node_key(n0 + c.xa, t0 + s), node_key(n0 + c.xb, t0 + s));
      F2 u[2];
      if constexpr (FORCE == FORCE_NONE) {
        const NoForce F[2] = {};
        fuse_collide<L, FORCE>(g, F, R, key, u);
      } else {
        const float *fp = A.force + (long long)(wy ? min(max(q, 0), A.ny - 1) : yq) * A.px;
        const F2 F[2] = {fuse_load(fp, c), fuse_load(fp + A.plane, c)};
        fuse_collide<L, FORCE>(g, F, R, key, u);
      }
      if constexpr (SAVE) {
        if (s == 0 && q >= y0 && q < y1) {
          float *p = A.usave + (long long)q * A.px + c0;
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            if (out_a) p[a * A.plane] = u[a].x;
            if (out_b) p[a * A.plane + 1] = u[a].y;
          }
        }
      }
    }
    if (it < 2 * (K - 1)) continue;
    float *po = fout + (long long)(r - (K - 1)) * A.px + c0;
    // 2: a pair as one access, 1: a pair in two, 0: the odd row's last node
    auto store_row = [&](auto how) {
#pragma unroll
      for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          float *p = po + ((long long)(s < 2 ? s + 1 : 0) * Q + i) * A.plane;
          if constexpr (how == 2) {
            __stcs(reinterpret_cast<float2 *>(p), g[s][i].f2());
          } else {
            __stcs(p, g[s][i].x);
            if constexpr (how == 1) __stcs(p + 1, g[s][i].y);
          }
        }
    };
    if (out_b) {
      if (A.pairs) store_row(std::integral_constant<int, 2>{});
      else store_row(std::integral_constant<int, 1>{});
    } else if (out_a) {
      store_row(std::integral_constant<int, 0>{});
    }
  }
}

// The lattice of a launch's arguments.
template <class L>
__device__ __forceinline__ FuseLattice fuse_lattice(const DevArgs &A) {
  FuseLattice G;
  G.fin = static_cast<const float *>(A.fin);
  G.fout = static_cast<float *>(A.fout);
  G.plane = A.plane;
  G.nx = A.nx;
  G.ny = A.ny;
  G.px = A.px;
  G.pairs = true;  // the pitch is a multiple of 32
  G.wx = A.wall[0] != 0;
  G.wy = A.wall[1] != 0;
  G.lid = A.lid != 0;
  G.lid_u[0] = float(2.0 * L::w(L::UP) * A.lid_u[0]);
  G.lid_u[1] = float(2.0 * L::w(L::UP) * A.lid_u[1]);
  G.force = static_cast<const float *>(A.force);
  G.s1 = A.s1f;
  G.s2 = A.s2f;
  G.key0 = (uint32_t)A.key_base;
  G.t0 = launch_step(A);
  G.usave = nullptr;
  return G;
}

template <int K, int Q> constexpr int fuse_slots() { return (K - 1) * 3 * Q * 32; }  // float2 per warp

template <class L, int K, bool WALLS, int FORCE>
__global__ void __launch_bounds__(32 * kFuseWarps, kFuseBlocks)
    k_update_fused2d(const DevArgs A, int strips, int seg_rows, int nseg) {
  extern __shared__ float2 fuse_smem[];
  const int item = blockIdx.x * kFuseWarps + (threadIdx.x >> 5);
  if (item >= strips * nseg) return;  // the whole warp
  const int strip = item % strips, seg = item / strips;
  fuse_march<L, K, WALLS, FORCE, false>(fuse_lattice<L>(A), strip, seg * seg_rows, min((seg + 1) * seg_rows, A.ny),
                                        fuse_smem + (threadIdx.x >> 5) * fuse_slots<K, L::Q>() + (threadIdx.x & 31));
}

// Rows per segment for one wave of w = 1 .. wmax warps per SM sub-partition
// (items(rows): warps that segments of that many rows make).  A warp does K
// rows + K (K - 1) row updates (the second term fills and drains the
// pipeline), each in a time of about 1.7 + w: measured at 1024^2, K = 4:
// 0.57 / 0.76 / 1.0 / 1.2 us for w = 1 .. 4.  Long segments waste less, many
// warps hide more; large lattices take the most warps, small ones fewer
// (256^2: 3.65 us per update with w = 1 against 4.17 with w = 2 .. 4;
// 1024^2: 20.0, 14.5, 14.0, 14.1, at a build that now takes 13.1).
template <int K, class Items>
int fuse_rows(int ny, int wmax, Items items) {
  int best_rows = ny;
  double best = 0.0;
  for (int w = 1; w <= std::max(1, wmax); ++w) {
    int lo = std::min(ny, 2), hi = ny;  // fewest rows that fit one wave (the longest when none does)
    while (lo < hi) {
      const int mid = (lo + hi) / 2;
      if (items(mid) <= 4LL * w * kSMs) hi = mid;
      else lo = mid + 1;
    }
    const double cost = (lo + K - 1.0) * (1.7 + w);
    if (best == 0.0 || cost < best) {
      best = cost;
      best_rows = lo;
    }
  }
  return best_rows;
}

template <class L, int K, bool WALLS, int FORCE>
cudaError_t launch_fused2d(const DevArgs &a, cudaStream_t s) {
  constexpr size_t smem = (size_t)kFuseWarps * fuse_slots<K, L::Q>() * sizeof(float2);
  static const int per_sm = [] {  // resident blocks per SM of this build
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_update_fused2d<L, K, WALLS, FORCE>, 32 * kFuseWarps,
                                                      smem) != cudaSuccess)
      cudaGetLastError();
    return n > 0 ? n : 1;
  }();
  const int strips = (a.nx + fuse_out<K>() - 1) / fuse_out<K>();
  const int seg_rows = fuse_rows<K>(a.ny, per_sm * kFuseWarps / 4, [&](int rows) {
    return (long long)strips * ((a.ny + rows - 1) / rows);
  });
  const int nseg = (a.ny + seg_rows - 1) / seg_rows;
  const long long items = (long long)strips * nseg;
  k_update_fused2d<L, K, WALLS, FORCE>
      <<<(unsigned)((items + kFuseWarps - 1) / kFuseWarps), 32 * kFuseWarps, smem, s>>>(a, strips, seg_rows, nseg);
  return cudaGetLastError();
}

template <class L, int K>
cudaError_t update_fused2d(bool walls, const DevArgs &a, cudaStream_t s) {
  if (a.scheme2)
    return walls ? launch_fused2d<L, K, true, FORCE_SCHEME2>(a, s) : launch_fused2d<L, K, false, FORCE_SCHEME2>(a, s);
  if (a.force)
    return walls ? launch_fused2d<L, K, true, FORCE_EQ321>(a, s) : launch_fused2d<L, K, false, FORCE_EQ321>(a, s);
  return walls ? launch_fused2d<L, K, true, FORCE_NONE>(a, s) : launch_fused2d<L, K, false, FORCE_NONE>(a, s);
}

}  // namespace mdf
