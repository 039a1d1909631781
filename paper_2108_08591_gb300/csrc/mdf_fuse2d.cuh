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
// 4096^2 152 / 301, 2048^2 42.1 / 80, 1024^2 14.2 / 22.6, 256^2 3.7 / 6.2;
// 4095^2 153 / (scalar kernel) 330; walls and lid 170 at 4096^2.  K = 4 is
// bound by the FP32 and integer pipes (issue 58 %, the f32x2 operations take
// two slots of theirs): 219 instructions per update and node, of which 1.14
// x is rim.  K = 2 would stay at HBM's 150 us.
#pragma once

#include "mdf_kernels.cuh"

namespace mdf {

constexpr int kFuseWarps = 2;  // independent warps per block
constexpr int kSMs = 152;      // of a GB300
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
__device__ __forceinline__ void fuse_collide(F2 (&g)[3][L::Q], const TF (&F)[2], const Rates<F2> &R, uint2 key) {
  F2 u[2], Pp, gv[2][L::Q];
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

template <class L, int K, bool WALLS, int FORCE>
__global__ void __launch_bounds__(32 * kFuseWarps, kFuseBlocks)
    k_update_fused2d(const DevArgs A, int strips, int seg_rows, int nseg) {
  static_assert(L::D == 2 && K >= 2, "2D, at least two updates");
  constexpr int Q = L::Q, H = fuse_halo<K>(), OUT = fuse_out<K>();
  const int lane = threadIdx.x & 31;
  const int item = blockIdx.x * kFuseWarps + (threadIdx.x >> 5);
  if (item >= strips * nseg) return;  // the whole warp
  const int strip = item % strips, seg = item / strips;
  const int y0 = seg * seg_rows, y1 = min(y0 + seg_rows, A.ny);
  const bool wx = WALLS && A.wall[0], wy = WALLS && A.wall[1];

  const int c0 = strip * OUT - H + 2 * lane;
  FuseCols c;
  c.xa = c0 < 0 ? (c0 % A.nx + A.nx) % A.nx : c0 % A.nx;
  c.xb = c.xa + 1 == A.nx ? 0 : c.xa + 1;
  // an odd row is not a whole number of pairs: where the strip leaves it,
  // the wrapped columns are read one by one (behind an x wall they are not
  // used, so any column will do)
  c.vec = (A.nx & 1) == 0 || wx || (strip * OUT - H >= 0 && strip * OUT - H + 64 <= A.nx);
  if (c.vec && (c.xa & 1)) c.xa = c.xb = 0;  // odd nx behind an x wall
  c.w0a = wx && c0 == 0;
  c.w0b = false;  // c0 is even
  c.wall = wx && (strip * OUT - H <= 0 || strip * OUT - H + 64 >= A.nx);
  c.w1a = wx && c0 == A.nx - 1;
  c.w1b = wx && c0 + 1 == A.nx - 1;
  const bool out_a = lane >= H / 2 && lane < 32 - H / 2 && c0 < A.nx;
  const bool out_b = out_a && c0 + 1 < A.nx;

  const float *__restrict__ fin = static_cast<const float *>(A.fin);
  float *__restrict__ fout = static_cast<float *>(A.fout);
  const Rates<F2> R(F2(A.s1f, A.s1f), F2(A.s2f, A.s2f));
  const int t0 = launch_step(A);
  F2 lid[3][Q] = {};
  if (WALLS) {
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (L::c(i, 1) == -1) {
#pragma unroll
        for (int a = 0; a < 2; ++a) lid[a][i] = F2(2.0 * L::w(i) * A.lid_u[a]);
      }
  }

  // what update s + 1 still needs of update s, per lane, in shared memory:
  // the row directions of the row last computed, shifted, and the +y
  // direction of the last two rows (alternating slots)
  constexpr int NROW = Q - 2, SLOTS = 3 * (NROW + 2);
  extern __shared__ float2 fuse_smem[];
  float2 *const sb = fuse_smem + (threadIdx.x >> 5) * (K - 1) * SLOTS * 32 + lane;

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
      const uint32_t n0 = (uint32_t)A.key_base + (uint32_t)(yq * A.nx);
      const uint2 key = make_uint2(node_key(n0 + c.xa, t0 + s), node_key(n0 + c.xb, t0 + s));
      if constexpr (FORCE == FORCE_NONE) {
        const NoForce F[2] = {};
        fuse_collide<L, FORCE>(g, F, R, key);
      } else {
        const float *fp = static_cast<const float *>(A.force) + (long long)(wy ? min(max(q, 0), A.ny - 1) : yq) * A.px;
        const F2 F[2] = {fuse_load(fp, c), fuse_load(fp + A.plane, c)};
        fuse_collide<L, FORCE>(g, F, R, key);
      }
    }
    if (it < 2 * (K - 1)) continue;
    float *po = fout + (long long)(r - (K - 1)) * A.px + c0;
    auto store_row = [&](auto pair) {
#pragma unroll
      for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          float *p = po + ((long long)(s < 2 ? s + 1 : 0) * Q + i) * A.plane;
          if constexpr (pair) __stcs(reinterpret_cast<float2 *>(p), g[s][i].f2());
          else __stcs(p, g[s][i].x);
        }
    };
    if (out_b) store_row(std::true_type{});
    else if (out_a) store_row(std::false_type{});
  }
}

template <class L, int K, bool WALLS, int FORCE>
cudaError_t launch_fused2d(const DevArgs &a, cudaStream_t s) {
  constexpr size_t smem = (size_t)kFuseWarps * (K - 1) * 3 * L::Q * 32 * sizeof(float2);
  static const int per_sm = [] {  // resident blocks per SM of this build
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_update_fused2d<L, K, WALLS, FORCE>, 32 * kFuseWarps,
                                                      smem) != cudaSuccess)
      cudaGetLastError();
    return n > 0 ? n : 1;
  }();
  const int strips = (a.nx + fuse_out<K>() - 1) / fuse_out<K>();
  // Rows per segment, for one wave of w = 1 .. the resident warps per SM
  // sub-partition.  A warp does K rows + K (K - 1) row updates (the second
  // term fills and drains the pipeline), each in a time of about 1.7 + w:
  // measured at 1024^2, K = 4: 0.57 / 0.76 / 1.0 / 1.2 us for w = 1 .. 4.
  // Long segments waste less, many warps hide more; large lattices take the
  // most warps, small ones fewer (256^2: 3.65 us per update with w = 1
  // against 4.17 with w = 2 .. 4; 1024^2: 20.0, 14.5, 14.0, 14.1).
  int seg_rows = a.ny;
  double best = 0.0;
  for (int w = 1; w <= std::max(1, per_sm * kFuseWarps / 4); ++w) {
    const int want = std::max(1, kSMs * 4 * w / strips);
    const int rows = std::max((a.ny + want - 1) / want, std::min(a.ny, 2));
    const double cost = (rows + K - 1.0) * (1.7 + w);
    if (best == 0.0 || cost < best) {
      best = cost;
      seg_rows = rows;
    }
  }
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
