// Two updates of a 3D FP32 lattice in one pass over memory.
//
// The single update is bound by HBM (224 B per node, D3Q7).  Here every
// population is read once and written once per two updates.  A block of
// kF3Rows warps owns a tile of 64 columns (two x-adjacent nodes per lane, one
// FP32 pair) x kF3Rows rows, one row per warp, and marches along z.  In
// iteration r it pulls plane r from memory, does update 1 on it, then update
// 2 on plane r - 1, which it stores.  Update 2 of plane q pulls, of what
// update 1 left,
//   - the directions along x and the rest direction from its own row of plane
//     q (x neighbours by warp shuffle), carried one iteration,
//   - the directions along y from the neighbouring warps' rows of plane q,
//   - the direction along +z from plane q - 1, carried two iterations,
//   - the direction along -z from plane q + 1, computed just now.
// What is carried sits in shared memory.  Only the y directions are read by
// another warp; they alternate between two buffers, so one barrier per plane
// orders the writes of one iteration before the reads of the next.  The price
// is redundant work at the tile's rim: 60 of 64 columns and kF3Rows - 2 rows
// are stored (the outer two rows skip update 2), and a z segment starts one
// plane early and ends one late.
//
// The arithmetic per node is the single update's (the same templates on the
// type F2, the same dither draws), so the bits are those of two single
// updates.
//
// Measured (GB300, us per update against the single one): 512^3 3637 / 4633,
// 480 x 480 x 200 1226 / 1590, 256^3 534 / 584, 190 x 202 x 178 with walls
// and a lid 269 / 351, periodic 242 / 255.  Bound by the FP32 and integer
// pipes (590 instructions per update and node at 256^3, where the tiles do
// 1.5 x the work) and by the barriers: issue 47 %.  The 128 registers that two
// blocks per SM leave are not quite enough: the D3Q7 forms spill 24 B (periodic)
// to 84 B (walls and a force) of stores, the D3Q6 ones none to 120 B.  Requesting the next plane
// with cp.async (548 at 256^3), and prefetching it to L2 (578), gained
// nothing.  fuse3_plan says where it pays.
#pragma once

#include "mdf_fuse2d.cuh"

namespace mdf {

// Warps per block (one row of the tile each) and blocks per SM.  Two blocks of
// 8 run past each other's barriers and loads: 536 / 3647 us per update at
// 256^3 / 512^3 against 548 / 3802 for one of 16, though they work on 8 rows
// for 6 stored (16 for 14); one of 12 552 / 3951.
constexpr int kF3Rows = kFuse3Rows, kF3Blocks = 2;
constexpr int kF3Out = kF3Rows - 2;
// slots of 32 float2 per warp: row directions, two y directions (two
// buffers), the +z direction (two planes), of four sets
template <class L> constexpr int fuse3_slots() { return 4 * (L::Q - 4) + 4 * 2 * 2 + 4 * 2; }

template <class L, bool WALLS, int FORCE>
__global__ void __launch_bounds__(32 * kF3Rows, kF3Blocks)
    k_update_fused3d(const DevArgs A, int tiles_x, int tiles_y, int seg) {
  static_assert(L::D == 3, "3D");
  constexpr int Q = L::Q, H = fuse_halo<2>(), OUT = fuse_out<2>(), NROW = Q - 4;
  extern __shared__ float2 fuse3_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tx = blockIdx.x % tiles_x, t2 = blockIdx.x / tiles_x;
  const int ty = t2 % tiles_y, z0 = t2 / tiles_y * seg, z1 = min(z0 + seg, A.nz);
  const bool wx = WALLS && A.wall[0], wy = WALLS && A.wall[1], wz = WALLS && A.wall[2];

  // columns: as in fuse_march
  const int c0 = tx * OUT - H + 2 * lane;
  FuseCols c;
  c.xa = c0 < 0 ? (c0 % A.nx + A.nx) % A.nx : c0 % A.nx;
  c.xb = c.xa + 1 == A.nx ? 0 : c.xa + 1;
  c.vec = (A.nx & 1) == 0 || wx || (tx * OUT - H >= 0 && tx * OUT - H + 64 <= A.nx);
  if (c.vec && (c.xa & 1)) c.xa = c.xb = 0;  // odd nx behind an x wall
  c.w0a = wx && c0 == 0;
  c.w0b = false;
  c.wall = wx && (tx * OUT - H <= 0 || tx * OUT - H + 64 >= A.nx);
  c.w1a = wx && c0 == A.nx - 1;
  c.w1b = wx && c0 + 1 == A.nx - 1;
  // this warp's row; rows beyond a wall are computed on clamped data, not used
  const int yu = ty * kF3Out - 1 + warp;
  const int y = wy ? min(max(yu, 0), A.ny - 1) : (yu % A.ny + A.ny) % A.ny;
  const int ym = y == 0 ? A.ny - 1 : y - 1, yp = y == A.ny - 1 ? 0 : y + 1;
  const bool ylo = wy && yu == 0, yhi = wy && yu == A.ny - 1;
  const bool second = warp > 0 && warp < kF3Rows - 1 && yu < A.ny;  // rows that update 2 runs on
  const bool out_a = second && lane >= H / 2 && lane < 32 - H / 2 && c0 < A.nx;
  const bool out_b = out_a && c0 + 1 < A.nx;

  const float *__restrict__ fin = static_cast<const float *>(A.fin);
  float *__restrict__ fout = static_cast<float *>(A.fout);
  const Rates<F2> R(F2(A.s1f, A.s1f), F2(A.s2f, A.s2f));
  const int t0 = launch_step(A);
  float lid[3] = {0.f, 0.f, 0.f};
  if (WALLS) {
#pragma unroll
    for (int a = 0; a < 3; ++a) lid[a] = float(2.0 * L::w(L::UP) * A.lid_u[a]);
  }

  // shared memory: own slots, and the neighbouring warps' y slots
  constexpr int WSTRIDE = fuse3_slots<L>() * 32;
  float2 *const own = fuse3_smem + warp * WSTRIDE + lane;
  constexpr int YOFF = 4 * NROW * 32, ZOFF = YOFF + 16 * 32;

  auto collide = [&](F2(&g)[4][Q], int z, int s) {
    const uint32_t n0 = (uint32_t)A.key_base + ((uint32_t)z * (uint32_t)A.ny + (uint32_t)y) * (uint32_t)A.nx;
    const uint2 key = make_uint2(node_key(n0 + c.xa, t0 + s), node_key(n0 + c.xb, t0 + s));
    F2 u[3], Pp, gv[3][Q], r;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int i = 0; i < Q; ++i) gv[a][i] = g[a][i];
    if constexpr (FORCE == FORCE_NONE) {
      const NoForce F[3] = {};
      node_moments<L, F2, false>(gv, F, u, Pp);
#pragma unroll
      for (int a = 0; a < 3; ++a) relax_velocity_set<L, F2, true>(g[a], a, u, Pp, R, F[a], key);
    } else {
      const int zc = wz ? min(max(z, 0), A.nz - 1) : z;
      const float *fp = static_cast<const float *>(A.force) + ((long long)zc * A.ny + y) * A.px;
      const F2 F[3] = {fuse_load(fp, c), fuse_load(fp + A.plane, c), fuse_load(fp + 2 * A.plane, c)};
      node_moments<L, F2, FORCE == FORCE_SCHEME2>(gv, F, u, Pp);
#pragma unroll
      for (int a = 0; a < 3; ++a) relax_velocity_set<L, F2, true>(g[a], a, u, Pp, R, F[a], key);
    }
    relax_rho_set<L, F2>(g[3], u, R, r);
  };

  const int iters = z1 - z0 + 2;
  for (int it = 0; it < iters; ++it) {
    const int r = z0 - 1 + it;
    F2 g[4][Q];
    {  // update 1 of plane r from memory
      const int zr = wz ? min(max(r, 0), A.nz - 1) : wrap(r, A.nz);
      const int zm = zr == 0 ? A.nz - 1 : zr - 1, zp = zr == A.nz - 1 ? 0 : zr + 1;
      const bool zlo = wz && r == 0, zhi = wz && r == A.nz - 1;
      const float *p0 = fin + ((long long)zr * A.ny + y) * A.px;
      const float *pym = fin + ((long long)zr * A.ny + ym) * A.px, *pyp = fin + ((long long)zr * A.ny + yp) * A.px;
      const float *pzm = fin + ((long long)zm * A.ny + y) * A.px, *pzp = fin + ((long long)zp * A.ny + y) * A.px;
      auto load_plane = [&](auto vec) {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const long long set = (long long)(s < 3 ? s + 1 : 0) * Q;  // velocity sets, then alpha = 0
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            // behind a y or z wall: the node's own opposite direction
            const bool wall = WALLS && ((L::c(i, 1) == 1 && ylo) || (L::c(i, 1) == -1 && yhi) ||
                                        (L::c(i, 2) == 1 && zlo) || (L::c(i, 2) == -1 && zhi));
            const float *p = wall ? p0 + (set + L::opp(i)) * A.plane
                                  : (L::c(i, 1) == 1    ? pym
                                     : L::c(i, 1) == -1 ? pyp
                                     : L::c(i, 2) == 1  ? pzm
                                     : L::c(i, 2) == -1 ? pzp
                                                        : p0) + (set + i) * A.plane;
            if constexpr (vec) g[s][i] = F2(__ldg(reinterpret_cast<const float2 *>(p + c.xa)));
            else g[s][i] = F2(__ldg(p + c.xa), __ldg(p + c.xb));
          }
        }
      };
      if (c.vec) load_plane(std::true_type{});
      else load_plane(std::false_type{});
      if (WALLS && (ylo || yhi || zlo || zhi)) {
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            if ((L::c(i, 1) == 1 && ylo) || (L::c(i, 1) == -1 && yhi) || (L::c(i, 2) == 1 && zlo)) g[s][i] = -g[s][i];
            if (L::c(i, 2) == -1 && zhi) {
              g[s][i] = -g[s][i];
              if (s < 3 && A.lid) g[s][i] += F2(lid[s < 3 ? s : 0], lid[s < 3 ? s : 0]);
            }
          }
      }
#pragma unroll
      for (int s = 0; s < 4; ++s) fuse_shift_row<L, WALLS>(g[s], c);
      collide(g, wz ? r : wrap(r, A.nz), 0);
    }
    // keep plane r of update 1, assemble the pull of plane q = r - 1
    const int q = r - 1, b = it & 1;
    float2 *const yw = own + YOFF + b * 8 * 32;                     // this plane's y directions
    const float2 *const yr = own + YOFF + (b ^ 1) * 8 * 32;         // plane q's, own row
    float2 *const zu = own + ZOFF + b * 4 * 32;                     // +z of plane q - 1, then of plane r
    float2 *const zv = own + ZOFF + (b ^ 1) * 4 * 32;               // +z of plane q
    const bool run = it >= 2 && second;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      F2 n[Q];
      if (run) {
        int k = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          if (L::c(i, 1) == 1) {  // from the row below; its own -y direction behind a wall
            n[i] = F2(ylo ? yr[(4 + s) * 32] : yr[s * 32 - WSTRIDE]);
            if (WALLS && ylo) n[i] = -n[i];
          } else if (L::c(i, 1) == -1) {
            n[i] = F2(yhi ? yr[s * 32] : yr[(4 + s) * 32 + WSTRIDE]);
            if (WALLS && yhi) n[i] = -n[i];
          } else if (L::c(i, 2) == 1) {
            n[i] = F2(zu[s * 32]);
          } else if (L::c(i, 2) == -1) {
            n[i] = g[s][i];
            if (WALLS && wz && q == A.nz - 1) {
              n[i] = -F2(zv[s * 32]);
              if (s < 3 && A.lid) n[i] += F2(lid[s < 3 ? s : 0], lid[s < 3 ? s : 0]);
            }
          } else {
            n[i] = F2(own[(s * NROW + k++) * 32]);
          }
        }
      }
      if (WALLS && wz && q == -1) {  // plane 0 pulls its own -z direction back
#pragma unroll
        for (int i = 0; i < Q; ++i)
          if (L::c(i, 2) == -1) zv[s * 32] = (-g[s][i]).f2();
      }
      fuse_shift_row<L, WALLS>(g[s], c);
      int k = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        if (L::c(i, 1) == 1) yw[s * 32] = g[s][i].f2();
        else if (L::c(i, 1) == -1) yw[(4 + s) * 32] = g[s][i].f2();
        else if (L::c(i, 2) == 1) zu[s * 32] = g[s][i].f2();
        else if (L::c(i, 2) == 0) own[(s * NROW + k++) * 32] = g[s][i].f2();
        if (run) g[s][i] = n[i];
      }
    }
    if (run) {
      collide(g, wz ? q : wrap(q, A.nz), 1);
      float *po = fout + ((long long)q * A.ny + yu) * A.px + c0;
      auto store_plane = [&](auto pair) {
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            float *p = po + ((long long)(s < 3 ? s + 1 : 0) * Q + i) * A.plane;
            if constexpr (pair) __stcs(reinterpret_cast<float2 *>(p), g[s][i].f2());
            else __stcs(p, g[s][i].x);
          }
      };
      if (out_b) store_plane(std::true_type{});
      else if (out_a) store_plane(std::false_type{});
    }
    __syncthreads();
  }
}

template <class L, bool WALLS, int FORCE>
cudaError_t launch_fused3d(const DevArgs &a, cudaStream_t s) {
  constexpr size_t smem = (size_t)kF3Rows * fuse3_slots<L>() * 32 * sizeof(float2);
  static OncePerDevice once;
  const cudaError_t set = allow_smem(once, k_update_fused3d<L, WALLS, FORCE>, smem);
  if (set != cudaSuccess) return set;
  const int tx = (a.nx + fuse_out<2>() - 1) / fuse_out<2>(), ty = (a.ny + kF3Out - 1) / kF3Out;
  const int seg = fuse3_plan(a.nx, a.ny, a.nz).seg;
  const long long blocks = (long long)tx * ty * ((a.nz + seg - 1) / seg);
  k_update_fused3d<L, WALLS, FORCE><<<(unsigned)blocks, 32 * kF3Rows, smem, s>>>(a, tx, ty, seg);
  return cudaGetLastError();
}

template <class L>
cudaError_t update_fused3d(bool walls, const DevArgs &a, cudaStream_t s) {
  if (a.scheme2)
    return walls ? launch_fused3d<L, true, FORCE_SCHEME2>(a, s) : launch_fused3d<L, false, FORCE_SCHEME2>(a, s);
  if (a.force)
    return walls ? launch_fused3d<L, true, FORCE_EQ321>(a, s) : launch_fused3d<L, false, FORCE_EQ321>(a, s);
  return walls ? launch_fused3d<L, true, FORCE_NONE>(a, s) : launch_fused3d<L, false, FORCE_NONE>(a, s);
}

}  // namespace mdf
