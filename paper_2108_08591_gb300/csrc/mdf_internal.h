// Host/device interface between the C-ABI layer (mdf_api.cu) and the
// per-lattice kernel translation units.  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "mdf_device.h"

namespace mdf {

// Everything a kernel launch needs, as plain pointers and sizes.
struct DevArgs {
  const void *fin;               // current populations (post-collision, pre-stream)
  void *fout;                    // next populations
  const uint8_t *mask;           // link mask [plane] or null (periodic)
  const void *force;             // [d][plane] body force (compute type) or null
  int scheme2;                   // 1: Scheme II forcing (Eq. 2-3c, 2-7a) with a force set
  int aa;                        // 0: two buffers, pull; in-place AA pattern: 1 even, 2 odd phase
  const void *min;               // moments [K][plane] read (equilibrium-shifted storage)
  void *mout;                    // moments written
  int nx, ny, nz, px;            // grid and padded x pitch
  long long plane;               // px * ny * nz
  int with_rho;                  // 1: set 0 is the alpha = 0 set
  int vx;                        // x-nodes per thread of the update kernel (1: scalar)
  int block;                     // threads per block of the update kernel
  double s1, s2;                 // relaxation rates (s0 never acts: m0 = m0eq)
  float s1f, s2f;                // the same rates rounded to FP32 on the host
  double lid_u[3];               // lid velocity
  int wall[3], lid;              // walls per axis, lid on the + face of the last axis
  // derived-field outputs (dense [N] layout), each nullable
  double *P, *u, *rho, *G, *div, *S, *sigma, *omega;
  // init inputs (dense FP64 on the device); Gin [d][d][N] nullable
  const double *Pin, *uin, *Gin;
  // reductions
  double *partials;              // [blocks][k] block partial sums
  double *uprev;                 // [d][N] previous velocity (residual)
  double *result;                // [k] final sums
  int *nonfinite;                // set to 1 when a non-finite value is met
  // dithered rounding of FP32 storage: time step = *clock + tk; the node
  // key is that of global node index key_base + dense local index
  const int *clock;              // device step counter of the launch group
  int tk;                        // this launch's offset in its group
  long long key_base;            // global index of local node 0 (slabs)
};

enum Mode { MODE_STEP = 0, MODE_STEP_FIELDS = 1, MODE_FIELDS = 2 };
enum Storage { ST_F32 = 0, ST_F16 = 1, ST_BF16 = 2, ST_F64 = 3, ST_F16EQ = 4, ST_BF16EQ = 5 };
enum ReduceKind { RED_SUMS = 0, RED_RESIDUAL = 1 };

// Block width along x of the auxiliary kernels, and the largest block of the
// update kernels (their width is a launch parameter).
constexpr int kBlockX = 128;
constexpr int kMaxBlock = 256;
// Blocks of the grid-stride reduction pass (a multiple of the 152 SMs).
constexpr int kReduceBlocks = 152 * 4;
constexpr int kReduceThreads = 256;

// Per-lattice launchers (mdf_d2q5.cu, mdf_d3q7.cu).

cudaError_t launch_update_d2q5(int storage, int mode, bool walls, const DevArgs &a,
                               cudaStream_t s);
cudaError_t launch_init_d2q5(int storage, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_reduce_d2q5(int storage, bool walls, int kind, const DevArgs &a,
                               cudaStream_t s);
cudaError_t launch_update_d3q7(int storage, int mode, bool walls, const DevArgs &a,
                               cudaStream_t s);
cudaError_t launch_init_d3q7(int storage, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_reduce_d3q7(int storage, bool walls, int kind, const DevArgs &a,
                               cudaStream_t s);

cudaError_t launch_mask_d2q5(const int wall[3], int lid, const DevArgs &a, uint8_t *mask,
                             cudaStream_t s);
cudaError_t launch_mask_d3q7(const int wall[3], int lid, const DevArgs &a, uint8_t *mask,
                             cudaStream_t s);

// Lattices without a rest direction (mdf_d2q4.cu, mdf_d3q6.cu): the
// rest-shifted storage types only.
cudaError_t launch_update_d2q4(int storage, int mode, bool walls, const DevArgs &a,
                               cudaStream_t s);
cudaError_t launch_init_d2q4(int storage, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_reduce_d2q4(int storage, bool walls, int kind, const DevArgs &a,
                               cudaStream_t s);
cudaError_t launch_mask_d2q4(const int wall[3], int lid, const DevArgs &a, uint8_t *mask,
                             cudaStream_t s);
cudaError_t launch_update_d3q6(int storage, int mode, bool walls, const DevArgs &a,
                               cudaStream_t s);
cudaError_t launch_init_d3q6(int storage, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_reduce_d3q6(int storage, bool walls, int kind, const DevArgs &a,
                               cudaStream_t s);
cudaError_t launch_mask_d3q6(const int wall[3], int lid, const DevArgs &a, uint8_t *mask,
                             cudaStream_t s);

// Two fused updates of a 3D lattice (mdf_fuse3d.cuh): planes per z segment,
// and whether they pay.  Blocks of kFuse3Rows rows (two fewer stored) x 64
// columns (60 stored), two per SM; a block is counted at 5.2 us per plane and
// 1.2 planes to fill.  The lines are in that count per node, where the pair
// and two single updates took the same time over 30 boxes of 49 .. 315 nodes
// a side (D3Q7): 69 ps; 76 with walls, whose mask slows the single update
// more (41 -> 49 ps a node at 235 x 118 x 161); 60 with a force, which slows the
// pair by 13 % there and the two by 3 %; 66 with both.  128^3 (92 us the pair, 74 the
// two) and smaller boxes stay single, 60 x 60 x 200 (31 / 37), 190 x 202 x 178
// (242 / 255) and 145 x 267 x 175 (526 / 562) go fused; of walled boxes with a
// force, 192 x 229 x 78 (358 / 301) stays single and 235 x 118 x 161
// (388 / 437) goes fused.
constexpr int kSMs = 152;  // of a GB300
constexpr int kFuse3Rows = 8;
struct Fuse3Plan {
  int seg;
  double us;  // of two updates
};
inline Fuse3Plan fuse3_plan(int nx, int ny, int nz) {
  const long long tiles = (long long)((nx + 59) / 60) * ((ny + kFuse3Rows - 3) / (kFuse3Rows - 2));
  Fuse3Plan p{nz, 0.0};
  for (int k = nz; k >= 1; k = k > 1 ? (k * 15 / 16 > 1 ? k * 15 / 16 : 1) : 0) {
    const long long blocks = tiles * ((nz + k - 1) / k);
    const double us = 5.2 * (double)((blocks + 2 * kSMs - 1) / (2 * kSMs)) * (k + 1.2);
    if (p.us == 0.0 || us < p.us) p = {k, us};
  }
  return p;
}
inline bool fuse3_pays(int nx, int ny, int nz, bool walls, bool force) {
  const double ps = walls ? (force ? 66.0 : 76.0) : (force ? 60.0 : 69.0);
  return fuse3_plan(nx, ny, nz).us < 1e-6 * ps * nx * (double)ny * nz;
}

constexpr int kFuseWarps = 2;  // independent warps per block of the 2D fused kernel

// The resident kernel's launches (mdf_res2d.cuh).
constexpr int kResThreads = 512;
constexpr int kResMaxCluster = 16;                // needs the non-portable size
// Most nodes of a CTA.  Up to here the resident kernel is the faster one: us
// per update against fused launches, 16^2 0.62 / 3.1, 64^2 0.75 / 3.1 (and
// 4.2 in launches of one), 96^2 1.47 / 3.1, 128^2 (1024 nodes a CTA) 1.98 /
// 3.2; at 144^2 (1296) 2.95 / 3.2 and at 170^2 3.37 / 3.4 it no longer pays
// for its start.
constexpr int kResMaxNodes = 1200;
constexpr int kResMaxSteps = 1 << 14;  // updates of one launch
// Fewest updates that pay for reading and writing the lattice once more than
// a fused launch would: with two nodes a thread four (128^2: 4.7 us per update
// against 5.8 of single ones; with two updates 8.4 against 7.5).
inline int res_min_steps(int nodes) { return nodes > kResThreads ? 4 : 2; }

// CTAs of a cluster for nx x ny nodes, and the shared memory of each; 0 when
// it does not fit.
struct ResShape {
  int ctas, rows;  // rows: the most of a CTA
  size_t smem;
};
inline ResShape res_shape(int nx, int ny, int q, int nsets) {
  const int c = std::min(ny, kResMaxCluster), rows = (ny + c - 1) / c;
  if ((long long)rows * nx > kResMaxNodes) return {0, 0, 0};
  return {c, rows, 2ull * nsets * q * rows * (size_t)nx * sizeof(float)};
}

// Threads of a CTA for its nodes: whole warps, a node each, or two each (as a
// pair) beyond the limit.
inline bool res_pairs(int nodes) { return nodes > kResThreads; }
inline int res_threads(int nodes) {
  const int n = res_pairs(nodes) ? (nodes + 1) / 2 : nodes;
  return std::min(kResThreads, (n + 31) / 32 * 32);
}

// K updates in one launch (FP32, two buffers, all d + 1 sets): 2 or 4 in 2D
// (ny >= K), 2 in 3D.
cudaError_t launch_fused_d2q5(int K, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_fused_d2q4(int K, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_fused_d3q7(int K, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_fused_d3q6(int K, bool walls, const DevArgs &a, cudaStream_t s);

// `steps` updates (at most 16384) of a small 2D FP32 lattice in one launch of
// one thread-block cluster (mdf_res2d.cuh), and the fewest updates for which
// that pays (0: it does not fit).
cudaError_t launch_resident_d2q5(int steps, bool walls, const DevArgs &a, cudaStream_t s);
cudaError_t launch_resident_d2q4(int steps, bool walls, const DevArgs &a, cudaStream_t s);
int resident_steps_d2q5(int nx, int ny, int nsets);
int resident_steps_d2q4(int nx, int ny, int nsets);

// The launchers of one lattice (resident: 2D only).
struct LatticeLaunch {
  cudaError_t (*update)(int storage, int mode, bool walls, const DevArgs &a, cudaStream_t s);
  cudaError_t (*init)(int storage, bool walls, const DevArgs &a, cudaStream_t s);
  cudaError_t (*reduce)(int storage, bool walls, int kind, const DevArgs &a, cudaStream_t s);
  cudaError_t (*mask)(const int wall[3], int lid, const DevArgs &a, uint8_t *mask, cudaStream_t s);
  cudaError_t (*fused)(int K, bool walls, const DevArgs &a, cudaStream_t s);
  cudaError_t (*resident)(int steps, bool walls, const DevArgs &a, cudaStream_t s);
  int (*resident_steps)(int nx, int ny, int nsets);
};
inline const LatticeLaunch *lattice_launch(int d, int q) {
  static const LatticeLaunch d2q5{launch_update_d2q5, launch_init_d2q5, launch_reduce_d2q5, launch_mask_d2q5,
                                  launch_fused_d2q5, launch_resident_d2q5, resident_steps_d2q5};
  static const LatticeLaunch d3q7{launch_update_d3q7, launch_init_d3q7, launch_reduce_d3q7, launch_mask_d3q7,
                                  launch_fused_d3q7, nullptr, nullptr};
  static const LatticeLaunch d2q4{launch_update_d2q4, launch_init_d2q4, launch_reduce_d2q4, launch_mask_d2q4,
                                  launch_fused_d2q4, launch_resident_d2q4, resident_steps_d2q4};
  static const LatticeLaunch d3q6{launch_update_d3q6, launch_init_d3q6, launch_reduce_d3q6, launch_mask_d3q6,
                                  launch_fused_d3q6, nullptr, nullptr};
  if (d == 2) return q == 5 ? &d2q5 : q == 4 ? &d2q4 : nullptr;
  if (d == 3) return q == 7 ? &d3q7 : q == 6 ? &d3q6 : nullptr;
  return nullptr;
}

// Sets the device step counter read by the update kernels of a launch group.
cudaError_t launch_set_clock(int *clock, int value, cudaStream_t s);
// Second reduction pass: sums `nblocks` x `k` partials in a fixed order.
cudaError_t launch_reduce_final(const DevArgs &a, int nblocks, int k, cudaStream_t s);
// Dense FP64 [d][N] -> padded [d][plane] in FP32 (f64 = false) or FP64.
cudaError_t launch_pad_force(const double *src, void *dst, bool f64, int d, int nx, int ny,
                             int nz, int px, cudaStream_t s);

}  // namespace mdf
