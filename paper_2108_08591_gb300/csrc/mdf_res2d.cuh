// A small 2D FP32 lattice kept on chip for all updates of a call.
//
// What bounds a small lattice is not memory but the launch and the latency
// of each update (64^2: 4.2 us per update in launches of one, 3.1 in fused
// launches of four, for 0.03 us of arithmetic).  Here one thread-block cluster
// holds the whole lattice: each CTA a run of rows, all populations in two
// buffers of its shared memory.  An update pulls from one buffer, its edge
// rows from the neighbouring CTAs' shared memory, collides and stores into
// the other; one cluster barrier ends it.  Global memory is read once before
// the first update and written once after the last.
//
// The arithmetic per node is the scalar kernel's (collide_node with the same
// dither draws), so the bits are those of single updates.
#pragma once

#include <cooperative_groups.h>

#include "mdf_fuse2d.cuh"

namespace mdf {

constexpr int kResMaxTeamNodes = 1800;  // of a CTA in a batch of cavities
constexpr size_t kResMaxSmem = 2ull * 15 * kResMaxTeamNodes * sizeof(float);  // of a CTA
// Where a node's populations come from: one pointer per direction (set 0,
// current buffer; local or of a neighbouring CTA), and what the walls make of
// the value.
template <int Q> struct ResPull {
  const float *q[Q];
  unsigned neg;  // bit i: bounced back, negated
  bool lid;      // the -y direction bounces off the lid
};

// `steps` updates of lattice G by this thread's cluster; rcap: rows a CTA's
// buffers are laid out for.  PAIR: a thread takes its nodes two at a time as
// the lanes of an FP32 pair (any two: every access is a 4-byte one), for CTAs
// with more nodes than threads, which the issue slots bound; with a node a
// thread the latency of one collision does, and the scalar form is shorter.
// The lattice is held by CTAs first .. first + C - 1 of the cluster, of which
// this is CTA first + rank; the barriers are the whole cluster's.  nodes = 0
// (G.ny = 0) takes part in them alone.
template <class L, bool WALLS, int FORCE, bool PAIR>
__device__ __forceinline__ void res_run(const FuseLattice &G, bool with_rho, int steps, bool save, int rcap,
                                        float *buf, int first, int C, int rank) {
  namespace cg = cooperative_groups;
  using TC = typename std::conditional<PAIR, F2, float>::type;
  constexpr int Q = L::Q, NP = PAIR ? 2 : 1;
  const cg::cluster_group cl = cg::this_cluster();
  const int base = G.ny / C, extra = G.ny - base * C;
  const int rows = base + (rank < extra ? 1 : 0), y0 = rank * base + min(rank, extra);
  const int lo = rank == 0 ? C - 1 : rank - 1, hi = rank == C - 1 ? 0 : rank + 1;
  const int lo_last = base + (lo < extra ? 1 : 0) - 1;
  const bool wx = WALLS && G.wx, wy = WALLS && G.wy;
  const int stride = rcap * G.nx;  // of a direction
  const int pops = (2 + (with_rho ? 1 : 0)) * Q;
  const int half = pops * stride;  // of a buffer
  const int T = (int)blockDim.x, tid = (int)threadIdx.x;
  const int nodes = rows * G.nx;
  const int dy = T / G.nx, dx = T - dy * G.nx;  // a thread's step through its nodes
  const int yf = tid / G.nx, xf = tid - yf * G.nx;
  auto advance = [&](int &x, int &y) {
    x += dx;
    y += dy;
    if (x >= G.nx) { x -= G.nx; ++y; }
  };

  {
    int y = yf, x = xf;
    for (int k = tid; k < nodes; k += T, advance(x, y)) {
      const float *src = G.fin + (long long)(y0 + y) * G.px + x;
      float v[3 * Q];
#pragma unroll
      for (int p = 0; p < 3 * Q; ++p) v[p] = p < pops ? __ldg(src + (long long)p * G.plane) : 0.f;
#pragma unroll
      for (int p = 0; p < 3 * Q; ++p)
        if (p < pops) buf[p * stride + k] = v[p];
    }
  }
  cl.sync();
  const float *const rlo = cl.map_shared_rank(buf, first + lo) + lo_last * G.nx;  // row y0 - 1
  const float *const rhi = cl.map_shared_rank(buf, first + hi);                 // row y0 + rows
  const Rates<TC> R(TC(G.s1), TC(G.s2));

  for (int s = 0; s < steps; ++s) {
    const int b = (s & 1) * half;
    float *const out = buf + (half - b);
    int y = yf, x = xf;
    for (int k = tid; k < nodes;) {
      ResPull<Q> P[NP];
      int kk[NP], node[NP];
      uint32_t key[NP];
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const bool past = j > 0 && k >= nodes;  // an odd last node: its pair repeats it
        if (past) {
          kk[j] = kk[0];
          node[j] = node[0];
          key[j] = key[0];
          P[j] = P[0];
          continue;
        }
        const float *const r0 = buf + b + (k - x);
        const float *const rm = y > 0 ? r0 - G.nx : rlo + b;
        const float *const rp = y < rows - 1 ? r0 + G.nx : rhi + b;
        const int xm = x == 0 ? G.nx - 1 : x - 1, xp = x == G.nx - 1 ? 0 : x + 1;
        P[j].neg = 0u;
        P[j].lid = false;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const float *p = (L::c(i, 1) == 1 ? rm : L::c(i, 1) == -1 ? rp : r0) +
                           (L::c(i, 0) == 1 ? xm : L::c(i, 0) == -1 ? xp : x) + i * stride;
          if (WALLS && moving<L>(i)) {  // the node's own opposite direction, negated
            const bool wall = L::c(i, 0) == 1    ? wx && x == 0
                              : L::c(i, 0) == -1 ? wx && x == G.nx - 1
                              : L::c(i, 1) == 1  ? wy && y0 + y == 0
                                                 : wy && y0 + y == G.ny - 1;
            if (wall) {
              p = r0 + x + L::opp(i) * stride;
              P[j].neg |= 1u << i;
              if (L::c(i, 1) == -1) P[j].lid = G.lid;
            }
          }
          P[j].q[i] = p;
        }
        kk[j] = k;
        node[j] = (y0 + y) * G.px + x;
        key[j] = node_key(G.key0 + (uint32_t)((y0 + y) * G.nx + x), G.t0 + s);
        k += T;
        advance(x, y);
      }
      TC g[2][Q], h[Q];
      auto pull = [&](TC(&v)[Q], int set, int e) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          float w[NP];
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            w[j] = P[j].q[i][set * Q * stride];
            if (WALLS && moving<L>(i)) {
              if ((P[j].neg >> i) & 1u) w[j] = -w[j];
              if (e >= 0 && L::c(i, 1) == -1 && P[j].lid) w[j] += G.lid_u[e >= 0 ? e : 0];
            }
          }
          if constexpr (PAIR) v[i] = F2(w[0], w[1]);
          else v[i] = w[0];
        }
      };
      pull(g[0], with_rho ? 1 : 0, 0);
      pull(g[1], with_rho ? 2 : 1, 1);
      if (with_rho) pull(h, 0, -1);
      typename NodeKey<TC>::T kt;
      if constexpr (PAIR) kt = make_uint2(key[0], key[1]);
      else kt = key[0];
      TC u[2], Pp;
      auto relax = [&](const auto &F) {
        node_moments<L, TC, FORCE == FORCE_SCHEME2>(g, F, u, Pp);
#pragma unroll
        for (int a = 0; a < 2; ++a) relax_velocity_set<L, TC, true>(g[a], a, u, Pp, R, F[a], kt);
      };
      if constexpr (FORCE == FORCE_NONE) {
        const NoForce F[2] = {};
        relax(F);
      } else {
        TC F[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const float *f = G.force + a * G.plane;
          if constexpr (PAIR) F[a] = F2(__ldg(f + node[0]), __ldg(f + node[1]));
          else F[a] = __ldg(f + node[0]);
        }
        relax(F);
      }
      if (with_rho) {
        TC r;
        relax_rho_set<L, TC>(h, u, R, r);
      }
      auto lane = [](TC v, int j) {
        if constexpr (PAIR) return j == 0 ? v.x : v.y;
        else return v;
      };
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        if (save && s == 0) {
#pragma unroll
          for (int a = 0; a < 2; ++a) G.usave[a * G.plane + node[j]] = lane(u[a], j);
        }
        float *o = out + kk[j];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          o[((with_rho ? 1 : 0) * Q + i) * stride] = lane(g[0][i], j);
          o[((with_rho ? 2 : 1) * Q + i) * stride] = lane(g[1][i], j);
          if (with_rho) o[i * stride] = lane(h[i], j);
        }
      }
    }
    cl.sync();  // every pull of this update is done, every store visible
  }

  const float *const last = buf + (steps & 1) * half;
  int y = yf, x = xf;
  for (int k = tid; k < nodes; k += T, advance(x, y)) {
    float *dst = G.fout + (long long)(y0 + y) * G.px + x;
#pragma unroll
    for (int p = 0; p < 3 * Q; ++p)
      if (p < pops) dst[(long long)p * G.plane] = last[p * stride + k];
  }
}

template <class L, bool WALLS, int FORCE, bool PAIR>
__global__ void __launch_bounds__(kResThreads) k_resident2d(const DevArgs A, int steps, int rcap) {
  extern __shared__ float res_smem[];
  const cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  res_run<L, WALLS, FORCE, PAIR>(fuse_lattice<L>(A), A.with_rho != 0, steps, false, rcap, res_smem, 0,
                                 (int)cl.num_blocks(), (int)cl.block_rank());
}

template <class Kernel, class... Args>
cudaError_t res_launch(Kernel kernel, int clusters, const ResShape &r, int threads, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * r.ctas));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = r.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)r.ctas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}
// Shared memory and cluster size beyond the defaults.
template <class Kernel>
cudaError_t res_configure(Kernel kernel) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResMaxSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

// Clusters of the largest size that the device holds at once.
template <class Kernel>
cudaError_t res_clusters(Kernel kernel, int threads, size_t smem, int *n) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kResMaxCluster);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kResMaxCluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(n, kernel, &cfg);
}
// Whether the current device runs clusters of the largest size (configures
// the kernel for them).
template <class Kernel>
bool res_available(OncePerDevice &once, Kernel kernel) {
  const cudaError_t e = once([&] {
    int n = 0;
    cudaError_t s = res_configure(kernel);
    if (s == cudaSuccess) s = res_clusters(kernel, kResThreads, kResMaxSmem, &n);
    return s != cudaSuccess || n > 0 ? s : cudaErrorNotSupported;
  });
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess;
}

template <class L, bool WALLS, int FORCE, bool PAIR>
cudaError_t launch_resident2d_p(const ResShape &r, const DevArgs &a, int steps, cudaStream_t s) {
  static OncePerDevice once;
  const cudaError_t set = once([] { return res_configure(k_resident2d<L, WALLS, FORCE, PAIR>); });
  if (set != cudaSuccess) return set;
  return res_launch(k_resident2d<L, WALLS, FORCE, PAIR>, 1, r, res_threads(r.rows * a.nx), s, a, steps, r.rows);
}

template <class L, bool WALLS, int FORCE>
cudaError_t launch_resident2d(const DevArgs &a, int steps, cudaStream_t s) {
  const ResShape r = res_shape(a.nx, a.ny, L::Q, 2 + a.with_rho);
  if (!r.ctas) return cudaErrorInvalidValue;
  return res_pairs(r.rows * a.nx) ? launch_resident2d_p<L, WALLS, FORCE, true>(r, a, steps, s)
                                  : launch_resident2d_p<L, WALLS, FORCE, false>(r, a, steps, s);
}

template <class L>
cudaError_t update_resident2d(bool walls, const DevArgs &a, int steps, cudaStream_t s) {
  if (a.scheme2)
    return walls ? launch_resident2d<L, true, FORCE_SCHEME2>(a, steps, s)
                 : launch_resident2d<L, false, FORCE_SCHEME2>(a, steps, s);
  if (a.force)
    return walls ? launch_resident2d<L, true, FORCE_EQ321>(a, steps, s)
                 : launch_resident2d<L, false, FORCE_EQ321>(a, steps, s);
  return walls ? launch_resident2d<L, true, FORCE_NONE>(a, steps, s)
               : launch_resident2d<L, false, FORCE_NONE>(a, steps, s);
}

}  // namespace mdf
