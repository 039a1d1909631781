// Forward 3x3 convolution on the 5th-generation tensor cores: persistent
// CTAs fed by the Tensor Memory Accelerator.
//
// What bounded the staged-halo kernel (mdf_nn_halo.cuh, kept for other
// alignments and for the tile overrides): one CTA per tile, whose four
// cp.async warps waited for the weights of every (16-channel chunk, tap) in
// turn; the tensor pipe was 8.5 % busy on the 32 -> 32 layer.  Here
//   - a CTA stays on its SM and walks over tiles, so filling the pipeline,
//     the barriers and TMEM are paid once, and the next tiles' loads run
//     under the current tile's MMAs and epilogue;
//   - the weights of its output channels stay in shared memory for every
//     tile where they fit (else they are loaded with each channel chunk);
//   - one thread loads: one TMA box for the zero-padded input halo of a tile
//     and chunk, one per tap for the weights (four warps of cp.async, two
//     units in flight behind the one signalled, took twice as long over the
//     network's layers: 785 us against 413);
//   - two to four accumulators in TMEM and two groups of four epilogue warps,
//     each taking every other tile: an epilogue (~400 instructions a warp,
//     one after the other) takes longer than the MMAs of a narrow tile.
//
// Geometry (as in the halo kernel).  The image is cut into column strips of
// TW <= 64 columns; a strip with a one-pixel border, row pitch P = TW + 2,
// is a 1D array of positions.  Output (r, c) of a strip is position o = r P
// + c (columns c >= TW are discarded) and tap (kh, kw) of it reads padded
// position o + kh P + kw.  A tile is M = 128 MT consecutive positions from
// o0 on; its halo box is the RB whole padded rows that hold them, which one
// TMA box (KC channels x P columns x RB rows; zeros outside the image)
// brings in as consecutive rows of 2 KC bytes, swizzled at that width.  Every
// tap is then the same K-major matrix from another start row: the swizzle is
// a function of the shared-memory address, which the tensor cores apply to
// the addresses they form, so the start may be any row.
//
// The sum over K runs over groups of 16 channels (32 on deep layers), the
// taps within a group: the order of the halo kernel's chunks, so the two give
// the same bits.  (Any other order is as accurate, but a rounding that flips
// in one layer travels through all that follow.)
//
// Measured (GB300, 8 samples, BF16 out, us against the halo kernel): 256^2
// 32 -> 32 22.8 / 42.0, 96 -> 32 48.8 / 91.7, 32 -> 96 30.9 / 127.7; 128^2
// 64 -> 64 16.5 / 29.4, 192 -> 64 34.5 / 65.7; 64^2 384 -> 128 24.5 / 73.2
// (1183 TFLOP/s); 32^2 256 -> 256 12.8 / 41.5.  With 32 output channels an
// MMA takes ~54 cycles to read its A rows (16 of them arithmetic); the
// full-resolution layers are held by the epilogues (E ~ 6400 cycles a tile)
// and stay 2 - 2.5 x above the time of their bytes.
//
// Every wait is bounded; after a time-out the CTA raises the error flag,
// waits (bounded) for the boxes and MMAs it issued, and frees TMEM.
#pragma once

#include "mdf_nn_wgrad_tc.cuh"

namespace mdfnn {

constexpr int PC_EPI = 8;                      // epilogue warps, in two groups
constexpr int PC_THREADS = 32 * (PC_EPI + 2);  // then the MMA and the TMA warp
constexpr int PC_MAX_STAGES = 6, PC_MAX_ACC = 4;

struct PersArgs {
  int P, TW, strips, tiles;  // strip pitch and width, strips, tiles per strip and image
  int RB;                    // padded rows of a halo box
  int ntiles;                // B strips tiles
  int per_cta, extra;        // tiles per CTA; the first `extra` CTAs take one more
  int BN;                    // output channels per CTA (multiple of 16, at most 128)
  int stages, resident;      // ring depth; 1: the weights stay in shared memory
  int accs, tcols;           // accumulators (2 or 4), TMEM columns
  int group;                 // channels summed before the next tap's (16 or 32)
};

// Padded rows that the reads of a tile can touch: positions o0 .. o0 + M - 1
// shifted by up to 2 P + 2, with o0 anywhere in its row.
__host__ __device__ constexpr int pers_rows(int MT, int P) { return (128 * MT + 3 * P) / P + 1; }
__host__ __device__ constexpr uint32_t pers_halo_bytes(int KC, int P, int RB) {
  return (uint32_t)(((long long)KC * 2 * P * RB + 1023) / 1024 * 1024);
}
__host__ __device__ constexpr uint32_t pers_w_bytes(int KC, int BN) { return 9u * (uint32_t)BN * KC * 2u; }
// Weights of all chunks (resident) or of every stage, the halo ring, the
// bias, the barriers; 1 KB of slack for the 1024-byte alignment.
__host__ __device__ inline size_t pers_smem_bytes(int Cin, int KC, int P, int RB, int BN, int stages, int resident) {
  const size_t w = (pers_w_bytes(KC, BN) + 1023) / 1024 * 1024;
  return 1024 + (resident ? (size_t)(Cin / KC) : (size_t)stages) * w + (size_t)stages * pers_halo_bytes(KC, P, RB) +
         (size_t)BN * 4 + (2 * PC_MAX_STAGES + 2 * PC_MAX_ACC + 1) * 8 + 16;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2,
                                            uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void st_global_32b(void *p, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// One lane's pixel row of 16 accumulator columns: bias, ReLU, store.
__device__ __forceinline__ void pers_store16(const ConvArgs &a, const float *bias, float *v, size_t m, int oc,
                                             bool vb, bool vf) {
  if (a.bias)
#pragma unroll
    for (int e = 0; e < 16; e += 4) {
      const float4 b = *reinterpret_cast<const float4 *>(bias + e);
      v[e] += b.x; v[e + 1] += b.y; v[e + 2] += b.z; v[e + 3] += b.w;
    }
  if (a.relu)
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = fmaxf(v[e], 0.f);
  if (a.y) {
    bf16 *dst = a.y + m * a.ldy + a.yoff + oc;
    if (vb && oc + 16 <= a.Cout) {
      uint32_t p[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) p[e] = pack_bf16(v[2 * e], v[2 * e + 1]);
      st_global_32b(dst, p);
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e)
        if (oc + e < a.Cout) dst[e] = __float2bfloat16_rn(v[e]);
    }
  }
  if (a.yf) {
    float *dst = a.yf + m * a.ldy + a.yoff + oc;
    if (vf && oc + 16 <= a.Cout) {
      uint32_t p[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int e = 0; e < 8; ++e) p[e] = __float_as_uint(v[8 * h + e]);
        st_global_32b(dst + 8 * h, p);
      }
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e)
        if (oc + e < a.Cout) dst[e] = v[e];
    }
  }
}

template <int KC, int MT>
__global__ void __launch_bounds__(PC_THREADS)
    k_conv_fwd_pers(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap, ConvArgs a,
                    PersArgs g, int *err) {
  static_assert(KC == 16 || KC == 32 || KC == 64, "channel chunk");
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int NC = a.Cin / KC, S = g.stages;
  const uint32_t hbytes = pers_halo_bytes(KC, g.P, g.RB), hbox = (uint32_t)(KC * 2 * g.P * g.RB);
  const uint32_t wtap = (uint32_t)g.BN * KC * 2, wbox = 9 * wtap, wslot = (wbox + 1023) / 1024 * 1024;
  const uint32_t w0 = smem_u32(smem), h0 = w0 + (g.resident ? (uint32_t)NC : (uint32_t)S) * wslot;
  float *sbias = reinterpret_cast<float *>(smem + (h0 - w0) + (size_t)S * hbytes);
  uint64_t *full = reinterpret_cast<uint64_t *>(sbias + g.BN);
  uint64_t *empty = full + PC_MAX_STAGES;
  uint64_t *tfull = empty + PC_MAX_STAGES;
  uint64_t *tempty = tfull + PC_MAX_ACC;
  uint64_t *done = tempty + PC_MAX_ACC;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = blockIdx.y * g.BN;
  const long long limit = 2000000000LL;
  // this CTA's tiles: a contiguous run, so that no role divides per tile
  const int t0 = (int)blockIdx.x * g.per_cta + min((int)blockIdx.x, g.extra);
  const int t1 = t0 + g.per_cta + ((int)blockIdx.x < g.extra ? 1 : 0);

  if (warp == PC_EPI) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)g.tcols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    for (int k = 0; k < S; ++k) {
      mbar_init(&full[k], 1);
      mbar_init(&empty[k], 1);
    }
    for (int k = 0; k < g.accs; ++k) {
      mbar_init(&tfull[k], 1);
      mbar_init(&tempty[k], 128);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  for (int k = tid; k < g.BN; k += PC_THREADS) sbias[k] = a.bias && n0 + k < a.Cout ? a.bias[n0 + k] : 0.f;
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = *tmem_slot;

  bool ok = true;
  if (warp == PC_EPI + 1) {
    if (lane == 0) {
      // ---------------- loads: unit u = (tile, chunk) into stage u % S
      int u = 0, tile = t0 % g.tiles, strip = t0 / g.tiles % g.strips, b = t0 / g.tiles / g.strips;
      for (int t = t0; t < t1 && ok; ++t) {
        const int row0 = tile * 128 * MT / g.P, col0 = strip * g.TW;
        for (int c = 0; c < NC; ++c, ++u) {
          const int s = u % S;
          if (u >= S && !mbar_wait(&empty[s], (uint32_t)((u / S - 1) & 1), limit)) {
            ok = false;
            break;
          }
          const bool weights = !g.resident || u < NC;
          mbar_expect_tx(&full[s], hbox + (weights ? wbox : 0u));
          tma_load_4d(h0 + (uint32_t)s * hbytes, &xmap, c * KC, col0 - 1, row0 - 1, b, &full[s]);
          if (weights) {
            const uint32_t dst = w0 + (uint32_t)(g.resident ? c : s) * wslot;
            for (int k = 0; k < 9; ++k) tma_load_3d(dst + k * wtap, &wmap, c * KC, k, n0, &full[s]);
          }
        }
        if (++tile == g.tiles) {
          tile = 0;
          if (++strip == g.strips) {
            strip = 0;
            ++b;
          }
        }
      }
      // every box issued has landed before the CTA can leave
      for (int i = u > S ? u - S : 0; i < u; ++i)
        if (!mbar_wait(&full[i % S], (uint32_t)((i / S) & 1), limit)) ok = false;
    }
  } else if (warp == PC_EPI) {
    if (lane == 0) {
      // ---------------- MMAs
      const uint32_t idesc = umma_idesc_bf16(128, g.BN);
      const uint64_t swz = (uint64_t)umma_swizzle(2 * KC) << 61;
      int u = 0, acc = 0, used = 0, o0 = t0 % g.tiles * 128 * MT;
      for (int t = t0; t < t1 && ok; ++t) {
        if (used && !mbar_wait(&tempty[acc], (uint32_t)((used - 1) & 1), limit)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        const uint32_t off = (uint32_t)(o0 % g.P);  // o0 in its row
        const uint32_t d = tmem + (uint32_t)(acc * MT * g.BN);
        for (int c = 0; c < NC; ++c, ++u) {
          const int s = u % S;
          if (!mbar_wait(&full[s], (uint32_t)((u / S) & 1), limit)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;\n");
          const uint64_t hd = umma_smem_desc(h0 + (uint32_t)s * hbytes, 16, 16 * KC) | swz;
          const uint64_t wd = umma_smem_desc(w0 + (uint32_t)(g.resident ? c : s) * wslot, 16, 16 * KC) | swz;
          // channel groups of G, the taps within a group, K = 16 steps within a tap
          auto mmas = [&](auto group) {
            constexpr int G = decltype(group)::value;
#pragma unroll
            for (int q = 0; q < KC / G; ++q)
#pragma unroll
              for (int k = 0; k < 9; ++k) {
                const uint32_t row = off + (uint32_t)(k / 3 * g.P + k % 3);
#pragma unroll
                for (int ks = q * (G / 16); ks < (q + 1) * (G / 16); ++ks)
#pragma unroll
                  for (int mt = 0; mt < MT; ++mt)
                    tc_mma(d + (uint32_t)(mt * g.BN), hd + (uint64_t)((row + 128 * mt) * (KC / 8) + 2 * ks),
                           wd + (uint64_t)(k * (wtap >> 4) + 2 * ks), idesc, (c | q | k | (ks % (G / 16))) ? 1u : 0u);
              }
          };
          if constexpr (KC >= 32) {
            if (g.group == 32) mmas(std::integral_constant<int, 32>{});
            else mmas(std::integral_constant<int, 16>{});
          } else {
            mmas(std::integral_constant<int, 16>{});
          }
          tc_commit(&empty[s]);
        }
        if (ok) tc_commit(&tfull[acc]);
        if (++acc == g.accs) {
          acc = 0;
          ++used;
        }
        o0 += 128 * MT;
        if (o0 == g.tiles * 128 * MT) o0 = 0;
      }
      tc_commit(done);  // arrives once every MMA issued above has completed
      if (!mbar_wait(done, 0u, limit)) ok = false;
    }
  } else {
    // ---------------- epilogue: warps 0-3 take the CTA's even tiles, 4-7 the
    // odd ones; warp w holds positions 32 (w & 3) .. of each M tile
    const bool vb = a.y && (((a.ldy | a.yoff) & 15) == 0) && (((uintptr_t)a.y & 31) == 0);
    const bool vf = a.yf && (((a.ldy | a.yoff) & 7) == 0) && (((uintptr_t)a.yf & 31) == 0);
    const int half = warp >> 2, quad = warp & 3;
    const int q128 = 128 / g.P, m128 = 128 - q128 * g.P;  // 128 positions in rows and columns
    int tile = t0 % g.tiles, strip = t0 / g.tiles % g.strips, b = t0 / g.tiles / g.strips;
    int acc = 0, used = 0;
    int o = tile * 128 * MT + quad * 32 + lane, r = o / g.P, cc = o - r * g.P;  // this lane's position
    for (int t = t0; t < t1; ++t) {
      const bool mine = ((t - t0) & 1) == half;
      if (mine) {
        if (!mbar_wait(&tfull[acc], (uint32_t)(used & 1), limit)) ok = false;
        if (!__all_sync(0xffffffffu, ok)) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n");
      }
      const int col0 = strip * g.TW, TWs = min(g.TW, a.W - col0);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        if (mine) {
          const size_t m = ((size_t)b * a.H + r) * a.W + col0 + cc;
          const bool live = r < a.H && cc < TWs;
          const uint32_t d = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)((acc * MT + mt) * g.BN);
          int c0 = 0;
#pragma unroll 1
          for (; c0 + 32 <= g.BN; c0 += 32) {
            float v[32];
            tc_ld<32>(d + c0, v);
            if (live && n0 + c0 < a.Cout) pers_store16(a, sbias + c0, v, m, n0 + c0, vb, vf);
            if (live && n0 + c0 + 16 < a.Cout) pers_store16(a, sbias + c0 + 16, v + 16, m, n0 + c0 + 16, vb, vf);
          }
          if (c0 < g.BN) {
            float v[16];
            tc_ld<16>(d + c0, v);
            if (live && n0 + c0 < a.Cout) pers_store16(a, sbias + c0, v, m, n0 + c0, vb, vf);
          }
        }
        r += q128;
        cc += m128;
        if (cc >= g.P) {
          cc -= g.P;
          ++r;
        }
      }
      if (mine) {
        asm volatile("tcgen05.fence::before_thread_sync;\n");
        mbar_arrive(&tempty[acc]);
      }
      if (++acc == g.accs) {
        acc = 0;
        ++used;
      }
      if (++tile == g.tiles) {
        tile = 0;
        o = quad * 32 + lane;
        r = o / g.P;
        cc = o - r * g.P;
        if (++strip == g.strips) {
          strip = 0;
          ++b;
        }
      }
    }
  }
  if (!ok) atomicExch(err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  if (warp == PC_EPI) {
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"((uint32_t)g.tcols));
  }
}

}  // namespace mdfnn
