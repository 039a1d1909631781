// Kernels of the warm-start network: 3x3 convolutions as implicit GEMMs on
// the BF16 tensor cores (mma.sync m16n8k16, FP32 accumulation; operands
// staged in shared memory by cp.async and fed by ldmatrix), and the
// element-wise pieces (ReLU gradient, 2x2 average pooling, nearest 2x
// upsampling, MSE, Adam).  Activations are NHWC BF16; convolution weights
// are [Cout][3][3][Cin] BF16 with FP32 master copies.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace mdfnn {

typedef __nv_bfloat16 bf16;

// ---------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// 16-byte global -> shared copy; valid = false writes 16 zero bytes.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, bool valid) {
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(smem)), "l"(gmem),
               "r"(n));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
// D += A (16x16, row-major) * B (16x8, column-major), BF16 in, FP32 out.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------
// Forward convolution: y[m][o] = sum_k A[m][k] W[o][k] (+ bias, ReLU), with
// m = (b, h, w) a pixel, k = (kh, kw, i) and A the zero-padded 3x3 window
// (im2col, formed on the fly).  Tile 64 pixels x 64 outputs x 32 of K per
// step, 4 warps of 32 x 32, double-buffered.  Needs Cin % 8 == 0.
// ---------------------------------------------------------------------------
struct ConvArgs {
  const bf16 *x;      // [B][H][W][Cin]
  const bf16 *w;      // [Cout][9 * Cin]
  const float *bias;  // [Cout] or null
  bf16 *y;            // output (BF16), element [m][yoff + o] with row stride ldy; nullable
  float *yf;          // output (FP32), same indexing; nullable
  int B, H, W, Cin, Cout;
  int ldy, yoff;
  int relu;
};

constexpr int CBM = 64, CBN = 64, CBK = 32, CSK = CBK + 8;  // padded smem rows (80 B)

__global__ void __launch_bounds__(128) k_conv_fwd(ConvArgs a) {
  __shared__ __align__(128) bf16 sA[2][CBM][CSK];
  __shared__ __align__(128) bf16 sB[2][CBN][CSK];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * CBM, n0 = blockIdx.y * CBN;
  const int HW = a.H * a.W, M = a.B * HW, K = 9 * a.Cin;
  const int KT = (K + CBK - 1) / CBK;
  const int q = tid & 3;  // 16-byte chunk within a 32-wide row
  int prow[2], pb[2], ph[2], pw[2];
  bool pv[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    prow[j] = (tid >> 2) + 32 * j;
    const int m = m0 + prow[j];
    pv[j] = m < M;
    const int mm = pv[j] ? m : 0;
    pb[j] = mm / HW;
    const int rem = mm - pb[j] * HW;
    ph[j] = rem / a.W;
    pw[j] = rem - ph[j] * a.W;
  }
  auto load = [&](int kt, int buf) {
    const int k = kt * CBK + q * 8;
    const bool kv = k < K;
    const int tap = kv ? k / a.Cin : 0, ci = kv ? k - tap * a.Cin : 0;
    const int kh = tap / 3, kw = tap - kh * 3;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int hh = ph[j] + kh - 1, ww = pw[j] + kw - 1;
      const bool v = pv[j] && kv && hh >= 0 && hh < a.H && ww >= 0 && ww < a.W;
      const bf16 *src = v ? a.x + ((size_t)(pb[j] * a.H + hh) * a.W + ww) * a.Cin + ci : a.x;
      cp_async16(&sA[buf][prow[j]][q * 8], src, v);
      const int co = n0 + prow[j];
      const bool wv = kv && co < a.Cout;
      cp_async16(&sB[buf][prow[j]][q * 8], wv ? a.w + (size_t)co * K + k : a.w, wv);
    }
    cp_async_commit();
  };
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  load(0, 0);
  for (int kt = 0; kt < KT; ++kt) {
    if (kt + 1 < KT) {
      load(kt + 1, (kt + 1) & 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int buf = kt & 1;
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      uint32_t af[2][4], bfr[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
        ldsm_x4(af[mt], &sA[buf][wm + mt * 16 + (lane & 15)][ks * 16 + (lane >> 4) * 8]);
#pragma unroll
      for (int np = 0; np < 2; ++np)
        ldsm_x4(bfr[np], &sB[buf][wn + np * 16 + (lane & 7) + (lane >> 4) * 8][ks * 16 + ((lane >> 3) & 1) * 8]);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
          mma16816(acc[mt][nt], af[mt], bfr[nt >> 1][(nt & 1) * 2], bfr[nt >> 1][(nt & 1) * 2 + 1]);
    }
    __syncthreads();
  }
  // epilogue: rows lane/4 (+8), column pairs (lane%4)*2
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int m = m0 + wm + mt * 16 + (lane >> 2) + half * 8;
      if (m >= M) continue;
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        const int o = n0 + wn + nt * 8 + (lane & 3) * 2;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (o + e >= a.Cout) continue;
          float v = acc[mt][nt][half * 2 + e];
          if (a.bias) v += a.bias[o + e];
          if (a.relu) v = fmaxf(v, 0.f);
          const size_t at = (size_t)m * a.ldy + a.yoff + o + e;
          if (a.y) a.y[at] = __float2bfloat16_rn(v);
          if (a.yf) a.yf[at] = v;
        }
      }
    }
}

// ---------------------------------------------------------------------------
// Weight gradient: dW[o][k] = sum_m dZ[m][o] A[m][k], the sum over pixels
// split into `splits` slices whose partials are reduced in a fixed order.
// Tile 64 outputs x 64 of K, 32 pixels per step; both operands go through
// ldmatrix.trans (pixels are the reduction index).  Needs Cin, Cout % 8 == 0.
// ---------------------------------------------------------------------------
struct WgradArgs {
  const bf16 *x;   // [B][H][W][Cin] layer input
  const bf16 *dz;  // [B][H][W][Cout] gradient of the pre-activation
  float *part;     // [splits][Cout][9 * Cin]
  int B, H, W, Cin, Cout;
  int pix_per_split;
};

constexpr int WBP = 32, WSK = 64 + 8;  // pixels per step; padded smem rows (144 B)

__global__ void __launch_bounds__(128) k_conv_wgrad(WgradArgs a) {
  __shared__ __align__(128) bf16 sD[2][WBP][WSK];
  __shared__ __align__(128) bf16 sX[2][WBP][WSK];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int k0 = blockIdx.x * 64, o0 = blockIdx.y * 64, split = blockIdx.z;
  const int HW = a.H * a.W, M = a.B * HW, K = 9 * a.Cin;
  const int pbeg = split * a.pix_per_split;
  const int pend = min(M, pbeg + a.pix_per_split);
  const int steps = (pend - pbeg + WBP - 1) / WBP;
  const int q = tid & 7, r0 = tid >> 3;  // chunk q of rows r0, r0 + 16
  // the im2col column of this thread's chunk
  const int kc = k0 + q * 8;
  const bool kv = kc < K;
  const int tap = kv ? kc / a.Cin : 0, ci = kv ? kc - tap * a.Cin : 0;
  const int kh = tap / 3, kw = tap - kh * 3;
  const int oc = o0 + q * 8;
  const bool ov = oc < a.Cout;
  auto load = [&](int s, int buf) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = r0 + 16 * j;
      const int m = pbeg + s * WBP + r;
      const bool mv = m < pend;
      const int mm = mv ? m : 0;
      const int b = mm / HW, rem = mm - b * HW, h = rem / a.W, w = rem - h * a.W;
      cp_async16(&sD[buf][r][q * 8], mv && ov ? a.dz + (size_t)mm * a.Cout + oc : a.dz, mv && ov);
      const int hh = h + kh - 1, ww = w + kw - 1;
      const bool xv = mv && kv && hh >= 0 && hh < a.H && ww >= 0 && ww < a.W;
      cp_async16(&sX[buf][r][q * 8], xv ? a.x + ((size_t)(b * a.H + hh) * a.W + ww) * a.Cin + ci : a.x, xv);
    }
    cp_async_commit();
  };
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
  const int wo = (warp >> 1) * 32, wk = (warp & 1) * 32;
  if (steps > 0) load(0, 0);
  for (int s = 0; s < steps; ++s) {
    if (s + 1 < steps) {
      load(s + 1, (s + 1) & 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int buf = s & 1;
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      uint32_t af[2][4], bfr[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)  // A' = dZ^T: rows outputs, columns pixels
        ldsm_x4_t(af[mt], &sD[buf][ks * 16 + (lane & 7) + (lane >> 4) * 8][wo + mt * 16 + ((lane >> 3) & 1) * 8]);
#pragma unroll
      for (int np = 0; np < 2; ++np)  // B' = im2col: reduction over pixels, columns K
        ldsm_x4_t(bfr[np], &sX[buf][ks * 16 + (lane & 7) + ((lane >> 3) & 1) * 8][wk + np * 16 + (lane >> 4) * 8]);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
          mma16816(acc[mt][nt], af[mt], bfr[nt >> 1][(nt & 1) * 2], bfr[nt >> 1][(nt & 1) * 2 + 1]);
    }
    __syncthreads();
  }
  float *out = a.part + (size_t)split * a.Cout * K;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int o = o0 + wo + mt * 16 + (lane >> 2) + half * 8;
      if (o >= a.Cout) continue;
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        const int k = k0 + wk + nt * 8 + (lane & 3) * 2;
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (k + e < K) out[(size_t)o * K + k + e] = acc[mt][nt][half * 2 + e];
      }
    }
}

// dst[i] = sum_s part[s][i], fixed order.  A block takes COLS columns of V
// consecutive elements and deals the splits to its ROWS thread rows, so that
// a small n with many splits (9216 elements, 152 splits for a 32 -> 32
// layer; 32 elements, 608 splits for its bias) does not wait for one load
// after another.
template <int V, int COLS, int ROWS>
__global__ void __launch_bounds__(COLS *ROWS)
    k_sum_splits(const float *__restrict__ part, int splits, long long n, float *__restrict__ dst) {
  __shared__ float sh[ROWS][COLS * V + 1];
  const int tx = threadIdx.x % COLS, ty = threadIdx.x / COLS;
  const long long i = ((long long)blockIdx.x * COLS + tx) * V;
  float s[V] = {};
  if (i < n) {
#pragma unroll 8
    for (int k = ty; k < splits; k += ROWS) {
      const float *p = part + (long long)k * n + i;
      if constexpr (V == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
        s[0] += v.x; s[1] += v.y; s[2] += v.z; s[3] += v.w;
      } else {
        s[0] += __ldg(p);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < V; ++j) sh[ty][tx * V + j] = s[j];
  __syncthreads();
  for (int c = threadIdx.x; c < COLS * V; c += COLS * ROWS) {
    const long long e = (long long)blockIdx.x * COLS * V + c;
    if (e >= n) continue;
    float t = sh[0][c];
#pragma unroll
    for (int k = 1; k < ROWS; ++k) t += sh[k][c];
    dst[e] = t;
  }
}

// Eight BF16 channels as one 16-byte access.
struct Bf8 {
  uint4 v;
  __device__ __forceinline__ float2 get(int k) const {
    return __bfloat1622float2(reinterpret_cast<const __nv_bfloat162 *>(&v)[k]);
  }
  __device__ __forceinline__ void set(int k, float2 f) {
    reinterpret_cast<__nv_bfloat162 *>(&v)[k] = __floats2bfloat162_rn(f.x, f.y);
  }
};
__device__ __forceinline__ Bf8 ld8(const bf16 *p) { return {__ldg(reinterpret_cast<const uint4 *>(p))}; }
__device__ __forceinline__ void st8(bf16 *p, const Bf8 &b) { *reinterpret_cast<uint4 *>(p) = b.v; }

// dz = dy (x) relu'(y) (RELU; else dz = dy, not written) and the bias
// gradient's partial sums: part[block][c] = sum over the block's rows of
// dz[.][c].  C % 8 == 0, 16-byte aligned rows.  A thread keeps one vector of
// 8 channels and walks down its rows, so a warp reads whole rows; the block
// then adds its threads of one vector in a fixed order.  (Summed by one block
// per channel, 2 bytes per row and thread, the bias gradients of the 256^2,
// 8-sample network took 5.7 of its 7.0 ms.)
constexpr int kBiasThreads = 256;
template <bool RELU>
__global__ void __launch_bounds__(kBiasThreads)
    k_relu_bias(const bf16 *dy, int lddy, int dyoff, const bf16 *y, int ldy, int yoff, bf16 *dz, long long M, int C,
                long long rows, float *__restrict__ part) {
  __shared__ float sh[kBiasThreads][9];
  const int nv = C / 8;
  const int per = nv < kBiasThreads ? nv : kBiasThreads;  // vectors per pass over the columns
  const int groups = kBiasThreads / per;                  // rows in flight
  const int g = threadIdx.x / per, v0 = threadIdx.x - g * per;
  const long long m0 = (long long)blockIdx.x * rows, m1 = m0 + rows < M ? m0 + rows : M;
  for (int vb = 0; vb < nv; vb += per) {
    const int v = vb + v0;
    float acc[8] = {};
    if (g < groups && v < nv) {
#pragma unroll 4
      for (long long m = m0 + g; m < m1; m += groups) {
        Bf8 d = ld8(dy + m * lddy + dyoff + v * 8);
        if constexpr (RELU) {
          const Bf8 o = ld8(y + m * ldy + yoff + v * 8);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 f = d.get(k), r = o.get(k);
            d.set(k, make_float2(r.x > 0.f ? f.x : 0.f, r.y > 0.f ? f.y : 0.f));
          }
          st8(dz + m * C + v * 8, d);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 f = d.get(k);
          acc[2 * k] += f.x;
          acc[2 * k + 1] += f.y;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) sh[threadIdx.x][k] = acc[k];
    __syncthreads();
    for (int e = threadIdx.x; e < per * 8; e += kBiasThreads) {
      const int vv = e / 8, k = e - vv * 8;
      if (vb + vv >= nv) continue;
      float t = 0.f;
      for (int q = 0; q < groups; ++q) t += sh[q * per + vv][k];
      part[(long long)blockIdx.x * C + (vb + vv) * 8 + k] = t;
    }
  }
}

// Wt[i][t'][o] = W[o][t][i] with t' = 8 - t (spatial flip): the data gradient
// of a convolution is the forward convolution of dZ with Wt.  All layers of a
// list in one launch, by 32 x 32 tiles through shared memory so that both
// sides are read and written along their rows.
constexpr int kFlipLayers = 32;
struct FlipList {
  int n;
  int tile0[kFlipLayers + 1];  // first tile of each layer
  int cin[kFlipLayers], cout[kFlipLayers];
  long long off[kFlipLayers];  // element offset of the layer in w and in wt
};
__global__ void __launch_bounds__(256) k_flip_weights(const bf16 *__restrict__ w, bf16 *__restrict__ wt, FlipList f) {
  __shared__ bf16 sh[32][33];
  int l = 0;
  while (l + 1 < f.n && (int)blockIdx.x >= f.tile0[l + 1]) ++l;
  const int Cin = f.cin[l], Cout = f.cout[l], ti = (Cin + 31) / 32;
  int r = (int)blockIdx.x - f.tile0[l];
  const int t = r % 9;
  r /= 9;
  const int i0 = (r % ti) * 32, o0 = (r / ti) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  w += f.off[l];
  wt += f.off[l];
  for (int k = ty; k < 32; k += 8)
    if (o0 + k < Cout && i0 + tx < Cin) sh[k][tx] = w[((long long)(o0 + k) * 9 + t) * Cin + i0 + tx];
  __syncthreads();
  for (int k = ty; k < 32; k += 8)
    if (i0 + k < Cin && o0 + tx < Cout) wt[((long long)(i0 + k) * 9 + (8 - t)) * Cout + o0 + tx] = sh[tx][k];
}

// ---------------------------------------------------------------------------
// Element-wise pieces (strided channel slices: element [m][off + c]).  Each
// thread moves one vector of 8 channels (C % 8 == 0, 16-byte aligned rows);
// blockIdx.x is an image row, blockIdx.y a run of 256 vectors of it.  One
// 2-byte element per thread with its 64-bit divisions ran at a tenth of HBM
// (upsampling 32^2 .. 128^2 to 256^2, 8 samples: 282 us).
// ---------------------------------------------------------------------------
// out[b][h][w][c] = mean of the 2x2 block of in (in: H x W, slice [off, off+C))
__global__ void __launch_bounds__(256) k_avgpool2(const bf16 *in, int ldi, int ioff, int H, int W, int C, bf16 *out) {
  const int nv = C / 8, Wo = W / 2, Ho = H / 2;
  const int e = blockIdx.y * 256 + threadIdx.x;
  if (e >= Wo * nv) return;
  const int wo = e / nv, c = (e - wo * nv) * 8;
  const int b = blockIdx.x / Ho, ho = blockIdx.x - b * Ho;
  Bf8 q[2][2], o;
#pragma unroll
  for (int dh = 0; dh < 2; ++dh)
#pragma unroll
    for (int dw = 0; dw < 2; ++dw)
      q[dh][dw] = ld8(in + (((long long)b * H + 2 * ho + dh) * W + 2 * wo + dw) * ldi + ioff + c);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = q[j >> 1][j & 1].get(k);
      s.x += f.x;
      s.y += f.y;
    }
    o.set(k, make_float2(0.25f * s.x, 0.25f * s.y));
  }
  st8(out + ((long long)blockIdx.x * Wo + wo) * C + c, o);
}

// dx[m][c] = dpool[parent(m)][c] / 4 + dskip[m][soff + c]   (dx: H x W, contiguous C)
__global__ void __launch_bounds__(256)
    k_avgpool2_bwd_add(const bf16 *dpool, const bf16 *dskip, int lds, int soff, int H, int W, int C, bf16 *dx) {
  const int nv = C / 8;
  const int e = blockIdx.y * 256 + threadIdx.x;
  if (e >= W * nv) return;
  const int w = e / nv, c = (e - w * nv) * 8;
  const int b = blockIdx.x / H, h = blockIdx.x - b * H;
  const Bf8 p = ld8(dpool + (((long long)b * (H / 2) + h / 2) * (W / 2) + w / 2) * C + c);
  const long long m = (long long)blockIdx.x * W + w;
  const Bf8 s = ld8(dskip + m * lds + soff + c);
  Bf8 o;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 f = p.get(k), g = s.get(k);
    o.set(k, make_float2(0.25f * f.x + g.x, 0.25f * f.y + g.y));
  }
  st8(dx + m * C + c, o);
}

// out[b][2h+i][2w+j][c] = in[b][h][w][c], into a slice of width C at column 0
// of rows of stride ldo.  blockIdx.x: an input row; H, W: the input's.
__global__ void __launch_bounds__(256) k_upsample2(const bf16 *in, int H, int W, int C, bf16 *out, int ldo) {
  const int nv = C / 8;
  const int e = blockIdx.y * 256 + threadIdx.x;
  if (e >= W * nv) return;
  const int w = e / nv, c = (e - w * nv) * 8;
  const int b = blockIdx.x / H, h = blockIdx.x - b * H;
  const Bf8 v = ld8(in + ((long long)blockIdx.x * W + w) * C + c);
  bf16 *o = out + (((long long)b * 2 * H + 2 * h) * 2 * W + 2 * w) * ldo + c;
  st8(o, v);
  st8(o + ldo, v);
  o += (long long)2 * W * ldo;
  st8(o, v);
  st8(o + ldo, v);
}

// d[b][h][w][c] = sum of the 2x2 children of dup (slice [0, C) of stride ldu)
__global__ void __launch_bounds__(256) k_upsample2_bwd(const bf16 *dup, int ldu, int H, int W, int C, bf16 *d) {
  const int nv = C / 8;
  const int e = blockIdx.y * 256 + threadIdx.x;
  if (e >= W * nv) return;
  const int w = e / nv, c = (e - w * nv) * 8;
  const int b = blockIdx.x / H, h = blockIdx.x - b * H;
  Bf8 q[2][2], o;
#pragma unroll
  for (int dh = 0; dh < 2; ++dh)
#pragma unroll
    for (int dw = 0; dw < 2; ++dw)
      q[dh][dw] = ld8(dup + (((long long)b * 2 * H + 2 * h + dh) * 2 * W + 2 * w + dw) * ldu + c);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = q[j >> 1][j & 1].get(k);
      s.x += f.x;
      s.y += f.y;
    }
    o.set(k, s);
  }
  st8(d + ((long long)blockIdx.x * W + w) * C + c, o);
}

// MSE over the first `cv` of `cp` channels: per-block partial loss (FP64)
// and dy = 2 (y - t) / (M cv) for those channels, 0 for the padding.  One
// thread per pixel (of 16 channels, 3 of them used in the study's network):
// only the used channels are read, and one block in 16 of before reduces.
__global__ void __launch_bounds__(256) k_mse(const float *y, int cp, const float *t, int cv, long long M, bf16 *dy,
                                             double *part) {
  __shared__ double sh[8];
  const long long m = (long long)blockIdx.x * 256 + threadIdx.x;
  double l = 0.0;
  if (m < M) {
    for (int c0 = 0; c0 < cp; c0 += 8) {
      Bf8 o;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float g[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c = c0 + 2 * k + j;
          g[j] = 0.f;
          if (c < cv) {
            const float d = y[m * cp + c] - t[m * cv + c];
            l += (double)d * d;
            g[j] = 2.f * d / (float)(M * cv);
          }
        }
        o.set(k, make_float2(g[0], g[1]));
      }
      st8(dy + m * cp + c0, o);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) l += sh[w];
    part[blockIdx.x] = l;
  }
}

// Adam (Kingma & Ba 2015) on FP32 master parameters, with the BF16 copy.
__global__ void k_adam(float *p, const float *g, float *m, float *v, bf16 *pb, long long n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  p[i] = pi;
  if (pb) pb[i] = __float2bfloat16_rn(pi);
}

// y = x in BF16; VEC: 8 elements per thread (n % 8 == 0, 16-byte aligned).
template <bool VEC>
__global__ void __launch_bounds__(256) k_f32_to_bf16(const float *x, bf16 *y, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if constexpr (VEC) {
    if (i * 8 >= n) return;
    const float4 a = __ldg(reinterpret_cast<const float4 *>(x) + 2 * i);
    const float4 b = __ldg(reinterpret_cast<const float4 *>(x) + 2 * i + 1);
    Bf8 o;
    o.set(0, make_float2(a.x, a.y));
    o.set(1, make_float2(a.z, a.w));
    o.set(2, make_float2(b.x, b.y));
    o.set(3, make_float2(b.z, b.w));
    st8(y + i * 8, o);
  } else {
    if (i < n) y[i] = __float2bfloat16_rn(x[i]);
  }
}

}  // namespace mdfnn
