// fvna_net.cu -- the learned sub-grid correction (not in the paper): three
// 3x3 convolutions with zero padding, 3 -> 32 -> 32 -> 3 channels, ReLU after
// the first two,
//     y[o,i,j] = b[o] + sum_c sum_{u,v} w[o,c,u,v] x[c, i+u-1, j+v-1].
//
// Forward: BF16 tensor-core implicit GEMM (mma.sync m16n8k16, FP32
// accumulation).  A CTA owns an 8 x 32 pixel tile; each warp one 32-pixel row
// (two m-tiles of 16 pixels).  The input tile plus a 1-pixel halo sits in
// shared memory channel-innermost (pixel stride 40 bf16 = 80 bytes, so the
// eight rows an ldmatrix reads fall in distinct bank groups); K runs over the
// nine taps times the input channels.  The 3-channel first layer builds its
// (pixels x 32) im2col tile in shared memory instead.  Hidden activations are
// stored as BF16, pixel-major with 32 channels; network input and output are
// FP32 channel planes.
// Backward (training): FP32 CUDA-core kernels on pixel tiles for the input and
// weight gradients, then Adam on FP32 master weights, which are re-packed to
// BF16.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <new>

#include "../../include/fvna.h"
#include "fvna_net.h"

namespace fvna {

constexpr int NET_TH = 8;             // tile rows (one warp per row)
constexpr int NET_TW = 32;            // tile columns
constexpr int NET_PIX = NET_TH * NET_TW;
constexpr int NET_HALO_W = NET_TW + 2;
constexpr int NET_HALO_H = NET_TH + 2;
constexpr int CH = 32;                // hidden channels
constexpr int CPAD = 40;              // padded channel stride of shared tiles
constexpr int KH = 9 * CH;            // K of the hidden layers (288)
constexpr int KPAD = KH + 8;          // padded K stride of shared weights (296)
constexpr int K1 = 32;                // K of the first layer (27 taps x channels, padded)

// ---------------------------------------------------------------------------
// PTX helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void ldsm_x4(unsigned addr, unsigned &r0, unsigned &r1, unsigned &r2,
                                        unsigned &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(unsigned addr, unsigned &r0, unsigned &r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r0), "=r"(r1)
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float d[4], unsigned a0, unsigned a1, unsigned a2,
                                         unsigned a3, unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------
// Forward convolution on tensor cores.
//   MODE 0: input = FP32 planes (3 channels) times in_scale, output BF16 hidden + ReLU
//   MODE 1: input = BF16 hidden, output BF16 hidden + ReLU
//   MODE 2: input = BF16 hidden, output FP32 planes (3 channels); if apply,
//           the planes receive += out_scale * y instead of y
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(256) k_net_conv(NetConvArgs a) {
  constexpr int NT = MODE == 2 ? 1 : 4;           // n-tiles of 8 output channels
  constexpr int KS = MODE == 0 ? K1 / 16 : KH / 16;  // k-steps of 16
  constexpr int WROWS = NT * 8;
  constexpr int WSTRIDE = MODE == 0 ? K1 + 8 : KPAD;
  __shared__ __align__(16) __nv_bfloat16 s_in[NET_HALO_H * NET_HALO_W * CPAD];  // also im2col
  __shared__ __align__(16) __nv_bfloat16 s_w[WROWS * WSTRIDE];
  if (a.done && *a.done) return;   // the step of this domain was not taken
  if (a.step && a.every > 1 && (*a.step + 1) % a.every != 0) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.z;
  const int i0 = blockIdx.y * NET_TH, j0 = blockIdx.x * NET_TW;
  const int H = a.h, W = a.w;

  // weights: [n][k] rows of the packed BF16 matrix
  {
    const int kk = MODE == 0 ? K1 : KH;
    for (int e = tid; e < WROWS * kk / 8; e += 256) {
      int n = e / (kk / 8), k8 = e - n * (kk / 8);
      uint4 v = reinterpret_cast<const uint4 *>(a.wmat + (size_t)n * kk)[k8];
      *reinterpret_cast<uint4 *>(&s_w[n * WSTRIDE + k8 * 8]) = v;
    }
  }
  if (MODE == 0) {
    // 3-channel FP32 input tile -> BF16, then the im2col tile (pixels x 32)
    __shared__ __nv_bfloat16 s_x3[NET_HALO_H * NET_HALO_W * 4];
    for (int e = tid; e < NET_HALO_H * NET_HALO_W; e += 256) {
      int r = e / NET_HALO_W, cc = e - r * NET_HALO_W;
      int gi = i0 + r - 1, gj = j0 + cc - 1;
      float v[3] = {0.f, 0.f, 0.f};
      if (gi >= 0 && gi < H && gj >= 0 && gj < W) {
        size_t off = (size_t)b * a.in_bstride + (size_t)gi * a.in_pitch + gj;
        for (int c = 0; c < 3; c++) v[c] = a.in[off + (size_t)c * a.in_pstride] * a.in_scale;
      }
      for (int c = 0; c < 3; c++) s_x3[e * 4 + c] = __float2bfloat16_rn(v[c]);
      s_x3[e * 4 + 3] = __float2bfloat16_rn(0.f);
    }
    __syncthreads();
    for (int e = tid; e < NET_PIX * K1; e += 256) {
      int p = e / K1, k = e - p * K1;
      int r = p / NET_TW, cc = p - r * NET_TW;
      __nv_bfloat16 v = __float2bfloat16_rn(0.f);
      if (k < 27) {
        int t = k / 3, c = k - t * 3;
        v = s_x3[((r + t / 3) * NET_HALO_W + cc + t % 3) * 4 + c];
      }
      s_in[p * CPAD + k] = v;
    }
  } else {
    // BF16 hidden input tile with halo (zero outside the image)
    for (int e = tid; e < NET_HALO_H * NET_HALO_W * 4; e += 256) {
      int pix = e >> 2, q = e & 3;
      int r = pix / NET_HALO_W, cc = pix - r * NET_HALO_W;
      int gi = i0 + r - 1, gj = j0 + cc - 1;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (gi >= 0 && gi < H && gj >= 0 && gj < W)
        v = reinterpret_cast<const uint4 *>(a.hin + (((size_t)b * H + gi) * W + gj) * CH)[q];
      *reinterpret_cast<uint4 *>(&s_in[pix * CPAD + q * 8]) = v;
    }
  }
  __syncthreads();

  float acc[2][NT][4];
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int nt = 0; nt < NT; nt++)
#pragma unroll
      for (int q = 0; q < 4; q++) acc[mt][nt][q] = 0.f;

  const int mi = lane >> 3, mr = lane & 7;
#pragma unroll 2
  for (int ks = 0; ks < KS; ks++) {
    unsigned af[2][4];
#pragma unroll
    for (int mt = 0; mt < 2; mt++) {
      int m = mt * 16 + mr + (mi & 1) * 8;      // pixel within the warp's 32
      int kof = (mi >> 1) * 8;
      const __nv_bfloat16 *src;
      if (MODE == 0) {
        src = &s_in[(warp * NET_TW + m) * CPAD + ks * 16 + kof];
      } else {
        int tap = ks >> 1, half = ks & 1;
        int u = tap / 3, v = tap - u * 3;
        src = &s_in[((warp + u) * NET_HALO_W + m + v) * CPAD + half * 16 + kof];
      }
      ldsm_x4(smem_u32(src), af[mt][0], af[mt][1], af[mt][2], af[mt][3]);
    }
#pragma unroll
    for (int nt = 0; nt < NT; nt++) {
      unsigned b0, b1;
      const __nv_bfloat16 *src = &s_w[(nt * 8 + mr) * WSTRIDE + ks * 16 + (mi & 1) * 8];
      ldsm_x2(smem_u32(src), b0, b1);
#pragma unroll
      for (int mt = 0; mt < 2; mt++)
        mma_bf16(acc[mt][nt], af[mt][0], af[mt][1], af[mt][2], af[mt][3], b0, b1);
    }
  }

  // epilogue: bias, ReLU, store
  const int g = lane >> 2, tig = lane & 3;
  const int gi = i0 + warp;
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      int gj = j0 + mt * 16 + g + hh * 8;
      if (gi >= H || gj >= W) continue;
#pragma unroll
      for (int nt = 0; nt < NT; nt++) {
        int ch = nt * 8 + tig * 2;
        if (MODE == 2 && ch >= 3) continue;
        float y0 = acc[mt][nt][hh * 2] + a.bias[ch];
        float y1 = acc[mt][nt][hh * 2 + 1] + (MODE == 2 && ch + 1 >= 3 ? 0.f : a.bias[ch + 1]);
        if (MODE != 2) {
          y0 = fmaxf(y0, 0.f);
          y1 = fmaxf(y1, 0.f);
          __nv_bfloat162 v = __floats2bfloat162_rn(y0, y1);
          *reinterpret_cast<__nv_bfloat162 *>(a.hout + (((size_t)b * H + gi) * W + gj) * CH + ch) = v;
        } else {
          if (a.apply && (gj < a.band || gj >= W - a.band || gi < a.band || gi >= H - a.band))
            continue;
          size_t off = (size_t)b * a.out_bstride + (size_t)gi * a.out_pitch + gj;
          if (ch < 3) {
            float *o = a.out + off + (size_t)ch * a.out_pstride;
            *o = a.apply ? *o + a.out_scale * y0 : y0;
          }
          if (ch + 1 < 3) {
            float *o = a.out + off + (size_t)(ch + 1) * a.out_pstride;
            *o = a.apply ? *o + a.out_scale * y1 : y1;
          }
        }
      }
    }
}

// ---------------------------------------------------------------------------
// The three layers in one kernel, for a forward whose output does not overlap
// its input.  Persistent blocks keep all weights in shared memory and take
// tiles of 8 x 32 pixels: the input with a ring of three pixels, the first
// activation with a ring of two and the second with a ring of one are made in
// shared memory, so neither activation is read back (both are still written,
// for a backward).  The rings cost a third more tensor instructions (2,088 of
// m16n8k16 a tile against 1,568).  Shared memory bounds it (70 % of its
// cycles, the tensor pipe 48 %), so a warp holds three 16-pixel m-tiles of the
// hidden layer for each weight fragment, keeps the first and the last layer's
// weights in registers and shares the last layer's pixels between two rows.
// Every sum runs over k in the order of k_net_conv: the bits are the same.  One
// 2048 x 512 field: 157 us in three kernels (39 + 77 + 41), 127 us in this one.
// ---------------------------------------------------------------------------
constexpr int F1H = NET_TH + 4, F1W = NET_TW + 4, F1P = F1H * F1W;   // first activation
constexpr int F2H = NET_TH + 2, F2W = NET_TW + 2, F2P = F2H * F2W;   // second activation
constexpr int FXH = NET_TH + 6, FXW = NET_TW + 6;                    // input
constexpr int F1M = F1P / 16, F2M = (F2P + 15) / 16;
static_assert(F1P % 16 == 0 && F2M <= 24, "m-tiles");
constexpr int K1S = K1 + 8;
constexpr int FUSED_SMEM =
    (32 * K1S + 40 * KPAD + FXH * FXW * 4 + F1P * CPAD + F2M * 16 * CPAD) * (int)sizeof(__nv_bfloat16) +
    64 * (int)sizeof(float);

struct NetFusedArgs {
  int B, H, W;
  const float *x;
  float in_scale;
  const __nv_bfloat16 *w1, *w2, *w3;
  const float *b1, *b2, *b3;
  __nv_bfloat16 *h1, *h2;
  float *y;
};

// two n-tiles' B fragments of one k-step: rows n of the weights w (stride ws)
__device__ __forceinline__ void b_frags(const __nv_bfloat16 *w, int ws, int n0, int k, int lane,
                                        unsigned b[4]) {
  const int mi = lane >> 3, mr = lane & 7;
  ldsm_x4(smem_u32(&w[(n0 + (mi >> 1) * 8 + mr) * ws + k + (mi & 1) * 8]), b[0], b[1], b[2], b[3]);
}
// bias, ReLU and rounding of one m-tile's 32 channels into a shared activation
// tile (zero outside the image; a tile well inside asks no pixel)
__device__ __forceinline__ void put_hidden(const float acc[4][4], const float *bias, __nv_bfloat16 *s,
                                           int p0, int width, bool inside, int i0, int j0, int H,
                                           int W, int lane) {
  unsigned keep[2] = {~0u, ~0u};
  if (!inside) {
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      const int p = p0 + (lane >> 2) + hh * 8, gi = i0 + p / width, gj = j0 + p % width;
      keep[hh] = gi >= 0 && gi < H && gj >= 0 && gj < W ? ~0u : 0u;
    }
  }
  unsigned v[2][4];
#pragma unroll
  for (int nt = 0; nt < 4; nt++) {
    const float2 b = *reinterpret_cast<const float2 *>(bias + nt * 8 + (lane & 3) * 2);
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      // the rounding keeps the sign, so the maximum may follow it
      const float2 r = __fadd2_rn(make_float2(acc[nt][hh * 2], acc[nt][hh * 2 + 1]), b);
      const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(r.x, r.y), __floats2bfloat162_rn(0.f, 0.f));
      v[hh][nt] = *reinterpret_cast<const unsigned *>(&h) & keep[hh];
    }
  }
  const unsigned at = smem_u32(s + (p0 + (lane & 7)) * CPAD + (lane >> 3) * 8);
#pragma unroll
  for (int hh = 0; hh < 2; hh++)
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(
                     at + hh * 8 * CPAD * 2),
                 "r"(v[hh][0]), "r"(v[hh][1]), "r"(v[hh][2]), "r"(v[hh][3])
                 : "memory");
}
// the tile's own pixels of a shared activation (ring r, width w) to global memory
__device__ __forceinline__ void store_hidden(const __nv_bfloat16 *s, int r, int w, __nv_bfloat16 *h,
                                             int b, int i0, int j0, int H, int W, int tid) {
  const int q = tid & 3, j = (tid >> 2) & 31, i = tid >> 7;
  if (j0 + j >= W) return;
  const uint4 *from = reinterpret_cast<const uint4 *>(s + ((i + r) * w + j + r) * CPAD) + q;
  uint4 *to = reinterpret_cast<uint4 *>(h + (((size_t)b * H + i0 + i) * W + j0 + j) * CH) + q;
#pragma unroll
  for (int k = 0; k < NET_TH / 2; k++)
    if (i0 + i + 2 * k < H) to[(size_t)k * 2 * W * (CH / 8)] = from[k * 2 * w * (CPAD / 8)];
}
// input pixels of tile (b, i0, j0): loads, and rounded stores
struct InPixels {
  float v[3][3];
  __device__ __forceinline__ void load(const NetFusedArgs &a, int b, int i0, int j0, int tid) {
    const long long hw = (long long)a.H * a.W;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const int e = tid + k * 256, gi = i0 + e / FXW - 3, gj = j0 + e % FXW - 3;
      const bool in = e < FXH * FXW && gi >= 0 && gi < a.H && gj >= 0 && gj < a.W;
      const float *q = a.x + 3 * b * hw + (long long)gi * a.W + gj;
#pragma unroll
      for (int c = 0; c < 3; c++) v[k][c] = in ? q[c * hw] : 0.f;
    }
  }
  __device__ __forceinline__ void store(const NetFusedArgs &a, __nv_bfloat16 *s, int tid) const {
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const int e = tid + k * 256;
      if (e >= FXH * FXW) continue;
      const __nv_bfloat162 lo = __floats2bfloat162_rn(v[k][0] * a.in_scale, v[k][1] * a.in_scale);
      const __nv_bfloat162 hi = __floats2bfloat162_rn(v[k][2] * a.in_scale, 0.f);
      uint2 u;
      u.x = *reinterpret_cast<const unsigned *>(&lo);
      u.y = *reinterpret_cast<const unsigned *>(&hi);
      *reinterpret_cast<uint2 *>(&s[e * 4]) = u;
    }
  }
};

__global__ void __launch_bounds__(256, 2) k_net_fused(NetFusedArgs a) {
  extern __shared__ __align__(16) __nv_bfloat16 fs[];
  __nv_bfloat16 *const s_w1 = fs, *const s_w2 = s_w1 + 32 * K1S, *const s_w3 = s_w2 + 32 * KPAD;
  __nv_bfloat16 *const s_h1 = s_w3 + 8 * KPAD, *const s_h2 = s_h1 + F1P * CPAD;
  __nv_bfloat16 *const s_x = s_h2 + F2M * 16 * CPAD;
  float *const s_b = reinterpret_cast<float *>(s_x + FXH * FXW * 4);   // b1, b2
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, H = a.H, W = a.W;
  const int mi = lane >> 3, mr = lane & 7, tig = lane & 3, g = lane >> 2;
  for (int e = tid; e < 32 * K1 / 8; e += 256)
    *reinterpret_cast<uint4 *>(&s_w1[e / (K1 / 8) * K1S + e % (K1 / 8) * 8]) =
        reinterpret_cast<const uint4 *>(a.w1)[e];
  for (int e = tid; e < 40 * KH / 8; e += 256) {      // w2 and w3 (32 and 8 rows)
    const uint4 v = e < 32 * KH / 8 ? reinterpret_cast<const uint4 *>(a.w2)[e]
                                    : reinterpret_cast<const uint4 *>(a.w3)[e - 32 * KH / 8];
    *reinterpret_cast<uint4 *>(&s_w2[e / (KH / 8) * KPAD + e % (KH / 8) * 8]) = v;
  }
  if (tid < 64) s_b[tid] = tid < 32 ? a.b1[tid] : a.b2[tid - 32];
  // input offsets of this lane's eight k pairs of the first layer; k >= 27 reads
  // the zero that pads a pixel
  int koff[2][2][2];
#pragma unroll
  for (int q = 0; q < 8; q++) {
    const int k = (q >> 2) * 16 + ((q >> 1) & 1) * 8 + tig * 2 + (q & 1), t = k / 3;
    koff[q >> 2][(q >> 1) & 1][q & 1] = k < 27 ? ((t / 3) * FXW + t % 3) * 4 + k % 3 : 3;
  }
  const int tw = (W + NET_TW - 1) / NET_TW, th = (H + NET_TH - 1) / NET_TH;
  const long long tiles = (long long)a.B * tw * th, hw = (long long)H * W;
  // tile t of batch b at (i0, j0)
  auto tile = [&](long long t, int &b, int &i0, int &j0) {
    b = (int)(t / (tw * th));
    const int r = (int)(t - (long long)b * tw * th);
    i0 = r / tw * NET_TH;
    j0 = (r - r / tw * tw) * NET_TW;
  };
  int b, i0, j0;
  tile(blockIdx.x, b, i0, j0);
  InPixels in;
  in.load(a, b, i0, j0, tid);
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    in.store(a, s_x, tid);
    __syncthreads();
    const bool inside = i0 >= 2 && j0 >= 2 && i0 + NET_TH + 2 <= H && j0 + NET_TW + 2 <= W;
    // first activation on 12 x 36 pixels
    const unsigned short *const xs = reinterpret_cast<const unsigned short *>(s_x);
    unsigned wf[2][2][4];
#pragma unroll
    for (int q = 0; q < 4; q++) b_frags(s_w1, K1S, (q & 1) * 16, (q >> 1) * 16, lane, wf[q >> 1][q & 1]);
#pragma unroll 2
    for (int mt = warp; mt < F1M; mt += 8) {
      float acc[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; nt++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[nt][q] = 0.f;
      const int pa = mt * 16 + g, pb = pa + 8;
      const unsigned short *const xa = xs + (pa / F1W * FXW + pa % F1W) * 4;
      const unsigned short *const xb = xs + (pb / F1W * FXW + pb % F1W) * 4;
#pragma unroll
      for (int ks = 0; ks < 2; ks++) {
        unsigned af[4];
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int o0 = koff[ks][h][0], o1 = koff[ks][h][1];
          af[2 * h] = xa[o0] | (unsigned)xa[o1] << 16;
          af[2 * h + 1] = xb[o0] | (unsigned)xb[o1] << 16;
        }
#pragma unroll
        for (int n2 = 0; n2 < 2; n2++) {
          const unsigned *bf = wf[ks][n2];
          mma_bf16(acc[2 * n2], af[0], af[1], af[2], af[3], bf[0], bf[1]);
          mma_bf16(acc[2 * n2 + 1], af[0], af[1], af[2], af[3], bf[2], bf[3]);
        }
      }
      put_hidden(acc, s_b, s_h1, mt * 16, F1W, inside, i0 - 2, j0 - 2, H, W, lane);
    }
    __syncthreads();
    store_hidden(s_h1, 2, F1W, a.h1, b, i0, j0, H, W, tid);
    // second activation on 10 x 34 pixels: m-tiles warp, warp + 8, warp + 16
    {
      float acc[3][4][4];
      unsigned row[3];
      const bool third = warp + 16 < F2M;
#pragma unroll
      for (int m = 0; m < 3; m++) {
        int p = (warp + 8 * m) * 16 + mr + (mi & 1) * 8;
        p = p < F2P ? p : F2P - 1;
        row[m] = smem_u32(&s_h1[(p / F2W * F1W + p % F2W) * CPAD + (mi >> 1) * 8]);
#pragma unroll
        for (int nt = 0; nt < 4; nt++)
#pragma unroll
          for (int q = 0; q < 4; q++) acc[m][nt][q] = 0.f;
      }
#pragma unroll 1
      for (int ty = 0; ty < 3; ty++)
#pragma unroll
        for (int q = 0; q < 6; q++) {      // the row's three taps, two k-steps each
          const unsigned off = ((ty * F1W + (q >> 1)) * CPAD + (q & 1) * 16) * 2;
          unsigned bf[2][4], af[4];
          b_frags(s_w2, KPAD, 0, ty * 96 + q * 16, lane, bf[0]);
          b_frags(s_w2, KPAD, 16, ty * 96 + q * 16, lane, bf[1]);
#pragma unroll
          for (int m = 0; m < 3; m++) {
            if (m == 2 && !third) break;
            ldsm_x4(row[m] + off, af[0], af[1], af[2], af[3]);
#pragma unroll
            for (int nt = 0; nt < 4; nt++)
              mma_bf16(acc[m][nt], af[0], af[1], af[2], af[3], bf[nt >> 1][(nt & 1) * 2],
                       bf[nt >> 1][(nt & 1) * 2 + 1]);
          }
        }
#pragma unroll
      for (int m = 0; m < 3; m++) {
        if (m == 2 && !third) break;
        put_hidden(acc[m], s_b + 32, s_h2, (warp + 8 * m) * 16, F2W, inside, i0 - 1, j0 - 1, H, W,
                   lane);
      }
    }
    __syncthreads();
    store_hidden(s_h2, 1, F2W, a.h2, b, i0, j0, H, W, tid);
    // the next tile's input is on its way during the output layer
    const int ob = b, oi = i0 + (warp >> 1) * 2, oj = j0 + (warp & 1) * 16;
    if (t + gridDim.x < tiles) {
      tile(t + gridDim.x, b, i0, j0);
      in.load(a, b, i0, j0, tid);
    }
    // output: two rows of 16 pixels a warp, which share the fragments of the
    // two middle ones of the four rows that they read
    float acc[2][4];
    unsigned w3f[9][4];                  // both k-steps of each tap
#pragma unroll
    for (int m = 0; m < 2; m++)
#pragma unroll
      for (int q = 0; q < 4; q++) acc[m][q] = 0.f;
#pragma unroll
    for (int tap = 0; tap < 9; tap++)
      ldsm_x4(smem_u32(&s_w3[mr * KPAD + tap * 32 + mi * 8]), w3f[tap][0], w3f[tap][1], w3f[tap][2],
              w3f[tap][3]);
    const unsigned base = smem_u32(
        &s_h2[((warp >> 1) * 2 * F2W + (warp & 1) * 16 + mr + (mi & 1) * 8) * CPAD + (mi >> 1) * 8]);
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
      for (int q = 0; q < 6; q++) {
        unsigned af[4];
        ldsm_x4(base + ((r * F2W + (q >> 1)) * CPAD + (q & 1) * 16) * 2, af[0], af[1], af[2], af[3]);
#pragma unroll
        for (int m = 0; m < 2; m++)
          if (r >= m && r - m < 3) {
            const unsigned *bf = w3f[(r - m) * 3 + (q >> 1)] + (q & 1) * 2;
            mma_bf16(acc[m], af[0], af[1], af[2], af[3], bf[0], bf[1]);
          }
      }
    if (tig < 2) {
#pragma unroll
      for (int m = 0; m < 2; m++)
#pragma unroll
        for (int hh = 0; hh < 2; hh++) {
          const int gi = oi + m, gj = oj + g + hh * 8;
          if (gi >= H || gj >= W) continue;
          float *o = a.y + (3 * ob + 2 * tig) * hw + (long long)gi * W + gj;
          o[0] = acc[m][hh * 2] + a.b3[2 * tig];
          if (tig == 0) o[hw] = acc[m][hh * 2 + 1] + a.b3[1];
        }
    }
  }
}

// ---------------------------------------------------------------------------
// Parameter packing: FP32 master parameters (w[o][c][u][v] per layer, then
// biases) -> BF16 matrices [n][k], k = tap*CIN + c (first layer: tap*3 + c,
// padded to 32), rows beyond the output channels zero (last layer: 8 rows).
// ---------------------------------------------------------------------------
__global__ void k_net_pack(const float *params, __nv_bfloat16 *w1, __nv_bfloat16 *w2,
                           __nv_bfloat16 *w3) {
  const float *p1 = params + NET_OFF_W1, *p2 = params + NET_OFF_W2, *p3 = params + NET_OFF_W3;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 32 * K1 + 32 * KH + 8 * KH;
       e += gridDim.x * blockDim.x) {
    if (e < 32 * K1) {
      int n = e / K1, k = e - n * K1;
      float v = 0.f;
      if (k < 27) { int t = k / 3, c = k - t * 3; v = p1[(n * 3 + c) * 9 + t]; }
      w1[e] = __float2bfloat16_rn(v);
    } else if (e < 32 * K1 + 32 * KH) {
      int f = e - 32 * K1, n = f / KH, k = f - n * KH;
      int t = k / CH, c = k - t * CH;
      w2[f] = __float2bfloat16_rn(p2[(n * CH + c) * 9 + t]);
    } else {
      int f = e - 32 * K1 - 32 * KH, n = f / KH, k = f - n * KH;
      int t = k / CH, c = k - t * CH;
      w3[f] = __float2bfloat16_rn(n < 3 ? p3[(n * CH + c) * 9 + t] : 0.f);
    }
  }
}

// ---------------------------------------------------------------------------
// Training kernels (FP32 CUDA cores).  Blocks take pixel tiles of the batch (16
// columns, 8 or 16 rows) in turn; a tile of one operand and the tile with a 1-pixel ring of
// the other are staged in shared memory, and each thread keeps 27 to 36 sums
// in registers, so that a shared load feeds about ten multiply-adds and the
// FP32 pipes are the bound.  Pixels outside the image count as zero.  The
// gradient of the second activation is FP32, pixel-major with 32 channels
// like the activation; that of the first never leaves the block that makes
// it.  A weight gradient is a sum over all pixels: every block adds up its
// tiles and writes one partial sum per weight (part, one row of parameters a
// block), and k_net_reduce adds the rows in binary64.
// A step on eight 128 x 128 crops: 4.6 ms when each pair of channels was one
// block that read the whole batch with strided loads, now 0.25 ms (the
// gradient of layer 3 31 us, of layer 2 64, of layers 2 and 1 to their inputs 74,
// the rows 8; the FP32 pipes would take 12, 32 and 36).
// ---------------------------------------------------------------------------
constexpr int BT = 16;                  // tile columns
constexpr int BR = BT + 2;              // with the ring
constexpr int BTHREADS = 256;
constexpr int HP = CH + 1;              // padded channel stride

struct NetBwdArgs {
  int B, H, W;
  const float *gy;                      // gradient of the output, planes
  const float *x;                       // network input, planes
  float in_scale;
  const __nv_bfloat16 *h1, *h2, *w2, *w3;
  float *gh2;                           // gradient of the second activation
  float *part;                          // partial sums, FVNA_NET_PARAMS a block
};

template <int TH> struct BTile {
  int b, i0, j0;
  __device__ __forceinline__ BTile(const NetBwdArgs &a, int t) {
    const int tw = (a.W + BT - 1) / BT, th = (a.H + TH - 1) / TH;
    b = t / (tw * th);
    const int r = t - b * tw * th;
    i0 = r / tw * TH;
    j0 = (r - r / tw * tw) * BT;
  }
};
template <int TH> __host__ __device__ __forceinline__ long long bwd_tiles(const NetBwdArgs &a) {
  return (long long)a.B * ((a.H + TH - 1) / TH) * ((a.W + BT - 1) / BT);
}
// pixel offset of ring position e (0 .. (TH + 2) BR - 1), or -1 outside the image
template <int TH>
__device__ __forceinline__ long long ring_pixel(const NetBwdArgs &a, const BTile<TH> &t, int e) {
  const int gi = t.i0 + e / BR - 1, gj = t.j0 + e % BR - 1;
  if (gi < 0 || gi >= a.H || gj < 0 || gj >= a.W) return -1;
  return ((long long)t.b * a.H + gi) * a.W + gj;
}
// three FP32 planes with the ring, as float4 per pixel
template <bool ROUND, int TH>
__device__ __forceinline__ void load_planes(const NetBwdArgs &a, const BTile<TH> &t, const float *p,
                                            float scale, float4 *s) {
  const long long hw = (long long)a.H * a.W;
  for (int e = threadIdx.x; e < (TH + 2) * BR; e += BTHREADS) {
    const long long o = ring_pixel(a, t, e);
    float v[3] = {0.f, 0.f, 0.f};
    if (o >= 0) {
      const float *q = p + (o - t.b * hw) + 3 * t.b * hw;
      for (int c = 0; c < 3; c++)
        v[c] = ROUND ? __bfloat162float(__float2bfloat16_rn(q[c * hw] * scale)) : q[c * hw];
    }
    s[e] = make_float4(v[0], v[1], v[2], 0.f);
  }
}
// a BF16 activation with the ring, [pixel][channel] at stride `stride`
template <int TH>
__device__ __forceinline__ void load_hidden(const NetBwdArgs &a, const BTile<TH> &t,
                                            const __nv_bfloat16 *h, float *s, int stride) {
  for (int e = threadIdx.x; e < (TH + 2) * BR * 4; e += BTHREADS) {
    const long long o = ring_pixel(a, t, e >> 2);
    uint4 v = make_uint4(0, 0, 0, 0);
    if (o >= 0) v = reinterpret_cast<const uint4 *>(h + o * CH)[e & 3];
    float *d = s + (e >> 2) * stride + (e & 3) * 8;
    const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; k++) {
      d[2 * k] = __uint_as_float(u[k] << 16);
      d[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u);
    }
  }
}
// sums[n] of every (warp, lane) added over the warps; f(k, lane, sum) stores
// them.  s: 8 * n * 32 floats of shared memory.
template <int N, class F>
__device__ __forceinline__ void over_warps(const float (&sums)[N], float *s, F f) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; k++) s[(warp * N + k) * 32 + lane] = sums[k];
  __syncthreads();
  for (int e = threadIdx.x; e < N * 32; e += BTHREADS) {
    float v = 0.f;
    for (int w = 0; w < 8; w++) v += s[w * N * 32 + e];
    f(e >> 5, e & 31, v);
  }
}

// Layer 3: its weight gradient, gw3[o][c][u][v] = sum g[o][i][j]
// h2[c][i+u-1][j+v-1], lane = c, and the gradient of h2, gh2[c][i][j] =
// [h2 > 0] sum_o sum_{u,v} w3[o][c][u][v] g[o][i-u+1][j-v+1], thread = pixel.
constexpr int BWD3_TH = 16;
constexpr int BWD3_SMEM = (BR * BR * 4 + BR * BR * HP + 27 * CH) * 4;
__global__ void __launch_bounds__(BTHREADS) k_net_bwd3(NetBwdArgs a) {
  constexpr int TH = BWD3_TH;
  extern __shared__ __align__(16) float sm[];
  float4 *const sg = reinterpret_cast<float4 *>(sm);
  float *const sh = sm + BR * BR * 4, *const sw = sh + BR * BR * HP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < 27 * CH; e += BTHREADS)      // [o * 9 + tap][c]
    sw[e] = __bfloat162float(a.w3[(e / (9 * CH)) * KH + e % (9 * CH)]);
  float acc[30];
#pragma unroll
  for (int k = 0; k < 30; k++) acc[k] = 0.f;
  const int nt = (int)bwd_tiles<TH>(a);
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const BTile<TH> tl(a, t);
    __syncthreads();
    load_planes<false>(a, tl, a.gy, 1.f, sg);
    load_hidden(a, tl, a.h2, sh, HP);
    __syncthreads();
    for (int rr = 0; rr < 2; rr++) {
      const int r = 2 * warp + rr;
      float x[3][BR];
#pragma unroll
      for (int p = 0; p < BT; p++) {
#pragma unroll
        for (int u = 0; u < 3; u++) {
          if (p == 0) {
            x[u][0] = sh[(r + u) * BR * HP + lane];
            x[u][1] = sh[((r + u) * BR + 1) * HP + lane];
          }
          x[u][p + 2] = sh[((r + u) * BR + p + 2) * HP + lane];
        }
        const float4 g4 = sg[(r + 1) * BR + p + 1];
        const float g[3] = {g4.x, g4.y, g4.z};
#pragma unroll
        for (int o = 0; o < 3; o++) {
#pragma unroll
          for (int k = 0; k < 9; k++) acc[o * 9 + k] = fmaf(g[o], x[k / 3][p + k % 3], acc[o * 9 + k]);
          acc[27 + o] += g[o];
        }
      }
    }
    const int i = tid / BT, j = tid % BT;
    float g[27];
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const float4 v = sg[(i + 2 - k / 3) * BR + j + 2 - k % 3];
      g[k] = v.x; g[9 + k] = v.y; g[18 + k] = v.z;
    }
    const float *const hp = sh + ((i + 1) * BR + j + 1) * HP;
    const bool in = tl.i0 + i < a.H && tl.j0 + j < a.W;
    float *const dst = a.gh2 + (((size_t)tl.b * a.H + tl.i0 + i) * a.W + tl.j0 + j) * CH;
#pragma unroll 2
    for (int c = 0; c < CH; c += 4) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 27; k++) {
        const float4 w = *reinterpret_cast<const float4 *>(sw + k * CH + c);
        s.x = fmaf(w.x, g[k], s.x);
        s.y = fmaf(w.y, g[k], s.y);
        s.z = fmaf(w.z, g[k], s.z);
        s.w = fmaf(w.w, g[k], s.w);
      }
      s.x = hp[c] > 0.f ? s.x : 0.f;
      s.y = hp[c + 1] > 0.f ? s.y : 0.f;
      s.z = hp[c + 2] > 0.f ? s.z : 0.f;
      s.w = hp[c + 3] > 0.f ? s.w : 0.f;
      if (in) *reinterpret_cast<float4 *>(dst + c) = s;
    }
  }
  float *const part = a.part + (size_t)blockIdx.x * FVNA_NET_PARAMS;
  over_warps(acc, sm, [&](int k, int c, float v) {
    if (k < 27) part[NET_OFF_W3 + ((k / 9) * CH + c) * 9 + k % 9] = v;
    else if (c == 0) part[NET_OFF_B3 + k - 27] = v;
  });
}

// Layer 2's weight gradient, gw2[o][c][u][v] = sum gh2[o][i][j]
// h1[c][i+u-1][j+v-1]: lane = c, a warp for four channels o, all nine taps.
constexpr int BWD2_TH = 8;
constexpr int BWD2_SMEM = (BWD2_TH * BT * CH + (BWD2_TH + 2) * BR * CH) * 4;
__global__ void __launch_bounds__(BTHREADS, 3) k_net_bwd2(NetBwdArgs a) {
  constexpr int TH = BWD2_TH;
  extern __shared__ __align__(16) float sm[];
  float *const sg = sm, *const sh = sm + TH * BT * CH;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float acc[4][9], sb[4];
#pragma unroll
  for (int o = 0; o < 4; o++) {
    sb[o] = 0.f;
#pragma unroll
    for (int k = 0; k < 9; k++) acc[o][k] = 0.f;
  }
  const int nt = (int)bwd_tiles<TH>(a);
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const BTile<TH> tl(a, t);
    __syncthreads();
    for (int e = tid; e < TH * BT * 8; e += BTHREADS) {
      const int p = e >> 3, gi = tl.i0 + p / BT, gj = tl.j0 + p % BT;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (gi < a.H && gj < a.W)
        v = reinterpret_cast<const float4 *>(a.gh2 + (((size_t)tl.b * a.H + gi) * a.W + gj) * CH)[e & 7];
      reinterpret_cast<float4 *>(sg)[e] = v;
    }
    load_hidden(a, tl, a.h1, sh, CH);
    __syncthreads();
    for (int r = 0; r < TH; r++) {
      float x[3][BR];
#pragma unroll
      for (int p = 0; p < BT; p++) {
#pragma unroll
        for (int u = 0; u < 3; u++) {
          if (p == 0) {
            x[u][0] = sh[(r + u) * BR * CH + lane];
            x[u][1] = sh[((r + u) * BR + 1) * CH + lane];
          }
          x[u][p + 2] = sh[((r + u) * BR + p + 2) * CH + lane];
        }
        const float4 g4 = *reinterpret_cast<const float4 *>(sg + (r * BT + p) * CH + warp * 4);
        const float g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
        for (int o = 0; o < 4; o++) {
#pragma unroll
          for (int k = 0; k < 9; k++) acc[o][k] = fmaf(g[o], x[k / 3][p + k % 3], acc[o][k]);
          sb[o] += g[o];
        }
      }
    }
  }
  float *const part = a.part + (size_t)blockIdx.x * FVNA_NET_PARAMS;
#pragma unroll
  for (int o = 0; o < 4; o++) {
#pragma unroll
    for (int k = 0; k < 9; k++) part[NET_OFF_W2 + ((warp * 4 + o) * 9 + k) * CH + lane] = acc[o][k];
    if (lane == 0) part[NET_OFF_B2 + warp * 4 + o] = sb[o];
  }
}

// The gradient of h1, [h1 > 0] sum_o sum_{u,v} w2[o][c][u][v]
// gh2[o][i-u+1][j-v+1] (a thread: four pixels of a row, eight channels; a
// warp one group of channels, so that the weights are broadcast loads), then
// layer 1's weight gradient from it, gw1[o][c][u][v] = sum gh1[o][i][j]
// x[c][i+u-1][j+v-1], lane = o.
constexpr int GROW = 20;                // padded row of the transposed gradient
constexpr int BWD1_TH = 16;
constexpr int GPLANE = (BWD1_TH + 2) * GROW + 4;   // padded plane: 4 GPLANE = 16 mod 32 banks
constexpr int BWD1_SMEM = (CH * GPLANE + CH * 9 * CH + (BWD1_TH + 2) * BR * 4) * 4;
static_assert(CH * GPLANE >= BWD1_TH * BT * HP && CH * 9 * CH >= 8 * 28 * 32, "shared memory reuse");
__global__ void __launch_bounds__(BTHREADS, 2) k_net_bwd1(NetBwdArgs a) {
  constexpr int TH = BWD1_TH, RR = TH + 2;
  extern __shared__ __align__(16) float sm[];
  float *const sg = sm;                              // gh2 [o][row][col], then gh1 [pixel][o]
  float *const sw = sg + CH * GPLANE;             // [o * 9 + tap][c]
  float4 *const sx = reinterpret_cast<float4 *>(sw + CH * 9 * CH);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < CH * 9 * CH; e += BTHREADS) sw[e] = __bfloat162float(a.w2[e]);
  float acc[28];
#pragma unroll
  for (int k = 0; k < 28; k++) acc[k] = 0.f;
  // eight lanes read rows r and r + 4, whose 16-byte pieces fall in different banks
  const int c0 = (warp >> 1) * 8, col = (lane & 3) * 4;
  const int row = (warp & 1) * 8 + (lane >> 3) + (lane & 4);
  const int nt = (int)bwd_tiles<TH>(a);
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const BTile<TH> tl(a, t);
    __syncthreads();
    for (int e = tid; e < RR * BR * 8; e += BTHREADS) {
      const long long o = ring_pixel(a, tl, e >> 3);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (o >= 0) v = reinterpret_cast<const float4 *>(a.gh2 + o * CH)[e & 7];
      float *d = sg + (e & 7) * 4 * GPLANE + (e >> 3) / BR * GROW + (e >> 3) % BR;
      d[0] = v.x;
      d[GPLANE] = v.y;
      d[2 * GPLANE] = v.z;
      d[3 * GPLANE] = v.w;
    }
    load_planes<true>(a, tl, a.x, a.in_scale, sx);
    __syncthreads();
    float s[4][8];
#pragma unroll
    for (int p = 0; p < 4; p++)
#pragma unroll
      for (int k = 0; k < 8; k++) s[p][k] = 0.f;
#pragma unroll 1
    for (int o = 0; o < CH; o++) {
#pragma unroll
      for (int u = 0; u < 3; u++) {
        const float *gp = sg + o * GPLANE + (row + 2 - u) * GROW + col;
        const float4 ga = *reinterpret_cast<const float4 *>(gp);
        const float2 gb = *reinterpret_cast<const float2 *>(gp + 4);
        const float g[6] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y};
#pragma unroll
        for (int v = 0; v < 3; v++) {
          const float4 *wp = reinterpret_cast<const float4 *>(sw + (o * 9 + u * 3 + v) * CH + c0);
          const float4 wa = wp[0], wb = wp[1];
          const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int p = 0; p < 4; p++)
#pragma unroll
            for (int k = 0; k < 8; k++) s[p][k] = fmaf(w[k], g[p + 2 - v], s[p][k]);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 4; p++) {
      const int gi = tl.i0 + row, gj = tl.j0 + col + p;
      uint4 h = make_uint4(0, 0, 0, 0);
      if (gi < a.H && gj < a.W)
        h = *reinterpret_cast<const uint4 *>(a.h1 + (((size_t)tl.b * a.H + gi) * a.W + gj) * CH + c0);
      const unsigned hu[4] = {h.x, h.y, h.z, h.w};
      float *d = sg + (row * BT + col + p) * HP + c0;
#pragma unroll
      for (int k = 0; k < 8; k++) {
        const float hv = __uint_as_float(k & 1 ? hu[k >> 1] & 0xffff0000u : hu[k >> 1] << 16);
        d[k] = hv > 0.f ? s[p][k] : 0.f;
      }
    }
    __syncthreads();
    for (int r = 2 * warp; r < 2 * warp + 2; r++) {
#pragma unroll 4
      for (int p = 0; p < BT; p++) {
        const float g = sg[(r * BT + p) * HP + lane];
#pragma unroll
        for (int k = 0; k < 9; k++) {
          const float4 x = sx[(r + k / 3) * BR + p + k % 3];
          acc[k] = fmaf(g, x.x, acc[k]);
          acc[9 + k] = fmaf(g, x.y, acc[9 + k]);
          acc[18 + k] = fmaf(g, x.z, acc[18 + k]);
        }
        acc[27] += g;
      }
    }
  }
  float *const part = a.part + (size_t)blockIdx.x * FVNA_NET_PARAMS;
  over_warps(acc, sw, [&](int k, int o, float v) {
    if (k < 27) part[NET_OFF_W1 + (o * 3 + k / 9) * 9 + k % 9] = v;
    else part[NET_OFF_B1 + o] = v;
  });
}

// grads[e] = sum over the blocks' rows: eight rows at a time in pairs, these
// in binary64 (which a GB300 adds at a sixty-fourth of the FP32 rate); n1, n2,
// n3 rows hold the parameters of layers 1, 2, 3 (layer 2's weights as [o][tap][c],
// the order its kernel stores coalesced).  32 parameters and sixteen slices of
// rows a block.
__global__ void __launch_bounds__(512) k_net_reduce(const float *part, float *grads, int n1, int n2,
                                                    int n3) {
  __shared__ double s[16][32];
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  double v = 0.0;
  if (e < FVNA_NET_PARAMS) {
    const int n = e < NET_OFF_W2 ? n1 : e < NET_OFF_W3 ? n2 : n3;
    for (int b = slice; b < n; b += 128) {
      float p[8];
#pragma unroll
      for (int k = 0; k < 8; k++)
        p[k] = b + 16 * k < n ? part[(size_t)(b + 16 * k) * FVNA_NET_PARAMS + e] : 0.f;
      v += (double)(((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7])));
    }
  }
  s[slice][lane] = v;
  __syncthreads();
  if (slice == 0 && e < FVNA_NET_PARAMS) {
    for (int k = 1; k < 16; k++) v += s[k][lane];
    const int f = e - NET_OFF_W2;
    const bool w2 = e >= NET_OFF_W2 && e < NET_OFF_B2;
    grads[w2 ? NET_OFF_W2 + (f / (9 * CH) * CH + f % CH) * 9 + f / CH % 9 : e] = (float)v;
  }
}

// loss = mean over the pixels at least `margin` from the image edge of
// (y - t)^2, g = 2 (y - t) / N there and 0 elsewhere
// edges (device, batch x 4: top, bottom, left, right margins) overrides the
// uniform margin per image side: 0 where a crop side is an edge of the field.
__global__ void k_net_count(int B, int H, int W, int margin, const int *edges, long long *nin) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  long long s = 0;
  for (int b = 0; b < B; b++) {
    int t = edges ? edges[4 * b] : margin, bo = edges ? edges[4 * b + 1] : margin;
    int l = edges ? edges[4 * b + 2] : margin, r = edges ? edges[4 * b + 3] : margin;
    s += (long long)(H - t - bo) * (W - l - r);
  }
  *nin = s;
}

// grid: x over the pixels of a plane, y over the planes (batch x 3)
__global__ void k_net_mse(const float *y, const float *t, float *g, int H, int W, int planes,
                          int margin, const int *edges, const long long *nin_p, double *loss) {
  const long long nin = *nin_p;
  const int hw = H * W;
  double s = 0.0;
  for (int p = blockIdx.y; p < planes; p += gridDim.y) {
    const int b = p / 3;
    const int mt = edges ? edges[4 * b] : margin, mb = edges ? edges[4 * b + 1] : margin;
    const int ml = edges ? edges[4 * b + 2] : margin, mr = edges ? edges[4 * b + 3] : margin;
    const size_t o = (size_t)p * hw;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < hw; e += gridDim.x * blockDim.x) {
      const int i = e / W, j = e - i * W;
      const bool in = i >= mt && i < H - mb && j >= ml && j < W - mr;
      const float d = in ? y[o + e] - t[o + e] : 0.f;
      g[o + e] = 2.f * d / (float)nin;
      s += (double)d * d;
    }
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) s += red[w];
    atomicAdd(loss, s / (double)nin);
  }
}

__global__ void k_net_adam(float *p, const float *g, float *m, float *v, int n, float lr,
                           float b1, float b2, float eps, float c1, float c2) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  float gg = g[e];
  float mm = b1 * m[e] + (1.f - b1) * gg;
  float vv = b2 * v[e] + (1.f - b2) * gg * gg;
  m[e] = mm;
  v[e] = vv;
  p[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

}  // namespace fvna

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
using namespace fvna;

struct fvna_net {
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;  // FP32 master, Adam
  __nv_bfloat16 *w1 = nullptr, *w2 = nullptr, *w3 = nullptr;            // packed BF16
  __nv_bfloat16 *h1 = nullptr, *h2 = nullptr;                           // activations
  float *y = nullptr, *g3 = nullptr, *gh2 = nullptr;
  float *part = nullptr;                // the training kernels' partial sums
  int blocks[3] = {0, 0, 0};            // their persistent grids (layers 1, 2, 3)
  int fused_blocks = 0;                 // the fused forward's
  double *loss = nullptr;
  long long *nin = nullptr;
  long long cap_pix = 0;  // capacity of the activation buffers (B*H*W)
  int adam_t = 0;
};

namespace {

int cerr(cudaError_t e) {
  if (e == cudaSuccess) return FVNA_OK;
  return e == cudaErrorMemoryAllocation ? FVNA_ERR_OOM : FVNA_ERR_CUDA;
}
#define NCK(x)                          \
  do {                                  \
    cudaError_t e_ = (x);               \
    if (e_ != cudaSuccess) return cerr(e_); \
  } while (0)

void net_free_buffers(fvna_net *n) {
  cudaFree(n->h1); cudaFree(n->h2); cudaFree(n->y); cudaFree(n->g3);
  cudaFree(n->gh2);
  n->h1 = n->h2 = nullptr;
  n->y = n->g3 = n->gh2 = nullptr;
  n->cap_pix = 0;
}

int net_reserve(fvna_net *n, long long pix) {
  if (pix <= n->cap_pix) return FVNA_OK;
  net_free_buffers(n);
  NCK(cudaMalloc(&n->h1, (size_t)pix * CH * sizeof(__nv_bfloat16)));
  NCK(cudaMalloc(&n->h2, (size_t)pix * CH * sizeof(__nv_bfloat16)));
  NCK(cudaMalloc(&n->y, (size_t)pix * 3 * sizeof(float)));
  NCK(cudaMalloc(&n->g3, (size_t)pix * 3 * sizeof(float)));
  NCK(cudaMalloc(&n->gh2, (size_t)pix * CH * sizeof(float)));
  n->cap_pix = pix;
  return FVNA_OK;
}

// forward of a batch of planes into the network's own activations
int net_forward(fvna_net *n, int B, int H, int W, const float *x, float in_scale, float *y,
                cudaStream_t s) {
  const long long hw = (long long)H * W;
  if (!n->fused_blocks) {
    int dev = 0, sms = 0, occ = 0;
    NCK(cudaGetDevice(&dev));
    NCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    NCK(cudaFuncSetAttribute(k_net_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, FUSED_SMEM));
    NCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_net_fused, 256, FUSED_SMEM));
    n->fused_blocks = (occ > 0 ? occ : 1) * sms;
  }
  const int th = (H + NET_TH - 1) / NET_TH;
  const long long tiles = (long long)B * th * ((W + NET_TW - 1) / NET_TW);
  // The layers one by one where the output overlaps the input (a block's halo
  // would read what another one has written), and for many tiles with less than
  // two fifths of their pixels in the image, where the fused kernel's rings cost
  // more than its one pass saves (60,000 images of 1 x 1 1.38 ms against 1.57, 8,192 of
  // 9 x 33 0.88 against 0.98; full tiles 0.33 against 0.27, half-full ones alike).
  // A call of few tiles is three launches' latency against one's.
  const bool overlap = x < y + 3 * B * hw && y < x + 3 * B * hw;
  const bool sparse = tiles > n->fused_blocks && 5 * B * hw < 2 * tiles * NET_PIX;
  if (overlap || (sparse && B <= 65535 && th <= 65535)) {   // (grid limits of the layers)
    NCK(net_forward_launch(n, B, H, W, x, hw, W, 3 * hw, in_scale, y, hw, W, 3 * hw, 0, 1.f, n->h1,
                           n->h2, s));
    return FVNA_OK;
  }
  NetFusedArgs a;
  a.B = B; a.H = H; a.W = W;
  a.x = x; a.in_scale = in_scale; a.y = y;
  a.w1 = n->w1; a.w2 = n->w2; a.w3 = n->w3;
  a.b1 = n->params + NET_OFF_B1; a.b2 = n->params + NET_OFF_B2; a.b3 = n->params + NET_OFF_B3;
  a.h1 = n->h1; a.h2 = n->h2;
  k_net_fused<<<(int)(tiles < n->fused_blocks ? tiles : n->fused_blocks), 256, FUSED_SMEM, s>>>(a);
  NCK(cudaGetLastError());
  return FVNA_OK;
}

// the partial-sum rows, and the grids that fill the device
int net_reserve_part(fvna_net *n) {
  if (n->part) return FVNA_OK;
  int dev = 0, sms = 0;
  NCK(cudaGetDevice(&dev));
  NCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  void (*const k[3])(NetBwdArgs) = {k_net_bwd1, k_net_bwd2, k_net_bwd3};
  const int smem[3] = {BWD1_SMEM, BWD2_SMEM, BWD3_SMEM};
  int most = 1;
  for (int l = 0; l < 3; l++) {
    int occ = 0;
    NCK(cudaFuncSetAttribute(k[l], cudaFuncAttributeMaxDynamicSharedMemorySize, smem[l]));
    NCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k[l], BTHREADS, smem[l]));
    n->blocks[l] = (occ > 0 ? occ : 1) * sms;
    most = n->blocks[l] > most ? n->blocks[l] : most;
  }
  NCK(cudaMalloc(&n->part, (size_t)most * FVNA_NET_PARAMS * sizeof(float)));
  return FVNA_OK;
}

}  // namespace

namespace fvna {

cudaError_t net_pack(fvna_net *n, cudaStream_t s) {
  k_net_pack<<<64, 256, 0, s>>>(n->params, n->w1, n->w2, n->w3);
  return cudaGetLastError();
}

// The three forward launches.  in: FP32 planes (plane stride, pitch, batch
// stride in elements); out: FP32 planes (or the same planes with apply).
cudaError_t net_forward_launch(const fvna_net *n, int B, int H, int W, const float *in,
                               long long in_pstride, int in_pitch, long long in_bstride,
                               float in_scale, float *out, long long out_pstride, int out_pitch,
                               long long out_bstride, int apply, float out_scale,
                               __nv_bfloat16 *h1, __nv_bfloat16 *h2, cudaStream_t s,
                               const int *done, const long long *step, int every,
                               int band) {
  dim3 grid((W + NET_TW - 1) / NET_TW, (H + NET_TH - 1) / NET_TH, B);
  NetConvArgs a;
  std::memset(&a, 0, sizeof a);
  a.h = H; a.w = W;
  a.in = in; a.in_pstride = in_pstride; a.in_pitch = in_pitch; a.in_bstride = in_bstride;
  a.in_scale = in_scale;
  a.done = done;
  a.step = step;
  a.every = every;
  a.band = band;
  a.wmat = n->w1; a.bias = n->params + NET_OFF_B1; a.hout = h1;
  k_net_conv<0><<<grid, 256, 0, s>>>(a);
  a.hin = h1; a.wmat = n->w2; a.bias = n->params + NET_OFF_B2; a.hout = h2;
  k_net_conv<1><<<grid, 256, 0, s>>>(a);
  a.hin = h2; a.wmat = n->w3; a.bias = n->params + NET_OFF_B3;
  a.out = out; a.out_pstride = out_pstride; a.out_pitch = out_pitch; a.out_bstride = out_bstride;
  a.apply = apply; a.out_scale = out_scale;
  k_net_conv<2><<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace fvna

extern "C" {

int fvna_net_create(const float *params, fvna_net **out) {
  if (!out || !params) return FVNA_ERR_ARG;
  *out = nullptr;
  fvna_net *n = new (std::nothrow) fvna_net();
  if (!n) return FVNA_ERR_OOM;
  cudaError_t e = cudaMalloc(&n->params, 4 * FVNA_NET_PARAMS * sizeof(float));
  if (e == cudaSuccess) {
    n->grads = n->params + FVNA_NET_PARAMS;
    n->m = n->grads + FVNA_NET_PARAMS;
    n->v = n->m + FVNA_NET_PARAMS;
    e = cudaMalloc(&n->w1, (size_t)(32 * K1 + 32 * KH + 8 * KH) * sizeof(__nv_bfloat16));
  }
  if (e == cudaSuccess) {
    n->w2 = n->w1 + 32 * K1;
    n->w3 = n->w2 + 32 * KH;
    e = cudaMalloc(&n->loss, sizeof(double));
  }
  if (e == cudaSuccess) e = cudaMalloc(&n->nin, sizeof(long long));
  if (e == cudaSuccess)
    e = cudaMemcpy(n->params, params, FVNA_NET_PARAMS * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, 2 * FVNA_NET_PARAMS * sizeof(float));
  if (e == cudaSuccess) e = net_pack(n, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    fvna_net_destroy(n);
    return cerr(e);
  }
  *out = n;
  return FVNA_OK;
}

void fvna_net_destroy(fvna_net *n) {
  if (!n) return;
  cudaDeviceSynchronize();
  net_free_buffers(n);
  cudaFree(n->params);
  cudaFree(n->part);
  cudaFree(n->w1);
  cudaFree(n->loss);
  cudaFree(n->nin);
  delete n;
}

int fvna_net_params(fvna_net *n, float *dst, const float *src) {
  if (!n || (!dst && !src)) return FVNA_ERR_ARG;
  if (src) {
    NCK(cudaMemcpy(n->params, src, FVNA_NET_PARAMS * sizeof(float), cudaMemcpyHostToDevice));
    NCK(net_pack(n, 0));
  }
  if (dst) NCK(cudaMemcpy(dst, n->params, FVNA_NET_PARAMS * sizeof(float), cudaMemcpyDeviceToHost));
  NCK(cudaDeviceSynchronize());
  return FVNA_OK;
}

int fvna_net_forward(fvna_net *n, int B, int H, int W, const float *x, float in_scale, float *y,
                     unsigned short *h1_out, unsigned short *h2_out, void *stream) {
  if (!n || !x || !y || B < 1 || H < 1 || W < 1) return FVNA_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = net_reserve(n, (long long)B * H * W);
  if (rc != FVNA_OK) return rc;
  long long hw = (long long)H * W;
  rc = net_forward(n, B, H, W, x, in_scale, y, s);
  if (rc != FVNA_OK) return rc;
  size_t hb = (size_t)B * hw * CH * sizeof(__nv_bfloat16);
  if (h1_out) NCK(cudaMemcpyAsync(h1_out, n->h1, hb, cudaMemcpyDeviceToDevice, s));
  if (h2_out) NCK(cudaMemcpyAsync(h2_out, n->h2, hb, cudaMemcpyDeviceToDevice, s));
  NCK(cudaStreamSynchronize(s));
  return FVNA_OK;
}

int fvna_net_backward(fvna_net *n, int B, int H, int W, const float *x, float in_scale,
                      const float *gy, float *grads, void *stream) {
  if (!n || !x || !gy || B < 1 || H < 1 || W < 1) return FVNA_ERR_ARG;
  if ((long long)B * H * W > n->cap_pix) return FVNA_ERR_ARG;  // needs the forward's activations
  cudaStream_t s = (cudaStream_t)stream;
  int rc = net_reserve_part(n);
  if (rc != FVNA_OK) return rc;
  NetBwdArgs a;
  a.B = B; a.H = H; a.W = W;
  a.gy = gy; a.x = x; a.in_scale = in_scale;
  a.h1 = n->h1; a.h2 = n->h2; a.w2 = n->w2; a.w3 = n->w3;
  a.gh2 = n->gh2; a.part = n->part;
  const long long tiles[3] = {bwd_tiles<BWD1_TH>(a), bwd_tiles<BWD2_TH>(a), bwd_tiles<BWD3_TH>(a)};
  if (tiles[0] > 0x7fffffff || tiles[1] > 0x7fffffff) return FVNA_ERR_ARG;
  int nb[3];
  for (int k = 0; k < 3; k++) nb[k] = (int)(tiles[k] < n->blocks[k] ? tiles[k] : n->blocks[k]);
  k_net_bwd3<<<nb[2], BTHREADS, BWD3_SMEM, s>>>(a);
  k_net_bwd2<<<nb[1], BTHREADS, BWD2_SMEM, s>>>(a);
  k_net_bwd1<<<nb[0], BTHREADS, BWD1_SMEM, s>>>(a);
  k_net_reduce<<<(FVNA_NET_PARAMS + 31) / 32, 512, 0, s>>>(n->part, n->grads, nb[0], nb[1], nb[2]);
  NCK(cudaGetLastError());
  if (grads) NCK(cudaMemcpyAsync(grads, n->grads, FVNA_NET_PARAMS * sizeof(float), cudaMemcpyDeviceToDevice, s));
  NCK(cudaStreamSynchronize(s));
  return FVNA_OK;
}

int fvna_net_train_step(fvna_net *n, int B, int H, int W, const float *x, float in_scale,
                        const float *target, int margin, const int *edges, float lr, double *loss,
                        void *stream) {
  if (!n || !x || !target || B < 1 || H < 1 || W < 1 || !(lr > 0.f)) return FVNA_ERR_ARG;
  if (margin < 0 || 2 * margin >= H || 2 * margin >= W) return FVNA_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = net_reserve(n, (long long)B * H * W);
  if (rc != FVNA_OK) return rc;
  long long hw = (long long)H * W;
  rc = net_forward(n, B, H, W, x, in_scale, n->y, s);
  if (rc != FVNA_OK) return rc;
  NCK(cudaMemsetAsync(n->loss, 0, sizeof(double), s));
  k_net_count<<<1, 32, 0, s>>>(B, H, W, margin, edges, n->nin);
  const long long px = (hw + 255) / 256;
  const dim3 grid((unsigned)(px < 64 ? px : 64), (unsigned)(3LL * B < 4096 ? 3 * B : 4096));
  k_net_mse<<<grid, 256, 0, s>>>(n->y, target, n->g3, H, W, 3 * B, margin, edges, n->nin, n->loss);
  NCK(cudaGetLastError());
  rc = fvna_net_backward(n, B, H, W, x, in_scale, n->g3, nullptr, stream);
  if (rc != FVNA_OK) return rc;
  n->adam_t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  float c1 = 1.f - powf(b1, (float)n->adam_t), c2 = 1.f - powf(b2, (float)n->adam_t);
  k_net_adam<<<(FVNA_NET_PARAMS + 255) / 256, 256, 0, s>>>(n->params, n->grads, n->m, n->v,
                                                           FVNA_NET_PARAMS, lr, b1, b2, 1e-8f, c1, c2);
  NCK(cudaGetLastError());
  NCK(net_pack(n, s));
  if (loss) NCK(cudaMemcpyAsync(loss, n->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
  NCK(cudaStreamSynchronize(s));
  return FVNA_OK;
}

}  // extern "C"
