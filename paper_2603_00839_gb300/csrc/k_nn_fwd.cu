// Forward 3x3 convolutions of the warm-start network on a shared-memory tile
// (the general implicit GEMM for other channel counts is in k_nn.cu).
//
// Both kernels sum in the order of the general one: k = (tap, channel) in
// steps of 16 through one accumulator, K cut into the same slices, whose sums
// are added in order; so every layer's result is the same bit for bit whichever
// kernel runs it.
#include <cuda_bf16.h>

#include "nn_internal.cuh"
#include "nn_mma.cuh"
#include "rtg_internal.cuh"

namespace rtg {
namespace nn {

constexpr int FT_A = 8, FT_B = 16;   // output pixels of a CTA

struct FwdEpilogue {
  const float* bias;
  float* rout;          // act(conv + b), channels last (or null)
  const float* skip;    // added to it for out (or null)
  float* out;           // channels last, or planar (or null)
  const float* planar;  // not null: out = planar + result in the solver's planar layout
  int relu;
};

__device__ __forceinline__ void fwd_store(const FwdEpilogue& ep, float v, int c, int cout, int64_t pix, int n, int HW,
                                          int64_t in_img) {
  v += ep.bias ? ep.bias[c] : 0.f;
  if (ep.relu) v = fmaxf(v, 0.f);
  if (ep.planar != nullptr) {
    const int64_t o = (static_cast<int64_t>(n) * cout + c) * HW + in_img;
    ep.out[o] = ep.planar[o] + v;
    return;
  }
  const int64_t o = pix * cout + c;
  if (ep.rout != nullptr) ep.rout[o] = v;
  if (ep.out != nullptr) ep.out[o] = ep.skip ? v + ep.skip[o] : v;
}

// Channels in whole steps of 16.  CTA: 8 x 16 output pixels x BN channels;
// the input tile with its halo is converted to BF16 once (a patch entry was
// gathered from global memory and rounded for each of its nine taps before),
// an up-sampled input is kept at its stored resolution (a third of the
// pixels); the weights of a tap arrive with cp.async while the tap before is
// multiplied; all operands go through ldmatrix.  Eight warps, 4 along the
// pixels x 2 along the channels (8 x 1 for BN = 8).  SPLIT: K is cut every
// `kchunk` values and the slices are added in a second accumulator.
// 512 x 512, 64 -> 32 channels from an up-sampled input: 69.8 us (138 TFLOP/s),
// warps waiting for the tile's loads (long scoreboard 3.4 an instruction; tensor
// pipe 22 % busy, four CTAs an SM by registers).  Inference on one 512 x 512
// image, every layer on the general kernel: 912 us; with this one 314.
template <int BN, bool SPLIT>
__global__ void __launch_bounds__(256)
k_conv_tile(const float* __restrict__ x, const __nv_bfloat16* __restrict__ wt, FwdEpilogue ep, int H, int W, int C,
            int stride, int cout, int up, int kchunk, int tilesb) {
  extern __shared__ __align__(16) unsigned char ft_smem[];
  const int PC = C + 8;   // pitch of a pixel and of a weight row: an odd number of 16-byte pieces
  const int hr = up ? FT_A / 2 + 2 : (FT_A - 1) * stride + 3;   // stored rows and columns of the tile
  const int hc = up ? FT_B / 2 + 2 : (FT_B - 1) * stride + 3;
  __nv_bfloat16* tile = reinterpret_cast<__nv_bfloat16*>(ft_smem);   // [hr * hc][PC]
  __nv_bfloat16* Bs = tile + hr * hc * PC;                           // [2][BN][PC]
  constexpr int WN = BN >= 16 ? 2 : 1, WM = 8 / WN;                  // warps
  constexpr int MT = 8 / WM, NT = BN / (8 * WN);                     // m16 tiles (tile rows), n8 tiles per warp
  const int Ho = H / stride, Wo = W / stride;
  const int Hs = up ? H / 2 : H, Ws = up ? W / 2 : W;
  const int n = blockIdx.z, a0 = (blockIdx.x / tilesb) * FT_A, b0 = (blockIdx.x % tilesb) * FT_B;
  const int n0 = blockIdx.y * BN;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const int wm = (warp % WM) * MT, wn = (warp / WM) * 8 * NT;
  const int cpc = C / 8;
  auto load_w = [&](int tap, int buf) {   // one cp.async group
    __nv_bfloat16* dst = Bs + buf * BN * PC;
    for (int e = tid; e < BN * cpc; e += 256) {
      const int o = e / cpc, c = (e - o * cpc) * 8;
      const bool v = n0 + o < cout;
      const __nv_bfloat16* src = v ? wt + (static_cast<int64_t>(n0 + o) * 9 + tap) * C + c : wt;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(dst + o * PC + c)), "l"(src),
                   "r"(v ? 16 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  load_w(0, 0);
  {   // the input tile: stored row / column of the tile's origin
    const int y0 = up ? a0 / 2 - 1 : a0 * stride - 1, x0 = up ? b0 / 2 - 1 : b0 * stride - 1;
    // four pieces of eight channels per round, their loads in flight together
    for (int e0 = tid; e0 < hr * hc * cpc; e0 += 4 * 256) {
      float4 p[4], q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * 256, pix = e / cpc, c = (e - pix * cpc) * 8;
        const int y = y0 + pix / hc, xx = x0 + pix % hc;
        p[u] = q[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < hr * hc * cpc && y >= 0 && y < Hs && xx >= 0 && xx < Ws) {
          const float4* s4 = reinterpret_cast<const float4*>(x + ((static_cast<int64_t>(n) * Hs + y) * Ws + xx) * C + c);
          p[u] = s4[0];
          q[u] = s4[1];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * 256, pix = e / cpc, c = (e - pix * cpc) * 8;
        if (e < hr * hc * cpc)
          *reinterpret_cast<uint4*>(tile + pix * PC + c) =
              make_uint4(pack_bf16(p[u].x, p[u].y), pack_bf16(p[u].z, p[u].w), pack_bf16(q[u].x, q[u].y),
                         pack_bf16(q[u].z, q[u].w));
      }
    }
  }
  float acc[MT][NT][4], tot[SPLIT ? MT : 1][SPLIT ? NT : 1][4];
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int b = 0; b < NT; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        acc[a][b][c] = 0.f;
        if constexpr (SPLIT) tot[a][b][c] = 0.f;
      }
  const int mi = lane >> 3, r8 = lane & 7;
  const int pb = (mi & 1) * 8 + r8;   // this lane's row of the A tiles: output column
  int k = 0, next_cut = kchunk;
  for (int tap = 0; tap < 9; ++tap) {
    const int ky = tap / 3, kx = tap - 3 * ky;
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();   // the tap's weights (and the tile) are there, the other buffer is free
    if (tap < 8) load_w(tap + 1, (tap + 1) & 1);
    const __nv_bfloat16* B = Bs + (tap & 1) * BN * PC;
    uint32_t arow[MT];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      const int a = wm + mt;
      // tile row / column of input pixel (s a + ky - 1, s b + kx - 1)
      const int row = up ? (a + ky + 1) >> 1 : a * stride + ky, col = up ? (pb + kx + 1) >> 1 : pb * stride + kx;
      arow[mt] = smem_addr(tile + (row * hc + col) * PC + (mi >> 1) * 8);
    }
    const uint32_t brow = smem_addr(B + (wn + (BN >= 16 ? (mi >> 1) * 8 : 0) + r8) * PC + (mi & 1) * 8);
    for (int c = 0; c < C; c += 16) {
      if constexpr (SPLIT) {
        if (k == next_cut) {
#pragma unroll
          for (int a = 0; a < MT; ++a)
#pragma unroll
            for (int b = 0; b < NT; ++b)
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                tot[a][b][q] += acc[a][b][q];
                acc[a][b][q] = 0.f;
              }
          next_cut += kchunk;
        }
        k += 16;
      }
      uint32_t a[MT][4];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) ldsm_x4(a[mt], arow[mt] + c * 2);
      if constexpr (BN >= 16) {
#pragma unroll
        for (int nt = 0; nt < NT; nt += 2) {
          uint32_t b[4];
          ldsm_x4(b, brow + (nt * 8 * PC + c) * 2);
#pragma unroll
          for (int mt = 0; mt < MT; ++mt) {
            mma_k16(acc[mt][nt], a[mt], b[0], b[1]);
            mma_k16(acc[mt][nt + 1], a[mt], b[2], b[3]);
          }
        }
      } else {
        uint32_t b[4];   // (the upper pair repeats the lower)
        ldsm_x4(b, brow + c * 2);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) mma_k16(acc[mt][0], a[mt], b[0], b[1]);
      }
    }
  }
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    const int a = a0 + wm + mt;
    if (a >= Ho) continue;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int b = b0 + gid + 8 * h;
        if (b >= Wo) continue;
        const int64_t in_img = static_cast<int64_t>(a) * Wo + b;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int c = n0 + wn + nt * 8 + tig * 2 + q;
          if (c >= cout) continue;
          float v = acc[mt][nt][2 * h + q];
          if constexpr (SPLIT) v = tot[mt][nt][2 * h + q] + v;
          fwd_store(ep, v, c, cout, static_cast<int64_t>(n) * Ho * Wo + in_img, n, Ho * Wo, in_img);
        }
      }
  }
}

// The input layer: three channels, K = 27 patch entries padded to 32.  CTA: 8
// x 16 pixels; a thread's eight patch entries sit at fixed offsets from its
// pixel in the BF16 tile, so a fragment is eight 2-byte shared loads.  planar:
// x in the solver's planar layout.  Bound by the output's stores.
template <int BN>
__global__ void __launch_bounds__(256)
k_conv_in3(const float* __restrict__ x, const __nv_bfloat16* __restrict__ wt, FwdEpilogue ep, int H, int W, int stride,
           int cout, int planar, int tilesb) {
  constexpr int HR = (FT_A - 1) * 2 + 3, HC = (FT_B - 1) * 2 + 3;   // stride 2's tile
  __shared__ __nv_bfloat16 tile[HR * HC * 3];
  __shared__ __align__(4) __nv_bfloat16 Bs[BN][34];
  const int hr = (FT_A - 1) * stride + 3, hc = (FT_B - 1) * stride + 3;
  const int Ho = H / stride, Wo = W / stride;
  const int n = blockIdx.z, a0 = (blockIdx.x / tilesb) * FT_A, b0 = (blockIdx.x % tilesb) * FT_B;
  const int n0 = blockIdx.y * BN;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
  for (int e = tid; e < BN * 32; e += 256) {
    const int o = e >> 5, k = e & 31;
    Bs[o][k] = (n0 + o < cout && k < 27) ? wt[static_cast<int64_t>(n0 + o) * 27 + k] : __float2bfloat16(0.f);
  }
  for (int e = tid; e < hr * hc * 3; e += 256) {
    int pix, c;
    if (planar) {
      c = e / (hr * hc);
      pix = e - c * hr * hc;
    } else {
      pix = e / 3;
      c = e - 3 * pix;
    }
    const int y = a0 * stride - 1 + pix / hc, xx = b0 * stride - 1 + pix % hc;
    float v = 0.f;
    if (y >= 0 && y < H && xx >= 0 && xx < W)
      v = planar ? x[((static_cast<int64_t>(n) * 3 + c) * H + y) * W + xx]
                 : x[((static_cast<int64_t>(n) * H + y) * W + xx) * 3 + c];
    tile[pix * 3 + c] = __float2bfloat16(v);
  }
  __syncthreads();
  // offsets of this thread's patch entries: k = 16 s + 2 tig + {0, 1, 8, 9}, s = 0, 1
  int off[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int k = min(26, 16 * (u >> 2) + 2 * tig + (u & 1) + 8 * ((u >> 1) & 1));
    off[u] = ((k / 9) * hc + (k % 9) / 3) * 3 + k % 3;
  }
  const unsigned short* tl = reinterpret_cast<const unsigned short*>(tile);
  const int a = warp;   // warp w: tile row w, 16 pixels
  float acc[BN / 8][4];
#pragma unroll
  for (int b = 0; b < BN / 8; ++b)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[b][c] = 0.f;
  // entries past the 27: zeros, as in the general kernel (a real value there would
  // meet a zero weight, and an infinite one would make a NaN of it)
  const uint32_t tail = tig == 0 ? 0xffffffffu : (tig == 1 ? 0xffffu : 0u);   // k = 24 + 2 tig, + 1
  const unsigned short* p0 = tl + (a * stride * hc + gid * stride) * 3;
  const unsigned short* p1 = p0 + 8 * stride * 3;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    uint32_t af[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // k pair, then k pair + 8
      const int u = 4 * s + 2 * h;
      af[2 * h] = static_cast<uint32_t>(p0[off[u]]) | static_cast<uint32_t>(p0[off[u + 1]]) << 16;
      af[2 * h + 1] = static_cast<uint32_t>(p1[off[u]]) | static_cast<uint32_t>(p1[off[u + 1]]) << 16;
      if (u == 6) {
        af[2 * h] &= tail;
        af[2 * h + 1] &= tail;
      }
    }
#pragma unroll
    for (int nt = 0; nt < BN / 8; ++nt) {
      const uint32_t b0r = *reinterpret_cast<const uint32_t*>(&Bs[nt * 8 + gid][16 * s + 2 * tig]);
      const uint32_t b1r = *reinterpret_cast<const uint32_t*>(&Bs[nt * 8 + gid][16 * s + 2 * tig + 8]);
      mma_k16(acc[nt], af, b0r, b1r);
    }
  }
  if (a0 + a >= Ho) return;
#pragma unroll
  for (int nt = 0; nt < BN / 8; ++nt)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int b = b0 + gid + 8 * h;
      if (b >= Wo) continue;
      const int64_t in_img = static_cast<int64_t>(a0 + a) * Wo + b;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int c = n0 + nt * 8 + tig * 2 + q;
        if (c < cout)
          fwd_store(ep, acc[nt][2 * h + q], c, cout, static_cast<int64_t>(n) * Ho * Wo + in_img, n, Ho * Wo, in_img);
      }
    }
}

static size_t tile_smem(int bn, int C, int stride, bool up) {
  const int hr = up ? FT_A / 2 + 2 : (FT_A - 1) * stride + 3, hc = up ? FT_B / 2 + 2 : (FT_B - 1) * stride + 3;
  return (size_t(hr) * hc + size_t(2) * bn) * (C + 8) * 2;
}

// The tile kernels take three channels, or whole steps of 16 channels whose
// tile fits shared memory and 16-byte aligned operands (an up-sampled input
// also an even grid); anything else runs the general kernel.
int conv_tile_kind(const float* x, const __nv_bfloat16* w, int H, int W, int C, int stride, int bn, bool up) {
  if (C == 3 && !up && stride <= 2) return 1;
  if (C % 16 != 0 || reinterpret_cast<uintptr_t>(x) % 16 != 0 || reinterpret_cast<uintptr_t>(w) % 16 != 0) return 0;
  if (up && (stride != 1 || H % 2 || W % 2)) return 0;
  return tile_smem(bn, C, stride, up) <= size_t(220) * 1024 ? 2 : 0;
}

cudaError_t conv_tile(int kind, const float* x, const __nv_bfloat16* w, const float* bias, float* r, const float* skip,
                      float* out, const float* planar_add, bool planar_in, int N, int H, int W, int C, int stride,
                      int cout, bool relu, bool up, int bn, int kchunk, cudaStream_t s) {
  const int Ho = H / stride, Wo = W / stride;
  const int ta = (Ho + FT_A - 1) / FT_A, tb = (Wo + FT_B - 1) / FT_B;
  const bool split = kchunk < 9 * C;
  // fewer channels per CTA where the tiles alone leave SMs idle (32 x 32 tiles at
  // 128 channels: 32 CTAs of 128, 128 of 32); the result does not depend on it
  while (bn > 32 && int64_t(ta) * tb * N * ((cout + bn - 1) / bn) < 152) bn /= 2;
  const size_t smem = tile_smem(bn, C, stride, up);
  for (int n0 = 0; n0 < N; n0 += 65535) {   // the grid's z limit
    const int nn = N - n0 < 65535 ? N - n0 : 65535;
    const int64_t io = int64_t(n0) * (up ? H / 2 : H) * (up ? W / 2 : W) * C, oo = int64_t(n0) * Ho * Wo * cout;
    const FwdEpilogue ep{bias,           r ? r + oo : nullptr,
                         skip ? skip + oo : nullptr, out ? out + oo : nullptr,
                         planar_add ? planar_add + oo : nullptr, relu ? 1 : 0};
    const dim3 grid(ta * tb, (cout + bn - 1) / bn, nn);
    cudaError_t e = cudaSuccess;
#define RTG_TILE_CASE(B_)                                                                                         \
  if (bn == B_) {                                                                                                 \
    if (kind == 1) {                                                                                              \
      k_conv_in3<B_><<<grid, 256, 0, s>>>(x + io, w, ep, H, W, stride, cout, planar_in ? 1 : 0, tb);               \
    } else if (split) {                                                                                           \
      e = set_smem(k_conv_tile<B_, true>, smem);                                                                  \
      if (e != cudaSuccess) return e;                                                                             \
      k_conv_tile<B_, true><<<grid, 256, smem, s>>>(x + io, w, ep, H, W, C, stride, cout, up ? 1 : 0, kchunk, tb); \
    } else {                                                                                                      \
      e = set_smem(k_conv_tile<B_, false>, smem);                                                                 \
      if (e != cudaSuccess) return e;                                                                             \
      k_conv_tile<B_, false><<<grid, 256, smem, s>>>(x + io, w, ep, H, W, C, stride, cout, up ? 1 : 0, kchunk, tb); \
    }                                                                                                             \
  }
    RTG_TILE_CASE(8) RTG_TILE_CASE(32) RTG_TILE_CASE(64) RTG_TILE_CASE(128)
#undef RTG_TILE_CASE
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace nn
}  // namespace rtg
