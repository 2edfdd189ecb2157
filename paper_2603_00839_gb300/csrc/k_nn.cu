// Kernels of the learned warm start (a convolutional encoder-decoder that
// predicts X_0 and log(lambda) from C).  Activations are FP32 and channels
// last (N, H, W, C); 3x3 convolutions with zero padding 1 run on BF16
// tensor cores with FP32 accumulation; here the forward pass, an implicit
// GEMM that gathers its patches from the activations, and the small kernels
// (layout changes, pooling, the lambda head, Adam).  The convolutions'
// gradients and the loss are in k_nn_bwd.cu.
#include <cuda_bf16.h>

#include "nn_internal.cuh"
#include "nn_mma.cuh"

namespace rtg {
namespace nn {

static unsigned grid_of(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 32) b = 152 * 32;
  return static_cast<unsigned>(b < 1 ? 1 : b);
}

// ------------------------------------------------------------------ implicit-GEMM convolution
// Forward 3x3 convolution without a materialised im2col: the A tile (128
// output pixels x 32 of the 9 c_in patch entries) is gathered from the
// channels-last input while the previous tile is multiplied.  When
// c_in % 32 == 0 a 32-wide K slice is one tap and 32 consecutive channels,
// i.e. 8 float4 per pixel; otherwise (the 3-channel input layer) entries are
// gathered one by one.  Weights (c_out x K, BF16) come in 16-byte pieces
// when K % 8 == 0.  The epilogue adds the bias, applies the ReLU and the skip
// sum and stores FP32: r = act(acc + b) (optional), out = r + skip.
// Eight warps; warp w owns output rows 16w..16w+15 and all BN channels.
constexpr int CBM = 128, CBK = 32, CPAD = 8;

// up = 1: x holds the half-resolution tensor (H/2 x W/2) and the layer
// reads its nearest x2 up-sampling without materialising it.  gridDim.z > 1
// splits K: slice z writes its raw sums to part + z * M * cout and the
// epilogue runs in k_conv_split_epilogue.
template <int BN>
__global__ void __launch_bounds__(256, BN <= 64 ? 3 : 2)
k_conv_fwd(const float* __restrict__ x, const __nv_bfloat16* __restrict__ wt, const float* __restrict__ bias,
           float* __restrict__ rout, const float* __restrict__ skip, float* __restrict__ out, int N, int H, int W,
           int C, int stride, int cout, int relu, int up, int kchunk, float* __restrict__ part) {
  __shared__ __align__(16) __nv_bfloat16 As[2][CBM][CBK + CPAD];
  __shared__ __align__(16) __nv_bfloat16 Bs[2][BN][CBK + CPAD];
  constexpr int NB = (BN * 4 + 255) / 256;   // 16-byte weight pieces per thread
  const int Ho = H / stride, Wo = W / stride;
  const int M = N * Ho * Wo, Kfull = 9 * C;
  const int kbeg = blockIdx.z * kchunk;
  const int K = min(Kfull, kbeg + kchunk);   // this slice covers [kbeg, K)
  const int Hs = up ? H / 2 : H, Ws = up ? W / 2 : W, sh = up ? 1 : 0;   // stored input grid
  const int m0 = blockIdx.x * CBM, n0 = blockIdx.y * BN;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const bool fastA = (C % 32) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const bool fastB = (Kfull % 8) == 0;
  float4 ra[4];
  float rs[16];
  uint4 rb[NB];
  auto load_tiles = [&](int k0) {
    if (fastA) {
      const int tap = k0 / C, c0 = k0 - tap * C, ky = tap / 3, kx = tap - ky * 3;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = tid + q * 256, row = e >> 3, piece = e & 7;
        const int m = m0 + row;
        ra[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m < M) {
          const int j = m % Wo, i = (m / Wo) % Ho, n = m / (Wo * Ho);
          const int yy = stride * i + ky - 1, xx = stride * j + kx - 1;
          if (yy >= 0 && yy < H && xx >= 0 && xx < W)
            ra[q] = *reinterpret_cast<const float4*>(
                x + ((static_cast<int64_t>(n) * Hs + (yy >> sh)) * Ws + (xx >> sh)) * C + c0 + piece * 4);
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int e = tid + q * 256, row = e >> 5, kk = e & 31;
        const int m = m0 + row, k = k0 + kk;
        rs[q] = 0.f;
        if (m < M && k < K) {
          const int c = k % C, t = k / C, kx = t % 3, ky = t / 3;
          const int j = m % Wo, i = (m / Wo) % Ho, n = m / (Wo * Ho);
          const int yy = stride * i + ky - 1, xx = stride * j + kx - 1;
          if (yy >= 0 && yy < H && xx >= 0 && xx < W)
            rs[q] = x[((static_cast<int64_t>(n) * Hs + (yy >> sh)) * Ws + (xx >> sh)) * C + c];
        }
      }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + q * 256, row = e >> 2, piece = e & 3;
      rb[q] = make_uint4(0u, 0u, 0u, 0u);
      if (row < BN && n0 + row < cout) {
        const int k = k0 + piece * 8;
        if (fastB && k + 8 <= K) {
          rb[q] = *reinterpret_cast<const uint4*>(wt + static_cast<int64_t>(n0 + row) * Kfull + k);
        } else {
          __nv_bfloat16 t8[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            t8[u] = (k + u < K) ? wt[static_cast<int64_t>(n0 + row) * Kfull + k + u] : __float2bfloat16(0.f);
          rb[q] = *reinterpret_cast<const uint4*>(t8);
        }
      }
    }
  };
  auto store_tiles = [&](int buf) {
    if (fastA) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = tid + q * 256, row = e >> 3, piece = e & 7;
        __nv_bfloat162 h0 = __floats2bfloat162_rn(ra[q].x, ra[q].y);
        __nv_bfloat162 h1 = __floats2bfloat162_rn(ra[q].z, ra[q].w);
        uint2 v;
        v.x = *reinterpret_cast<uint32_t*>(&h0);
        v.y = *reinterpret_cast<uint32_t*>(&h1);
        *reinterpret_cast<uint2*>(&As[buf][row][piece * 4]) = v;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int e = tid + q * 256, row = e >> 5, kk = e & 31;
        As[buf][row][kk] = __float2bfloat16(rs[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + q * 256, row = e >> 2, piece = e & 3;
      if (row < BN) *reinterpret_cast<uint4*>(&Bs[buf][row][piece * 8]) = rb[q];
    }
  };
  float acc[BN / 8][4];
#pragma unroll
  for (int a = 0; a < BN / 8; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[a][c] = 0.f;
  load_tiles(kbeg);
  store_tiles(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = kbeg; k0 < K; k0 += CBK) {
    const bool more = k0 + CBK < K;
    if (more) load_tiles(k0 + CBK);   // in flight during the products
#pragma unroll
    for (int kk = 0; kk < CBK; kk += 16) {
      uint32_t af[4];
      const int r = warp * 16 + gid;
      af[0] = *reinterpret_cast<const uint32_t*>(&As[buf][r][kk + tig * 2]);
      af[1] = *reinterpret_cast<const uint32_t*>(&As[buf][r + 8][kk + tig * 2]);
      af[2] = *reinterpret_cast<const uint32_t*>(&As[buf][r][kk + tig * 2 + 8]);
      af[3] = *reinterpret_cast<const uint32_t*>(&As[buf][r + 8][kk + tig * 2 + 8]);
#pragma unroll
      for (int nt = 0; nt < BN / 8; ++nt) {
        const uint32_t b0 = *reinterpret_cast<const uint32_t*>(&Bs[buf][nt * 8 + gid][kk + tig * 2]);
        const uint32_t b1 = *reinterpret_cast<const uint32_t*>(&Bs[buf][nt * 8 + gid][kk + tig * 2 + 8]);
        mma_k16(acc[nt], af, b0, b1);
      }
    }
    if (more) {
      store_tiles(buf ^ 1);   // the other buffer: nobody reads it during this step
      __syncthreads();
      buf ^= 1;
    }
  }
#pragma unroll
  for (int nt = 0; nt < BN / 8; ++nt)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = m0 + warp * 16 + gid + h * 8;
      if (m >= M) continue;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int c = n0 + nt * 8 + tig * 2 + q;
        if (c >= cout) continue;
        if (gridDim.z > 1) {
          part[(static_cast<int64_t>(blockIdx.z) * M + m) * cout + c] = acc[nt][2 * h + q];
          continue;
        }
        float v = acc[nt][2 * h + q] + (bias ? bias[c] : 0.f);
        if (relu) v = fmaxf(v, 0.f);
        const int64_t o = static_cast<int64_t>(m) * cout + c;
        if (rout != nullptr) rout[o] = v;
        if (out != nullptr) out[o] = skip ? v + skip[o] : v;
      }
    }
}

// Epilogue of a K-split convolution: sum the slices in order, then bias,
// activation and skip as in k_conv_fwd.
__global__ void k_conv_split_epilogue(const float* __restrict__ part, const float* __restrict__ bias,
                                      float* __restrict__ rout, const float* __restrict__ skip,
                                      float* __restrict__ out, int64_t MC, int cout, int nz, int relu) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < MC;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    float v = 0.f;
    for (int z = 0; z < nz; ++z) v += part[static_cast<int64_t>(z) * MC + i];
    v += bias ? bias[i % cout] : 0.f;
    if (relu) v = fmaxf(v, 0.f);
    if (rout != nullptr) rout[i] = v;
    if (out != nullptr) out[i] = skip ? v + skip[i] : v;
  }
}

// Tiles of a forward convolution and the slices of K (whole 32-wide steps) that
// fill the GPU when the tiles alone leave SMs idle; slices > 1 need slices * M *
// cout floats of scratch.
struct FwdSplit {
  int bn, mtiles, ntiles, splits, kchunk;
};
static FwdSplit fwd_split(int N, int H, int W, int C, int stride, int cout, bool may_split, int64_t part_floats) {
  const int M = N * (H / stride) * (W / stride), K = 9 * C;
  FwdSplit f;
  f.bn = cout <= 8 ? 8 : (cout <= 32 ? 32 : (cout <= 64 ? 64 : 128));
  f.mtiles = (M + CBM - 1) / CBM;
  f.ntiles = (cout + f.bn - 1) / f.bn;
  f.splits = 1;
  if (may_split && f.mtiles * f.ntiles < 152) {
    f.splits = (304 + f.mtiles * f.ntiles - 1) / (f.mtiles * f.ntiles);
    const int ksteps = (K + CBK - 1) / CBK;
    if (f.splits > ksteps / 2) f.splits = ksteps / 2 > 1 ? ksteps / 2 : 1;
    while (f.splits > 1 && int64_t(f.splits) * M * cout > part_floats) --f.splits;
  }
  f.kchunk = (K + f.splits - 1) / f.splits;
  f.kchunk = ((f.kchunk + CBK - 1) / CBK) * CBK;
  f.splits = (K + f.kchunk - 1) / f.kchunk;
  return f;
}

int64_t conv_fwd_scratch(int N, int H, int W, int C, int stride, int cout) {
  // (the slices before rounding K to whole steps: the bound of the search above)
  const FwdSplit f = fwd_split(N, H, W, C, stride, cout, true, int64_t(1) << 62);
  const int64_t per = int64_t(N) * (H / stride) * (W / stride) * cout;
  const int64_t most = (304 + f.mtiles * f.ntiles - 1) / (f.mtiles * f.ntiles);
  return f.splits > 1 ? (most > f.splits ? most : f.splits) * per : 0;
}

cudaError_t conv_fwd(const float* x, const __nv_bfloat16* w, const float* bias, float* r, const float* skip,
                     float* out, int N, int H, int W, int C, int stride, int cout, bool relu, bool up,
                     float* part, int64_t part_floats, cudaStream_t s, bool planar_in, const float* planar_add) {
  const int M = N * (H / stride) * (W / stride);
  const FwdSplit f = fwd_split(N, H, W, C, stride, cout, part != nullptr, part_floats);
  const int bn = f.bn, mtiles = f.mtiles, ntiles = f.ntiles, splits = f.splits, kchunk = f.kchunk;
  // the tile kernels read an input tile once for all taps; they cut K where the
  // slices would, so the choice does not change the result
  if (const int kind = conv_tile_kind(x, w, H, W, C, stride, bn, up))
    return conv_tile(kind, x, w, bias, r, skip, out, planar_add, planar_in, N, H, W, C, stride, cout, relu, up, bn,
                     kchunk, s);
  if (planar_in || planar_add != nullptr) return cudaErrorInvalidValue;
  dim3 grid(mtiles, ntiles, splits);
  const int rl = relu ? 1 : 0, u = up ? 1 : 0;
#define RTG_CONV_CASE(B_)                                                                                   \
  if (bn == B_)                                                                                             \
    k_conv_fwd<B_><<<grid, 256, 0, s>>>(x, w, bias, r, skip, out, N, H, W, C, stride, cout, rl, u, kchunk, part);
  RTG_CONV_CASE(8) RTG_CONV_CASE(32) RTG_CONV_CASE(64) RTG_CONV_CASE(128)
#undef RTG_CONV_CASE
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || splits == 1) return e;
  const int64_t MC = int64_t(M) * cout;
  k_conv_split_epilogue<<<grid_of(MC), 256, 0, s>>>(part, bias, r, skip, out, MC, cout, splits, rl);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ elementwise
// solver layout (per image x fastest, then y, then channel) <-> channels last
__global__ void k_to_nhwc(const float* __restrict__ src, float* __restrict__ dst, int64_t pixels, int HW, int C) {
  for (int64_t p = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; p < pixels;
       p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t n = p / HW;
    for (int c = 0; c < C; ++c) dst[p * C + c] = src[(n * (C - 1) + c) * HW + p];   // image n starts at n C HW
  }
}

// dst (solver layout) = base (solver layout) + src (channels last)
__global__ void k_from_nhwc_add(const float* __restrict__ src, const float* __restrict__ base,
                                float* __restrict__ dst, int N, int H, int W, int C) {
  const int64_t total = static_cast<int64_t>(N) * H * W * C;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < total;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int x = static_cast<int>(e % W);
    const int y = static_cast<int>((e / W) % H);
    const int c = static_cast<int>((e / (static_cast<int64_t>(W) * H)) % C);
    const int n = static_cast<int>(e / (static_cast<int64_t>(W) * H * C));
    dst[e] = base[e] + src[((static_cast<int64_t>(n) * H + y) * W + x) * C + c];
  }
}

// g[n, c] = mean over pixels of e[n, ., ., c] in two fixed-order stages:
// block (n, b) sums the pixels of slice b for every channel (consecutive
// threads read consecutive channels), then one block per image adds the
// slices and applies the head loglam[n] = w . g[n] + b.
constexpr int POOL_SLICES = 32;
__global__ void k_pool_part(const float* __restrict__ e, float* __restrict__ part, int HW, int C) {
  const int n = blockIdx.x, b = blockIdx.y;
  const int p0 = static_cast<int>((static_cast<int64_t>(HW) * b) / POOL_SLICES);
  const int p1 = static_cast<int>((static_cast<int64_t>(HW) * (b + 1)) / POOL_SLICES);
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float v = 0.f;
#pragma unroll 16
    for (int p = p0; p < p1; ++p) v += e[(static_cast<int64_t>(n) * HW + p) * C + c];
    part[(static_cast<int64_t>(n) * POOL_SLICES + b) * C + c] = v;
  }
}

__global__ void k_pool_head(const float* __restrict__ part, const float* __restrict__ w, const float* __restrict__ b,
                            float* __restrict__ g, float* __restrict__ loglam, int HW, int C) {
  const int n = blockIdx.x;
  __shared__ float red[256];
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float v = 0.f;
    for (int s2 = 0; s2 < POOL_SLICES; ++s2) v += part[(static_cast<int64_t>(n) * POOL_SLICES + s2) * C + c];
    g[static_cast<int64_t>(n) * C + c] = v / HW;
  }
  __syncthreads();
  float v = 0.f;
  for (int c = threadIdx.x; c < C; c += blockDim.x) v += w[c] * g[static_cast<int64_t>(n) * C + c];
  red[threadIdx.x] = v;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) loglam[n] = red[0] + b[0];
}

// Lambda head backward: dw[c] = sum_n g[n, c] dloglam[n], db = sum_n dloglam[n];
// de[n, p, c] += dloglam[n] w[c] / HW
__global__ void k_head_back(const float* __restrict__ g, const float* __restrict__ dll, const float* __restrict__ w,
                            float* __restrict__ dw, float* __restrict__ db, int N, int C) {
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float v = 0.f;
    for (int n = 0; n < N; ++n) v += g[static_cast<int64_t>(n) * C + c] * dll[n];
    dw[c] = v;
  }
  if (threadIdx.x == 0) {
    float v = 0.f;
    for (int n = 0; n < N; ++n) v += dll[n];
    db[0] = v;
  }
}

__global__ void k_head_back_spread(const float* __restrict__ dll, const float* __restrict__ w, float* __restrict__ de,
                                   int N, int HW, int C) {
  const int64_t total = static_cast<int64_t>(N) * HW * C;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < total;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(e % C);
    const int n = static_cast<int>(e / (static_cast<int64_t>(HW) * C));
    de[e] += dll[n] * w[c] / HW;
  }
}

// Adam on the FP32 master weights; the BF16 copy used by the GEMMs follows.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       __nv_bfloat16* __restrict__ pb, int64_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    if (pb != nullptr) pb[i] = __float2bfloat16(w);
  }
}

__global__ void k_to_bf16(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, int64_t n) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    y[i] = __float2bfloat16(x[i]);
}

#define NN_EW(kernel, n, ...)                                 \
  do {                                                        \
    kernel<<<grid_of(n), 256, 0, s>>>(__VA_ARGS__);           \
    return cudaGetLastError();                                \
  } while (0)

cudaError_t to_nhwc(const float* src, float* dst, int N, int H, int W, int C, cudaStream_t s) {
  NN_EW(k_to_nhwc, int64_t(N) * H * W, src, dst, int64_t(N) * H * W, H * W, C);
}
cudaError_t from_nhwc_add(const float* src, const float* base, float* dst, int N, int H, int W, int C,
                          cudaStream_t s) {
  NN_EW(k_from_nhwc_add, int64_t(N) * H * W * C, src, base, dst, N, H, W, C);
}
cudaError_t pool_head(const float* e, const float* w, const float* b, float* g, float* loglam, float* part, int N,
                      int HW, int C, cudaStream_t s) {
  k_pool_part<<<dim3(N, POOL_SLICES), 128, 0, s>>>(e, part, HW, C);
  k_pool_head<<<N, 256, 0, s>>>(part, w, b, g, loglam, HW, C);
  return cudaGetLastError();
}
cudaError_t head_back(const float* g, const float* dll, const float* w, float* dw, float* db, float* de, int N,
                      int HW, int C, cudaStream_t s) {
  k_head_back<<<1, 256, 0, s>>>(g, dll, w, dw, db, N, C);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  NN_EW(k_head_back_spread, int64_t(N) * HW * C, dll, w, de, N, HW, C);
}
cudaError_t adam(float* p, const float* g, float* m, float* v, __nv_bfloat16* pb, int64_t n, float lr, float b1,
                 float b2, float eps, float c1, float c2, cudaStream_t s) {
  NN_EW(k_adam, n, p, g, m, v, pb, n, lr, b1, b2, eps, c1, c2);
}
cudaError_t to_bf16(const float* x, __nv_bfloat16* y, int64_t n, cudaStream_t s) {
  NN_EW(k_to_bf16, n, x, y, n);
}

}  // namespace nn
}  // namespace rtg
