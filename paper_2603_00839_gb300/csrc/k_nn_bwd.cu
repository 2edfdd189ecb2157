// Backward kernels of the warm-start network (channels last, FP32
// activations, BF16 tensor-core products with FP32 accumulation): the
// gradient of a layer's output (ReLU mask, BF16 copy, bias gradient), the
// data and weight gradients of a 3x3 convolution, and the loss.
//
// Neither gradient materialises patches.  A patch matrix is nine times the
// activation (302 MB in BF16 for 16 images of 128 x 128 at 64 channels, 604 MB
// in FP32 for its gradient), so writing and reading it bound both products;
// here the nine taps read the same tile (data gradient) or gather through L2
// (weight gradient).
#include <cuda_bf16.h>

#include "nn_internal.cuh"
#include "nn_mma.cuh"
#include "rtg_internal.cuh"

namespace rtg {
namespace nn {

// ------------------------------------------------------------------ output gradient
// dzb = bf16(dz), dz = dy * (mask > 0) (mask null: dz = dy), and with `part`
// the column sums of dz: block t takes the rows t, t + 256, ..., all threads
// load (U rows of a column each, in flight together) and one thread per column
// adds them in row order; part[t][cols], then k_colsum_tree.  The order is kept
// whatever the parallelism: Adam divides by the gradients' size, so a change
// of rounding in an entry near zero would change its first step's sign.
// blockIdx.y: column chunk of `cw` <= 256 columns.
constexpr int MG_U = 8;
__global__ void __launch_bounds__(256)
k_mask_grad_db(const float* __restrict__ dy, const float* __restrict__ mask, __nv_bfloat16* __restrict__ dzb,
               float* __restrict__ part, int64_t rows, int cols, int cw) {
  __shared__ float sh[MG_U * 256];
  const int c0 = blockIdx.y * cw, width = min(cw, cols - c0);
  const int lpc = 256 / width;                       // rows loaded side by side
  const int kk = threadIdx.x / width, col = c0 + threadIdx.x % width;
  const int64_t nk = blockIdx.x < rows ? (rows - blockIdx.x + 255) / 256 : 0;   // this block's rows
  float sum = 0.f;
  for (int64_t k0 = 0; k0 < nk; k0 += MG_U * lpc) {
    float g[MG_U], m[MG_U];
#pragma unroll
    for (int u = 0; u < MG_U; ++u) {
      const int64_t k = k0 + u * lpc + kk;
      g[u] = 0.f;
      m[u] = 1.f;
      if (kk < lpc && k < nk) {
        const int64_t at = (blockIdx.x + 256 * k) * cols + col;
        g[u] = dy[at];
        if (mask != nullptr) m[u] = mask[at];
      }
    }
#pragma unroll
    for (int u = 0; u < MG_U; ++u) {
      const int64_t k = k0 + u * lpc + kk;
      if (!(m[u] > 0.f)) g[u] = 0.f;
      if (kk < lpc && k < nk) dzb[(blockIdx.x + 256 * k) * cols + col] = __float2bfloat16(g[u]);
      if (kk < lpc) sh[(u * lpc + kk) * width + threadIdx.x % width] = g[u];
    }
    if (part == nullptr) continue;
    __syncthreads();
    if (threadIdx.x < width) {
      const int64_t left = nk - k0;
      const int cnt = static_cast<int>(left < MG_U * lpc ? left : MG_U * lpc);
#pragma unroll 16
      for (int q = 0; q < cnt; ++q) sum += sh[q * width + threadIdx.x];
    }
    __syncthreads();
  }
  if (part != nullptr && threadIdx.x < width) part[static_cast<int64_t>(blockIdx.x) * cols + c0 + threadIdx.x] = sum;
}

// db[c] = tree over the 256 partial sums of column c.
__global__ void __launch_bounds__(256) k_colsum_tree(const float* __restrict__ part, float* __restrict__ db, int cols) {
  __shared__ float red[256];
  red[threadIdx.x] = part[static_cast<int64_t>(threadIdx.x) * cols + blockIdx.x];
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) db[blockIdx.x] = red[0];
}

// out[i] = sum over z < nz of part[z * len + i], in order (as above): up to 16
// loads in flight per thread.
__global__ void __launch_bounds__(128)
k_sum_slices(const float* __restrict__ part, float* __restrict__ out, int64_t len, int nz) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * 128 + threadIdx.x;
  if (i >= len) return;
  float v = 0.f;
  int z = 0;
  for (; z + 16 <= nz; z += 16) {
    float t[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) t[u] = part[static_cast<int64_t>(z + u) * len + i];
#pragma unroll
    for (int u = 0; u < 16; ++u) v += t[u];
  }
#pragma unroll 4
  for (; z < nz; ++z) v += part[static_cast<int64_t>(z) * len + i];
  out[i] = v;
}

static bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

cudaError_t mask_grad(const float* dy, const float* mask, __nv_bfloat16* dzb, float* db, float* part, int64_t rows,
                      int cols, cudaStream_t s) {
  float* pt = db != nullptr ? part : nullptr;
  const int cw = cols < 256 ? cols : 256;
  k_mask_grad_db<<<dim3(256, (cols + cw - 1) / cw), 256, 0, s>>>(dy, mask, dzb, pt, rows, cols, cw);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || pt == nullptr) return e;
  k_colsum_tree<<<cols, 256, 0, s>>>(part, db, cols);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ weight gradient
// dw[o, tap, c] = sum over output pixels p of dz[p, o] x[p + tap, c], as a GEMM
// with M = output channels, N = (tap, input channel) and K = pixels.  CTA tile
// BM x 64, K in stages of 128 pixels (64 for BM = 128), double buffered (with
// stages of 32 the loads' latency was most of a stage): dz rows arrive with
// 16-byte loads, the patch entries are gathered from x (FP32, rounded to BF16
// on the way) while the stage before is multiplied; both operands lie [k][.]
// in shared memory and are read with transposing ldmatrix.  gridDim.z splits
// the pixels; slice z writes part[z].  16 x 128 x 128, all eight layers: 2.93
// ms of GEMM (scalar loads) and 2.16 ms of im2col before.
constexpr int DW_BN = 64;
template <int BM>
__host__ __device__ constexpr int dw_bk() { return BM >= 128 ? 64 : 128; }
template <int BM>
constexpr size_t dw_smem() { return size_t(2) * dw_bk<BM>() * (BM + 8 + DW_BN + 8) * 2; }

template <int BM>
__global__ void __launch_bounds__(256)
k_conv_dw(const float* __restrict__ x, const __nv_bfloat16* __restrict__ dzb, float* __restrict__ part, int N, int H,
          int W, int C, int stride, int cout, int up, int kchunk, int vecx) {
  constexpr int BK = dw_bk<BM>(), PA = BM + 8, PB = DW_BN + 8;
  extern __shared__ __align__(16) unsigned char dw_sm[];
  __nv_bfloat16(*As)[BK][PA] = reinterpret_cast<__nv_bfloat16(*)[BK][PA]>(dw_sm);
  __nv_bfloat16(*Bs)[BK][PB] = reinterpret_cast<__nv_bfloat16(*)[BK][PB]>(dw_sm + size_t(2) * BK * PA * 2);
  constexpr int WM = BM >= 64 ? 4 : 2, WN = 8 / WM;          // warps along M and N
  constexpr int MT = BM / (16 * WM), NT = DW_BN / (8 * WN);  // m16 and n8 tiles per warp
  constexpr int ACH = BK * BM / 8;                        // 16-byte pieces of an A stage
  constexpr int AP = (ACH + 255) / 256, BP = BK / 32;        // pieces per thread
  const int Ho = H / stride, Wo = W / stride;
  const int M = N * Ho * Wo, K9 = 9 * C;
  const int n0 = blockIdx.x * DW_BN, m0 = blockIdx.y * BM;
  const int kbeg = blockIdx.z * kchunk, kend = min(M, kbeg + kchunk);
  const int Hs = up ? H / 2 : H, Ws = up ? W / 2 : W;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const int wm = (warp % WM) * 16 * MT, wn = (warp / WM) * 8 * NT;
  const bool veca = cout % 8 == 0;
  // this thread's pieces of a B stage: eight columns of every 32nd pixel
  const int brow = tid >> 3, j0 = n0 + (tid & 7) * 8;
  const int tap0 = j0 / C, ch0 = j0 - tap0 * C, ky0 = tap0 / 3, kx0 = tap0 - 3 * ky0;   // (vecx: all eight)
  int ent[8];   // otherwise: channel, ky and kx of each (negative: past K9)
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int jj = j0 + k, tap = jj / C;
    ent[k] = jj < K9 ? (jj - tap * C) << 4 | (tap / 3) << 2 | tap % 3 : -1;
  }
  uint4 ra[AP], rb[BP];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < AP; ++q) {
      const int e = tid + q * 256, row = e / (BM / 8), o = m0 + (e % (BM / 8)) * 8;
      ra[q] = make_uint4(0u, 0u, 0u, 0u);
      if (e >= ACH || k0 + row >= kend || o >= cout) continue;
      const __nv_bfloat16* src = dzb + static_cast<int64_t>(k0 + row) * cout + o;
      if (veca) {
        ra[q] = *reinterpret_cast<const uint4*>(src);
      } else {
        const unsigned short* u = reinterpret_cast<const unsigned short*>(src);
        uint32_t h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) h[k] = o + k < cout ? u[k] : 0u;
        ra[q] = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
      }
    }
    if (vecx) {   // eight channels of one tap
      float4 fa[BP], fb[BP];
#pragma unroll
      for (int q = 0; q < BP; ++q) {
        fa[q] = fb[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int p = k0 + brow + 32 * q;
        if (p >= kend || j0 >= K9) continue;
        const int j = p % Wo, t1 = p / Wo, i = t1 % Ho, n = t1 / Ho;
        const int yy = stride * i + ky0 - 1, xx = stride * j + kx0 - 1;
        if (yy < 0 || yy >= H || xx < 0 || xx >= W) continue;
        const float4* s4 = reinterpret_cast<const float4*>(
            x + ((static_cast<int64_t>(n) * Hs + (yy >> up)) * Ws + (xx >> up)) * C + ch0);
        fa[q] = s4[0];
        fb[q] = s4[1];
      }
#pragma unroll
      for (int q = 0; q < BP; ++q)
        rb[q] = make_uint4(pack_bf16(fa[q].x, fa[q].y), pack_bf16(fa[q].z, fa[q].w), pack_bf16(fb[q].x, fb[q].y),
                           pack_bf16(fb[q].z, fb[q].w));
      return;
    }
#pragma unroll
    for (int q = 0; q < BP; ++q) {
      const int p = k0 + brow + 32 * q;
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = 0.f;
      if (p < kend) {
        const int j = p % Wo, t1 = p / Wo, i = t1 % Ho, n = t1 / Ho;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int yy = stride * i + (ent[k] >> 2 & 3) - 1, xx = stride * j + (ent[k] & 3) - 1;
          if (ent[k] >= 0 && yy >= 0 && yy < H && xx >= 0 && xx < W)
            v[k] = x[((static_cast<int64_t>(n) * Hs + (yy >> up)) * Ws + (xx >> up)) * C + (ent[k] >> 4)];
        }
      }
      rb[q] = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < AP; ++q) {
      const int e = tid + q * 256;
      if (e < ACH) *reinterpret_cast<uint4*>(&As[buf][e / (BM / 8)][(e % (BM / 8)) * 8]) = ra[q];
    }
#pragma unroll
    for (int q = 0; q < BP; ++q) *reinterpret_cast<uint4*>(&Bs[buf][brow + 32 * q][(tid & 7) * 8]) = rb[q];
  };
  float acc[MT][NT][4];
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int b = 0; b < NT; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
  load(kbeg);
  store(0);
  __syncthreads();
  const int mi = lane >> 3, r8 = lane & 7;
  int buf = 0;
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
    const bool more = k0 + BK < kend;
    if (more) load(k0 + BK);
#pragma unroll 2
    for (int kk = 0; kk < BK; kk += 16) {
      uint32_t a[MT][4];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
        ldsm_x4_t(a[mt], smem_addr(&As[buf][kk + (mi >> 1) * 8 + r8][wm + mt * 16 + (mi & 1) * 8]));
#pragma unroll
      for (int nt = 0; nt < NT; nt += 2) {
        uint32_t b[4];
        ldsm_x4_t(b, smem_addr(&Bs[buf][kk + (mi & 1) * 8 + r8][wn + nt * 8 + (mi >> 1) * 8]));
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          mma_k16(acc[mt][nt], a[mt], b[0], b[1]);
          mma_k16(acc[mt][nt + 1], a[mt], b[2], b[3]);
        }
      }
    }
    if (more) {
      store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
  float* out = part + static_cast<int64_t>(blockIdx.z) * cout * K9;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int o = m0 + wm + mt * 16 + gid + h * 8, j = n0 + wn + nt * 8 + tig * 2;
        if (o >= cout) continue;
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (j + q < K9) out[static_cast<int64_t>(o) * K9 + j + q] = acc[mt][nt][2 * h + q];
      }
}

// Slices of the pixels: about 2048 each, at most 64.
int conv_dw_splits(int N, int H, int W, int stride) {
  const int64_t sp = int64_t(N) * (H / stride) * (W / stride) / 2048;
  return static_cast<int>(sp < 1 ? 1 : (sp > 64 ? 64 : sp));
}

cudaError_t conv_dw(const float* x, const __nv_bfloat16* dzb, float* dw, int N, int H, int W, int C, int stride,
                    int cout, bool up, float* part, cudaStream_t s) {
  const int64_t M = int64_t(N) * (H / stride) * (W / stride), len = int64_t(cout) * 9 * C;
  int splits = conv_dw_splits(N, H, W, stride);
  int64_t kchunk = (M + splits - 1) / splits;
  kchunk = (kchunk + 31) / 32 * 32;
  splits = static_cast<int>((M + kchunk - 1) / kchunk);
  float* dst = splits > 1 ? part : dw;
  const int vecx = C % 8 == 0 && aligned16(x) ? 1 : 0, u = up ? 1 : 0;
  // fewer output channels per CTA where the tiles and slices leave SMs idle
  const int64_t ntile = (9 * C + DW_BN - 1) / DW_BN;
  int bm = cout <= 32 ? 32 : (cout <= 64 ? 64 : 128);
  while (bm > 32 && ntile * ((cout + bm - 1) / bm) * splits < 152) bm /= 2;
  const dim3 grid(static_cast<unsigned>(ntile), (cout + bm - 1) / bm, splits);
  const int kc = static_cast<int>(kchunk);
  cudaError_t e = cudaSuccess;
#define RTG_DW_CASE(B_)                                                                                       \
  if (bm == B_) {                                                                                             \
    e = set_smem(k_conv_dw<B_>, dw_smem<B_>());                                                               \
    if (e != cudaSuccess) return e;                                                                           \
    k_conv_dw<B_><<<grid, 256, dw_smem<B_>(), s>>>(x, dzb, dst, N, H, W, C, stride, cout, u, kc, vecx);       \
  }
  RTG_DW_CASE(32) RTG_DW_CASE(64) RTG_DW_CASE(128)
#undef RTG_DW_CASE
  e = cudaGetLastError();
  if (e != cudaSuccess || splits == 1) return e;
  k_sum_slices<<<static_cast<unsigned>((len + 127) / 128), 128, 0, s>>>(part, dw, len, splits);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ data gradient
// dx[y, x, c] = sum over taps of sum over o of dz[(y + 1 - ky) / s, (x + 1 - kx) / s, o] w[o, ky, kx, c].
// CTA: 8 x 16 pixels (of one parity class when the stride is 2: the class
// fixes which taps meet it) x BN input channels; the tile of dz with its halo
// lies in shared memory in BF16, the nine taps read it shifted, and each tap's
// weights (K = output channels, up to 128 at a time) arrive with cp.async
// while the tap before is multiplied.  Warp w owns a 2 x 8 patch of pixels
// and all BN channels.  Each tap has its own accumulator, added to the sum in
// tap order.  Epilogue: out = v, out = addend + v, or (up2) the sum of each
// 2 x 2 block of pixels, the gradient of a nearest x2 up-sampling.  16 x 128 x
// 128, seven layers: 0.9 ms of GEMM and 1.12 ms of col2im before.
constexpr int DX_TA = 8, DX_TB = 16, DX_PIX = (DX_TA + 2) * (DX_TB + 2);

template <int BN>
__global__ void __launch_bounds__(256)
k_conv_dx(const __nv_bfloat16* __restrict__ dzb, const __nv_bfloat16* __restrict__ wt, const float* __restrict__ addend,
          float* __restrict__ out, int H, int W, int C, int stride, int cout, int up2, int kp, int tilesb, int vecw) {
  extern __shared__ __align__(16) unsigned char dx_smem[];
  const int PH = kp + 8;                                  // pitch of a halo pixel (an odd number of 16-byte pieces)
  constexpr int PB = BN + 8;
  __nv_bfloat16* halo = reinterpret_cast<__nv_bfloat16*>(dx_smem);   // [DX_PIX][PH]
  __nv_bfloat16* Bs = halo + DX_PIX * PH;                            // [2][kp][PB]
  const int Ho = H / stride, Wo = W / stride;
  const int nclass = stride * stride;
  const int n = blockIdx.z / nclass, cls = blockIdx.z % nclass, py = cls / stride, px = cls % stride;
  const int a0 = (blockIdx.x / tilesb) * DX_TA, b0 = (blockIdx.x % tilesb) * DX_TB;
  const int n0 = blockIdx.y * BN;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const int nchunk = (cout + kp - 1) / kp;
  const bool vecz = cout % 8 == 0;
  const int kpc = kp / 8;                                 // 16-byte pieces per pixel
  auto load_halo = [&](int chunk) {
    for (int e = tid; e < DX_PIX * kpc; e += 256) {
      const int pix = e / kpc, o = chunk * kp + (e % kpc) * 8;
      const int i = a0 - 1 + pix / (DX_TB + 2), j = b0 - 1 + pix % (DX_TB + 2);
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (i >= 0 && i < Ho && j >= 0 && j < Wo && o < cout) {
        const __nv_bfloat16* src = dzb + ((static_cast<int64_t>(n) * Ho + i) * Wo + j) * cout + o;
        if (vecz) {
          v = *reinterpret_cast<const uint4*>(src);
        } else {
          const unsigned short* u = reinterpret_cast<const unsigned short*>(src);
          uint32_t h[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) h[k] = o + k < cout ? u[k] : 0u;
          v = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
        }
      }
      *reinterpret_cast<uint4*>(halo + pix * PH + (e % kpc) * 8) = v;
    }
  };
  auto load_w = [&](int tap, int chunk, int buf) {   // one cp.async group
    __nv_bfloat16* dst = Bs + buf * kp * PB;
    for (int e = tid; e < kp * (BN / 8); e += 256) {
      const int k = e / (BN / 8), c = n0 + (e % (BN / 8)) * 8, o = chunk * kp + k;
      const __nv_bfloat16* src = wt + (static_cast<int64_t>(o) * 9 + tap) * C + c;
      __nv_bfloat16* d = dst + k * PB + (e % (BN / 8)) * 8;
      if (vecw) {   // C a multiple of 8: a piece lies inside the row or past it
        const bool v = o < cout && c < C;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(d)), "l"(v ? src : wt),
                     "r"(v ? 16 : 0)
                     : "memory");
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) d[q] = (o < cout && c + q < C) ? src[q] : __float2bfloat16(0.f);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  // the taps that meet this parity class, in order
  auto next_tap = [&](int t) {
    for (; t < 9; ++t)
      if (stride == 1 || ((py + 1 - t / 3) % 2 == 0 && (px + 1 - t % 3) % 2 == 0)) break;
    return t;
  };
  float v[BN / 8][4];
#pragma unroll
  for (int a = 0; a < BN / 8; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) v[a][c] = 0.f;
  if (nchunk == 1) load_halo(0);
  const int mi = lane >> 3, r8 = lane & 7;
  const int aw = (warp >> 1) * 2, bw = (warp & 1) * 8;
  int tap = next_tap(0), buf = 0;
  load_w(tap, 0, 0);
  while (tap < 9) {
    const int after = next_tap(tap + 1);
    const int da = stride == 1 ? 1 - tap / 3 : (py + 1 - tap / 3) / 2, db = stride == 1 ? 1 - tap % 3 : (px + 1 - tap % 3) / 2;
    float acc[BN / 8][4];
#pragma unroll
    for (int a = 0; a < BN / 8; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][c] = 0.f;
    for (int ch = 0; ch < nchunk; ++ch) {
      if (nchunk > 1) {
        __syncthreads();   // the chunk before has been multiplied
        load_halo(ch);
      }
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      __syncthreads();     // weights and halo are there, and the other weight buffer is free
      if (ch + 1 < nchunk) load_w(tap, ch + 1, buf ^ 1);
      else if (after < 9) load_w(after, 0, buf ^ 1);
      const __nv_bfloat16* B = Bs + buf * kp * PB;
      // lane's row of the A tiles: pixel (mi & 1) * 8 + r8 of the warp's patch, shifted by the tap
      const __nv_bfloat16* arow =
          halo + ((aw + (mi & 1) + da + 1) * (DX_TB + 2) + bw + r8 + db + 1) * PH + (mi >> 1) * 8;
      for (int kk = 0; kk < kp; kk += 16) {
        uint32_t a[4];
        ldsm_x4(a, smem_addr(arow + kk));
#pragma unroll
        for (int nt = 0; nt < BN / 8; nt += 2) {
          uint32_t b[4];
          ldsm_x4_t(b, smem_addr(B + (kk + (mi & 1) * 8 + r8) * PB + nt * 8 + (mi >> 1) * 8));
          mma_k16(acc[nt], a, b[0], b[1]);
          mma_k16(acc[nt + 1], a, b[2], b[3]);
        }
      }
      buf ^= 1;
    }
#pragma unroll
    for (int a = 0; a < BN / 8; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[a][c] += acc[a][c];
    tap = after;
  }
  const int b = b0 + bw + gid;
#pragma unroll
  for (int nt = 0; nt < BN / 8; ++nt) {
    const int c = n0 + nt * 8 + tig * 2;
    if (up2) {
      float top[2], bot[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        top[q] = v[nt][q] + __shfl_xor_sync(0xffffffffu, v[nt][q], 4);          // pixels gid and gid ^ 1
        bot[q] = v[nt][2 + q] + __shfl_xor_sync(0xffffffffu, v[nt][2 + q], 4);
      }
      if ((gid & 1) == 0 && a0 + aw < H && b < W) {
        const int64_t o = ((static_cast<int64_t>(n) * (H / 2) + (a0 + aw) / 2) * (W / 2) + b / 2) * C + c;
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (c + q < C) out[o + q] = top[q] + bot[q];
      }
      continue;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int a = a0 + aw + h;
      if (a >= Ho || b >= Wo) continue;
      const int64_t o = ((static_cast<int64_t>(n) * H + stride * a + py) * W + stride * b + px) * C + c;
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (c + q < C) out[o + q] = addend != nullptr ? addend[o + q] + v[nt][2 * h + q] : v[nt][2 * h + q];
    }
  }
}

cudaError_t conv_dx(const __nv_bfloat16* dzb, const __nv_bfloat16* w, const float* addend, float* dx, int N, int H,
                    int W, int C, int stride, int cout, bool up2, cudaStream_t s) {
  int bn = C <= 32 ? 32 : (C <= 64 ? 64 : 128);
  int kp = (cout + 15) / 16 * 16;
  if (kp > 128) kp = 128;
  const int Ho = H / stride, Wo = W / stride;
  const int ta = (Ho + DX_TA - 1) / DX_TA, tb = (Wo + DX_TB - 1) / DX_TB;
  // fewer input channels per CTA where all of them leave most SMs idle (4 x 4 pixels,
  // 1024 channels: 8 CTAs of 128); the result does not depend on it
  while (bn > 32 && int64_t(ta) * tb * stride * stride * N * ((C + bn - 1) / bn) < 76) bn /= 2;
  const size_t smem = (size_t(DX_PIX) * (kp + 8) + size_t(2) * kp * (bn + 8)) * 2;
  const int vecw = C % 8 == 0 && aligned16(w) ? 1 : 0, u = up2 ? 1 : 0;
  const int per = 65535 / (stride * stride);   // images of one launch (the grid's z limit)
  for (int n0 = 0; n0 < N; n0 += per) {
    const int nn = N - n0 < per ? N - n0 : per;
    const int64_t xo = int64_t(n0) * H * W * C / (up2 ? 4 : 1);
    const __nv_bfloat16* dz = dzb + int64_t(n0) * Ho * Wo * cout;
    const float* ad = addend != nullptr ? addend + xo : nullptr;
    const dim3 grid(ta * tb, (C + bn - 1) / bn, nn * stride * stride);
    cudaError_t e = cudaSuccess;
#define RTG_DX_CASE(B_)                                                                                          \
  if (bn == B_) {                                                                                                \
    e = set_smem(k_conv_dx<B_>, smem);                                                                           \
    if (e != cudaSuccess) return e;                                                                              \
    k_conv_dx<B_><<<grid, 256, smem, s>>>(dz, w, ad, dx + xo, H, W, C, stride, cout, u, kp, tb, vecw);           \
  }
    RTG_DX_CASE(32) RTG_DX_CASE(64) RTG_DX_CASE(128)
#undef RTG_DX_CASE
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ------------------------------------------------------------------ loss
// Loss of the batch and the output gradients: per image ||X0 - X*||^2 /
// ||X*||^2 + (loglam - logmu)^2, averaged; dout = 2 (X0 - X*) / (||X*||^2 N)
// (channels last), dloglam = 2 (loglam - logmu) / N.  X0 and X* in solver
// layout.  Three launches: sums per image and slice (FP64), the scalars, the
// gradient; one block did it all in 3.08 ms for 16 x 128 x 128.
constexpr int LOSS_SLICES = 32;

__global__ void __launch_bounds__(256)
k_loss_part(const float* __restrict__ X0, const float* __restrict__ Xs, double* __restrict__ part, int64_t per) {
  __shared__ double red[2][8];
  const int n = blockIdx.y, sl = blockIdx.x;
  const int64_t e0 = per * sl / LOSS_SLICES, e1 = per * (sl + 1) / LOSS_SLICES;
  double a = 0.0, b = 0.0;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const double xs = Xs[n * per + e], d = static_cast<double>(X0[n * per + e]) - xs;
    a = fma(d, d, a);
    b = fma(xs, xs, b);
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = a;
    red[1][threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int q = 0; q < 8; ++q) s += red[threadIdx.x][q];
    part[(static_cast<int64_t>(n) * LOSS_SLICES + sl) * 2 + threadIdx.x] = s;
  }
}

// One block: the images' sums, the loss and the scale 2 / (||X*||^2 N) of each image's gradient.
__global__ void __launch_bounds__(256)
k_loss_scalars(const double* __restrict__ part, const float* __restrict__ loglam, const float* __restrict__ logmu,
               float* __restrict__ dloglam, double* __restrict__ scale, double* __restrict__ loss, int N) {
  __shared__ double term[256];
  double t = 0.0;
  for (int n = threadIdx.x; n < N; n += blockDim.x) {
    double a = 0.0, b = 0.0;
    for (int q = 0; q < LOSS_SLICES; ++q) {
      a += part[(static_cast<int64_t>(n) * LOSS_SLICES + q) * 2];
      b += part[(static_cast<int64_t>(n) * LOSS_SLICES + q) * 2 + 1];
    }
    const double dl = static_cast<double>(loglam[n]) - logmu[n];
    t += a / b + dl * dl;
    scale[n] = 2.0 / (b * N);
    dloglam[n] = static_cast<float>(2.0 * dl / N);
  }
  term[threadIdx.x] = t;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) term[threadIdx.x] += term[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = term[0] / N;
}

__global__ void __launch_bounds__(256)
k_loss_grad(const float* __restrict__ X0, const float* __restrict__ Xs, const double* __restrict__ scale,
            float* __restrict__ dout, int H, int W, int C) {
  const int n = blockIdx.y, HW = H * W;
  const int64_t per = static_cast<int64_t>(HW) * C;
  const double f = scale[n];
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < HW; p += gridDim.x * blockDim.x)
    for (int c = 0; c < C; ++c) {
      const int64_t e = n * per + static_cast<int64_t>(c) * HW + p;
      dout[n * per + static_cast<int64_t>(p) * C + c] =
          static_cast<float>(f * (static_cast<double>(X0[e]) - Xs[e]));
    }
}

int64_t loss_scratch_doubles(int N) { return int64_t(N) * (2 * LOSS_SLICES + 1); }

cudaError_t loss(const float* X0, const float* Xs, const float* loglam, const float* logmu, float* dout,
                 float* dloglam, double* out, double* scratch, int N, int H, int W, int C, cudaStream_t s) {
  double* scale = scratch + int64_t(N) * 2 * LOSS_SLICES;
  k_loss_part<<<dim3(LOSS_SLICES, N), 256, 0, s>>>(X0, Xs, scratch, int64_t(H) * W * C);
  k_loss_scalars<<<1, 256, 0, s>>>(scratch, loglam, logmu, dloglam, scale, out, N);
  int64_t b = (int64_t(H) * W + 255) / 256;
  if (b > 1024) b = 1024;
  k_loss_grad<<<dim3(static_cast<unsigned>(b), N), 256, 0, s>>>(X0, Xs, scale, dout, H, W, C);
  return cudaGetLastError();
}

}  // namespace nn
}  // namespace rtg
