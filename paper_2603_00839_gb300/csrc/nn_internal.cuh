// Internal interface of the warm-start network kernels (k_nn.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rtg {
namespace nn {

// dz = dy * (mask > 0) (mask null: dz = dy) in BF16, db[c] = its FP32 column
// sums over the rows (db null: none; part: 256 * cols floats).
cudaError_t mask_grad(const float* dy, const float* mask, __nv_bfloat16* dzb, float* db, float* part, int64_t rows,
                      int cols, cudaStream_t s);
// Gradients of a 3x3 convolution on an H x W grid (padding 1).  Weights: dw
// (cout, 3, 3, C); x as for conv_fwd (up: stored at half resolution); part:
// conv_dw_splits(...) * cout * 9 C floats when that is over 1.
// Data: dx (N, H, W, C) = addend + gradient (addend may be null); up2: the 2 x 2
// block sums of the gradient instead, (N, H / 2, W / 2, C).
int conv_dw_splits(int N, int H, int W, int stride);
cudaError_t conv_dw(const float* x, const __nv_bfloat16* dzb, float* dw, int N, int H, int W, int C, int stride,
                    int cout, bool up, float* part, cudaStream_t s);
cudaError_t conv_dx(const __nv_bfloat16* dzb, const __nv_bfloat16* w, const float* addend, float* dx, int N, int H,
                    int W, int C, int stride, int cout, bool up2, cudaStream_t s);
cudaError_t to_nhwc(const float* src, float* dst, int N, int H, int W, int C, cudaStream_t s);
cudaError_t from_nhwc_add(const float* src, const float* base, float* dst, int N, int H, int W, int C,
                          cudaStream_t s);
// part: N * 32 * C floats of scratch
cudaError_t pool_head(const float* e, const float* w, const float* b, float* g, float* loglam, float* part, int N,
                      int HW, int C, cudaStream_t s);
// Implicit-GEMM 3x3 convolution forward with fused bias, ReLU and skip:
// r = act(conv(x) + b) (if r), out = r + skip (if out; skip may be null).
// H x W is the grid the convolution reads; up: x is stored at H/2 x W/2 and
// read through its nearest x2 up-sampling.  part (part_floats floats, may be
// null) lets small layers split K across CTAs.
// planar_in: x in the solver's planar layout (C = 3 only); planar_add: out, in
// that layout too, = planar_add + act(conv(x) + b) (channel counts of the tile kernels only).
cudaError_t conv_fwd(const float* x, const __nv_bfloat16* w, const float* bias, float* r, const float* skip,
                     float* out, int N, int H, int W, int C, int stride, int cout, bool relu, bool up,
                     float* part, int64_t part_floats, cudaStream_t s, bool planar_in = false,
                     const float* planar_add = nullptr);
// k_nn_fwd.cu: 0: the general kernel runs the layer; else the kind for conv_tile.
int conv_tile_kind(const float* x, const __nv_bfloat16* w, int H, int W, int C, int stride, int bn, bool up);
cudaError_t conv_tile(int kind, const float* x, const __nv_bfloat16* w, const float* bias, float* r, const float* skip,
                      float* out, const float* planar_add, bool planar_in, int N, int H, int W, int C, int stride,
                      int cout, bool relu, bool up, int bn, int kchunk, cudaStream_t s);
// floats of scratch that lets conv_fwd split K as far as it would
int64_t conv_fwd_scratch(int N, int H, int W, int C, int stride, int cout);
// scratch: loss_scratch_doubles(N)
cudaError_t loss(const float* X0, const float* Xs, const float* loglam, const float* logmu, float* dout,
                 float* dloglam, double* out, double* scratch, int N, int H, int W, int C, cudaStream_t s);
int64_t loss_scratch_doubles(int N);
cudaError_t head_back(const float* g, const float* dll, const float* w, float* dw, float* db, float* de, int N,
                      int HW, int C, cudaStream_t s);
cudaError_t adam(float* p, const float* g, float* m, float* v, __nv_bfloat16* pb, int64_t n, float lr, float b1,
                 float b2, float eps, float c1, float c2, cudaStream_t s);
cudaError_t to_bf16(const float* x, __nv_bfloat16* y, int64_t n, cudaStream_t s);

}  // namespace nn
}  // namespace rtg
