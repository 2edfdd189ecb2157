// Philox4x64-10, the generator of the Rademacher sketch signs (the random
// projections Theta_k of Section 3; k_sketch.cu expands them).
//
// Philox4x64-10 is written from its published definition (Salmon, Moraes,
// Dror, Shaw, "Parallel random numbers: as easy as 1, 2, 3", SC'11): the
// round maps (x0,x1,x2,x3) with key (k0,k1) to
// (hi(M1 x2) ^ x1 ^ k0, lo(M1 x2), hi(M0 x0) ^ x3 ^ k1, lo(M0 x0)); after
// each round the key is bumped by the Weyl constants.  Stream word w is
// lane w%4 of the block with counter (w/4 + 1, 0, 0, 0) and key
// (seed, problem_id); sign e is bit e%64 of word e/64, a set bit meaning -1.
#include "rtg_internal.cuh"
#include "philox.cuh"

namespace rtg {

__global__ void k_philox_words(uint64_t seed, uint64_t pid, int64_t n_words, uint64_t* out) {
  int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;   // one Philox block per thread
  if (4 * b >= n_words) return;
  uint64_t r[4];
  philox4x64_10(static_cast<uint64_t>(b) + 1, 0, 0, 0, seed, pid, r);
  for (int l = 0; l < 4; ++l)
    if (4 * b + l < n_words) out[4 * b + l] = r[l];
}

cudaError_t launch_philox_words(uint64_t seed, uint64_t pid, int64_t n_words, uint64_t* out,
                                cudaStream_t s) {
  if (n_words <= 0) return cudaSuccess;
  int64_t blocks = (n_words + 3) / 4;
  k_philox_words<<<(unsigned)((blocks + 127) / 128), 128, 0, s>>>(seed, pid, n_words, out);
  return cudaGetLastError();
}

}  // namespace rtg
