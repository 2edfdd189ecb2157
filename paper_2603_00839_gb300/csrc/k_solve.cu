// Reduced solves and solution assembly of RTG-GMRES.
//
// The Givens QR of the step kernels already holds Hbar_k = Omega^T [R; 0]
// and Omega^T beta e1 = g, so
//   ||beta e1 - Hbar y||^2 + mu ||y||^2 = ||g_{0:k} - R y||^2 + g_k^2 + mu ||y||^2.
// Projected Tikhonov (Eq. 12S) is solved in the stacked form of Eq. 13,
// min || [R; sqrt(mu) I] y - [g_{0:k}; 0] ||, by Householder reflections
// that use the structure (column j touches row j of R and rows 0..j of the
// sqrt(mu) I block), then back substitution.  GCV (Section 3, "Parameter
// selection via GCV"): the numerator is ||Hbar y_mu - beta e1||^2; the
// trace is tr(I - Hbar (Hbar^T Hbar + mu I)^{-1} Hbar^T) = 1 + mu ||R_mu^{-1}||_F^2
// (k+1 minus k plus mu tr((R_mu^T R_mu)^{-1})).  One CTA per candidate mu;
// the last CTA to finish picks the smallest GCV (ties: the larger mu).
// Everything here is FP64.
#include "gs_common.cuh"
#include "queue.cuh"

namespace rtg {

// Four warps per candidate mu.  An FP64 warp instruction occupies its SM
// sub-partition's FP64 unit for about 64 cycles on this GPU, so the cost of
// this kernel is the number of FP64 warp instructions each sub-partition
// issues one after another: the columns of a reflection are dealt over the
// warps and its rows over the lanes, every warp takes the pivot column's norm
// itself (no exchange before the update), and the square root and the
// quotients are Newton-Raphson refinements of FP32 seeds (tk_reflector; sqrt()
// and two divisions take over 30 FP64 instructions).  Back substitution
// and residual (warp 0) run beside the trace's inverse (warps 1 to 3).
constexpr int TK_THREADS = 128;
constexpr int TK_WARPS = TK_THREADS / 32;

// 2^-e x by the exponent field (x and the result normal).
__device__ __forceinline__ double tk_scale(double x, int e) {
  return __hiloint2double(__double2hiint(x) - (e << 20), __double2loint(x));
}

// Double value of a normal positive float, and the float of a double in [1, 4)
// with its low bits cut, in the integer pipes (a conversion between the two
// types takes about as long as a dozen FP64 instructions).
__device__ __forceinline__ double tk_widen(float f) {
  const uint32_t b = __float_as_uint(f);
  return __hiloint2double(static_cast<int>((b >> 3) + ((1023u - 127u) << 20)), static_cast<int>(b << 29));
}
__device__ __forceinline__ float tk_narrow(double x) {
  const uint32_t h = static_cast<uint32_t>(__double2hiint(x));
  return __uint_as_float(((h - ((1023u - 127u) << 20)) << 3) | (static_cast<uint32_t>(__double2loint(x)) >> 29));
}

// Householder reflector of a column (alpha; a part of squared norm sigma > 0):
// nrm = sqrt(q), q = alpha^2 + sigma; v0 = alpha + sgn nrm; tau = 2 / (v0^2 +
// sigma); the new pivot -sgn nrm as its reciprocal pinv.  From an FP32 seed of
// y = 1 / sqrt(q) (relative error below 2^-21) one step of third order, y (1 +
// e / 2 + 3 e^2 / 8) with e = 1 - q y^2, leaves 5 e^3 / 16 < 2^-61; nrm = q y.
// tau starts at y^2 / h, h = 1 + |alpha| y, with an FP32 reciprocal of h, and is
// corrected to third order by 1 - (v0^2 + sigma) tau / 2: what counts for the
// error is that tau fits the rounded v0.  Mean error of the solution, over random
// triangles of 1 to 100 columns: 0.77 to 0.87 of that with sqrt() and divisions
// (with tau from y and h alone 2.6 times for one column, 1.3 for twelve).
// Beyond 2^+-900, and for NaN, the plain operations.
__device__ __forceinline__ void tk_reflector(double alpha, double sigma, double& v0, double& tau, double& pinv) {
  const double q = fma(alpha, alpha, sigma);
  const int hi = __double2hiint(q);
  double nrm;
  if (hi < ((1023 - 900) << 20) || hi >= ((1023 + 900) << 20)) {
    nrm = sqrt(q);
    v0 = fabs(alpha) + nrm;
    tau = 2.0 / fma(v0, v0, sigma);
    pinv = 1.0 / nrm;
  } else {
    const int e = ((hi >> 20) - 1023) & ~1;
    const double a = tk_scale(q, e);   // [1, 4)
    const double y0 = tk_widen(rsqrtf(tk_narrow(a)));
    const double r = fma(-(a * y0), y0, 1.0);
    const double y = tk_scale(fma(y0, r * fma(0.375, r, 0.5), y0), e / 2);
    const double t = (y * y) * tk_widen(__frcp_rn(tk_narrow(fma(fabs(alpha), y, 1.0))));   // (h in [1, 2])
    nrm = q * y;
    pinv = y;
    v0 = fabs(alpha) + nrm;
    const double f = fma(-fma(v0, v0, sigma), tk_scale(t, 1), 1.0);
    tau = fma(t, fma(f, f, f), t);
  }
  if (alpha >= 0.0) {
    pinv = -pinv;
  } else {
    v0 = -v0;
  }
}

// Back substitution with the unit upper-triangular U D^{-1} (U's columns
// already multiplied by rinv; leading dimension ldu) by one warp: b becomes
// D y.  rinv is 0 for a zero pivot: y_i = 0, the smallest-norm least-squares
// choice on that direction.
__device__ void back_subst(const double* U, int ldu, double* b, int k) {
  const int lane = threadIdx.x & 31;
  if (k <= 32) {   // b in the lanes' registers
    double v = lane < k ? b[lane] : 0.0;
    for (int i = k - 1; i > 0; --i) {
      const double bi = __shfl_sync(0xffffffffu, v, i);
      if (lane < i) v = fma(-U[lane + static_cast<int64_t>(ldu) * i], bi, v);
    }
    if (lane < k) b[lane] = v;
    __syncwarp();
    return;
  }
  for (int i = k - 1; i > 0; --i) {
    __syncwarp();
    const double bi = b[i];
    for (int t = lane; t < i; t += 32) b[t] = fma(-U[t + static_cast<int64_t>(ldu) * i], bi, b[t]);
  }
  __syncwarp();
}

// mode 0: least squares (mu = 0); 1: fixed mu = lambda; 2: GCV over the grid.
// Working set per CTA (tk_scratch_doubles(m) doubles): T and B, both
// (m+1) x (m+1) with row stride m+1, then y and rinv.  T holds R (becoming
// R_mu) with g_{0:k} as column k; B holds the sqrt(mu) I block with its
// right-hand side (0) as column k, and after the factorisation the
// inverse R_mu^{-1} is built in it.  With in_smem the working set is the
// CTA's dynamic shared memory, else the per-CTA global scratch.
__global__ void __launch_bounds__(TK_THREADS)
k_tikhonov(Work w0, const SolveDesc* desc0, int mode, double* scratch0, int in_smem, const int* gate) {
  const int64_t bo = bidx(w0.b).off;
  const Work w = w0.at(bo);
  const SolveDesc* desc = bsh(desc0, bo);
  double* scratch = bsh(scratch0, bo);
  Ctl* ctl = w.ctl;
  gate = bsh(gate, bo);
  if (gate != nullptr && *gate) return;
  // a GCV plan whose descriptor carries lambda > 0 (the learned warm start's
  // prediction) solves with that fixed mu on its first block
  if (mode == 2 && desc->lambda > 0.0) {
    if (blockIdx.x != 0) return;
    mode = 1;
  }
  const int k = ctl->j;
  const int m = w.m, ld = m + 1;
  __shared__ double wsum[TK_WARPS];
  __shared__ int am_last;
  extern __shared__ __align__(16) double tk_smem[];
  if (k == 0) {
    if (threadIdx.x == 0 && blockIdx.x == 0) ctl->mu = (mode == 1) ? desc->lambda : 0.0;
    return;
  }
  const double mu = (mode == 0) ? 0.0 : (mode == 1 ? desc->lambda : desc->mu_grid[blockIdx.x]);
  const int lm = m + 1;
  double* T = in_smem ? tk_smem : scratch + static_cast<int64_t>(blockIdx.x) * tk_scratch_doubles(m);
  double* Bm = T + lm * lm;
  double* y = Bm + lm * lm;
  double* rinv = y + lm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const double smu = sqrt(mu);
  for (int idx = tid; idx < k * (k + 1); idx += TK_THREADS) {
    const int col = idx / k, i = idx - col * k;
    T[i + lm * col] = (col == k) ? w.g[i] : (i <= col ? w.R[i + static_cast<int64_t>(ld) * col] : 0.0);
    Bm[i + lm * col] = (i == col) ? smu : 0.0;
  }
  __syncthreads();
  if (mode != 0) {
    // Householder on column j: rows {j of T} U {0..j of B}; row j of B is
    // still sqrt(mu), rows 0..j-1 were filled by the earlier reflections.
    // Slot 0 of every warp is the pivot column, slot c > 0 its column
    // j + 1 + warp + 4 (c - 1) (column k: the right-hand side); a warp covers
    // cw slots at a time and 32 / cw stripes of rows.
    for (int j = 0; j < k; ++j) {
      const int slots = 1 + ((k - j + TK_WARPS - 1) >> 2);
      const int cw = slots >= 32 ? 32 : 1 << (32 - __clz(slots - 1));
      const int nst = 32 / cw, st = lane / cw, cs = lane % cw;
      const double* Bj = Bm + lm * j;
      const double alpha = T[j + lm * j];   // row j of T is this step's alone
      double v0 = 0.0, tau = 0.0;
      bool refl = false;
      for (int c0 = 0; c0 < slots; c0 += cw) {
        const int c = c0 + cs;
        const int own = j + 1 + warp + TK_WARPS * (c - 1);
        const bool in = c > 0 && c < slots && own <= k;
        const int col = in ? own : j;
        double* Bc = Bm + lm * col;
        const double tj = T[j + lm * col];
        double a = 0.0;
        for (int i = st; i <= j; i += nst) a = fma(Bj[i], Bc[i], a);
        for (int o = cw; o < 32; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (c0 == 0) {
          const double sigma = __shfl_sync(0xffffffffu, a, 0);
          double pinv = 0.0;
          refl = sigma != 0.0;
          if (refl) {
            tk_reflector(alpha, sigma, v0, tau, pinv);
          } else if (alpha != 0.0) {
            pinv = 1.0 / alpha;
          }
          if (tid == 0) rinv[j] = pinv;
        }
        __syncwarp();   // every lane has read row j of its column
        if (refl && in) {
          const double wv = tau * fma(v0, tj, a);
          if (st == 0) T[j + lm * col] = fma(-wv, v0, tj);
          for (int i = st; i <= j; i += nst) Bc[i] = fma(-wv, Bj[i], Bc[i]);
        }
      }
      __syncthreads();
    }
  } else {
    for (int i = tid; i < k; i += TK_THREADS) {
      const double piv = T[i + lm * i];
      rinv[i] = (piv != 0.0) ? 1.0 / piv : 0.0;
    }
    __syncthreads();
  }
  // U D^{-1} in place of U above the diagonal, and I in B
  for (int idx = tid; idx < k * k; idx += TK_THREADS) {
    const int col = idx / k, i = idx - col * k;
    if (mode == 2) Bm[i + lm * col] = (i == col) ? 1.0 : 0.0;
    if (i < col) T[i + lm * col] *= rinv[col];
  }
  __syncthreads();
  if (warp == 0) {
    double* b = T + lm * k;
    back_subst(T, lm, b, k);
    for (int i = lane; i < k; i += 32) y[i] = b[i] * rinv[i];
    __syncwarp();
    if (mode == 2) {   // residual ||g_{0:k} - R y||^2 + g_k^2 with the unregularised R
      double part = 0.0;
      for (int i = lane; i < k; i += 32) {
        double r0 = w.g[i], r1 = 0.0;
        int jj = i;
        for (; jj + 1 < k; jj += 2) {
          r0 -= w.R[i + static_cast<int64_t>(ld) * jj] * y[jj];
          r1 -= w.R[i + static_cast<int64_t>(ld) * (jj + 1)] * y[jj + 1];
        }
        if (jj < k) r0 -= w.R[i + static_cast<int64_t>(ld) * jj] * y[jj];
        const double r = r0 + r1;
        part = fma(r, r, part);
      }
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (lane == 0) wsum[0] = fma(w.g[k], w.g[k], part);
    }
  } else if (mode == 2) {
    // ||Z||_F^2 with Z = R_mu^{-1}: right-looking substitution on W = I
    // (stored in B), rows of Z from the last up; row l of Z is
    // W[l, l:] / R_mu[l,l].
    constexpr int NT = TK_THREADS - 32;
    const int id = tid - 32;
    for (int l = k - 1; l > 0; --l) {
      const int nc = k - l;
      for (int idx = id; idx < l * nc; idx += NT) {
        const int i = idx / nc, col = l + (idx - i * nc);
        Bm[i + lm * col] = fma(-T[i + lm * l], Bm[l + lm * col], Bm[i + lm * col]);
      }
      asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
    }
    double inv2 = 0.0;
    for (int idx = id; idx < k * k; idx += NT) {
      const int col = idx / k, i = idx - col * k;
      if (i <= col) {
        const double z = Bm[i + lm * col] * rinv[i];
        inv2 = fma(z, z, inv2);
      }
    }
    for (int o = 16; o > 0; o >>= 1) inv2 += __shfl_xor_sync(0xffffffffu, inv2, o);
    if (lane == 0) wsum[warp] = inv2;
  }
  __syncthreads();
  if (mode == 2) {
    if (tid == 0) {
      const double trace = fma(mu, wsum[1] + wsum[2] + wsum[3], 1.0);
      w.gcv[blockIdx.x] = wsum[0] / (trace * trace);
    }
    for (int i = tid; i < k; i += TK_THREADS) w.ysel[static_cast<int64_t>(blockIdx.x) * m + i] = y[i];
    __syncthreads();
    if (tid == 0) am_last = (ticket_acq_rel(w.counter, gridDim.x - 1) == gridDim.x - 1);
    __syncthreads();
    if (!am_last) return;
    __shared__ int best;
    // the smallest value, of equal ones the larger mu, of equal ones the first;
    // the values are not negative, so their bits order them, and a NaN
    // (anywhere but in front) never wins
    if (warp == 0) {
      unsigned long long bv = ~0ull, bm = 0ull;
      int bi = lane;
      if (lane < static_cast<int>(gridDim.x)) {
        bv = static_cast<unsigned long long>(__double_as_longlong(__ldcg(w.gcv + lane)));
        bm = static_cast<unsigned long long>(__double_as_longlong(desc->mu_grid[lane]));
        bm = (bm >> 63) ? ~bm : (bm | (1ull << 63));
        if (lane == 0 && (bv << 1) > (0x7ffull << 53)) {
          bv = 0ull;
          bm = ~0ull;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ov = __shfl_xor_sync(0xffffffffu, bv, o), om = __shfl_xor_sync(0xffffffffu, bm, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov < bv || (ov == bv && (om > bm || (om == bm && oi < bi)))) {
          bv = ov;
          bm = om;
          bi = oi;
        }
      }
      if (lane == 0) {
        best = bi;
        ctl->mu = desc->mu_grid[bi];
        ctl->gcv_best = __ldcg(w.gcv + bi);
      }
    }
    __syncthreads();
    for (int i = tid; i < k; i += TK_THREADS) w.y[i] = __ldcg(w.ysel + static_cast<int64_t>(best) * m + i);
    return;
  }
  for (int i = tid; i < k; i += TK_THREADS) w.y[i] = y[i];
  if (tid == 0) ctl->mu = mu;
}

// X = X0 + sum_{i<k} y_i V_i  (Eq. 10S); after a restart X holds the iterate
// the cycle started from and takes the place of X0 (elementwise in place)
template <typename T>
__global__ void k_assemble(Work w0, PtrRef X0r0, PtrRef Xr0, const int* gate) {
  const int64_t bo = bidx(w0.b).off;
  const Work w = w0.at(bo);
  const PtrRef X0r = X0r0.at(bo), Xr = Xr0.at(bo);
  gate = bsh(gate, bo);
  if (gate != nullptr && *gate) return;
  const int k = w.ctl->j;
  __shared__ T ys[kMaxK];
  for (int i = threadIdx.x; i < k; i += blockDim.x) ys[i] = coef_as<T>(w.y[i]);
  __syncthreads();
  T* X = Xr.get<T>();
  const T* X0 = w.ctl->cycle > 0 ? X : X0r.get<const T>();
  const T* V = static_cast<const T*>(w.V);
  const int64_t n = w.n;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n;
       o += (int64_t)gridDim.x * blockDim.x) {
    T v = (X0 != nullptr) ? X0[o] : static_cast<T>(0);
    for (int i = 0; i < k; ++i) v += ys[i] * V[static_cast<int64_t>(i) * n + o];
    X[o] = v;
  }
}

__global__ void k_finalize(Work w0, InfoDev* info0) {
  const int64_t bo = bidx(w0.b).off;
  const Work w = w0.at(bo);
  InfoDev* info = bsh(info0, bo);
  const Ctl* c = w.ctl;
  const int t = threadIdx.x;
  if (t == 0) {
    info->iters = c->iters_total;
    info->restarts = c->cycle;
    info->breakdown = c->breakdown;
    info->converged = c->converged;
    info->status = c->status;
    info->k = c->j;
    info->beta = c->beta0;
    info->mu = c->mu;
    info->rho_final = c->rho;
    info->true_rel_resid = c->true_rr;
    info->true_rel_resid_theta = c->true_th;
  }
  for (int i = t; i < c->iters_total && i < kMaxK; i += blockDim.x) info->rho_hist[i] = w.rho_hist[i];
  for (int i = t; i < kMaxMu; i += blockDim.x) info->gcv[i] = w.gcv[i];
}

// Holds the stream until the host has queued a whole kernel group (phase
// timing): one thread polls a flag in mapped host memory.  The wait is
// bounded (limit_ns of globaltimer; phase timing gives 10 s, room for the
// lazy loading of modules on a first launch); on expiry the kernel records
// RTG_ERR_TIMEOUT in *status and returns, so the stream never stalls.
__global__ void k_gate(const volatile unsigned* flag, unsigned want, volatile unsigned* status,
                       unsigned long long limit_ns) {
  unsigned long long t0;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  while (*flag < want) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > limit_ns) {
      *status = RTG_ERR_TIMEOUT;
      return;
    }
    __nanosleep(500);
  }
}

cudaError_t launch_gate(const unsigned* flag, unsigned want, unsigned* status, cudaStream_t s,
                        unsigned long long limit_ns) {
  k_gate<<<1, 1, 0, s>>>(flag, want, status, limit_ns);
  return cudaGetLastError();
}

static unsigned ew_grid(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  return static_cast<unsigned>(b < 1 ? 1 : b);
}

cudaError_t launch_tikhonov(const Work& w, const FinishOpts& f, cudaStream_t s, const int* gate) {
  const unsigned blocks = (f.mode == 2) ? static_cast<unsigned>(f.n_mu) : 1u;
  const size_t sm = static_cast<size_t>(tk_scratch_doubles(w.m)) * sizeof(double);
  const int in_smem = sm <= size_t(200) * 1024 ? 1 : 0;
  if (in_smem) {
    cudaError_t e = set_smem(k_tikhonov, sm);
    if (e != cudaSuccess) return e;
  }
  k_tikhonov<<<dim3(blocks, 1, w.b.n), TK_THREADS, in_smem ? sm : 0, s>>>(w, f.desc, f.mode,
                                                                         w.ysel + kMaxMu * w.m, in_smem, gate);
  return cudaGetLastError();
}

// X = X0 + sum_{i<k} y_i V_i with V in BF16 (FP32 arithmetic, 8 values per load);
// X0 after a restart as in k_assemble
__global__ void k_assemble_bf16(Work w0, PtrRef X0r0, PtrRef Xr0, const int* gate) {
  const int64_t bo = bidx(w0.b).off;
  const Work w = w0.at(bo);
  const PtrRef X0r = X0r0.at(bo), Xr = Xr0.at(bo);
  gate = bsh(gate, bo);
  if (gate != nullptr && *gate) return;
  const int k = w.ctl->j;
  __shared__ float ys[kMaxK];
  for (int i = threadIdx.x; i < k; i += blockDim.x) ys[i] = coef_as<float>(w.y[i]);
  __syncthreads();
  float* X = Xr.get<float>();
  const float* X0 = w.ctl->cycle > 0 ? X : X0r.get<const float>();
  const uint4* V8 = static_cast<const uint4*>(w.V);
  const int64_t n8 = w.n / 8;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n8;
       o += (int64_t)gridDim.x * blockDim.x) {
    float acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = (X0 != nullptr) ? X0[8 * o + q] : 0.f;
    for (int i = 0; i < k; ++i) {
      const uint4 v = V8[static_cast<int64_t>(i) * n8 + o];
      const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        acc[2 * q] = fmaf(ys[i], __uint_as_float(w4[q] << 16), acc[2 * q]);
        acc[2 * q + 1] = fmaf(ys[i], __uint_as_float(w4[q] & 0xffff0000u), acc[2 * q + 1]);
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) X[8 * o + q] = acc[q];
  }
}

cudaError_t launch_assemble(const Work& w, PtrRef X0, PtrRef X, cudaStream_t s, const int* gate) {
  if (w.vdtype == RTG_BF16) {
    k_assemble_bf16<<<dim3(ew_grid(w.n / 8 + 1), 1, w.b.n), 256, 0, s>>>(w, X0, X, gate);
    return cudaGetLastError();
  }
  if (w.dtype == RTG_F64) k_assemble<double><<<dim3(ew_grid(w.n), 1, w.b.n), 256, 0, s>>>(w, X0, X, gate);
  else k_assemble<float><<<dim3(ew_grid(w.n), 1, w.b.n), 256, 0, s>>>(w, X0, X, gate);
  return cudaGetLastError();
}

// Final residual of the Block GMRES algorithm (Section 4.4, its last steps:
// R_m = C - A *_N X_m and its Theta-norm).  R (in the V_0 slot) and S(R) (in
// Spart) come from the apply and sketch launched before this kernel.  Each
// block sums R.R, C.C (grid-stride over n) and S(R).S(R) (over d) in
// float-float (FP32) or FP64, writes one row of three partial sums, and the
// last block adds the rows in a fixed order.
template <typename T>
__global__ void __launch_bounds__(256) k_true_resid(Work w0, PtrRef Cr0) {
  const int64_t bo = bidx(w0.b).off;
  const Work w = w0.at(bo);
  const T* C = Cr0.at(bo).get<const T>();
  const T* R = static_cast<const T*>(w.V);
  const T* SR = static_cast<const T*>(w.Spart);
  __shared__ double red[8][3];
  __shared__ int am_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  DotAcc<T> rr, cc, ss;
  for (int64_t o = t0; o < w.n; o += stride) {
    const T r = R[o], c = C[o];
    rr.add(r, r);
    cc.add(c, c);
  }
  for (int64_t o = t0; o < w.d; o += stride) {
    const T v = SR[o];
    ss.add(v, v);
  }
  const double a = rr.warp_total(), b = cc.warp_total(), c = ss.warp_total();
  if (lane == 0) {
    red[warp][0] = a;
    red[warp][1] = b;
    red[warp][2] = c;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double v = 0.0;
    for (int u = 0; u < 8; ++u) v += red[u][threadIdx.x];
    w.part[static_cast<int64_t>(blockIdx.x) * 3 + threadIdx.x] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) am_last = (ticket_acq_rel(w.counter + 1, gridDim.x - 1) == gridDim.x - 1);
  __syncthreads();
  if (!am_last) return;
  if (warp == 0) {   // lane l sums rows l, l + 32, ...; then a fixed warp tree
    double s3[3] = {0.0, 0.0, 0.0};
    for (unsigned r = lane; r < gridDim.x; r += 32)
      for (int q = 0; q < 3; ++q) s3[q] += __ldcg(w.part + static_cast<int64_t>(r) * 3 + q);
    for (int q = 0; q < 3; ++q) s3[q] = warp_sum(s3[q]);
    if (lane == 0) {
      Ctl* ctl = w.ctl;
      ctl->true_rr = s3[1] > 0.0 ? sqrt(s3[0] / s3[1]) : (s3[0] > 0.0 ? INFINITY : 0.0);
      ctl->true_th = ctl->beta0 > 0.0 ? sqrt(s3[2]) / ctl->beta0 : (s3[2] > 0.0 ? INFINITY : 0.0);
    }
  }
}

cudaError_t launch_true_resid(const Work& w, PtrRef C, cudaStream_t s) {
  // rows of three partial sums must fit the partial-sum buffer
  int64_t blocks = ew_grid(w.n / 4 + 1);
  const int64_t cap = static_cast<int64_t>(w.part_rows) * (2 * w.m + 4) / 3;
  if (blocks > cap) blocks = cap;
  if (blocks > 304) blocks = 304;
  if (blocks < 1) blocks = 1;
  const dim3 g(static_cast<unsigned>(blocks), 1, static_cast<unsigned>(w.b.n));
  if (w.dtype == RTG_F64) k_true_resid<double><<<g, 256, 0, s>>>(w, C);
  else k_true_resid<float><<<g, 256, 0, s>>>(w, C);
  return cudaGetLastError();
}

// Learned warm start: ||S(R_0)|| and ||S(C)|| (float-float sums over the d
// sketch entries, one block), then the decision: fall back to X_0 = 0 with
// GCV when the prediction's sketched residual is not below the cold start's,
// else keep X_0, take lambda = exp(predicted log lambda) and rescale the stop
// level so that both stop at ||S(C - Phi X)|| <= tol ||S(C)||.
__global__ void __launch_bounds__(1024) k_ws_decide(const float* SR, const float* SC, int64_t d,
                                                    const float* loglam, double tol, WsDecision* dec) {
  __shared__ double red[32][2];
  DotAcc<float> r, c;
  for (int64_t i = threadIdx.x; i < d; i += blockDim.x) {
    const float a = SR[i], b = SC[i];
    r.add(a, a);
    c.add(b, b);
  }
  const double rr = r.warp_total(), cc = c.warp_total();
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = rr;
    red[threadIdx.x >> 5][1] = cc;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double sr = 0.0, sc = 0.0;
  for (int u = 0; u < (int)(blockDim.x >> 5); ++u) {
    sr += red[u][0];
    sc += red[u][1];
  }
  sr = sqrt(sr);
  sc = sqrt(sc);
  const bool warm = isfinite(sr) && sr < sc;
  dec->fell_back = warm ? 0 : 1;
  dec->sC = sc;
  dec->sR = sr;
  if (warm) {
    const double ll = static_cast<double>(*loglam);
    dec->lambda = isfinite(ll) ? exp(fmin(fmax(ll, -40.0), 20.0)) : 1e-3;
    dec->tol = sr > 0.0 ? tol * sc / sr : tol;
  } else {
    dec->lambda = -1.0;
    dec->tol = tol;
  }
}

__global__ void k_ws_zero_if(const WsDecision* dec, float* X, int64_t n) {
  if (!dec->fell_back) return;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n; o += (int64_t)gridDim.x * blockDim.x)
    X[o] = 0.f;
}

__global__ void k_ws_write_desc(const WsDecision* dec, SolveDesc* desc) {
  desc->tol = dec->tol;
  desc->lambda = dec->lambda;
}

cudaError_t launch_ws_decide(const float* SR, const float* SC, int64_t d, const float* loglam, double tol,
                             WsDecision* dec, cudaStream_t s) {
  k_ws_decide<<<1, 1024, 0, s>>>(SR, SC, d, loglam, tol, dec);
  return cudaGetLastError();
}

cudaError_t launch_ws_zero_if(const WsDecision* dec, float* X, int64_t n, cudaStream_t s) {
  k_ws_zero_if<<<ew_grid(n), 256, 0, s>>>(dec, X, n);
  return cudaGetLastError();
}

cudaError_t launch_ws_write_desc(const WsDecision* dec, SolveDesc* desc, cudaStream_t s) {
  k_ws_write_desc<<<1, 1, 0, s>>>(dec, desc);
  return cudaGetLastError();
}

// Work queue of a batched solve: a graph branch takes the next problem of
// its class with one atomic increment of the class's counter and copies that
// problem's descriptor into its own, which its kernels read.  With `done`
// set, the branch first returns the info record of the problem it has just
// solved to that problem's place.  The branch's loop condition is 1 while
// the class has problems left, else 0 (the branch then ends).  A nested loop
// condition keeps its value from one pass of the outer loop's body to the
// next, so the solve's own loop condition is set to 1 for the new problem
// (the first problem of a launch starts from the condition's default, 1).
__global__ void k_queue_next(QueueArgs q, int done) {
  __shared__ int next;
  const int cur = *q.cur;
  if (done && cur >= 0) {
    const uint64_t* src = reinterpret_cast<const uint64_t*>(q.my_info);
    uint64_t* dst = reinterpret_cast<uint64_t*>(q.info + cur);
    for (int i = threadIdx.x; i < int(sizeof(InfoDev) / 8); i += blockDim.x) dst[i] = src[i];
  }
  __syncthreads();   // every thread has read *q.cur
  if (threadIdx.x == 0) {
    const unsigned k = atomicAdd(q.counter, 1u);
    next = k < static_cast<unsigned>(q.n) ? static_cast<int>(k) : -1;
    *q.cur = next;
    cudaGraphSetConditional(static_cast<cudaGraphConditionalHandle>(q.cond), next >= 0 ? 1u : 0u);
    if (next >= 0 && q.use_inner) cudaGraphSetConditional(static_cast<cudaGraphConditionalHandle>(q.inner), 1u);
  }
  __syncthreads();
  if (next >= 0) {
    const uint64_t* src = reinterpret_cast<const uint64_t*>(q.desc + next);
    uint64_t* dst = reinterpret_cast<uint64_t*>(q.my_desc);
    for (int i = threadIdx.x; i < int(sizeof(SolveDesc) / 8); i += blockDim.x) dst[i] = src[i];
  }
}
static_assert(sizeof(SolveDesc) % 8 == 0 && sizeof(InfoDev) % 8 == 0, "records are copied as 8-byte words");

cudaError_t launch_queue_next(const QueueArgs& q, int done, cudaStream_t s) {
  k_queue_next<<<1, 128, 0, s>>>(q, done);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const Work& w, InfoDev* info, cudaStream_t s) {
  k_finalize<<<dim3(1, 1, w.b.n), 256, 0, s>>>(w, info);
  return cudaGetLastError();
}

}  // namespace rtg
