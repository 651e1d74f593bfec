// ISGO importance weights and statistics (Eq. isgo of arXiv:2011.12453, read as the
// covariance gradient), the plain gradient step, and the device Philox used by the
// sampler exposed for bit-exact checks.  All reductions are float64 in a fixed order.
#include <cmath>

#include "common.cuh"

namespace gna {

static __device__ int s_isgo_status;

// Blocks of 128 threads, at most one per SM: up to 19456 samples a thread has one, which is where
// the FP64 exponentials and logarithms want them -- spread over the chip's FP64 pipes (with 1024
// samples per block of 256 threads the two passes took 34 + 29 us at 4096 samples, with these
// blocks and no separate combining kernels in between about a third of that).
constexpr int kRedThreads = 128;
constexpr int kRedBlocks = 152;

// Fixed-order block reductions of N doubles per thread (results in every thread): butterflies
// within the warps, then the warps in order.
template <bool MAX, int N>
__device__ void block_reduce(double* v, double* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < N; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double y = __shfl_xor_sync(0xffffffffu, v[i], o);
      v[i] = MAX ? fmax(v[i], y) : v[i] + y;
    }
    if (lane == 0) sm[i * (kRedThreads / 32) + warp] = v[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double x = sm[i * (kRedThreads / 32)];
    for (int w = 1; w < kRedThreads / 32; ++w) {
      const double y = sm[i * (kRedThreads / 32) + w];
      x = MAX ? fmax(x, y) : x + y;
    }
    v[i] = x;
  }
  __syncthreads();
}

__device__ inline double log_weight(const double* lp, const double* lp0, const double* counts, int64_t x) {
  double lw = 2.0 * (lp[2 * x] - lp0[2 * x]);
  if (counts) lw += log(counts[x]);
  return lw;
}

// pass 1: per block (m_b, sum exp(lw - m_b), sum exp(lw - m_b) E); done (when not NULL) is the
// counter of pass 2's blocks, reset here
__global__ void __launch_bounds__(kRedThreads) k_isgo_pass1(const double* lp, const double* lp0, const double* counts,
                                                            const double* E, int64_t B, double* part, int* done) {
  __shared__ double sm[3 * kRedThreads / 32];
  const int64_t x0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  const double lw0 = x0 < B ? log_weight(lp, lp0, counts, x0) : -INFINITY;
  double m = lw0;
  for (int64_t x = x0 + step; x < B; x += step) m = fmax(m, log_weight(lp, lp0, counts, x));
  block_reduce<true, 1>(&m, sm);
  double s[3] = {0.0, 0.0, 0.0};
  if (m > -INFINITY) {
    for (int64_t x = x0; x < B; x += step) {
      const double w = exp((x == x0 ? lw0 : log_weight(lp, lp0, counts, x)) - m);
      s[0] += w;
      s[1] += w * E[2 * x];
      s[2] += w * E[2 * x + 1];
    }
  }
  block_reduce<false, 3>(s, sm);
  if (threadIdx.x == 0) {
    part[4 * blockIdx.x + 0] = m;
    part[4 * blockIdx.x + 1] = s[0];
    part[4 * blockIdx.x + 2] = s[1];
    part[4 * blockIdx.x + 3] = s[2];
    if (blockIdx.x == 0 && done) *done = 0;
  }
}

// The blocks' partials combined: g = (m, S, S_re, S_im), the same in every thread.
__device__ void combine1(const double* part, int nb, double* g, double* sm) {
  double m = -INFINITY;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) m = fmax(m, part[4 * b]);
  block_reduce<true, 1>(&m, sm);
  double s[3] = {0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const double mb = part[4 * b];
    const double f = mb > -INFINITY ? exp(mb - m) : 0.0;
    s[0] += f * part[4 * b + 1];
    s[1] += f * part[4 * b + 2];
    s[2] += f * part[4 * b + 3];
  }
  block_reduce<false, 3>(s, sm);
  g[0] = m;
  g[1] = s[0];
  g[2] = s[1];
  g[3] = s[2];
}

// a shard's (m, S, S Re Ebar, S Im Ebar)
__global__ void __launch_bounds__(kRedThreads) k_isgo_combine1(const double* part, int nb, double* gsum) {
  __shared__ double sm[3 * kRedThreads / 32];
  double g[4];
  combine1(part, nb, g, sm);
  if (threadIdx.x < 4) gsum[threadIdx.x] = threadIdx.x == 0 ? g[0] : threadIdx.x == 1 ? g[1] : threadIdx.x == 2 ? g[2] : g[3];
}

// stats = (Re Ebar, Im Ebar, var, ess) from the blocks' (var, q, n), or with raw != NULL the shard's
// sums only
__device__ void combine2(const double* part2, int nb, double er, double ei, double* stats, double* raw, double* sm) {
  double s[3] = {0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    s[0] += part2[3 * b];
    s[1] += part2[3 * b + 1];
    s[2] += part2[3 * b + 2];
  }
  block_reduce<false, 3>(s, sm);
  if (threadIdx.x != 0) return;
  if (raw) {
    raw[0] = s[0];
    raw[1] = s[1];
    raw[2] = s[2];
    return;
  }
  stats[0] = er;
  stats[1] = ei;
  stats[2] = s[0];
  stats[3] = 1.0 / s[1];
  if (!isfinite(er) || !isfinite(ei) || !isfinite(s[0]) || !isfinite(s[1])) atomicOr(&s_isgo_status, 2);
  // degenerate reweighting (the failure the paper warns of: a few samples carry the
  // weights and the gradient is dominated by them): IS-ESS below 1% of the copies
  else if (1.0 / s[1] < 0.01 * s[2]) atomicOr(&s_isgo_status, 4);
}

__global__ void __launch_bounds__(kRedThreads) k_isgo_combine2(const double* part2, int nb, double* raw) {
  __shared__ double sm[3 * kRedThreads / 32];
  combine2(part2, nb, 0.0, 0.0, nullptr, raw, sm);
}

// pass 2: p, cotangents, per block sum p |E - Ebar|^2 and sum p^2 / c.  global4 = (m, S, Re Ebar,
// Im Ebar) of all shards, or NULL: every block combines pass 1's partials itself, and the block
// that finishes last the others' sums into stats.
__global__ void __launch_bounds__(kRedThreads) k_isgo_pass2(const double* lp, const double* lp0, const double* counts,
                                                            const double* E, int64_t B, const double* global4,
                                                            const double* part, int nb, double* cot, double* part2,
                                                            double* stats, int* done) {
  __shared__ double sm[3 * kRedThreads / 32];
  __shared__ int s_last;
  double g[4];
  if (global4) {
    for (int i = 0; i < 4; ++i) g[i] = global4[i];
  } else {
    combine1(part, nb, g, sm);
    g[2] /= g[1];
    g[3] /= g[1];
  }
  double s[3] = {0.0, 0.0, 0.0};
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < B; x += (int64_t)gridDim.x * blockDim.x) {
    const double p = exp(log_weight(lp, lp0, counts, x) - g[0]) / g[1];
    const double dr = E[2 * x] - g[2], di = E[2 * x + 1] - g[3], c = counts ? counts[x] : 1.0;
    s[0] += p * (dr * dr + di * di);
    s[1] += counts ? p * p / c : p * p;
    s[2] += c;
    if (cot) {
      cot[2 * x] = 2.0 * p * dr;
      cot[2 * x + 1] = 2.0 * p * di;
    }
  }
  block_reduce<false, 3>(s, sm);
  if (threadIdx.x == 0) {
    part2[3 * blockIdx.x] = s[0];
    part2[3 * blockIdx.x + 1] = s[1];
    part2[3 * blockIdx.x + 2] = s[2];
    s_last = 0;
    if (stats) {
      __threadfence();
      s_last = atomicAdd(done, 1) == (int)gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  combine2(part2, nb, g[2], g[3], stats, nullptr, sm);
}

static int isgo_blocks(int64_t B) {
  const int64_t nb = (B + kRedThreads - 1) / kRedThreads;
  return (int)(nb < 1 ? 1 : nb > kRedBlocks ? kRedBlocks : nb);
}

size_t isgo_weights_ws(int64_t B) {
  const int nb = isgo_blocks(B);
  return align_up((size_t)nb * 4 * 8) + align_up((size_t)nb * 3 * 8) + align_up(4 * 8);
}

gna_status isgo_weights_launch(const double* lp, const double* lp0, const double* E, const double* counts, int64_t B,
                               double* cot, double* stats, void* ws, cudaStream_t st) {
  const int nb = isgo_blocks(B);
  unsigned char* w = (unsigned char*)ws;
  double* part = (double*)w;
  w += align_up((size_t)nb * 4 * 8);
  double* part2 = (double*)w;
  w += align_up((size_t)nb * 3 * 8);
  int* done = (int*)w;
  k_isgo_pass1<<<nb, kRedThreads, 0, st>>>(lp, lp0, counts, E, B, part, done);
  k_isgo_pass2<<<nb, kRedThreads, 0, st>>>(lp, lp0, counts, E, B, nullptr, part, nb, cot, part2, stats, done);
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

// Sample-sharded form: the shard's (m, S, S Re Ebar, S Im Ebar) ...
gna_status isgo_partials_launch(const double* lp, const double* lp0, const double* E, const double* counts, int64_t B,
                                double* part4, void* ws, cudaStream_t st) {
  const int nb = isgo_blocks(B);
  double* part = (double*)ws;
  k_isgo_pass1<<<nb, kRedThreads, 0, st>>>(lp, lp0, counts, E, B, part, nullptr);
  k_isgo_combine1<<<1, kRedThreads, 0, st>>>(part, nb, part4);
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

// ... and, given the global (m, S, Re Ebar, Im Ebar), the shard's cotangents and (var, q, n) sums.
gna_status isgo_finish_launch(const double* lp, const double* lp0, const double* E, const double* counts, int64_t B,
                              const double* global4, double* cot, double* part3, void* ws, cudaStream_t st) {
  const int nb = isgo_blocks(B);
  double* part2 = (double*)ws;
  k_isgo_pass2<<<nb, kRedThreads, 0, st>>>(lp, lp0, counts, E, B, global4, nullptr, nb, cot, part2, nullptr, nullptr);
  k_isgo_combine2<<<1, kRedThreads, 0, st>>>(part2, nb, part3);
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

template <typename T>
__global__ void k_sgd(T* theta, const double* grad, double lr, int P) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < P) theta[p] = (T)((double)theta[p] - lr * grad[p]);
}

gna_status sgd_launch(int prec, void* theta, const double* grad, double lr, int P, cudaStream_t st) {
  if (prec == GNA_PREC_FP64)
    k_sgd<double><<<(P + 255) / 256, 256, 0, st>>>((double*)theta, grad, lr, P);
  else
    k_sgd<float><<<(P + 255) / 256, 256, 0, st>>>((float*)theta, grad, lr, P);
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

__global__ void k_philox(const uint64_t* keys, const uint64_t* ctrs, int64_t n, uint64_t* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const U64x4 r = philox4x64_10(keys[2 * i], keys[2 * i + 1], U64x4{ctrs[4 * i], ctrs[4 * i + 1], ctrs[4 * i + 2], ctrs[4 * i + 3]});
  out[4 * i] = r.x;
  out[4 * i + 1] = r.y;
  out[4 * i + 2] = r.z;
  out[4 * i + 3] = r.w;
}

gna_status philox_launch(const uint64_t* keys, const uint64_t* ctrs, int64_t n, uint64_t* out, cudaStream_t st) {
  if (n == 0) return GNA_OK;
  k_philox<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(keys, ctrs, n, out);
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

gna_status isgo_read_status(int* flags, int clear) {
  int v = 0;
  GNA_CUDA_TRY(cudaMemcpyFromSymbol(&v, s_isgo_status, sizeof(int)));
  *flags |= v;
  if (clear) {
    int z = 0;
    GNA_CUDA_TRY(cudaMemcpyToSymbol(s_isgo_status, &z, sizeof(int)));
  }
  return GNA_OK;
}

}  // namespace gna
