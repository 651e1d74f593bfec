// Learned exchange proposal: the network 9 -> 64 -> 64 -> 1 (tanh hidden units) that
// scores an exchange of site i with its antiparallel neighbour j from local spin
// features, its training step (mean squared error against the plain exchange's log
// acceptance min(0, 2 Re Delta_e), hand-written reverse mode, Adam), and batched logits.
// Not part of arXiv:2011.12453; it proposes moves for the paper's MCMC step.
//
// Rows are (configuration b, bond e, orientation o): o = 0 scores i -> j, o = 1 scores
// j -> i for e = (i, j).  Only antiparallel bonds have rows: a block walks its (configuration,
// range of bonds) items, queues the features of their rows and runs the network on 128 rows at a
// time.
//
// Bound: FP32 multiply-add issue (27 k operations a row: 9 x 64 and 64 x 64 forward, the same
// twice in reverse).  Every product is tiled in registers: a thread owns 8 rows x 4 units (or 4 x 4
// entries of dW2), two rows to a packed multiply-add, activations in shared memory with the rows
// contiguous, so 16 packed multiply-adds stand against 3 shared loads (one multiply-add against
// two loads, masked rows of the parallel bonds included, took 6.06 ms for 4096 configurations
// of a random graph of 65 sites; this 0.48).  Weight gradients stay in the registers of the one
// thread that owns them for the whole launch (fixed order, no atomics); per-CTA partials are
// reduced in float64 by a second kernel.
#include "common.cuh"
#include "frag.cuh"
#include "prop.cuh"

namespace gna {

constexpr int kPropThreads = 256;
constexpr int kRows = 128;            // rows of the network at a time
constexpr int kLd = kRows + 4;        // row stride of a unit's activations: 4 mod 32 words
constexpr int kChunk = kPropThreads;  // bonds looked over at a time

struct PropArgs {
  DevGraph g;
  const int8_t* spins;     // [B][N]
  const float* dlogpsi;    // [B][E] (training) or NULL
  const float* params;     // [kPropParams]
  int64_t B;
  int parts;               // items per configuration (ranges of bonds)
  float* logits;           // [B][E][2] (logits)
  double* partial;         // [grid][kPropParams + 2] (training): gradient sums, loss sum, row count
};

// Shared memory in floats.  Units are permuted, position 4 c + j holding unit c + 16 j, so that a
// thread's four units load as 16 bytes and store without bank conflicts.
constexpr int kSW1 = 0;                       // [9][64] permuted columns
constexpr int kSb1 = kSW1 + kPropIn * kPropHid;
constexpr int kSW2 = kSb1 + kPropHid;         // [64][64] permuted columns
constexpr int kSb2 = kSW2 + kPropHid * kPropHid;
constexpr int kSw3 = kSb2 + kPropHid;
constexpr int kSW2T = kSw3 + kPropHid;        // [k][permuted m] = W2[m][k]
constexpr int kSPhi = kSW2T + kPropHid * kPropHid;  // [10][kLd] features, then ones for the rows in use
constexpr int kSH1 = kSPhi + (kPropIn + 1) * kLd;   // [64][kLd]
constexpr int kSD = kSH1 + kPropHid * kLd;          // [64][kLd] dZ2
constexpr int kSTgt = kSD + kPropHid * kLd;         // [kRows] targets
constexpr int kSIdx = kSTgt + kRows;                // [kRows] int64 row indices
constexpr int kSList = kSIdx + 2 * kRows;           // [kChunk] antiparallel bonds of the chunk
constexpr int kSCfg = kSList + kChunk;              // [N] neighbour-spin sums, [N] means, [N] spins (int8)

// tanh of two values: Lambert's continued fraction up to |x| = 1 (relative error below 1e-7), beyond
// it (X - 1)/(X + 1) with X = exp(2 |x|); one reciprocal either way.
__device__ __forceinline__ uint64_t tanh2(uint64_t x) {
  const uint64_t z = f2_mul(x, x);
  const uint64_t w = f2_mul(x, f2_fma(z, f2_fma(z, f2_dup(1.f / 15.f), f2_dup(7.f)), f2_dup(63.f)));
  const uint64_t Q = f2_fma(z, f2_add(z, f2_dup(28.f)), f2_dup(63.f));
  float v[2], n[2], d[2];
  f2_unpack(x, v[0], v[1]);
  f2_unpack(w, n[0], n[1]);
  f2_unpack(Q, d[0], d[1]);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float X = __expf(fminf(2.f * fabsf(v[i]), 40.f));
    const bool far = fabsf(v[i]) > 1.f;
    n[i] = far ? copysignf(X - 1.f, v[i]) : n[i];
    d[i] = far ? X + 1.f : d[i];
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d[i]));
    n[i] *= r;
  }
  return f2_pack(n[0], n[1]);
}

// acc[j][p] (4 units x 4 row pairs) += sum_k A[k][rows] B[k][unit j]: A rows contiguous, B permuted.
template <int K>
__device__ __forceinline__ void prop_gemm(const float* A, const float* B, int tr, int tc, uint64_t (*acc)[4]) {
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(A + k * kLd + tr * 8);
    const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(A + k * kLd + tr * 8 + 4);
    const float4 w = *reinterpret_cast<const float4*>(B + k * kPropHid + tc * 4);
    const uint64_t wd[4] = {f2_dup(w.x), f2_dup(w.y), f2_dup(w.z), f2_dup(w.w)};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[j][0] = f2_fma(a0.x, wd[j], acc[j][0]);
      acc[j][1] = f2_fma(a0.y, wd[j], acc[j][1]);
      acc[j][2] = f2_fma(a1.x, wd[j], acc[j][2]);
      acc[j][3] = f2_fma(a1.y, wd[j], acc[j][3]);
    }
  }
}

// A thread's four units of 8 rows to (or from) a [64][kLd] array.
__device__ __forceinline__ void prop_store(float* S, int tr, int tc, const uint64_t (*v)[4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float* o = S + (tc + 16 * j) * kLd + tr * 8;
    *reinterpret_cast<ulonglong2*>(o) = make_ulonglong2(v[j][0], v[j][1]);
    *reinterpret_cast<ulonglong2*>(o + 4) = make_ulonglong2(v[j][2], v[j][3]);
  }
}

// A thread's gradient sums over the launch.
struct PropAcc {
  float w2[4][4];        // dW2[mi + 16 i][ki + 16 j]
  float w1[4];           // threads < 160: row f = tid / 16 of [dW1; db1], units ki + 16 j
  uint64_t b2[4], w3[4]; // by unit, row pairs
  float b3, loss, count;
};

// The network on the queued rows [0, n): logits out, or the gradient sums of the training loss.
template <bool GRAD>
__device__ void prop_rows(const PropArgs& a, float* sm, float b3, int n, PropAcc& g) {
  const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
  uint64_t acc[4][4];
  __syncthreads();  // the queue is complete
  // hidden layer 1
  {
    const float4 b = *reinterpret_cast<const float4*>(sm + kSb1 + tc * 4);
    const float bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[j][p] = f2_dup(bb[j]);
  }
  prop_gemm<kPropIn>(sm + kSPhi, sm + kSW1, tr, tc, acc);
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[j][p] = tanh2(acc[j][p]);
  prop_store(sm + kSH1, tr, tc, acc);
  __syncthreads();
  // hidden layer 2 and the logits
  {
    const float4 b = *reinterpret_cast<const float4*>(sm + kSb2 + tc * 4);
    const float bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[j][p] = f2_dup(bb[j]);
  }
  prop_gemm<kPropHid>(sm + kSH1, sm + kSW2, tr, tc, acc);
  const float4 w3v = *reinterpret_cast<const float4*>(sm + kSw3 + tc * 4);
  const float w3[4] = {w3v.x, w3v.y, w3v.z, w3v.w};
  uint64_t z[4] = {0, 0, 0, 0};
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      acc[j][p] = tanh2(acc[j][p]);
      z[p] = f2_fma(acc[j][p], f2_dup(w3[j]), z[p]);
    }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) z[p] = f2_add(z[p], __shfl_xor_sync(0xffffffffu, z[p], o));
  if (!GRAD) {
    const int64_t* idx = reinterpret_cast<const int64_t*>(sm + kSIdx);
    if (tc == 0)
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        float z0, z1;
        f2_unpack(z[p], z0, z1);
        const int r = tr * 8 + 2 * p;
        if (r < n) a.logits[idx[r]] = z0 + b3;
        if (r + 1 < n) a.logits[idx[r + 1]] = z1 + b3;
      }
    __syncthreads();
    return;
  }
  uint64_t dl[4];  // d loss / d logit, 0 past the last row
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int r = tr * 8 + 2 * p;
    const float2 t = *reinterpret_cast<const float2*>(sm + kSTgt + r);
    float z0, z1;
    f2_unpack(z[p], z0, z1);
    const float e0 = r < n ? z0 + b3 - t.x : 0.f, e1 = r + 1 < n ? z1 + b3 - t.y : 0.f;
    dl[p] = f2_pack(2.f * e0, 2.f * e1);
    if (tc == 0) {
      g.loss += e0 * e0 + e1 * e1;
      g.b3 += 2.f * (e0 + e1);
    }
  }
  // dZ2 = dlogit w3 (1 - H2^2), and the sums of w3 and b2
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint64_t h = acc[j][p];
      g.w3[j] = f2_fma(dl[p], h, g.w3[j]);
      const uint64_t s = f2_fma(f2_mul(h, h), f2_dup(-1.f), f2_dup(1.f));
      acc[j][p] = f2_mul(f2_mul(dl[p], f2_dup(w3[j])), s);
      g.b2[j] = f2_add(g.b2[j], acc[j][p]);
    }
  prop_store(sm + kSD, tr, tc, acc);
  __syncthreads();
  // dW2 += H1^T dZ2: entries (mi + 16 i, ki + 16 j), even and odd rows apart within the tile
  {
    const int mi = tr, ki = tc;
    uint64_t s[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[i][j] = 0;
#pragma unroll 2
    for (int r = 0; r < kRows; r += 4) {
      ulonglong2 h[4], d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        h[i] = *reinterpret_cast<const ulonglong2*>(sm + kSH1 + (mi + 16 * i) * kLd + r);
        d[i] = *reinterpret_cast<const ulonglong2*>(sm + kSD + (ki + 16 * i) * kLd + r);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = f2_fma(h[i].y, d[j].y, f2_fma(h[i].x, d[j].x, s[i][j]));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float x, y;
        f2_unpack(s[i][j], x, y);
        g.w2[i][j] += x + y;
      }
  }
  // dZ1 = (dZ2 W2^T) (1 - H1^2), over H1
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[j][p] = 0;
  prop_gemm<kPropHid>(sm + kSD, sm + kSW2T, tr, tc, acc);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float* o = sm + kSH1 + (tc + 16 * j) * kLd + tr * 8;
    const ulonglong2 h0 = *reinterpret_cast<const ulonglong2*>(o), h1 = *reinterpret_cast<const ulonglong2*>(o + 4);
    const uint64_t h[4] = {h0.x, h0.y, h1.x, h1.y};
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[j][p] = f2_mul(acc[j][p], f2_fma(f2_mul(h[p], h[p]), f2_dup(-1.f), f2_dup(1.f)));
  }
  __syncthreads();  // every read of H1 is done
  prop_store(sm + kSH1, tr, tc, acc);
  __syncthreads();
  // [dW1; db1] += [phi; 1]^T dZ1
  if (tid < 16 * (kPropIn + 1)) {
    const float* f = sm + kSPhi + tr * kLd;
    uint64_t s[4] = {0, 0, 0, 0};
#pragma unroll 4
    for (int r = 0; r < kRows; r += 4) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(f + r);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const ulonglong2 d = *reinterpret_cast<const ulonglong2*>(sm + kSH1 + (tc + 16 * j) * kLd + r);
        s[j] = f2_fma(x.y, d.y, f2_fma(x.x, d.x, s[j]));
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float x, y;
      f2_unpack(s[j], x, y);
      g.w1[j] += x + y;
    }
  }
  if (tid == 0) g.count += (float)n;
  __syncthreads();
}

template <bool GRAD>
__global__ void __launch_bounds__(kPropThreads, 2) k_prop(const __grid_constant__ PropArgs a) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_cnt[kPropThreads / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const DevGraph& g = a.g;
  const int N = g.n, E = g.E;
  for (int i = tid; i < kPropIn * kPropHid; i += kPropThreads)
    sm[kSW1 + i] = a.params[kPropOW1 + (i & ~63) + ((i & 63) >> 2) + 16 * (i & 3)];
  for (int i = tid; i < kPropHid; i += kPropThreads) {
    const int u = (i >> 2) + 16 * (i & 3);
    sm[kSb1 + i] = a.params[kPropOb1 + u];
    sm[kSb2 + i] = a.params[kPropOb2 + u];
    sm[kSw3 + i] = a.params[kPropOw3 + u];
  }
  for (int i = tid; i < kPropHid * kPropHid; i += kPropThreads) {
    const int u = ((i & 63) >> 2) + 16 * (i & 3);
    sm[kSW2 + i] = a.params[kPropOW2 + (i & ~63) + u];
    sm[kSW2T + i] = a.params[kPropOW2 + u * kPropHid + (i >> 6)];
  }
  for (int i = tid; i < (kPropIn + 1) * kLd; i += kPropThreads) sm[kSPhi + i] = 0.f;
  for (int i = tid; i < kRows; i += kPropThreads) sm[kSTgt + i] = 0.f;
  const float b3 = a.params[kPropOb3];
  PropAcc acc;
  if (GRAD) memset(&acc, 0, sizeof(acc));
  float* n1 = sm + kSCfg;
  float* q = n1 + N;
  int8_t* s = reinterpret_cast<int8_t*>(q + N);
  int* list = reinterpret_cast<int*>(sm + kSList);
  int64_t* idx = reinterpret_cast<int64_t*>(sm + kSIdx);
  int queued = 0;
  for (int64_t item = blockIdx.x; item < a.B * a.parts; item += gridDim.x) {
    const int64_t b = item / a.parts;
    const int part = (int)(item - b * a.parts);
    const int e_lo = (int)((int64_t)E * part / a.parts), e_hi = (int)((int64_t)E * (part + 1) / a.parts);
    __syncthreads();
    for (int v = tid; v < N; v += kPropThreads) s[v] = a.spins[b * N + v];
    __syncthreads();
    for (int v = tid; v < N; v += kPropThreads) {
      const int k0 = __ldg(g.row_ptr + v), k1 = __ldg(g.row_ptr + v + 1);
      float x = 0.f;
      for (int k = k0; k < k1; ++k) x += (float)s[__ldg(g.col + k)];
      n1[v] = x;
      q[v] = k1 > k0 ? x / (float)(k1 - k0) : 0.f;
    }
    for (int c0 = e_lo; c0 < e_hi; c0 += kChunk) {
      // the chunk's antiparallel bonds, in order
      const int e = c0 + tid;
      bool anti = false;
      if (e < e_hi) anti = s[__ldg(g.edges + 2 * e)] != s[__ldg(g.edges + 2 * e + 1)];
      const unsigned mask = __ballot_sync(0xffffffffu, anti);
      if (lane == 0) s_cnt[warp] = __popc(mask);
      __syncthreads();
      int before = 0, cnt = 0;
      for (int w = 0; w < kPropThreads / 32; ++w) {
        before += w < warp ? s_cnt[w] : 0;
        cnt += s_cnt[w];
      }
      if (anti) list[before + __popc(mask & ((1u << lane) - 1u))] = e;
      if (!GRAD && e < e_hi && !anti)
        a.logits[(b * E + e) * 2] = a.logits[(b * E + e) * 2 + 1] = __int_as_float(0x7fc00000);
      __syncthreads();
      for (int pos = 0; pos < cnt;) {
        const int take = min(cnt - pos, (kRows - queued) / 2);
        if (tid < 2 * take) {
          const int bond = list[pos + (tid >> 1)], o = tid & 1, r = queued + tid;
          const int i = __ldg(g.edges + 2 * bond + o), j = __ldg(g.edges + 2 * bond + 1 - o);
          const int ki0 = __ldg(g.row_ptr + i), ki1 = __ldg(g.row_ptr + i + 1);
          const int kj0 = __ldg(g.row_ptr + j), kj1 = __ldg(g.row_ptr + j + 1);
          const int di = ki1 - ki0, dj = kj1 - kj0;
          const float si = (float)s[i], sj = (float)s[j];
          float bi = 0.f, bj = 0.f;
          for (int k = ki0; k < ki1; ++k) {
            const int u = __ldg(g.col + k);
            if (u != j) bi += q[u];
          }
          for (int k = kj0; k < kj1; ++k) {
            const int u = __ldg(g.col + k);
            if (u != i) bj += q[u];
          }
          float* f = sm + kSPhi + r;
          f[0] = si;
          f[kLd] = sj;
          f[2 * kLd] = (float)__ldg(g.J + bond);
          f[3 * kLd] = 1.f / (float)di;
          f[4 * kLd] = 1.f / (float)dj;
          f[5 * kLd] = (n1[i] - sj) / (float)max(di - 1, 1);
          f[6 * kLd] = (n1[j] - si) / (float)max(dj - 1, 1);
          f[7 * kLd] = di > 1 ? bi / (float)(di - 1) : 0.f;
          f[8 * kLd] = dj > 1 ? bj / (float)(dj - 1) : 0.f;
          f[9 * kLd] = 1.f;
          if (GRAD)
            sm[kSTgt + r] = fminf(0.f, 2.f * a.dlogpsi[b * E + bond]);
          else
            idx[r] = (b * E + bond) * 2 + o;
        }
        queued += 2 * take;
        pos += take;
        if (queued == kRows) {
          prop_rows<GRAD>(a, sm, b3, kRows, acc);
          queued = 0;
        }
      }
      __syncthreads();
    }
  }
  if (queued > 0) prop_rows<GRAD>(a, sm, b3, queued, acc);
  if (!GRAD) return;
  // the block's sums: rows of dW2 and dW1 from their owners, the others over the 16 row groups
  double* out = a.partial + (size_t)blockIdx.x * (kPropParams + 2);
  const int tr = tid >> 4, tc = tid & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) out[kPropOW2 + (tr + 16 * i) * kPropHid + tc + 16 * j] = (double)acc.w2[i][j];
  if (tid < 16 * (kPropIn + 1))
#pragma unroll
    for (int j = 0; j < 4; ++j) out[(tr < kPropIn ? kPropOW1 + tr * kPropHid : kPropOb1) + tc + 16 * j] = (double)acc.w1[j];
  __syncthreads();
  float* red = sm + kSH1;  // [16 row groups][2][64], then [16][2]
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float x, y;
    f2_unpack(acc.b2[j], x, y);
    red[(tr * 2) * kPropHid + tc + 16 * j] = x + y;
    f2_unpack(acc.w3[j], x, y);
    red[(tr * 2 + 1) * kPropHid + tc + 16 * j] = x + y;
  }
  if (tc == 0) {
    red[2048 + tr] = acc.b3;
    red[2064 + tr] = acc.loss;
  }
  __syncthreads();
  if (tid < 2 * kPropHid) {
    double t = 0.0;
    for (int r = 0; r < 16; ++r) t += (double)red[r * 128 + tid];
    out[tid < kPropHid ? kPropOb2 + tid : kPropOw3 + tid - kPropHid] = t;
  } else if (tid < 2 * kPropHid + 2) {
    double t = 0.0;
    for (int r = 0; r < 16; ++r) t += (double)red[2048 + 16 * (tid - 2 * kPropHid) + r];
    out[tid == 2 * kPropHid ? kPropOb3 : kPropParams] = t;
  }
  if (tid == 0) out[kPropParams + 1] = (double)acc.count;
}

// grad = (sum over CTAs of the partials) / count; loss likewise.  Fixed order, float64.
__global__ void k_prop_reduce(const double* partial, int grid, double* grad, double* loss) {
  const int p = blockIdx.x * 32 + (threadIdx.x & 31);
  const double s = sum_partials(partial, grid, kPropParams + 2, p, p <= kPropParams);
  const double n = sum_partials(partial, grid, kPropParams + 2, kPropParams + 1, true);
  if (threadIdx.x >= 32 || p > kPropParams) return;
  const double inv = n > 0.0 ? 1.0 / n : 0.0;
  if (p < kPropParams)
    grad[p] = s * inv;
  else if (loss)
    *loss = s * inv;
}

// Adam (Kingma & Ba 2015), step t >= 1.
__global__ void k_adam(float* params, float* m, float* v, const double* grad, int P, int t, double lr, double b1,
                       double b2, double eps) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const double g = grad[p];
  const double mm = b1 * (double)m[p] + (1.0 - b1) * g;
  const double vv = b2 * (double)v[p] + (1.0 - b2) * g * g;
  m[p] = (float)mm;
  v[p] = (float)vv;
  const double mh = mm / (1.0 - pow(b1, (double)t));
  const double vh = vv / (1.0 - pow(b2, (double)t));
  params[p] = (float)((double)params[p] - lr * mh / (sqrt(vh) + eps));
}

// Items (configuration, range of bonds) for two blocks on every SM: whole configurations while
// there are enough of them, ranges of at least 32 bonds otherwise.
static int prop_parts(int64_t B, int E, int sms) {
  int64_t parts = (2 * (int64_t)sms + B - 1) / B;
  const int64_t most = (E + 31) / 32;
  if (parts > most) parts = most;
  return parts < 1 ? 1 : (int)parts;
}
static int prop_grid(int64_t B, int E, int* parts) {
  DeviceInfo di;
  *parts = 1;
  if (device_info(&di) != GNA_OK) return 1;
  *parts = prop_parts(B, E, di.sms);
  const int64_t items = B * *parts, grid = 2 * (int64_t)di.sms;
  return (int)(items < grid ? (items < 1 ? 1 : items) : grid);
}

size_t prop_workspace(const gna_graph* g, int64_t B) {
  int parts;
  return align_up((size_t)prop_grid(B, g->d.E, &parts) * (kPropParams + 2) * sizeof(double));
}

static gna_status prop_run(bool grad, const gna_graph* g, const int8_t* spins, const float* dlogpsi, int64_t B,
                           const float* params, float* logits, double* partial, int* grid, cudaStream_t st) {
  PropArgs a;
  a.g = g->d;
  a.spins = spins;
  a.dlogpsi = dlogpsi;
  a.params = params;
  a.B = B;
  a.logits = logits;
  a.partial = partial;
  *grid = prop_grid(B, g->d.E, &a.parts);
  const int smem = kSCfg * 4 + g->d.n * 8 + (g->d.n + 15) / 16 * 16;
  const void* k = grad ? (const void*)k_prop<true> : (const void*)k_prop<false>;
  DeviceInfo di;
  gna_status s = device_info(&di);
  if (s == GNA_OK) s = allow_smem(k, (uint64_t)di.smem_optin - 64);
  if (s != GNA_OK) return s;
  void* args[] = {&a};
  GNA_CUDA_TRY(cudaLaunchKernel(k, dim3(*grid), dim3(kPropThreads), args, smem, st));
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

gna_status prop_grad_launch(const gna_graph* g, const int8_t* spins, const float* dlogpsi, int64_t B,
                            const float* params, double* grad, double* loss, void* ws, cudaStream_t st) {
  int grid = 0;
  const gna_status s = prop_run(true, g, spins, dlogpsi, B, params, nullptr, (double*)ws, &grid, st);
  if (s != GNA_OK) return s;
  k_prop_reduce<<<(kPropParams + 1 + 31) / 32, 32 * kSumRows, 0, st>>>((double*)ws, grid, grad, loss);
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

gna_status prop_logits_launch(const gna_graph* g, const int8_t* spins, int64_t B, const float* params, float* logits,
                              cudaStream_t st) {
  int grid = 0;
  return prop_run(false, g, spins, nullptr, B, params, logits, nullptr, &grid, st);
}

gna_status prop_adam_launch(float* params, float* m, float* v, const double* grad, int t, double lr,
                            cudaStream_t st) {
  k_adam<<<(kPropParams + 255) / 256, 256, 0, st>>>(params, m, v, grad, kPropParams, t, lr, 0.9, 0.999, 1e-8);
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

}  // namespace gna
