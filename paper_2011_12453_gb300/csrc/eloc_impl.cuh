// Incremental local energy, one warp per tile of 16 rows, for models whose balls fit shared
// memory: the kernel templates of eloc.cu (BF16X2, with log Psi) and eloc32.cu (FP32, tanh and
// ReLU + layer norm).  tc.cu and simt.cu have the general kernels, tc.cu the numerics of the
// difference form ( layer l changes by dY^l = [A_hat dH^{l-1} ; dH^{l-1}] W on ball_l(e) and
// dH^l = f(Y^l + dY^l) - f(Y^l)).
//
// The product comes before the gather.  Gathering is linear, so
//   dY^l_v = a_v sum_{u ~ v} (a_u Z_u[:F]) + Z_v[F:],   Z = dH^{l-1} [W[:F] | W[F:]],
// with a_v = 1/sqrt(d_v).  Compared with multiplying the gathered rows [A_hat dH ; dH] W this
//   - multiplies the rows of ball_{l-1} instead of those of ball_l (7 + 17 + 32 of
//     7 + 17 + 32 + 52 rows a bond on Kagome; none for layer 1, whose two rows are +-(d W)
//     with the one vector d = emb(-1) - emb(+1), multiplied once per CTA in float32),
//   - splits F values of a row into hi + lo instead of 2F, and
//   - needs no neighbour weights: a sum of rows, scaled at both ends.
// A tile's dH comes out of the epilogue in the registers that the next product reads
// (frag.cuh), so dH is never stored; only Z passes through shared memory, in float32.
//
// Bound: instruction issue (tiles of 16 x F; no dense tensor or DRAM limit is near).  A bond is
// worked on by a unit of one or a few warps, as many units as shared memory holds, because
// the work between two row exchanges is a few hundred instructions: with 128-row tiles on
// tcgen05 every layer paid two block barriers and an MMA round trip (barrier 2.5 stalls per
// instruction, 93 instructions per 32 features of a row).  One-warp units meet nobody.
// Measured (local energy with log Psi, tensor-memory kernel before, this one after): Kagome
// 108, L 4, F 32, 16384 configurations 33.9 -> 14.7 ms; triangular 144, L 4, F 48, 4001: 38.0 ->
// 18.4 ms; Kagome 432, L 6, F 64, 512: 26.9 -> 18.6 ms; the error of the energies against 64 bits
// falls 3 to 5 times at weight scale 0.1.
#pragma once

#include <cfloat>

#include "eloc.cuh"
#include "frag.cuh"

namespace gna {

constexpr int kElThreads = 512;
constexpr int kReadout = 512;  // threads of the forward call's readout, whose order of sums is kept
constexpr int kElWarps = kElThreads / 32;

// Arithmetic of a kernel.  EL_X2: W is a BF16 parameter (one term), the forward's operands hi + lo
// as in the forward call.  EL_F32: W in float32 as three BF16 terms; a product of two float32
// values keeps the six products of terms above 2^-24 of it, the large one added with rounding --
// float32 accuracy (over 17 updates of FP32 models the energies' errors against 64 bits are 1e-8 to 2e-6,
// in 15 of them below those of simt.cu's recomputing kernel) at a fraction of the instructions of
// 2 F fused multiply-adds a feature.  EL_F32_LN: the same with f = ReLU +
// layer norm, which couples a row's features: they lie in four lanes, two shuffles a sum.
enum ElMode { EL_X2 = 0, EL_F32 = 1, EL_F32_LN = 2 };
template <int MODE>
struct ElSum {
  typedef double T;
};
template <>
struct ElSum<EL_X2> {
  typedef float T;
};
__host__ __device__ constexpr int el_wterms(int mode) { return mode == EL_X2 ? 1 : 3; }

struct ElArgs {
  DevGraph g;
  Dims m;
  const float* theta;
  const int8_t* spins;
  int64_t B;
  double* logpsi;
  double* eloc;
  float* dlogpsi;
  float* gU;   // [grid][2][L][N][ldu], L2-resident: exp(2 Y) of the CTA's configuration, then Y where that
               // is out of range; with layer norm Y, then H
  float* gH;   // [grid][2][N][ldh] when the forward's rows are in the workspace
  int h_smem;
  int units, uw;                    // units per CTA, warps per unit
  int nbuf;                         // staged tables: 2 (the next bond's travel meanwhile) or 1
  uint32_t oW, obias, oemb, owr, obr, oav, oz0, ospin, olist, orp, owf, ocol, ored, ounit;
  uint32_t otab, tab_bytes;         // a unit's staged tables at otab + h * tab_bytes (never overlaid: rows past
  uint32_t urec[2], upair[2], usum; // a ball's last one are looked up in what an earlier bond left there)
  uint32_t unit_bytes, uz[2];       // a unit's Z buffers at ounit + h * unit_bytes
  uint32_t oH;                      // the forward's rows in shared memory (over the units)
};

__host__ __device__ constexpr int el_ldh(int F) { return F + (F % 32 == 0 ? 16 : 0); }
__host__ __device__ constexpr int el_ldu(int F) { return F + (F % 32 == 0 ? 4 : 0); }

__device__ __forceinline__ void el_bar(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// What the incremental step needs of a cached unit, in one float32: E = exp(2 Y).  H = (E - 1)/(E + 1),
// and 1 - H^2 = 4 E/(1 + E)^2 keeps its relative precision at saturation.  Where E leaves
// [kElTiny, kElCap) (Y outside -42.6 .. 43.4) it is 0 to kElTiny, kElCap or not a number, and Y itself
// is kept beside the cache: a swing of more than 1 is then taken from Y (el_dtanh2_out), a smaller
// one changes H by less than 1e-35.
constexpr float kElCap = 5e37f, kElTiny = 1e-37f;
__device__ __forceinline__ float el_cache(float y) {
  const float e = expf(2.f * y);
  return e > kElCap ? kElCap : e;  // (not fminf: what is not a number stays one)
}
__device__ __forceinline__ bool el_cached(float E) { return E >= kElTiny && E < kElCap; }
// Four features' cache entries at U, and their Y at U + to_y where one of them needs it (true then).
__device__ __forceinline__ bool el_store_cache(float* U, size_t to_y, float y0, float y1, float y2, float y3) {
  const float4 e = make_float4(el_cache(y0), el_cache(y1), el_cache(y2), el_cache(y3));
  *reinterpret_cast<float4*>(U) = e;
  if (el_cached(e.x) && el_cached(e.y) && el_cached(e.z) && el_cached(e.w)) return false;
  *reinterpret_cast<float4*>(U + to_y) = make_float4(y0, y1, y2, y3);
  return true;
}

// The packed constants of el_dtanh2 and of the operand split.  Made by volatile assembly so
// that they stay in registers: left to itself the compiler builds each of them anew, two
// moves a use, which was a quarter of a tile's instructions.
struct ElConst {
  uint64_t c63, c7, c15th, c28, half, m1;
};
__device__ __forceinline__ uint64_t el_keep(float a) {
  uint64_t r;
  asm volatile("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}

// dH = tanh(Y + x) - tanh(Y) = t (1 - H^2)/(1 + H t), t = tanh(x), for |x| <= 1.  tanh is the
// fifth convergent of Lambert's continued fraction (relative error below 1e-7 at |x| = 1),
// t = w/Q with z = x^2, w = x (63 + 7 z + z^2/15), Q = 63 + 28 z + z^2, which needs no
// division of its own: with c = (1 + E)/2, dH = E w / (c (Q c + w (c - 1))).
__device__ __forceinline__ uint64_t el_dtanh2(const ElConst& k, uint64_t x, uint64_t E) {
  const uint64_t z = f2_mul(x, x);
  const uint64_t w = f2_mul(x, f2_fma(z, f2_fma(z, k.c15th, k.c7), k.c63));
  const uint64_t Q = f2_fma(z, f2_add(z, k.c28), k.c63);
  const uint64_t c = f2_fma(E, k.half, k.half);
  const uint64_t den = f2_mul(c, f2_fma(w, f2_add(c, k.m1), f2_mul(Q, c)));
  float d0, d1, r0, r1;
  f2_unpack(den, d0, d1);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(d0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(d1));
  return f2_mul(E, f2_mul(w, f2_pack(r0, r1)));  // (den overflows from E = 1e18 on: r = 0, as dH is there)
}
// The same for |x| > 1: with X = exp(-2 |x|), dH = 2 E/(1 + E) (1 - X)/(X + E) for x > 0 and
// -2 E/(1 + E) (1 - X)/(1 + E X) for x < 0, in which nothing cancels or overflows, whichever way
// the unit swings (E within the cached range).
__device__ __forceinline__ float el_dtanh_far(float x, float E) {
  const float X = expf(-2.f * fabsf(x));
  float r0, r1;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(1.f + E));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(x > 0.f ? X + E : fmaf(E, X, 1.f)));
  return copysignf(2.f * (E * r0) * ((1.f - X) * r1), x);
}
__device__ __forceinline__ uint64_t el_dtanh2_far(const ElConst& k, uint64_t x, uint64_t E) {
  float x0, x1, e0, e1, d0, d1;
  f2_unpack(el_dtanh2(k, x, E), d0, d1);
  f2_unpack(x, x0, x1);
  f2_unpack(E, e0, e1);
  return f2_pack(fabsf(x0) > 1.f ? el_dtanh_far(x0, e0) : d0, fabsf(x1) > 1.f ? el_dtanh_far(x1, e1) : d1);
}
// And outside the cached range, where tanh Y = sgn Y = +-1: dH = -2 sgn Y/(1 + exp(2 sgn Y (Y + x))).
__device__ __forceinline__ float el_dtanh_out(float x, float y) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.f + expf(2.f * copysignf(1.f, y) * (y + x))));
  return copysignf(2.f, -y) * r;
}
// el_dtanh2_far's d, put right where a unit of the pair is out of range (its Y at py).
__device__ __forceinline__ uint64_t el_dtanh2_out(uint64_t d, uint64_t x, uint64_t E, const float* py) {
  float x0, x1, e0, e1, d0, d1;
  f2_unpack(d, d0, d1);
  f2_unpack(x, x0, x1);
  f2_unpack(E, e0, e1);
  if (fabsf(x0) > 1.f && !el_cached(e0)) d0 = el_dtanh_out(x0, py[0]);
  if (fabsf(x1) > 1.f && !el_cached(e1)) d1 = el_dtanh_out(x1, py[1]);
  return f2_pack(d0, d1);
}

template <int FC>
struct ElCtx {
  const ElArgs* a;
  const uint4* Wf;
  const float *bias, *emb, *wr, *br, *av, *z0;
  int8_t* spin;
  uint16_t* list;
  const int* rp;
  const float* wf;
  const uint16_t* col;
  ElConst k;
  // 1: some unit of the configuration is out of the cache's range (in shared memory; as a value it was
  // a register of the whole tile and 7 % of a local energy on a random graph of 77 sites, F 32)
  int* out;
};

// Forward of the configuration in c.spin: Y^1..Y^L into the cache, H^L left in the row
// buffer that is returned when want_h.  X = [A_hat H ; H] as hi + lo operands, FP32 rows, in
// the order of the forward call's kernel (bit-identical log Psi).
template <int FC>
__device__ const float* el_forward_x2(const ElCtx<FC>& c, float* U, float* Hb, bool want_h) {
  constexpr int F = 16 * FC, LDH = el_ldh(F), LDU = el_ldu(F);
  const int N = c.a->m.N, L = c.a->m.L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  float* Hp = Hb;
  float* Hn = Hb + (size_t)N * LDH;
  for (int i = threadIdx.x; i < N * (F / 4); i += kElThreads) {
    const int v = i / (F / 4), f = (i % (F / 4)) * 4;
    *reinterpret_cast<float4*>(Hp + (size_t)v * LDH + f) =
        *reinterpret_cast<const float4*>(c.emb + (c.spin[v] > 0 ? 0 : F) + f);
  }
  __syncthreads();
  for (int l = 1; l <= L; ++l) {
    for (int t = warp; t * 16 < N; t += kElWarps) {
      uint32_t hi[2 * FC][4], lo[2 * FC][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v = min(16 * t + g + 8 * h, N - 1);
        float acc[FC][4];
#pragma unroll
        for (int k = 0; k < FC; ++k) acc[k][0] = acc[k][1] = acc[k][2] = acc[k][3] = 0.f;
        for (int k = c.rp[v]; k < c.rp[v + 1]; ++k) {
          const float w = c.wf[k];
          const float* x = Hp + (size_t)c.col[k] * LDH + 4 * q;
#pragma unroll
          for (int cc = 0; cc < FC; ++cc) {
            const float4 y = *reinterpret_cast<const float4*>(x + 16 * cc);
            acc[cc][0] = fmaf(w, y.x, acc[cc][0]);
            acc[cc][1] = fmaf(w, y.y, acc[cc][1]);
            acc[cc][2] = fmaf(w, y.z, acc[cc][2]);
            acc[cc][3] = fmaf(w, y.w, acc[cc][3]);
          }
        }
        const float* self = Hp + (size_t)v * LDH + 4 * q;
#pragma unroll
        for (int cc = 0; cc < FC; ++cc) {
          split2(c.k.m1, acc[cc][0], acc[cc][1], hi[cc][h], lo[cc][h]);
          split2(c.k.m1, acc[cc][2], acc[cc][3], hi[cc][2 + h], lo[cc][2 + h]);
          const float4 y = *reinterpret_cast<const float4*>(self + 16 * cc);
          split2(c.k.m1, y.x, y.y, hi[FC + cc][h], lo[FC + cc][h]);
          split2(c.k.m1, y.z, y.w, hi[FC + cc][2 + h], lo[FC + cc][2 + h]);
        }
      }
#pragma unroll
      for (int co = 0; co < FC; ++co) {
        float D[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
#pragma unroll
        for (int kc = 0; kc < 2 * FC; ++kc) {
          const uint4 b = c.Wf[(kc * FC + co) * 32 + lane];
          mma_16816(D[0], hi[kc], b.x, b.y);
          mma_16816(D[1], hi[kc], b.z, b.w);
        }
#pragma unroll
        for (int kc = 0; kc < 2 * FC; ++kc) {
          const uint4 b = c.Wf[(kc * FC + co) * 32 + lane];
          mma_16816(D[0], lo[kc], b.x, b.y);
          mma_16816(D[1], lo[kc], b.z, b.w);
        }
        const float4 bs = *reinterpret_cast<const float4*>(c.bias + 16 * co + 4 * q);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int v = 16 * t + g + 8 * h;
          if (v >= N) continue;
          const float y0 = D[0][2 * h] + bs.x, y1 = D[0][2 * h + 1] + bs.y;
          const float y2 = D[1][2 * h] + bs.z, y3 = D[1][2 * h + 1] + bs.w;
          float* u = U + ((size_t)(l - 1) * N + v) * LDU + 16 * co + 4 * q;
          if (el_store_cache(u, (size_t)L * N * LDU, y0, y1, y2, y3)) *c.out = 1;
          if (l < L || want_h)
            *reinterpret_cast<float4*>(Hn + (size_t)v * LDH + 16 * co + 4 * q) =
                make_float4(tanhf(y0), tanhf(y1), tanhf(y2), tanhf(y3));
        }
      }
    }
    __syncthreads();
    float* t2 = Hp;
    Hp = Hn;
    Hn = t2;
  }
  return Hp;
}

// Row-wise ReLU + layer norm of a tile row's values (FC x 4 in each of four lanes), in place:
// (r - mean r)/sqrt(var r + 1e-6), r = max(y, 0).
template <int FC>
__device__ __forceinline__ void el_relu_ln(float (*y)[4]) {
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < FC; ++c)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      y[c][i] = fmaxf(y[c][i], 0.f);
      s += y[c][i];
    }
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  const float mu = s * (1.f / (16 * FC));
  float v = 0.f;
#pragma unroll
  for (int c = 0; c < FC; ++c)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      y[c][i] -= mu;
      v = fmaf(y[c][i], y[c][i], v);
    }
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  const float inv = 1.f / sqrtf(fmaf(v, 1.f / (16 * FC), 1e-6f));
#pragma unroll
  for (int c = 0; c < FC; ++c)
#pragma unroll
    for (int i = 0; i < 4; ++i) y[c][i] *= inv;
}

// Products with a W of three terms (FP32 models), in two steps.  The tensor cores truncate a sum
// where FP32 arithmetic rounds it, so a long chain drifts: the five small products of every K step
// come first, in one chain (D), then each large one, hi x W's first term, from zero and added with
// rounding.  D[2 i], D[2 i + 1]: column tiles of output chunk i.
template <int FC>
__device__ __forceinline__ void el_mma_small(float (*D)[4], const uint32_t* hi, const uint32_t* mid, const uint32_t* lo,
                                             const uint4* Wf, int at, bool first) {
  const int lane = threadIdx.x & 31;
  const uint4 w2 = Wf[(2 * 2 * FC * FC + at) * 32 + lane];
  if (first) {
    mma_16816_first(D[0], hi, w2.x, w2.y);
    mma_16816_first(D[1], hi, w2.z, w2.w);
  } else {
    mma_16816(D[0], hi, w2.x, w2.y);
    mma_16816(D[1], hi, w2.z, w2.w);
  }
  const uint4 w1 = Wf[(2 * FC * FC + at) * 32 + lane];
  mma_16816(D[0], mid, w1.x, w1.y);
  mma_16816(D[1], mid, w1.z, w1.w);
  const uint4 w0 = Wf[at * 32 + lane];
  mma_16816(D[0], lo, w0.x, w0.y);
  mma_16816(D[1], lo, w0.z, w0.w);
  mma_16816(D[0], hi, w1.x, w1.y);
  mma_16816(D[1], hi, w1.z, w1.w);
  mma_16816(D[0], mid, w0.x, w0.y);
  mma_16816(D[1], mid, w0.z, w0.w);
}
template <int FC>
__device__ __forceinline__ void el_mma_large(float (*D)[4], const uint32_t* hi, const uint4* Wf, int at) {
  const uint4 w0 = Wf[at * 32 + (threadIdx.x & 31)];
  float T[2][4];
  mma_16816_first(T[0], hi, w0.x, w0.y);
  mma_16816_first(T[1], hi, w0.z, w0.w);
#pragma unroll
  for (int i = 0; i < 8; ++i) D[i / 4][i % 4] += T[i / 4][i % 4];
}

// Forward of an FP32 model: the cache of every layer (exp(2 Y), or Y and H with layer norm).
template <int FC, int MODE>
__device__ void el_forward_f32(const ElCtx<FC>& c, float* U, float* Hb) {
  constexpr int F = 16 * FC, LDH = el_ldh(F), LDU = el_ldu(F);
  const int N = c.a->m.N, L = c.a->m.L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  float* Hp = Hb;
  float* Hn = Hb + (size_t)N * LDH;
  float* Hc = U + (size_t)L * N * LDU;  // layer norm only
  for (int i = threadIdx.x; i < N * (F / 4); i += kElThreads) {
    const int v = i / (F / 4), f = (i % (F / 4)) * 4;
    *reinterpret_cast<float4*>(Hp + (size_t)v * LDH + f) =
        *reinterpret_cast<const float4*>(c.emb + (c.spin[v] > 0 ? 0 : F) + f);
  }
  __syncthreads();
  for (int l = 1; l <= L; ++l) {
    for (int t = warp; t * 16 < N; t += kElWarps) {
      float acc[2][FC][4];
      const float* self[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v = min(16 * t + g + 8 * h, N - 1);
        self[h] = Hp + (size_t)v * LDH + 4 * q;
#pragma unroll
        for (int k = 0; k < FC; ++k) acc[h][k][0] = acc[h][k][1] = acc[h][k][2] = acc[h][k][3] = 0.f;
        for (int k = c.rp[v]; k < c.rp[v + 1]; ++k) {
          const float w = c.wf[k];
          const float* x = Hp + (size_t)c.col[k] * LDH + 4 * q;
#pragma unroll
          for (int cc = 0; cc < FC; ++cc) {
            const float4 y = *reinterpret_cast<const float4*>(x + 16 * cc);
            acc[h][cc][0] = fmaf(w, y.x, acc[h][cc][0]);
            acc[h][cc][1] = fmaf(w, y.y, acc[h][cc][1]);
            acc[h][cc][2] = fmaf(w, y.z, acc[h][cc][2]);
            acc[h][cc][3] = fmaf(w, y.w, acc[h][cc][3]);
          }
        }
      }
      float D[2 * FC][4];
#pragma unroll
      for (int step = 0; step < 4 * FC; ++step) {  // the small products of all K steps, then the large ones
        const int kc = step % (2 * FC);
        uint32_t hi[4], mid[4], lo[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 s = kc < FC ? make_float4(acc[h][kc % FC][0], acc[h][kc % FC][1], acc[h][kc % FC][2], acc[h][kc % FC][3])
                                   : *reinterpret_cast<const float4*>(self[h] + 16 * (kc % FC));
          split3(c.k.m1, s.x, s.y, hi[h], mid[h], lo[h]);
          split3(c.k.m1, s.z, s.w, hi[2 + h], mid[2 + h], lo[2 + h]);
        }
#pragma unroll
        for (int co = 0; co < FC; ++co) {
          if (step < 2 * FC)
            el_mma_small<FC>(D + 2 * co, hi, mid, lo, c.Wf, kc * FC + co, kc == 0);
          else
            el_mma_large<FC>(D + 2 * co, hi, c.Wf, kc * FC + co);
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v = 16 * t + g + 8 * h;
        float y[FC][4];
#pragma unroll
        for (int co = 0; co < FC; ++co) {
          const float4 bs = *reinterpret_cast<const float4*>(c.bias + 16 * co + 4 * q);
          y[co][0] = D[2 * co][2 * h] + bs.x;
          y[co][1] = D[2 * co][2 * h + 1] + bs.y;
          y[co][2] = D[2 * co + 1][2 * h] + bs.z;
          y[co][3] = D[2 * co + 1][2 * h + 1] + bs.w;
          float* u = U + ((size_t)(l - 1) * N + v) * LDU + 16 * co + 4 * q;
          if (v < N && MODE == EL_F32_LN)
            *reinterpret_cast<float4*>(u) = make_float4(y[co][0], y[co][1], y[co][2], y[co][3]);
          else if (v < N && el_store_cache(u, (size_t)L * N * LDU, y[co][0], y[co][1], y[co][2], y[co][3]))
            *c.out = 1;
        }
        if (MODE == EL_F32_LN) el_relu_ln<FC>(y);  // (shuffles: every lane)
        if (v < N)
#pragma unroll
          for (int co = 0; co < FC; ++co) {
            const float4 hv = MODE == EL_F32_LN ? make_float4(y[co][0], y[co][1], y[co][2], y[co][3])
                                                : make_float4(tanhf(y[co][0]), tanhf(y[co][1]), tanhf(y[co][2]), tanhf(y[co][3]));
            if (MODE == EL_F32_LN) *reinterpret_cast<float4*>(Hc + ((size_t)(l - 1) * N + v) * LDU + 16 * co + 4 * q) = hv;
            if (l < L) *reinterpret_cast<float4*>(Hn + (size_t)v * LDH + 16 * co + 4 * q) = hv;
          }
      }
    }
    __syncthreads();
    float* t2 = Hp;
    Hp = Hn;
    Hn = t2;
  }
}

// Shared memory by byte offset (the offsets select between buffers at run time; addressed
// from the array itself every access is a shared-memory one with 32-bit arithmetic).
extern __shared__ __align__(128) unsigned char el_smem[];
template <typename T>
__device__ __forceinline__ const T& el_sh(uint32_t off) {
  return *reinterpret_cast<const T*>(el_smem + off);
}
template <typename T>
__device__ __forceinline__ T& el_shw(uint32_t off) {
  return *reinterpret_cast<T*>(el_smem + off);
}

// Byte offset of row p of a Z buffer, and of its chunk c (16 floats).  A row is Z[:F] then
// Z[F:], with neighbouring chunks of odd rows exchanged: two rows that share a quarter of a
// 16-byte load then lie in different halves of the banks unless their positions have the same
// parity.  The staged positions are s = 4 p + (p & 1), which is the row's offset in units of 64
// bytes at F = 32.
template <int FC>
__device__ __forceinline__ uint32_t el_zrow(uint32_t p) {
  return p * (128 * FC) + (p & 1u) * 64;
}
template <int FC>
__device__ __forceinline__ uint32_t el_zpos(uint32_t s) {
  return FC == 2 ? s * 64 : (s >> 2) * (128 * FC) + (s & 1u) * 64;
}
__device__ __forceinline__ uint32_t el_zchunk(uint32_t row, int c) { return (c & 1 ? row ^ 64u : row) + (c & ~1) * 64; }

__device__ __forceinline__ float el_max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// One tile of 16 rows of a bond's ball_l: rows 16 t + g and + 8.
//   zin: Z of the sp rows of ball_{l-1}, then a zero row, which stands for every row outside
//   the ball; zout: Z of the n rows of ball_l for the next layer; Ul: the layer's cache (to_h
//   floats on: its H with layer norm, else Y of the units out of the cache's range).
// The stages are kept apart (look-ups, gather, difference, product), each a block without
// branches over all of the thread's values: a warp hides most of its own latency that way.
template <int FC, int NP, int MODE, bool LAST>
__device__ __forceinline__ void el_tile(const ElCtx<FC>& c, uint32_t rec, uint32_t pairs, int t, int n, int sp,
                                        uint32_t zin, uint32_t zout, const float* Ul, size_t to_h, float& sre, float& sim) {
  constexpr int F = 16 * FC, LDU = el_ldu(F);
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const uint32_t sp2 = (uint32_t)(4 * sp + (sp & 1)) * 0x10001u, zq = zin + 16 * q;
  const int row0 = 16 * t + g;
  // look-ups
  // (rows past the ball's last one find an earlier bond's entries: their results are dropped)
  uint32_t pp[2], zrow[2];
  int np[2];
  float av[2];
  const float* ur[2];
  const uint32_t zr0 = row0 * (128 * FC) + (g & 1) * 64;  // el_zrow(row0); row0 + 8 has the same parity
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int row = row0 + 8 * h;
    const int2 rc = el_sh<int2>(rec + row * 8);
    const int v = rc.x & 0xFFFF;
    np[h] = rc.x >> 16;
    pp[h] = pairs + (NP > 0 ? NP * row : rc.y) * 4;
    zrow[h] = zq + (row < sp ? zr0 + h * (1024 * FC) : el_zrow<FC>(sp));
    av[h] = c.av[v];
    ur[h] = Ul + v * LDU + 4 * q;
  }
  // gather
  uint64_t x[2][FC][2];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int cc = 0; cc < FC; ++cc) x[h][cc][0] = x[h][cc][1] = 0;
  auto add_pair = [&](int h, uint32_t w) {
    const uint32_t p = __vminu2(w, sp2);
    const uint32_t z0 = zq + el_zpos<FC>(p & 0xFFFFu), z1 = zq + el_zpos<FC>(p >> 16);
#pragma unroll
    for (int cc = 0; cc < FC; ++cc) {
      const ulonglong2 y0 = el_sh<ulonglong2>(el_zchunk(z0, cc)), y1 = el_sh<ulonglong2>(el_zchunk(z1, cc));
      x[h][cc][0] = f2_add(x[h][cc][0], f2_add(y0.x, y1.x));
      x[h][cc][1] = f2_add(x[h][cc][1], f2_add(y0.y, y1.y));
    }
  };
  if (NP > 0) {
#pragma unroll
    for (int j = 0; j < NP; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) add_pair(h, el_sh<uint32_t>(pp[h] + 4 * j));
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll 1
      for (int j = 0; j < np[h]; ++j) add_pair(h, el_sh<uint32_t>(pp[h] + 4 * j));
  }
  float zmax = 0.f;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int cc = 0; cc < FC; ++cc) {
      const ulonglong2 y = el_sh<ulonglong2>(el_zchunk(zrow[h], FC + cc));
      x[h][cc][0] = f2_fma(f2_dup(av[h]), x[h][cc][0], y.x);
      x[h][cc][1] = f2_fma(f2_dup(av[h]), x[h][cc][1], y.y);
      float x0, x1, x2, x3;
      f2_unpack(x[h][cc][0], x0, x1);
      f2_unpack(x[h][cc][1], x2, x3);
      zmax = el_max3(el_max3(zmax, fabsf(x0), fabsf(x1)), fabsf(x2), fabsf(x3));
    }
  // dH in place of x (what is not a number stays one)
  if (MODE == EL_F32_LN) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float y[FC][4];
#pragma unroll
      for (int cc = 0; cc < FC; ++cc) {
        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(ur[h] + 16 * cc);
        f2_unpack(f2_add(x[h][cc][0], e.x), y[cc][0], y[cc][1]);
        f2_unpack(f2_add(x[h][cc][1], e.y), y[cc][2], y[cc][3]);
      }
      el_relu_ln<FC>(y);
#pragma unroll
      for (int cc = 0; cc < FC; ++cc) {
        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(ur[h] + to_h + 16 * cc);
        x[h][cc][0] = f2_fma(e.x, c.k.m1, f2_pack(y[cc][0], y[cc][1]));
        x[h][cc][1] = f2_fma(e.y, c.k.m1, f2_pack(y[cc][2], y[cc][3]));
      }
    }
  } else if (!__any_sync(0xffffffffu, zmax > 1.f)) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int cc = 0; cc < FC; ++cc) {
        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(ur[h] + 16 * cc);
        x[h][cc][0] = el_dtanh2(c.k, x[h][cc][0], e.x);
        x[h][cc][1] = el_dtanh2(c.k, x[h][cc][1], e.y);
      }
  } else {  // some unit of the tile swings further than the series reaches
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int cc = 0; cc < FC; ++cc) {
        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(ur[h] + 16 * cc);
        uint64_t d0 = el_dtanh2_far(c.k, x[h][cc][0], e.x), d1 = el_dtanh2_far(c.k, x[h][cc][1], e.y);
        if (*c.out) {
          d0 = el_dtanh2_out(d0, x[h][cc][0], e.x, ur[h] + to_h + 16 * cc);
          d1 = el_dtanh2_out(d1, x[h][cc][1], e.y, ur[h] + to_h + 16 * cc + 2);
        }
        x[h][cc][0] = d0;
        x[h][cc][1] = d1;
      }
  }
  const bool ok0 = row0 < n, ok1 = row0 + 8 < n;
  if (LAST) {  // this thread's part of Delta = sum_v dH_v . w_r
    float pre[2] = {0.f, 0.f}, pim[2] = {0.f, 0.f};
#pragma unroll
    for (int cc = 0; cc < FC; ++cc) {
      const float4* w = reinterpret_cast<const float4*>(c.wr + 2 * (16 * cc + 4 * q));
      const float4 wa = w[0], wb = w[1];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float d0, d1, d2, d3;
        f2_unpack(x[h][cc][0], d0, d1);
        f2_unpack(x[h][cc][1], d2, d3);
        pre[h] += d0 * wa.x + d1 * wa.z + d2 * wb.x + d3 * wb.z;
        pim[h] += d0 * wa.y + d1 * wa.w + d2 * wb.y + d3 * wb.w;
      }
    }
    sre += (ok0 ? pre[0] : 0.f) + (ok1 ? pre[1] : 0.f);
    sim += (ok0 ? pim[0] : 0.f) + (ok1 ? pim[1] : 0.f);
    return;
  }
  // product: dH in three BF16 parts, so that its rounding adds nothing to the FP32 rows (two
  // parts, as the forward has, left errors 1.4 times those of splitting the gathered rows)
  uint32_t hi[FC][4], mid[FC][4], lo[FC][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int cc = 0; cc < FC; ++cc) {
      float d0, d1, d2, d3;
      f2_unpack(x[h][cc][0], d0, d1);
      f2_unpack(x[h][cc][1], d2, d3);
      split3(c.k.m1, d0, d1, hi[cc][h], mid[cc][h], lo[cc][h]);
      split3(c.k.m1, d2, d3, hi[cc][2 + h], mid[cc][2 + h], lo[cc][2 + h]);
    }
  const uint32_t o0 = zout + 16 * q + zr0, o1 = o0 + 1024 * FC;
  // output chunks j < FC are Z[:F] (message, scaled by a_u), the others Z[F:] (self); two at a
  // time, so that four chains of products overlap
#pragma unroll
  for (int j = 0; j < 2 * FC; j += 2) {
    float D[4][4];
    if (MODE == EL_X2) {
#pragma unroll
      for (int kc = 0; kc < FC; ++kc) {
        const uint4 b0 = c.Wf[((j / FC * FC + kc) * FC + j % FC) * 32 + lane];
        const uint4 b1 = c.Wf[(((j + 1) / FC * FC + kc) * FC + (j + 1) % FC) * 32 + lane];
        const uint32_t* terms[3] = {lo[kc], mid[kc], hi[kc]};
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          if (kc == 0 && x == 0) {
            mma_16816_first(D[0], terms[x], b0.x, b0.y);
            mma_16816_first(D[1], terms[x], b0.z, b0.w);
            mma_16816_first(D[2], terms[x], b1.x, b1.y);
            mma_16816_first(D[3], terms[x], b1.z, b1.w);
          } else {
            mma_16816(D[0], terms[x], b0.x, b0.y);
            mma_16816(D[1], terms[x], b0.z, b0.w);
            mma_16816(D[2], terms[x], b1.x, b1.y);
            mma_16816(D[3], terms[x], b1.z, b1.w);
          }
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int o = ((j + i) / FC * FC) * FC + (j + i) % FC;
#pragma unroll
        for (int kc = 0; kc < FC; ++kc) el_mma_small<FC>(D + 2 * i, hi[kc], mid[kc], lo[kc], c.Wf, o + kc * FC, kc == 0);
#pragma unroll
        for (int kc = 0; kc < FC; ++kc) el_mma_large<FC>(D + 2 * i, hi[kc], c.Wf, o + kc * FC);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float(*d)[4] = D + 2 * i;
      ulonglong2 y0 = make_ulonglong2(f2_pack(d[0][0], d[0][1]), f2_pack(d[1][0], d[1][1]));
      ulonglong2 y1 = make_ulonglong2(f2_pack(d[0][2], d[0][3]), f2_pack(d[1][2], d[1][3]));
      if (j + i < FC) {
        y0 = make_ulonglong2(f2_mul(y0.x, f2_dup(av[0])), f2_mul(y0.y, f2_dup(av[0])));
        y1 = make_ulonglong2(f2_mul(y1.x, f2_dup(av[1])), f2_mul(y1.y, f2_dup(av[1])));
      }
      if (ok0) el_shw<ulonglong2>(el_zchunk(o0, j + i)) = y0;
      if (ok1) el_shw<ulonglong2>(el_zchunk(o1, j + i)) = y1;
    }
  }
}

template <int FC, int NP, int MODE>
__global__ void __launch_bounds__(kElThreads, 1) k_eloc(const __grid_constant__ ElArgs a) {
  unsigned char* const smem = el_smem;
  __shared__ int s_cnt[kElWarps], s_out;
  __shared__ double s_diag[kElWarps], s_e[2 * kElWarps];
  constexpr int F = 16 * FC, LDH = el_ldh(F), LDU = el_ldu(F);
  const int N = a.m.N, L = a.m.L, E = a.m.E;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  ElCtx<FC> c;
  c.a = &a;
  c.Wf = (const uint4*)(smem + a.oW);
  c.bias = (const float*)(smem + a.obias);
  c.emb = (const float*)(smem + a.oemb);
  c.wr = (const float*)(smem + a.owr);
  c.br = (const float*)(smem + a.obr);
  c.av = (const float*)(smem + a.oav);
  c.z0 = (const float*)(smem + a.oz0);
  c.spin = (int8_t*)(smem + a.ospin);
  c.list = (uint16_t*)(smem + a.olist);
  c.rp = (const int*)(smem + a.orp);
  c.wf = (const float*)(smem + a.owf);
  c.col = (const uint16_t*)(smem + a.ocol);
  c.out = &s_out;
  c.k = {el_keep(63.f), el_keep(7.f), el_keep(1.f / 15.f), el_keep(28.f), el_keep(0.5f), el_keep(-1.f)};
  float* red = (float*)(smem + a.ored);
  const float* th = a.theta;
  const float* W = th + a.m.oW;
  // parameters and graph: once per CTA
  for (int i = tid; i < el_wterms(MODE) * 2 * FC * FC * 32; i += kElThreads)
    ((uint4*)c.Wf)[i] = make_wfrag<FC, MODE == EL_F32>(W, (i / (FC * 32)) % (2 * FC), (i / 32) % FC, i & 31, i / (2 * FC * FC * 32));
  for (int i = tid; i < F; i += kElThreads) ((float*)c.bias)[i] = th[a.m.ob + i];
  if (MODE != EL_F32_LN) {
    for (int i = tid; i < 2 * F; i += kElThreads) ((float*)c.emb)[i] = tanhf(th[a.m.oWe + i] + th[a.m.obe + i % F]);
  } else if (warp < 2) {  // one embedding row per warp, 4 FC features in each of its first four lanes (and copies)
    float y[FC][4];
#pragma unroll
    for (int cc = 0; cc < FC; ++cc)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int f = 16 * cc + 4 * (lane & 3) + i;
        y[cc][i] = th[a.m.oWe + warp * F + f] + th[a.m.obe + f];
      }
    el_relu_ln<FC>(y);
    if (lane < 4)
#pragma unroll
      for (int cc = 0; cc < FC; ++cc)
#pragma unroll
        for (int i = 0; i < 4; ++i) ((float*)c.emb)[warp * F + 16 * cc + 4 * lane + i] = y[cc][i];
  }
  for (int i = tid; i < (F + 2) * 2; i += kElThreads) ((float*)c.wr)[i] = th[a.m.owr + i];
  if (tid < 2) ((float*)c.br)[tid] = th[a.m.obr + tid];
  for (uint32_t i = tid; i < a.units * a.tab_bytes / 16; i += kElThreads) el_shw<uint4>(a.otab + 16 * i) = make_uint4(0, 0, 0, 0);
  __syncthreads();
  for (int v = tid; v < N; v += kElThreads) {
    const int d = __ldg(a.g.row_ptr + v + 1) - __ldg(a.g.row_ptr + v);
    // FP32: rounded once, as the forward's weights are; the BF16X2 operands (2^-16) do not see its last bit
    ((float*)c.av)[v] = d > 0 ? (MODE == EL_X2 ? 1.f / sqrtf((float)d) : (float)(1.0 / sqrt((double)d))) : 0.f;
  }
  // Z^0 of a row that changes from up to down: (emb(-1) - emb(+1)) [W[:F] | W[F:]]
  for (int i = tid; i < 2 * F; i += kElThreads) {
    const int f = i % F, top = i < F ? 0 : F;
    float z = 0.f;
    for (int k = 0; k < F; ++k) {
      const float w = MODE == EL_F32 ? finite_w(W[(size_t)(top + k) * F + f]) : W[(size_t)(top + k) * F + f];
      z = fmaf(c.emb[F + k] - c.emb[k], MODE == EL_X2 ? __bfloat162float(__float2bfloat16_rn(w)) : w, z);
    }
    ((float*)c.z0)[i] = z;
  }
  const size_t to_h = (size_t)L * N * LDU;
  float* U = a.gU + (size_t)blockIdx.x * to_h * 2;
  float* Hb = a.h_smem ? (float*)(smem + a.oH) : a.gH + (size_t)blockIdx.x * 2 * N * LDH;

  // this thread's unit
  const int uthreads = a.uw * 32, h = warp / a.uw, uwarp = warp % a.uw, utid = tid - h * uthreads;
  const bool active = h < a.units;
  const uint32_t uo = a.ounit + (uint32_t)(active ? h : 0) * a.unit_bytes;
  const uint32_t ut = a.otab + (uint32_t)(active ? h : 0) * a.tab_bytes;
  auto unit_sync = [&]() {
    if (a.uw == 1)
      __syncwarp();
    else
      el_bar(1 + h, uthreads);
  };
  __syncthreads();

  for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) {
    for (int v = tid; v < N; v += kElThreads) c.spin[v] = a.spins[b * N + v];
    // the forward's adjacency, over the units' space
    for (int v = tid; v <= N; v += kElThreads) ((int*)c.rp)[v] = __ldg(a.g.row_ptr + v);
    for (int i = tid; i < 2 * E; i += kElThreads) {
      ((float*)c.wf)[i] = __ldg(a.g.wf + i);
      ((uint16_t*)c.col)[i] = (uint16_t)__ldg(a.g.col + i);
    }
    if (a.dlogpsi)
      for (int e = tid; e < E; e += kElThreads) a.dlogpsi[b * E + e] = 0.f;
    if (tid == 0) s_out = 0;
    __syncthreads();
    const float* HL = nullptr;
    if (MODE == EL_X2)
      HL = el_forward_x2<FC>(c, U, Hb, a.logpsi != nullptr);
    else
      el_forward_f32<FC, MODE>(c, U, Hb);
    if (MODE == EL_X2 && a.logpsi) {
      // the readout in the order of the forward call: kReadout / F interleaved site strides
      const int parts = kReadout / F, f = tid % F, p = tid / F;
      if (p < parts) {
        float acc = 0.f;
        for (int v = p; v < N; v += parts) acc += HL[(size_t)v * LDH + f];
        red[p * F + f] = acc;
      }
      __syncthreads();
      if (warp == 0) {
        float re = 0.f, im = 0.f;
        for (int ff = lane; ff < F; ff += 32) {
          float s = 0.f;
          for (int pp = 0; pp < parts; ++pp) s += red[pp * F + ff];
          re += s * c.wr[2 * ff];
          im += s * c.wr[2 * ff + 1];
        }
        re = warp_sum_f(re);
        im = warp_sum_f(im);
        int up = 0;
        for (int v = lane; v < N; v += 32) up += c.spin[v] > 0;
        up = warp_sum_f(up);
        if (lane == 0) {
          const int dn = N - up;
          a.logpsi[2 * b] = (double)(re + (float)up * c.wr[2 * F] + (float)dn * c.wr[2 * (F + 1)] + c.br[0]);
          a.logpsi[2 * b + 1] = (double)(im + (float)up * c.wr[2 * F + 1] + (float)dn * c.wr[2 * (F + 1) + 1] + c.br[1]);
        }
      }
    }
    // antiparallel bonds (in order) and the diagonal energy, 512 bonds at a time
    double diag = 0.0;
    int na = 0;
    for (int base = 0; base < E; base += kElThreads) {
      const int e = base + tid;
      bool anti = false;
      if (e < E) {
        const int2 ij = __ldg(reinterpret_cast<const int2*>(a.g.edges) + e);
        const int si = c.spin[ij.x], sj = c.spin[ij.y];
        anti = si != sj;
        diag += bond_diag(a.g, e, si, sj);
      }
      const unsigned mask = __ballot_sync(0xffffffffu, anti);
      if (lane == 0) s_cnt[warp] = __popc(mask);
      __syncthreads();
      int before = na, all = na;
      for (int w = 0; w < kElWarps; ++w) {
        const int x = s_cnt[w];
        before += w < warp ? x : 0;
        all += x;
      }
      if (anti) c.list[before + __popc(mask & ((1u << lane) - 1u))] = (uint16_t)e;
      na = all;
      __syncthreads();
    }
    diag = warp_sum_f(diag);
    if (lane == 0) s_diag[warp] = diag;
    // the units' shares of the bonds (equal up to one), a bond at a time
    double er = 0.0, ei = 0.0;  // lane 0 of a unit's first warp: the terms of its bonds
    if (active) {
      const int b_lo = (int)((int64_t)na * h / a.units), b_hi = (int)((int64_t)na * (h + 1) / a.units);
      // lane i holds int i of a bond's record (DevGraph::bond_info); every warp its own
      auto load_info = [&](int i) { return i < b_hi ? __ldg(a.g.bond_info + c.list[i] * 32 + lane) : 0; };
      auto field = [&](int x, int i) { return __shfl_sync(0xffffffffu, x, i); };
      auto stage = [&](int info, int buf) {  // the rows and neighbour pairs of a bond
        const int rows2 = (field(info, 8 + L) + 1) / 2, pairs4 = (field(info, 16 + L) + 3) / 4;
        const int* gr = a.g.rec + 2 * (size_t)field(info, 0);
        const uint32_t* gp = a.g.pairs + field(info, 1);
        for (int i = utid; i < rows2; i += uthreads) cp_async16(smem + ut + a.urec[buf] + 16 * i, gr + 4 * i);
        for (int i = utid; i < pairs4; i += uthreads) cp_async16(smem + ut + a.upair[buf] + 16 * i, gp + 4 * i);
      };
      int cur = load_info(b_lo), nxt = load_info(b_lo + 1);
      if (b_lo < b_hi) stage(cur, 0);
      for (int i = b_lo; i < b_hi; ++i) {
        const int buf = a.nbuf == 2 ? (i - b_lo) & 1 : 0;
        cp_async_wait_all();
        const int cur_i = field(cur, 4), cur_j = field(cur, 5);
        // Z^0: rows i and j of the bond, then the zero row
        for (int k = utid; k < 3 * (F / 2); k += uthreads) {
          const int r = k / (F / 2), ch = (k % (F / 2)) / 4, f = (k % (F / 2)) * 4;
          float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
          if (r < 2) {
            const int v = r ? cur_j : cur_i;
            const float s = (c.spin[v] > 0 ? 1.f : -1.f) * (f < F ? c.av[v] : 1.f);
            y = *reinterpret_cast<const float4*>(c.z0 + f);
            y = make_float4(s * y.x, s * y.y, s * y.z, s * y.w);
          }
          el_shw<float4>(el_zchunk(uo + a.uz[0] + el_zrow<FC>(r), ch) + (k & 3) * 16) = y;
        }
        unit_sync();
        if (a.nbuf == 2 && i + 1 < b_hi) stage(nxt, buf ^ 1);
        const int next2 = load_info(i + 2);
        float sre = 0.f, sim = 0.f;
        int sp = 2;
        for (int l = 1; l <= L; ++l) {
          const int n = field(cur, 8 + l), tiles = (n + 15) / 16;
          const uint32_t zin = uo + a.uz[(l - 1) & 1], zout = uo + a.uz[l & 1];
          const uint32_t rec = ut + a.urec[buf], pr = ut + a.upair[buf];
          const float* Ul = U + (size_t)(l - 1) * N * LDU;
          if (l < L) {
            for (int k = utid; k < F / 2; k += uthreads)
              el_shw<float4>(zout + n * (128 * FC) + 16 * k) = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int t = uwarp; t < tiles; t += a.uw)
              el_tile<FC, NP, MODE, false>(c, rec, pr, t, n, sp, zin, zout, Ul, to_h, sre, sim);
          } else {
            for (int t = uwarp; t < tiles; t += a.uw)
              el_tile<FC, NP, MODE, true>(c, rec, pr, t, n, sp, zin, zout, Ul, to_h, sre, sim);
          }
          unit_sync();
          sp = n;
        }
        if (a.nbuf == 1 && i + 1 < b_hi) stage(nxt, 0);
        // Delta (fixed order) and the bond's term Jxy/2 exp(Delta)
        // (FP32: summed in float64, since Delta may be many times its terms' rounding)
        typedef typename ElSum<MODE>::T S;
        S dre = warp_sum_f((S)sre), dim = warp_sum_f((S)sim);
        if (a.uw > 1) {
          if (lane == 0) {
            el_shw<S>(ut + a.usum + uwarp * 16) = dre;
            el_shw<S>(ut + a.usum + uwarp * 16 + 8) = dim;
          }
          unit_sync();
        }
        const int j_lo = field(cur, 2), j_hi = field(cur, 3);
        if (uwarp == 0 && lane == 0) {
          for (int w = 1; w < a.uw; ++w) {
            dre += el_sh<S>(ut + a.usum + w * 16);
            dim += el_sh<S>(ut + a.usum + w * 16 + 8);
          }
          const float xr = (float)dre, xi = (float)dim;
          float amp = expf(xr), sn, cs;
          sincosf(xi, &sn, &cs);
          if (MODE != EL_X2) {  // the parts of Delta below float32
            if (amp <= FLT_MAX) amp = fmaf(amp, (float)(dre - (S)xr), amp);
            const float lo = (float)(dim - (S)xi), s0 = sn;
            sn = fmaf(cs, lo, sn);
            cs = fmaf(-s0, lo, cs);
          }
          const double hJ = 0.5 * __hiloint2double(j_hi, j_lo);
          er += hJ * (double)(amp * cs);
          ei += hJ * (double)(amp * sn);
          if (a.dlogpsi) a.dlogpsi[b * E + c.list[i]] = xr;
        }
        cur = nxt;
        nxt = next2;
      }
    }
    if (lane == 0) {
      s_e[2 * warp] = er;
      s_e[2 * warp + 1] = ei;
    }
    __syncthreads();
    if (tid == 0) {
      double re = 0.0, im = 0.0, d = 0.0;
      for (int w = 0; w < kElWarps; ++w) {
        d += s_diag[w];
        re += s_e[2 * w];
        im += s_e[2 * w + 1];
      }
      a.eloc[2 * b] = d + re;
      a.eloc[2 * b + 1] = im;
    }
  }
}

// The kernel of NP neighbour pairs a row for F features.
template <int NP, int MODE>
const void* el_kernel_np(int F) {
  switch (F) {
    case 16:
      return (const void*)k_eloc<1, NP, MODE>;
    case 32:
      return (const void*)k_eloc<2, NP, MODE>;
    case 48:
      return (const void*)k_eloc<3, NP, MODE>;
    default:
      return (const void*)k_eloc<4, NP, MODE>;
  }
}
const void* el_kernel_f32(int np, int F, int mode);  // eloc32.cu

}  // namespace gna
