// Metropolis pair-exchange sweeps of BF16 models (plain moves): a warp per chain.
//
// The move rule is the one of the other samplers: step t of chain c draws
// Philox4x64-10(key = (seed, c), counter = (t, 0, 0, 0)), bond e = hi64(r0 |E|); a parallel
// bond is a rejected no-op, an antiparallel one is accepted iff
// (r1 >> 40) 2^-24 < exp(2 Re Delta).  Delta is the difference propagation of the local energy:
// per layer X = [A_hat dH ; dH] on the bond's ball in BF16, dY = X W accumulated in FP32,
// dH = tanh(Y + dY) - tanh(Y) in FP32.  The decisions are a chain's trajectory, so the order
// of every sum is fixed: the message over the neighbours in CSR order, K steps of 16 features
// of the message and then of the row itself, a row's readout feature by feature, the rows
// by (row mod 32) and then across the lanes.
//
// What bounds it: about 9 tiles of 16 rows a proposal (Kagome 108, L 4), each a few hundred
// instructions -- neighbour rows gathered and unpacked, two exponential-type functions and a
// reciprocal per unit -- against 16 matrix instructions, so the issue slots and the latency
// of one tile after the other (6700 instructions a proposal, 43 % of them integer; issue slots
// 40 % busy with 7 warps an SM).  Pools of chains that shared 128-row tcgen05 tiles spent their time
// in barriers and TMEM round trips instead: Kagome 108, L 4, F 32, 16384 chains 25.5 ms against 10.2,
// a twelve-site lattice with 1024 chains 1.08 ms against 0.18 for three sweeps.
// Hence: a warp owns a chain and runs its tiles without any barrier; products are mma.sync (bit-identical to tcgen05 in this order, frag.cuh), their
// results become the next layer's input without leaving the thread's features; W stays in
// registers up to F = 32; Y rows are loaded (L2) before the tile's gather; the Y + dY rows of a
// proposal wait in shared memory and are copied to Y on acceptance; lanes draw 32 steps of
// random words at once and the next antiparallel proposal is found by a ballot.
#include <cuda_bf16.h>

#include "frag.cuh"
#include "mtile.cuh"

namespace gna {
namespace {

// Most warps a block, and with it the registers of a thread (128 or 168): F = 32 keeps W in
// registers and gains from the larger set (Kagome 108, L 4, 16384 chains: 10.2 ms with 168, 11.0
// with 128; the shared memory holds 11 warps either way); the other widths gain more from 16 warps
// (F = 16 6.4 against 7.2 ms; triangular 144, L 4, F = 64, 4096 chains: 15.8 against 18.4).
__host__ __device__ constexpr int mt_warps(int FC) { return FC == 2 ? 12 : 16; }
// Fewest warps a block worth keeping the Y + dY rows in shared memory for.  Kagome 108, L 4,
// F = 64, 8192 chains: 19.2 ms with 5 warps and shared rows, 17.1 with 16 and rows in the workspace;
// F = 32, 16384 chains: 11.0 with 11 and shared rows, 11.2 with 16 without.
constexpr int kMtEnough = 6;

struct MtArgs {
  DevGraph g;
  Dims m;
  const float* theta;
  int8_t* chain_spins;
  int64_t C;
  int n_sweeps, record_every;
  uint64_t seed, step0;
  int8_t* samples_out;
  double* logpsi_out;
  int32_t* n_acc;
  double* trace;
  unsigned char* ws;
  uint64_t ws_warp;           // workspace bytes per warp: Y^1..Y^L, two BF16 layers, what is not shared
  uint64_t w_h, w_dh, w_yn;   // byte offsets in it
  // shared memory (bytes); per warp from owarp
  uint32_t oW, obias, oemb, owr, owp, owf, owarp, warp_bytes;
  uint32_t p_spin, p_rec, p_pair, p_buf, p_dh[2], p_yn;
  uint32_t g_dh1;             // second dH buffer from w_dh when the workspace holds them
  int dh_smem, yn_smem;
  int warps;
  int yrow[kMaxL + 2];        // first row of layer l in the Y + dY rows
};

__device__ __forceinline__ float mt_tanh(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float mt_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float mt_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t mt_pack(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// acc (two pairs) += w * four BF16 features
__device__ __forceinline__ void mt_fma4(uint64_t* acc, uint64_t w, uint2 x) {
  acc[0] = f2_fma(f2_pack(__uint_as_float(x.x << 16), __uint_as_float(x.x & 0xFFFF0000u)), w, acc[0]);
  acc[1] = f2_fma(f2_pack(__uint_as_float(x.y << 16), __uint_as_float(x.y & 0xFFFF0000u)), w, acc[1]);
}
__device__ __forceinline__ void mt_pack4(const uint64_t* acc, uint32_t& lo, uint32_t& hi) {
  float a, b;
  f2_unpack(acc[0], a, b);
  lo = mt_pack(a, b);
  f2_unpack(acc[1], a, b);
  hi = mt_pack(a, b);
}

__host__ __device__ constexpr int mt_ldh(int F) { return F + 8; }  // BF16 rows
__host__ __device__ constexpr int mt_ldd(int F) { return F + 4; }  // last layer's dH rows (FP32)

// 16-byte chunk j of row r of the Y + dY rows: for F a multiple of 32, pairs of rows would meet
// in the same banks, so odd rows swap neighbouring groups of four chunks.
template <int FC>
__device__ __forceinline__ int mt_yn(int r, int j) {
  return r * 4 * FC + (FC % 2 == 0 ? j ^ ((r & 1) << 2) : j);
}

// tanh(y + d) - tanh(y) by the full rule: with e = exp(-2|y|), t = tanh d,
// 4 e t / ((1 + e)((1 + e) + sgn(y)(1 - e) t)), and the direct difference where the unit swings
// across saturation and the denominator vanishes.
__device__ __noinline__ float mt_dtanh_full(float y, float d) {
  const float e = __expf(-2.f * fabsf(y));
  const float sg = y < 0.f ? -1.f : 1.f;
  const float tt = fabsf(d) < 0.5f ? mt_tanh(d) : tanhf(d);
  const float ope = 1.f + e;
  const float den = ope * (ope + sg * (1.f - e) * tt);
  return den > 1e-3f ? __fdividef(4.f * e * tt, den) : tanhf(y + d) - tanhf(y);
}

// The same for two units by the common case (|d| < 0.5, denominator > 1e-3); mx, mn collect what
// decides whether it applies.
__device__ __forceinline__ void mt_dtanh2(uint64_t one, uint64_t m1, uint64_t four, float y0, float y1, float d0,
                                          float d1, float& o0, float& o1, float& mx, float& mn) {
  constexpr float k = -2.8853900817779268f;  // -2 log2 e
  const uint64_t e = f2_pack(mt_ex2(fabsf(y0) * k), mt_ex2(fabsf(y1) * k));
  const uint64_t t = f2_pack(mt_tanh(d0), mt_tanh(d1));
  const uint64_t ope = f2_add(e, one);
  float a, b;
  f2_unpack(f2_fma(e, m1, one), a, b);
  const uint64_t den = f2_mul(ope, f2_fma(f2_pack(copysignf(a, y0), copysignf(b, y1)), t, ope));
  float n0, n1;
  f2_unpack(den, n0, n1);
  f2_unpack(f2_mul(f2_mul(f2_mul(e, four), t), f2_pack(mt_rcp(n0), mt_rcp(n1))), o0, o1);
  mx = fmaxf(mx, fmaxf(fabsf(d0), fabsf(d1)));
  mn = fminf(mn, fminf(n0, n1));
}

template <int FC, bool REG>
struct MtW {  // B fragments of W in registers or shared memory
  uint4 r[REG ? 2 * FC * FC : 1];
  const uint4* s;
  __device__ __forceinline__ uint4 at(int i, int lane) const { return REG ? r[REG ? i : 0] : s[i * 32 + lane]; }
};

// D = X W for output chunk co: D[0] (columns 4q, 4q + 1 of the chunk), D[1] (4q + 2, 4q + 3);
// [0..1] row g, [2..3] row g + 8.
template <int FC, bool REG>
__device__ __forceinline__ void mt_product(const MtW<FC, REG>& W, const uint32_t (*A)[4], int co, int lane, float (*D)[4]) {
#pragma unroll
  for (int kc = 0; kc < 2 * FC; ++kc) {
    const uint4 b = W.at(kc * FC + co, lane);
    if (kc == 0) {
      mma_16816_first(D[0], A[0], b.x, b.y);
      mma_16816_first(D[1], A[0], b.z, b.w);
    } else {
      mma_16816(D[0], A[kc], b.x, b.y);
      mma_16816(D[1], A[kc], b.z, b.w);
    }
  }
}

// Forward of the warp's configuration: Y^1..Y^L (FP32).
template <int FC>
__device__ __noinline__ void mt_forward(const MtArgs& a, const float* bias, const float* emb, const int* wp,
                                        const float2* wf, const uint4* Ws, const int8_t* sp, float* Y,
                                        __nv_bfloat16* H) {
  constexpr int F = 16 * FC, LDH = mt_ldh(F);
  const int N = a.m.N, L = a.m.L;
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  MtW<FC, false> W;
  W.s = Ws;
  for (int i = lane; i < N * (F / 4); i += 32) {
    const int v = i / (F / 4), f = (i % (F / 4)) * 4;
    const float4 x = *reinterpret_cast<const float4*>(emb + (sp[v] > 0 ? 0 : F) + f);
    *reinterpret_cast<uint2*>(H + (size_t)v * LDH + f) = make_uint2(mt_pack(x.x, x.y), mt_pack(x.z, x.w));
  }
  __syncwarp();
  for (int l = 1; l <= L; ++l) {
    const __nv_bfloat16* hp = H + (size_t)((l - 1) & 1) * N * LDH + 4 * q;
    __nv_bfloat16* hn = H + (size_t)(l & 1) * N * LDH + 4 * q;
    for (int t = 0; t < N; t += 16) {
      uint32_t A[2 * FC][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v = min(t + g + 8 * h, N - 1);
        uint64_t acc[FC][2];
#pragma unroll
        for (int c = 0; c < FC; ++c) acc[c][0] = acc[c][1] = 0;
        const int k0 = __ldg(a.g.row_ptr + v), dg = __ldg(a.g.row_ptr + v + 1) - k0;
        const float* w = reinterpret_cast<const float*>(wf + wp[v]);
        for (int k = 0; k < dg; ++k) {
          const uint64_t w2 = f2_dup(w[k]);
          const __nv_bfloat16* x = hp + (size_t)__ldg(a.g.col + k0 + k) * LDH;
#pragma unroll
          for (int c = 0; c < FC; ++c) mt_fma4(acc[c], w2, *reinterpret_cast<const uint2*>(x + 16 * c));
        }
#pragma unroll
        for (int c = 0; c < FC; ++c) {
          mt_pack4(acc[c], A[c][h], A[c][2 + h]);
          const uint2 x = *reinterpret_cast<const uint2*>(hp + (size_t)v * LDH + 16 * c);
          A[FC + c][h] = x.x;
          A[FC + c][2 + h] = x.y;
        }
      }
#pragma unroll
      for (int co = 0; co < FC; ++co) {
        float D[2][4];
        mt_product(W, A, co, lane, D);
        const float4 b = *reinterpret_cast<const float4*>(bias + 16 * co + 4 * q);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int v = t + g + 8 * h;
          if (v >= N) continue;
          const float4 y = make_float4(D[0][2 * h] + b.x, D[0][2 * h + 1] + b.y, D[1][2 * h] + b.z, D[1][2 * h + 1] + b.w);
          *reinterpret_cast<float4*>(Y + ((size_t)(l - 1) * N + v) * F + 16 * co + 4 * q) = y;
          if (l < L)
            *reinterpret_cast<uint2*>(hn + (size_t)v * LDH + 16 * co) =
                make_uint2(mt_pack(mt_tanh(y.x), mt_tanh(y.y)), mt_pack(mt_tanh(y.z), mt_tanh(y.w)));
        }
      }
    }
    __syncwarp();
  }
}

// log Psi from Y^L and the spins: per-thread partial sums of the block that has 512 / units
// threads (units = 2 up to F = 16, else 4), added in float64.
template <int FC>
__device__ __noinline__ void mt_record(const MtArgs& a, const float* wr, const int8_t* sp, const float* YL, int64_t ch,
                                       int rec) {
  constexpr int F = 16 * FC, kPart = FC == 1 ? 256 : 128;
  const int N = a.m.N, lane = threadIdx.x & 31;
  if (a.samples_out)
    for (int v = lane; v < N; v += 32) a.samples_out[((size_t)rec * a.C + ch) * N + v] = sp[v];
  if (!a.logpsi_out) return;
  double zr = 0.0, zi = 0.0;
  for (int p = lane; p < kPart; p += 32) {
    float re = 0.f, im = 0.f;
    for (int i = p; i < N * F; i += kPart) {
      const float hv = tanhf(YL[i]);
      const int f = i % F;
      re += hv * wr[2 * f];
      im += hv * wr[2 * f + 1];
    }
    zr += (double)re;
    zi += (double)im;
  }
  int up = 0;
  for (int v = lane; v < N; v += 32) up += sp[v] > 0;
  zr = warp_sum_f(zr);
  zi = warp_sum_f(zi);
  up = warp_sum_f(up);
  if (lane == 0) {
    const float* br = wr + 2 * (F + 2);
    const int dn = N - up;
    double* o = a.logpsi_out + ((size_t)rec * a.C + ch) * 2;
    o[0] = zr + (double)up * wr[2 * F] + (double)dn * wr[2 * (F + 1)] + (double)br[0];
    o[1] = zi + (double)up * wr[2 * F + 1] + (double)dn * wr[2 * (F + 1) + 1] + (double)br[1];
  }
}

extern __shared__ __align__(128) unsigned char mt_smem[];

// GEN: the dH rows or the Y + dY rows live in the workspace (graphs whose balls are large).
template <int FC, bool GEN>
__global__ void __launch_bounds__(mt_warps(FC) * 32, 1) k_mt_metro(const MtArgs a) {
  constexpr int F = 16 * FC, LDH = mt_ldh(F), LDD = mt_ldd(F);
  const int N = a.m.N, L = a.m.L, E = a.m.E;
  const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
  const float* th = a.theta;
  float* bias = (float*)(mt_smem + a.obias);
  float* emb = (float*)(mt_smem + a.oemb);
  float* wr = (float*)(mt_smem + a.owr);  // [F + 2][2], then br[2], then the real parts [F]
  int* wp = (int*)(mt_smem + a.owp);
  float2* wf = (float2*)(mt_smem + a.owf);
  for (int i = tid; i < F; i += nthr) bias[i] = th[a.m.ob + i];
  for (int i = tid; i < 2 * F; i += nthr) emb[i] = tanhf(th[a.m.oWe + i] + th[a.m.obe + i % F]);
  for (int i = tid; i < (F + 2) * 2; i += nthr) wr[i] = th[a.m.owr + i];
  if (tid < 2) wr[2 * (F + 2) + tid] = th[a.m.obr + tid];
  float* wre = wr + 2 * (F + 2) + 4;
  for (int i = tid; i < F; i += nthr) wre[i] = th[a.m.owr + 2 * i];
  for (int i = tid; i < 2 * FC * FC * 32; i += nthr)
    ((uint4*)(mt_smem + a.oW))[i] = make_wfrag<FC>(th + a.m.oW, i / (FC * 32), (i / 32) % FC, i & 31, 0);
  if (warp == 0) {  // first pair of each vertex: a running sum, 32 vertices at a time
    int base = 0;
    for (int v0 = 0; v0 < N; v0 += 32) {
      const int v = v0 + lane;
      const int n = v < N ? (__ldg(a.g.row_ptr + v + 1) - __ldg(a.g.row_ptr + v) + 1) / 2 : 0;
      int x = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
      }
      if (v < N) wp[v] = base + x - n;
      base += __shfl_sync(0xffffffffu, x, 31);
    }
  }
  __syncthreads();
  for (int v = tid; v < N; v += nthr) {
    const int k0 = __ldg(a.g.row_ptr + v), dg = __ldg(a.g.row_ptr + v + 1) - k0;
    for (int j = 0; 2 * j < dg; ++j)
      wf[wp[v] + j] = make_float2(__ldg(a.g.wf + k0 + 2 * j), 2 * j + 1 < dg ? __ldg(a.g.wf + k0 + 2 * j + 1) : 0.f);
  }
  __syncthreads();
  constexpr bool kWReg = FC <= 2;
  MtW<FC, kWReg> W;
  W.s = (const uint4*)(mt_smem + a.oW);
  if (kWReg)
#pragma unroll
    for (int i = 0; i < (kWReg ? 2 * FC * FC : 1); ++i) W.r[i] = W.s[i * 32 + lane];

  // this warp's parts of shared memory and of the workspace
  unsigned char* sm = mt_smem + a.owarp + (uint32_t)warp * a.warp_bytes;
  int8_t* sp = (int8_t*)(sm + a.p_spin);
  int2* rec = (int2*)(sm + a.p_rec);
  uint32_t* pairs = (uint32_t*)(sm + a.p_pair);
  float* dbuf = (float*)(sm + a.p_buf);
  const int64_t gw = (int64_t)blockIdx.x * a.warps + warp, nw = (int64_t)gridDim.x * a.warps;
  unsigned char* ws = a.ws + (size_t)gw * a.ws_warp;
  float* Y = (float*)ws;
  __nv_bfloat16* H = (__nv_bfloat16*)(ws + a.w_h);
  unsigned char *dh0 = sm + a.p_dh[0], *dh1 = sm + a.p_dh[1];
  float4* yn = (float4*)(sm + a.p_yn);
  if (GEN) {
    if (!a.dh_smem) {
      dh0 = ws + a.w_dh;
      dh1 = dh0 + a.g_dh1;
    }
    if (!a.yn_smem) yn = (float4*)(ws + a.w_yn);
  }
  const uint64_t one = f2_dup(1.f), m1 = f2_dup(-1.f), four = f2_dup(4.f);
  const int64_t n_steps = (int64_t)a.n_sweeps * N;
  const int64_t rec_steps = a.record_every > 0 ? (int64_t)a.record_every * N : INT64_MAX;

  for (int64_t ch = gw; ch < a.C; ch += nw) {
    for (int v = lane; v < N; v += 32) sp[v] = a.chain_spins[ch * N + v];
    __syncwarp();
    mt_forward<FC>(a, bias, emb, wp, wf, (const uint4*)(mt_smem + a.oW), sp, Y, H);
    int accepted = 0, nrec = 0;
    int64_t wbase = -64, next_rec = rec_steps;
    uint64_t r1 = 0;             // this lane's step wbase + lane: uniform word, bond and its ends
    int be = 0, bi = 0, bj = 0;
    for (int64_t k = 0; k < n_steps;) {
      // 1. the next antiparallel proposal (the steps before it are rejected no-ops)
      if (k >= wbase + 32) {
        wbase = k;
        const U64x4 w = philox4x64_10(a.seed, (uint64_t)ch, U64x4{a.step0 + (uint64_t)(k + lane), 0, 0, 0});
        r1 = w.y;
        be = (int)__umul64hi(w.x, (uint64_t)E);
        bi = __ldg(a.g.edges + 2 * be);
        bj = __ldg(a.g.edges + 2 * be + 1);
      }
      const int64_t lim = min(min(wbase + 32, n_steps), next_rec);
      const bool in = wbase + lane >= k && wbase + lane < lim;
      const uint32_t anti = __ballot_sync(0xffffffffu, in && sp[bi] != sp[bj]);
      const int src = anti ? __ffs(anti) - 1 : 0;
      const int64_t stop = anti ? wbase + src : lim;
      if (a.trace && in && wbase + lane < stop) {
        double* tr = a.trace + ((size_t)ch * n_steps + wbase + lane) * 4;
        tr[0] = (double)be;
        tr[1] = 0.0;
        tr[2] = __longlong_as_double(0x7ff8000000000000ll);
        tr[3] = 1.0;
      }
      k = stop;
      if (anti) {
        const int e = __shfl_sync(0xffffffffu, be, src), i = __shfl_sync(0xffffffffu, bi, src),
                  j = __shfl_sync(0xffffffffu, bj, src);
        // 2. the bond's rows and neighbour positions, and dH^0
        const int info = __ldg(a.g.bond_info + 32 * (size_t)e + lane);
        const int rec0 = __shfl_sync(0xffffffffu, info, 0), pair0 = __shfl_sync(0xffffffffu, info, 1);
        const int RL = __shfl_sync(0xffffffffu, info, 8 + L), np = __shfl_sync(0xffffffffu, info, 16 + L);
        {
          const int2* src_r = reinterpret_cast<const int2*>(a.g.rec) + rec0;
          for (int x = lane; 2 * x < RL; x += 32) cp_async16(rec + 2 * x, src_r + 2 * x);
          const uint32_t* src_p = a.g.pairs + pair0;
          for (int x = lane; 4 * x < np; x += 32) cp_async16(pairs + 4 * x, src_p + 4 * x);
          const int si = sp[i] > 0 ? 0 : F, sj = sp[j] > 0 ? 0 : F;
          __nv_bfloat16* d = (__nv_bfloat16*)dh0;
          for (int f = lane; f < F; f += 32) {
            d[f] = __float2bfloat16_rn(emb[sj + f] - emb[si + f]);
            d[LDH + f] = __float2bfloat16_rn(emb[si + f] - emb[sj + f]);
            d[2 * LDH + f] = __float2bfloat16_rn(0.f);
          }
          cp_async_wait_all();
        }
        __syncwarp();
        // 3. the layers, tiles of 16 rows
        float dre = 0.f;
        int sprev = 2;
        for (int l = 1; l <= L; ++l) {
          const int R = __shfl_sync(0xffffffffu, info, 8 + l);
          const __nv_bfloat16* dp = (const __nv_bfloat16*)((l - 1) & 1 ? dh1 : dh0) + 4 * q;
          __nv_bfloat16* dn = (__nv_bfloat16*)(l & 1 ? dh1 : dh0) + 4 * q;
          if (l < L && lane < 4)
#pragma unroll
            for (int c = 0; c < FC; ++c) *reinterpret_cast<uint2*>(dn + (size_t)R * LDH + 16 * c) = make_uint2(0u, 0u);
          const float* Yl = Y + (size_t)(l - 1) * N * F + 4 * q;
          for (int t = 0; t < R; t += 16) {
            uint32_t A[2 * FC][4];
            float4 y[2][FC];
            int2 rr[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              rr[h] = rec[min(t + g + 8 * h, R - 1)];
              const float* yr = Yl + (rr[h].x & 0xFFFF) * F;
#pragma unroll
              for (int c = 0; c < FC; ++c) y[h][c] = *reinterpret_cast<const float4*>(yr + 16 * c);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int r = t + g + 8 * h;
              uint64_t acc[FC][2];
#pragma unroll
              for (int c = 0; c < FC; ++c) acc[c][0] = acc[c][1] = 0;
              const int n2 = (int)((uint32_t)rr[h].x >> 16);
              const float2* w = wf + wp[rr[h].x & 0xFFFF];
              const uint32_t* pr = pairs + rr[h].y;
              // positions outside ball_{l-1} read the row of zeros behind it: the zero products
              // leave the sums unchanged
              for (int p = 0; p < n2; ++p) {
                const uint32_t pp = pr[p];
                const float2 ww = w[p];
                const __nv_bfloat16* x0 = dp + min((int)((pp & 0xFFFFu) >> 2), sprev) * LDH;
                const __nv_bfloat16* x1 = dp + min((int)(pp >> 18), sprev) * LDH;
                const uint64_t w0 = f2_dup(ww.x), w1 = f2_dup(ww.y);
#pragma unroll
                for (int c = 0; c < FC; ++c) {
                  mt_fma4(acc[c], w0, *reinterpret_cast<const uint2*>(x0 + 16 * c));
                  mt_fma4(acc[c], w1, *reinterpret_cast<const uint2*>(x1 + 16 * c));
                }
              }
              const __nv_bfloat16* xs = dp + min(r, sprev) * LDH;
#pragma unroll
              for (int c = 0; c < FC; ++c) {
                mt_pack4(acc[c], A[c][h], A[c][2 + h]);
                const uint2 x = *reinterpret_cast<const uint2*>(xs + 16 * c);
                A[FC + c][h] = x.x;
                A[FC + c][2 + h] = x.y;
              }
            }
#pragma unroll
            for (int co = 0; co < FC; ++co) {
              float D[2][4];
              mt_product(W, A, co, lane, D);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const int r = t + g + 8 * h;
                const float4 yy = y[h][co];
                const float d0 = D[0][2 * h], d1 = D[0][2 * h + 1], d2 = D[1][2 * h], d3 = D[1][2 * h + 1];
                float o0, o1, o2, o3, mx = 0.f, mn = 1.f;
                mt_dtanh2(one, m1, four, yy.x, yy.y, d0, d1, o0, o1, mx, mn);
                mt_dtanh2(one, m1, four, yy.z, yy.w, d2, d3, o2, o3, mx, mn);
                if (!(mx < 0.5f) || !(mn > 1e-3f)) {
                  o0 = mt_dtanh_full(yy.x, d0);
                  o1 = mt_dtanh_full(yy.y, d1);
                  o2 = mt_dtanh_full(yy.z, d2);
                  o3 = mt_dtanh_full(yy.w, d3);
                }
                if (r < R) {
                  yn[mt_yn<FC>(a.yrow[l] + r, 4 * co + q)] = make_float4(yy.x + d0, yy.y + d1, yy.z + d2, yy.w + d3);
                  if (l < L)
                    *reinterpret_cast<uint2*>(dn + r * LDH + 16 * co) = make_uint2(mt_pack(o0, o1), mt_pack(o2, o3));
                }
                if (l == L)
                  *reinterpret_cast<float4*>(dbuf + (g + 8 * h) * LDD + 16 * co + 4 * q) = make_float4(o0, o1, o2, o3);
              }
            }
            if (l == L) {
              // a row's Re dH . w_r feature by feature, the row in lane (row mod 32)
              __syncwarp();
              if (lane >> 4 == ((t >> 4) & 1) && t + (lane & 15) < R) {
                const float4* d = reinterpret_cast<const float4*>(dbuf + (lane & 15) * LDD);
                float s = 0.f;
#pragma unroll
                for (int f4 = 0; f4 < F / 4; ++f4) {
                  const float4 x = d[f4], w = reinterpret_cast<const float4*>(wre)[f4];
                  s = fmaf(x.x, w.x, s);
                  s = fmaf(x.y, w.y, s);
                  s = fmaf(x.z, w.z, s);
                  s = fmaf(x.w, w.w, s);
                  if (FC == 1 && f4 == 1) {  // F = 16: the two chunks of 8 one after the other
                    dre += s;
                    s = 0.f;
                  }
                }
                dre += s;
              }
              __syncwarp();
            }
          }
          sprev = R;
          __syncwarp();
        }
        // 4. the decision
        dre = warp_sum_f(dre);
        const uint64_t u1 = __shfl_sync(0xffffffffu, r1, src);
        const bool acc = (float)(u1 >> 40) * 0x1.0p-24f < expf(2.0f * dre);
        if (a.trace && lane == 0) {
          double* tr = a.trace + ((size_t)ch * n_steps + k) * 4;
          tr[0] = (double)e;
          tr[1] = acc ? 1.0 : 0.0;
          tr[2] = (double)dre;
          tr[3] = 1.0;
        }
        if (acc) {
          ++accepted;
          for (int l = 1; l <= L; ++l) {
            const int R = __shfl_sync(0xffffffffu, info, 8 + l);
            float* Yl = Y + (size_t)(l - 1) * N * F;
#pragma unroll 4
            for (int x = lane; x < R * 4 * FC; x += 32) {
              const int r = x / (4 * FC), c = x - r * 4 * FC;
              *reinterpret_cast<float4*>(Yl + (rec[r].x & 0xFFFF) * F + 4 * c) = yn[mt_yn<FC>(a.yrow[l] + r, c)];
            }
          }
          if (lane == 0) {
            const int8_t s = sp[i];
            sp[i] = sp[j];
            sp[j] = s;
          }
        }
        __syncwarp();
        ++k;
      }
      // 5. the sample of a completed sweep
      if (k == next_rec) {
        mt_record<FC>(a, wr, sp, Y + (size_t)(L - 1) * N * F, ch, nrec++);
        next_rec += rec_steps;
      }
    }
    for (int v = lane; v < N; v += 32) a.chain_spins[ch * N + v] = sp[v];
    if (lane == 0 && a.n_acc) a.n_acc[ch] += accepted;
    __syncwarp();
  }
}

struct MtPlan {
  MtArgs a;
  int grid = 0;
  uint32_t smem = 0;
  size_t ws_bytes = 0;
};

const void* mt_kernel(int F, bool gen) {
  switch (F / 16) {
    case 1: return gen ? (const void*)k_mt_metro<1, true> : (const void*)k_mt_metro<1, false>;
    case 2: return gen ? (const void*)k_mt_metro<2, true> : (const void*)k_mt_metro<2, false>;
    case 3: return gen ? (const void*)k_mt_metro<3, true> : (const void*)k_mt_metro<3, false>;
    default: return gen ? (const void*)k_mt_metro<4, true> : (const void*)k_mt_metro<4, false>;
  }
}

// Shared-memory layout with the dH rows and the Y + dY rows in it or not: fills the offsets, the
// workspace per warp and the bytes a block takes before its warps' parts.
void mt_layout(const gna_graph* g, const Dims& m, bool dh_smem, bool yn_smem, MtArgs* a) {
  const int F = m.F, N = m.N, L = m.L, FC = F / 16;
  uint64_t o = 0;
  auto take = [&](uint64_t bytes) {
    const uint64_t r = o;
    o = (o + bytes + 15) / 16 * 16;
    return r;
  };
  uint64_t npairs = 0;
  for (int v = 0; v < N; ++v) npairs += (g->h_row_ptr[v + 1] - g->h_row_ptr[v] + 1) / 2;
  a->oW = (uint32_t)take((uint64_t)2 * FC * FC * 512);
  a->obias = (uint32_t)take(F * 4);
  a->oemb = (uint32_t)take(2 * F * 4);
  a->owr = (uint32_t)take((2 * (F + 2) + 4 + F) * 4);
  a->owp = (uint32_t)take((uint64_t)(N + 1) * 4);
  a->owf = (uint32_t)take(npairs * 8);
  a->owarp = (uint32_t)o;
  o = 0;
  a->dh_smem = dh_smem;
  a->yn_smem = yn_smem;
  const uint64_t buf = (uint64_t)16 * mt_ldd(F) * 4;
  uint64_t dh[2] = {0, 0}, rows = 0;  // rows of the even and the odd layers' dH and a row of zeros
  for (int l = 0; l < L; ++l) {
    const uint64_t b = (uint64_t)(g->max_ball[l] + 1) * mt_ldh(F) * 2;
    if (b > dh[l & 1]) dh[l & 1] = b;
  }
  for (int l = 1; l <= L; ++l) {
    a->yrow[l] = (int)rows;
    rows += g->max_ball[l];
  }
  a->p_spin = (uint32_t)take(N);
  a->p_rec = (uint32_t)take((uint64_t)(g->max_ball[L] + 1) / 2 * 16);
  a->p_pair = (uint32_t)take((uint64_t)(g->max_pairs[L] + 3) / 4 * 16);
  if (dh_smem) {
    // the last layer's rows take the place of the dH of layer L - 2, which nothing reads any more
    if (buf > dh[L & 1]) dh[L & 1] = buf;
    a->p_dh[0] = (uint32_t)take(dh[0]);
    a->p_dh[1] = (uint32_t)take(dh[1]);
    a->p_buf = a->p_dh[L & 1];
  } else {
    a->p_buf = (uint32_t)take(buf);
  }
  if (yn_smem) a->p_yn = (uint32_t)take(rows * F * 4);
  a->warp_bytes = (uint32_t)o;
  o = 0;
  take((uint64_t)L * N * F * 4);
  a->w_h = take((uint64_t)2 * N * mt_ldh(F) * 2);
  if (!dh_smem) {
    a->w_dh = take(dh[0]);
    a->g_dh1 = (uint32_t)(take(dh[1]) - a->w_dh);
  }
  if (!yn_smem) a->w_yn = take(rows * F * 4);
  a->ws_warp = (o + 127) / 128 * 128;
}

gna_status mt_plan(const gna_graph* g, const Dims& m, int64_t C, MtPlan* p) {
  if (m.F % 16 != 0 || m.F < 16 || m.F > 64 || m.L < 1 || !m.shared || m.act != GNA_ACT_TANH || m.E < 1 || !g->pack_ok)
    return GNA_ERR_UNSUPPORTED;
  DeviceInfo di;
  gna_status st = device_info(&di);
  if (st != GNA_OK) return st;
  const uint64_t budget = (uint64_t)di.smem_optin - 64;
  MtArgs& a = p->a;
  memset(&a, 0, sizeof(a));
  // rows in shared memory while enough warps fit, else the Y + dY rows, then also the dH rows, in
  // the workspace
  int warps = 0, form = 0;
  for (; form < 3; ++form) {
    mt_layout(g, m, form < 2, form < 1, &a);
    warps = a.owarp > budget ? 0 : (int)((budget - a.owarp) / a.warp_bytes);
    if (warps >= (form == 2 ? 1 : kMtEnough)) break;
  }
  if (form == 3) return GNA_ERR_UNSUPPORTED;
  if (warps > mt_warps(m.F / 16)) warps = mt_warps(m.F / 16);
  // equal shares of the chains: the rounds that the most warps need, with as few warps as do them
  const int most = warps;
  const int64_t per_sm = (C + di.sms - 1) / di.sms;
  const int64_t rounds = (per_sm + warps - 1) / warps;
  warps = (int)((per_sm + rounds - 1) / rounds);
  a.warps = warps;
  p->smem = a.owarp + (uint32_t)warps * a.warp_bytes;
  if ((st = allow_smem(mt_kernel(m.F, form > 0), budget)) != GNA_OK) return st;
  const int64_t need = (C + warps - 1) / warps;
  p->grid = (int)(need < di.sms ? need : di.sms);
  // (the bytes of any number of chains up to C: fewer chains may be more warps)
  const int64_t slots = C + most - 1 < (int64_t)di.sms * most ? C + most - 1 : (int64_t)di.sms * most;
  p->ws_bytes = align_up((size_t)slots * a.ws_warp);
  return GNA_OK;
}

}  // namespace

gna_status mt_workspace(const gna_graph* g, const Dims& m, int64_t C, size_t* bytes) {
  if (C == 0) {
    *bytes = 0;
    return GNA_OK;
  }
  MtPlan p;
  gna_status st = mt_plan(g, m, C, &p);
  if (st == GNA_OK) *bytes = p.ws_bytes;
  return st;
}

gna_status mt_run(const MetroCall& mc, void* ws, size_t ws_bytes, cudaStream_t stream) {
  if (mc.C == 0 || mc.n_sweeps == 0) return GNA_OK;
  MtPlan p;
  gna_status st = mt_plan(mc.g, mc.m, mc.C, &p);
  if (st != GNA_OK) return st;
  if (ws_bytes < p.ws_bytes || !ws) return GNA_ERR_WORKSPACE;
  MtArgs& a = p.a;
  a.g = mc.g->d;
  a.m = mc.m;
  a.theta = (const float*)mc.theta;
  a.chain_spins = mc.chain_spins;
  a.C = mc.C;
  a.n_sweeps = mc.n_sweeps;
  a.record_every = mc.record_every;
  a.seed = mc.seed;
  a.step0 = mc.step0;
  a.samples_out = mc.samples_out;
  a.logpsi_out = mc.logpsi_out;
  a.n_acc = mc.n_acc;
  a.trace = mc.trace;
  a.ws = (unsigned char*)ws;
  void* args[] = {&a};
  GNA_CUDA_TRY(cudaLaunchKernel(mt_kernel(mc.m.F, !(a.dh_smem && a.yn_smem)), dim3(p.grid), dim3(a.warps * 32), args,
                                p.smem, stream));
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

}  // namespace gna
