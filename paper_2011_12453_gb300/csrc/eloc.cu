// Incremental local energy (and log Psi) with split BF16 operands, one warp per tile of 16
// rows: the BF16X2 path of gna_local_energy and gna_local_energy_logpsi for models whose
// balls fit shared memory (tc.cu has the general kernel and the numerics of the difference
// form: layer l changes by dY^l = [A_hat dH^{l-1} ; dH^{l-1}] W on ball_l(e) and
// dH^l = tanh(Y^l + dY^l) - tanh(Y^l)).
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
// 108, L 4, F 32, 16384 configurations 33.9 -> 14.4 ms; triangular 144, L 4, F 48, 4001: 38.0 ->
// 18.7 ms; Kagome 432, L 6, F 64, 512: 26.9 -> 18.2 ms; the error of the energies against 64 bits
// falls 3 to 5 times at weight scale 0.1.
#include <climits>
#include <cstring>

#include "eloc.cuh"
#include "frag.cuh"

namespace gna {

constexpr int kElThreads = 512;
constexpr int kReadout = 512;  // threads of the forward call's readout, whose order of sums is kept
constexpr int kElWarps = kElThreads / 32;
struct ElArgs {
  DevGraph g;
  Dims m;
  const float* theta;
  const int8_t* spins;
  int64_t B;
  double* logpsi;
  double* eloc;
  float* dlogpsi;
  float* gU;   // [grid][L][N][ldu] exp(2 Y) of the CTA's configuration (L2-resident)
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

// What the incremental step needs of a cached unit, in one float32: E = exp(2 Y), at most
// kElCap (Y = 43.7; zero below Y = -52).  H = (E - 1)/(E + 1), and 1 - H^2 = 4 E/(1 + E)^2 keeps its
// relative precision at saturation.
constexpr float kElCap = 5e37f;
__device__ __forceinline__ float el_cache(float y) { return fminf(__expf(2.f * y), kElCap); }

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
// the unit swings (one that lies outside the cached range stays where it is).
__device__ __forceinline__ float el_dtanh_far(float x, float E) {
  const float X = expf(-2.f * fabsf(x));
  float r0, r1;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(1.f + E));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(x > 0.f ? fmaxf(X + E, 1e-37f) : fmaf(E, X, 1.f)));
  return E < kElCap ? copysignf(2.f * (E * r0) * ((1.f - X) * r1), x) : 0.f;
}

__device__ __forceinline__ uint64_t el_dtanh2_far(const ElConst& k, uint64_t x, uint64_t E) {
  float x0, x1, e0, e1, d0, d1;
  f2_unpack(el_dtanh2(k, x, E), d0, d1);
  f2_unpack(x, x0, x1);
  f2_unpack(E, e0, e1);
  return f2_pack(fabsf(x0) > 1.f ? el_dtanh_far(x0, e0) : d0, fabsf(x1) > 1.f ? el_dtanh_far(x1, e1) : d1);
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
};

// Forward of the configuration in c.spin: u of Y^1..Y^L into the cache, H^L left in the row
// buffer that is returned when want_h.  X = [A_hat H ; H] as hi + lo operands, FP32 rows, in
// the order of the forward call's kernel (bit-identical log Psi).
template <int FC>
__device__ const float* el_forward(const ElCtx<FC>& c, float* U, float* Hb, bool want_h) {
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
          *reinterpret_cast<float4*>(U + ((size_t)(l - 1) * N + v) * LDU + 16 * co + 4 * q) =
              make_float4(el_cache(y0), el_cache(y1), el_cache(y2), el_cache(y3));
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

// Shared memory by byte offset (the offsets select between buffers at run time; addressed
// from the array itself every access is a shared-memory one with 32-bit arithmetic).
extern __shared__ __align__(1024) unsigned char el_smem[];
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
//   the ball; zout: Z of the n rows of ball_l for the next layer.
// The stages are kept apart (look-ups, gather, difference, product), each a block without
// branches over all of the thread's values: a warp hides most of its own latency that way.
template <int FC, int NP, bool LAST>
__device__ __forceinline__ void el_tile(const ElCtx<FC>& c, uint32_t rec, uint32_t pairs, int t, int n, int sp,
                                        uint32_t zin, uint32_t zout, const float* Ul, float& sre, float& sim) {
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
  if (!__any_sync(0xffffffffu, zmax > 1.f)) {
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
        x[h][cc][0] = el_dtanh2_far(c.k, x[h][cc][0], e.x);
        x[h][cc][1] = el_dtanh2_far(c.k, x[h][cc][1], e.y);
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
#pragma unroll
    for (int kc = 0; kc < FC; ++kc) {
      const uint4 b0 = c.Wf[((j / FC * FC + kc) * FC + j % FC) * 32 + lane];
      const uint4 b1 = c.Wf[(((j + 1) / FC * FC + kc) * FC + (j + 1) % FC) * 32 + lane];
      if (kc == 0) {
        mma_16816_first(D[0], lo[kc], b0.x, b0.y);
        mma_16816_first(D[1], lo[kc], b0.z, b0.w);
        mma_16816_first(D[2], lo[kc], b1.x, b1.y);
        mma_16816_first(D[3], lo[kc], b1.z, b1.w);
      } else {
        mma_16816(D[0], lo[kc], b0.x, b0.y);
        mma_16816(D[1], lo[kc], b0.z, b0.w);
        mma_16816(D[2], lo[kc], b1.x, b1.y);
        mma_16816(D[3], lo[kc], b1.z, b1.w);
      }
      mma_16816(D[0], mid[kc], b0.x, b0.y);
      mma_16816(D[1], mid[kc], b0.z, b0.w);
      mma_16816(D[2], mid[kc], b1.x, b1.y);
      mma_16816(D[3], mid[kc], b1.z, b1.w);
      mma_16816(D[0], hi[kc], b0.x, b0.y);
      mma_16816(D[1], hi[kc], b0.z, b0.w);
      mma_16816(D[2], hi[kc], b1.x, b1.y);
      mma_16816(D[3], hi[kc], b1.z, b1.w);
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

template <int FC, int NP>
__global__ void __launch_bounds__(kElThreads, 1) k_eloc(const __grid_constant__ ElArgs a) {
  unsigned char* const smem = el_smem;
  __shared__ int s_cnt[kElWarps];
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
  c.k = {el_keep(63.f), el_keep(7.f), el_keep(1.f / 15.f), el_keep(28.f), el_keep(0.5f), el_keep(-1.f)};
  float* red = (float*)(smem + a.ored);
  const float* th = a.theta;
  const float* W = th + a.m.oW;
  // parameters and graph: once per CTA
  for (int i = tid; i < 2 * FC * FC * 32; i += kElThreads)
    ((uint4*)c.Wf)[i] = make_wfrag<FC>(W, i / (FC * 32), (i / 32) % FC, i & 31);
  for (int i = tid; i < F; i += kElThreads) ((float*)c.bias)[i] = th[a.m.ob + i];
  for (int i = tid; i < 2 * F; i += kElThreads) ((float*)c.emb)[i] = tanhf(th[a.m.oWe + i] + th[a.m.obe + i % F]);
  for (int i = tid; i < (F + 2) * 2; i += kElThreads) ((float*)c.wr)[i] = th[a.m.owr + i];
  if (tid < 2) ((float*)c.br)[tid] = th[a.m.obr + tid];
  for (uint32_t i = tid; i < a.units * a.tab_bytes / 16; i += kElThreads) el_shw<uint4>(a.otab + 16 * i) = make_uint4(0, 0, 0, 0);
  __syncthreads();
  for (int v = tid; v < N; v += kElThreads) {
    const int d = __ldg(a.g.row_ptr + v + 1) - __ldg(a.g.row_ptr + v);
    ((float*)c.av)[v] = d > 0 ? 1.f / sqrtf((float)d) : 0.f;
  }
  // Z^0 of a row that changes from up to down: (emb(-1) - emb(+1)) [W[:F] | W[F:]]
  for (int i = tid; i < 2 * F; i += kElThreads) {
    const int f = i % F, top = i < F ? 0 : F;
    float z = 0.f;
    for (int k = 0; k < F; ++k)
      z = fmaf(c.emb[F + k] - c.emb[k], __bfloat162float(__float2bfloat16_rn(W[(size_t)(top + k) * F + f])), z);
    ((float*)c.z0)[i] = z;
  }
  float* U = a.gU + (size_t)blockIdx.x * L * N * LDU;
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
    __syncthreads();
    const float* HL = el_forward<FC>(c, U, Hb, a.logpsi != nullptr);
    if (a.logpsi) {
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
              el_tile<FC, NP, false>(c, rec, pr, t, n, sp, zin, zout, Ul, sre, sim);
          } else {
            for (int t = uwarp; t < tiles; t += a.uw)
              el_tile<FC, NP, true>(c, rec, pr, t, n, sp, zin, zout, Ul, sre, sim);
          }
          unit_sync();
          sp = n;
        }
        if (a.nbuf == 1 && i + 1 < b_hi) stage(nxt, 0);
        // Delta (fixed order) and the bond's term Jxy/2 exp(Delta)
        sre = warp_sum_f(sre);
        sim = warp_sum_f(sim);
        if (a.uw > 1) {
          if (lane == 0) el_shw<float2>(ut + a.usum + uwarp * 8) = make_float2(sre, sim);
          unit_sync();
        }
        const int j_lo = field(cur, 2), j_hi = field(cur, 3);
        if (uwarp == 0 && lane == 0) {
          for (int w = 1; w < a.uw; ++w) {
            const float2 p = el_sh<float2>(ut + a.usum + w * 8);
            sre += p.x;
            sim += p.y;
          }
          const float amp = expf(sre);
          float sn, cs;
          sincosf(sim, &sn, &cs);
          const double hJ = 0.5 * __hiloint2double(j_hi, j_lo);
          er += hJ * (double)(amp * cs);
          ei += hJ * (double)(amp * sn);
          if (a.dlogpsi) a.dlogpsi[b * E + c.list[i]] = sre;
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

// ---------------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------------
struct ElPlan {
  ElArgs a;
  int grid = 0;
  uint32_t smem = 0;
  size_t ws_bytes = 0, u_bytes = 0;
};

// Every row of a graph whose sites all have 3 or 4 (5 or 6) neighbours has two (three)
// neighbour pairs: the gather loop is then unrolled.
template <int NP>
static const void* el_kernel_np(int F) {
  switch (F) {
    case 16:
      return (const void*)k_eloc<1, NP>;
    case 32:
      return (const void*)k_eloc<2, NP>;
    case 48:
      return (const void*)k_eloc<3, NP>;
    default:
      return (const void*)k_eloc<4, NP>;
  }
}
static int el_np(const gna_graph* g) {
  const int np = (g->max_deg + 1) / 2;
  return (g->min_deg + 1) / 2 == np && (np == 2 || np == 3) ? np : 0;
}
static const void* el_kernel(const gna_graph* g, int F) {
  const int np = el_np(g);
  return np == 2 ? el_kernel_np<2>(F) : np == 3 ? el_kernel_np<3>(F) : el_kernel_np<0>(F);
}

// Shared-memory layout of one choice of units and warps; returns its total in bytes.
static uint64_t el_layout(const gna_graph* g, const Dims& m, int units, int uw, int nbuf, ElArgs* a) {
  const int F = m.F, N = m.N, L = m.L;
  uint64_t o = 0;
  auto take = [&](uint64_t bytes) {
    o = (o + 15) / 16 * 16;
    const uint64_t r = o;
    o += bytes;
    return (uint32_t)r;
  };
  a->units = units;
  a->uw = uw;
  a->nbuf = nbuf;
  a->oW = take((uint64_t)2 * F * F * 2);
  a->obias = take(F * 4);
  a->oemb = take(2 * F * 4);
  a->owr = take((F + 2) * 2 * 4);
  a->obr = take(8);
  a->oav = take((uint64_t)N * 4);
  a->oz0 = take(2 * F * 4);
  a->ospin = take(N);
  a->olist = take((uint64_t)m.E * 2);
  // one unit: Z of even and odd layers (the ball's rows and the zero row), staged tables
  uint64_t zr[2] = {3, 0};
  for (int l = 1; l < L; ++l) {
    const uint64_t rows = (uint64_t)g->max_ball[l] + 1;
    if (rows > zr[l & 1]) zr[l & 1] = rows;
  }
  uint64_t u = 0;
  auto utake = [&](uint64_t bytes) {
    const uint64_t r = u;
    u = (u + bytes + 127) / 128 * 128;
    return (uint32_t)r;
  };
  const int np = el_np(g);
  const uint64_t nrec = (uint64_t)(g->max_ball[L] + 15) / 16 * 16;
  const uint64_t npairs = np > 0 ? nrec * np : (uint64_t)(g->max_pairs[L] + 3) / 4 * 4;
  for (int i = 0; i < 2; ++i) a->urec[i] = i < nbuf ? utake(nrec * 8) : 0;
  for (int i = 0; i < 2; ++i) a->upair[i] = i < nbuf ? utake(npairs * 4) : 0;
  a->usum = utake((uint64_t)uw * 8);
  const uint64_t tab = u;
  u = 0;
  for (int i = 0; i < 2; ++i) a->uz[i] = utake(zr[i] * 2 * F * 4);
  if (u > UINT32_MAX / kElWarps || tab > UINT32_MAX / kElWarps) return UINT64_MAX;
  a->tab_bytes = (uint32_t)tab;
  a->unit_bytes = (uint32_t)u;
  a->otab = take((uint64_t)units * tab);
  // the forward's adjacency, readout scratch and (where they fit) two row buffers share the
  // units' space
  o = (o + 127) / 128 * 128;
  a->ounit = (uint32_t)o;
  a->orp = take((uint64_t)(N + 1) * 4);
  a->owf = take((uint64_t)2 * m.E * 4);
  a->ocol = take((uint64_t)2 * m.E * 2);
  a->ored = take(kReadout * 4);
  a->oH = take(0);
  const uint64_t end = (uint64_t)a->ounit + (uint64_t)units * u;
  if (o > end) return UINT64_MAX;
  a->h_smem = o + (uint64_t)2 * N * el_ldh(F) * 4 <= end;
  o = end;
  return o;
}

static gna_status el_plan(const gna_graph* g, const Dims& m, int64_t B, ElPlan* p) {
  if (m.F % 16 != 0 || m.F > 64 || m.L < 1 || !m.shared || m.act != GNA_ACT_TANH || !g->pack_ok || m.E < 1 ||
      m.E > 0xFFFF)
    return GNA_ERR_UNSUPPORTED;
  DeviceInfo di;
  gna_status st = device_info(&di);
  if (st != GNA_OK) return st;
  if (di.cc < 100) return GNA_ERR_UNSUPPORTED;
  const uint64_t budget = (uint64_t)di.smem_optin - 512;  // static variables
  memset(&p->a, 0, sizeof(p->a));
  // For each number of warps a unit may have, as many units as fit.  The time of a bond is its
  // rounds of tiles, each the longer the more warps share the SM: fitted to sweeps of the
  // choices on three lattices and a random graph (Kagome 108, F 32: 15 units of one warp 2.12
  // ms per 2432 configurations, 8 of two 2.34; triangular 144, F 48: 5 of three 5.03, 7 of two
  // 5.22, per 1216; Kagome 432, F 64: 3 of five 7.18, 2 of six 8.78, per 304).  More warps with
  // fewer registers each did not pay (640 and 768 threads: 5 and 13 % slower).  One table
  // buffer instead of two only where it makes room for another unit.
  double best = 1e300;
  int bu = 0, bw = 0, bn = 0;
  ElArgs t;
  memset(&t, 0, sizeof(t));
  for (int uw = 1; uw <= 8; ++uw) {
    double rounds = uw > 1 ? 0.05 * (m.L + 2) : 0.0;
    for (int l = 1; l <= m.L; ++l) rounds += ((g->max_ball[l] + 15) / 16 + uw - 1) / uw;
    for (int nbuf = 2; nbuf >= 1; --nbuf) {
      int units = uw > 1 && kElWarps / uw > 15 ? 15 : kElWarps / uw;  // 15 named barriers beside the block's
      while (units > 0 && el_layout(g, m, units, uw, nbuf, &t) > budget) --units;
      if (units == 0) continue;
      const double cost = rounds / units * (1.0 + 0.12 * units * uw) * (nbuf == 1 ? 1.02 : 1.0);
      if (cost < best) {
        best = cost;
        bu = units;
        bw = uw;
        bn = nbuf;
      }
    }
  }
  if (bu == 0) return GNA_ERR_UNSUPPORTED;
  p->smem = (uint32_t)el_layout(g, m, bu, bw, bn, &p->a);
  const void* kfn = el_kernel(g, m.F);
  GNA_CUDA_TRY(cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p->smem));
  int64_t grid = di.sms;
  if (grid > B) grid = B;
  p->grid = (int)(grid < 1 ? 1 : grid);
  p->u_bytes = align_up((size_t)p->grid * m.L * m.N * el_ldu(m.F) * sizeof(float));
  p->ws_bytes = p->u_bytes + (p->a.h_smem ? 0 : align_up((size_t)p->grid * 2 * m.N * el_ldh(m.F) * sizeof(float)));
  return GNA_OK;
}

gna_status el_workspace(const gna_graph* g, const Dims& m, int64_t B, size_t* bytes) {
  if (B == 0) {
    *bytes = 0;
    return GNA_OK;
  }
  ElPlan p;
  gna_status st = el_plan(g, m, B, &p);
  if (st != GNA_OK) return st;
  *bytes = p.ws_bytes;
  return GNA_OK;
}

gna_status el_run(const TcCall& call, void* ws, size_t ws_bytes, cudaStream_t stream) {
  ElPlan p;
  gna_status st = el_plan(call.g, call.m, call.B, &p);
  if (st != GNA_OK) return st;
  if (ws_bytes < p.ws_bytes || (p.ws_bytes > 0 && !ws)) return GNA_ERR_WORKSPACE;
  ElArgs& a = p.a;
  a.g = call.g->d;
  a.m = call.m;
  a.theta = call.theta;
  a.spins = call.spins;
  a.B = call.B;
  a.logpsi = call.logpsi;
  a.eloc = call.eloc;
  a.dlogpsi = call.dlogpsi;
  a.gU = (float*)ws;
  a.gH = a.h_smem ? nullptr : (float*)((unsigned char*)ws + p.u_bytes);
  void* args[] = {&a};
  GNA_CUDA_TRY(cudaLaunchKernel(el_kernel(call.g, call.m.F), dim3(p.grid), dim3(kElThreads), args, p.smem, stream));
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

}  // namespace gna
