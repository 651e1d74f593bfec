// Metropolis pair-exchange sweeps with one warp per chain (plain moves).
//
// Sampling P ~ |Psi|^2 (scaling section of arXiv:2011.12453) needs, per proposed exchange
// of an antiparallel pair (i, j), the ratio Psi(s')/Psi(s).  It is computed by propagating
// the change of the node features through the GCN layers of Eq. (gcn), restricted to the
// nested neighbourhoods ball_l(e) of the bond:
//   dH^0 = rows i, j of the embedding difference;
//   dY^l = [A_hat dH^{l-1} ; dH^{l-1}] W   (the bias cancels; zero outside ball_l),
//   dH^l = tanh(Y^l + dY^l) - tanh(Y^l) = t (1 - H^2)/(1 + H t),  t = tanh(dY^l),
//   Delta log Psi = w_r[:F] . sum_v dH^L_v.
// The chain keeps the pre-activations Y^1..Y^L of its current state (in a per-warp slice of
// the workspace, L2-resident); an accepted move adds dY^l to the rows of ball_l.
//
// A warp owns a chain at a time: no block barriers, only warp-synchronous steps, so the
// latency of one chain's step is hidden behind the other warps' chains.  Lanes own
// feature columns (f = lane, lane + 32).  The Philox words of 32 consecutive steps are
// drawn at once, one step per lane, and broadcast by shuffles.
#include <climits>
#include <cmath>

#include "common.cuh"
#include "frag.cuh"
#include "metro.cuh"
#include "prop.cuh"

namespace gna {

constexpr int kMetroMaxWarps = 16;  // chains per CTA at most (fewer when shared memory is short)

template <typename T>
struct MetroArgs {
  DevGraph g;
  Dims m;
  int maxball[kMaxL + 1];
  int off_dh[kMaxL + 1];  // per-warp smem element offsets (elements of T) of dH^l rows, l < L
  int off_dy[kMaxL + 1];  // workspace element offsets of dY^l rows (l = 1..L) in the warp slot
  int off_x;              // per-warp smem element offset of the 4 staged dX rows (4 x 2F)
  int off_meta;           // per-warp smem byte offset of the row metadata
  int max_rows, max_span; // capacity of the metadata arrays (rows of ball_L, their neighbours)
  int warp_bytes;         // shared-memory bytes per warp
  int prop_rows;          // capacity of the proposal row arrays (4 x max degree, 0 without a network)
  int nwarps;             // warps (chains in flight) per CTA
  const T* theta;
  int8_t* chain_spins;
  int64_t C;
  int32_t n_sweeps, record_every;
  uint64_t seed, step0;
  int8_t* samples_out;
  double* logpsi_out;
  int32_t* n_acc;
  double* trace;
  T* gws;          // per warp slot: Y^1..Y^L [L][N][F], two H scratch layers [2][N][F], dY rows
  size_t ws_elems; // elements per warp slot
  const float* prop;  // learned proposal network or NULL (plain moves)
  double prop_eps;
};

__device__ __forceinline__ double m_tanh(double x) { return tanh(x); }
// float tanh: odd Taylor series through x^13 for |x| < 0.5 (truncation below 5e-7
// relative), else sgn(x) (1 - e)/(1 + e) with e = exp(-2|x|).
__device__ __forceinline__ float m_tanh(float x) {
  const float ax = fabsf(x);
  if (ax < 0.5f) {
    const float x2 = x * x;
    float p = 21844.f / 6081075.f;
    p = fmaf(p, x2, -1382.f / 155925.f);
    p = fmaf(p, x2, 62.f / 2835.f);
    p = fmaf(p, x2, -17.f / 315.f);
    p = fmaf(p, x2, 2.f / 15.f);
    p = fmaf(p, x2, -1.f / 3.f);
    return fmaf(p * x2, x, x);
  }
  const float e = __expf(-2.f * ax);
  return copysignf(__fdividef(1.f - e, 1.f + e), x);
}
__device__ __forceinline__ double m_exp(double x) { return exp(x); }
__device__ __forceinline__ float m_exp(float x) { return __expf(x); }
__device__ __forceinline__ double m_div(double a, double b) { return a / b; }
__device__ __forceinline__ float m_div(float a, float b) { return __fdividef(a, b); }

__device__ __forceinline__ void load4(const float* p, float* v) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x;
  v[1] = t.y;
  v[2] = t.z;
  v[3] = t.w;
}
__device__ __forceinline__ void load4(const double* p, double* v) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  const double2 b = *reinterpret_cast<const double2*>(p + 2);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}

template <typename T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// dH = tanh(y + dy) - tanh(y), in the stable form t (1 - H^2)/(1 + H t) built from
// e = exp(-2|y|); falls back to the direct difference when 1 + H t is small (a unit
// swinging across saturation, where dH is O(1) and the difference has no cancellation).
template <typename T>
__device__ __noinline__ T dtanh_far(T y, T dy) {
  return m_tanh(y + dy) - m_tanh(y);
}
template <typename T>
__device__ __forceinline__ T dtanh(T y, T dy) {
  const T e = m_exp((T)-2 * fabs(y));
  const T t = m_tanh(dy);
  const T sg = y < (T)0 ? (T)-1 : (T)1;
  const T ope = (T)1 + e;
  const T den = ope * (ope + sg * ((T)1 - e) * t);
  return den > (T)1e-3 ? m_div((T)4 * e * t, den) : dtanh_far(y, dy);
}

template <typename T>
__device__ inline bool m_accept_log(uint64_t r1, T log_ratio);
template <>
__device__ inline bool m_accept_log<double>(uint64_t r1, double log_ratio) {
  return (double)(r1 >> 11) * 0x1.0p-53 < exp(log_ratio);
}
template <>
__device__ inline bool m_accept_log<float>(uint64_t r1, float log_ratio) {
  return (float)(r1 >> 40) * 0x1.0p-24f < expf(log_ratio);
}

// Row index in [r0, r1) whose partner is `other`.
__device__ __forceinline__ int row_of(const int* ro, int r0, int r1, int other) {
  for (int r = r0; r < r1; ++r)
    if (ro[r] == other) return r;
  return r0;
}

template <typename T>
__device__ inline bool m_accept(uint64_t r1, T dre);
template <>
__device__ inline bool m_accept<double>(uint64_t r1, double dre) {
  return (double)(r1 >> 11) * 0x1.0p-53 < exp(2.0 * dre);
}
template <>
__device__ inline bool m_accept<float>(uint64_t r1, float dre) {
  return (float)(r1 >> 40) * 0x1.0p-24f < expf(2.0f * dre);
}


// ---- learned exchange proposal, evaluated by one warp ----------------------------------
__device__ __forceinline__ int spin_x(const int8_t* sp, int v, int a, int b) {
  return v == a ? sp[b] : (v == b ? sp[a] : sp[v]);
}

template <typename T>
__device__ T nsum(const DevGraph& g, const int8_t* sp, int v, int a, int b) {
  T acc = 0;
  const int k1 = __ldg(g.row_ptr + v + 1);
  for (int k = __ldg(g.row_ptr + v); k < k1; ++k) acc += (T)spin_x(sp, __ldg(g.col + k), a, b);
  return acc;
}

// Features of the ordered pair (i, j) in s, or in s with (a, b) exchanged when a >= 0.
template <typename T>
__device__ void pair_phi(const DevGraph& g, const int8_t* sp, int i, int j, int a, int b, T* f) {
  const int ki0 = __ldg(g.row_ptr + i), ki1 = __ldg(g.row_ptr + i + 1);
  const int kj0 = __ldg(g.row_ptr + j), kj1 = __ldg(g.row_ptr + j + 1);
  const int di = ki1 - ki0, dj = kj1 - kj0;
  const T si = (T)spin_x(sp, i, a, b), sj = (T)spin_x(sp, j, a, b);
  T Jij = 0, bi = 0, bj = 0;
  int ci = 0, cj = 0;
  for (int k = ki0; k < ki1; ++k) {
    const int u = __ldg(g.col + k);
    if (u == j) {
      Jij = (T)__ldg(g.J + __ldg(g.col_edge + k));
      continue;
    }
    bi += nsum<T>(g, sp, u, a, b) / (T)(__ldg(g.row_ptr + u + 1) - __ldg(g.row_ptr + u));
    ++ci;
  }
  for (int k = kj0; k < kj1; ++k) {
    const int u = __ldg(g.col + k);
    if (u == i) continue;
    bj += nsum<T>(g, sp, u, a, b) / (T)(__ldg(g.row_ptr + u + 1) - __ldg(g.row_ptr + u));
    ++cj;
  }
  f[0] = si;
  f[1] = sj;
  f[2] = Jij;
  f[3] = (T)1 / (T)di;
  f[4] = (T)1 / (T)dj;
  f[5] = (nsum<T>(g, sp, i, a, b) - sj) / (T)max(di - 1, 1);
  f[6] = (nsum<T>(g, sp, j, a, b) - si) / (T)max(dj - 1, 1);
  f[7] = ci ? bi / (T)ci : (T)0;
  f[8] = cj ? bj / (T)cj : (T)0;
}

// Sums of two products in the roundings that these logits have always had.
__device__ __forceinline__ float m_dot2(float a, float b, float c, float d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); }
__device__ __forceinline__ double m_dot2(double a, double b, double c, double d) { return __fma_rn(a, b, __dmul_rn(c, d)); }
__device__ __forceinline__ float m_dot2_last(float a, float b, float c, float d) {
  return __fmaf_rn(c, d, __fmul_rn(a, b));
}
__device__ __forceinline__ double m_dot2_last(double a, double b, double c, double d) {
  return __fma_rn(c, d, __dmul_rn(a, b));
}
template <typename T>
__device__ __noinline__ T m_tanh_call(T x) {
  return m_tanh(x);
}

// Logits of rows r < n of (rc[r] -> ro[r]) evaluated in the state selected by rx[r]
// (0: s, 1: s with (pa, pb) exchanged).  Returns the logit of row `lane` (and row lane+32).
// Four rows (float32) share the loads of the weights.  Not inlined (nor what else the proposal calls): a
// step passes through all of the kernel's code, which has to stay in the instruction caches.
template <typename T>
struct Logits {
  T lg0, lg1;
};
template <typename T>
__device__ __noinline__ Logits<T> warp_logits(const DevGraph& g, const int8_t* sp, const T* P, const int* rc,
                                              const int* ro, const int* rx, int n, int pa, int pb) {
  constexpr int kLogitRows = sizeof(T) == 4 ? 4 : 1;  // at a time; float64 has no registers for more
  const int lane = threadIdx.x & 31;
  const T* W1 = P + kPropOW1;
  const T* b1 = P + kPropOb1;
  const T* W2 = P + kPropOW2;
  const T* b2 = P + kPropOb2;
  const T* w3 = P + kPropOw3;
  Logits<T> out{0, 0};
  for (int base = 0; base < n; base += 32) {
    T f[kPropIn];
    const int r = base + lane;
    if (r < n) {
      pair_phi<T>(g, sp, rc[r], ro[r], rx[r] ? pa : -1, rx[r] ? pb : -1, f);
    } else {
#pragma unroll
      for (int q = 0; q < kPropIn; ++q) f[q] = 0;
    }
    const int cnt = min(32, n - base);
    for (int rr = 0; rr < cnt; rr += kLogitRows) {
      // hidden layer 1 (units lane, lane + 32) of rows base + rr ..
      T h0[kLogitRows], h1[kLogitRows], y0[kLogitRows], y1[kLogitRows];
#pragma unroll
      for (int i = 0; i < kLogitRows; ++i) {
        T z0 = b1[lane], z1 = b1[lane + 32];
#pragma unroll
        for (int q = 0; q < kPropIn; ++q) {
          const T x = __shfl_sync(0xffffffffu, f[q], rr + i);
          z0 += x * W1[q * kPropHid + lane];
          z1 += x * W1[q * kPropHid + lane + 32];
        }
        h0[i] = m_tanh_call(z0);
        h1[i] = m_tanh_call(z1);
        y0[i] = b2[lane];
        y1[i] = b2[lane + 32];
      }
      // hidden layer 2
#pragma unroll 2
      for (int q = 0; q < 32; ++q) {
        const T wa0 = W2[q * kPropHid + lane], wb0 = W2[(q + 32) * kPropHid + lane];
        const T wa1 = W2[q * kPropHid + lane + 32], wb1 = W2[(q + 32) * kPropHid + lane + 32];
#pragma unroll
        for (int i = 0; i < kLogitRows; ++i) {
          const T xa = __shfl_sync(0xffffffffu, h0[i], q);
          const T xb = __shfl_sync(0xffffffffu, h1[i], q);
          y0[i] += m_dot2(xa, wa0, xb, wb0);
          y1[i] += m_dot2(xa, wa1, xb, wb1);
        }
      }
#pragma unroll
      for (int i = 0; i < kLogitRows; ++i) {
        T z = m_dot2_last(m_tanh_call(y0[i]), w3[lane], m_tanh_call(y1[i]), w3[lane + 32]);
        z = wsum(z) + P[kPropOb3];
        if (lane == rr + i) {
          if (base == 0)
            out.lg0 = z;
          else
            out.lg1 = z;
        }
      }
    }
  }
  return out;
}

// Softmax probability of row `target_row` among rows [r0, r1) whose logits sit in lanes.
template <typename T>
__device__ __noinline__ T warp_softmax_prob(T lg0, T lg1, int r0, int r1, int target_row) {
  const int lane = threadIdx.x & 31;
  T zmax = -(T)INFINITY;
  for (int r = r0; r < r1; ++r) {
    const T z = __shfl_sync(0xffffffffu, r < 32 ? lg0 : lg1, r & 31);
    zmax = z > zmax ? z : zmax;
  }
  T sum = 0, pt = 0;
  for (int r = r0; r < r1; ++r) {
    const T z = __shfl_sync(0xffffffffu, r < 32 ? lg0 : lg1, r & 31);
    const T w = m_exp(z - zmax);
    sum += w;
    if (r == target_row) pt = w;
  }
  (void)lane;
  return pt / sum;
}

// Appends the antiparallel neighbours of i (in CSR order) as rows (i -> u, x); all lanes
// write the same values (warp-uniform), returns the new count.
__device__ __noinline__ int push_rows(const DevGraph& g, const int8_t* sp, int i, int x, int pa, int pb, int* rc, int* ro, int* rx,
                         int n) {
  const int a = x ? pa : -1, b = x ? pb : -1;
  const int si = spin_x(sp, i, a, b);
  const int k1 = __ldg(g.row_ptr + i + 1);
  for (int k = __ldg(g.row_ptr + i); k < k1; ++k) {
    const int u = __ldg(g.col + k);
    if (spin_x(sp, u, a, b) != si) {
      rc[n] = i;
      ro[n] = u;
      rx[n] = x;
      ++n;
    }
  }
  return n;
}

// Elements of the block's parameters: W (not with r8), its transpose, biases, embedding, readout.
__host__ __device__ inline size_t metro_param_elems(int F, bool r8) {
  const size_t n = (r8 ? 0 : (size_t)2 * F * (F + 1)) + (size_t)F * (2 * F + 4) + F + 2 * F + (F + 2) * 2 + 2;
  return (n + 3) / 4 * 4;
}
__host__ __device__ inline int metro_meta_ints(int rows, int span) { return (3 * rows + span + 5) / 4 * 4; }

// One layer of a proposal for one column a lane: rows [0, R) in groups of 8.  xs [2F][8]: the group's
// dX = [A_hat dH ; dH], feature k of rows 0..3 and 4..7 as two 16-byte halves that swap places
// every four k (the lanes' stores then spread over the banks).  Positions outside ball_{l-1} read the row of
// zeros behind it.  pre: the lane's part of Re Delta at the last layer.
__device__ __forceinline__ void metro_rows8(float* xs, const float* wt, const float* swr, const float* dprev,
                                            float* dcur, float* dyl, const float* Y, const int* mv, const int* mdeg,
                                            const int* mnb, const int2* nbw, int F, int R, int sprev, bool last,
                                            float& pre) {
  const int lane = threadIdx.x & 31;
  const bool has = lane < F;
  const int f = has ? lane : 0;
  for (int rb = 0; rb < R; rb += 8) {
    float yc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) yc[q] = Y[(size_t)mv[min(rb + q, R - 1)] * F + f];
    // two rows a turn: unrolled over all eight, this loop and the last one did not stay in the
    // instruction caches (with 14 warps at different places of the step)
#pragma unroll 1
    for (int p = 0; p < 4; ++p) {
      float ag[2], sf[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = min(rb + 2 * p + h, R - 1);
        const int2* nb = nbw + mnb[r];
        const int dg = mdeg[r];
        float s = 0.f;
#pragma unroll 1
        for (int t = 0; t < dg; ++t) {
          const int2 n = nb[t];
          s = fmaf(__int_as_float(n.y), dprev[min(n.x, sprev) * F + f], s);
        }
        ag[h] = s;
        sf[h] = dprev[min(r, sprev) * F + f];
      }
      if (has) {
        float2* x = reinterpret_cast<float2*>(xs);
        const int half = p >> 1;
        x[4 * lane + 2 * (half ^ ((lane >> 2) & 1)) + (p & 1)] = make_float2(ag[0], ag[1]);
        x[4 * (F + lane) + 2 * (half ^ (((F + lane) >> 2) & 1)) + (p & 1)] = make_float2(sf[0], sf[1]);
      }
    }
    __syncwarp();
    uint64_t acc[4] = {0, 0, 0, 0};
    const ulonglong2* x2 = reinterpret_cast<const ulonglong2*>(xs);
#pragma unroll 1
    for (int k = 0; k < 2 * F; k += 8) {
      float w[8];
      load4(wt + k, w);
      load4(wt + k + 4, w + 4);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint64_t w2 = f2_dup(w[u]);
        const ulonglong2 a = x2[2 * (k + u) + (u >> 2)], b = x2[2 * (k + u) + ((u >> 2) ^ 1)];
        acc[0] = f2_fma(a.x, w2, acc[0]);
        acc[1] = f2_fma(a.y, w2, acc[1]);
        acc[2] = f2_fma(b.x, w2, acc[2]);
        acc[3] = f2_fma(b.y, w2, acc[3]);
      }
    }
    __syncwarp();
#pragma unroll 1
    for (int r = rb; r < R && r < rb + 8; r += 2) {
      float ys[2];
      f2_unpack(acc[0], ys[0], ys[1]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!has || r + h >= R) break;
        const float d = dtanh(yc[h], ys[h]);
        dyl[(size_t)(r + h) * F + lane] = ys[h];
        if (last)
          pre += d * swr[2 * lane];
        else
          dcur[(size_t)(r + h) * F + lane] = d;
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) acc[i] = acc[i + 1];
#pragma unroll
      for (int i = 0; i < 6; ++i) yc[i] = yc[i + 2];
    }
  }
}

// log(a) - log(b)
__device__ __noinline__ double m_log_ratio(double a, double b) { return log(a) - log(b); }

// PROP: learned moves.  NF: feature columns of a lane (F <= 32 NF).  For one column of float32
// with F a multiple of 4 the layers take 8 rows at a time in packed multiply-adds (R8).
//
// What bounds it: instructions (some 30000 a learned step on a random graph of 65 sites, L 3, F 32) and
// their supply -- every warp is at another place of a step that was longer than the instruction
// caches (6 of 11 stall cycles an instruction).  So the learned and the plain kernel are apart,
// one-column code is not carried through two, rare and repeated pieces are calls, loops over a
// group's rows are rolled, and four rows of the network share the loads of its weights.  One sweep of
// 4096 chains with learned moves: 37.6 -> 21.7 ms; plain FP32 sweep of 4096 chains on Kagome 108,
// L 4, F 32: 18.2 -> 12.1; the two-column kernel gains from the calls alone (F 64, learned 10.4 -> 6.4).
template <typename T, bool PROP, int NF>
__global__ void __launch_bounds__(32 * kMetroMaxWarps) k_metro_warp(const MetroArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool R8 = sizeof(T) == 4 && NF == 1;
  const DevGraph& g = a.g;
  const Dims& m = a.m;
  const int N = m.N, F = m.F, L = m.L, E = m.E;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ldw = F + 1;
  // block-shared parameters: W (2F x F) and its transpose Wt (F x (2F + 4)) for 128-bit row loads
  const int ldt = 2 * F + 4;
  T* sW = (T*)smem;                  // [2F][F+1], not with R8
  T* sWt = sW + (R8 ? 0 : 2 * F * ldw);         // [F][2F+4]
  T* sb = sWt + F * ldt;             // [F]
  T* semb = sb + F;                  // [2][F]
  T* swr = semb + 2 * F;             // [(F+2)][2]
  T* sbr = swr + (F + 2) * 2;        // [2]
  const size_t param_pad = metro_param_elems(F, R8);
  T* sP = (T*)smem + param_pad;  // proposal network (when used)
  const size_t prop_pad = PROP ? ((size_t)kPropParams + 3) / 4 * 4 : 0;
  T* wbase = sP + prop_pad;
  unsigned char* wb = (unsigned char*)wbase + (size_t)warp * a.warp_bytes;
  T* wsm = (T*)wb;                                   // this warp's dH rows and staged dX rows
  T* sX = wsm + a.off_x;                             // [4][2F]
  int* mv = (int*)(wb + a.off_meta);                 // vertex of ball row r
  int* mdeg = mv + a.max_rows;                       // its degree
  int* mnb = mdeg + a.max_rows;                      // offset of its neighbour entries
  int* npos = mnb + a.max_rows;                      // per neighbour entry: position in the ball
  T* nwt = (T*)(mv + metro_meta_ints(a.max_rows, a.max_span));  // ... and normalised weight
  int2* nbw = (int2*)(mv + (3 * a.max_rows + 1) / 2 * 2);  // R8: both (position, weight bits)
  int* prc = (int*)(nwt + a.max_span);               // proposal rows: centre, partner, exchanged
  int* pro = prc + a.prop_rows;
  int* prx = pro + a.prop_rows;
  int8_t* spin = (int8_t*)(prx + a.prop_rows);
  const T* th = a.theta;
  for (int i = threadIdx.x; i < 2 * F * F; i += blockDim.x) {
    if (!R8) sW[(i / F) * ldw + i % F] = th[m.oW + i];
    sWt[(i % F) * ldt + i / F] = th[m.oW + i];
  }
  for (int i = threadIdx.x; i < F; i += blockDim.x) sb[i] = th[m.ob + i];
  for (int i = threadIdx.x; i < 2 * F; i += blockDim.x) semb[i] = m_tanh(th[m.oWe + i] + th[m.obe + i % F]);
  for (int i = threadIdx.x; i < (F + 2) * 2; i += blockDim.x) swr[i] = th[m.owr + i];
  if (threadIdx.x < 2) sbr[threadIdx.x] = th[m.obr + threadIdx.x];
  if (PROP)
    for (int i = threadIdx.x; i < kPropParams; i += blockDim.x) sP[i] = (T)a.prop[i];
  __syncthreads();

  const int64_t gwarp = (int64_t)blockIdx.x * a.nwarps + warp;
  const int64_t nwarps = (int64_t)gridDim.x * a.nwarps;
  T* Ybase = a.gws + (size_t)gwarp * a.ws_elems;  // Y^l at Ybase + (l-1)*N*F
  T* Hs0 = Ybase + (size_t)L * N * F;
  T* Hs1 = Hs0 + (size_t)N * F;
  T* dYg = Ybase;  // dY^l rows at dYg + off_dy[l]
  const int f0 = lane, f1 = lane + 32;
  const bool has0 = f0 < F, has1 = NF > 1 && f1 < F;
  const int64_t n_steps = (int64_t)a.n_sweeps * N;
  const int n_rec = a.record_every > 0 ? a.n_sweeps / a.record_every : 0;

  for (int64_t ch = gwarp; ch < a.C; ch += nwarps) {
    for (int v = lane; v < N; v += 32) spin[v] = a.chain_spins[ch * N + v];
    __syncwarp();
    // ---- forward: Y^1..Y^L of the chain's state (H scratch ping-pong) ----
    for (int v = 0; v < N; ++v) {
      const int c = spin[v] > 0 ? 0 : 1;
      if (has0) Hs0[(size_t)v * F + f0] = semb[c * F + f0];
      if (has1) Hs0[(size_t)v * F + f1] = semb[c * F + f1];
    }
    __syncwarp();
    for (int l = 1; l <= L; ++l) {
      const T* Hp = (l & 1) ? Hs0 : Hs1;
      T* Hn = (l & 1) ? Hs1 : Hs0;
      T* Y = Ybase + (size_t)(l - 1) * N * F;
      for (int v = 0; v < N; ++v) {
        T ag0 = 0, ag1 = 0;
        const int k1 = __ldg(g.row_ptr + v + 1);
        for (int k = __ldg(g.row_ptr + v); k < k1; ++k) {
          const T w = (T)__ldg(g.wd + k);
          const T* hu = Hp + (size_t)__ldg(g.col + k) * F;
          if (has0) ag0 += w * hu[f0];
          if (has1) ag1 += w * hu[f1];
        }
        const T sf0 = has0 ? Hp[(size_t)v * F + f0] : (T)0, sf1 = has1 ? Hp[(size_t)v * F + f1] : (T)0;
        T y0 = has0 ? sb[f0] : (T)0, y1 = has1 ? sb[f1] : (T)0;
        if (R8) {
          const T* wt = sWt + (size_t)(has0 ? f0 : 0) * ldt;
          for (int k4 = 0; k4 < F; k4 += 4) {
            T wa[4], wb[4];
            load4(wt + k4, wa);
            load4(wt + F + k4, wb);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const T av = __shfl_sync(0xffffffffu, ag0, k4 + u);
              const T sv = __shfl_sync(0xffffffffu, sf0, k4 + u);
              y0 += av * wa[u] + sv * wb[u];
            }
          }
        } else
        for (int kk = 0; kk < F; ++kk) {
          const T av = __shfl_sync(0xffffffffu, kk < 32 ? ag0 : ag1, kk & 31);
          const T sv = __shfl_sync(0xffffffffu, kk < 32 ? sf0 : sf1, kk & 31);
          if (has0) y0 += av * sW[kk * ldw + f0] + sv * sW[(F + kk) * ldw + f0];
          if (has1) y1 += av * sW[kk * ldw + f1] + sv * sW[(F + kk) * ldw + f1];
        }
        if (has0) {
          Y[(size_t)v * F + f0] = y0;
          Hn[(size_t)v * F + f0] = m_tanh(y0);
        }
        if (has1) {
          Y[(size_t)v * F + f1] = y1;
          Hn[(size_t)v * F + f1] = m_tanh(y1);
        }
      }
      __syncwarp();
    }
    int accepts = 0;
    uint64_t w0 = 0, w1 = 0, w2 = 0, w3 = 0;  // Philox words of step (k0 + lane)
    for (int64_t k = 0; k < n_steps; ++k) {
      if ((k & 31) == 0) {
        const U64x4 w = philox4x64_10(a.seed, (uint64_t)ch, U64x4{a.step0 + (uint64_t)(k + lane), 0, 0, 0});
        w0 = w.x;
        w1 = w.y;
        w2 = w.z;
        w3 = w.w;
      }
      const uint64_t r0 = __shfl_sync(0xffffffffu, w0, (int)(k & 31));
      const uint64_t r1 = __shfl_sync(0xffffffffu, w1, (int)(k & 31));
      int e = -1, kind = 1;
      bool move = false;
      T logq = 0;
      if (!PROP) {
        e = (int)__umul64hi(r0, (uint64_t)E);
        move = spin[__ldg(g.edges + 2 * e)] != spin[__ldg(g.edges + 2 * e + 1)];
      } else {
        const uint64_t r2 = __shfl_sync(0xffffffffu, w2, (int)(k & 31));
        const uint64_t r3 = __shfl_sync(0xffffffffu, w3, (int)(k & 31));
        const T eps = (T)a.prop_eps;
        int pi = -1, pj = -1, n = 0;
        T pij = 0, lg0 = 0, lg1 = 0;
        if ((double)(r3 >> 40) * 0x1.0p-24 < a.prop_eps) {
          e = (int)__umul64hi(r0, (uint64_t)E);
          pi = __ldg(g.edges + 2 * e);
          pj = __ldg(g.edges + 2 * e + 1);
          move = spin[pi] != spin[pj];
          if (move) n = push_rows(g, spin, pi, 0, pi, pj, prc, pro, prx, 0);
        } else {
          kind = 2;
          pi = (int)__umul64hi(r2, (uint64_t)N);
          const int n1 = push_rows(g, spin, pi, 0, -1, -1, prc, pro, prx, 0);
          __syncwarp();
          if (n1 > 0) {
            // the partner j ~ pi_i(. | s), by the categorical uniform (r3 mod 2^32) 2^-32
            const Logits<T> lg = warp_logits<T>(g, spin, sP, prc, pro, prx, n1, -1, -1);
            lg0 = lg.lg0;
            lg1 = lg.lg1;
            T zmax = -(T)INFINITY;
            for (int r = 0; r < n1; ++r) {
              const T z = __shfl_sync(0xffffffffu, r < 32 ? lg0 : lg1, r & 31);
              zmax = z > zmax ? z : zmax;
            }
            T sum = 0;
            for (int r = 0; r < n1; ++r) sum += m_exp(__shfl_sync(0xffffffffu, r < 32 ? lg0 : lg1, r & 31) - zmax);
            const T uc = (T)((double)(r3 & 0xFFFFFFFFull) * 0x1.0p-32);
            T cum = 0;
            int pick = n1 - 1;
            for (int r = 0; r < n1; ++r) {
              const T pr = m_exp(__shfl_sync(0xffffffffu, r < 32 ? lg0 : lg1, r & 31) - zmax) / sum;
              cum += pr;
              if (uc < cum) {
                pick = r;
                pij = pr;
                break;
              }
              if (r == n1 - 1) pij = pr;
            }
            pj = pro[pick];
            const int k1 = __ldg(g.row_ptr + pi + 1);
            for (int kk = __ldg(g.row_ptr + pi); kk < k1; ++kk)
              if (__ldg(g.col + kk) == pj) e = __ldg(g.col_edge + kk);
            move = true;
          }
          __syncwarp();
        }
        if (move) {
          // the exact mixture proposal density both ways: q(s -> s') and q(s' -> s)
          int g0 = n;  // rows [0, g0): cand(i, s) (plain moves only)
          n = push_rows(g, spin, pj, 0, pi, pj, prc, pro, prx, n);
          const int g1 = n;
          n = push_rows(g, spin, pi, 1, pi, pj, prc, pro, prx, n);
          const int g2 = n;
          n = push_rows(g, spin, pj, 1, pi, pj, prc, pro, prx, n);
          __syncwarp();
          const Logits<T> lg = warp_logits<T>(g, spin, sP, prc, pro, prx, n, pi, pj);
          lg0 = lg.lg0;
          lg1 = lg.lg1;
          const T p_ij = kind == 1 ? warp_softmax_prob<T>(lg0, lg1, 0, g0, row_of(pro, 0, g0, pj)) : pij;
          const T p_ji = warp_softmax_prob<T>(lg0, lg1, g0, g1, row_of(pro, g0, g1, pi));
          const T p_ij2 = warp_softmax_prob<T>(lg0, lg1, g1, g2, row_of(pro, g1, g2, pj));
          const T p_ji2 = warp_softmax_prob<T>(lg0, lg1, g2, n, row_of(pro, g2, n, pi));
          const T wl = ((T)1 - eps) / (T)N, wp = eps / (T)E;
          logq = (T)m_log_ratio((double)(wl * (p_ij2 + p_ji2) + wp), (double)(wl * (p_ij + p_ji) + wp));
        }
      }
      double* tr = a.trace ? a.trace + ((size_t)ch * n_steps + k) * 4 : nullptr;
      if (!move) {
        if (tr && lane == 0) {
          tr[0] = (double)e;
          tr[1] = 0.0;
          tr[2] = __longlong_as_double(0x7ff8000000000000ll);
          tr[3] = (double)kind;
        }
      } else {
        const int i = __ldg(g.edges + 2 * e), j = __ldg(g.edges + 2 * e + 1);
        const int bo = __ldg(g.ball_off + e);
        const int* bsz = g.ball_size + (size_t)e * (g.Lmax + 1);
        // layer 0: dH^0 rows (i, j)
        {
          T* d0 = wsm + a.off_dh[0];
          const int ci = spin[i] > 0 ? 0 : 1, cj = spin[j] > 0 ? 0 : 1;
          if (has0) {
            d0[f0] = semb[cj * F + f0] - semb[ci * F + f0];
            d0[F + f0] = semb[ci * F + f0] - semb[cj * F + f0];
          }
          if (has1) {
            d0[f1] = semb[cj * F + f1] - semb[ci * F + f1];
            d0[F + f1] = semb[ci * F + f1] - semb[cj * F + f1];
          }
          if (R8 && has0) d0[2 * F + f0] = 0;
          __syncwarp();
        }
        // row metadata of ball_L(e): vertex, degree, neighbour positions and weights
        const int RL = __ldg(bsz + L);
        const int nb_base = __ldg(g.row_nbr + bo);
        for (int r = lane; r < RL; r += 32) {
          const int v = __ldg(g.ball_vert + bo + r);
          const int k0 = __ldg(g.row_ptr + v), dg = __ldg(g.row_ptr + v + 1) - k0;
          const int o = __ldg(g.row_nbr + bo + r) - nb_base;
          mv[r] = v;
          mdeg[r] = dg;
          mnb[r] = o;
          for (int t = 0; t < dg; ++t) {
            const int p = __ldg(g.nbr_pos + nb_base + o + t);
            const T w = (T)__ldg(g.wd + k0 + t);
            if (R8) {
              nbw[o + t] = make_int2(p, __float_as_int((float)w));
            } else {
              npos[o + t] = p;
              nwt[o + t] = w;
            }
          }
        }
        __syncwarp();
        T pre = 0;
        for (int l = 1; l <= L; ++l) {
          const int sprev = __ldg(bsz + l - 1), R = __ldg(bsz + l);
          const T* dprev = wsm + a.off_dh[l - 1];
          T* dcur = l < L ? wsm + a.off_dh[l] : nullptr;
          T* dyl = dYg + a.off_dy[l];
          const T* Y = Ybase + (size_t)(l - 1) * N * F;
          if constexpr (R8) {
            if (l < L && has0) dcur[(size_t)R * F + f0] = 0;
            metro_rows8(sX, sWt + (size_t)(has0 ? f0 : 0) * ldt, swr, dprev, dcur, dyl, Y, mv, mdeg, mnb, nbw, F, R,
                        sprev, l == L, pre);
          } else
          for (int rb = 0; rb < R; rb += 4) {
            // stage dX = [A_hat dH^{l-1} ; dH^{l-1}] of rows rb..rb+3 (zeros past R)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int r = rb + q;
              T ag0 = 0, ag1 = 0, sf0 = 0, sf1 = 0;
              if (r < R) {
                const int o = mnb[r], dg = mdeg[r];
                for (int t = 0; t < dg; ++t) {
                  const int p = npos[o + t];
                  if (p < sprev) {
                    const T w = nwt[o + t];
                    if (has0) ag0 += w * dprev[(size_t)p * F + f0];
                    if (has1) ag1 += w * dprev[(size_t)p * F + f1];
                  }
                }
                if (r < sprev) {
                  if (has0) sf0 = dprev[(size_t)r * F + f0];
                  if (has1) sf1 = dprev[(size_t)r * F + f1];
                }
              }
              T* x = sX + q * 2 * F;
              if (has0) {
                x[f0] = ag0;
                x[F + f0] = sf0;
              }
              if (has1) {
                x[f1] = ag1;
                x[F + f1] = sf1;
              }
            }
            __syncwarp();
            // prefetch the cached pre-activations of the 4 rows (hidden behind the GEMM)
            T yc0[4], yc1[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int r = rb + q < R ? rb + q : R - 1;
              const T* yr = Y + (size_t)mv[r] * F;
              yc0[q] = has0 ? yr[f0] : (T)0;
              yc1[q] = has1 ? yr[f1] : (T)0;
            }
            // dY = dX W for the 4 rows (lane: output columns f0, f1), 4 inputs per load
            T y00 = 0, y10 = 0, y20 = 0, y30 = 0, y01 = 0, y11 = 0, y21 = 0, y31 = 0;
            const T* wt0 = sWt + (size_t)(has0 ? f0 : 0) * ldt;
            const T* wt1 = sWt + (size_t)(has1 ? f1 : 0) * ldt;
#pragma unroll 2
            for (int q = 0; q < 2 * F; q += 4) {
              T xa[4], xb[4], xc[4], xd[4], wa[4], wb[4];
              load4(sX + q, xa);
              load4(sX + 2 * F + q, xb);
              load4(sX + 4 * F + q, xc);
              load4(sX + 6 * F + q, xd);
              load4(wt0 + q, wa);
              if (has1) load4(wt1 + q, wb);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                y00 += xa[u] * wa[u];
                y10 += xb[u] * wa[u];
                y20 += xc[u] * wa[u];
                y30 += xd[u] * wa[u];
                if (has1) {
                  y01 += xa[u] * wb[u];
                  y11 += xb[u] * wb[u];
                  y21 += xc[u] * wb[u];
                  y31 += xd[u] * wb[u];
                }
              }
            }
            __syncwarp();
            const T ys0[4] = {y00, y10, y20, y30};
            const T ys1[4] = {y01, y11, y21, y31};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int r = rb + q;
              if (r >= R) break;
              if (has0) {
                const T d = dtanh(yc0[q], ys0[q]);
                dyl[(size_t)r * F + f0] = ys0[q];
                if (l < L)
                  dcur[(size_t)r * F + f0] = d;
                else
                  pre += d * swr[2 * f0];
              }
              if (has1) {
                const T d = dtanh(yc1[q], ys1[q]);
                dyl[(size_t)r * F + f1] = ys1[q];
                if (l < L)
                  dcur[(size_t)r * F + f1] = d;
                else
                  pre += d * swr[2 * f1];
              }
            }
          }
          __syncwarp();
        }
        const T dre = wsum(pre);
        T value;
        bool acc;
        if (PROP) {
          value = (T)2 * dre + logq;
          acc = m_accept_log<T>(r1, value);
        } else {
          value = dre;
          acc = m_accept<T>(r1, dre);
        }
        if (tr && lane == 0) {
          tr[0] = (double)e;
          tr[1] = acc ? 1.0 : 0.0;
          tr[2] = (double)value;
          tr[3] = (double)kind;
        }
        if (acc) {
          ++accepts;
          for (int l = 1; l <= L; ++l) {
            const int R = __ldg(bsz + l);
            const T* dy = dYg + a.off_dy[l];
            T* Y = Ybase + (size_t)(l - 1) * N * F;
            // four rows' loads before their stores (a ball's vertices are distinct)
            for (int r = 0; r < R; r += 4) {
              T y0[4], y1[4];
              int v[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int rr = r + q < R ? r + q : R - 1;
                v[q] = mv[rr];
                y0[q] = has0 ? Y[(size_t)v[q] * F + f0] + dy[(size_t)rr * F + f0] : (T)0;
                y1[q] = has1 ? Y[(size_t)v[q] * F + f1] + dy[(size_t)rr * F + f1] : (T)0;
              }
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                if (r + q >= R) break;
                if (has0) Y[(size_t)v[q] * F + f0] = y0[q];
                if (has1) Y[(size_t)v[q] * F + f1] = y1[q];
              }
            }
          }
          if (lane == 0) {
            const int8_t t = spin[i];
            spin[i] = spin[j];
            spin[j] = t;
          }
        }
        __syncwarp();
      }
      if ((k + 1) % N == 0 && a.record_every > 0) {
        const int sweep = (int)((k + 1) / N);
        if (sweep % a.record_every == 0) {
          const int rec = sweep / a.record_every - 1;
          if (rec < n_rec) {
            if (a.samples_out)
              for (int v = lane; v < N; v += 32) a.samples_out[((size_t)rec * a.C + ch) * N + v] = spin[v];
            if (a.logpsi_out) {
              // log Psi = sum_v [tanh(Y^L_v) ; onehot_v] . w_r + b_r
              const T* YL = Ybase + (size_t)(L - 1) * N * F;
              T z0 = 0, z1 = 0;
              int up = 0;
              for (int v = 0; v < N; ++v) {
                if (has0) z0 += L > 0 ? m_tanh(YL[(size_t)v * F + f0]) : semb[(spin[v] > 0 ? 0 : 1) * F + f0];
                if (has1) z1 += L > 0 ? m_tanh(YL[(size_t)v * F + f1]) : semb[(spin[v] > 0 ? 0 : 1) * F + f1];
                up += spin[v] > 0;
              }
              T re = (has0 ? z0 * swr[2 * f0] : (T)0) + (has1 ? z1 * swr[2 * f1] : (T)0);
              T im = (has0 ? z0 * swr[2 * f0 + 1] : (T)0) + (has1 ? z1 * swr[2 * f1 + 1] : (T)0);
              re = wsum(re);
              im = wsum(im);
              if (lane == 0) {
                const int dn = N - up;
                a.logpsi_out[((size_t)rec * a.C + ch) * 2] =
                    (double)(re + (T)up * swr[2 * F] + (T)dn * swr[2 * (F + 1)] + sbr[0]);
                a.logpsi_out[((size_t)rec * a.C + ch) * 2 + 1] =
                    (double)(im + (T)up * swr[2 * F + 1] + (T)dn * swr[2 * (F + 1) + 1] + sbr[1]);
              }
            }
          }
        }
      }
    }
    for (int v = lane; v < N; v += 32) a.chain_spins[ch * N + v] = spin[v];
    if (lane == 0 && a.n_acc) a.n_acc[ch] += accepts;
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------------
struct MetroPlan {
  int grid = 0;
  int smem = 0;
  int nwarps = 0;
  int warp_bytes = 0;
  int off_dh[kMaxL + 1] = {0};
  int off_dy[kMaxL + 1] = {0};
  int off_x = 0, off_meta = 0, max_rows = 0, max_span = 0, prop_rows = 0;
  size_t ws_elems = 0;
  size_t ws_bytes = 0;
};

// Columns a lane: one (with the packed rows) for F <= 32 and a multiple of 4.
static int metro_nf(int F) { return F <= 32 && F % 4 == 0 ? 1 : 2; }

template <typename T>
static const void* metro_kernel(int F, bool prop) {
  if (metro_nf(F) == 1)
    return prop ? (const void*)k_metro_warp<T, true, 1> : (const void*)k_metro_warp<T, false, 1>;
  return prop ? (const void*)k_metro_warp<T, true, 2> : (const void*)k_metro_warp<T, false, 2>;
}

template <typename T>
static gna_status metro_plan(const gna_graph* g, const Dims& m, int64_t C, int with_prop, MetroPlan* p) {
  // dX and W^T rows are read 4 features at a time, which needs 2F to be a multiple of 4
  if (m.L < 1 || m.F > 64 || m.F % 2 != 0) return GNA_ERR_UNSUPPORTED;
  // one W in shared memory for every layer: models with a W per layer take the CTA-per-chain sampler
  if (!m.shared && m.L > 1) return GNA_ERR_UNSUPPORTED;
  if (with_prop && g->max_deg > 16) return GNA_ERR_UNSUPPORTED;
  p->prop_rows = with_prop ? 4 * (g->max_deg > 0 ? g->max_deg : 1) : 0;
  DeviceInfo di;
  gna_status st = device_info(&di);
  if (st != GNA_OK) return st;
  const int F = m.F, L = m.L;
  const bool r8 = sizeof(T) == 4 && metro_nf(F) == 1;
  // per-warp shared memory: dH rows (l < L), 4 staged dX rows, row metadata, spins
  int o = 0;
  for (int l = 0; l < L; ++l) {
    p->off_dh[l] = o;
    o += (g->max_ball[l] + (r8 ? 1 : 0)) * F;  // r8: and a row of zeros
  }
  o = (o + 3) / 4 * 4;
  p->off_x = o;
  o += (r8 ? 8 : 4) * 2 * F;
  size_t bytes = (size_t)o * sizeof(T);
  bytes = (bytes + 15) / 16 * 16;
  p->off_meta = (int)bytes;
  p->max_rows = g->max_ball[L];
  p->max_span = g->max_span[L];
  const int meta_ints = metro_meta_ints(p->max_rows, p->max_span);  // keeps the weights 16-byte aligned
  bytes += (size_t)meta_ints * 4 + (size_t)p->max_span * sizeof(T) + (size_t)3 * p->prop_rows * 4 + (size_t)m.N;
  p->warp_bytes = (int)((bytes + 15) / 16 * 16);
  // per-warp workspace slot: Y^1..Y^L, two H scratch layers, dY^1..dY^L rows
  size_t e = (size_t)(L + 2) * m.N * F;
  for (int l = 1; l <= L; ++l) {
    p->off_dy[l] = (int)e;
    e += (size_t)g->max_ball[l] * F;
  }
  p->ws_elems = (e + 31) / 32 * 32;
  const size_t param_bytes = (metro_param_elems(F, r8) + (with_prop ? ((size_t)kPropParams + 3) / 4 * 4 : 0)) * sizeof(T);
  auto smem_for = [&](int nw) { return param_bytes + (size_t)nw * p->warp_bytes; };
  int nw = kMetroMaxWarps;
  while (nw > 0 && smem_for(nw) > (size_t)di.smem_optin - 1024) --nw;
  if (nw < 2) return GNA_ERR_UNSUPPORTED;
  // equal shares: the rounds over the chains that the most warps need, with as few warps as do them
  const int most = nw;
  const int64_t per_sm = (C + di.sms - 1) / di.sms, rounds = (per_sm + nw - 1) / nw;
  nw = (int)((per_sm + rounds - 1) / rounds);
  p->nwarps = nw;
  p->smem = (int)smem_for(nw);
  const void* kern = metro_kernel<T>(F, with_prop != 0);
  if ((st = allow_smem(kern, (uint64_t)di.smem_optin - 1024)) != GNA_OK) return st;
  int occ = 0;
  GNA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 32 * nw, p->smem));
  if (occ > kMetroMaxWarps / nw) occ = kMetroMaxWarps / nw;
  if (occ < 1) occ = 1;
  int64_t grid = (int64_t)di.sms * occ;
  const int64_t need = (C + nw - 1) / nw;
  if (grid > need) grid = need;
  if (grid < 1) grid = 1;
  p->grid = (int)grid;
  // The bytes of any number of chains up to C (fewer chains may be more warps): at most the warps that fit
  // an SM's shared memory, kMetroMaxWarps of them, or the chains with a last block part empty.
  int64_t slots = ((int64_t)di.smem_optin - (int64_t)param_bytes) / p->warp_bytes;
  slots = di.sms * (slots < kMetroMaxWarps ? slots : kMetroMaxWarps);
  if (slots > C + most - 1) slots = C + most - 1;
  p->ws_bytes = align_up((size_t)slots * p->ws_elems * sizeof(T));
  return GNA_OK;
}

gna_status metro_workspace(const gna_graph* g, const Dims& m, int prec, int64_t C, int with_prop, size_t* bytes) {
  if (C == 0) {
    *bytes = 0;
    return GNA_OK;
  }
  MetroPlan p;
  gna_status st = prec == GNA_PREC_FP64 ? metro_plan<double>(g, m, C, with_prop, &p)
                                        : metro_plan<float>(g, m, C, with_prop, &p);
  if (st != GNA_OK) return st;
  *bytes = p.ws_bytes;
  return GNA_OK;
}

template <typename T>
static gna_status metro_launch_t(const MetroCall& mc, void* ws, size_t ws_bytes, cudaStream_t stream) {
  MetroPlan p;
  gna_status st = metro_plan<T>(mc.g, mc.m, mc.C, mc.prop != nullptr, &p);
  if (st != GNA_OK) return st;
  if (ws_bytes < p.ws_bytes || !ws) return GNA_ERR_WORKSPACE;
  MetroArgs<T> a;
  a.g = mc.g->d;
  a.m = mc.m;
  for (int l = 0; l <= kMaxL; ++l) {
    a.maxball[l] = (l <= mc.m.L && l <= mc.g->d.Lmax) ? mc.g->max_ball[l] : 0;
    a.off_dh[l] = p.off_dh[l];
    a.off_dy[l] = p.off_dy[l];
  }
  a.off_x = p.off_x;
  a.off_meta = p.off_meta;
  a.max_rows = p.max_rows;
  a.max_span = p.max_span;
  a.warp_bytes = p.warp_bytes;
  a.prop_rows = p.prop_rows;
  a.prop = mc.prop;
  a.prop_eps = mc.prop_eps;
  a.nwarps = p.nwarps;
  a.theta = (const T*)mc.theta;
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
  a.gws = (T*)ws;
  a.ws_elems = p.ws_elems;
  void* args[] = {&a};
  GNA_CUDA_TRY(cudaLaunchKernel(metro_kernel<T>(mc.m.F, mc.prop != nullptr), dim3(p.grid), dim3(32 * p.nwarps), args,
                                p.smem, stream));
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

gna_status metro_run(const MetroCall& mc, int prec, void* ws, size_t ws_bytes, cudaStream_t stream) {
  if (mc.C == 0 || mc.n_sweeps == 0) return GNA_OK;
  return prec == GNA_PREC_FP64 ? metro_launch_t<double>(mc, ws, ws_bytes, stream)
                               : metro_launch_t<float>(mc, ws, ws_bytes, stream);
}

}  // namespace gna
