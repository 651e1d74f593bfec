// Float64 Metropolis sweeps (plain moves) and incremental local energy of tanh models with
// shared weights.  The exchange of a pair is propagated as in eloc.cu, product before gather:
//   dY^l_v = a_v sum_{u ~ v} (a_u Z_u[:F]) + Z_v[F:],  Z = dH^{l-1} [W[:F] | W[F:]],  a_v = 1/sqrt(d_v),
// with Z^0 = +-(emb(-1) - emb(+1)) [W[:F] | W[F:]] multiplied once per CTA.
//
// Bound: the FP64 pipe (2 lanes a clock and SM; a warp instruction takes 16 SM clocks).  What
// counts is the number of FP64 warp instructions and that no SM's pipe stands idle:
//   - the rows of ball_{l-1} are multiplied instead of those of ball_l (Kagome 2x2x3, L 2: 7 rows
//     a bond instead of 19);
//   - tanh(Y + x) - tanh(Y) comes from a rational tanh(x) and the cached H = tanh Y and 1 - H^2 with
//     one reciprocal (13 instructions an element, 20 with the updates of H and 1 - H^2 and 5 more when an
//     accepted move keeps them; exp, tanh and a division took 70);
//   - a warp holds 32 / F rows of F <= 16 features, not one;
//   - blocks of four warps, so that 1024 chains reach every SM (16 chains a block filled 64 SMs).
// Ten sweeps of 1024 chains, Kagome 2x2x3, L 2, F 16: 23.9 -> 3.01 ms (the general kernels before, these
// after); update of 1024 configurations 1.00 -> 0.88.
#include <climits>
#include <cmath>
#include <cstring>

#include "dbl.cuh"

namespace gna {

namespace {

constexpr int kDbThreads = 128;
constexpr int kDbWarps = kDbThreads / 32;
constexpr int kDbBatch = 256;  // bonds of the local energy whose Delta are kept at a time

struct DbArgs {
  DevGraph g;
  Dims m;
  const double* theta;
  int units, uw;      // units per CTA, warps per unit
  int lpr, fpl;       // lanes per row (a power of two), features per lane
  uint32_t oW, ob, oemb, owr, obr, oav, oz0, olist, ores, ounit;
  uint32_t unit_bytes, uz[2], ud, usum, uspin;
  double* ws;
  size_t ws_unit;     // doubles per unit (sampler) or per CTA (local energy)
  size_t off_new[kMaxL + 1], off_h;  // within it: new rows of layer l, the forward's row buffers
  // sampler
  int8_t* chain_spins;
  int64_t B;          // chains or configurations
  int n_sweeps, record_every;
  uint64_t seed, step0;
  int8_t* samples_out;
  double* logpsi_out;
  int32_t* n_acc;
  double* trace;
  // local energy
  const int8_t* spins;
  double* eloc;
  float* dlogpsi;
};

extern __shared__ __align__(16) unsigned char db_smem[];

struct DbCtx {
  const DbArgs* a;
  const double *W, *b, *emb, *wr, *br, *av, *z0;
  int lane, f, row_in_warp, rows_per_warp;
};

__device__ __forceinline__ double db_rcp(double d) {
  double r;  // about 20 bits; the cubic step leaves 60
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double db_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// H = tanh y and S = 1 - H^2 (its relative precision kept at saturation) from e = exp(-2 |y|).
__device__ __forceinline__ double2 db_cache(double y) {
  const double e = exp(-2.0 * fabs(y)), r = db_rcp(1.0 + e);
  return make_double2(copysign((1.0 - e) * r, y), 4.0 * e * (r * r));
}

// dH = tanh(Y + x) - tanh(Y) = t S/(1 + H t), t = tanh x, from H = tanh Y and S = 1 - H^2; NEXT also
// the new H and S = S (1 - t^2)/(1 + H t)^2.  t = w/Q by a convergent of Lambert's continued
// fraction: the sixth (relative error 4e-17 up to |x| = 1/4) or the ninth (3e-17 up to 1), chosen
// for the whole warp.  Beyond 1 from X = exp(-2 |x|), with 1 + H t summed without cancellation; where S
// is below kDbTiny (|Y| > 345; or not a number) it no longer says how far out the unit is, tanh Y = sgn Y
// and dH = -2 sgn Y/(1 + exp(2 sgn Y (Y + x))), from Y at *py.
constexpr double kDbTiny = 1e-300;
__device__ __forceinline__ bool db_cached(double S) { return S >= kDbTiny; }
template <bool NEXT>
__device__ __forceinline__ double db_dtanh(double x, double2 hs, const double* py, double2& next) {
  const int hx = __double2hiint(x) & 0x7fffffff;
  const double z = x * x, H = hs.x, S = hs.y;
  double w, Q;
  if (!__any_sync(0xffffffffu, hx > 0x3fd00000)) {
    w = x * fma(z, fma(z, 21.0, 1260.0), 10395.0);
    Q = fma(z, fma(z, z + 210.0, 4725.0), 10395.0);
  } else {
    w = x * fma(z, fma(z, fma(z, z + 990.0, 135135.0), 4729725.0), 34459425.0);
    Q = fma(z, fma(z, fma(z, fma(z, 45.0, 13860.0), 945945.0), 16216200.0), 34459425.0);
  }
  const double r = db_rcp(fma(H, w, Q)), u = S * r;
  double d = w * u;
  if (NEXT) next = make_double2(H + d, (u * r) * ((Q - w) * (Q + w)));
  if (hx > 0x3ff00000) {  // (also what is not a number, which stays one)
    const bool in = db_cached(S);
    const double y = in ? 0.0 : *py, sg = copysign(1.0, y);
    const double X = exp(in ? -2.0 * fabs(x) : 2.0 * sg * (y + x)), x1 = 1.0 / (1.0 + X);
    if (in) {
      const double t = copysign((1.0 - X) * x1, x), ah = fabs(H);
      const double D = (x < 0.0) == (H < 0.0) ? 1.0 + ah * fabs(t) : S / (1.0 + ah) + ah * (2.0 * X * x1);
      const double v = S / D;  // (D is at least half of S)
      d = t * v;
      if (NEXT) next = make_double2(H + d, v / D * (4.0 * X * (x1 * x1)));
    } else {
      d = -2.0 * sg * x1;
      if (NEXT) next = make_double2(sg * (X - 1.0) * x1, 4.0 * (X * x1) * x1);
    }
    if (x != x) d = x;
  }
  return d;
}

// The pair (H, S) of a move that is kept, back on S = 1 - H^2.  The factors of db_dtanh leave it by a
// rounding, and the next ones enlarge what it is off: left alone it grew 1.5 times a sweep, until after some
// 100 sweeps (Kagome 2x2x3, weight scale 0.3) H had no correct digit.  H decides below 0.75 and S above,
// where it has the digits; what is left is a random walk of roundings, like that of Y (1e-14 after 10^4 moves).
__device__ __forceinline__ double2 db_settle(double h, double s) {
  if (fabs(h) < 0.75)
    s = fma(-h, h, 1.0);
  else
    h = fma(0.5 * fma(-h, h, 1.0 - s), h, h);
  return make_double2(h, s);
}

// FINITE_W: an infinite weight becomes one that saturates tanh as well, so that a unit whose input does not change
// stays out of the energy (0 w = 0), as where the rows are recomputed.
template <bool FINITE_W>
__device__ void db_setup(const DbArgs& a, DbCtx& c) {
  const int F = a.m.F, N = a.m.N;
  const double* th = a.theta;
  double* W = (double*)(db_smem + a.oW);
  double* b = (double*)(db_smem + a.ob);
  double* emb = (double*)(db_smem + a.oemb);
  double* wr = (double*)(db_smem + a.owr);
  double* br = (double*)(db_smem + a.obr);
  double* av = (double*)(db_smem + a.oav);
  double* z0 = (double*)(db_smem + a.oz0);
  for (int i = threadIdx.x; i < 2 * F * F; i += blockDim.x) {
    const double w = th[a.m.oW + i];
    W[i] = FINITE_W && fabs(w) == INFINITY ? copysign(1e200, w) : w;
  }
  for (int i = threadIdx.x; i < F; i += blockDim.x) b[i] = th[a.m.ob + i];
  for (int i = threadIdx.x; i < 2 * F; i += blockDim.x) emb[i] = tanh(th[a.m.oWe + i] + th[a.m.obe + i % F]);
  for (int i = threadIdx.x; i < (F + 2) * 2; i += blockDim.x) wr[i] = th[a.m.owr + i];
  if (threadIdx.x < 2) br[threadIdx.x] = th[a.m.obr + threadIdx.x];
  for (int v = threadIdx.x; v < N; v += blockDim.x) {
    const int d = __ldg(a.g.row_ptr + v + 1) - __ldg(a.g.row_ptr + v);
    av[v] = d > 0 ? 1.0 / sqrt((double)d) : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * F; i += blockDim.x) {
    const int f = i % F, top = i < F ? 0 : F;
    double z = 0.0;
    for (int k = 0; k < F; ++k) z = fma(emb[F + k] - emb[k], W[(top + k) * F + f], z);
    z0[i] = z;
  }
  __syncthreads();
  c.a = &a;
  c.W = W;
  c.b = b;
  c.emb = emb;
  c.wr = wr;
  c.br = br;
  c.av = av;
  c.z0 = z0;
  c.lane = threadIdx.x & 31;
  c.f = c.lane & (a.lpr - 1);
  c.row_in_warp = c.lane / a.lpr;
  c.rows_per_warp = 32 / a.lpr;
}

// One row of features times W: out[j] = sum_k x_k W[k][f + 32 j], x broadcast from shared memory.
template <int FPL>
__device__ __forceinline__ void db_rowmul(const double* x, const double* W, int F, const int* fs, double* out) {
#pragma unroll 4
  for (int k = 0; k < F; ++k) {
    const double y = x[k];
#pragma unroll
    for (int j = 0; j < FPL; ++j) out[j] = fma(y, W[k * F + fs[j]], out[j]);
  }
}

// Forward of spins sp by `nwarps` warps (this one is `warp`): (H, 1 - H^2) of every layer into the cache, and
// Y (all of it with KEEP_Y, else of the units whose 1 - H^2 does not say how far out they are).  Hb: two row
// buffers [N][F]; xs: this warp's staging rows [rows_per_warp][2 F].
template <int FPL, bool KEEP_Y, typename Sync>
__device__ const double* db_forward(const DbCtx& c, const int8_t* sp, double* Yc, double2* Hc, double* Hb, double* xs,
                                    int warp, int nwarps, Sync sync) {
  const DbArgs& a = *c.a;
  const int N = a.m.N, F = a.m.F, L = a.m.L, R = c.rows_per_warp;
  const DevGraph& g = a.g;
  double* Hp = Hb;
  double* Hn = Hb + (size_t)N * F;
  int fs[FPL];
  bool has[FPL];
#pragma unroll
  for (int j = 0; j < FPL; ++j) {
    has[j] = c.f + 32 * j < F;
    fs[j] = has[j] ? c.f + 32 * j : 0;
  }
  for (int v = warp * R + c.row_in_warp; v < N; v += nwarps * R)
#pragma unroll
    for (int j = 0; j < FPL; ++j)
      if (has[j]) Hp[(size_t)v * F + fs[j]] = c.emb[(sp[v] > 0 ? 0 : F) + fs[j]];
  sync();
  double* x = xs + c.row_in_warp * 2 * F;
  for (int l = 1; l <= L; ++l) {
    for (int v0 = warp * R; v0 < N; v0 += nwarps * R) {
      const int v = min(v0 + c.row_in_warp, N - 1);
      double ag[FPL], y[FPL];
#pragma unroll
      for (int j = 0; j < FPL; ++j) ag[j] = 0.0;
      const int k1 = __ldg(g.row_ptr + v + 1);
      for (int k = __ldg(g.row_ptr + v); k < k1; ++k) {
        const double w = __ldg(g.wd + k);
        const double* h = Hp + (size_t)__ldg(g.col + k) * F;
#pragma unroll
        for (int j = 0; j < FPL; ++j) ag[j] = fma(w, h[fs[j]], ag[j]);
      }
#pragma unroll
      for (int j = 0; j < FPL; ++j) {
        y[j] = c.b[fs[j]];
        if (has[j]) {
          x[fs[j]] = ag[j];
          x[F + fs[j]] = Hp[(size_t)v * F + fs[j]];
        }
      }
      __syncwarp();
      db_rowmul<FPL>(x, c.W, F, fs, y);
      db_rowmul<FPL>(x + F, c.W + F * F, F, fs, y);
#pragma unroll
      for (int j = 0; j < FPL; ++j) {
        if (has[j] && v0 + c.row_in_warp < N) {
          const size_t i = ((size_t)(l - 1) * N + v) * F + fs[j];
          const double2 hs = db_cache(y[j]);
          if (KEEP_Y || !db_cached(hs.y)) Yc[i] = y[j];
          Hc[i] = hs;
          Hn[(size_t)v * F + fs[j]] = hs.x;
        }
      }
      __syncwarp();
    }
    sync();
    double* t = Hp;
    Hp = Hn;
    Hn = t;
  }
  return Hp;
}

// Delta log Psi of exchanging the ends of the bond whose record is in `info` (lane i holds int i of
// DevGraph::bond_info): this warp's lanes' parts of (Re, Im when IM).  NEXT: the rows' new Y, H
// and 1 - H^2 into the unit's new rows.  uo: byte offset of the unit's shared memory.
template <int FPL, bool NEXT, bool IM, typename Sync>
__device__ __forceinline__ void db_delta(const DbCtx& c, int info, const int8_t* sp, const double* Yc, const double2* Hc,
                                         double* wsu, uint32_t uo, int uwarp, Sync sync, double& sre, double& sim) {
  const DbArgs& a = *c.a;
  const int N = a.m.N, F = a.m.F, L = a.m.L, R = c.rows_per_warp, uthreads = a.uw * 32;
  const DevGraph& g = a.g;
  auto field = [&](int i) { return __shfl_sync(0xffffffffu, info, i); };
  const int* rec = g.rec + 2 * (size_t)field(0);
  const uint32_t* pairs = g.pairs + field(1);
  const int bi = field(4), bj = field(5);
  double* z[2] = {(double*)(db_smem + uo + a.uz[0]), (double*)(db_smem + uo + a.uz[1])};
  double* ds = (double*)(db_smem + uo + a.ud) + (uwarp * R + c.row_in_warp) * F;
  int fs[FPL];
  bool has[FPL];
#pragma unroll
  for (int j = 0; j < FPL; ++j) {
    has[j] = c.f + 32 * j < F;
    fs[j] = has[j] ? c.f + 32 * j : 0;
  }
  for (int i = uwarp * 32 + c.lane; i < 6 * F; i += uthreads) {  // Z^0: rows i and j, then the zero row
    const int r = i / (2 * F), k = i - r * 2 * F, v = r ? bj : bi;
    z[0][i] = r < 2 ? (sp[v] > 0 ? c.z0[k] : -c.z0[k]) * (k < F ? c.av[v] : 1.0) : 0.0;
  }
  sync();
  int prev = 2;
  for (int l = 1; l <= L; ++l) {
    const int n = field(8 + l);
    const double* zi = (l & 1) ? z[0] : z[1];
    double* zo = (l & 1) ? z[1] : z[0];
    for (int r0 = uwarp * R; r0 < n; r0 += a.uw * R) {
      const int r = min(r0 + c.row_in_warp, n - 1);
      const bool ok = r0 + c.row_in_warp < n;
      const int2 rc = __ldg(reinterpret_cast<const int2*>(rec) + r);
      const int v = rc.x & 0xFFFF, np = rc.x >> 16;
      double x[FPL], dv[FPL];
#pragma unroll
      for (int j = 0; j < FPL; ++j) x[j] = 0.0;
      for (int k = 0; k < np; ++k) {
        const uint32_t w = __ldg(pairs + rc.y + k);
        const int p0 = min((int)(w & 0xFFFFu) >> 2, prev), p1 = min((int)(w >> 18), prev);
#pragma unroll
        for (int j = 0; j < FPL; ++j) {
          x[j] += zi[p0 * 2 * F + fs[j]];
          x[j] += zi[p1 * 2 * F + fs[j]];
        }
      }
      const double av = c.av[v];
      const size_t ci = ((size_t)(l - 1) * N + v) * F;
#pragma unroll
      for (int j = 0; j < FPL; ++j) {
        x[j] = fma(av, x[j], zi[min(r, prev) * 2 * F + F + fs[j]]);
        double2 nx;
        dv[j] = db_dtanh<NEXT>(x[j], Hc[ci + fs[j]], Yc + ci + fs[j], nx);
        if (NEXT && ok && has[j]) {
          const double Yn = Yc[ci + fs[j]] + x[j];
          // far out, where 1 - H^2 nears the end of the exponents, from Y itself
          if ((__double2hiint(Yn) & 0x7fffffff) >= 0x4062c000) nx = db_cache(Yn);  // |Y| >= 150
          double* nw = wsu + a.off_new[l] + ((size_t)r * F + fs[j]) * 3;
          nw[0] = Yn;
          nw[1] = nx.x;
          nw[2] = nx.y;
        }
      }
      if (l == L) {
#pragma unroll
        for (int j = 0; j < FPL; ++j)
          if (ok && has[j]) {
            sre = fma(dv[j], c.wr[2 * fs[j]], sre);
            if (IM) sim = fma(dv[j], c.wr[2 * fs[j] + 1], sim);
          }
        continue;
      }
#pragma unroll
      for (int j = 0; j < FPL; ++j)
        if (has[j]) ds[fs[j]] = dv[j];
      __syncwarp();
      double zt[FPL], zb[FPL];
#pragma unroll
      for (int j = 0; j < FPL; ++j) zt[j] = zb[j] = 0.0;
      db_rowmul<FPL>(ds, c.W, F, fs, zt);
      db_rowmul<FPL>(ds, c.W + F * F, F, fs, zb);
#pragma unroll
      for (int j = 0; j < FPL; ++j)
        if (ok && has[j]) {
          zo[(size_t)r * 2 * F + fs[j]] = av * zt[j];
          zo[(size_t)r * 2 * F + F + fs[j]] = zb[j];
        }
      __syncwarp();
    }
    if (l < L)
      for (int i = uwarp * 32 + c.lane; i < 2 * F; i += uthreads) zo[(size_t)n * 2 * F + i] = 0.0;
    sync();
    prev = n;
  }
}

// ---------------------------------------------------------------------------------
// Metropolis sweeps: a unit of warps runs a chain at a time (the move rule of the other samplers)
// ---------------------------------------------------------------------------------
template <int FPL>
__global__ void __launch_bounds__(kDbThreads) k_db_metro(const __grid_constant__ DbArgs a) {
  DbCtx c;
  db_setup<false>(a, c);
  const int N = a.m.N, F = a.m.F, L = a.m.L, E = a.m.E, lane = c.lane;
  const int warp = threadIdx.x >> 5, h = warp / a.uw, uwarp = warp % a.uw, uthreads = a.uw * 32, utid = threadIdx.x - h * uthreads;
  if (h >= a.units) return;
  const uint32_t uo = a.ounit + (uint32_t)h * a.unit_bytes;
  int8_t* sp = (int8_t*)(db_smem + uo + a.uspin);
  double* sum = (double*)(db_smem + uo + a.usum);
  auto sync = [&]() {
    if (a.uw == 1)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(1 + h), "r"(uthreads) : "memory");
  };
  double* wsu = a.ws + ((size_t)blockIdx.x * a.units + h) * a.ws_unit;
  const size_t NF = (size_t)N * F;
  double2* Hc = (double2*)wsu;
  double* Yc = wsu + 2 * L * NF;
  const int64_t n_steps = (int64_t)a.n_sweeps * N, rec_steps = (int64_t)a.record_every * N;
  const int64_t n_rec = a.record_every > 0 ? a.n_sweeps / a.record_every : 0;
  for (int64_t ch = (int64_t)blockIdx.x * a.units + h; ch < a.B; ch += (int64_t)gridDim.x * a.units) {
    for (int v = utid; v < N; v += uthreads) sp[v] = a.chain_spins[ch * N + v];
    sync();
    db_forward<FPL, true>(c, sp, Yc, Hc, wsu + a.off_h, (double*)(db_smem + uo + a.uz[0]) + (size_t)uwarp * c.rows_per_warp * 2 * F, uwarp,
                    a.uw, sync);
    int accepts = 0;
    int64_t base = -32, k = 0, rec = 0;
    int e = 0, ei = 0, ej = 0;  // this lane's step base + lane
    uint64_t r1 = 0;
    while (k < n_steps) {
      if (k >= base + 32) {
        base = k;
        const U64x4 w = philox4x64_10(a.seed, (uint64_t)ch, U64x4{a.step0 + (uint64_t)(base + lane), 0, 0, 0});
        e = (int)__umul64hi(w.x, (uint64_t)E);
        r1 = w.y;
        const int2 ij = __ldg(reinterpret_cast<const int2*>(a.g.edges) + e);
        ei = ij.x;
        ej = ij.y;
      }
      int64_t stop = min(base + 32, n_steps);
      if (rec < n_rec) stop = min(stop, (rec + 1) * rec_steps);
      const int64_t s = base + lane;
      const bool in = s >= k && s < stop;
      const unsigned mask = __ballot_sync(0xffffffffu, in && sp[ei] != sp[ej]);
      const int64_t ks = mask ? base + __ffs(mask) - 1 : stop;
      if (a.trace && uwarp == 0 && in && s < ks) {  // parallel bonds: rejected steps
        double* tr = a.trace + ((size_t)ch * n_steps + s) * 4;
        tr[0] = (double)e;
        tr[1] = 0.0;
        tr[2] = __longlong_as_double(0x7ff8000000000000ll);
        tr[3] = 1.0;
      }
      k = ks;
      if (mask) {
        const int src = __ffs(mask) - 1;
        const int eb = __shfl_sync(0xffffffffu, e, src);
        const uint64_t u1 = __shfl_sync(0xffffffffu, r1, src);
        const int info = __ldg(a.g.bond_info + (size_t)eb * 32 + lane);
        double dre = 0.0, dim = 0.0;
        db_delta<FPL, true, false>(c, info, sp, Yc, Hc, wsu, uo, uwarp, sync, dre, dim);
        dre = db_sum(dre);
        if (a.uw > 1) {
          if (lane == 0) sum[uwarp] = dre;
          sync();
          dre = 0.0;
          for (int w = 0; w < a.uw; ++w) dre += sum[w];
        }
        // u < exp(2 Delta): the float32 exponential decides unless it is too close to u
        const double u = (double)(u1 >> 11) * 0x1.0p-53;
        bool acc = dre >= 0.0;
        if (!acc) {
          const double ef = (double)expf((float)(2.0 * dre));
          acc = u < ef * (1.0 - 1e-5);
          if (!acc && !(u > ef * (1.0 + 1e-5) + 1e-37)) acc = u < exp(2.0 * dre);
        }
        if (a.trace && utid == 0) {
          double* tr = a.trace + ((size_t)ch * n_steps + k) * 4;
          tr[0] = (double)eb;
          tr[1] = acc ? 1.0 : 0.0;
          tr[2] = dre;
          tr[3] = 1.0;
        }
        if (acc) {
          ++accepts;
          const int* rc = a.g.rec + 2 * (size_t)__shfl_sync(0xffffffffu, info, 0);
          for (int l = 1; l <= L; ++l) {
            const int n = __shfl_sync(0xffffffffu, info, 8 + l) * F;
            const double* nw = wsu + a.off_new[l];
            for (int i = utid; i < n; i += uthreads) {
              const int r = i / F;
              const size_t o = (size_t)(l - 1) * NF + (size_t)(__ldg(rc + 2 * r) & 0xFFFF) * F + (i - r * F);
              Yc[o] = nw[3 * i];
              Hc[o] = db_settle(nw[3 * i + 1], nw[3 * i + 2]);
            }
          }
          if (utid == 0) {
            const int i = __ldg(a.g.edges + 2 * eb), j = __ldg(a.g.edges + 2 * eb + 1);
            const int8_t t = sp[i];
            sp[i] = sp[j];
            sp[j] = t;
          }
        }
        sync();
        ++k;
      }
      if (rec < n_rec && k == (rec + 1) * rec_steps) {
        if (a.samples_out)
          for (int v = utid; v < N; v += uthreads) a.samples_out[((size_t)rec * a.B + ch) * N + v] = sp[v];
        if (a.logpsi_out) {
          const double2* HL = Hc + (L - 1) * NF;
          double re = 0.0, im = 0.0;
          for (int i = utid; i < (int)NF; i += uthreads) {
            const int f = i % F;
            const double hv = HL[i].x;
            re = fma(hv, c.wr[2 * f], re);
            im = fma(hv, c.wr[2 * f + 1], im);
          }
          re = db_sum(re);
          im = db_sum(im);
          if (a.uw > 1) {
            if (lane == 0) {
              sum[2 * uwarp] = re;
              sum[2 * uwarp + 1] = im;
            }
            sync();
            re = im = 0.0;
            for (int w = 0; w < a.uw; ++w) {
              re += sum[2 * w];
              im += sum[2 * w + 1];
            }
          }
          int up = 0;
          for (int v = lane; v < N; v += 32) up += sp[v] > 0;
          up = __reduce_add_sync(0xffffffffu, up);
          if (utid == 0) {
            double* o = a.logpsi_out + ((size_t)rec * a.B + ch) * 2;
            o[0] = re + (double)up * c.wr[2 * F] + (double)(N - up) * c.wr[2 * (F + 1)] + c.br[0];
            o[1] = im + (double)up * c.wr[2 * F + 1] + (double)(N - up) * c.wr[2 * (F + 1) + 1] + c.br[1];
          }
        }
        ++rec;
        sync();
      }
    }
    for (int v = utid; v < N; v += uthreads) a.chain_spins[ch * N + v] = sp[v];
    if (utid == 0 && a.n_acc) a.n_acc[ch] += accepts;
    sync();
  }
}

// ---------------------------------------------------------------------------------
// Incremental local energy: a CTA per configuration, its units take the antiparallel bonds in turn
// ---------------------------------------------------------------------------------
template <int FPL>
__global__ void __launch_bounds__(kDbThreads) k_db_eloc(const __grid_constant__ DbArgs a) {
  __shared__ int s_cnt[kDbWarps];
  __shared__ double s_e[3 * kDbWarps];
  DbCtx c;
  db_setup<true>(a, c);
  const int N = a.m.N, F = a.m.F, L = a.m.L, E = a.m.E, lane = c.lane;
  const int warp = threadIdx.x >> 5, h = warp / a.uw, uwarp = warp % a.uw, uthreads = a.uw * 32;
  const bool active = h < a.units;
  const uint32_t uo = a.ounit + (uint32_t)(active ? h : 0) * a.unit_bytes;
  double* sum = (double*)(db_smem + uo + a.usum);
  int8_t* sp = (int8_t*)(db_smem + a.ounit + a.uspin);  // the first unit's: one configuration per CTA
  uint16_t* list = (uint16_t*)(db_smem + a.olist);
  auto sync = [&]() {
    if (a.uw == 1)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(1 + h), "r"(uthreads) : "memory");
  };
  double* wsu = a.ws + (size_t)blockIdx.x * a.ws_unit;
  double2* Hc = (double2*)wsu;
  double* Yc = wsu + 2 * L * (size_t)N * F;
  for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) {
    for (int v = threadIdx.x; v < N; v += kDbThreads) sp[v] = a.spins[b * N + v];
    if (a.dlogpsi)
      for (int e = threadIdx.x; e < E; e += kDbThreads) a.dlogpsi[b * E + e] = 0.f;
    __syncthreads();
    db_forward<FPL, false>(c, sp, Yc, Hc, wsu + a.off_h,
                    (double*)(db_smem + a.ounit + (size_t)(a.units - 1) * a.unit_bytes + a.ud) + (size_t)warp * c.rows_per_warp * 2 * F,
                    warp, kDbWarps, [] { __syncthreads(); });
    // antiparallel bonds in order, and the diagonal energy
    double diag = 0.0;
    int na = 0;
    for (int base = 0; base < E; base += kDbThreads) {
      const int e = base + (int)threadIdx.x;
      bool anti = false;
      if (e < E) {
        const int2 ij = __ldg(reinterpret_cast<const int2*>(a.g.edges) + e);
        const int si = sp[ij.x], sj = sp[ij.y];
        anti = si != sj;
        diag += bond_diag(a.g, e, si, sj);
      }
      const unsigned mask = __ballot_sync(0xffffffffu, anti);
      if (lane == 0) s_cnt[warp] = __popc(mask);
      __syncthreads();
      int before = na, all = na;
      for (int w = 0; w < kDbWarps; ++w) {
        before += w < warp ? s_cnt[w] : 0;
        all += s_cnt[w];
      }
      if (anti) list[before + __popc(mask & ((1u << lane) - 1u))] = (uint16_t)e;
      na = all;
      __syncthreads();
    }
    // Delta of up to kDbBatch bonds at a time, then one warp's worth of exponentials for 32 of them
    double er = 0.0, ei = 0.0;
    double2* res = (double2*)(db_smem + a.ores);
    for (int b0 = 0; b0 < na; b0 += kDbBatch) {
      const int nb = min(kDbBatch, na - b0);
      if (active)
        for (int i = h; i < nb; i += a.units) {
          const int e = list[b0 + i];
          const int info = __ldg(a.g.bond_info + (size_t)e * 32 + lane);
          double dre = 0.0, dim = 0.0;
          db_delta<FPL, false, true>(c, info, sp, Yc, Hc, nullptr, uo, uwarp, sync, dre, dim);
          dre = db_sum(dre);
          dim = db_sum(dim);
          if (a.uw > 1) {
            if (lane == 0) {
              sum[2 * uwarp] = dre;
              sum[2 * uwarp + 1] = dim;
            }
            sync();
            dre = dim = 0.0;
            for (int w = 0; w < a.uw; ++w) {
              dre += sum[2 * w];
              dim += sum[2 * w + 1];
            }
            sync();
          }
          if (uwarp == 0 && lane == 0) {
            res[i] = make_double2(dre, dim);
            if (a.dlogpsi) a.dlogpsi[b * E + e] = (float)dre;
          }
        }
      __syncthreads();
      for (int i = threadIdx.x; i < nb; i += kDbThreads) {
        const double2 d = res[i];
        const double amp = exp(d.x), hJ = 0.5 * __ldg(a.g.J + list[b0 + i]);
        double sn = 0.0, cs = 1.0;
        if (d.y != 0.0) sincos(d.y, &sn, &cs);
        er += hJ * (amp * cs);
        ei += hJ * (amp * sn);
      }
      __syncthreads();
    }
    diag = db_sum(diag);
    if (warp * 32 < na) {  // (warps without a term keep their zeros)
      er = db_sum(er);
      ei = db_sum(ei);
    }
    if (lane == 0) {
      s_e[warp] = diag;
      s_e[kDbWarps + warp] = er;
      s_e[2 * kDbWarps + warp] = ei;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double d = 0.0, re = 0.0, im = 0.0;
      for (int w = 0; w < kDbWarps; ++w) {
        d += s_e[w];
        re += s_e[kDbWarps + w];
        im += s_e[2 * kDbWarps + w];
      }
      a.eloc[2 * b] = d + re;
      a.eloc[2 * b + 1] = im;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------------
struct DbPlan {
  DbArgs a;
  int grid = 0;
  uint32_t smem = 0;
  size_t ws_bytes = 0;
};

const void* db_kernel(bool eloc, int F) {
  if (eloc) return F > 32 ? (const void*)k_db_eloc<2> : (const void*)k_db_eloc<1>;
  return F > 32 ? (const void*)k_db_metro<2> : (const void*)k_db_metro<1>;
}

// Shared memory of a CTA with `units` units of `uw` warps, in bytes.
uint64_t db_layout(const gna_graph* g, const Dims& m, bool eloc, int units, int uw, DbArgs* a) {
  const int F = m.F, N = m.N, L = m.L;
  a->units = units;
  a->uw = uw;
  a->lpr = 1;
  while (a->lpr < F && a->lpr < 32) a->lpr *= 2;
  a->fpl = (F + 31) / 32;
  const int R = 32 / a->lpr;
  uint64_t o = 0;
  auto take = [&](uint64_t bytes) {
    const uint64_t r = o;
    o = (o + bytes + 15) / 16 * 16;
    return (uint32_t)r;
  };
  a->oW = take((uint64_t)2 * F * F * 8);
  a->ob = take((uint64_t)F * 8);
  a->oemb = take((uint64_t)2 * F * 8);
  a->owr = take((uint64_t)(F + 2) * 2 * 8);
  a->obr = take(16);
  a->oav = take((uint64_t)N * 8);
  a->oz0 = take((uint64_t)2 * F * 8);
  a->olist = eloc ? take((uint64_t)m.E * 2) : 0;
  a->ores = eloc ? take((uint64_t)kDbBatch * 16) : 0;
  uint64_t zr[2] = {3, 0};
  for (int l = 1; l < L; ++l) {
    const uint64_t rows = (uint64_t)g->max_ball[l] + 1;
    if (rows > zr[l & 1]) zr[l & 1] = rows;
  }
  // the sampler's forward stages its rows in the Z space, the local energy's (all warps of the
  // CTA) in the last unit's product rows, which are made large enough
  const uint64_t stage = (uint64_t)uw * R * 2;
  if (zr[0] + zr[1] < stage) zr[1] = stage - zr[0];
  uint64_t u = 0;
  auto utake = [&](uint64_t bytes) {
    const uint64_t r = u;
    u = (u + bytes + 15) / 16 * 16;
    return (uint32_t)r;
  };
  for (int i = 0; i < 2; ++i) a->uz[i] = utake(zr[i] * 2 * F * 8);
  a->ud = utake((uint64_t)(eloc ? 2 * kDbWarps : uw) * R * F * 8);
  a->usum = utake((uint64_t)uw * 16);
  a->uspin = utake(N);
  if (u > UINT32_MAX / kDbWarps) return UINT64_MAX;
  a->unit_bytes = (uint32_t)u;
  a->ounit = take((uint64_t)units * u);
  return o;
}

gna_status db_plan(const gna_graph* g, const Dims& m, bool eloc, int64_t B, DbPlan* p) {
  if (m.L < 1 || m.F > 64 || !m.shared || m.act != GNA_ACT_TANH || m.E < 1 || m.E > 0xFFFF) return GNA_ERR_UNSUPPORTED;
  DeviceInfo di;
  gna_status st = device_info(&di);
  if (st != GNA_OK) return st;
  const uint64_t budget = (uint64_t)di.smem_optin - 512;
  DbArgs& a = p->a;
  memset(&a, 0, sizeof(a));
  // one warp per chain (bond) while there are enough of them for the four FP64 pipes of every SM,
  // else the block's warps share fewer
  int uw = 1;
  if (!eloc && B * 2 <= (int64_t)di.sms * kDbWarps) uw = B > di.sms ? 2 : 4;
  uint64_t smem = 0;
  for (; uw <= kDbWarps; uw *= 2) {
    smem = db_layout(g, m, eloc, kDbWarps / uw, uw, &a);
    if (smem <= budget) break;
  }
  if (uw > kDbWarps) return GNA_ERR_UNSUPPORTED;
  p->smem = (uint32_t)smem;
  const void* k = db_kernel(eloc, m.F);
  if ((st = allow_smem(k, budget)) != GNA_OK) return st;
  int occ = 0;
  GNA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kDbThreads, p->smem));
  if (occ < 1) occ = 1;
  if (occ > 4) occ = 4;  // four warps of each pipe keep it busy; more only need more workspace
  int64_t grid = (int64_t)di.sms * occ;
  const int64_t need = eloc ? B : (B + a.units - 1) / a.units;
  if (grid > need) grid = need;
  p->grid = (int)(grid < 1 ? 1 : grid);
  const size_t NF = (size_t)m.N * m.F;
  size_t o = 3 * m.L * NF;  // (H, 1 - H^2), then Y
  if (!eloc)
    for (int l = 1; l <= m.L; ++l) {
      a.off_new[l] = o;
      o += (size_t)3 * g->max_ball[l] * m.F;
    }
  a.off_h = o;
  o += 2 * NF;
  a.ws_unit = (o + 1) / 2 * 2;
  p->ws_bytes = align_up((size_t)p->grid * (eloc ? 1 : a.units) * a.ws_unit * sizeof(double));
  return GNA_OK;
}

gna_status db_size(const gna_graph* g, const Dims& m, bool eloc, int64_t B, size_t* bytes) {
  if (B == 0) {
    *bytes = 0;
    return GNA_OK;
  }
  DbPlan p;
  gna_status st = db_plan(g, m, eloc, B, &p);
  if (st == GNA_OK) *bytes = p.ws_bytes;
  return st;
}

gna_status db_launch(DbPlan& p, bool eloc, void* ws, size_t ws_bytes, cudaStream_t stream) {
  if (ws_bytes < p.ws_bytes || !ws) return GNA_ERR_WORKSPACE;
  p.a.ws = (double*)ws;
  void* args[] = {&p.a};
  GNA_CUDA_TRY(cudaLaunchKernel(db_kernel(eloc, p.a.m.F), dim3(p.grid), dim3(kDbThreads), args, p.smem, stream));
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

}  // namespace

gna_status db_metro_workspace(const gna_graph* g, const Dims& m, int64_t C, size_t* bytes) {
  return db_size(g, m, false, C, bytes);
}
gna_status db_eloc_workspace(const gna_graph* g, const Dims& m, int64_t B, size_t* bytes) {
  return db_size(g, m, true, B, bytes);
}

gna_status db_metro_run(const MetroCall& mc, void* ws, size_t ws_bytes, cudaStream_t stream) {
  DbPlan p;
  gna_status st = db_plan(mc.g, mc.m, false, mc.C, &p);
  if (st != GNA_OK) return st;
  DbArgs& a = p.a;
  a.g = mc.g->d;
  a.m = mc.m;
  a.theta = (const double*)mc.theta;
  a.chain_spins = mc.chain_spins;
  a.B = mc.C;
  a.n_sweeps = mc.n_sweeps;
  a.record_every = mc.record_every;
  a.seed = mc.seed;
  a.step0 = mc.step0;
  a.samples_out = mc.samples_out;
  a.logpsi_out = mc.logpsi_out;
  a.n_acc = mc.n_acc;
  a.trace = mc.trace;
  return db_launch(p, false, ws, ws_bytes, stream);
}

gna_status db_eloc_run(const SimtCall& sc, void* ws, size_t ws_bytes, cudaStream_t stream) {
  DbPlan p;
  gna_status st = db_plan(sc.g, sc.m, true, sc.B, &p);
  if (st != GNA_OK) return st;
  DbArgs& a = p.a;
  a.g = sc.g->d;
  a.m = sc.m;
  a.theta = (const double*)sc.theta;
  a.spins = sc.spins;
  a.B = sc.B;
  a.eloc = sc.eloc;
  a.dlogpsi = sc.dlogpsi;
  return db_launch(p, true, ws, ws_bytes, stream);
}

}  // namespace gna
