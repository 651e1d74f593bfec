// log Psi of BF16X2 models: the forward of a configuration in tiles of 16 sites, one warp each.
//
// Per layer a warp gathers X = [A_hat H ; H] of its sites in FP32, splits it into hi + lo BF16
// operands in its registers and multiplies by W with mma.sync (frag.cuh); H^l is tanh of the result
// plus the bias, in FP32 rows of shared memory.  Sums are in the order of the tcgen05 forward
// (tc.cu) and of the local energy's own (eloc_impl.cuh): the results are the same bits.
//
// What bounds it: one configuration is L dependent layers of some 100 rows, so latency -- of the
// parameters' loads, then per layer of one gather, 4 FC products and a barrier, where the tcgen05
// form pays a fence, an mbarrier round trip and a TMEM read besides.  With a block of as many warps as
// a configuration has tiles (at most 8, so that several blocks share an SM; 16 while every block has
// an SM to itself), no warp waits for another's second tile.
// Triangular 144, L 4, F 48: 1000 configurations 87 us against some 270, 4001 configurations and
// their gradient 4.29 -> 3.59 ms.  One configuration through the library is bound by the host's call:
// Kagome 108, L 4, F 32 takes 34 to 37 us with either kernel.
#include <cstring>

#include "eloc_impl.cuh"
#include "fwd.cuh"

namespace gna {
namespace {

struct FxArgs {
  DevGraph g;
  Dims m;
  const float* theta;
  const int8_t* spins;
  int64_t B;
  double* logpsi;
  float* gH;  // [grid][2][N][ldh] when the rows are in the workspace
  int h_smem;
  uint32_t oW, obias, oemb, owr, obr, ospin, orp, owf, ocol, ored, oH;
};

extern __shared__ __align__(128) unsigned char fx_smem[];

template <int FC>
__global__ void __launch_bounds__(512, 1) k_fwd_x2(const FxArgs a) {
  constexpr int F = 16 * FC, LDH = el_ldh(F), kParts = kReadout / F;
  const int N = a.m.N, L = a.m.L;
  const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, nwarps = nthr >> 5, lane = tid & 31;
  const int g = lane >> 2, q = lane & 3;
  const float* th = a.theta;
  uint4* Wf = (uint4*)(fx_smem + a.oW);
  float* bias = (float*)(fx_smem + a.obias);
  float* emb = (float*)(fx_smem + a.oemb);
  float* wr = (float*)(fx_smem + a.owr);
  float* br = (float*)(fx_smem + a.obr);
  int8_t* spin = (int8_t*)(fx_smem + a.ospin);
  int* rp = (int*)(fx_smem + a.orp);
  float* wf = (float*)(fx_smem + a.owf);
  uint16_t* col = (uint16_t*)(fx_smem + a.ocol);
  float* red = (float*)(fx_smem + a.ored);
  for (int i = tid; i < 2 * FC * FC * 32; i += nthr) Wf[i] = make_wfrag<FC>(th + a.m.oW, i / (FC * 32), (i / 32) % FC, i & 31, 0);
  for (int i = tid; i < F; i += nthr) bias[i] = th[a.m.ob + i];
  for (int i = tid; i < 2 * F; i += nthr) emb[i] = tanhf(th[a.m.oWe + i] + th[a.m.obe + i % F]);
  for (int i = tid; i < (F + 2) * 2; i += nthr) wr[i] = th[a.m.owr + i];
  if (tid < 2) br[tid] = th[a.m.obr + tid];
  for (int i = tid; i <= N; i += nthr) rp[i] = __ldg(a.g.row_ptr + i);
  for (int i = tid; i < 2 * a.m.E; i += nthr) {
    wf[i] = __ldg(a.g.wf + i);
    col[i] = (uint16_t)__ldg(a.g.col + i);
  }
  const uint64_t m1 = f2_dup(-1.f);
  float* Hb = a.h_smem ? (float*)(fx_smem + a.oH) : a.gH + (size_t)blockIdx.x * 2 * N * LDH;

  for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) {
    for (int v = tid; v < N; v += nthr) spin[v] = a.spins[b * N + v];
    __syncthreads();
    float* Hp = Hb;
    float* Hn = Hb + (size_t)N * LDH;
    for (int i = tid; i < N * (F / 4); i += nthr) {
      const int v = i / (F / 4), f = (i % (F / 4)) * 4;
      *reinterpret_cast<float4*>(Hp + (size_t)v * LDH + f) =
          *reinterpret_cast<const float4*>(emb + (spin[v] > 0 ? 0 : F) + f);
    }
    __syncthreads();
    for (int l = 1; l <= L; ++l) {
      for (int t = warp; t * 16 < N; t += nwarps) {
        uint32_t hi[2 * FC][4], lo[2 * FC][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int v = min(16 * t + g + 8 * h, N - 1);
          float acc[FC][4];
#pragma unroll
          for (int c = 0; c < FC; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.f;
          const int k1 = rp[v + 1];
          for (int k = rp[v]; k < k1; ++k) {
            const float w = wf[k];
            const float* x = Hp + (size_t)col[k] * LDH + 4 * q;
#pragma unroll
            for (int c = 0; c < FC; ++c) {
              const float4 y = *reinterpret_cast<const float4*>(x + 16 * c);
              acc[c][0] = fmaf(w, y.x, acc[c][0]);
              acc[c][1] = fmaf(w, y.y, acc[c][1]);
              acc[c][2] = fmaf(w, y.z, acc[c][2]);
              acc[c][3] = fmaf(w, y.w, acc[c][3]);
            }
          }
          const float* self = Hp + (size_t)v * LDH + 4 * q;
#pragma unroll
          for (int c = 0; c < FC; ++c) {
            split2(m1, acc[c][0], acc[c][1], hi[c][h], lo[c][h]);
            split2(m1, acc[c][2], acc[c][3], hi[c][2 + h], lo[c][2 + h]);
            const float4 y = *reinterpret_cast<const float4*>(self + 16 * c);
            split2(m1, y.x, y.y, hi[FC + c][h], lo[FC + c][h]);
            split2(m1, y.z, y.w, hi[FC + c][2 + h], lo[FC + c][2 + h]);
          }
        }
#pragma unroll
        for (int co = 0; co < FC; ++co) {
          float D[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
#pragma unroll
          for (int kc = 0; kc < 2 * FC; ++kc) {
            const uint4 w = Wf[(kc * FC + co) * 32 + lane];
            mma_16816(D[0], hi[kc], w.x, w.y);
            mma_16816(D[1], hi[kc], w.z, w.w);
          }
#pragma unroll
          for (int kc = 0; kc < 2 * FC; ++kc) {
            const uint4 w = Wf[(kc * FC + co) * 32 + lane];
            mma_16816(D[0], lo[kc], w.x, w.y);
            mma_16816(D[1], lo[kc], w.z, w.w);
          }
          const float4 bs = *reinterpret_cast<const float4*>(bias + 16 * co + 4 * q);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int v = 16 * t + g + 8 * h;
            if (v < N)
              *reinterpret_cast<float4*>(Hn + (size_t)v * LDH + 16 * co + 4 * q) =
                  make_float4(tanhf(D[0][2 * h] + bs.x), tanhf(D[0][2 * h + 1] + bs.y), tanhf(D[1][2 * h] + bs.z),
                              tanhf(D[1][2 * h + 1] + bs.w));
          }
        }
      }
      __syncthreads();
      float* x = Hp;
      Hp = Hn;
      Hn = x;
    }
    // readout: kParts interleaved site strides per feature, added in order
    for (int i = tid; i < kParts * F; i += nthr) {
      float s = 0.f;
      for (int v = i / F; v < N; v += kParts) s += Hp[(size_t)v * LDH + i % F];
      red[i] = s;
    }
    __syncthreads();
    if (warp == 0) {
      float re = 0.f, im = 0.f;
      for (int f = lane; f < F; f += 32) {
        float s = 0.f;
        for (int p = 0; p < kParts; ++p) s += red[p * F + f];
        re += s * wr[2 * f];
        im += s * wr[2 * f + 1];
      }
      re = warp_sum_f(re);
      im = warp_sum_f(im);
      int up = 0;
      for (int v = lane; v < N; v += 32) up += spin[v] > 0;
      up = warp_sum_f(up);
      if (lane == 0) {
        const int dn = N - up;
        a.logpsi[2 * b] = (double)(re + (float)up * wr[2 * F] + (float)dn * wr[2 * (F + 1)] + br[0]);
        a.logpsi[2 * b + 1] = (double)(im + (float)up * wr[2 * F + 1] + (float)dn * wr[2 * (F + 1) + 1] + br[1]);
      }
    }
    __syncthreads();
  }
}

struct FxPlan {
  FxArgs a;
  const void* kernel = nullptr;
  int grid = 0, warps = 0;
  uint32_t smem = 0, smem_limit = 0;
  size_t ws_bytes = 0;
};

gna_status fx_plan(const gna_graph* g, const Dims& m, int64_t B, FxPlan* p) {
  if (m.F % 16 != 0 || m.F < 16 || m.F > 64 || m.L < 1 || !m.shared || m.act != GNA_ACT_TANH) return GNA_ERR_UNSUPPORTED;
  DeviceInfo di;
  gna_status st = device_info(&di);
  if (st != GNA_OK) return st;
  const int F = m.F, N = m.N;
  FxArgs& a = p->a;
  memset(&a, 0, sizeof(a));
  uint64_t o = 0;
  auto take = [&](uint64_t bytes) {
    const uint64_t r = o;
    o = (o + bytes + 15) / 16 * 16;
    return (uint32_t)r;
  };
  a.oW = take((uint64_t)2 * (F / 16) * (F / 16) * 512);
  a.obias = take(F * 4);
  a.oemb = take(2 * F * 4);
  a.owr = take((F + 2) * 2 * 4);
  a.obr = take(8);
  a.ospin = take(N);
  a.orp = take((uint64_t)(N + 1) * 4);
  a.owf = take((uint64_t)2 * m.E * 4);
  a.ocol = take((uint64_t)2 * m.E * 2);
  a.ored = take(kReadout * 4);
  const uint64_t rows = (uint64_t)2 * N * el_ldh(F) * 4, budget = di.smem_optin;
  a.h_smem = o + rows <= budget;
  if (a.h_smem) a.oH = take(rows);
  if (o > budget) return GNA_ERR_UNSUPPORTED;
  p->smem = (uint32_t)o;
  p->smem_limit = (uint32_t)budget;
  // tiles of 16 sites in equal rounds
  const int tiles = (N + 15) / 16, most = B <= di.sms ? 16 : 8, rounds = (tiles + most - 1) / most;
  p->warps = (tiles + rounds - 1) / rounds;
  if (p->warps < 4) p->warps = 4;
  switch (F / 16) {
    case 1: p->kernel = (const void*)k_fwd_x2<1>; break;
    case 2: p->kernel = (const void*)k_fwd_x2<2>; break;
    case 3: p->kernel = (const void*)k_fwd_x2<3>; break;
    default: p->kernel = (const void*)k_fwd_x2<4>;
  }
  // blocks that share an SM: 16 warps of 128 registers, its shared memory with 1 KiB a block
  const int64_t by_smem = (int64_t)((di.smem_optin + 1024) / (p->smem + 1024)), by_regs = 16 / p->warps;
  int64_t occ = by_smem < by_regs ? by_smem : by_regs;
  if (occ < 1) occ = 1;
  p->grid = (int)(B < di.sms * occ ? B : di.sms * occ);
  p->ws_bytes = a.h_smem ? 0 : align_up((size_t)p->grid * rows);
  return GNA_OK;
}

}  // namespace

gna_status fx_workspace(const gna_graph* g, const Dims& m, int64_t B, size_t* bytes) {
  *bytes = 0;
  if (B == 0) return GNA_OK;
  FxPlan p;
  gna_status st = fx_plan(g, m, B, &p);
  if (st == GNA_OK) *bytes = p.ws_bytes;
  return st;
}

gna_status fx_run(const gna_graph* g, const Dims& m, const float* theta, const int8_t* spins, int64_t B, double* logpsi,
                  void* ws, size_t ws_bytes, cudaStream_t stream) {
  if (B == 0) return GNA_OK;
  FxPlan p;
  gna_status st = fx_plan(g, m, B, &p);
  if (st != GNA_OK) return st;
  if (p.ws_bytes && (ws_bytes < p.ws_bytes || !ws)) return GNA_ERR_WORKSPACE;
  p.a.g = g->d;
  p.a.m = m;
  p.a.theta = theta;
  p.a.spins = spins;
  p.a.B = B;
  p.a.logpsi = logpsi;
  p.a.gH = (float*)ws;
  if ((st = allow_smem(p.kernel, p.smem_limit)) != GNA_OK) return st;
  void* args[] = {&p.a};
  GNA_CUDA_TRY(cudaLaunchKernel(p.kernel, dim3(p.grid), dim3(32 * p.warps), args, p.smem, stream));
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

}  // namespace gna
