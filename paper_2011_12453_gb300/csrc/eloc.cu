// Incremental local energy on warp tiles (eloc_impl.cuh): the BF16X2 kernels, and the plan and
// launch of all of them.
#include <cstring>

#include "eloc_impl.cuh"

namespace gna {

// ---------------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------------
struct ElPlan {
  ElArgs a;
  const void* kernel = nullptr;
  int grid = 0;
  uint32_t smem = 0;
  size_t ws_bytes = 0, u_bytes = 0;
};

// Every row of a graph whose sites all have 3 or 4 (5 or 6) neighbours has two (three)
// neighbour pairs: the gather loop is then unrolled (two only for FP32).
static int el_np(const gna_graph* g, int mode) {
  const int np = (g->max_deg + 1) / 2;
  return (g->min_deg + 1) / 2 == np && (np == 2 || (np == 3 && mode == EL_X2)) ? np : 0;
}
static const void* el_kernel(const gna_graph* g, int F, int mode) {
  const int np = el_np(g, mode);
  if (mode != EL_X2) return el_kernel_f32(np, F, mode);
  return np == 2 ? el_kernel_np<2, EL_X2>(F) : np == 3 ? el_kernel_np<3, EL_X2>(F) : el_kernel_np<0, EL_X2>(F);
}

// Shared-memory layout of one choice of units and warps; returns its total in bytes.
static uint64_t el_layout(const gna_graph* g, const Dims& m, int units, int uw, int nbuf, int mode, ElArgs* a) {
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
  a->oW = take((uint64_t)el_wterms(mode) * 2 * F * F * 2);
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
  const int np = el_np(g, mode);
  const uint64_t nrec = (uint64_t)(g->max_ball[L] + 15) / 16 * 16;
  const uint64_t npairs = np > 0 ? nrec * np : (uint64_t)(g->max_pairs[L] + 3) / 4 * 4;
  for (int i = 0; i < 2; ++i) a->urec[i] = i < nbuf ? utake(nrec * 8) : 0;
  for (int i = 0; i < 2; ++i) a->upair[i] = i < nbuf ? utake(npairs * 4) : 0;
  a->usum = utake((uint64_t)uw * 16);
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

static gna_status el_plan(const gna_graph* g, const Dims& m, int64_t B, bool f32, ElPlan* p) {
  const int mode = !f32 ? EL_X2 : m.act == GNA_ACT_RELU_LN ? EL_F32_LN : EL_F32;
  if (m.F % 16 != 0 || m.F > 64 || m.L < 1 || !m.shared || (m.act != GNA_ACT_TANH && !f32) || !g->pack_ok ||
      m.E < 1 || m.E > 0xFFFF)
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
      while (units > 0 && el_layout(g, m, units, uw, nbuf, mode, &t) > budget) --units;
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
  p->smem = (uint32_t)el_layout(g, m, bu, bw, bn, mode, &p->a);
  const void* kfn = el_kernel(g, m.F, mode);
  p->kernel = kfn;
  if ((st = allow_smem(kfn, budget)) != GNA_OK) return st;
  int64_t grid = di.sms;
  if (grid > B) grid = B;
  p->grid = (int)(grid < 1 ? 1 : grid);
  p->u_bytes = align_up((size_t)p->grid * 2 * m.L * m.N * el_ldu(m.F) * sizeof(float));
  p->ws_bytes = p->u_bytes + (p->a.h_smem ? 0 : align_up((size_t)p->grid * 2 * m.N * el_ldh(m.F) * sizeof(float)));
  return GNA_OK;
}

gna_status el_workspace(const gna_graph* g, const Dims& m, int64_t B, bool f32, size_t* bytes) {
  if (B == 0) {
    *bytes = 0;
    return GNA_OK;
  }
  ElPlan p;
  gna_status st = el_plan(g, m, B, f32, &p);
  if (st != GNA_OK) return st;
  *bytes = p.ws_bytes;
  return GNA_OK;
}

gna_status el_run(const TcCall& call, bool f32, void* ws, size_t ws_bytes, cudaStream_t stream) {
  ElPlan p;
  gna_status st = el_plan(call.g, call.m, call.B, f32, &p);
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
  GNA_CUDA_TRY(cudaLaunchKernel(p.kernel, dim3(p.grid), dim3(kElThreads), args, p.smem, stream));
  GNA_CUDA_TRY(cudaGetLastError());
  return GNA_OK;
}

}  // namespace gna
