"""A workspace that is large enough for a batch is large enough for every smaller one."""
import ctypes

import numpy as np
import pytest

from paper_2011_12453_gb300 import build as B, gna, workloads as W

pytestmark = pytest.mark.gpu

MODELS = [(gna.PREC_FP64, 16, gna.ACT_TANH), (gna.PREC_FP32, 16, gna.ACT_TANH), (gna.PREC_FP32, 16, gna.ACT_RELU_LN),
          (gna.PREC_FP32, 48, gna.ACT_TANH), (gna.PREC_BF16, 32, gna.ACT_TANH), (gna.PREC_BF16X2, 32, gna.ACT_TANH),
          (gna.PREC_BF16X2, 64, gna.ACT_TANH)]


@pytest.fixture(scope="module")
def torch():
    import torch as t

    B.build()
    t.cuda.set_device(0)
    return t


@pytest.mark.parametrize("gname", ["kagome2", "kagome6", "er65"])
@pytest.mark.parametrize("prec,F,act", MODELS)
def test_size_never_falls(torch, gname, prec, F, act):
    g = W.erdos_renyi(65, 0.06, seed=5) if gname == "er65" else W.kagome(int(gname[-1]))
    graph, model = gna.Graph.from_workload(g, 3), gna.Model(F, 3, prec, act=act)
    for op in (gna.OP_FORWARD, gna.OP_ELOC_FULL, gna.OP_ELOC_INCR, gna.OP_METROPOLIS, gna.OP_BACKWARD, gna.OP_ISGO_WEIGHTS,
               gna.OP_ISGO_GRAD, gna.OP_METROPOLIS_LEARNED, gna.OP_ELOC_LOGPSI):
        sizes = np.array([gna.workspace_size(graph, model, op, n) for n in range(0, 2600)])
        assert np.all(np.diff(sizes) >= 0), (op, np.nonzero(np.diff(sizes) < 0)[0][:4] + 1)


@pytest.mark.parametrize("prec", [gna.PREC_BF16X2, gna.PREC_FP32])
def test_fewer_chains_run_in_a_larger_number_s_workspace(torch, prec):
    # with 152 SMs, 11 or 12 warps each: one round of 11 (or 12) warps an SM, against two of 6 (or 7)
    g = W.kagome(6)
    graph, model = gna.Graph.from_workload(g, 4), gna.Model(32, 4, prec)
    theta = torch.tensor(W.random_theta(32, 4, seed=1), dtype=torch.float32, device="cuda")
    sizes = {n: gna.workspace_size(graph, model, gna.OP_METROPOLIS, n) for n in range(1, 2600)}
    large = min(range(1400, 2600), key=lambda n: sizes[n])
    ws = torch.empty(sizes[large], dtype=torch.uint8, device="cuda")
    for n in (large - 1, 1, 64):
        ch = torch.tensor(W.random_spins(g.n_sites, n, seed=4), device="cuda")
        want = ch.clone()
        gna.metropolis_sweep(graph, model, theta, want, 1, 0, 7, 0)
        st = gna.lib().gna_metropolis_sweep(graph.handle, ctypes.byref(model.desc), theta.data_ptr(), ch.data_ptr(), n, 1, 0, 7, 0,
                                            None, 0.0, None, None, None, None, ws.data_ptr(), ws.numel(),
                                            torch.cuda.current_stream().cuda_stream)
        assert st == gna.GNA_OK and torch.equal(ch, want)
