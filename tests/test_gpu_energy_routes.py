"""Local energies on routes that the other tests' shapes do not reach, against the FP64 oracle: FP64 with more
antiparallel bonds than one batch of 256, the per-bond values of the FP64 kernel, the degree factors of FP32
models, and the tensor-memory kernel for split operands, which takes shallow models on many sites."""
import numpy as np
import pytest

from oracle import gcn, heisenberg as hz
from paper_2011_12453_gb300 import build as B, gna, workloads as W

import bounds as BD
import scales as SC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t

    B.build()
    t.cuda.set_device(0)
    yield t
    gna.debug_wait_limit(None)
    gna.device_status(clear=True)


def _isolated():
    r = W.ring(9)
    return W.Graph(10, r.edges, r.J, "ring9_plus_isolated")


@pytest.mark.parametrize("name,F,L,scale,B_", [("two", 8, 1, 0.3, 3), ("isolated", 33, 2, 0.3, 3), ("bipartite", 64, 2, 2.0, 3),
                                               ("kagome3", 16, 3, 2.0, 3), ("tri14", 8, 2, 0.3, 2), ("tri14", 40, 1, 0.3, 1)])
def test_fp64_bond_ratios(torch, name, F, L, scale, B_):
    # 1e-9 of the terms, and the float32 rounding of the stored ratio
    g = {"two": W.two_site, "isolated": _isolated, "bipartite": lambda: W.complete_bipartite(3, 14), "kagome3": lambda: W.kagome(3),
         "tri14": lambda: W.triangular(14, 14)}[name]()
    th = W.random_theta(F, L, seed=2, scale=scale)
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_FP64)
    s = W.random_spins(g.n_sites, B_, seed=3)
    E, dl = gna.local_energy(graph, model, torch.tensor(th, device="cuda"), torch.tensor(s, device="cuda"), gna.ELOC_INCREMENTAL,
                             bonds=True)
    E, dl = E.cpu().numpy(), dl.cpu().numpy()
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    psi = lambda x: gcn.logpsi_complex(th, F, L, Ah, x)  # noqa: E731
    d = hz.bond_log_ratios(psi, g.edges, s)
    anti = ~np.isnan(d.real)
    if name == "tri14":
        assert anti.sum(axis=1).min() > 256
    want = np.where(anti, d.real, 0.0)
    assert np.all(dl[~anti] == 0.0)
    assert np.all(np.abs(dl - want) <= 2.0 ** -23 * np.abs(want) + 1e-9 * np.maximum(SC.delta_scale(th, F, L, Ah, g.edges, s), 1.0))
    err = np.abs(E[:, 0] + 1j * E[:, 1] - hz.local_energy(psi, g.edges, g.J, s))
    assert np.all(err <= 1e-9 * np.maximum(SC.eloc_scale(th, F, L, Ah, g.edges, g.J, s), 1.0)), err


@pytest.mark.parametrize("n,F", [(1000, 16), (1500, 32)])
def test_shallow_split_operand_model_on_many_sites(torch, n, F):
    g, L = W.ring(n), 1
    theta = torch.tensor(W.random_theta(F, L, seed=F, scale=0.3), dtype=torch.float32, device="cuda")
    th = theta.double().cpu().numpy()
    w = slice(3 * F, 3 * F + 2 * F * F)
    th[w] = BD.bf16_round(th[w])
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_BF16X2)
    Ah = gcn.norm_adjacency(gcn.adjacency(n, g.edges))
    s = W.random_spins(n, 2, seed=3, n_up=12)
    st = torch.tensor(s, device="cuda")
    gna.device_status(clear=True)
    E, dl = gna.local_energy(graph, model, theta, st, gna.ELOC_INCREMENTAL, bonds=True)
    assert torch.equal(gna.local_energy_logpsi(graph, model, theta, st)[1], gna.forward(graph, model, theta, st))
    assert gna.device_status(clear=True) == 0
    delta, bd, eb = BD.bond_bounds(th, F, L, Ah, g.edges, g.J, s, "bf16x2")
    anti = ~np.isnan(delta.real)
    want_d = np.where(anti, delta.real, 0.0)
    got_d = dl.cpu().numpy()
    assert np.all(got_d[~anti] == 0.0) and np.all(np.abs(got_d - want_d) <= bd + 2.0 ** -23 * np.abs(want_d))
    want = hz.local_energy(lambda x: gcn.logpsi_complex(th, F, L, Ah, x), g.edges, g.J, s)
    err = np.abs(E.cpu().numpy()[:, 0] + 1j * E.cpu().numpy()[:, 1] - want)
    assert np.all(err <= eb + 2.0 ** -21 * SC.eloc_scale(th, F, L, Ah, g.edges, g.J, s)), err
    # only that kernel has waits that can be limited
    gna.debug_wait_limit(0)
    gna.local_energy(graph, model, theta, st, gna.ELOC_INCREMENTAL)
    gna.debug_wait_limit(None)
    assert gna.device_status(clear=True) & 1
