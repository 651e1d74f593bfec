"""The split-operand local energy (one warp per tile of 16 rows, eloc.cu) at the sizes where its
tiles, neighbour pairs and units can go wrong, against the FP64 oracle on BF16-rounded W: balls
that end on, just before and just after a multiple of 16 rows, one layer and eight, degrees 0 to
14 (odd ones too: half-filled pairs), the unrolled pair counts 2 and 3, and weights large enough
that units swing further than the tanh series reaches.

Tolerance: the derived bound on each Delta and each sample of tests/bounds.py, plus the float32
rounding of the returned Delta and of each term, as for the other local-energy tests.  The same
tiles in FP32 (tanh, and ReLU + layer norm): 1e-5 of the terms' magnitude (tests/scales.py)."""
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
    return t


def _isolated():
    r = W.ring(9)
    return W.Graph(10, r.edges, r.J, "ring9_plus_isolated")


GRAPHS = {"two": W.two_site, "ring15": lambda: W.ring(15), "ring40": lambda: W.ring(40), "isolated": _isolated,
          "complete9": lambda: W.complete(9), "bipartite": lambda: W.complete_bipartite(3, 14),
          "kagome3": lambda: W.kagome(3), "tri5": lambda: W.triangular(5, 5), "er30": lambda: W.erdos_renyi(30, 0.2, seed=5)}

# (graph, F, L, weight scale).  Ring balls have 2 + 2 l rows: 16 at l = 7, 18 at l = 8
CASES = [("two", 16, 1, 0.3), ("ring15", 32, 1, 0.3), ("ring40", 16, 8, 0.3), ("ring40", 32, 7, 0.3), ("ring40", 48, 6, 0.3),
         ("isolated", 64, 3, 0.3), ("complete9", 32, 2, 0.3), ("bipartite", 48, 3, 0.1), ("bipartite", 16, 2, 1.5),
         ("kagome3", 64, 5, 0.1), ("kagome3", 32, 3, 1.5), ("tri5", 16, 2, 0.3), ("tri5", 64, 3, 1.5), ("er30", 32, 4, 0.3)]


@pytest.mark.parametrize("name,F,L,scale", CASES)
def test_tiles_against_the_oracle(torch, name, F, L, scale):
    g = GRAPHS[name]()
    th = W.random_theta(F, L, seed=F + L, scale=scale)
    theta = torch.tensor(th, dtype=torch.float32, device="cuda")
    th = theta.double().cpu().numpy()
    w = slice(3 * F, 3 * F + 2 * F * F)
    th[w] = theta[w].to(torch.bfloat16).double().cpu().numpy()
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_BF16X2)
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    s = W.random_spins(g.n_sites, 7, seed=3)
    st = torch.tensor(s, device="cuda")
    gna.device_status(clear=True)
    E, dl = gna.local_energy(graph, model, theta, st, gna.ELOC_INCREMENTAL, bonds=True)
    E2, lp = gna.local_energy_logpsi(graph, model, theta, st)
    assert gna.device_status(clear=True) == 0
    assert np.array_equal(E.cpu().numpy(), E2.cpu().numpy())
    assert np.array_equal(lp.cpu().numpy(), gna.forward(graph, model, theta, st).cpu().numpy())
    delta, bd, eb = BD.bond_bounds(th, F, L, Ah, g.edges, g.J, s, "bf16x2")
    anti = ~np.isnan(delta.real)
    want_d = np.where(anti, delta.real, 0.0)
    got_d = dl.cpu().numpy()
    assert np.all(got_d[~anti] == 0.0)
    assert np.all(np.abs(got_d - want_d) <= bd + 2.0 ** -23 * np.abs(want_d)), np.max(np.abs(got_d - want_d) - bd)
    want = hz.local_energy(lambda x: gcn.logpsi_complex(th, F, L, Ah, x), g.edges, g.J, s)
    terms = 0.5 * np.abs(np.where(anti, g.J[None, :], 0.0)) * np.abs(np.exp(np.where(anti, delta, 0.0)))
    err = np.abs(E.cpu().numpy()[:, 0] + 1j * E.cpu().numpy()[:, 1] - want)
    assert np.all(err <= eb + 2.0 ** -21 * terms.sum(axis=1) + 1e-12 * np.abs(want)), err


def test_bonds_without_antiparallel_partners(torch):
    # every unit idle, and fewer antiparallel bonds than units
    g = W.kagome(3)
    graph, model = gna.Graph.from_workload(g, 3), gna.Model(32, 3, gna.PREC_BF16X2)
    theta = torch.tensor(W.random_theta(32, 3, seed=1, scale=0.3), dtype=torch.float32, device="cuda")
    s = np.ones((3, g.n_sites), dtype=np.int8)
    s[1, 4] = -1
    s[2, :] = -1
    E = gna.local_energy(graph, model, theta, torch.tensor(s, device="cuda"), gna.ELOC_INCREMENTAL).cpu().numpy()
    assert E[0, 0] == E[2, 0] == 0.25 * g.J.sum() and E[0, 1] == E[2, 1] == 0.0
    th = theta.double().cpu().numpy()
    w = slice(3 * 32, 3 * 32 + 2 * 32 * 32)
    th[w] = theta[w].to(torch.bfloat16).double().cpu().numpy()
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    _, _, eb = BD.bond_bounds(th, 32, 3, Ah, g.edges, g.J, s[1:2], "bf16x2")
    want = hz.local_energy(lambda x: gcn.logpsi_complex(th, 32, 3, Ah, x), g.edges, g.J, s[1:2])
    assert abs(E[1, 0] + 1j * E[1, 1] - want[0]) <= eb[0] + 2.0 ** -21 * 0.25 * g.J.sum()


@pytest.mark.parametrize("act", ["tanh", "relu_ln"])
@pytest.mark.parametrize("name,F,L,scale", [("two", 16, 1, 0.3), ("ring40", 16, 8, 0.3), ("ring40", 32, 7, 0.3),
                                            ("isolated", 64, 3, 0.3), ("complete9", 32, 2, 0.3), ("bipartite", 48, 3, 0.1),
                                            ("kagome3", 64, 3, 0.3), ("kagome3", 16, 3, 1.0), ("tri5", 48, 2, 0.3),
                                            ("er30", 32, 4, 0.3)])
def test_fp32_tiles_against_the_oracle(torch, name, F, L, scale, act):
    g = GRAPHS[name]()
    one = np.ones(g.n_edges)
    xxz = (one, -0.7 * one, 0.5 * one, 0.25 * one) if act == "relu_ln" else None
    theta = torch.tensor(W.random_theta(F, L, seed=F + L, scale=scale), dtype=torch.float32, device="cuda")
    th = theta.double().cpu().numpy()
    graph = gna.Graph(g.n_sites, g.edges, g.J, L, xxz=xxz)
    model = gna.Model(F, L, gna.PREC_FP32, act=gna.ACT_RELU_LN if act == "relu_ln" else gna.ACT_TANH)
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    s = W.random_spins(g.n_sites, 7, seed=3)
    E, dl = gna.local_energy(graph, model, theta, torch.tensor(s, device="cuda"), gna.ELOC_INCREMENTAL, bonds=True)
    psi = lambda x: gcn.logpsi_complex(th, F, L, Ah, x, True, act)  # noqa: E731
    kw = {"xxz": xxz} if xxz is not None else {}
    want = hz.local_energy(psi, g.edges, g.J, s, **kw)
    err = np.abs(E.cpu().numpy()[:, 0] + 1j * E.cpu().numpy()[:, 1] - want)
    assert np.all(err <= 1e-5 * np.maximum(SC.eloc_scale(th, F, L, Ah, g.edges, g.J, s, act=act, **kw), 1.0)), err
    d = hz.bond_log_ratios(psi, g.edges, s)
    want_d = np.where(np.isnan(d.real), 0.0, d.real)
    lim = 1e-5 * np.maximum(SC.delta_scale(th, F, L, Ah, g.edges, s, act=act), 1.0) + 2.0 ** -24 * np.abs(want_d)
    assert np.all(np.abs(dl.cpu().numpy() - want_d) <= lim), np.max(np.abs(dl.cpu().numpy() - want_d) - lim)
