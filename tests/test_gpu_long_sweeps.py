"""Samplers that carry a chain's features from move to move: after hundreds of sweeps in one call they are
still those of the configuration.

FP64: the recorded log Psi against gna.forward of the recorded samples, and the log ratios of the last steps
against the oracle.  Every accepted move adds roundings of some 1e-16 to each feature it touches; 1e3
sweeps are some 1e4 of them, as a random walk 1e-14, times the 200 features' weights: 1e-10 of the terms'
magnitude leaves two orders.  FP32 alike (6e-8 each): 1e-3."""
import numpy as np
import pytest

from oracle import gcn, heisenberg as hz
from paper_2011_12453_gb300 import build as B, gna, workloads as W

import scales as SC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t

    B.build()
    t.cuda.set_device(0)
    return t


@pytest.mark.parametrize("prec,tol", [(gna.PREC_FP64, 1e-10), (gna.PREC_FP32, 1e-3)])
@pytest.mark.parametrize("F,L,scale,C,sweeps", [(16, 2, 0.1, 40, 1000), (16, 2, 0.3, 200, 400), (16, 3, 1.0, 40, 400),
                                                (48, 2, 0.3, 700, 200), (16, 2, 3.0, 40, 400)])
def test_features_after_many_sweeps(torch, prec, tol, F, L, scale, C, sweeps):
    g = W.kagome(2)
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, prec)
    theta = torch.tensor(W.random_theta(F, L, seed=3, scale=scale), dtype=model.theta_dtype(), device="cuda")
    th = theta.double().cpu().numpy()
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    ch = torch.tensor(W.random_spins(g.n_sites, C, seed=4), device="cuda")
    samples, lp, _, _ = gna.metropolis_sweep(graph, model, theta, ch, sweeps, sweeps // 4, 7, 0)
    for r in range(4):
        x = samples[r].contiguous()
        want = gna.forward(graph, model, theta, x).cpu().numpy()
        sc = np.maximum(SC.logpsi_scale(th, F, L, Ah, x[:8].cpu().numpy()).max(), 1.0)
        assert np.abs(lp[r].cpu().numpy() - want).max() <= tol * sc, r


@pytest.mark.parametrize("scale", [0.3, 1.0])
def test_fp64_ratios_after_many_sweeps(torch, scale):
    g, F, L, C, sweeps = W.kagome(2), 16, 2, 3, 400
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_FP64)
    th = W.random_theta(F, L, seed=3, scale=scale)
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    s0 = W.random_spins(g.n_sites, C, seed=4)
    tr = gna.metropolis_sweep(graph, model, torch.tensor(th, device="cuda"), torch.tensor(s0, device="cuda"), sweeps, 0, 7, 0,
                              trace=True)[3].cpu().numpy()
    states, bonds, got = [], [], []
    for c in range(C):
        s = s0[c].copy()
        for k, (e, acc, v, _) in enumerate(tr[c]):
            i, j = g.edges[int(e)]
            if s[i] == s[j]:
                continue
            if k >= tr.shape[1] - 40:
                states.append(s.copy())
                bonds.append(int(e))
                got.append(v)
            if acc:
                s[[i, j]] = s[[j, i]]
    states, r = np.stack(states), np.arange(len(bonds))
    want = hz.bond_log_ratios(lambda x: gcn.logpsi_complex(th, F, L, Ah, x), g.edges, states).real[r, bonds]
    lim = 1e-10 * np.maximum(SC.delta_scale(th, F, L, Ah, g.edges, states)[r, bonds], 1.0)
    assert len(bonds) > 20 and np.all(np.abs(np.array(got) - want) <= lim), np.max(np.abs(np.array(got) - want) - lim)
