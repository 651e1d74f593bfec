"""Samplers of models with a W and b per layer, against the FP64 oracle: every proposal's log ratio (the plain
move's Re Delta) and the recorded log Psi.  FP64 1e-9 and FP32 1e-5 of the terms' magnitude
(tests/scales.py), as the other parity tests; the learned moves' records only, against gna.forward."""
import numpy as np
import pytest

from oracle import gcn, heisenberg as hz
from paper_2011_12453_gb300 import build as B, gna, workloads as W

import scales as SC

pytestmark = pytest.mark.gpu

PREC = {"fp64": (gna.PREC_FP64, 1e-9), "fp32": (gna.PREC_FP32, 1e-5)}


@pytest.fixture(scope="module")
def torch():
    import torch as t

    B.build()
    t.cuda.set_device(0)
    return t


def _model(torch, g, F, L, prec):
    theta = torch.tensor(W.random_theta(F, L, seed=F + L, scale=0.3, shared=False), device="cuda",
                         dtype=torch.float64 if prec == "fp64" else torch.float32)
    return gna.Graph.from_workload(g, L), gna.Model(F, L, PREC[prec][0], shared=False), theta


@pytest.mark.parametrize("prec", list(PREC))
@pytest.mark.parametrize("F,L", [(16, 1), (16, 2), (48, 3)])
def test_plain_moves(torch, prec, F, L):
    g, tol = W.kagome(2), PREC[prec][1]
    graph, model, theta = _model(torch, g, F, L, prec)
    th = theta.double().cpu().numpy()
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    s0 = W.random_spins(g.n_sites, 5, seed=4)
    ch = torch.tensor(s0, device="cuda")
    samples, lp, _, tr = gna.metropolis_sweep(graph, model, theta, ch, 2, 1, 7, 0, trace=True)
    tr = tr.cpu().numpy()
    x = samples[-1].cpu().numpy()
    sc = np.maximum(SC.logpsi_scale(th, F, L, Ah, x, False), 1.0)
    assert np.all(np.abs(lp[-1].cpu().numpy() - gcn.logpsi(th, F, L, Ah, x, False)) <= tol * sc)
    states, bonds, got = [], [], []
    for c in range(5):
        s = s0[c].copy()
        for e, acc, v, _ in tr[c]:
            i, j = g.edges[int(e)]
            if s[i] == s[j]:
                continue
            states.append(s.copy())
            bonds.append(int(e))
            got.append(v)
            if acc:
                s[[i, j]] = s[[j, i]]
    states, r = np.stack(states), np.arange(len(bonds))
    want = hz.bond_log_ratios(lambda y: gcn.logpsi_complex(th, F, L, Ah, y, False), g.edges, states).real[r, bonds]
    lim = tol * np.maximum(SC.delta_scale(th, F, L, Ah, g.edges, states, False)[r, bonds], 1.0)
    assert np.all(np.abs(np.array(got) - want) <= lim)


@pytest.mark.parametrize("prec", list(PREC))
def test_learned_moves(torch, prec):
    g, F, L = W.erdos_renyi(20, 0.2, seed=5), 16, 2
    graph, model, theta = _model(torch, g, F, L, prec)
    p32 = torch.tensor(W.random_proposal_params(3, 0.5), dtype=torch.float32, device="cuda")
    ch = torch.tensor(W.random_spins(g.n_sites, 9, seed=4), device="cuda")
    samples, lp, _, _ = gna.metropolis_sweep(graph, model, theta, ch, 2, 2, 7, 0, proposal=p32)
    want = gna.forward(graph, model, theta, samples[-1].contiguous())
    assert (lp[-1] - want).abs().max().item() <= PREC[prec][1] * max(1.0, want.abs().max().item()) * 10
