"""Units far outside tanh's range, and parameters that are not a number, in the difference form of the
local energy and the samplers, against the FP64 oracle.

An exchange may carry a unit from one side of zero to the other however far out it was: tanh(Y + dY) -
tanh(Y) is then +-2 although 1 - tanh^2(Y) is zero in the arithmetic.  In test_swings feature 1 of the embedding is
+-0.995 and feature 0 of layer 1 is A times the site's own feature 1 plus B, so that an exchange swings
feature 0 of its two sites between A + B and -A + B.

Tolerances: FP32 1e-5 of the terms' magnitude and BF16X2 the derived bounds (tests/bounds.py), as the other
local-energy tests; FP64 1e-9 of it.  At weight scale 3 nearly all units are saturated and a few are
steep: FP32 as above plus eight times the largest change of Delta among four sets of parameters that are each
moved by up to one part in 2^23 (what rounding the parameters once more would do)."""
import numpy as np
import pytest

from oracle import gcn, heisenberg as hz
from paper_2011_12453_gb300 import build as B, gna, workloads as W

import bounds as BD
import scales as SC

pytestmark = pytest.mark.gpu

PREC = {"fp32": gna.PREC_FP32, "bf16x2": gna.PREC_BF16X2, "fp64": gna.PREC_FP64}


@pytest.fixture(scope="module")
def torch():
    import torch as t

    B.build()
    t.cuda.set_device(0)
    yield t
    gna.device_status(clear=True)


def _swinging(F, L, A, b):
    th = W.random_theta(F, L, seed=F, scale=0.3)
    th[1], th[F + 1], th[2 * F + 1] = 3.0, -3.0, 0.0  # W_e and b_e of feature 1
    th[3 * F + (F + 1) * F] = A  # W: feature 0 from the site's own feature 1
    th[3 * F + 2 * F * F] = b    # and its bias
    return th


def _rounded(torch, th, F, prec):
    theta = torch.tensor(th, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
    th = theta.double().cpu().numpy()
    if prec == "bf16x2":
        w = slice(3 * F, 3 * F + 2 * F * F)
        th[w] = BD.bf16_round(th[w])
    return theta, th


@pytest.mark.parametrize("prec,A,b", [("fp32", 56.0, -5.0), ("fp32", 200.0, 60.0), ("bf16x2", 56.0, -5.0), ("bf16x2", 128.0, 60.0),
                                      ("fp64", 56.0, -5.0), ("fp64", 450.0, -20.0)])
@pytest.mark.parametrize("F,L", [(16, 1), (32, 2)])
def test_swings(torch, prec, A, b, F, L):
    g = W.kagome(3)
    theta, th = _rounded(torch, _swinging(F, L, A, b), F, prec)
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, PREC[prec])
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    s = W.random_spins(g.n_sites, 5, seed=3)
    st = torch.tensor(s, device="cuda")
    E, dl = gna.local_energy(graph, model, theta, st, gna.ELOC_INCREMENTAL, bonds=True)
    assert torch.equal(E, gna.local_energy_logpsi(graph, model, theta, st)[0])
    E, dl = E.cpu().numpy(), dl.cpu().numpy()
    psi = lambda x: gcn.logpsi_complex(th, F, L, Ah, x)  # noqa: E731
    d = hz.bond_log_ratios(psi, g.edges, s)
    want_d = np.where(np.isnan(d.real), 0.0, d.real)
    want = hz.local_energy(psi, g.edges, g.J, s)
    err = np.abs(E[:, 0] + 1j * E[:, 1] - want)
    if prec == "bf16x2":
        _, bd, eb = BD.bond_bounds(th, F, L, Ah, g.edges, g.J, s, "bf16x2")
        terms = SC.eloc_scale(th, F, L, Ah, g.edges, g.J, s)
        assert np.all(np.abs(dl - want_d) <= bd + 2.0 ** -23 * np.abs(want_d)), np.max(np.abs(dl - want_d) - bd)
        assert np.all(err <= eb + 2.0 ** -21 * terms), err
    else:
        tol = 1e-5 if prec == "fp32" else 1e-9
        assert np.all(err <= tol * np.maximum(SC.eloc_scale(th, F, L, Ah, g.edges, g.J, s), 1.0)), err
        lim = tol * np.maximum(SC.delta_scale(th, F, L, Ah, g.edges, s), 1.0) + 2.0 ** -24 * np.abs(want_d)
        assert np.all(np.abs(dl - want_d) <= lim), np.max(np.abs(dl - want_d) - lim)


@pytest.mark.parametrize("prec,A,b", [("fp32", 56.0, -5.0), ("bf16x2", 56.0, -5.0), ("fp64", 450.0, -20.0)])
def test_swings_in_the_samplers(torch, prec, A, b):
    # every proposal's Delta (the later ones start from rows that accepted moves have carried across)
    F, L = 16, 2
    g = W.kagome(2)
    theta, th = _rounded(torch, _swinging(F, L, A, b), F, prec)
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, PREC[prec])
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    s0 = W.random_spins(g.n_sites, 4, seed=3)
    tr = gna.metropolis_sweep(graph, model, theta, torch.tensor(s0, device="cuda"), 4, 0, 5, 0, trace=True)[3].cpu().numpy()
    states, bonds, got = [], [], []
    for c in range(4):
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
    d = hz.bond_log_ratios(lambda x: gcn.logpsi_complex(th, F, L, Ah, x), g.edges, np.stack(states))
    want = d.real[np.arange(len(bonds)), bonds]
    if prec == "bf16x2":  # (the sampler multiplies in BF16)
        lim = BD.bond_bounds(th, F, L, Ah, g.edges, g.J, np.stack(states), "bf16")[1][np.arange(len(bonds)), bonds]
    else:
        lim = (1e-5 if prec == "fp32" else 1e-9) * np.maximum(SC.delta_scale(th, F, L, Ah, g.edges, np.stack(states)), 1.0)
        lim = lim[np.arange(len(bonds)), bonds]
    assert len(bonds) > 50 and np.all(np.abs(np.array(got) - want) <= lim), np.max(np.abs(np.array(got) - want) - lim)


@pytest.mark.parametrize("F,L", [(32, 3), (64, 2)])
def test_fp32_local_energy_at_weight_scale_3(torch, F, L):
    g = W.kagome(3)
    theta, th = _rounded(torch, W.random_theta(F, L, seed=F + L, scale=3.0), F, "fp32")
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_FP32)
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    s = W.random_spins(g.n_sites, 3, seed=3)
    dl = gna.local_energy(graph, model, theta, torch.tensor(s, device="cuda"), gna.ELOC_INCREMENTAL, bonds=True)[1].cpu().numpy()

    def ratios(t):
        d = hz.bond_log_ratios(lambda x: gcn.logpsi_complex(t, F, L, Ah, x), g.edges, s).real
        return np.where(np.isnan(d), 0.0, d)

    want, rng, moved = ratios(th), np.random.default_rng(0), 0.0
    for _ in range(4):
        moved = np.maximum(moved, np.abs(ratios(th * (1.0 + 2.0 ** -23 * rng.uniform(-1, 1, th.size))) - want))
    lim = 1e-5 * np.maximum(SC.delta_scale(th, F, L, Ah, g.edges, s), 1.0) + 8.0 * moved
    assert np.all(np.abs(dl - want) <= lim), np.max(np.abs(dl - want) - lim)


@pytest.mark.parametrize("prec", list(PREC))
@pytest.mark.parametrize("name,scale", [("kagome2", 0.3), ("kagome2", 2.0), ("two", None)])
def test_a_bias_that_is_not_a_number_shows_in_the_energy(torch, prec, name, scale):
    # "two": the only rows are the exchanged pair's, and the feature swings by more than 100
    F, L = 16, 2 if scale else 1
    g = W.kagome(2) if scale else W.two_site()
    th = W.random_theta(F, L, seed=1, scale=scale) if scale else _swinging(F, L, 56.0, -5.0)
    theta, _ = _rounded(torch, th, F, prec)
    theta[3 * F + 2 * F * F] = float("nan")  # b of feature 0
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, PREC[prec])
    s = torch.tensor(W.random_spins(g.n_sites, 8, seed=1), device="cuda")
    E = gna.local_energy(graph, model, theta, s, gna.ELOC_INCREMENTAL)
    assert torch.isnan(E[:, 0]).all()


def test_a_ratio_beyond_float32_makes_the_energy_infinite(torch):
    # real log Psi (Im w_r = 0) with ratios of up to exp(+-several hundred), summed with positive J
    F, L = 16, 2
    g = W.kagome(2)
    th = W.random_theta(F, L, seed=1, scale=0.3)
    o = 4 * F + 2 * F * F
    th[o:o + 2 * F:2] *= 1000.0
    th[o + 1:o + 2 * F:2] = 0.0
    theta, th = _rounded(torch, th, F, "fp32")
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_FP32)
    s = W.random_spins(g.n_sites, 40, seed=1)
    st = torch.tensor(s, device="cuda")
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    d = np.nanmax(hz.bond_log_ratios(lambda x: gcn.logpsi_complex(th, F, L, Ah, x), g.edges, s).real, axis=1)
    assert (d > 95).sum() > 10 and not ((d > 80) & (d < 95)).any()
    for mode in (gna.ELOC_FULL, gna.ELOC_INCREMENTAL):
        E = gna.local_energy(graph, model, theta, st, mode)[:, 0].cpu().numpy()
        assert np.array_equal(np.isposinf(E), d > 95) and np.isfinite(E[d < 80]).all()


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-9)])
@pytest.mark.parametrize("F,L,sign", [(16, 1, 1.0), (32, 3, -1.0)])
def test_an_infinite_weight_saturates_its_unit(torch, prec, tol, F, L, sign):
    # as in the recomputing mode: tanh(+-inf) = +-1, and where the unit's input does not change its 0 x inf is no term
    g = W.kagome(3)
    theta, th = _rounded(torch, W.random_theta(F, L, seed=F, scale=0.3), F, prec)
    theta[3 * F + 7] = sign * float("inf")
    th[3 * F + 7] = sign * 1e30
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, PREC[prec])
    s = W.random_spins(g.n_sites, 5, seed=3)
    st = torch.tensor(s, device="cuda")
    full = gna.local_energy(graph, model, theta, st, gna.ELOC_FULL)
    E = gna.local_energy(graph, model, theta, st, gna.ELOC_INCREMENTAL)
    assert torch.isfinite(full).all()
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    lim = 2 * tol * np.maximum(SC.eloc_scale(th, F, L, Ah, g.edges, g.J, s), 1.0)
    assert np.all((E - full).abs().cpu().numpy().max(axis=1) <= lim)
