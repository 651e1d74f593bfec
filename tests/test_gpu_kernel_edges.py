"""Kernels whose work is split over warps, tiles of 16 or 128 rows and a few blocks, at the sizes where
the split can go wrong, against the FP64 oracle.

- BF16 sampler (mtile.cu): balls on either side of a multiple of 16 rows, odd degrees, isolated
  sites, one layer and six, chains that do not fill a block, and the graphs whose rows move from
  shared memory to the workspace.  Bonds, no-ops and decisions are replayed exactly with the
  oracle's Philox words; Delta within 2e-3 (the BF16 tolerance of the other sampler tests at weight
  scale 0.1, where the balls are as large; per-row roundings of 2^-9 add as in a random walk).
- FP64 sampler and local energy (dbl.cu): F that is no multiple of 16 or 32, one, two and four warps a
  chain, weights large enough for swings across saturation.  1e-9: float64 sums of some
  thousand terms, with the margin of the other FP64 tests.
- Importance weights (isgo.cu): batches around one block, around the whole first pass (152 blocks
  of 128) and with counts.  1e-11 relative: float64 sums of 4e4 positive terms.
- Proposal gradient (prop.cu): configurations without antiparallel bonds, a number of rows on either
  side of the 128-row tiles, few configurations (several parts each).  1e-4 of the largest
  entry, as the other gradient test (FP32 network)."""
import numpy as np
import pytest

from oracle import gcn, heisenberg as hz, isgo, proposal as P, sampler
from paper_2011_12453_gb300 import build as B, gna, workloads as W

from bounds import bf16_round

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


GRAPHS = {"two": W.two_site, "ring40": lambda: W.ring(40), "isolated": _isolated, "complete9": lambda: W.complete(9),
          "bipartite": lambda: W.complete_bipartite(3, 14), "kagome2": lambda: W.kagome(2), "kagome3": lambda: W.kagome(3),
          "kagome6": lambda: W.kagome(6), "tri14": lambda: W.triangular(14, 14), "er30": lambda: W.erdos_renyi(30, 0.2, seed=5)}


def _replay(g, s0, tr, final, seed, step0, prec):
    """Checks bonds, no-ops and decisions of every step; returns [(state, bond, Delta)] of the proposals."""
    out, near = [], 0
    for c in range(s0.shape[0]):
        s = s0[c].copy()
        for k in range(tr.shape[1]):
            w = sampler.step_words(seed, c, step0 + k)
            e = sampler.bond_index(w[0], g.n_edges)
            assert int(tr[c, k, 0]) == e and tr[c, k, 3] == 1.0
            i, j = g.edges[e]
            if s[i] == s[j]:
                assert np.isnan(tr[c, k, 2]) and tr[c, k, 1] == 0
                continue
            out.append((s.copy(), e, tr[c, k, 2]))
            u = sampler.uniform(w[1], prec)
            if abs(float(u) - np.exp(2 * tr[c, k, 2])) < 1e-6:
                near += 1
            else:
                assert bool(tr[c, k, 1]) == sampler.accept(u, tr[c, k, 2], prec)
            if tr[c, k, 1]:
                s[[i, j]] = s[[j, i]]
        assert np.array_equal(s, final[c])
    assert near <= 2 + s0.shape[0] // 16
    return out


def _sweep(torch, g, F, L, prec, scale, C, sweeps, seed=31, step0=77):
    th = W.random_theta(F, L, seed=F + L, scale=scale)
    model = gna.Model(F, L, prec)
    theta = torch.tensor(th, dtype=model.theta_dtype(), device="cuda")
    th = theta.double().cpu().numpy()
    graph = gna.Graph.from_workload(g, L)
    s0 = W.random_spins(g.n_sites, C, seed=4)
    ch = torch.tensor(s0, device="cuda")
    _, _, acc, tr = gna.metropolis_sweep(graph, model, theta, ch, sweeps, 0, seed, step0, trace=True)
    tr, final = tr.cpu().numpy(), ch.cpu().numpy()
    assert np.array_equal(acc.cpu().numpy(), tr[:, :, 1].sum(axis=1))
    # the same chains without a trace and with a record after each sweep
    ch2 = torch.tensor(s0, device="cuda")
    samples, lp, acc2, _ = gna.metropolis_sweep(graph, model, theta, ch2, sweeps, 1, seed, step0)
    assert torch.equal(ch2, ch) and torch.equal(acc2, acc) and torch.equal(samples[-1], ch)
    want = gna.forward(graph, model, theta, samples[-1].contiguous()).cpu().numpy()
    tol = 1e-9 if prec == gna.PREC_FP64 else 2e-2
    assert np.abs(lp[-1].cpu().numpy() - want).max() <= tol * max(1.0, np.abs(want).max())
    return th, s0, tr, final


def _deltas(th, F, L, g, props, n):
    pick = np.random.default_rng(0).choice(len(props), size=min(n, len(props)), replace=False)
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    d = hz.bond_log_ratios(lambda x: gcn.logpsi_complex(th, F, L, Ah, x), g.edges, np.stack([props[p][0] for p in pick]))
    want = d.real[np.arange(len(pick)), [props[p][1] for p in pick]]
    return np.array([props[p][2] for p in pick]), want


@pytest.mark.parametrize("name,F,L,C,sweeps", [
    ("two", 16, 1, 3, 20), ("ring40", 16, 8, 5, 1), ("ring40", 48, 7, 2, 1), ("isolated", 64, 2, 153, 1),
    ("complete9", 32, 2, 5, 4), ("bipartite", 48, 3, 4, 3), ("kagome3", 32, 5, 5, 2), ("er30", 64, 4, 3, 2),
    ("kagome6", 64, 4, 3, 1), ("tri14", 64, 6, 2, 1)])
def test_bf16_sampler(torch, name, F, L, C, sweeps):
    g = GRAPHS[name]()
    th, s0, tr, final = _sweep(torch, g, F, L, gna.PREC_BF16, 0.1, C, sweeps)
    props = _replay(g, s0, tr, final, 31, 77, "fp32")
    w = slice(3 * F, 3 * F + 2 * F * F)
    th[w] = bf16_round(th[w])
    got, want = _deltas(th, F, L, g, props, 12 if g.n_sites < 100 else 3)
    assert np.abs(got - want).max() <= 2e-3


@pytest.mark.parametrize("F,C,scale", [(8, 1, 0.3), (33, 160, 0.3), (64, 700, 0.3), (16, 5, 2.0)])
def test_fp64_sampler(torch, F, C, scale):
    g = W.kagome(2)
    th, s0, tr, final = _sweep(torch, g, F, 2, gna.PREC_FP64, scale, C, 2)
    n = min(C, 16)
    props = _replay(g, s0[:n], tr[:n], final[:n], 31, 77, "fp64")
    got, want = _deltas(th, F, 2, g, props, 20)
    assert np.abs(got - want).max() <= 1e-9 * max(1.0, np.abs(want).max())


@pytest.mark.parametrize("name,F,L,scale", [("two", 8, 1, 0.3), ("isolated", 33, 2, 0.3), ("bipartite", 64, 2, 2.0), ("kagome3", 16, 3, 2.0)])
def test_fp64_local_energy(torch, name, F, L, scale):
    g = GRAPHS[name]()
    th = W.random_theta(F, L, seed=2, scale=scale)
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_FP64)
    s = W.random_spins(g.n_sites, 3, seed=3)
    E, dl = gna.local_energy(graph, model, torch.tensor(th, device="cuda"), torch.tensor(s, device="cuda"), gna.ELOC_INCREMENTAL,
                             bonds=True)
    Ah = gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges))
    fn = lambda x: gcn.logpsi_complex(th, F, L, Ah, x)
    want = hz.local_energy(fn, g.edges, g.J, s)
    d = hz.bond_log_ratios(fn, g.edges, s)
    i, j = g.edges[:, 0], g.edges[:, 1]
    terms = np.abs(np.asarray(g.J)) / 2 * np.exp(np.where(s[:, i] != s[:, j], d.real, 0.0))
    mag = terms.sum(axis=1) + np.abs(np.asarray(g.J)).sum()
    got = E.cpu().numpy()
    assert (np.abs(got[:, 0] + 1j * got[:, 1] - want) <= 1e-9 * mag).all()


@pytest.mark.parametrize("n", [1, 127, 129, 128 * 152, 128 * 152 + 1, 40000])
@pytest.mark.parametrize("counts", [False, True])
def test_isgo_weights(torch, n, counts):
    rng = np.random.default_rng(n)
    lp, lp0, E = rng.normal(size=(n, 2)), rng.normal(size=(n, 2)), rng.normal(size=(n, 2))
    c = rng.integers(1, 9, size=n) if counts else None
    t = lambda x: torch.tensor(x, device="cuda")
    for _ in range(2):  # the second call starts from what the first left behind
        cot, stats = gna.isgo_weights(t(lp), t(lp0), t(E), t(c.astype(np.float64)) if counts else None)
    p = isgo.weights(lp, lp0, c)
    Ebar, var, ess = isgo.statistics(p, E[:, 0] + 1j * E[:, 1], c)
    want = np.array([Ebar.real, Ebar.imag, var, ess])
    assert np.abs(stats.cpu().numpy() - want).max() <= 1e-11 * max(1.0, np.abs(want).max())
    wc = isgo.cotangents(p, E[:, 0] + 1j * E[:, 1], Ebar)
    assert np.abs(cot.cpu().numpy() - wc).max() <= 1e-11 * np.abs(p).max() * 10


@pytest.mark.parametrize("name,n,n_up", [("two", 1, None), ("two", 129, None), ("ring40", 3, None), ("kagome2", 1, None),
                                         ("kagome2", 61, None), ("er30", 2, 1), ("bipartite", 5, None), ("ring40", 40, 0)])
def test_proposal_gradient(torch, name, n, n_up):
    g = GRAPHS[name]()
    graph = gna.Graph.from_workload(g, 1)
    p32 = torch.tensor(W.random_proposal_params(3, 0.5), dtype=torch.float32, device="cuda")
    s = W.random_spins(g.n_sites, n, seed=4, n_up=n_up)
    if n > 2:
        s[n // 2] = 1  # a configuration without antiparallel bonds
    dl = np.random.default_rng(5).normal(scale=0.5, size=(n, g.n_edges)).astype(np.float32)
    grad, loss = gna.proposal_grad(graph, torch.tensor(s, device="cuda"), torch.tensor(dl, device="cuda"), p32)
    phi, tgt = P.training_rows(P.Topology(g.n_sites, g.edges, g.J), s, dl.astype(np.float64))
    if len(tgt) == 0:
        assert torch.all(grad == 0) and loss.item() == 0
        return
    want_loss, want = P.loss_and_grad(p32.double().cpu().numpy(), phi, tgt)
    assert abs(loss.item() - want_loss) <= 1e-4 * abs(want_loss)
    np.testing.assert_allclose(grad.cpu().numpy(), want, rtol=0, atol=1e-4 * np.abs(want).max())


@pytest.mark.parametrize("name,F,L,C", [("kagome2", 5, 2, 3), ("kagome2", 10, 2, 40), ("er30", 20, 3, 5), ("isolated", 32, 2, 7),
                                        ("complete9", 4, 1, 9), ("kagome3", 32, 3, 5), ("er30", 48, 2, 3)])
def test_fp32_sampler(torch, name, F, L, C):
    # Delta in FP32: 1e-4 of its size or of one (rounding 6e-8 of each of some thousand terms)
    g = GRAPHS[name]()
    th, s0, tr, final = _sweep(torch, g, F, L, gna.PREC_FP32, 0.3, C, 2)
    props = _replay(g, s0, tr, final, 31, 77, "fp32")
    got, want = _deltas(th, F, L, g, props, 20)
    assert np.abs(got - want).max() <= 1e-4 * max(1.0, np.abs(want).max())


@pytest.mark.parametrize("name,F,L", [("er30", 32, 3), ("er30", 20, 2), ("complete9", 16, 2), ("kagome3", 48, 2), ("kagome2", 5, 2)])
def test_fp32_learned_moves_as_fp64(torch, name, F, L):
    # the first step of 400 chains: the same bond and kind as the FP64 sampler's (checked against the
    # oracle elsewhere), the log acceptance ratio within 1e-4 of its size or of one; a chain may
    # pick another partner where its uniform lies within 1e-6 of a probability (at most 2 of 400)
    g = GRAPHS[name]()
    th32 = torch.tensor(W.random_theta(F, L, seed=7, scale=0.3), dtype=torch.float32, device="cuda")
    p32 = torch.tensor(W.random_proposal_params(3, 0.5), dtype=torch.float32, device="cuda")
    graph = gna.Graph.from_workload(g, L)
    s0 = W.random_spins(g.n_sites, 400, seed=4)
    tr = {}
    for prec, th in ((gna.PREC_FP32, th32), (gna.PREC_FP64, th32.double())):
        ch = torch.tensor(s0, device="cuda")
        tr[prec] = gna.metropolis_sweep(graph, gna.Model(F, L, prec), th, ch, 1, 0, 31, 0, trace=True, proposal=p32)[3].cpu().numpy()[:, 0]
        x = ch.cpu().numpy()
        assert np.array_equal((x > 0).sum(axis=1), (s0 > 0).sum(axis=1))
    a, b = tr[gna.PREC_FP32], tr[gna.PREC_FP64]
    same = a[:, 0] == b[:, 0]
    assert same.sum() >= 398 and np.array_equal(a[:, 3], b[:, 3])
    assert np.array_equal(np.isnan(a[same, 2]), np.isnan(b[same, 2]))
    ok = same & ~np.isnan(b[:, 2])
    assert ok.sum() > 100
    assert (np.abs(a[ok, 2] - b[ok, 2]) <= 1e-4 * np.maximum(1.0, np.abs(b[ok, 2]))).all()


@pytest.mark.parametrize("name,F,L,n", [("two", 16, 1, 1), ("isolated", 64, 3, 5), ("ring40", 48, 2, 153), ("kagome6", 32, 4, 1),
                                        ("kagome6", 64, 2, 700), ("tri14", 64, 2, 400), ("bipartite", 16, 3, 17)])
def test_bf16x2_forward(torch, name, F, L, n):
    # against the forward inside the local energy (the same sums: equal), and on a few
    # configurations against the oracle: 2^-16 operands, some hundred sites, as the other forward tests
    g = GRAPHS[name]()
    theta = torch.tensor(W.random_theta(F, L, seed=F, scale=0.3), dtype=torch.float32, device="cuda")
    graph, model = gna.Graph.from_workload(g, L), gna.Model(F, L, gna.PREC_BF16X2)
    s = W.random_spins(g.n_sites, n, seed=9)
    st = torch.tensor(s, device="cuda")
    lp = gna.forward(graph, model, theta, st)
    assert torch.equal(lp, gna.local_energy_logpsi(graph, model, theta, st)[1])
    th = theta.double().cpu().numpy()
    w = slice(3 * F, 3 * F + 2 * F * F)
    th[w] = bf16_round(th[w])
    want = gcn.logpsi(th, F, L, gcn.norm_adjacency(gcn.adjacency(g.n_sites, g.edges)), s[-3:])
    assert np.abs(lp[-3:].cpu().numpy() - want).max() <= 2e-4 * max(1.0, np.abs(want).max())
