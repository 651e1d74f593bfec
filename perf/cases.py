"""What is timed of this framework: calls of its public entry points (paper_2011_12453_gb300.gna
and .vmc) over the sizes that the repository's own configurations, tests and benchmark use.

The work of a user is variational Monte Carlo: Metropolis sweeps of many chains, the local
energy and log Psi of their samples, the reweighted energy gradient and an update of the
parameters, and, with the learned proposal, its training step.  The kinds of case are those
calls: "forward", "eloc" (local energy with log Psi), "update" (one ISGO gradient and its SGD
step), "sweep" (plain or learned moves), "backward" (log Psi through autograd) and "proposal"
(gradient of the proposal network).

The library writes energies, log Psi and gradients into float64 containers whatever the
model's arithmetic; a pass returns them in the type that the model computes in (float32 for
FP32, BF16 and BF16X2 models, whose parameters are float32; float64 for FP64 models).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2011_12453_gb300 import gna, vmc, workloads

PREC = {"fp64": gna.PREC_FP64, "fp32": gna.PREC_FP32, "bf16": gna.PREC_BF16, "bf16x2": gna.PREC_BF16X2}
PROPOSAL_EPS = 0.1
UPDATE_LR = 5e-4  # the step size of the repository's ISGO runs
HOPPING = 0.5     # bosons: t of the 12-site setups, V = 1
LN_EPS = 1e-6
HOT_CHUNK = 1 << 27  # float64 elements of one layer that the 64-bit reference holds at a time


def listed():
    return [
        # one configuration's log Psi: the smallest call there is, all latency
        dict(name="forward_one", kind="forward", lattice="kagome", size=6, L=4, F=32, prec="bf16x2", batch=1, scale=0.1),
        # the benchmark's local energy: Kagome 6x6x3, one sample of each of 16384 chains
        dict(name="eloc_kagome108", kind="eloc", lattice="kagome", size=6, L=4, F=32, prec="bf16x2", batch=16384, scale=0.1),
        # triangular 12x12, F = 48; a batch as grouping duplicates leaves it (odd)
        dict(name="eloc_triangular144", kind="eloc", lattice="triangular", size=12, L=4, F=48, prec="bf16x2", batch=4001, scale=0.1),
        # the largest system: Kagome 12x12x3, L = 6, F = 64, where balls cover hundreds of sites
        dict(name="eloc_kagome432", kind="eloc", lattice="kagome", size=12, L=6, F=64, prec="bf16x2", batch=512, scale=0.1),
        # one reuse update on an irregular graph with grouped samples (counts), parameters away from the start
        dict(name="update_random", kind="update", lattice="random", size=77, L=3, F=32, prec="bf16x2", batch=4096, scale=0.3),
        # one update of the paper's own model (hard-core bosons, ReLU + layer norm) on 108 sites, FP32
        dict(name="update_bosons108_fp32", kind="update", lattice="kagome", size=6, L=3, F=16, prec="fp32", batch=1024, scale=0.1, act="relu_ln"),
        # one update in FP64 on the 12-site lattice that exact diagonalisation checks
        dict(name="update_kagome12_fp64", kind="update", lattice="kagome", size=2, L=2, F=16, prec="fp64", batch=1024, scale=0.1),
        # the benchmark's sampling: one recorded sweep of 16384 chains, plain moves
        dict(name="sweep_kagome108", kind="sweep", lattice="kagome", size=6, L=4, F=32, prec="bf16x2", batch=16384, scale=0.1, sweeps=1),
        # FP64 sampling of the 12-site lattice: 1024 chains, ten sweeps a call
        dict(name="sweep_kagome12_fp64", kind="sweep", lattice="kagome", size=2, L=2, F=16, prec="fp64", batch=1024, scale=0.1, sweeps=10),
        # learned moves on a random graph, FP32
        dict(name="sweep_random_learned", kind="sweep", lattice="random", size=65, L=3, F=32, prec="fp32", batch=4096, scale=0.3, sweeps=1, learned=True),
        # log Psi and its parameter gradient through autograd, F = 48
        dict(name="backward_triangular144", kind="backward", lattice="triangular", size=12, L=4, F=48, prec="bf16x2", batch=4001, scale=0.3),
        # a training step's gradient of the proposal network on the chains of a random graph
        dict(name="proposal_random", kind="proposal", lattice="random", size=65, L=3, F=32, prec="fp32", batch=4096, scale=0.3),
    ]


# ---------------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------------

# Most operations of a drawn case, by kind and arithmetic, so that none costs more than the
# largest listed ones (the CUDA-core paths run at lower rates).
MOST_FLOPS = {"forward": 2e11, "eloc": 4e11, "update": 2e11, "sweep": 1.5e11, "backward": 2e11, "proposal": 4e10}
SLOWER = {"fp64": 0.02, "fp32": 0.1, "bf16": 1.0, "bf16x2": 1.0}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["forward", "eloc", "eloc", "update", "update", "sweep", "sweep", "backward", "proposal"])
    lattice = rng.choice(["kagome", "triangular", "random"])
    case = dict(kind=kind, lattice=lattice,
                size=rng.randint(2, 8) if lattice == "kagome" else rng.randint(4, 14) if lattice == "triangular" else rng.randint(32, 96),
                L=rng.randint(2, 4), F=rng.choice([16, 32, 48, 64]), scale=rng.choice([0.1, 0.3]))
    if kind == "proposal":
        case["prec"] = "fp32"
    elif kind == "sweep":
        case["prec"] = rng.choice(["bf16x2", "bf16x2", "fp32", "fp64"])
        case["sweeps"] = rng.randint(1, 3)
        if rng.random() < 0.3:
            case.update(prec="fp32", learned=True, sweeps=1, lattice="random", size=rng.randint(32, 96))
    else:
        case["prec"] = rng.choice(["bf16x2", "bf16x2", "bf16x2", "bf16", "fp32", "fp64"])
        if case["prec"] in ("fp32", "fp64") and kind == "update" and rng.random() < 0.5:
            case.update(act="relu_ln", scale=0.1)
    most = MOST_FLOPS[kind] * SLOWER[case["prec"]] * (case["F"] / 64.0 if case["prec"] in ("bf16", "bf16x2") else 1.0)
    one = work(dict(case, batch=1))["flops"]
    case["batch"] = _log_int(rng, 1 if kind != "proposal" else 8, int(max(8, min(16384, most / one))))
    return case


# ---------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------

def _lattice(case):
    if case["lattice"] == "kagome":
        return workloads.kagome(case["size"])
    if case["lattice"] == "triangular":
        return workloads.triangular(case["size"], case["size"])
    n = case["size"]
    return workloads.erdos_renyi(n, 4.0 / (n - 1), 1000 + n, J_range=(0.5, 1.5))


def _bonds(case, lat):
    """(Jz, Jxy, hz, c) of the bonds: Heisenberg, or hard-core bosons for the paper's model."""
    one = np.ones(lat.n_edges)
    if case.get("act") == "relu_ln":
        return one, -2.0 * HOPPING * one, 0.5 * one, 0.25 * one
    return lat.J, lat.J, 0.0 * one, 0.0 * one


class _Inputs:
    """Seeded inputs alone (no framework object): shared by prepare() and exact()."""

    def __init__(self, case, seed):
        dev = torch.device("cuda")
        g = torch.Generator(device=dev)
        g.manual_seed(int(seed))
        lat = _lattice(case)
        n, B, F = lat.n_sites, case["batch"], case["F"]
        dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
        theta = workloads.random_theta(F, case["L"], seed=int(seed) % (1 << 31), scale=case["scale"])
        if case.get("act") == "relu_ln":  # the paper's real one-unit head
            P = theta.size
            theta[P - 2 * (F + 3) + 1::2] = 0.0
        self.lat = lat
        self.theta = torch.tensor(theta, dtype=dtype, device=dev)
        keys = torch.rand((B, n), generator=g, device=dev)
        rank = keys.argsort(dim=1).argsort(dim=1)
        self.spins = torch.where(rank < n // 2, 1, -1).to(torch.int8).contiguous()  # S_z = 0 (odd n: one down more)
        if case["kind"] == "update":
            # the samples were drawn a few updates ago, at parameters close by
            step = torch.randn(self.theta.shape, generator=g, device=dev, dtype=torch.float64)
            if case.get("act") == "relu_ln":
                step = torch.where(self.theta.double() == 0, torch.zeros_like(step), step)
            self.theta_sampled = (self.theta.double() * (1.0 + 1e-3 * step)).to(dtype)
            self.counts = torch.randint(1, 4, (B,), generator=g, device=dev).double()
        if case["kind"] == "backward":
            # ISGO cotangents 2 p (E - mean E) at equal weights, of energies that vary with the configuration
            e = torch.tensor(np.asarray(lat.edges), dtype=torch.long, device=dev)
            J = torch.tensor(np.asarray(lat.J), dtype=torch.float64, device=dev)
            E = 0.1 * torch.randn((B, 2), generator=g, device=dev, dtype=torch.float64)
            E[:, 0] += (J / 4 * (self.spins[:, e[:, 0]] * self.spins[:, e[:, 1]])).sum(1)
            self.cot = (2.0 / B) * (E - E.mean(0, keepdim=True) if B > 1 else E)
        if case["kind"] == "proposal":
            self.dlogpsi = case["scale"] * torch.randn((B, lat.n_edges), generator=g, device=dev)
        if case["kind"] == "proposal" or case.get("learned"):
            self.params = torch.tensor(workloads.random_proposal_params(int(seed) % (1 << 31)), dtype=torch.float32, device=dev)


class _State:
    pass


def prepare(case, seed):
    x = _Inputs(case, seed)
    s = _State()
    s.kind, s.case = case["kind"], case
    act = gna.ACT_RELU_LN if case.get("act") == "relu_ln" else gna.ACT_TANH
    xxz = _bonds(case, x.lat) if act == gna.ACT_RELU_LN else None
    s.graph = gna.Graph(x.lat.n_sites, x.lat.edges, x.lat.J, case["L"], xxz=xxz)
    s.model = gna.Model(case["F"], case["L"], PREC[case["prec"]], act=act)
    s.theta, s.spins = x.theta, x.spins
    if s.kind == "update":
        s.start = x.theta.clone()
        s.logpsi0 = _logpsi_blocks(case, x.lat, x.theta_sampled, x.spins)
        s.counts = x.counts
    elif s.kind == "backward":
        s.theta.requires_grad_(True)
        s.cot = x.cot
    elif s.kind == "proposal":
        s.params, s.dlogpsi = x.params, x.dlogpsi
    elif s.kind == "sweep":
        s.chains = vmc.Chains(s.graph, s.model, s.theta, s.spins, seed=int(seed))
        s.proposal = x.params if case.get("learned") else None
    return s


def _computed(case, t):
    """t in the type that the model computes in."""
    return t if case["prec"] == "fp64" else t.float()


def run(s):
    c = s.case
    if s.kind == "forward":
        return _computed(c, gna.forward(s.graph, s.model, s.theta, s.spins))
    if s.kind == "eloc":
        E, lp = gna.local_energy_logpsi(s.graph, s.model, s.theta, s.spins)
        return {"eloc": _computed(c, E), "logpsi": _computed(c, lp)}
    if s.kind == "update":
        s.theta.copy_(s.start)  # back to the parameters the iteration keeps
        grad, stats = gna.isgo_grad(s.graph, s.model, s.theta, s.spins, s.logpsi0, counts=s.counts)
        gna.sgd_update(s.model, s.theta, grad, UPDATE_LR)
        return {"theta": s.theta, "stats": _computed(c, stats)}
    if s.kind == "sweep":
        samples, lp, accepted, _ = s.chains.sweep(c["sweeps"], record_every=c["sweeps"], proposal=s.proposal, eps=PROPOSAL_EPS)
        return {"samples": samples, "logpsi": _computed(c, lp), "accepted": accepted, "spins": s.chains.spins}
    if s.kind == "backward":
        lp = gna.gcn_logpsi(s.theta, s.spins, s.graph, s.model)
        (grad,) = torch.autograd.grad(lp, s.theta, s.cot)
        return {"logpsi": _computed(c, lp), "grad": grad}
    grad, loss = gna.proposal_grad(s.graph, s.spins, s.dlogpsi, s.params)
    return {"grad": grad.float(), "loss": loss.float()}


# ---------------------------------------------------------------------------------
# work that cannot be avoided
# ---------------------------------------------------------------------------------

def work(case):
    """Bytes: spins, parameters and results once.  Operations: the dense layers and the gathers
    of one forward per configuration, of the balls of every exchanged bond, and of the reverse
    pass, with the expected number of antiparallel bonds of a uniform S_z = 0 configuration."""
    lat = _lattice(case)
    n, E, F, L, B = lat.n_sites, lat.n_edges, case["F"], case["L"], case["batch"]
    real = 8 if case["prec"] == "fp64" else 4
    P = workloads.num_params(F, L)
    up = n // 2
    anti = E * 2.0 * up * (n - up) / (n * (n - 1.0))
    row = 4.0 * F * F + 2.0 * (2.0 * E / n) * F
    forward = L * n * row
    spins, par = float(B * n), float(P * real)
    if case["kind"] == "forward":
        return {"bytes": spins + par + 2 * B * real, "flops": B * forward}
    if case["kind"] == "backward":
        return {"bytes": spins + par * 2 + 2 * B * real + 2 * B * 8, "flops": B * 3 * forward}
    if case["kind"] == "proposal":
        rows = B * 2 * anti
        return {"bytes": spins + B * E * 4 + 2 * 4.0 * workloads.proposal_num_params(),
                "flops": rows * 2.0 * (2 * 9 * 64 + 3 * 64 * 64 + 2 * 64)}
    balls = gna.ball_sizes_host(n, lat.edges, L).astype(np.float64)  # [E][L+1]
    per_bond = float(balls[:, 1:].sum(1).mean()) * row
    if case["kind"] == "sweep":
        steps = case["sweeps"] * n
        flops = B * (forward + steps * anti / E * per_bond)
        if case.get("learned"):  # the pair's own candidates, before and after the exchange
            flops = B * (forward + steps * (per_bond + 4.0 * (2.0 * E / n) / 2 * 2 * (9 * 64 + 64 * 64 + 64)))
        return {"bytes": 3 * spins + par + 2 * B * real + 4 * B, "flops": flops}
    flops = B * (forward + anti * per_bond)
    if case["kind"] == "eloc":
        return {"bytes": spins + par + 4 * B * real, "flops": flops}
    return {"bytes": 2 * spins + 3 * par + 3 * 8 * B, "flops": flops + B * 3 * forward}


# ---------------------------------------------------------------------------------
# the same results in 64 bits, from plain torch
# ---------------------------------------------------------------------------------

def _params64(case, theta):
    """The parameter vector in 64 bits; W is a bfloat16 parameter of the tensor-core models."""
    F = case["F"]
    t = theta.detach().double().clone()
    if case["prec"] in ("bf16", "bf16x2"):
        w = slice(3 * F, 3 * F + 2 * F * F)
        t[w] = theta.detach()[w].to(torch.bfloat16).double()
    return t


def _neighbours(lat, dev):
    n = lat.n_sites
    nbr = [[] for _ in range(n)]
    for a, b in lat.edges.tolist():
        nbr[a].append(b)
        nbr[b].append(a)
    D = max(len(v) for v in nbr)
    idx = torch.zeros((D, n), dtype=torch.long)
    w = torch.zeros((D, n, 1), dtype=torch.float64)
    for v, us in enumerate(nbr):
        for k, u in enumerate(us):
            idx[k, v] = u
            w[k, v] = 1.0 / math.sqrt(len(us) * len(nbr[u]))
    return idx.to(dev), w.to(dev)


def _f(case, y):
    if case.get("act") != "relu_ln":
        return torch.tanh(y)
    r = torch.relu(y)
    d = r - r.mean(-1, keepdim=True)
    return d / torch.sqrt((d * d).mean(-1, keepdim=True) + LN_EPS)


def _logpsi(case, nb, t, spins):
    """log Psi [b][2] of Eq. (gcn), embedding and readout, for the parameters t in 64 bits."""
    F, L = case["F"], case["L"]
    idx, w = nb
    We, be, W, b = t[:2 * F].view(2, F), t[2 * F:3 * F], t[3 * F:3 * F + 2 * F * F].view(2 * F, F), t[3 * F + 2 * F * F:4 * F + 2 * F * F]
    o = 4 * F + 2 * F * F
    wr, br = t[o:o + 2 * (F + 2)].view(F + 2, 2), t[o + 2 * (F + 2):]
    up = spins > 0
    H = _f(case, We + be)[(~up).long()]
    for _ in range(L):
        M = w[0] * H[:, idx[0]]
        for k in range(1, idx.shape[0]):
            M = M + w[k] * H[:, idx[k]]
        H = _f(case, M @ W[:F] + H @ W[F:] + b)
    n_up = up.sum(1, keepdim=True).double()
    return H.sum(1) @ wr[:F] + n_up * wr[F] + (spins.shape[1] - n_up) * wr[F + 1] + br


def _logpsi_blocks(case, lat, theta, spins):
    nb, t = _neighbours(lat, spins.device), _params64(case, theta)
    step = max(1, HOT_CHUNK // (lat.n_sites * case["F"]))
    return torch.cat([_logpsi(case, nb, t, spins[i:i + step]) for i in range(0, spins.shape[0], step)])


def _eloc(case, lat, t, spins, lp):
    dev = spins.device
    nb = _neighbours(lat, dev)
    Jz, Jxy, hz, cb = (torch.tensor(np.asarray(a), dtype=torch.float64, device=dev) for a in _bonds(case, lat))
    e = torch.tensor(np.asarray(lat.edges), dtype=torch.long, device=dev)
    si, sj = spins[:, e[:, 0]].double(), spins[:, e[:, 1]].double()
    E = torch.zeros_like(lp)
    E[:, 0] = (Jz / 4 * si * sj + hz / 2 * (si + sj) + cb).sum(1)
    rows, bonds = torch.nonzero(si != sj, as_tuple=True)
    step = max(1, HOT_CHUNK // (lat.n_sites * case["F"]))
    for k in range(0, rows.numel(), step):
        r, b = rows[k:k + step], bonds[k:k + step]
        s = spins[r].clone()
        at = torch.arange(r.numel(), device=dev)
        s[at, e[b, 0]], s[at, e[b, 1]] = spins[r, e[b, 1]], spins[r, e[b, 0]]
        d = _logpsi(case, nb, t, s) - lp[r]
        amp = Jxy[b] / 2 * torch.exp(d[:, 0])
        E.index_add_(0, r, torch.stack([amp * torch.cos(d[:, 1]), amp * torch.sin(d[:, 1])], 1))
    return E


def _vjp(case, lat, t, spins, cot):
    nb = _neighbours(lat, spins.device)
    t = t.clone().requires_grad_(True)
    step = max(1, HOT_CHUNK // (8 * lat.n_sites * case["F"]))
    grad = torch.zeros_like(t)
    for i in range(0, spins.shape[0], step):
        lp = _logpsi(case, nb, t, spins[i:i + step])
        grad += torch.autograd.grad(lp, t, cot[i:i + step])[0]
    return grad.detach()


def _proposal(x):
    """Gradient and loss of the proposal network's training step."""
    lat, dev = x.lat, x.spins.device
    s = x.spins.double()
    n = lat.n_sites
    A = torch.zeros((n, n), dtype=torch.float64, device=dev)
    e = torch.tensor(np.asarray(lat.edges), dtype=torch.long, device=dev)
    A[e[:, 0], e[:, 1]] = 1.0
    A[e[:, 1], e[:, 0]] = 1.0
    d = A.sum(1)
    n1 = s @ A
    q = n1 / d
    qs = q @ A
    J = torch.tensor(np.asarray(lat.J), dtype=torch.float64, device=dev)
    feats, target = [], []
    for a, b in ((0, 1), (1, 0)):
        i, j = e[:, a], e[:, b]
        one = torch.ones_like(s[:, i])
        other = lambda v: torch.clamp(d[v] - 1, min=1)  # noqa: E731
        feats.append(torch.stack([s[:, i], s[:, j], J * one, one / d[i], one / d[j], (n1[:, i] - s[:, j]) / other(i), (n1[:, j] - s[:, i]) / other(j),
                                  (qs[:, i] - q[:, j]) / other(i), (qs[:, j] - q[:, i]) / other(j)], -1))
        target.append(torch.clamp(2.0 * x.dlogpsi.double(), max=0.0))
    anti = torch.cat([(s[:, e[:, 0]] != s[:, e[:, 1]])] * 2, 1)
    X, T = torch.cat(feats, 1)[anti], torch.cat(target, 1)[anti]
    p = x.params.double().requires_grad_(True)
    W1, b1, W2, b2, w3, b3 = p[:576].view(9, 64), p[576:640], p[640:4736].view(64, 64), p[4736:4800], p[4800:4864], p[4864]
    grad, loss = torch.zeros_like(p), 0.0
    for k in range(0, X.shape[0], 1 << 19):
        z = torch.tanh(torch.tanh(X[k:k + (1 << 19)] @ W1 + b1) @ W2 + b2) @ w3 + b3
        part = ((z - T[k:k + (1 << 19)]) ** 2).sum() / max(1, X.shape[0])
        grad = grad + torch.autograd.grad(part, p)[0]
        loss = loss + part.detach()
    return {"grad": grad.detach(), "loss": loss.reshape(1)}


def exact(case, seed):
    if case["kind"] == "sweep":
        return None  # accept decisions are made in the model's arithmetic
    flops = work(case)["flops"]
    if case["kind"] in ("eloc", "update"):  # every exchanged bond costs a whole forward here
        lat = _lattice(case)
        n = lat.n_sites
        flops = case["batch"] * lat.n_edges / 2 * case["L"] * n * (4.0 * case["F"] ** 2 + 120.0 * case["F"])
    if flops > 2e13:
        return None
    x = _Inputs(case, seed)
    if case["kind"] == "proposal":
        return _proposal(x)
    t = _params64(case, x.theta)
    lp = _logpsi_blocks(case, x.lat, x.theta, x.spins)
    if case["kind"] == "forward":
        return lp
    if case["kind"] == "backward":
        return {"logpsi": lp, "grad": _vjp(case, x.lat, t, x.spins, x.cot)}
    E = _eloc(case, x.lat, t, x.spins, lp)
    if case["kind"] == "eloc":
        return {"eloc": E, "logpsi": lp}
    lp0 = _logpsi_blocks(case, x.lat, x.theta_sampled, x.spins)
    p = torch.softmax(2.0 * (lp - lp0)[:, 0] + torch.log(x.counts), 0)
    mean = (p[:, None] * E).sum(0)
    dE = E - mean
    grad = _vjp(case, x.lat, t, x.spins, 2.0 * p[:, None] * dE)
    stats = torch.stack([mean[0], mean[1], (p * (dE * dE).sum(1)).sum(), 1.0 / (p * p / x.counts).sum()])
    return {"theta": x.theta.double() - UPDATE_LR * grad, "stats": stats}
