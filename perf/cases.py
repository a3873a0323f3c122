"""Performance cases of the QAOA / DQAOA path: what a program that uses this library has it do.

Ten kinds of work, each through the public entry points: the single-instance calls (build the
energies, run the layers, read <C> and the most probable bitstrings), the single-instance
gradient, a complex128 parameter grid, a batch of equal sub-QUBOs in one plan, the DQAOA cycle, the
DQAOA cycle fed by measured shots, one training step of an uneven batch, one large instance, a
served set of optimise-and-sample jobs, and measurement shots of a state.

Q entries are uniform on [-1, 1] (normal for the training batch), gamma uniform on [0, pi], beta on
[0, pi/2]: the distributions of the configurations in bench.py and synth/. <C>, gradients and
probabilities of a complex64 run are handed on in the precision of its parameters (float32), as a
training loop or a report does; the complex128 grid keeps float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_10531_gb300 as q
from paper_2506_10531_gb300 import serve, train

DEV = "cuda"


def listed():
    return [
        # one small QUBO through the single-instance calls: five launches, latency alone (n = 8 is
        # the smallest size of the uneven configuration)
        dict(name="single_n8", kind="single", n=8, p=1, k=4),
        # one QUBO of a size between the tiers, odd n: the same calls on a state of 4 MB
        dict(name="single_n19", kind="single", n=19, p=3, k=8),
        # the gradient of one instance, as an optimiser outside the library asks for it
        dict(name="grad_n20", kind="grad", n=20, p=4),
        # the plain configuration: a 256-point parameter grid of one n = 10 QUBO in complex128
        dict(name="grid_n10_z", kind="grid", n=10, p=1, points=256, k=8),
        # the sub-QUBOs of a Max-Cut sized cycle (500 of n = 12), solved as one plan for their most
        # probable bitstring (the measured candidate)
        dict(name="batch_n12", kind="batch", n=12, p=3, m=500, k=1),
        # larger sub-QUBOs (the paper goes to 28 variables), an odd number of them
        dict(name="batch_n17", kind="batch", n=17, p=5, m=101, k=2),
        # the headline configuration: three DQAOA cycles on a resident N = 1000 QUBO
        dict(name="cycle_n16", kind="cycle", N=1000, m=256, n=16, p=3, k=8, cycles=3),
        # the paper-literal cycle: sub-solutions read from measured shots
        dict(name="sampled_n12", kind="sampled", N=500, m=128, n=12, p=2, shots=1024),
        # one training step of an uneven batch (n 8..24, p 1..6): <C> and adjoint gradients
        dict(name="train_n8_24", kind="train", lo=8, hi=24, p=6, m=48, mix=3),
        # the large configuration: one n = 30 instance streamed through HBM
        dict(name="large_n30", kind="large", n=30, p=2, k=8),
        # the serving configuration at small size: jobs that arrive together, five Adam steps each
        dict(name="serve_n12_18", kind="serve", lo=12, hi=18, p=4, m=16, steps=5, k=2, mix=4),
        # measurement shots of one state
        dict(name="shots_n20", kind="shots", n=20, shots=65536),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(("single", "grad", "grid", "batch", "cycle", "sampled", "train", "large", "serve", "shots"))
    p = rng.randint(1, 6)
    if kind == "single":
        n = rng.randint(4, 22)
        return dict(kind=kind, n=n, p=p, k=rng.randint(1, 8))
    if kind == "grad":
        return dict(kind=kind, n=rng.randint(6, 22), p=p)
    if kind == "grid":
        return dict(kind=kind, n=rng.randint(6, 12), p=rng.randint(1, 3), points=logint(16, 400), k=rng.randint(1, 8))
    if kind == "batch":
        n = rng.randint(8, 17)
        return dict(kind=kind, n=n, p=p, m=logint(8, min(1000, 1 << (24 - n))), k=rng.randint(1, 2))
    if kind == "cycle":
        n = rng.randint(8, 17)
        N = logint(200, 1500)
        return dict(kind=kind, N=N, m=logint(16, min(512, 1 << (24 - n))), n=n, p=p, k=rng.randint(1, 8), cycles=3)
    if kind == "sampled":
        n = rng.randint(8, 15)
        return dict(kind=kind, N=logint(200, 1000), m=logint(16, 160), n=n, p=rng.randint(1, 3), shots=logint(64, 2048))
    if kind == "train":
        return dict(kind=kind, lo=8, hi=rng.randint(10, 23), p=p, m=rng.randint(8, 48), mix=rng.randrange(1 << 20))
    if kind == "large":
        return dict(kind=kind, n=rng.randint(24, 29), p=rng.randint(1, 3), k=rng.randint(1, 8))
    if kind == "serve":
        return dict(kind=kind, lo=10, hi=rng.randint(12, 18), p=rng.randint(1, 4), m=rng.randint(4, 24), steps=rng.randint(2, 6), k=2,
                    mix=rng.randrange(1 << 20))
    return dict(kind=kind, n=rng.randint(10, 24), shots=logint(256, 131072))


# ---- inputs, from the seed alone ----------------------------------------------------------------

def _rng(seed):
    return np.random.default_rng([int(seed), 2506])


def _sym(g, n, normal=False):
    v = g.standard_normal((n, n)) if normal else g.uniform(-1.0, 1.0, (n, n))
    return np.triu(v) + np.triu(v, 1).T


def _angles(g, p):
    return g.uniform(0.0, math.pi, p), g.uniform(0.0, math.pi / 2, p)


def _mix(case):
    """The (n, p) of an uneven batch's instances: both uniform, the case's own."""
    g = _rng(case["mix"])
    return [(int(g.integers(case["lo"], case["hi"] + 1)), int(g.integers(1, case["p"] + 1))) for _ in range(case["m"])]


def _inputs(case, seed):
    """Host inputs of a case."""
    g, kind = _rng(seed), case["kind"]
    if kind in ("single", "grad", "large", "shots"):
        p = case.get("p", 2)
        Q = _sym(g, case["n"]).astype(np.float32)
        ga, be = _angles(g, p)
        d = dict(Q=Q, params=np.concatenate([ga, be]).astype(np.float32))
        if kind == "shots":
            d["u"] = g.uniform(0.0, 1.0, case["shots"])
        return d
    if kind == "grid":
        # one QUBO, many parameter points (away from the degenerate ends of the grid, where every
        # probability is equal)
        Q = _sym(g, case["n"])
        par = [np.concatenate([g.uniform(0.05, math.pi - 0.05, case["p"]), g.uniform(0.05, math.pi / 2 - 0.05, case["p"])])
               for _ in range(case["points"])]
        return dict(Q=Q, params=np.stack(par))
    if kind == "batch":
        ga, be = _angles(g, case["p"])
        return dict(Q=np.stack([_sym(g, case["n"]) for _ in range(case["m"])]).astype(np.float32),
                    params=np.concatenate([ga, be]).astype(np.float32))
    if kind in ("cycle", "sampled"):
        ga, be = _angles(g, case["p"])
        d = dict(Q=_sym(g, case["N"]), x0=g.integers(0, 2, case["N"], dtype=np.uint8), gamma=ga, beta=be)
        if kind == "sampled":
            d["u"] = g.uniform(0.0, 1.0, (case["m"], case["shots"]))
        return d
    Qs, params = [], []
    for n, p in _mix(case):
        Qs.append(_sym(g, n, normal=kind == "train").astype(np.float32))
        ga, be = _angles(g, p)
        params.append((ga.astype(np.float32), be.astype(np.float32)))
    return dict(Qs=Qs, params=params)


_CTX = None


def _ctx():
    """The program's one library context."""
    global _CTX
    if _CTX is None:
        _CTX = q.qaoa_create(0)
    return _CTX


class _Owned:
    """A library handle that is given back with the state that holds it."""

    def __init__(self, handle, free):
        self.h, self._free = handle, free

    def __del__(self):
        try:
            torch.cuda.synchronize()
            self._free(self.h)
        except Exception:
            pass


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV)


def _plan(ctx, rows, qd, pd, count, k, dbl=False):
    """A forward plan with its output buffers."""
    ex = torch.zeros(count, dtype=torch.float64, device=DEV)
    idx = torch.zeros(count, k, dtype=torch.int64, device=DEV)
    prob = torch.zeros(count, k, dtype=torch.float64, device=DEV)
    io = q.make_io(qd, pd, expect=ex, topk_idx=idx, topk_prob=prob, k_stride=k)
    plan = q.qaoa_plan_create(ctx, q.make_insts(rows), io, dbl)
    return dict(io=io, plan=_Owned(plan, q.qaoa_plan_destroy), expect=ex, idx=idx, prob=prob)


def prepare(case, seed):
    torch.cuda.set_device(0)
    ctx, kind, d = _ctx(), case["kind"], _inputs(case, seed)
    s = dict(case=case, ctx=ctx, kind=kind)
    if kind in ("single", "grad", "shots"):
        n, p = case["n"], len(d["params"]) // 2
        q.qaoa_reserve(ctx, q.qaoa_workspace_bytes(n))
        par = _t(d["params"])
        s |= dict(n=n, p=p, Q=_t(d["Q"]), gamma=par[:p].clone(), beta=par[p:].clone(),
                  E=torch.empty(1 << n, device=DEV), expect=torch.empty(1, dtype=torch.float64, device=DEV))
        if kind == "grad":
            s |= dict(dgamma=torch.empty(p, dtype=torch.float64, device=DEV), dbeta=torch.empty(p, dtype=torch.float64, device=DEV))
            return s
        s["psi"] = torch.empty(1 << n, dtype=torch.complex64, device=DEV)
        if kind == "single":
            s |= dict(idx=torch.empty(case["k"], dtype=torch.int64, device=DEV),
                      prob=torch.empty(case["k"], dtype=torch.float64, device=DEV))
            return s
        q.qaoa_build_energies(ctx, n, s["Q"], s["E"])
        q.qaoa_run_layers(ctx, n, p, s["gamma"], s["beta"], s["E"], s["psi"])
        s |= dict(u=_t(d["u"]), out=torch.empty(case["shots"], dtype=torch.int64, device=DEV))
        return s
    if kind in ("grid", "batch", "large"):
        n, p, k = case["n"], case["p"], case["k"]
        m = case["points"] if kind == "grid" else case["m"] if kind == "batch" else 1
        qd, pd = _t(d["Q"]), _t(d["params"])
        rows = [(n, p, k, 0, 0 if kind == "grid" else i * n * n, 2 * p * i if kind == "grid" else 0, -1, -1) for i in range(m)]
        return s | dict(qd=qd, pd=pd) | _plan(ctx, rows, qd, pd, m, k, dbl=kind == "grid")
    if kind in ("cycle", "sampled"):
        sess = q.dqaoa_session_create(ctx, case["N"], case["m"], case["n"], case["p"], case.get("k", 1), q.DQAOA_RANDOM, True,
                                      d["gamma"], d["beta"])
        s |= dict(sess=_Owned(sess, q.dqaoa_session_destroy), Q=d["Q"], x0=d["x0"], u=d.get("u"), seed=int(seed))
        # the problem goes to the device with its first cycle; the cycles measured find it there
        q.dqaoa_session_cycle(sess, s["Q"], 1, s["x0"].copy(), s["seed"], 1 << 20)
        return s
    if kind == "train":
        batch = train.QAOABatch(ctx, d["Qs"], d["params"], grad=True)
        return s | dict(batch=batch, params=batch.params.clone())
    # serve
    reqs = [serve.Request(n=Q.shape[0], p=len(ga), Q=Q, params=np.concatenate([ga, be]), steps=case["steps"], lr=0.05)
            for Q, (ga, be) in zip(d["Qs"], d["params"])]
    srv = q.qaoa_server_create(ctx, 1 << 30, 64, case["k"])
    return s | dict(reqs=reqs, srv=_Owned(srv, q.qaoa_server_destroy))


def run(s):
    ctx, kind, case = s["ctx"], s["kind"], s["case"]
    if kind == "single":
        n, p, k = s["n"], s["p"], case["k"]
        q.qaoa_build_energies(ctx, n, s["Q"], s["E"])
        q.qaoa_run_layers(ctx, n, p, s["gamma"], s["beta"], s["E"], s["psi"])
        q.qaoa_expect(ctx, n, s["psi"], s["E"], s["expect"])
        q.qaoa_topk(ctx, n, s["psi"], k, s["idx"], s["prob"])
        return dict(energies=s["E"], state=s["psi"], expect=s["expect"].float(), idx=s["idx"], prob=s["prob"].float())
    if kind == "grad":
        n, p = s["n"], s["p"]
        q.qaoa_build_energies(ctx, n, s["Q"], s["E"])
        q.qaoa_grad(ctx, n, p, s["gamma"], s["beta"], s["E"], s["expect"], s["dgamma"], s["dbeta"])
        return dict(expect=s["expect"].float(), dgamma=s["dgamma"].float(), dbeta=s["dbeta"].float())
    if kind == "grid":
        q.qaoa_plan_launch(s["plan"].h)
        return dict(expect=s["expect"], idx=s["idx"], prob=s["prob"])
    if kind in ("batch", "large"):
        q.qaoa_plan_launch(s["plan"].h)
        return dict(expect=s["expect"].float(), idx=s["idx"], prob=s["prob"].float())
    if kind == "cycle":
        x, energies = s["x0"].copy(), []
        for c in range(case["cycles"]):
            e, _ = q.dqaoa_session_cycle(s["sess"].h, s["Q"], 0, x, s["seed"], c)
            energies.append(e)
        return dict(x=x, energies=energies)
    if kind == "sampled":
        x = s["x0"].copy()
        e, _ = q.dqaoa_session_cycle_sampled(s["sess"].h, s["Q"], 0, x, s["seed"], 0, s["u"])
        return dict(x=x, energy=e)
    if kind == "train":
        params = s["params"].detach().requires_grad_()
        ex = train.QAOAExpectation.apply(params, s["batch"])
        ex.sum().backward()
        return dict(expect=ex.detach().float(), grad=params.grad)
    if kind == "serve":
        rep = serve.serve_stream(ctx, s["reqs"], 0, 0, case["k"], server=s["srv"].h)
        res = [rep.results[i] for i in range(len(s["reqs"]))]
        return dict(expect=np.array([r.expect for r in res], dtype=np.float32),
                    params=np.concatenate([np.array(r.params[:2 * r.p], dtype=np.float32) for r in res]),
                    idx=np.array([list(r.topk_idx[:case["k"]]) for r in res], dtype=np.int64),
                    prob=np.array([list(r.topk_prob[:case["k"]]) for r in res], dtype=np.float32))
    q.qaoa_sample(ctx, case["n"], s["psi"], case["shots"], s["u"], s["out"])
    return s["out"]


# ---- what a pass cannot do without ------------------------------------------------------------

def _solve_flops(n, p):
    """Per instance: n rotations (4) and one cost phase with its sine and cosine (20) per amplitude
    and layer."""
    return (1 << n) * p * (4 * n + 20)


def work(case):
    kind = case["kind"]
    n, p, k = case.get("n", 0), case.get("p", 2), case.get("k", 1)
    D = 1 << n
    if kind == "single":      # Q and the angles in; energies, state, <C> and the top-k out
        return dict(bytes=4 * n * n + 8 * p + 4 * D + 8 * D + 8 + 16 * k, flops=_solve_flops(n, p) + 4 * D)
    if kind == "grad":        # forward, then both states undone with the inner products
        return dict(bytes=4 * n * n + 24 * p + 8, flops=3 * _solve_flops(n, p) + D * p * 4 * (n + 1))
    if kind == "grid":
        return dict(bytes=8 * n * n + case["points"] * (16 * p + 8 + 16 * k), flops=case["points"] * _solve_flops(n, p))
    if kind in ("batch", "large"):
        m = case.get("m", 1)
        return dict(bytes=m * (4 * n * n + 8 + 16 * k) + 8 * p, flops=m * _solve_flops(n, p))
    if kind == "cycle":       # the conditioned rows of the sub-QUBOs, per cycle
        c = case["cycles"]
        return dict(bytes=c * (8 * case["m"] * n * min(case["N"], 1 << 20) + case["N"]), flops=c * case["m"] * _solve_flops(n, p))
    if kind == "sampled":
        return dict(bytes=8 * case["m"] * n * case["N"] + 16 * case["m"] * case["shots"],
                    flops=case["m"] * (_solve_flops(n, p) + 4 * D))
    if kind in ("train", "serve"):
        steps, mix = case.get("steps", 1), _mix(case)
        return dict(bytes=sum(4 * v * v + 24 * l * steps for v, l in mix),
                    flops=sum(3 * _solve_flops(v, l) + (1 << v) * l * 4 * (v + 1) for v, l in mix) * steps)
    return dict(bytes=8 * D + 16 * case["shots"], flops=4 * D)


# ---- the same in 64 bits, in plain torch -------------------------------------------------------

def _energies64(Q):
    """z^T Q z for every z, by doubling."""
    Q = torch.as_tensor(np.asarray(Q, dtype=np.float64)).to(DEV)
    n = Q.shape[0]
    E = torch.zeros(1, dtype=torch.float64, device=DEV)
    for i in range(n):
        row = Q[i, i].reshape(1).clone()
        for j in range(i):
            row = torch.cat([row, row + (Q[i, j] + Q[j, i])])
        E = torch.cat([E, E + row])
    return E


def _mix64(psi, beta):
    c, s = math.cos(beta), math.sin(beta)
    for j in range(int(psi.numel()).bit_length() - 1):
        v = psi.view(-1, 2, 1 << j)
        a, b = v[:, 0], v[:, 1]
        a0 = a.clone()
        a.mul_(c).add_(b, alpha=complex(0.0, -s))
        b.mul_(c).add_(a0, alpha=complex(0.0, -s))


def _phase64(psi, E, gamma):
    step = 1 << 26
    for i in range(0, psi.numel(), step):
        th = E[i:i + step] * (-gamma)
        psi[i:i + step] *= torch.complex(torch.cos(th), torch.sin(th))


def _state64(E, gamma, beta):
    n = int(E.numel()).bit_length() - 1
    psi = torch.full((E.numel(),), 2.0 ** (-0.5 * n), dtype=torch.complex128, device=DEV)
    for ga, be in zip(gamma, beta):
        _phase64(psi, E, float(ga))
        _mix64(psi, float(be))
    return psi


def _read64(psi, E, k):
    pr = psi.real.square()
    pr += psi.imag.square()
    return (pr * E).sum(), torch.topk(pr, k).values


def _grad64(E, gamma, beta):
    psi = _state64(E, gamma, beta)
    ex = (psi.abs().square() * E).sum()
    lam = psi * E
    dg, db = np.zeros(len(gamma)), np.zeros(len(beta))
    for l in range(len(gamma) - 1, -1, -1):
        acc = 0.0
        for j in range(int(psi.numel()).bit_length() - 1):
            acc += torch.vdot(lam, psi.view(-1, 2, 1 << j).flip(1).reshape(-1)).imag.item()
        db[l] = 2.0 * acc
        _mix64(psi, -float(beta[l]))
        _mix64(lam, -float(beta[l]))
        dg[l] = 2.0 * torch.vdot(lam, psi * E).imag.item()
        _phase64(psi, E, -float(gamma[l]))
        _phase64(lam, E, -float(gamma[l]))
    return ex.item(), dg, db


def exact(case, seed):
    kind, d = case["kind"], _inputs(case, seed)
    if kind == "single":
        p = case["p"]
        E = _energies64(d["Q"])
        par = d["params"].astype(np.float64)
        psi = _state64(E, par[:p], par[p:])
        ex, pr = _read64(psi, E, case["k"])
        return dict(energies=E, state=psi, expect=ex.reshape(1), idx=None, prob=pr)
    if kind == "grad":
        p = case["p"]
        par = d["params"].astype(np.float64)
        ex, dg, db = _grad64(_energies64(d["Q"]), par[:p], par[p:])
        return dict(expect=np.array([ex]), dgamma=dg, dbeta=db)
    if kind in ("grid", "batch", "large"):
        p, k = case["p"], case["k"]
        m = case["points"] if kind == "grid" else case["m"] if kind == "batch" else 1
        Q = d["Q"].reshape(-1, case["n"], case["n"])
        par = d["params"].astype(np.float64).reshape(-1, 2 * p)
        exs, prs, E = [], [], None
        for i in range(m):
            if i < len(Q):
                E = _energies64(Q[i])
            v = par[i if len(par) > 1 else 0]
            ex, pr = _read64(_state64(E, v[:p], v[p:]), E, k)
            exs.append(ex)
            prs.append(pr)
        return dict(expect=torch.stack(exs), idx=None, prob=torch.stack(prs))
    if kind == "train":
        exs, gs = [], []
        for Q, (ga, be) in zip(d["Qs"], d["params"]):
            ex, dg, db = _grad64(_energies64(Q), ga.astype(np.float64), be.astype(np.float64))
            exs.append(ex)
            gs += [dg, db]
        return dict(expect=np.array(exs), grad=np.concatenate(gs))
    if kind == "serve":
        exs, prs, out = [], [], []
        for Q, (ga, be) in zip(d["Qs"], d["params"]):
            E, p = _energies64(Q), len(ga)
            v = np.concatenate([ga, be]).astype(np.float64)
            m1, m2 = np.zeros(2 * p), np.zeros(2 * p)
            for t in range(1, case["steps"] + 1):
                _, dg, db = _grad64(E, v[:p], v[p:])
                gr = np.concatenate([dg, db])
                m1, m2 = 0.9 * m1 + 0.1 * gr, 0.999 * m2 + 0.001 * gr * gr
                v = v - 0.05 * (m1 / (1 - 0.9 ** t)) / (np.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8)
            ex, pr = _read64(_state64(E, v[:p], v[p:]), E, case["k"])
            exs.append(ex)
            prs.append(pr)
            out.append(v)
        return dict(expect=torch.stack(exs), params=np.concatenate(out), idx=None, prob=torch.stack(prs))
    # cycles and shots return whole numbers (and the energies of them)
    return None
