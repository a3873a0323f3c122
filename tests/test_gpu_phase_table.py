"""Forward streaming passes that take phases and energies from Q itself: their states, <C> and top
probability against the complex128 plan and against the same passes reading an energy vector (a plan
that returns its energies), with one and two chunks of high qubits of every kind of window, two
instances with their own Q in a launch, large and wrapped phases, and terms that are not finite."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_10531_gb300 import build
    build.build()
    import paper_2506_10531_gb300 as qq
    return qq


def run(q, n, p, Qs, par, energies, dbl=False):
    m, D = len(Qs), 1 << n
    real, cplx = (torch.float64, torch.complex128) if dbl else (torch.float32, torch.complex64)
    qd = torch.as_tensor(np.concatenate([x.reshape(-1) for x in Qs]).astype(np.float32)).to("cuda", real)
    pd = torch.as_tensor(np.concatenate(par).astype(np.float32)).to("cuda", real)
    ex = torch.zeros(m, dtype=torch.float64, device="cuda")
    psi = torch.zeros(m * D, dtype=cplx, device="cuda")
    tp = torch.zeros(m, 1, dtype=torch.float64, device="cuda")
    ti = torch.zeros(m, 1, dtype=torch.int64, device="cuda")
    eb = torch.zeros(m * D if energies else 1, dtype=real, device="cuda")
    rows = [(n, p, 1, 0, i * n * n, i * 2 * p, i * D, i * D if energies else -1) for i in range(m)]
    io = q.make_io(qd, pd, expect=ex, topk_idx=ti, topk_prob=tp, k_stride=1, psi=psi, e=eb)
    ctx = q.qaoa_create(0)
    try:
        plan = q.qaoa_plan_create(ctx, q.make_insts(rows), io, dbl)
        q.qaoa_plan_launch(plan)
        torch.cuda.synchronize()
        q.qaoa_plan_check(plan)
        q.qaoa_plan_destroy(plan)
    finally:
        q.qaoa_destroy(ctx)
    return ex.cpu().numpy(), psi.cpu().numpy().reshape(m, D), tp.cpu().numpy()[:, 0], eb.cpu().numpy()


# (n, p, scale of Q): scale 1e3 takes phases through hundreds of turns, 1e7 through the reduction of
# terms beyond 5e5 turns. n = 14..22 have one chunk of 1..9 high qubits, 23 two; 15..17 run in clusters.
@pytest.mark.parametrize("n,p,scale", [(15, 1, 1.0), (16, 3, 1e3), (17, 2, 1.0), (18, 1, 1.0), (18, 3, 1.0), (19, 2, 1e3), (20, 1, 1e7), (21, 2, 1.0), (22, 2, 1.0),
                                       (23, 1, 1.0), (24, 2, 1.0)])
def test_table(q, n, p, scale):
    Qs = [scale * synth.symmetric_q(n, seed=60 + n + i) for i in range(2)]
    if n == 19:
        Qs[1] = np.triu(Qs[1]) * 2.0 - np.diag(np.diag(Qs[1]))   # W_ij from one triangle alone
    par = [np.concatenate(synth.random_params(p, seed=90 + i)) for i in range(2)]
    ea, pa, ta, _ = run(q, n, p, Qs, par, False)
    eb, pb, tb, E = run(q, n, p, Qs, par, True)
    ec, pc, tc, Ec = run(q, n, p, Qs, par, True, True)
    for i in range(2):
        Emax = np.abs(E[i << n:(i + 1) << n]).max()
        W = np.abs(Qs[i].astype(np.float32)).sum()
        ref = pc[i]
        assert np.abs(E[i << n:(i + 1) << n] - Ec[i << n:(i + 1) << n]).max() <= 32 * W * 2.0 ** -24
        # __sincosf 2^-21 and the angle's rounding 2^-23 a layer, n p mixer steps of 2^-22; the
        # FP32 sums of <C> 32 roundings
        tol = p * 2.0 ** -20 + n * p * 2.0 ** -22
        err = np.linalg.norm(pa[i].astype(np.complex128) - ref) / np.linalg.norm(ref)
        print(n, p, scale, i, err, tol)
        assert err <= tol
        assert abs(ea[i] - ec[i]) <= 2 * tol * Emax + 32 * W * 2.0 ** -24
        assert abs(ta[i] - tc[i]) <= 2 * tol
        if scale == 1.0:
            # read energies: gamma E off by half an ulp of FP32 E, the split factor, the reduction
            tole = tol + np.abs(par[i][:p]).sum() * Emax * 3 * 2.0 ** -24
            assert np.linalg.norm(pb[i].astype(np.complex128) - ref) <= tole * np.linalg.norm(ref)
            assert abs(eb[i] - ec[i]) <= 2 * tole * Emax + 32 * W * 2.0 ** -24


def test_not_finite(q):
    n, p = 18, 2
    par = [np.concatenate(synth.random_params(p, seed=5 + i)) for i in range(2)]
    for bad in (np.inf, np.nan):
        Qs = [synth.symmetric_q(n, seed=7 + i) for i in range(2)]
        Qs[1][3, 3] = bad
        ea, pa, _, _ = run(q, n, p, Qs, par, False)
        eb, pb, _, _ = run(q, n, p, Qs, par, True)
        assert np.isfinite(ea[0]) and np.isfinite(pa[0]).all()
        assert np.isnan(ea[1]) and np.isnan(eb[1])
        assert np.isnan(pa[1]).all() and np.isnan(pb[1]).all()
