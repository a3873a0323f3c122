"""Single complex64 states of 15..22 qubits through qaoa_run_layers and qaoa_grad (14..22): the tile
size changes with n up to 21 (tile bits 9..12, contiguous runs of 8 or 16 amplitudes) and with
22; and the energy build on both sides of its tile / row boundary, for every small n, for a
non-symmetric Q and an output at a 4-byte aligned address.

Tolerances: amplitudes within 1e-5 and gradients within 1e-5 max(max|d|, 1) max(1, n / 4) of the FP64
oracle (the library's stated bounds); energies: at most n(n+1)/2 FP32 roundings of partial sums
below sum |Q|: n(n+1)/2 2^-24 sum |Q|."""
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


@pytest.fixture(scope="module")
def ctx(q):
    c = q.qaoa_create(0)
    q.qaoa_reserve(c, q.qaoa_workspace_bytes(22))
    yield c
    q.qaoa_destroy(c)


@pytest.mark.parametrize("n,p", [(14, 2), (15, 1), (15, 4), (16, 3), (17, 2), (18, 3), (19, 2), (20, 2), (21, 1), (22, 1)])
def test_state_and_gradient(q, ctx, orc, n, p):
    Q32 = synth.symmetric_q(n, seed=30 + n).astype(np.float32)
    g, b = (v.astype(np.float32) for v in synth.random_params(p, seed=60 + n))
    E64 = orc.energies(Q32.astype(np.float64))
    E = torch.as_tensor(E64.astype(np.float32)).cuda()
    gd, bd = torch.as_tensor(g).cuda(), torch.as_tensor(b).cuda()
    Eo = E.cpu().numpy().astype(np.float64)
    psi = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    q.qaoa_run_layers(ctx, n, p, gd, bd, E, psi)
    ref = orc.state(n, g.astype(np.float64), b.astype(np.float64), Eo)
    assert np.max(np.abs(psi.cpu().numpy().astype(np.complex128) - ref)) <= 1e-5
    ex, dg, db = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (1, p, p))
    q.qaoa_grad(ctx, n, p, gd, bd, E, ex, dg, db)
    eo, dgo, dbo = orc.grad(n, g.astype(np.float64), b.astype(np.float64), Eo)
    scale = max(np.abs(dgo).max(), np.abs(dbo).max(), 1.0) * max(1.0, n / 4)
    assert np.max(np.abs(dg.cpu().numpy() - dgo)) <= 1e-5 * scale
    assert np.max(np.abs(db.cpu().numpy() - dbo)) <= 1e-5 * scale
    assert abs(ex.item() - eo) <= 1e-5 * np.abs(Q32).sum()


@pytest.mark.parametrize("n", [1, 2, 5, 7, 8, 9, 10, 11, 12, 17, 22, 23])
@pytest.mark.parametrize("dbl", [False, True])
@pytest.mark.parametrize("off", [0, 1])
def test_energy_tiles(q, ctx, orc, n, dbl, off):
    Q = synth.uniform_pm1(80 + n, n * n).reshape(n, n)          # not symmetric
    dt = torch.float64 if dbl else torch.float32
    Qd = torch.as_tensor(Q).to(dt).cuda()
    buf = torch.full(((1 << n) + 2,), float("nan"), dtype=dt, device="cuda")
    E = buf[off:off + (1 << n)]
    q.qaoa_build_energies(ctx, n, Qd, E, dbl=dbl)
    Q64 = Qd.cpu().numpy().astype(np.float64)
    Eo = orc.energies(Q64)
    tol = n * (n + 1) / 2 * (2.0 ** -53 if dbl else 2.0 ** -24) * np.abs(Q64).sum()
    assert np.max(np.abs(E.cpu().numpy().astype(np.float64) - Eo)) <= (2 * tol if dbl else tol)   # FP64: the oracle rounds too
    assert torch.isnan(buf[(1 << n) + off:]).all() and torch.isnan(buf[:off]).all()
