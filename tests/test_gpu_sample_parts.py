"""Shots (qaoa_sample) at the sizes where the part layout changes: fewer amplitudes than a row, one
coarse part, several, fine parts of 16 to 128 amplitudes, half-warp walks; states with long runs
of zero probability, a state at an 8-byte aligned address, odd shot counts; and the best shot of a
sub-QUBO whose entries lie below the FP32 filter's range.

Tolerance: the device adds 2^n FP64 probabilities by parts, the oracle in one running sum; both are
within 2^n 2^-53 of the exact sums (at most 2^-29 at n = 24, and in practice the rounding errors
average out), so a shot may take the neighbour of its index only where its target lies within
2^n 2^-53 of a CDF boundary."""
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
    yield c
    q.qaoa_destroy(c)


def sample(q, ctx, n, psi, u):
    z = torch.full((len(u),), -1, dtype=torch.int64, device="cuda")
    q.qaoa_sample(ctx, n, psi, len(u), torch.as_tensor(u).cuda(), z)
    torch.cuda.synchronize()
    return z.cpu().numpy().astype(np.uint64)


def check(orc, psi, u, zg):
    a = psi.astype(np.complex128)
    pr = orc.probs(a)
    zo = orc.sample_probs(pr, u)
    cdf = np.cumsum(pr)
    tol = len(pr) * 2.0 ** -53 * cdf[-1]
    assert np.all(pr[zg.astype(np.int64)] > 0)
    for i in np.nonzero(zg != zo)[0]:
        z, t = int(zg[i]), u[i] * cdf[-1]
        lo = cdf[z - 1] if z > 0 else 0.0
        assert lo - tol <= t <= cdf[z] + tol, (i, z, int(zo[i]))


@pytest.mark.parametrize("n,shots", [(2, 7), (3, 100), (4, 33), (5, 257), (9, 1000), (17, 1000), (21, 3001),
                                     (22, 513), (23, 3001), (24, 1025)])
def test_part_layouts(q, ctx, orc, n, shots):
    g = torch.Generator().manual_seed(n)
    psi = torch.randn(2 << n, generator=g).cuda()
    psi /= psi.norm()
    u = synth.uniform01(500 + n, shots)
    u[0], u[-1] = 0.0, 1.0 - 2.0 ** -53
    zg = sample(q, ctx, n, psi, u)
    check(orc, psi.cpu().numpy().view(np.complex64), u, zg)


@pytest.mark.parametrize("n", [6, 12, 19, 24])
def test_sparse_state_at_an_odd_address(q, ctx, orc, n):
    D = 1 << n
    at = np.unique((synth.uniform01(600 + n, 9) * D).astype(np.int64))
    at = at[at < D - D // 8]                  # an empty tail, empty parts in between
    v = np.zeros(D, dtype=np.complex64)
    v[at] = 1.0 + 0.5j
    v /= np.linalg.norm(v)
    buf = torch.zeros(2 * D + 2, device="cuda")
    buf[2:] = torch.as_tensor(v.view(np.float32)).cuda()
    u = synth.uniform01(601 + n, 515)
    u[0], u[1] = 0.0, 1.0 - 2.0 ** -53
    zg = sample(q, ctx, n, buf[2:], u)
    assert buf[2:].data_ptr() % 16 == 8
    check(orc, v, u, zg)
    assert set(zg.tolist()) <= set(at.tolist())


@pytest.mark.parametrize("scale", [1.0, 1e-36])
def test_best_shot_filter(q, orc, scale):
    # the chosen shot is the FP64 minimum, with the FP32 filter (scale 1) and without it
    N, m, k, shots = 60, 5, 9, 700
    Q = synth.symmetric_q(N, seed=71) * scale
    x = synth.bits(72, N)
    u = synth.uniform01(73, m * shots).reshape(m, shots)
    c = q.qaoa_create(0)
    try:
        s = q.dqaoa_session_create(c, N, m, k, 1, 1, q.DQAOA_RANDOM, True, [0.4], [0.5])
        q.dqaoa_session_cycle_sampled(s, Q, 1, x.copy(), 5, 0, u)
        z, best, _ = q.dqaoa_session_shots(s, m, k, shots)
        q.dqaoa_session_destroy(s)
    finally:
        q.qaoa_destroy(c)
    _, qs = orc.decompose(Q, x, m, k, 5, 0, conditioned=True)
    for j in range(m):
        ys = np.unique(z[j])
        es = np.array([float(b @ qs[j] @ b) for b in (((int(y) >> np.arange(k)) & 1).astype(np.float64) for y in ys)])
        assert float(es[ys == best[j]][0]) <= es.min() + 1e-13 * np.abs(qs[j]).sum(), j
