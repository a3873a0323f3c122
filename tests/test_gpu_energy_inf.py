"""Energies of a QUBO with infinite entries: E(z) is infinite (or, with both signs, NaN) exactly where z
holds the qubits of such an entry, and elsewhere the same number as without it -- for the energies
that plans return (built per tile of 2^11) and those of one-qubit and unaligned single calls."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_10531_gb300 as qq
    return qq


def energies(q, Q, how, dbl):
    n = Q.shape[0]
    dt = torch.float64 if dbl else torch.float32
    Qd = torch.as_tensor(Q).to(dt).cuda()
    ctx = q.qaoa_create(0)
    try:
        if how == "single":
            buf = torch.zeros((1 << n) + 1, dtype=dt, device="cuda")
            E = buf[1:]                                   # float: 4-byte aligned only
            q.qaoa_build_energies(ctx, n, Qd, E, dbl=dbl)
        else:
            E = torch.zeros(1 << n, dtype=dt, device="cuda")
            io = q.make_io(Qd, torch.full((2,), 0.3, dtype=dt, device="cuda"), e=E,
                           expect=torch.zeros(1, dtype=torch.float64, device="cuda"))
            q.qaoa_batch_run(ctx, q.make_insts([(n, 1, 0, 0, 0, 0, -1, 0)]), io, dbl=dbl)
        return E.cpu().numpy()
    finally:
        q.qaoa_destroy(ctx)


@pytest.mark.parametrize("n,how,dbl", [(1, "single", False), (1, "single", True), (12, "single", False),
                                        (18, "plan", False), (14, "plan", True)])
@pytest.mark.parametrize("where", ["low", "mixed", "high", "both_signs"])
def test_infinite_entries(q, n, how, dbl, where):
    Q = synth.symmetric_q(n, seed=70 + n)
    a, b = {"low": (0, min(3, n - 1)), "mixed": (min(2, n - 1), n - 1), "high": (n - 1, max(n - 2, 0)),
            "both_signs": (0, n - 1)}[where]
    Q[a, b] = 0.0
    base = energies(q, Q, how, dbl)
    z = np.arange(1 << n)
    hit = ((z >> a) & (z >> b) & 1).astype(bool)
    Q[a, b] = np.inf
    got = energies(q, Q, how, dbl)
    np.testing.assert_array_equal(got[~hit], base[~hit])
    assert np.all(got[hit] == np.inf)
    if where == "both_signs" and n > 2:
        Q[1, 1] = -np.inf
        got = energies(q, Q, how, dbl)
        one = ((z >> 1) & 1).astype(bool)
        np.testing.assert_array_equal(got[~hit & ~one], base[~hit & ~one])
        assert np.all(got[hit & ~one] == np.inf) and np.all(got[~hit & one] == -np.inf) and np.all(np.isnan(got[hit & one]))
