"""Top-k of states whose probabilities tie in their thousands: flat, one amplitude, two levels with the
larger one at scattered indices, and equal but for one rounding. The list (probability descending,
index ascending) is compared entry by entry with the ranking of the exact FP64 probabilities."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def states(n):
    D = 1 << n
    z = np.arange(D, dtype=np.uint64)
    hash_ = (z * np.uint64(0x9E3779B97F4A7C15)) >> np.uint64(40)
    a = np.float32(2.0 ** (-n / 2))
    flat = np.full(D, a, dtype=np.float32)
    one = np.zeros(D, dtype=np.float32)
    one[D // 2 + 1] = 1.0
    two = np.where(hash_ % np.uint64(3) == 0, a, a / np.float32(2)).astype(np.float32)
    near = np.where(hash_ % np.uint64(5) == 0, np.nextafter(a, np.float32(1)), a).astype(np.float32)
    return {"flat": flat, "one": one, "two": two, "near": near}


@pytest.mark.parametrize("dbl", [False, True])
@pytest.mark.parametrize("n", [2, 8, 11, 12, 13, 16, 21, 22])
@pytest.mark.parametrize("k", [1, 8, 16])
def test_ties(n, k, dbl):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_10531_gb300 as q
    k = min(k, 1 << n)
    ctx = q.qaoa_create(0)
    try:
        for name, re in states(n).items():
            psi = torch.as_tensor(re).cuda().to(torch.complex128 if dbl else torch.complex64)
            ti = torch.empty(k, dtype=torch.int64, device="cuda")
            tp = torch.empty(k, dtype=torch.float64, device="cuda")
            q.qaoa_topk(ctx, n, psi, k, ti, tp, dbl=dbl)
            p = re.astype(np.float64) ** 2
            best = np.lexsort((np.arange(p.size), -p))[:k]
            assert ti.tolist() == best.tolist(), name
            assert tp.tolist() == p[best].tolist(), name
    finally:
        q.qaoa_destroy(ctx)
