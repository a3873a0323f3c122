"""Shots whose uniform is 0 or -0 take the first amplitude that has any probability, however many lie before
it (in the same fine part, in an earlier one, in an earlier coarse part)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,first", [(1, 1), (3, 2), (6, 40), (8, 200), (9, 300), (12, 5), (12, 100), (12, 4095), (17, 70001), (21, 1500000), (25, 30000001)])
def test_zero_uniforms(n, first):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_10531_gb300 as q
    ctx = q.qaoa_create(0)
    try:
        psi = torch.full((1 << n,), 2.0 ** (-n / 2), dtype=torch.complex64, device="cuda")
        psi[:first] = 0
        u = torch.tensor([0.0, -0.0, 1e-300], dtype=torch.float64, device="cuda")
        out = torch.empty(3, dtype=torch.int64, device="cuda")
        q.qaoa_sample(ctx, n, psi, 3, u, out)
        assert out.tolist() == [first] * 3
    finally:
        q.qaoa_destroy(ctx)
