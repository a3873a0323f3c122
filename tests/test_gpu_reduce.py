"""The standalone reductions (qaoa_expect, qaoa_topk) at the edges of their block layout: one block
(n <= 12), several blocks, several rounds per block; flat, sparse and random states; states at an
8-byte aligned address.

<C> tolerance: products in FP32 (three roundings each, sums of eight), FP64 above: 16 2^-24
sum |psi|^2 |E|. Top-k: the library's probabilities are exact FP64 values of the FP32 amplitudes, so
indices and values equal the oracle's."""
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


def make(kind, D, seed):
    g = torch.Generator().manual_seed(seed)
    v = torch.zeros(2 * D)
    if kind == "random":
        v = torch.randn(2 * D, generator=g)
    elif kind == "flat":
        v[0::2] = 1.0
    elif kind == "levels":                  # many exact ties at a few levels
        v[0::2] = torch.randint(1, 4, (D,), generator=g).float()
    else:                                   # sparse: fewer nonzeros than k, then one more block's worth
        at = torch.unique((torch.rand(5, generator=g) * D).long())
        v[2 * at] = 1.0
    return v / v.norm()


@pytest.mark.parametrize("n,k", [(1, 2), (3, 8), (8, 16), (11, 5), (12, 16), (13, 1), (14, 16), (17, 7), (21, 16), (23, 3)])
@pytest.mark.parametrize("kind", ["random", "flat", "levels", "sparse"])
def test_reductions(q, orc, n, k, kind):
    D = 1 << n
    v = make(kind, D, 100 * n + k)
    E = torch.as_tensor(synth.uniform_pm1(n, D).astype(np.float32))
    buf = torch.zeros(2 * D + 2, device="cuda")
    buf[2:] = v.cuda()
    psi = buf[2:]                           # 8-byte aligned
    ex = torch.zeros(1, dtype=torch.float64, device="cuda")
    ti = torch.full((k,), -1, dtype=torch.int64, device="cuda")
    tp = torch.zeros(k, dtype=torch.float64, device="cuda")
    c = q.qaoa_create(0)
    try:
        q.qaoa_reserve(c, 1 << 20)
        q.qaoa_expect(c, n, psi, E.cuda(), ex)
        q.qaoa_topk(c, n, psi, k, ti, tp)
        torch.cuda.synchronize()
    finally:
        q.qaoa_destroy(c)
    a = v.numpy().view(np.complex64).astype(np.complex128)
    pr = orc.probs(a)
    oi, op = orc.topk_probs(pr, k)
    np.testing.assert_array_equal(ti.cpu().numpy().astype(np.uint64), oi)
    np.testing.assert_array_equal(tp.cpu().numpy(), op)
    e64 = E.numpy().astype(np.float64)
    assert abs(ex.item() - float(pr @ e64)) <= 16 * 2.0 ** -24 * float(pr @ np.abs(e64)) + 1e-15
