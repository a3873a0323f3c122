"""Cluster-streaming plans of few instances run in clusters of eight thread blocks, larger ones in
clusters of four: an instance's <C>, top-k list and state are the same bits either way (its tiles,
their arithmetic and the order of the <C> sum do not depend on the cluster)."""
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


def run(q, n, p, k, count, Qs, par):
    D = 1 << n
    qd, pd = torch.as_tensor(Qs[:count].reshape(-1)).cuda(), torch.as_tensor(par[:count].reshape(-1)).cuda()
    ex = torch.zeros(count, dtype=torch.float64, device="cuda")
    ti = torch.zeros(count, k, dtype=torch.int64, device="cuda")
    tp = torch.zeros(count, k, dtype=torch.float64, device="cuda")
    psi = torch.zeros(3 * D, dtype=torch.complex64, device="cuda")
    rows = [(n, p, k, 0, i * n * n, i * 2 * p, i * D if i < 3 else -1, -1) for i in range(count)]
    ctx = q.qaoa_create(0)
    try:
        plan = q.qaoa_plan_create(ctx, q.make_insts(rows), q.make_io(qd, pd, expect=ex, topk_idx=ti, topk_prob=tp,
                                                                     k_stride=k, psi=psi))
        for _ in range(2):
            q.qaoa_plan_launch(plan)
        torch.cuda.synchronize()
        q.qaoa_plan_check(plan)
        q.qaoa_plan_destroy(plan)
    finally:
        q.qaoa_destroy(ctx)
    m = min(count, 3)
    return ex[:m].tolist(), ti[:m].tolist(), tp[:m].tolist(), psi[:m * D].cpu().numpy().tobytes()


# counts of one wave of the wide clusters (at most 38 on 152 SMs) and of more than one of either
@pytest.mark.parametrize("n,p,k", [(15, 2, 3), (16, 1, 16), (16, 4, 1), (17, 2, 5), (17, 3, 8)])
def test_same_bits(q, n, p, k):
    total = 170
    Qs = np.stack([synth.symmetric_q(n, seed=300 + i) for i in range(total)]).astype(np.float32)
    par = np.stack([np.concatenate(synth.random_params(p, seed=500 + i)) for i in range(total)]).astype(np.float32)
    ref = run(q, n, p, k, total, Qs, par)
    for count in (3, 20, 36, 37, 60):
        assert run(q, n, p, k, count, Qs, par) == ref, count
    one = run(q, n, p, k, 1, Qs, par)
    assert one[:3] == tuple(r[:1] for r in ref[:3]) and one[3] == ref[3][:len(one[3])]
