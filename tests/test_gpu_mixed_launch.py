"""Plans whose streaming instances of several sizes, depths and kinds share their launches: every
instance's results equal, bit for bit, those of a plan that holds it alone (the kernels work tile by
tile and instance by instance), with and without gradients, with top-k of several lengths, at one
and at many tiles per instance, and with energies at an address the TMA passes cannot take (that
group runs by itself)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (n, p, k, grad)
SPECS = [(14, 1, 0, 1), (14, 4, 3, 1), (15, 2, 0, 1), (18, 1, 5, 0), (18, 1, 5, 0), (18, 3, 2, 0), (19, 2, 16, 0),
         (20, 2, 0, 1), (21, 2, 1, 1), (22, 1, 8, 0), (23, 1, 0, 1), (23, 2, 4, 0)]


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_10531_gb300 import build
    build.build()
    import paper_2506_10531_gb300 as qq
    return qq


def launch(q, ctx, specs, ids, e_shift=None):
    qp, pp, rows = [], [], []
    qo = po = eo = 0
    for (n, p, k, g), i in zip(specs, ids):
        qp.append(synth.symmetric_q(n, seed=700 + i).astype(np.float32).reshape(-1))
        ga, be = synth.random_params(p, seed=800 + i)
        pp.append(np.concatenate([ga, be]).astype(np.float32))
        e = -1
        if e_shift is not None and e_shift == i:
            e, eo = 2, (1 << n) + 2            # 8-byte aligned only
        rows.append((n, p, k, g, qo, po, -1, e))
        qo += n * n
        po += 2 * p
    m = len(specs)
    qd, pd = torch.as_tensor(np.concatenate(qp)).cuda(), torch.as_tensor(np.concatenate(pp)).cuda()
    ex = torch.zeros(m, dtype=torch.float64, device="cuda")
    ti = torch.zeros(m, 16, dtype=torch.int64, device="cuda")
    tp = torch.zeros(m, 16, dtype=torch.float64, device="cuda")
    gr = torch.zeros(po, dtype=torch.float64, device="cuda")
    eb = torch.zeros(max(eo, 1), device="cuda")
    io = q.make_io(qd, pd, expect=ex, topk_idx=ti, topk_prob=tp, k_stride=16, grad=gr, e=eb)
    plan = q.qaoa_plan_create(ctx, q.make_insts(rows), io)
    for _ in range(2):
        q.qaoa_plan_launch(plan)
    torch.cuda.synchronize()
    q.qaoa_plan_check(plan)
    q.qaoa_plan_destroy(plan)
    out, at = [], 0
    for j, (n, p, k, g) in enumerate(specs):
        out.append((ex[j].item(), ti[j, :k].tolist(), tp[j, :k].tolist(), gr[at:at + 2 * p].tolist() if g else None))
        at += 2 * p
    return out


@pytest.mark.parametrize("e_shift", [None, 5])
def test_mixed_equals_alone(q, e_shift):
    ctx = q.qaoa_create(0)
    try:
        both = launch(q, ctx, SPECS, range(len(SPECS)), e_shift)
        for i, s in enumerate(SPECS):
            alone = launch(q, ctx, [s], [i], e_shift)[0]
            assert both[i] == alone, (i, s)
    finally:
        q.qaoa_destroy(ctx)
