"""Forward batches whose launches give each block tiles in a row: instances of one and of several sizes,
more and fewer tiles than blocks, shares that end inside an instance (an odd number of instances), top-k
lists that several blocks of an instance contribute to. Every instance's results equal, bit for bit,
those of a plan that holds it alone, whose launches stride."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def launch(q, ctx, specs, ids):
    Q = np.concatenate([synth.symmetric_q(s[0], seed=300 + i).reshape(-1) for s, i in zip(specs, ids)]).astype(np.float32)
    par = np.concatenate([np.concatenate(synth.random_params(s[1], seed=400 + i)) for s, i in zip(specs, ids)]).astype(np.float32)
    rows, qo, po = [], 0, 0
    for n, p, k in specs:
        rows.append((n, p, k, 0, qo, po, -1, -1))
        qo, po = qo + n * n, po + 2 * p
    m = len(specs)
    ex = torch.zeros(m, dtype=torch.float64, device="cuda")
    ti = torch.zeros(m, 16, dtype=torch.int64, device="cuda")
    tp = torch.zeros(m, 16, dtype=torch.float64, device="cuda")
    io = q.make_io(torch.as_tensor(Q).cuda(), torch.as_tensor(par).cuda(), expect=ex, topk_idx=ti, topk_prob=tp, k_stride=16)
    plan = q.qaoa_plan_create(ctx, q.make_insts(rows), io)
    q.qaoa_plan_launch(plan)
    q.qaoa_plan_check(plan)
    q.qaoa_plan_destroy(plan)
    return [(ex[j].item(), ti[j, :s[2]].tolist(), tp[j, :s[2]].tolist()) for j, s in enumerate(specs)]


@pytest.mark.parametrize("specs", [[(18, 2, 3)] * 2, [(18, 3, 16)] * 23, [(19, 1, 1)] * 7, [(21, 2, 8)] * 3, [(24, 1, 4)] * 2,
                                    [(18, 1, 2), (20, 3, 5), (20, 3, 5), (23, 2, 1), (25, 1, 3), (18, 4, 0)]],
                         ids=["2x18", "23x18", "7x19", "3x21", "2x24", "mixed"])
def test_tiles_in_a_row(specs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_10531_gb300 as q
    ctx = q.qaoa_create(0)
    try:
        both = launch(q, ctx, specs, range(len(specs)))
        for i, s in enumerate(specs):
            assert both[i] == launch(q, ctx, [s], [i])[0], i
    finally:
        q.qaoa_destroy(ctx)
