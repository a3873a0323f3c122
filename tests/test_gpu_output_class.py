"""An instance of a batched plan gives the same bits whatever its neighbours return: pairs of streaming
instances of equal (n, p, k), of which only the first returns its energies, at a 16-byte or only 8-byte
aligned address (or at none: the reference). Forward runs and gradients."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def launch(q, ctx, n, p, k, grad, e_off, ids):
    """Instances `ids`; instance 0 returns its energies at element e_off (None: nobody does)."""
    Q = np.concatenate([synth.symmetric_q(n, seed=40 + i).reshape(-1) for i in ids]).astype(np.float32)
    par = np.concatenate([np.concatenate(synth.random_params(p, seed=50 + i)) for i in ids]).astype(np.float32)
    m = len(ids)
    e = torch.zeros((1 << n) + 4, device="cuda")
    rows = [(n, p, k, int(grad), j * n * n, 2 * p * j, -1, e_off if i == 0 and e_off is not None else -1)
            for j, i in enumerate(ids)]
    ex = torch.zeros(m, dtype=torch.float64, device="cuda")
    ti = torch.zeros(m, k, dtype=torch.int64, device="cuda")
    tp = torch.zeros(m, k, dtype=torch.float64, device="cuda")
    gr = torch.zeros(m, 2 * p, dtype=torch.float64, device="cuda")
    io = q.make_io(torch.as_tensor(Q).cuda(), torch.as_tensor(par).cuda(), expect=ex, topk_idx=ti, topk_prob=tp,
                   k_stride=k, grad=gr, e=e)
    q.qaoa_batch_run(ctx, q.make_insts(rows), io)
    return [(ex[j].item(), ti[j].tolist(), tp[j].tolist(), gr[j].tolist()) for j in range(m)]


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("n,p,k", [(18, 3, 4), (20, 1, 1)])
@pytest.mark.parametrize("e_off", [0, 2])
def test_a_neighbours_energies_change_nothing(n, p, k, grad, e_off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_10531_gb300 as q
    ctx = q.qaoa_create(0)
    try:
        pair = launch(q, ctx, n, p, k, grad, e_off, [0, 1])
        assert pair[1] == launch(q, ctx, n, p, k, grad, None, [1])[0]      # the neighbour, as alone
        assert pair[0] == launch(q, ctx, n, p, k, grad, e_off, [0])[0]
        none = launch(q, ctx, n, p, k, grad, None, [0, 1])
        assert none[1] == pair[1]
    finally:
        q.qaoa_destroy(ctx)


@pytest.mark.parametrize("n", [15, 16, 17])
def test_cluster_streaming_energies_at_any_address(n):
    """15..17 qubits: the address energies are returned to decides nothing (they leave by 4-byte stores)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_10531_gb300 as q
    ctx = q.qaoa_create(0)
    try:
        assert launch(q, ctx, n, 2, 4, False, 2, [0]) == launch(q, ctx, n, 2, 4, False, 0, [0]) == launch(q, ctx, n, 2, 4, False, None, [0])
    finally:
        q.qaoa_destroy(ctx)
