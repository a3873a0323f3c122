"""The norm of complex128 states of the batched plans, resident (n = 10, 12) and streamed (n = 14), for
mixer angles on both sides of pi / 4.

What a layer leaves on every amplitude alike is the factor of its shears, applied once: the rounded
factor puts 2^-53 on the amplitudes, 2 2^-53 on the squared norm. |+> starts with one rounding of
2^(-n/2) (none for even n). Everything else rounds amplitude by amplitude: n + 4 roundings of random
sign a layer, averaged over the 2^n amplitudes, put about 2^-53 sqrt(p (n + 4) / 2^n) on the squared
norm, 0.2 2^-53 at n = 10, p = 3; 3 2^-53 are allowed. Bound: (2 p + 3) 2^-53. A factor formed as the
n-th power of a rounded number is off by up to n roundings and more and fails it."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(10, 64), (12, 64), (14, 8)])
@pytest.mark.parametrize("p", [1, 3])
def test_norm_of_states(n, m, p):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_10531_gb300 as q
    ctx = q.qaoa_create(0)
    try:
        Q = synth.symmetric_q(n, seed=900 + n).reshape(-1)
        ga = np.pi * synth.uniform_pm1(901, m * p).reshape(m, p)
        be = np.pi / 2 * synth.uniform_pm1(902, m * p).reshape(m, p)
        par = torch.as_tensor(np.concatenate([ga, be], axis=1)).cuda()
        psi = torch.empty(m << n, dtype=torch.complex128, device="cuda")
        ex = torch.empty(m, dtype=torch.float64, device="cuda")
        rows = [(n, p, 0, 0, 0, 2 * p * i, i << n, -1) for i in range(m)]
        io = q.make_io(torch.as_tensor(Q).cuda(), par, expect=ex, psi=psi)
        q.qaoa_batch_run_z(ctx, q.make_insts(rows), io)
        a = psi.cpu().numpy().reshape(m, -1)
        sq = (a.real.astype(np.longdouble) ** 2 + a.imag.astype(np.longdouble) ** 2).sum(axis=1)
        off = np.abs((sq - 1).astype(np.float64))
        assert off.max() <= (2 * p + 3) * 2.0 ** -53, off.max() * 2.0 ** 53
    finally:
        q.qaoa_destroy(ctx)
