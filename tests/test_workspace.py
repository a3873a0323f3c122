"""The workspace of single-instance gradients, region by region: psi and lam, one <C> partial per tile of
the forward passes, four gradient partials per tile of the adjoint passes, at the tile sizes that
complex64 states of 14..21 qubits have for themselves (2^((n + 4) / 2) amplitudes, runs of 8), at the
batched ones above (2^13 forward, 2^12 adjoint, runs of 16) and at those of complex128 (2^12, 2^11).
Host arithmetic only, no GPU."""
import pytest


def align(x):
    return (x + 255) // 256 * 256


@pytest.mark.parametrize("dbl", [False, True])
@pytest.mark.parametrize("n", range(14, 27))
def test_gradient_workspace(n, dbl):
    from paper_2506_10531_gb300 import build
    build.build()
    import paper_2506_10531_gb300 as q
    small = not dbl and n <= 21
    tb, tba, run = ((n + 4) // 2, (n + 4) // 2, 3) if small else (12, 11, 4) if dbl else (13, 12, 4)
    windows = -(-(n - tba) // (tba - run))            # chunks of upper qubits beside the contiguous window
    passes = 1 + 64 * windows                         # for the deepest circuit, p = 64
    want = 2 * align((16 if dbl else 8) << n) + align(8 << (n - tb)) + align(passes * 32 << (n - tba))
    assert q.qaoa_workspace_bytes(n, dbl) == want
