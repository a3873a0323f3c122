"""A DQAOA cycle that fails at any of its waits or event records leaves x as it was and a session that
goes on as if the cycle had not been called: the retry, with the same x and without announcing Q
again, gives the x, energy and accept count of a session that never failed. The failures are error
codes made on the host: a preloaded stand-in for the CUDA calls a cycle waits and orders its work
with fails the n-th of them without calling the driver, in a process of its own."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <dlfcn.h>
static int left = -1;
void fail_call(int n) { left = n; }
static int now(void) { return left >= 0 && left-- == 0; }
#define WRAP(name, args, call) \
    int name args { \
        static int (*real) args; \
        if (!real) real = (int (*) args)dlsym(dlopen("libcudart.so.13", RTLD_LAZY), #name); \
        return now() ? 999 : real call; \
    }
WRAP(cudaEventSynchronize, (void* e), (e))
WRAP(cudaStreamSynchronize, (void* s), (s))
WRAP(cudaEventRecord, (void* e, void* s), (e, s))
"""

SCRIPT = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import synth
import paper_2506_10531_gb300 as q
shim = ctypes.CDLL(sys.argv[2])
k, sampled, changed = int(sys.argv[3]), int(sys.argv[4]), int(sys.argv[5])
N, m, K = 300, 160, 4
ctx = q.qaoa_create(0)
Q1, Q2, x0 = synth.symmetric_q(N, seed=1), synth.symmetric_q(N, seed=2), synth.bits(3, N)
u = synth.uniform01(4, m * 64).reshape(m, 64)
def session():
    s = q.dqaoa_session_create(ctx, N, m, k, 2, K, q.DQAOA_RANDOM, True, [0.4, 0.7], [0.6, 0.3])
    x = x0.copy()
    cycle(s, Q1, 1, x, 0)
    return s, x
def cycle(s, Q, qc, x, c):
    if sampled: return q.dqaoa_session_cycle_sampled(s, Q, qc, x, 5, c, u, 0)
    return q.dqaoa_session_cycle(s, Q, qc, x, 5, c, 0)
Q = Q2 if changed else Q1
s, x = session()
begin = x.copy()
want = cycle(s, Q, changed, x, 1), x.tobytes()
assert x.tobytes() != begin.tobytes()
q.dqaoa_session_destroy(s)
failed = 0
for n in range(100):
    s, x = session()
    assert x.tobytes() == begin.tobytes()
    shim.fail_call(n)
    try:
        got = cycle(s, Q, changed, x, 1), x.tobytes()
        shim.fail_call(-1)
        assert got == want
        break
    except q.QaoaError:
        shim.fail_call(-1)
        failed += 1
        assert x.tobytes() == begin.tobytes(), n
        got = cycle(s, Q, 0, x, 1), x.tobytes()
        assert got == want, n
    q.dqaoa_session_destroy(s)
assert 4 <= failed < 100, failed
print("failures", failed)
"""


@pytest.mark.parametrize("k,sampled,changed", [(15, 0, 0), (15, 0, 1), (10, 0, 1), (10, 1, 0), (10, 1, 1)])
def test_failed_cycle_leaves_no_trace(tmp_path, k, sampled, changed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    shim = tmp_path / "shim.so"
    (tmp_path / "shim.c").write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(shim), str(tmp_path / "shim.c"), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", SCRIPT, ROOT, str(shim), str(k), str(sampled), str(changed)],
                       capture_output=True, text=True, env=dict(os.environ, LD_PRELOAD=str(shim)), timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
