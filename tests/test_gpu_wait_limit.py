"""Kernels whose waits run out: with a limit of one poll a wait may be over
before its phase is, in any role of a kernel. The kernel must then let its own
copies and matrix instructions finish, report, and return: the status is OK (no
wait ran out; the result is then right) or TIMEOUT, and a call after it that
waits for nothing is right."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import numpy as np, torch, oracle
import workloads as wl
import paper_1705_06661_gb300 as ss
from tests.gpu_helpers import assert_bitexact, gpu_run
st = torch.cuda.current_stream().cuda_stream
coef = wl.table2(1)
P = wl.integers(7, (8, 8, 8, 5, 5, 5))
good = oracle.spinsum(P, 3, coef, factorized=True)

def check(call, result, want):
    # a call whose wait ran out leaves its output unspecified, but nothing else
    out = 0
    for k in range(30):
        call()
        try:
            ss.spinsum_check_status(st)
            assert_bitexact(result().cpu().numpy(), want, "no wait ran out")
        except ss.SpinsumError as e:
            assert "TIMEOUT" in str(e), e
            out += 1
        B = gpu_run(P, 3, coef, factorized=True)
        assert_bitexact(B, good, "the call after")
    print("ran out", out)
"""

CONTRACT = """
A = wl.integers(1, (30000, 1, 1, 6, 6, 6))
W = wl.integers(2, (32, 216))
a = ss.to_colmajor(torch.from_numpy(A).cuda())
w = ss.to_colmajor(torch.from_numpy(W).cuda())
c = ss.colmajor_empty((30000, 1, 1, 32))
check(lambda: ss.contract(a, coef, w, out=c, factorized=True), lambda: c, oracle.contract(A, 3, coef, W, factorized=True))
"""


def _run(body):
    env = dict(os.environ, SPINSUM_WAIT_LIMIT="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", HEAD + body], cwd=ROOT, env=env, capture_output=True, text=True, timeout=200)
    assert r.returncode == 0, r.stdout + r.stderr
    print(r.stdout)


def test_contraction():
    _run(CONTRACT)


TILED = """
for d, N in ((3, 96), (4, 28)):
    A = wl.integers(d, (N,) * d)
    coef_d = wl.table2({3: 1, 4: 5}[d])
    a = ss.to_colmajor(torch.from_numpy(A).cuda())
    b = ss.colmajor_like(a)
    check(lambda: ss.spinsum(a, coef_d, d=d, out=b, factorized=True), lambda: b, oracle.spinsum(A, d, coef_d, factorized=True))
"""


def test_tiled_kernel():
    _run(TILED)
