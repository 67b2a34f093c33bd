"""Pinned host tensors in the paper's layout (every index permuted), read and
written over the host link by the tiled kernel's plain loads and stores; and the
TMA-fed tiled kernel with an alpha that is no power of two."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact, assert_within, fp64_tol, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N", [(2, 70), (3, 32), (3, 19), (4, 12)])
@pytest.mark.parametrize("inplace", [False, True])
def test_pinned_paper_layout(d, N, inplace):
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    coef = np.array([[2.0, -1.0]]) if d == 2 else wl.table2({3: 1, 4: 5}[d])
    A = wl.integers(N, (N,) * d)
    want = oracle.spinsum(A, d, coef, factorized=True)
    t = torch.empty((N,) * d, dtype=torch.float64).pin_memory().permute(*reversed(range(d)))
    o = torch.empty((N,) * d, dtype=torch.float64).pin_memory().permute(*reversed(range(d)))
    t.copy_(torch.from_numpy(A))
    out = ss.spinsum_host(t, coef, out=None if inplace else o, d=d, factorized=True, inplace=inplace)
    torch.cuda.synchronize()
    assert_bitexact(out.numpy(), want)


@pytest.mark.parametrize("d,N", [(3, 24), (3, 50), (4, 16)])
def test_alpha_no_power_of_two(d, N):
    import oracle
    coef = wl.table2({3: 1, 4: 5}[d])
    A = wl.uniform(N, (N,) * d)
    for inplace in (False, True):
        got = gpu_run(A, d, coef, factorized=True, alpha=0.3, inplace=inplace)
        assert_within(got, oracle.spinsum(A, d, coef, factorized=True, alpha=0.3), fp64_tol(d, coef, True, A, 0.3))
