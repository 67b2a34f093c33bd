"""Row-major FP64 with magnitudes spread over decades within an orbit: every
output against the exact sum, relative to the sum of its own terms' magnitudes,
also where the operator has zero coefficients and an output takes none of the
orbit's large inputs.

Tolerance, in units of 2^-53 of sum |a x|: a group summed in FP64 rounds every
product and partial sum of the chain, at most 2 n + 2 times for n terms. A group
summed on the grid rounds its inputs to 2^(E - bits) and the result once; the
largest input of every output is at least 2^(E - k), so the grid's share is at
most sum|a| / min|a| * 2^(k + 53 - bits)."""
import math

import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import nterms

pytestmark = pytest.mark.gpu

# d, Table II row, S, O
CASES = [(3, 1, 40, 9), (3, 2, 40, 9), (3, 3, 5, 14), (4, 5, 12, 5), (4, 6, 9, 6), (4, 18, 7, 7)]


def _expanded(d, coef):
    import oracle
    return oracle.expand(d, coef)


def _exact(A, d, a):
    import oracle
    out = np.zeros(A.shape, dtype=np.longdouble)
    n = A.ndim - d
    for c, p in zip(a, oracle.perms(d)):
        if c != 0.0:
            q = np.argsort(np.asarray(p) - np.min(p))
            out += np.longdouble(c) * A.transpose(list(range(n)) + [n + k for k in q])
    return out


def _bound(d, coef, a):
    L = float(np.abs(a).sum()) if d == 4 else float(np.prod([np.abs(f).sum() for f in np.atleast_2d(coef)]))
    lg = math.ceil(math.log2(L))
    bits = min(60, 62 - lg) if d < 4 else (61 - lg if 2 ** lg > L else 60 - lg)
    nz = np.abs(a[a != 0])
    k = 0
    if nz.size < a.size:
        k = max(3, min(6, math.floor(bits - 53 - math.log2(math.sqrt((nz ** 2).sum()) / nz.min()) + 2)))
    return max(2 * nterms(d, coef, True) + 2, 2 + L / nz.min() * 2.0 ** (k + 53 - bits))


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("decades", [0, 2, 5, 10])
def test_error_relative_to_the_terms(case, decades):
    import torch
    import paper_1705_06661_gb300 as ss
    d, row, S, O = CASES[case]
    coef = wl.table2(row)
    a = _expanded(d, coef)
    shape = (S,) + (1,) * (d - 1) + (O,) * d
    A = wl.uniform(30 + case, shape) * 10.0 ** (-0.5 * decades * (1.0 + wl.uniform(60 + case, shape)))
    A[1] = np.where(wl.integers(5, shape)[1] > 0, A[1], 0.0)     # with zeros
    x = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    b = torch.empty_like(x)
    alpha = 0.3 if d == 3 else 1.0
    ss.spinsum(x, coef, d=d, out=b, factorized=True, alpha=alpha)
    got = b.cpu().numpy().astype(np.longdouble) / np.longdouble(alpha)
    Al = np.asarray(A, dtype=np.longdouble)
    want, terms = _exact(Al, d, a), _exact(np.abs(Al), d, np.abs(a))
    err = np.abs(got - want)
    # (alpha's multiplication: one more rounding)
    assert np.all(err <= (_bound(d, coef, a) + 1) * 2.0 ** -53 * terms), float(
        (err[terms > 0] / terms[terms > 0]).max() * 2.0 ** 53)
