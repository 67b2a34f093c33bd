"""What the tensor-core contraction's grids cost, against sums in extended
precision: inputs of one sign (a truncated grid would bias them), and slots of a
chunk that hold no tuple beside a very large element elsewhere."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _summed(A, d, a):
    """S(A) of A [S, O, .., O] in extended precision, expanded coefficients a."""
    import oracle
    out = np.zeros(A.shape, dtype=np.longdouble)
    for c, p in zip(a, oracle.perms(d)):
        if c != 0.0:
            q = np.argsort(np.asarray(p) - np.min(p))
            out += np.longdouble(c) * A.astype(np.longdouble).transpose([0] + [1 + k for k in q])
    return out


def _flat(x, d):
    """[n, O, .., O] -> [n, T], first permuted index fastest."""
    return x.transpose([0] + list(range(d, 0, -1))).reshape(x.shape[0], -1)


def _run(A, d, coef, W):
    """A [S, O, .., O], W [Y, O, .., O] -> C [S, Y]."""
    import torch
    import paper_1705_06661_gb300 as ss
    full = A.reshape(A.shape[:1] + (1,) * (d - 1) + A.shape[1:])
    a = ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(full)).cuda())
    w = ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(_flat(W, d))).cuda())
    C = ss.contract(a, coef, w, d=d, factorized=True)
    ss.spinsum_check_status(torch.cuda.current_stream().cuda_stream)
    return C.cpu().numpy().reshape(A.shape[0], W.shape[0])


def test_inputs_of_one_sign_are_not_biased():
    """Equal coefficients of 1-norm 126 leave 47 bits for A; every element in [1/2, 1) is rounded to 2^-47
    independently, so an error beyond 8 standard deviations (and the one rounding of the only chunk) is a bias."""
    d, O, S, Y = 3, 5, 400, 32
    coef = np.full((1, 6), 21.0)
    rng = np.random.default_rng(3)
    A = 0.5 + 0.5 * rng.random((S,) + (O,) * d)
    W = 0.5 + 0.5 * rng.random((Y,) + (O,) * d)
    want = _flat(_summed(A, d, coef[0]), d) @ _flat(W, d).astype(np.longdouble).T
    wsum = _flat(_summed(W, d, coef[0]), d)
    sigma = 2.0 ** -47 / 12 ** 0.5 * np.sqrt((wsum ** 2).sum(axis=1))
    err = np.abs(_run(A, d, coef, W) - want)
    # W is rounded to 2^-54 or finer, and digit pairs below 2^-56 of the largest product are left out
    assert np.all(err <= 8 * sigma + (2.0 ** -53 + 2.0 ** -51) * want)


def test_empty_slots_do_not_coarsen_a_chunk():
    """O = 6 leaves slots of the first chunk empty; the tuple (0, 0, 0) belongs to the second. W is zero there."""
    d, O, S, Y = 3, 6, 600, 20
    coef = wl.table2(1)
    rng = np.random.default_rng(4)
    A = rng.uniform(-1, 1, (S,) + (O,) * d)
    W = rng.uniform(-1, 1, (Y,) + (O,) * d)
    i, j, k = np.indices((O,) * d)
    W[:, (i == j) | (j == k) | (i == k)] = 0.0
    A[:, 0, 0, 0] = 2.0 ** 40
    import oracle
    Sx = _flat(_summed(A, d, oracle.expand(d, coef)), d)
    Wx = _flat(W, d).astype(np.longdouble)
    want, terms = Sx @ Wx.T, np.abs(Sx) @ np.abs(Wx).T
    # 12 * 2^-51 per element of A at most 1, of 120 tuples with sum |S W| above a tenth of them
    assert np.all(np.abs(_run(A, d, coef, W) - want) <= 2.0 ** -44 * terms)
