"""What the tensor-core contraction's grids cost, against sums in extended
precision: inputs of one sign (a truncated grid would bias them), slots of a
chunk that hold no tuple beside a very large element elsewhere, and magnitudes
spread over decades within a chunk."""
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


def _pair(A, d, coef, W):
    """The summation stored, then the contraction alone (both FP64), as _run."""
    import torch
    import paper_1705_06661_gb300 as ss
    full = A.reshape(A.shape[:1] + (1,) * (d - 1) + A.shape[1:])
    a = ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(full)).cuda())
    w = ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(_flat(W, d))).cuda())
    return ss.contract(ss.spinsum(a, coef, d=d, factorized=True), None, w, d=d).cpu().numpy().reshape(A.shape[0], W.shape[0])


def _spread(d, O, S, Y, decades, opposed, seed):
    """A and W with magnitudes spread over the decades, alike within an orbit; opposed: W large where A is small."""
    rng = np.random.default_rng(seed)
    A = rng.uniform(-1, 1, (S,) + (O,) * d)
    W = rng.uniform(-1, 1, (Y,) + (O,) * d)
    orb = np.sort(np.indices((O,) * d).reshape(d, -1), axis=0)
    key = np.ravel_multi_index(tuple(orb), (O,) * d).reshape((O,) * d)
    u = rng.random(O ** d)
    v = 1 - u if opposed else rng.random(O ** d)
    return A * 10.0 ** (-decades * u[key]), W * 10.0 ** (-decades * v[key])


CASES = [(3, 8, 300, 32, 1), (3, 11, 520, 40, 2), (4, 6, 300, 20, 5), (2, 30, 700, 33, "pair"), (3, 9, 400, 24, "random")]


def _coef(d, c):
    if c == "pair":
        return np.array([[2.0, -1.0]])
    return wl.random_coef(d, 17) if c == "random" else wl.table2(c)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("opposed", [False, True])
@pytest.mark.parametrize("decades", [0, 1, 4, 8])
def test_spread_magnitudes(case, opposed, decades):
    """Relative to sum |S W|, a sum of T rounded products has an error of at most about 8 sqrt(T) half units,
    and the grid of an orbit (2^-47 of its largest element or finer, times sum |a|) one of 8 / sqrt(T) of its sum.
    Magnitudes far apart are left to the FP64 kernel, so the result is that of the unfused pair bit for bit."""
    import oracle
    d, O, S, Y, c = case
    coef = _coef(d, c)
    A, W = _spread(d, O, S, Y, decades, opposed, 7)
    T, a = O ** d, oracle.expand(d, coef)
    got, pair = _run(A, d, coef, W), _pair(A, d, coef, W)
    Sx, Wx = _flat(_summed(A, d, a), d), _flat(W, d).astype(np.longdouble)
    want, terms = Sx @ Wx.T, np.abs(Sx) @ np.abs(Wx).T
    mx = np.abs(A)
    for p in oracle.perms(d):
        mx = np.maximum(mx, np.abs(A).transpose([0] + [1 + k for k in np.asarray(p) - np.min(p)]))
    grid = 2.0 ** -47 * np.abs(a).sum() * (_flat(mx, d) @ np.abs(_flat(W, d)).T)
    tol = 8 * T ** 0.5 * 2.0 ** -53 * terms + 8 / T ** 0.5 * grid
    assert np.all(np.abs(got - want) <= tol), float((np.abs(got - want) / tol).max())
    if decades >= 4:
        assert np.array_equal(got, pair)
    if decades == 0:
        assert not np.array_equal(got, pair)     # the tensor cores' rounding


def test_spread_rows_leave_the_others_alone():
    """Only the tiles of 128 rows and 32 columns that hold spread rows or columns change sides."""
    d, O, S, Y = 3, 8, 700, 70
    coef = wl.table2(1)
    A, W = _spread(d, O, S, Y, 0, False, 9)
    A8, W8 = _spread(d, O, S, Y, 8, True, 9)
    base = _run(A, d, coef, W)
    A[300] = A8[300]
    W[40] = W8[40]
    A[5, 2:4] = 0.0                                # zeros are no spread
    got, pair = _run(A, d, coef, W), _pair(A, d, coef, W)
    assert np.array_equal(got[256:384], pair[256:384]) and np.array_equal(got[:, 32:64], pair[:, 32:64])
    keep = np.r_[6:256, 384:S]
    assert np.array_equal(got[keep][:, :32], base[keep][:, :32]) and np.array_equal(got[keep][:, 64:], base[keep][:, 64:])
    assert not np.array_equal(got[:128, :32], pair[:128, :32])


def test_strict_equals_the_unfused_pair():
    """With STRICT a call of any size is FP64 throughout: that of the strict summation, stored and contracted."""
    import torch
    import paper_1705_06661_gb300 as ss
    d, O, S, Y = 3, 8, 300, 32
    A, W = _spread(d, O, S, Y, 0, False, 12)
    a = ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(A.reshape((S, 1, 1) + (O,) * d))).cuda())
    w = ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(_flat(W, d))).cuda())
    coef = wl.table2(1)
    got = ss.contract(a, coef, w, factorized=True, strict=True)
    pair = ss.contract(ss.spinsum(a, coef, factorized=True, strict=True), None, w)
    assert torch.equal(got, pair)
