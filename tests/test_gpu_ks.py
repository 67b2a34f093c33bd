"""The on-chip block kernel: tensors whose permuted indices form one dense
block per spectator position (torch-contiguous ones, and any other order of the
permuted indices), against the oracle at the edges of its range: the smallest
and largest blocks, odd and even extents, spectator counts that leave a ragged
last round, strided spectators, alpha/beta, in place, strict order, FP32, and
groups outside the fixed-point range."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact, assert_within, chain_norm, fp32_tol, nterms

pytestmark = pytest.mark.gpu

# d, spectator extents, O, coefficient chain
CASES = [
    (2, (3, 5), 8, "pair"), (2, (7, 1), 31, "pair"), (2, (2, 2), 100, "pair"),
    (3, (5, 3, 7), 4, 1), (3, (4, 3, 5), 5, 2), (3, (3, 3, 3), 12, 1), (3, (2, 5, 3), 16, "random"),
    (3, (1, 2, 2), 27, 3),
    (4, (3, 2, 3, 5), 3, 5), (4, (2, 3, 2, 2), 6, 6), (4, (2, 1, 2, 1), 9, "random"), (4, (1, 1, 2, 1), 12, 5),
]


def _coef(d, c):
    if c == "pair":
        return wl.coef_vector(2, [(2.0, "12"), (-1.0, "21")])[None, :]
    return wl.random_coef(d, 31) if c == "random" else wl.table2(c)


def _tol64(d, coef, A, alpha=1.0):
    # the grid contributes at most L max|A| 2^-52, the final rounding half a unit of at most
    # L max|A|; the oracle rounds every product and every partial sum of a chain once
    return (2 * nterms(d, coef, True) + 6) * 2.0 ** -53 * chain_norm(d, coef, True) * abs(alpha) * np.abs(A).max()


def _place(x, d, order, dtype):
    """x on the GPU with the permuted indices as one dense block, fastest, in the given memory order."""
    import torch
    n = 2 * d
    # memory order, slowest first: spectators, then the permuted indices as `order` says
    mem = list(range(d)) + [d + k for k in order]
    t = torch.from_numpy(np.ascontiguousarray(x.transpose(mem))).to("cuda", dtype)
    inv = [mem.index(k) for k in range(n)]
    return t.permute(*inv)


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("mode", ["plain", "beta", "inplace", "adjoint", "strict", "f32"])
def test_against_oracle(case, mode):
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    d, spec, O, c = CASES[case]
    coef = _coef(d, c)
    shape = spec + (O,) * d
    A = wl.uniform(40 + case, shape)
    B0 = wl.uniform(90 + case, shape)
    f32 = mode == "f32"
    if f32:
        A = A.astype(np.float32).astype(np.float64)
    dt = torch.float32 if f32 else torch.float64
    order = list(range(d)) if case % 2 else list(reversed(range(d)))
    alpha, beta = (-0.5, 0.75) if mode == "beta" else (1.0, 0.0)
    a = _place(A, d, order, dt)
    b = a if mode == "inplace" else _place(B0, d, order, dt)
    ss.spinsum(a, coef, d=d, out=b, factorized=True, adjoint=mode == "adjoint", strict=mode == "strict",
               alpha=alpha, beta=beta, inplace=mode == "inplace")
    got = b.cpu().numpy().astype(np.float64)
    if mode == "adjoint":
        want = oracle.spinsum_transpose(A, d, coef)
    else:
        want = oracle.spinsum(A, d, coef, factorized=True, alpha=alpha, beta=beta,
                              B=B0.copy(order="F") if mode == "beta" else None)
    if mode == "strict":
        assert_bitexact(got, want)
    elif f32:
        assert_within(got, want, fp32_tol(d, coef, True, A))
    else:
        extra = 2.0 ** -52 * abs(beta) * np.abs(B0).max()
        assert_within(got, want, _tol64(d, coef, A, alpha) + extra)


@pytest.mark.parametrize("case", [1, 4, 5, 8, 9])
def test_integer_inputs_and_strided_spectators(case):
    """Integer inputs are exact; the spectator offsets come from their own strides, and nothing
    outside the output's elements is written."""
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    d, spec, O, c = CASES[case]
    coef = _coef(d, c)
    shape = spec + (O,) * d
    A = wl.integers(60 + case, shape)
    big = (spec[0] + 2,) + spec[1:] + (O,) * d
    base = torch.full(big, 7.5, dtype=torch.float64, device="cuda")
    out = torch.full(big, 7.5, dtype=torch.float64, device="cuda")
    base[1:1 + spec[0]].copy_(torch.from_numpy(np.ascontiguousarray(A)))
    ss.spinsum(base[1:1 + spec[0]], coef, d=d, out=out[1:1 + spec[0]], factorized=True)
    assert_bitexact(out[1:1 + spec[0]].cpu().numpy(), oracle.spinsum(A, d, coef, factorized=True))
    assert bool((out[0] == 7.5).all()) and bool((out[-1] == 7.5).all())


@pytest.mark.parametrize("d,O,c", [(3, 6, 1), (4, 4, 5)])
def test_groups_outside_the_fixed_point_range(d, O, c):
    """Zeros, subnormals, huge values, infinities and NaN: groups that leave the range are summed
    in the reference order, bit for bit; their neighbours stay accurate."""
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    coef = _coef(d, c)
    spec = (2,) * d
    shape = spec + (O,) * d
    A = wl.uniform(5, shape)
    flat = A.reshape(2 ** d, -1)
    for row, v in enumerate([0.0, 5e-324, 1e300, 1e-300, np.inf, np.nan]):
        flat[row] = v if np.isfinite(v) else flat[row]
        if not np.isfinite(v):
            flat[row, 3] = v
    A = np.asfortranarray(flat.reshape(shape))
    a = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    b = torch.empty_like(a)
    ss.spinsum(a, coef, d=d, out=b, factorized=True)
    # the transform of d = 4 applies the expanded operator; the oracle's chain gives the same
    # infinities and NaN where the expansion has no zero coefficients
    want = oracle.spinsum(A, d, coef, factorized=True)
    got = b.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    fin = np.isfinite(want)
    scale = np.abs(np.where(np.isfinite(A), A, 0)).reshape(2 ** d, -1).max(axis=1)
    tol = (2 * nterms(d, coef, True) + 6) * 2.0 ** -53 * chain_norm(d, coef, True) * scale + 5e-324
    tol = np.broadcast_to(tol.reshape(spec + (1,) * d), shape)
    assert np.all(np.abs(got[fin] - want[fin]) <= tol[fin])
