"""The TMA-fed tiled kernel (the paper's layout with 16-byte strides, no beta
term): extents below, at and past one tile, a ragged last tile, several coarse
groups; every arithmetic it takes; in place; padded strides with untouched
gaps; groups outside the fixed-point range; and bit for bit the results of the
copying tiled kernel (reached through an unaligned base address)."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact, assert_within, fp32_tol, fp64_tol

pytestmark = pytest.mark.gpu

CASES = [(3, 2), (3, 8), (3, 10), (3, 30), (3, 72), (3, 132),
         (4, 2), (4, 4), (4, 6), (4, 16), (4, 22), (4, 36)]


def _coef(d):
    return {3: wl.table2(1), 4: wl.table2(5)}[d]


def _place(x, dtype, pad=0, offset=0):
    """x column-major on the GPU, rows padded by `pad` elements, the base `offset` elements into its allocation."""
    import torch
    d, n = x.ndim, x.shape[0]
    ld = [1]
    for _ in range(d - 1):
        ld.append((n + pad) if len(ld) == 1 else ld[-1] * n)
    base = torch.full((ld[-1] * n + offset + 8,), 7.5, dtype=dtype, device="cuda")
    t = base.as_strided(x.shape, ld, offset)
    t.copy_(torch.from_numpy(np.ascontiguousarray(x)))
    return base, t


@pytest.mark.parametrize("d,N", CASES)
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("inplace", [False, True])
def test_against_oracle_and_copying_kernel(d, N, dtype, inplace):
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    if dtype == "f32" and N % 4:
        N += 4 - N % 4
    dt = torch.float64 if dtype == "f64" else torch.float32
    coef = _coef(d)
    for A in (wl.integers(N, (N,) * d), wl.uniform(N + 1, (N,) * d)):
        if dtype == "f32":
            A = np.asfortranarray(A.astype(np.float32).astype(np.float64))
        want = oracle.spinsum(A, d, coef, factorized=True, alpha=-0.5)
        out = []
        for offset in (0, 1):   # an odd base takes the copying kernel
            _, a = _place(A, dt, offset=offset)
            b = a if inplace else _place(np.zeros_like(A), dt, offset=offset)[1]
            ss.spinsum(a, coef, d=d, out=b, factorized=True, alpha=-0.5, inplace=inplace)
            ss.spinsum_check_status(torch.cuda.current_stream().cuda_stream)
            out.append(b.cpu().numpy())
        assert_bitexact(out[0], out[1], "copying kernel")
        if dtype == "f64":
            assert_within(out[0], want, fp64_tol(d, coef, True, A, 0.5))
        else:
            assert_within(out[0].astype(np.float64), want, fp32_tol(d, coef, True, A))


@pytest.mark.parametrize("d,N,pad", [(3, 26, 2), (4, 14, 4)])
def test_gaps_stay_untouched(d, N, pad):
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    A = wl.integers(3, (N,) * d)
    _, a = _place(A, torch.float64, pad)
    base, b = _place(np.zeros_like(A), torch.float64, pad)
    ss.spinsum(a, _coef(d), d=d, out=b, factorized=True)
    assert_bitexact(b.cpu().numpy(), oracle.spinsum(A, d, _coef(d), factorized=True))
    b.fill_(7.5)
    assert bool((base == 7.5).all())


@pytest.mark.parametrize("d,N", [(3, 20), (4, 10)])
def test_groups_outside_the_fixed_point_range(d, N):
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    A = wl.uniform(8, (N,) * d)
    idx = tuple(np.random.default_rng(1).integers(0, N, (d, 60)))
    A[idx] = np.resize([0.0, 1e-300, 5e-324, 1e300, np.inf, np.nan], 60)
    _, a = _place(A, torch.float64)
    _, b = _place(np.zeros_like(A), torch.float64)
    ss.spinsum(a, _coef(d), d=d, out=b, factorized=True)
    with np.errstate(all="ignore"):
        want = oracle.spinsum(A, d, _coef(d), factorized=True)
    got = b.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    small = np.isfinite(want) & (np.abs(want) < 1e100)
    assert np.abs(got[small] - want[small]).max() <= fp64_tol(d, _coef(d), True, np.ones(1))
