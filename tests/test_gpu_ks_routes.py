"""Row-major tensors on both sides of the lines between the on-chip block
kernel and the general one (positions, tensor size, arithmetic), against the
oracle: every arithmetic that changes sides, with alpha and beta, and alpha no
power of two."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact, assert_within, chain_norm, fp32_tol, nterms

pytestmark = pytest.mark.gpu

# d, S, O, arithmetic: the general kernel's side, then the block kernel's
CASES = [
    (2, 300, 40, "fixed"), (2, 600, 40, "fixed"), (2, 340, 90, "mul"), (2, 2040, 16, "f32"), (2, 2100, 16, "f32"),
    (2, 500, 33, "strict"), (2, 2300, 63, "strict"),
    (3, 90, 20, "fixed"), (3, 97, 20, "fixed"), (3, 97, 27, "mul"), (3, 120, 9, "mul"), (3, 200, 14, "f32"),
    (3, 260, 14, "f32"), (3, 260, 15, "strict"),
    (4, 3, 7, "fixed"), (4, 250, 7, "fixed"), (4, 250, 6, "mul"), (4, 900, 9, "f32"), (4, 1700, 9, "f32"),
    (4, 300, 6, "strict"),
]


@pytest.mark.parametrize("d,S,O,mode", CASES)
def test_both_sides_against_oracle(d, S, O, mode):
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    coef = np.array([[2.0, -1.0]]) if d == 2 else wl.table2({3: 1, 4: 5}[d])
    shape = (S,) + (1,) * (d - 1) + (O,) * d
    f32 = mode == "f32"
    dt = torch.float32 if f32 else torch.float64
    alpha = 0.3 if mode == "mul" else -0.5

    def place(x):
        return torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dt)

    A, B0 = wl.uniform(11, shape), wl.uniform(12, shape)
    if f32:
        A, B0 = (np.asfortranarray(x.astype(np.float32).astype(np.float64)) for x in (A, B0))
    for beta in (0.0, 0.75):
        a, b = place(A), place(B0)
        ss.spinsum(a, coef, d=d, out=b, factorized=True, strict=mode == "strict", alpha=alpha, beta=beta)
        got = b.cpu().numpy().astype(np.float64)
        want = oracle.spinsum(A, d, coef, factorized=True, alpha=alpha, beta=beta, B=B0.copy(order="F"))
        if mode == "strict":
            assert_bitexact(got, want)
        elif f32:
            assert_within(got, want, fp32_tol(d, coef, True, A) + 2.0 ** -23 * beta * np.abs(B0).max())
        else:
            # the grid's share of the value, and a rounding of every term on the oracle's side
            tol = (2 * nterms(d, coef, True) + 8) * 2.0 ** -53 * chain_norm(d, coef, True) * abs(alpha) * np.abs(A).max()
            assert_within(got, want, tol + 2.0 ** -52 * beta * np.abs(B0).max())
    if mode in ("fixed", "f32"):
        Ai = wl.integers(13, shape)
        a, b = place(Ai), place(np.zeros(shape))
        ss.spinsum(a, coef, d=d, out=b, factorized=True)
        assert_bitexact(b.cpu().numpy().astype(np.float64), oracle.spinsum(Ai, d, coef, factorized=True))
