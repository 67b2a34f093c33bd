"""The beta term of the spectators-fastest kernels (their own instantiations)
and FP32 runs with 4-byte loads: spectator counts below, at and past one and
two chunks of a block, odd (no wide loads) and even, against the oracle."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact, assert_within, fp32_tol, fp64_tol, gpu_run

pytestmark = pytest.mark.gpu

SPECS = [(65, 1), (256, 1), (257, 1), (511, 1), (32, 32), (41, 63)]


@pytest.mark.parametrize("spec", SPECS)
@pytest.mark.parametrize("d,O,row", [(2, 6, 0), (3, 5, 1), (3, 4, 2), (4, 5, 5), (4, 4, 18)])
@pytest.mark.parametrize("mode", ["f64", "strict", "f32", "f32-beta0"])
def test_beta_against_oracle(spec, d, O, row, mode):
    import oracle
    coef = wl.table2(row) if row else wl.coef_vector(2, [(2.0, "12"), (-1.0, "21")])[None, :]
    shape = spec + (1,) * (d - 2) + (O,) * d
    A, B0 = wl.uniform(11, shape), wl.uniform(12, shape)
    f32 = mode.startswith("f32")
    if f32:
        A, B0 = (np.asfortranarray(x.astype(np.float32).astype(np.float64)) for x in (A, B0))
    beta = 0.0 if mode == "f32-beta0" else -0.375
    want = oracle.spinsum(A, d, coef, factorized=True, beta=beta, B=B0.copy(order="F"))
    got = gpu_run(A, d, coef, factorized=True, beta=beta, B0=B0, strict=mode == "strict", dtype="f32" if f32 else "f64")
    if mode == "strict":
        assert_bitexact(got, want)
    elif f32:
        assert_within(got, want, fp32_tol(d, coef, True, A) + 2.0 ** -23 * np.abs(B0).max())
    else:
        assert_within(got, want, fp64_tol(d, coef, True, A) + 2.0 ** -52 * np.abs(B0).max())
