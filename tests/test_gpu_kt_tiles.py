"""The contraction on the tensor cores with several tiles per CTA and a last
chunk of one stage (a chunk is 192 tuples in units of 24, a stage two units:
unit counts of 1 or 2 mod 8), so that the group of threads that fills a tile's
last chunk changes from tile to tile. The row scales of the chunks differ by
powers of two from row to row, so a scale of another chunk or tile shows; all
inputs are integers times powers of two, so the results are exact."""
import math

import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact

pytestmark = pytest.mark.gpu


def _units(d, O):
    # members of an orbit by equality pattern, and its number of distinct values
    m = {2: [(2, 2), (1, 1)], 3: [(6, 3), (3, 2), (3, 2), (1, 1)],
         4: [(24, 4), (12, 3), (12, 3), (12, 3), (6, 2), (4, 2), (4, 2), (1, 1)]}[d]
    return sum(-(-math.comb(O, nd) // (24 // mm)) for mm, nd in m)


def _inputs(d, S, O, Y, seed):
    T = O ** d
    A = wl.integers(seed, (S,) + (1,) * (d - 1) + (O,) * d)
    W = wl.integers(seed + 1, (Y, T))
    # tuples with equal indices (the last chunk among them) on a scale of their own in every row
    idx = np.indices((O,) * d)
    rep = np.zeros((O,) * d, dtype=bool)
    for a in range(d):
        for b in range(a):
            rep |= idx[a] == idx[b]
    f = 2.0 ** ((np.arange(S) * 5 // 3) % 9 - 4)
    A = A * np.where(rep, f.reshape((S,) + (1,) * (2 * d - 1)), 1.0)
    return np.asfortranarray(A), W


def _run(A, d, coef, W):
    import torch
    import paper_1705_06661_gb300 as ss
    Wd = ss.colmajor_empty(W.shape)
    Wd.copy_(torch.from_numpy(np.ascontiguousarray(W)))
    C = ss.contract(ss.to_colmajor(torch.from_numpy(A).cuda()), coef, Wd, d=d, factorized=True)
    ss.spinsum_check_status(torch.cuda.current_stream().cuda_stream)
    return C.cpu().numpy()


# d, spectators, O, columns: two to five tiles for each of 152 CTAs
CASES = [(3, 43003, 6, 32), (3, 22000, 6, 64), (2, 45000, 20, 32), (2, 61000, 14, 17)]


@pytest.mark.parametrize("d,S,O,Y", CASES)
def test_scales_of_a_one_stage_last_chunk(d, S, O, Y):
    import oracle
    assert _units(d, O) % 8 in (1, 2) and -(-S // 128) * -(-Y // 32) > 304
    coef = wl.table2(1) if d == 3 else np.array([[2.0, -1.0]])
    A, W = _inputs(d, S, O, Y, 7)
    want = oracle.contract(A, d, coef, W, factorized=True)
    assert_bitexact(_run(A, d, coef, W), want)
    # an infinity in W, in the last chunk's tuples, reaches its column of every row
    W[1, -1] = np.inf
    with np.errstate(all="ignore"):
        want = oracle.contract(A, d, coef, W, factorized=True)
    assert_bitexact(_run(A, d, coef, W), want)
