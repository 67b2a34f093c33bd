"""The contraction on the tensor cores: the edges of its 128-row tiles, 32-column
tiles and 144-tuple chunks against the oracle, inputs whose digits are all
extreme (the FP32 digit sums come closest to 2^24), chunks of very different
magnitude, and tiles whose scales leave the exponent range (recomputed in FP64)."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact, chain_norm

pytestmark = pytest.mark.gpu


def _coef(d, c):
    if c == "pair":
        return wl.coef_vector(2, [(2.0, "12"), (-1.0, "21")])[None, :]
    return wl.random_coef(d, 17) if c == "random" else wl.table2(c)


def _run(A, d, coef, W):
    import torch
    import paper_1705_06661_gb300 as ss
    Wd = ss.colmajor_empty(W.shape)
    Wd.copy_(torch.from_numpy(np.ascontiguousarray(W)))
    C = ss.contract(ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(A)).cuda()), coef, Wd, d=d, factorized=True)
    ss.spinsum_check_status(torch.cuda.current_stream().cuda_stream)
    return C.cpu().numpy()


def _tol(A, d, coef, W):
    # each summed value carries at most 1e-14 L max|A|; T roundings of partial sums on each side
    T = W.shape[1]
    return (1e-14 + 2 * T * 2.0 ** -53) * chain_norm(d, coef, True) * np.abs(A).max() * np.abs(W).sum(axis=1).max()


# d, spectators (S = 257, 512, 513, 516, several tiles per CTA), O (a partial unit, a
# partial stage, an exact chunk, several chunks), columns
CASES = [
    (3, (257, 1, 1), 6, 1, 5), (3, (8, 8, 8), 4, 1, 17), (3, (513, 1, 1), 5, 2, 31), (3, (8, 16, 4), 6, 1, 32), (3, (43, 12, 1), 13, "random", 33),
    (3, (33, 32, 31), 3, 3, 65), (2, (32, 16), 12, "pair", 20), (2, (129, 5), 30, "pair", 40),
    (4, (2, 3, 4, 25), 3, 5, 30), (4, (8, 8, 8, 1), 5, "random", 32), (4, (129, 1, 5, 1), 6, 6, 3),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_edges_against_oracle(case):
    import oracle
    d, spec, O, c, Y = CASES[case]
    coef = _coef(d, c)
    A = wl.uniform(20 + case, spec + (O,) * d)
    W = wl.uniform(50 + case, (Y, O ** d))
    want = oracle.contract(A, d, coef, W, factorized=True)
    err = np.abs(_run(A, d, coef, W) - want).max()
    assert err <= _tol(A, d, coef, W), err
    Ai, Wi = wl.integers(70 + case, A.shape), wl.integers(80 + case, W.shape)
    assert_bitexact(_run(Ai, d, coef, Wi), oracle.contract(Ai, d, coef, Wi, factorized=True))


def test_extreme_digits():
    """Every byte of every factor at its largest magnitude with one sign: any digit sum that FP32 could not
    hold would show at 2^-24 of the result; the bound is that of the FP64 sum."""
    import oracle
    d, O, spec = 3, 8, (16, 8, 4)
    coef = np.zeros((1, 6))
    coef[0, 0] = 1.0
    v = -float(int("80" * 6 + "8", 16) << 1) / 2.0 ** 53   # digits of -128 throughout
    A = np.full(spec + (O,) * d, v, order="F")
    W = np.full((32, O ** d), v, order="F")
    want = oracle.contract(A, d, coef, W, factorized=True)
    got = _run(A, d, coef, W)
    assert np.abs(got - want).max() <= 2 * O ** d * 2.0 ** -53 * O ** d * v * v


def test_scales_per_chunk_and_out_of_range():
    import oracle
    d, O, spec, Y = 3, 9, (64, 4, 2), 12
    coef = _coef(d, 1)
    A = wl.uniform(1, spec + (O,) * d)
    W = wl.uniform(2, (Y, O ** d))
    # rows and columns of very different magnitude stay accurate on their own scale
    rows = 2.0 ** np.linspace(-300, 100, 64)
    A1 = np.asfortranarray(A * rows.reshape(64, 1, 1, 1, 1, 1))
    W1 = np.asfortranarray(W * (2.0 ** np.linspace(-200, 200, Y))[:, None])
    want = oracle.contract(A1, d, coef, W1, factorized=True)
    got = _run(A1, d, coef, W1)
    base = _tol(A, d, coef, W)
    tol = base * rows.reshape(64, 1, 1, 1) * (2.0 ** np.linspace(-200, 200, Y))
    assert np.all(np.abs(got - want) <= tol)
    # infinities, NaN, huge, tiny and subnormal values, zero rows
    for v in (np.inf, np.nan, 1e300, 1e-300, 5e-324, 0.0):
        A2 = A.copy(order="F")
        A2[3, 1, 1] = v
        with np.errstate(all="ignore"):
            want = oracle.contract(A2, d, coef, W, factorized=True)
        got = _run(A2, d, coef, W)
        assert np.array_equal(np.isfinite(got), np.isfinite(want)), v
        other = np.ones(spec, dtype=bool)
        other[3, 1, 1] = False
        assert np.abs(got[other] - want[other]).max() <= base, v
        if np.isfinite(v) and np.isfinite(want).all():
            lim = (1e-14 + 2 * O ** d * 2.0 ** -53) * 12 * abs(v) * np.abs(W).sum(axis=1).max() + 1e-320
            assert np.abs(got[3, 1, 1] - want[3, 1, 1]).max() <= lim, v


def test_capture_and_streams():
    """The workspace is stream-ordered: a captured call replays on new inputs, and calls on two streams
    at once do not share it."""
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    d, O, spec, Y = 3, 7, (24, 8, 4), 20
    coef = _coef(d, 1)
    As = [wl.integers(5 + k, spec + (O,) * d) for k in range(2)]
    Ws = [wl.integers(15 + k, (Y, O ** d)) for k in range(2)]
    want = [oracle.contract(a, d, coef, w, factorized=True) for a, w in zip(As, Ws)]
    A, W = ss.colmajor_empty(As[0].shape), ss.colmajor_empty(Ws[0].shape)
    out = ss.colmajor_empty(spec + (Y,))

    def fill(a, w, k):
        a.copy_(torch.from_numpy(As[k]))
        w.copy_(torch.from_numpy(Ws[k]))

    fill(A, W, 0)
    ss.contract(A, coef, W, out=out, factorized=True)
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
        ss.contract(A, coef, W, out=out, factorized=True)
    torch.cuda.current_stream().wait_stream(s)
    for k in (1, 0, 1):
        fill(A, W, k)
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert_bitexact(out.cpu().numpy(), want[k], f"replay {k}")
    streams = [torch.cuda.Stream() for _ in range(2)]
    ins = []
    for k in range(2):
        a, w, c = ss.colmajor_empty(As[k].shape), ss.colmajor_empty(Ws[k].shape), ss.colmajor_empty(spec + (Y,))
        fill(a, w, k)
        ins.append((a, w, c))
    torch.cuda.synchronize()
    for _ in range(20):
        for k in range(2):
            ss.contract(ins[k][0], coef, ins[k][1], out=ins[k][2], factorized=True, stream=streams[k])
    torch.cuda.synchronize()
    for k in range(2):
        assert_bitexact(ins[k][2].cpu().numpy(), want[k], f"stream {k}")
