"""The tensor-core contraction's workspace: columns in slabs that fit what the
library's pool keeps."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_helpers import assert_bitexact

pytestmark = pytest.mark.gpu


def _place(x):
    import torch
    import paper_1705_06661_gb300 as ss
    return ss.to_colmajor(torch.from_numpy(np.ascontiguousarray(x)).cuda())


@pytest.mark.parametrize("d,O,S,Y", [(3, 30, 300, 133), (3, 16, 600, 2393)])
def test_columns_in_slabs(d, O, S, Y):
    """Many columns, at once and (75 columns of tiles, 70 at most) in slabs with a ragged last one; C
    padded beyond S; integers are exact, the device's free memory moves by no more than what the pool keeps, and tiles left to the FP64
    kernel (one row of spread magnitudes, an infinity in one column) are the right ones in every slab."""
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    coef = wl.table2({3: 1, 4: 5}[d])
    spec = (S,) + (1,) * (d - 1)
    A, W = wl.integers(1, spec + (O,) * d), wl.integers(2, (Y, O ** d))
    a, w = _place(A), _place(W)
    base = torch.full(((S + 5) * Y,), 7.5, dtype=torch.float64, device="cuda")
    out = base.as_strided(spec + (Y,), [1] + [S] * (d - 1) + [S + 5])
    torch.cuda.synchronize()
    ss.contract(a, coef, w, out=out, factorized=True)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        ss.contract(a, coef, w, out=out, factorized=True)
        torch.cuda.synchronize()
        assert abs(torch.cuda.mem_get_info()[0] - free0) <= 2 << 20
    ss.spinsum_check_status(torch.cuda.current_stream().cuda_stream)
    want = oracle.contract(A, d, coef, W, factorized=True)
    assert_bitexact(out.cpu().numpy(), want)
    assert bool((base.view(Y, S + 5)[:, S:] == 7.5).all())
    A[200] *= 2.0 ** -((np.arange(O ** d) % 40).reshape((1,) * (d - 1) + (O,) * d))
    W[Y - 2, 3] = np.inf
    with np.errstate(all="ignore"):
        want = oracle.contract(A, d, coef, W, factorized=True)
    got = ss.contract(_place(A), coef, _place(W), factorized=True).cpu().numpy()
    keep = np.arange(S) != 200
    assert_bitexact(got[keep], want[keep])
    assert np.array_equal(np.isfinite(got), np.isfinite(want))


def test_captured_graph_holds_kernels_only():
    """A captured call puts no allocation into the graph, so the graph can be instantiated twice, both
    instances can run, and it can be a child of another graph."""
    import ctypes
    import torch
    import oracle
    import paper_1705_06661_gb300 as ss
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(rc):
        assert rc == 0, rc

    d, O, S, Y = 3, 8, 400, 32
    coef = wl.table2(1)
    A, W = wl.integers(3, (S, 1, 1) + (O,) * d), wl.integers(4, (Y, O ** d))
    want = oracle.contract(A, d, coef, W, factorized=True)
    a, w, out = _place(A), _place(W), ss.colmajor_empty((S, 1, 1, Y))
    ss.contract(a, coef, w, out=out, factorized=True)     # the tensor-core path
    assert_bitexact(out.cpu().numpy(), want)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    h = ctypes.c_void_p(st.cuda_stream)
    ok(cu.cuStreamBeginCapture_v2(h, 0))
    try:
        ss.contract(a, coef, w, out=out, factorized=True, stream=st)
    finally:
        g = ctypes.c_void_p()
        rc = cu.cuStreamEndCapture(h, ctypes.byref(g))
    ok(rc)
    n = ctypes.c_size_t(0)
    ok(cu.cuGraphGetNodes(g, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    ok(cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)))
    for k in range(n.value):
        t = ctypes.c_int(-1)
        ok(cu.cuGraphNodeGetType(ctypes.c_void_p(nodes[k]), ctypes.byref(t)))
        assert t.value == 0                               # a kernel
    parent, child = ctypes.c_void_p(), ctypes.c_void_p()
    ok(cu.cuGraphCreate(ctypes.byref(parent), 0))
    ok(cu.cuGraphAddChildGraphNode(ctypes.byref(child), parent, None, ctypes.c_size_t(0), g))
    for graph in (g, g, parent):
        x = ctypes.c_void_p()
        ok(cu.cuGraphInstantiateWithFlags(ctypes.byref(x), graph, ctypes.c_ulonglong(0)))
        out.zero_()
        torch.cuda.synchronize()
        ok(cu.cuGraphLaunch(x, h))
        torch.cuda.synchronize()
        assert_bitexact(out.cpu().numpy(), want)


def test_launches_are_counted():
    """Three launches per slab on the tensor cores (digits of W, products, what is left to FP64), one on the
    FP64 path."""
    import torch
    import paper_1705_06661_gb300 as ss
    d, O, S = 3, 16, 600
    coef, a = wl.table2(1), _place(wl.integers(5, (S, 1, 1) + (O,) * d))
    for Y, strict, n in ((32, False, 3), (2393, False, 6), (32, True, 1)):
        w = _place(wl.integers(6, (Y, O ** d)))
        ss.spinsum_launch_count(reset=True)
        ss.contract(a, coef, w, factorized=True, strict=strict)
        assert ss.spinsum_launch_count(reset=True) == n
    torch.cuda.synchronize()


def test_captured_calls_keep_the_bits_and_give_the_workspace_back():
    """A replay gives the bits of the eager call, on new inputs too; the workspaces of destroyed graphs go
    back to the pool, whose size stays that of a few of them."""
    import torch
    import paper_1705_06661_gb300 as ss
    d, O, S, Y = 3, 30, 300, 64                            # 24 MB of digits
    coef = wl.table2(1)
    A = [_place(wl.uniform(7 + k, (S, 1, 1) + (O,) * d)) for k in range(2)]
    w = _place(wl.uniform(9, (Y, O ** d)))
    a, out = ss.colmajor_like(A[0]), ss.colmajor_empty((S, 1, 1, Y))
    want = [ss.contract(x, coef, w, factorized=True) for x in A]
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for k in range(16):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ss.contract(a, coef, w, out=out, factorized=True)
        a.copy_(A[k % 2])
        g.replay()
        assert torch.equal(out, want[k % 2])
        g.replay()
        del g
        assert torch.equal(ss.contract(A[1], coef, w, factorized=True), want[1])
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= 160 << 20
