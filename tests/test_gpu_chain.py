"""A batched plan run as a chain of overlapping single-problem launches (one of
the tuner's choices): forced through an autotune cache file, checked against
the oracle for even and odd spectator counts, FP32, beta, alpha, in place and a
problem of the general path, on a stream and in a replayed graph, with work
behind it in the stream that must see every result."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
import sys
import numpy as np, torch
import oracle, workloads as wl
import paper_1705_06661_gb300 as ss

def problems(dt):
    out = []
    for b, (V, O, row) in enumerate([(16, 6, 1), (17, 7, 2), (20, 5, 3), (13, 9, 4), (24, 4, 1), (21, 3, 2), (18, 2, 3)]):
        shape = (V, V - 1, V + 1 - b % 2) + (O,) * 3
        A, B = wl.uniform(900 + b, shape), wl.uniform(950 + b, shape)
        if dt == torch.float32:
            A, B = (np.asfortranarray(x.astype(np.float32).astype(np.float64)) for x in (A, B))
        inplace = b == 4
        beta = 0.5 if b in (1, 2) else 0.0
        alpha = 0.3 if b == 3 else 1.0
        place = lambda x: (torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dt) if b == 5
                           else ss.to_colmajor(torch.from_numpy(x).to("cuda", dt)))
        a = place(A)
        out.append(dict(A=a, B=None if inplace else place(B), coef=wl.table2(row), d=3, factorized=True, alpha=alpha,
                        beta=beta, host=(A, B)))
    return out

mode, dtype = sys.argv[1], sys.argv[2]
dt = torch.float64 if dtype == "f64" else torch.float32
ps = problems(dt)
plan = ss.Plan(ps, tune=True)
print(plan.describe())
if mode == "check":
    assert "launch-per-problem" in plan.describe() and "cached" in plan.describe(), plan.describe()
    for run in ("stream", "graph"):
        for p in ps:
            p["A"].copy_(torch.from_numpy(p["host"][0]))
            if p["B"] is not None:
                p["B"].copy_(torch.from_numpy(p["host"][1]))
        if run == "stream":
            plan.execute()
        else:
            g = torch.cuda.CUDAGraph()
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
                plan.execute()
            torch.cuda.current_stream().wait_stream(s)
            g.replay()
        copies = [(p["A"] if p["B"] is None else p["B"]).clone() for p in ps]   # right behind, in stream order
        torch.cuda.synchronize()
        for p, c in zip(ps, copies):
            A, B = p["host"]
            want = oracle.spinsum(A, 3, p["coef"], factorized=True, alpha=p["alpha"], beta=p["beta"],
                                  B=B.copy(order="F"))
            L = float(np.prod([np.abs(f).sum() for f in p["coef"]]))
            eps = 1e-14 if dt == torch.float64 else 14 * 2.0 ** -24
            err = np.abs(c.cpu().numpy() - want).max()
            assert err <= eps * L * np.abs(A).max() + eps * np.abs(B).max(), (run, A.shape, err)
    print("ok")
'''


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_chained_plan(tmp_path, dtype):
    cache = tmp_path / "tune"
    env = dict(os.environ, SPINSUM_AUTOTUNE_CACHE=str(cache), PYTHONPATH=ROOT)

    def run(mode):
        r = subprocess.run([sys.executable, "-c", PROGRAM, mode, dtype], cwd=ROOT, env=env, capture_output=True,
                           text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout

    run("tune")                                   # writes the problems' key
    lines = cache.read_text().splitlines()
    assert len(lines) == 1
    cache.write_text(lines[0].rsplit("\t", 1)[0] + "\t3 2 1\n")
    assert "ok" in run("check")
