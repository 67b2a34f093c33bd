"""The workloads that this library is timed on: what a coupled-cluster code asks
of it, through the public entry points of `paper_1705_06661_gb300`.

Kinds of case:
  spin      one spin summation of a CCSD/CCSDT/CCSDTQ tensor with the spectator
            indices fastest (the library's own layout): `spinsum`
  paper     the same on a dense N^d tensor, every index permuted, the first one
            at stride 1 (column-major): `spinsum`
  rowmajor  the same on a torch-contiguous tensor (last permuted index fastest)
  batch     many independent 3D blocks through one `Plan`
  autograd  `spinsum_autograd` forward, then its gradient
  contract  the summation fused into a contraction with a matrix: `contract`
  packed    `unpack` of packed antisymmetric storage, then `pack` of the result

Inputs are uniform in [-1, 1), the stand-in for amplitudes that the
repository's tests and benchmark use throughout.
"""
import itertools
import math
import random

import numpy as np
import torch

import paper_1705_06661_gb300 as ss

_T = {"f64": torch.float64, "f32": torch.float32}

# factor chains [F_1, .., F_k], B = F_1(F_2(..F_k(A))): every factor is twice the
# identity minus the permutations listed (one-line notation)
_CHAINS = {
    "row1": (3, [["213"], ["321", "132"]]),
    "row2": (3, [["321", "132"]]),
    "row3": (3, [["213", "132"]]),
    "row5": (4, [["2134"], ["3214", "1324"], ["4231", "1432", "1243"]]),
    "row6": (4, [["3214", "1324"], ["4231", "1432", "1243"]]),
    "row18": (4, [["4231", "1432", "1243"]]),
    "pair": (2, [["21"]]),
}
_CHAINS_OF = {d: sorted(k for k, v in _CHAINS.items() if v[0] == d) for d in (2, 3, 4)}


def _perms(d):
    return list(itertools.permutations(range(d)))


def _coef(name, d):
    """Coefficient chain [nfactors, d!] in lexicographic permutation order."""
    ps = _perms(d)
    if name.startswith("random"):          # one of -2, -1, 1, 2, 4 per permutation
        r = random.Random(int(name[6:]))
        return np.array([[r.choice([-2.0, -1.0, 1.0, 2.0, 4.0]) for _ in ps]])
    rows = []
    for names in _CHAINS[name][1]:
        v = np.zeros(len(ps))
        v[0] = 2.0
        for n in names:
            v[ps.index(tuple(int(c) - 1 for c in n))] -= 1.0
        rows.append(v)
    return np.stack(rows)


def _expand(chain, d):
    """The product of a chain as one coefficient vector."""
    ps = _perms(d)
    at = {p: k for k, p in enumerate(ps)}
    out = chain[0]
    for f in chain[1:]:
        nxt = np.zeros(len(ps))
        for a, p in enumerate(ps):
            for b, q in enumerate(ps):
                nxt[at[tuple(p[q[m]] for m in range(d))]] += out[a] * f[b]
        out = nxt
    return out


def _inverse(p):
    q = [0] * len(p)
    for m, v in enumerate(p):
        q[v] = m
    return tuple(q)


def _sum64(A, coef, d, adjoint=False):
    """sum_sigma a_sigma pi_sigma(A) over the last d dimensions, in FP64."""
    n = A.dim() - d
    out = torch.zeros_like(A, dtype=torch.float64)
    A = A.to(torch.float64)
    for c, p in zip(coef, _perms(d)):
        if c != 0.0:
            q = p if adjoint else _inverse(p)
            out.add_(A.permute(*range(n), *[n + k for k in q]), alpha=float(c))
    return out


def _uniform(shape, dtype, gen, order="F"):
    shape = tuple(shape)
    if order == "F":
        t = torch.rand(shape[::-1], dtype=dtype, device="cuda", generator=gen)
        t = t.permute(*reversed(range(len(shape))))
    else:
        t = torch.rand(shape, dtype=dtype, device="cuda", generator=gen)
    return t.mul_(2.0).sub_(1.0)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _spec(case):
    """The spectator extents, written as in "48x48x48" (none for the paper's layout)."""
    return tuple(int(v) for v in case["spec"].split("x") if v)


def _shape(case):
    return _spec(case) + (case["O"],) * case["d"]


def _blocks(case):
    r = random.Random(case["block_seed"])
    out = []
    for b in range(case["nblocks"]):
        v, o = r.randint(case["vmin"], case["vmax"]), r.randint(case["omin"], case["omax"])
        out.append(((v, v, v, o, o, o), ["row1", "row2", "row3", f"random{200 + b}"][b % 4]))
    return out


def listed():
    return [
        # the smallest call: a CCSDT block of a small molecule, 2 MB, dominated by latency
        dict(name="spin-3d-8", kind="spin", d=3, spec="8x8x8", O=8, dtype="f64", coef="row1", alpha=1.0, beta=0.0,
             inplace=False),
        # the CCSDT amplitude tensor of the benchmark: 48 virtual and 16 occupied orbitals
        dict(name="spin-3d-48x16", kind="spin", d=3, spec="48x48x48", O=16, dtype="f64", coef="row1", alpha=1.0,
             beta=0.0, inplace=False),
        # the CCSDTQ tensor of the benchmark, summed in place (2^-6 keeps repeated calls bounded)
        dict(name="spin-4d-12-inplace", kind="spin", d=4, spec="12x12x12x12", O=12, dtype="f64", coef="row5",
             alpha=0.015625, beta=0.0, inplace=True),
        # single-precision storage, odd extents everywhere, accumulated into a residual
        dict(name="spin-3d-f32-odd", kind="spin", d=3, spec="45x43x41", O=15, dtype="f32", coef="random7", alpha=1.0,
             beta=0.5, inplace=False),
        # the paper's own tensors: every index permuted
        dict(name="paper-3d-544", kind="paper", d=3, spec="", O=544, dtype="f64", coef="row1", alpha=1.0, beta=0.0,
             inplace=False),
        dict(name="paper-3d-271", kind="paper", d=3, spec="", O=271, dtype="f64", coef="row2", alpha=1.0, beta=0.0,
             inplace=False),
        dict(name="paper-4d-112", kind="paper", d=4, spec="", O=112, dtype="f64", coef="row5", alpha=1.0, beta=0.0,
             inplace=False),
        # a tensor as torch allocates it: the permuted indices fastest
        dict(name="rowmajor-3d-32x12", kind="rowmajor", d=3, spec="32x32x32", O=12, dtype="f64", coef="row1",
             alpha=1.0, beta=0.0, inplace=False),
        # the uneven symmetry blocks of one amplitude tensor, planned once and summed every iteration
        dict(name="batch-32", kind="batch", d=3, nblocks=32, block_seed=3, vmin=16, vmax=40, omin=6, omax=14,
             dtype="f64"),
        # a differentiable step: forward and gradient of a CCSDTQ tensor
        dict(name="autograd-4d-10", kind="autograd", d=4, spec="10x10x10x10", O=10, dtype="f64", coef="random105",
             alpha=1.0),
        # the summed amplitudes contracted with 32 columns of a matrix (what the summation feeds)
        dict(name="contract-3d-y32", kind="contract", d=3, spec="48x48x48", O=16, dtype="f64", coef="row1", Y=32),
        # packed antisymmetric storage, both directions
        dict(name="packed-3d-48x16", kind="packed", d=3, spec="48x48x48", O=16, dtype="f64"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _specs(rng, d, O, elements):
    """d spectator extents, uneven, for about `elements` elements in all."""
    v = max(1.0, (elements / O ** d) ** (1.0 / d))
    return [max(2, int(round(v * rng.uniform(0.75, 1.25)))) for _ in range(d)]


def draw(rng):
    kind = rng.choice(["spin", "spin", "paper", "paper", "rowmajor", "batch", "autograd", "contract", "packed"])
    cap = 4.0e8                                     # elements: below the largest listed tensor
    if kind == "batch":
        return dict(kind=kind, d=3, nblocks=_logint(rng, 4, 32), block_seed=rng.randrange(1000), vmin=16,
                    vmax=rng.randint(20, 38), omin=6, omax=rng.randint(8, 13), dtype=rng.choice(["f64", "f32"]))
    if kind == "paper":
        d = rng.choice([2, 3, 3, 4, 4])
        O = {2: (256, 12000), 3: (48, 540), 4: (16, 112)}[d]
        return dict(kind=kind, d=d, spec="", O=_logint(rng, *O), dtype=rng.choice(["f64", "f64", "f32"]),
                    coef=rng.choice(_CHAINS_OF[d] + ["random%d" % rng.randrange(100)]), alpha=1.0,
                    beta=rng.choice([0.0, 0.0, 0.5]), inplace=False)
    d = rng.choice([2, 3, 3, 4]) if kind in ("spin", "contract") else (3 if kind == "packed" else rng.choice([3, 4]))
    O = rng.randint(*{2: (16, 96), 3: (6, 16), 4: (5, 12)}[d])
    dtype = rng.choice(["f64", "f64", "f32"]) if kind in ("spin", "rowmajor") else "f64"
    if kind == "rowmajor":
        cap = 1.0e8
    spec = _specs(rng, d, O, math.exp(rng.uniform(math.log(2.0e5), math.log(cap))))
    while math.prod(spec) * O ** d > 4.5e8:
        spec[rng.randrange(d)] -= 1
    case = dict(kind=kind, d=d, spec="x".join(map(str, spec)), O=O, dtype=dtype)
    if kind != "packed":
        case["coef"] = rng.choice(_CHAINS_OF[d] + ["random%d" % rng.randrange(100)])
    if kind in ("spin", "rowmajor"):
        case.update(alpha=rng.choice([1.0, 1.0, -0.5]), beta=rng.choice([0.0, 0.0, 0.5]), inplace=False)
    if kind == "autograd":
        case["alpha"] = rng.choice([1.0, 0.25])
    if kind == "contract":
        case["Y"] = max(1, min(_logint(rng, 1, 64), int(1.2e10 / (math.prod(spec) * O ** d))))
    return case


def prepare(case, seed):
    g = _gen(seed)
    kind, d, dt = case["kind"], case["d"], _T[case["dtype"]]
    st = dict(case=case, d=d)
    if kind == "batch":
        probs = []
        for shape, name in _blocks(case):
            A = _uniform(shape, dt, g)
            probs.append(dict(A=A, B=ss.colmajor_empty(shape, dtype=dt), coef=_coef(name, 3), d=3, factorized=True))
        st["out"] = [p["B"] for p in probs]
        st["plan"] = ss.Plan(probs)
        return st
    shape = _shape(case)
    if kind == "packed":
        st["P"] = _uniform(shape[:d] + (math.comb(case["O"], d),), dt, g)
        return st
    st["coef"] = _coef(case["coef"], d)
    st["A"] = _uniform(shape, dt, g, "C" if kind == "rowmajor" else "F")
    if kind == "autograd":
        st["A"].requires_grad_(True)
        st["G"] = _uniform(shape, dt, g)
    elif kind == "contract":
        st["W"] = _uniform((case["Y"], case["O"] ** d), dt, g)
    elif not case["inplace"]:
        # the caller's output tensor; with beta it holds the residual that the sum is added to
        st["B"] = _uniform(shape, dt, g, "C" if kind == "rowmajor" else "F")
    return st


def run(state):
    case, d = state["case"], state["d"]
    kind = case["kind"]
    if kind == "batch":
        state["plan"].execute()
        return state["out"]
    if kind == "packed":
        B = ss.unpack(state["P"], d, case["O"])
        return [B, ss.pack(B, d)]
    if kind == "autograd":
        B = ss.spinsum_autograd(state["A"], state["coef"], d=d, alpha=case["alpha"])
        return [B.detach(), torch.autograd.grad(B, state["A"], state["G"])[0]]
    if kind == "contract":
        return ss.contract(state["A"], state["coef"], state["W"], d=d, factorized=True)
    if case["inplace"]:
        return ss.spinsum(state["A"], state["coef"], d=d, factorized=True, alpha=case["alpha"], inplace=True)
    return ss.spinsum(state["A"], state["coef"], d=d, factorized=True, alpha=case["alpha"], beta=case["beta"],
                      out=state["B"])


def work(case):
    kind, d = case["kind"], case["d"]
    es = 8 if case["dtype"] == "f64" else 4
    if kind == "batch":
        bl = _blocks(case)
        n = [math.prod(s) for s, _ in bl]
        return dict(bytes=2 * es * sum(n), flops=sum(2 * k * int(np.count_nonzero(_coef(c, 3))) for k, (_, c) in zip(n, bl)))
    n = math.prod(_shape(case))
    S, O = math.prod(_spec(case)), case["O"]
    if kind == "packed":
        p = S * math.comb(O, d)
        return dict(bytes=es * ((p + n) + 2 * p), flops=0)     # unpack reads P, writes B; pack reads and writes p
    terms = 2 * int(np.count_nonzero(_coef(case["coef"], d)))
    if kind == "contract":
        Y = case["Y"]
        return dict(bytes=es * (n + Y * O ** d + S * Y), flops=n * terms + 2 * n * Y)
    if kind == "autograd":
        return dict(bytes=4 * es * n, flops=2 * n * terms)
    return dict(bytes=es * n * (3 if case["beta"] else 2), flops=n * terms)


def exact(case, seed):
    st = prepare(case, seed) if case["kind"] != "batch" else None
    kind, d = case["kind"], case["d"]
    if kind == "batch":
        g = _gen(seed)
        return [_sum64(_uniform(shape, _T[case["dtype"]], g), _expand(_coef(name, 3), 3), 3)
                for shape, name in _blocks(case)]
    if kind == "packed":
        P, O = st["P"].to(torch.float64), case["O"]
        B = torch.zeros(_shape(case)[::-1], dtype=torch.float64, device="cuda")
        B = B.permute(*reversed(range(2 * d)))
        idx = sorted(itertools.combinations(range(O), d), key=lambda t: t[::-1])
        ix = torch.tensor(idx, device="cuda")
        for p in _perms(d):
            sign = round(np.linalg.det(np.eye(d)[list(p)]))
            B[(Ellipsis,) + tuple(ix[:, k] for k in p)] = sign * P
        return [B, P]
    co = _expand(_coef(case["coef"], d), d)
    A = st["A"].detach()
    if kind == "autograd":
        return [_sum64(A, co, d) * case["alpha"], _sum64(st["G"], co, d, adjoint=True) * case["alpha"]]
    if kind == "contract":
        S, T = math.prod(_spec(case)), case["O"] ** d
        X = _sum64(A, co, d)
        X = X.permute(*reversed(range(2 * d))).reshape(T, S)              # [t, s], s fastest
        C = st["W"].to(torch.float64) @ X                                  # [y, s]
        return C.reshape((case["Y"],) + _spec(case)[::-1]).permute(*reversed(range(d + 1)))
    out = _sum64(A, co, d) * case["alpha"]
    if case["beta"]:
        out = out + case["beta"] * st["B"].to(torch.float64)
    return out
