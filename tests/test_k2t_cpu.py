"""Exhaustive CPU check of the TMA-fed tiled kernel's lane map: the bodies of
`K2TShape<d>::elem` are read from the kernel source (integer expressions whose
operator precedence is the same in C++ and Python). Tiles lie unswizzled in
shared memory, so a double at in-tile offset c falls on bank pair
(sum_k c_k BL^k) mod 16. Checked for every d: elem is a bijection of the
element indices onto the tile, and for all d! permutations the 16 lanes of every
half warp fall on 16 different bank pairs."""
import itertools
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1705_06661_gb300", "csrc", "ss_k2t.cuh")


def _shape(d):
    text = open(SRC).read()
    i = text.index(f"struct K2TShape<{d}> {{")
    block = text[i:text.index("\n};", i)]
    bl, nt = map(int, re.search(r"static constexpr int BL = (\d+), NT = (\d+);", block).groups())
    head = "elem(int e, int (&w)[4]) {"
    j = block.index(head) + len(head)
    code = []
    for st in block[j:block.index("\n  }", j)].split(";"):
        st = re.sub(r"//[^\n]*", "", st).strip()
        if st.startswith("const int "):
            code.extend(p.strip() for p in st[len("const int "):].split(","))
        elif st:
            code.append(st)
    code = "\n".join(code)

    def elem(e):
        env = {"e": e, "w": [0, 0, 0, 0]}
        exec(code, {}, env)
        return env["w"][:d]

    return bl, nt, elem


@pytest.mark.parametrize("d", [3, 4])
def test_lane_map(d):
    bl, nt, elem = _shape(d)
    offs = [elem(e) for e in range(nt)]
    assert sorted(map(tuple, offs)) == sorted(itertools.product(range(bl), repeat=d))
    for tau in itertools.permutations(range(d)):
        for h in range(0, nt, 16):
            banks = {sum(w[tau[k]] * bl ** k for k in range(d)) % 16 for w in offs[h:h + 16]}
            assert len(banks) == 16, (d, tau, h)


@pytest.mark.parametrize("d,flip", [(3, {8: (2, 4)})])
def test_second_pass_flips_one_bit(d, flip):
    """The kernel derives the offsets of its second pass (element index bit 8)
    from the first pass's by flipping one bit of one coordinate."""
    _, nt, elem = _shape(d)
    for e in range(nt):
        w = elem(e & 255)
        for bit, (k, m) in flip.items():
            if e >> bit & 1:
                w[k] ^= m
        assert w == elem(e)
