"""The test that keeps every particle's stencil within the grid, compiled for the
host from the kernels' header: a particle far outside has a base cell at the end
of the 32-bit range (the conversion saturates), where adding the stencil's width
would wrap round and count it as inside. Compared with Python's integers."""
import ctypes as C
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2503_05046_gb300", "csrc", "common.cuh")
LO, HI = -2 ** 31, 2 ** 31 - 1


def function(text, name):
    at = text.index("__device__ __forceinline__", text.rindex("\n", 0, re.search(r"\b%s\(" % name, text).start()))
    depth, i = 0, text.index("{", at)
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            return text[at:i]


@pytest.fixture(scope="module")
def inside(tmp_path_factory):
    with open(HEADER) as f:
        text = f.read()
    d = tmp_path_factory.mktemp("stencil")
    src, lib = str(d / "s.cc"), str(d / "s.so")
    with open(src, "w") as f:
        f.write("#define __device__\n#define __forceinline__ static inline\n"
                "struct GridDev { int rx, ry, rz; };\nstruct Stencil { int base[3]; };\n" +
                function(text, "stencil_inside") +
                '\nextern "C" int inside(int bx, int by, int bz, int rx, int ry, int rz) {\n'
                "  GridDev g{rx, ry, rz};\n  Stencil s{{bx, by, bz}};\n  return stencil_inside(g, s);\n}\n")
    subprocess.run(["g++", "-O1", "-fwrapv", "-shared", "-fPIC", src, "-o", lib], check=True)
    return C.CDLL(lib).inside


@pytest.mark.parametrize("res", [(4, 8, 64), (320, 184, 64), (4096, 4, 4)])
def test_only_stencils_within_the_grid_count_as_inside(inside, res):
    for a in range(3):
        for b in (LO, LO + 1, -2 ** 30, -3, -1, 0, 1, res[a] - 4, res[a] - 3, res[a] - 2, res[a] - 1, res[a],
                  2 ** 30, HI - 3, HI - 2, HI - 1, HI):
            base = [0, 0, 0]
            base[a] = b
            want = all(0 <= c and c + 2 < r for c, r in zip(base, res))
            assert bool(inside(*base, *res)) == want, (base, res)


def test_base_cell_is_converted_after_its_correction():
    """The float's conversion saturates; an integer step after it would not."""
    with open(HEADER) as f:
        body = function(f.read(), "cell_coord")
    code = re.sub(r"//[^\n]*", "", body)
    assert code.rstrip().rstrip("}").rstrip().endswith("base = (int)b;")
    assert "base +=" not in code and "base -=" not in code
