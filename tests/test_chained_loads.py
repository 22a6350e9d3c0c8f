"""Kernels of the launch chain (set up while the kernel before them still runs)
read what earlier kernels write only after their first statement, the wait, and
only by ordinary loads: a load through the read-only path (__ldg, or what the
compiler makes of a const __restrict__ parameter) is defined only for data that
no one writes during the whole life of the kernel, and that begins before the
wait. Checked on the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_05046_gb300", "csrc")
FILES = sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu")))

# const __restrict__ parameters of chained kernels that only the host writes,
# ahead of the chain: argument records and work lists, the mesh, materials, pins
HOST_WRITTEN = {"args", "work", "order", "tris", "rest", "groups", "pinned", "ids", "v_pin"}


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernels(text):
    """(name, parameters, body) of each __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, start = text[m.end():i - 1], text.index("{", i)
        depth, i = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), params, text[start + 1:i - 1]


def _chained(text):
    return [k for k in _kernels(text) if "chain_begin()" in k[2]]


def test_the_chain_is_found():
    names = {k[0] for f in FILES for k in _chained(_source(f))}
    assert {"k_p2g_w", "k_grid_update_dense", "k_solve_small", "k_solve", "k_g2p", "k_permute"} <= names


@pytest.mark.parametrize("name", FILES)
def test_chained_kernels_wait_first(name):
    text = _source(name)
    chained = {k[0]: k[2] for k in _chained(text)}
    for kernel in re.findall(r"launch_chained\(\s*(\w+)", text):
        assert kernel in chained, "%s is launched into the chain and does not wait" % kernel
    for kernel, body in chained.items():
        before = body[:body.index("chain_begin()")]
        rest = re.sub(r"__shared__[^;]*;", "", before).strip()
        assert rest == "", "%s: a statement before the wait: %s" % (kernel, rest)


@pytest.mark.parametrize("name", FILES)
def test_chained_kernels_read_no_other_kernels_output_through_the_read_only_path(name):
    text = _source(name)
    for kernel, params, _ in _chained(text):
        for p in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", params):
            assert p in HOST_WRITTEN, "%s reads %s through a const __restrict__ parameter" % (kernel, p)
    # the bodies are device functions that several kernels share; backward.cu's
    # readers of the grid are ordinary launches, which start when the chain is done
    if name != "backward.cu" and _chained(text):
        assert "__ldg(" not in text, "%s: a chained kernel may take this load before the wait" % name
