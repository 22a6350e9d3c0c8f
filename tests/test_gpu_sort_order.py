"""The order that the particle sort leaves, read through the contact list: with
every particle inside one (very soft) half-space, each 32 neighbouring slots
register their 32 contacts side by side, in slot order. The list, put together
from those pieces, has to be the stable sort of the ids by a key computed here:
the bits of the block's Morton code that its axis has, then the cell within the
block. Domains of one to four passes, at the sizes where the launches change;
and a batch of uneven members of different domains."""
import numpy as np
import pytest

from paper_2503_05046_gb300 import scenes

pytestmark = pytest.mark.gpu


def sort_keys(x, grid):
    """(keys, bits)"""
    res = np.asarray(grid["res"])
    base = np.floor((x.astype(np.float64) - np.asarray(grid["origin"])) / grid["dx"] - 0.5).astype(np.int64)
    block, cell, top = base >> 2, base & 3, res // 4 - 1
    key, pos = np.zeros(len(x), np.int64), 0
    for bit in range(12):
        for a in range(3):
            if top[a] >> bit:
                key |= ((block[:, a] >> bit) & 1) << pos
                pos += 1
    if pos + 6 <= 32:
        key, pos = (key << 6) | (cell[:, 2] << 4) | (cell[:, 1] << 2) | cell[:, 0], pos + 6
    return key, pos


def scattered(n, res, seed=0):
    """n particles in the domain, none near a cell's face, a third of them in a
    few cells (equal keys)."""
    sc = scenes.sand_random(64, 4.0)
    sc["grid"] = dict(sc["grid"], res=res)
    if res[0] * res[1] * res[2] > 1 << 24:
        sc["grid"]["max_blocks"] = 8 * n + 1
    rng = np.random.default_rng(seed)
    base = np.stack([rng.integers(0, r - 2, n) for r in res], 1)
    few = rng.random(n) < 1 / 3
    base[few] = base[rng.integers(0, max(n // 500, 1), int(few.sum()))]
    dx, o = sc["grid"]["dx"], np.asarray(sc["grid"]["origin"], np.float64)
    x = (o + (base + 0.5 + rng.uniform(0.1, 0.9, (n, 3))) * dx).astype(np.float32)
    sc["groups"] = [dict(sc["groups"][0], x=x, v=np.zeros((n, 3), np.float32))]
    sc["bodies"] = [scenes.body(scenes.HALFSPACE, p=(0.0, 0.0, 50.0), k=1e-9, d=0.0)]
    return sc


def check_order(ids, sc):
    x = sc["groups"][0]["x"]
    n = len(x)
    assert len(ids) == n and np.array_equal(np.sort(ids), np.arange(n))
    key, bits = sort_keys(x, sc["grid"])
    want = np.argsort(key, kind="stable")
    pieces, place = [], np.empty(n, np.int64)
    place[want] = np.arange(n)
    at = 0
    while at < n:  # a piece: 32 ids, or the last one's n % 32
        short = n % 32 and place[ids[at]] // 32 == n // 32
        size = n % 32 if short else 32
        pieces.append(ids[at:at + size])
        at += size
    pieces.sort(key=lambda p: place[p[0]])
    assert np.array_equal(np.concatenate(pieces), want)
    return bits


@pytest.mark.parametrize("res,passes", [((4, 4, 8), 1), ((8, 8, 8), 2), ((64, 64, 64), 3), ((320, 16, 64), 3),
                                        ((1024, 512, 64), 4)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 1025, 8192, 8193, 70_001])
def test_sort_order(n, res, passes):
    from paper_2503_05046_gb300 import native
    sc = scattered(n, res, seed=n)
    sim = native.Sim(sc)
    try:
        sim.step(n_substeps=1, solver=native.solver_params(max_iters=1), check=False)
        bits = check_order(sim.contacts()[0], sc)
        assert -(-bits // 8) == passes
    finally:
        sim.close()


@pytest.mark.parametrize("n", [524_288, 524_289])
def test_sort_order_of_long_tiles(n):
    from paper_2503_05046_gb300 import native
    sc = scattered(n, (64, 64, 64))
    sim = native.Sim(sc, max_contacts=n)
    try:
        sim.step(n_substeps=1, solver=native.solver_params(max_iters=1), check=False)
        check_order(sim.contacts()[0], sc)
    finally:
        sim.close()


def test_batched_sort_order():
    from paper_2503_05046_gb300 import native
    sizes = (1, 8192, 33, 20_000, 1024)
    res = ((64, 64, 64), (4, 4, 8), (64, 64, 64), (320, 16, 64), (8, 8, 8))
    scs = [scattered(n, r, seed=n) for n, r in zip(sizes, res)]
    batch = native.Batch(scs)
    try:
        batch.sort()
        batch.step(scs[0]["h"], 1, native.solver_params(max_iters=1))
        batch.synchronize(stats=False)
        for sim, sc in zip(batch.sims, scs):
            check_order(sim.contacts()[0], sc)
    finally:
        batch.close()
