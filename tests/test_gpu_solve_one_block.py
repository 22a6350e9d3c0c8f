"""Which contact solves run in one thread block's shared memory: up to 320
contacts whose nodes fit, not one more, and none where the option excludes the
cluster; the two counts agree with the route in a batch as well."""
import ctypes as C

import numpy as np
import pytest

from paper_2503_05046_gb300 import scenes
from test_gpu_solve_small import slab

pytestmark = pytest.mark.gpu


def spread(side):
    """side x side contacts three cells apart: 27 nodes each"""
    sc = scenes.sand_slab(side, side, 1)
    sc["groups"][0]["x"][:, :2] *= np.float32(6.0)
    sc["bodies"] = sc["bodies"][:1]
    res = 4 * int(np.ceil((6.0 * side * 0.5 + 16) / 4))
    sc["grid"] = dict(sc["grid"], res=(res, res, sc["grid"]["res"][2]), origin=(-res * 0.005, -res * 0.005, -0.08))
    return sc


def routes(sim, contacts, **options):
    from paper_2503_05046_gb300 import native
    for name, value in options.items():
        native.mpm_set_option(sim.ctx, getattr(native, name), value)
    stats = sim.step(n_substeps=1)
    assert stats.contacts_max == contacts
    return native.mpm_get_one_block_solves(sim.ctx), stats.cluster_substeps


@pytest.mark.parametrize("contacts,one_block", [(1, 1), (32, 1), (319, 1), (320, 1), (321, 0), (512, 0)])
def test_by_contact_count(contacts, one_block):
    from paper_2503_05046_gb300 import native
    sim = native.Sim(slab(contacts))
    try:
        assert routes(sim, contacts) == (one_block, 1)
    finally:
        sim.close()


@pytest.mark.parametrize("side,one_block", [(8, 1), (14, 0)])
def test_by_nodes(side, one_block):
    """64 contacts have 1,728 nodes of their own; 196 have 5,292, over the table's 4,096"""
    from paper_2503_05046_gb300 import native
    sim = native.Sim(spread(side))
    try:
        assert routes(sim, side * side) == (one_block, 1)
    finally:
        sim.close()


def test_by_option():
    from paper_2503_05046_gb300 import native
    sim = native.Sim(slab(100))
    try:
        assert routes(sim, 100, OPT_CLUSTER_CONTACTS=0) == (0, 0)
    finally:
        sim.close()
    sim = native.Sim(slab(100))
    try:
        assert routes(sim, 100, OPT_CLUSTER_CONTACTS=99) == (0, 0)
    finally:
        sim.close()


def test_in_a_batch():
    from paper_2503_05046_gb300 import native
    counts = (1, 320, 321)
    batch = native.Batch([slab(c) for c in counts])
    try:
        batch.step(1e-4, 1, native.solver_params())
        _, _, stats = batch.synchronize()
        assert tuple(s["contacts_max"] for s in stats) == counts
        assert [native.mpm_get_one_block_solves(s.ctx) for s in batch.sims] == [1, 1, 0]
    finally:
        batch.close()


def test_arguments():
    from paper_2503_05046_gb300 import native
    n = C.c_int32()
    assert native.lib.mpm_get_one_block_solves(None, C.byref(n)) == native.ERR_INVALID_ARG
