"""The particle sort at the edges of its launch shapes: one particle, less and
more than a warp, one round and more of the one-block sort (1,024), its last
size and the first of the tiled sort (8,192, 8,193), the last size of the short
tiles and the first of the long ones (524,288, 524,289), in domains of one to
four passes (an elongated one has axes of different bit counts), and a batch of
uneven members, one of them of another domain. A step of no substeps sorts and
nothing else: the state read back in id order keeps every bit."""
import numpy as np
import pytest

from paper_2503_05046_gb300 import scenes

pytestmark = pytest.mark.gpu


def scattered(n, res, seed=0):
    """n particles all over a domain, and beyond its faces on every side"""
    sc = scenes.sand_random(64, 4.0, penetration=-0.02)
    sc["grid"] = dict(sc["grid"], res=res)
    rng = np.random.default_rng(seed)
    dx, o = sc["grid"]["dx"], np.asarray(sc["grid"]["origin"], np.float64)
    x = rng.uniform(o - 3 * dx, o + (np.asarray(res) + 3) * dx, (n, 3)).astype(np.float32)
    sc["groups"] = [dict(sc["groups"][0], x=x, v=rng.standard_normal((n, 3)).astype(np.float32))]
    return sc


def give_state(sim, n, seed=1):
    st = sim.get_particles()
    rng = np.random.default_rng(seed)
    st["C"] = rng.standard_normal((n, 3, 3)).astype(np.float32)
    st["F"] = (np.eye(3) + 0.01 * rng.standard_normal((n, 3, 3))).astype(np.float32)
    sim.set_particles(st["x"], st["v"], st["C"], st["F"])
    return st


@pytest.mark.parametrize("res", [(8, 8, 8), (64, 64, 64), (320, 16, 64)])
@pytest.mark.parametrize("n", [1, 31, 1024, 1025, 8192, 8193, 524288, 524289])
def test_sort_keeps_every_particle(n, res):
    from paper_2503_05046_gb300 import native
    sc = scattered(n, res)
    sim = native.Sim(sc)
    try:
        want = give_state(sim, n)
        for _ in range(2):  # both particle buffers
            sim.step(n_substeps=0)
            got = sim.get_particles()
            for key in want:
                assert np.array_equal(want[key], got[key]), key
    finally:
        sim.close()


def test_batched_sort_keeps_every_particle():
    from paper_2503_05046_gb300 import native
    sizes = (1, 8192, 33, 20_000, 1024)
    res = ((64, 64, 64), (8, 8, 8), (64, 64, 64), (320, 16, 64), (64, 64, 64))
    batch = native.Batch([scattered(n, r, seed=n) for n, r in zip(sizes, res)])
    try:
        want = [give_state(sim, n) for sim, n in zip(batch.sims, sizes)]
        for _ in range(2):
            batch.sort()
            for sim, w in zip(batch.sims, want):
                got = sim.get_particles()
                for key in w:
                    assert np.array_equal(w[key], got[key]), key
    finally:
        batch.close()


@pytest.mark.parametrize("n", [1, 31, 33, 257, 1000])
@pytest.mark.parametrize("field", ["x", "v", "C", "F"])
def test_one_field_set_and_read_in_id_order(n, field):
    """Records of three and nine floats at the edges of a warp and of a block,
    in an order that is not the ids': one field set, the others as they were,
    and read with the others left out."""
    from paper_2503_05046_gb300 import native
    sim = native.Sim(scattered(n, (64, 64, 64)))
    try:
        want = give_state(sim, n)
        sim.step(n_substeps=0)
        want[field] = want[field] + np.float32(0.25)
        native.mpm_set_particles(sim.ctx, **{{"C": "Cm"}.get(field, field): want[field]})
        got = sim.get_particles()
        for key in want:
            assert np.array_equal(want[key], got[key]), key
        one = np.empty_like(want[field])
        native.mpm_get_particles(sim.ctx, **{{"C": "Cm"}.get(field, field): one})
        assert np.array_equal(one, want[field])
    finally:
        sim.close()
