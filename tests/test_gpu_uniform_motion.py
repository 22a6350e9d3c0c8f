"""A body that moves as one, with a velocity whose components are powers of two,
keeps it bit for bit: a node's momentum is then its mass times the velocity,
whatever the order of its sums (scaling by a power of two commutes with every
rounding), the grid update divides with one rounding, and G2P gathers differences
that are all zero, so v stays and C is zero. Sums of w v_i round at the scale of
the velocity instead, and their C is some 1e-7 |v| 4 / dx. Tolerance: none."""
import numpy as np
import pytest

from paper_2503_05046_gb300 import scenes

pytestmark = pytest.mark.gpu
V = (0.5, -1.0, 2.0)


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("n", [1, 33, 1000, 30_000, 200_000])
def test_uniform_motion_is_kept(n, sparse):
    from paper_2503_05046_gb300 import native
    rng = np.random.default_rng(n)
    dx, side = 0.01, max(n / 4.0, 1.0) ** (1 / 3) * 0.01  # four particles per cell, at random
    x = rng.uniform(-side / 2, side / 2, (n, 3)).astype(np.float32)
    res = 4 * int(np.ceil((side / dx + 16) / 4))
    g = {"x": x, "v": np.tile(np.asarray(V, np.float32), (n, 1)), "vol": dx ** 3 / 4,
         "material": scenes.elastic(1e5, 0.3, 1000.0)}
    grid = {"dx": dx, "res": (res,) * 3, "origin": (-res * dx / 2,) * 3, "gravity": (0.0, 0.0, 0.0), "bc_layers": 3}
    if sparse:
        grid["max_blocks"] = (res // 4) ** 3 - 1
    sc = {"name": "uniform", "grid": grid, "groups": [g], "bodies": [], "h": 1e-4, "substeps": 4}
    sim = native.Sim(sc)
    try:
        for _ in range(3):
            sim.step()
        st = sim.get_particles()
        assert np.array_equal(st["v"], g["v"])
        assert not np.any(st["C"])
        assert np.array_equal(st["F"], np.tile(np.eye(3, dtype=np.float32), (n, 1, 1)))
    finally:
        sim.close()


def test_velocity_beyond_range_leaves_the_domain():
    """A particle whose momentum overflows leaves the domain and is reported: its
    velocity is infinite, not a NaN (whose cell is 0)."""
    from paper_2503_05046_gb300 import native
    x = np.zeros((1, 3), np.float32)
    g = {"x": x, "v": np.asarray([[3e38, 0.0, 0.0]], np.float32), "vol": 1.0, "material": scenes.elastic(1e5, 0.3, 1e6)}
    sc = {"name": "beyond", "grid": {"dx": 0.01, "res": (32,) * 3, "origin": (-0.16,) * 3, "gravity": (0.0, 0.0, 0.0),
                                     "bc_layers": 3}, "groups": [g], "bodies": [], "h": 1e-4, "substeps": 1}
    sim = native.Sim(sc)
    try:
        sim.step(check=False)
        code, _ = sim.step(check=False)
        assert code == native.ERR_OUT_OF_DOMAIN
        assert sim.get_particles()["v"][0, 0] == np.inf
    finally:
        sim.close()
