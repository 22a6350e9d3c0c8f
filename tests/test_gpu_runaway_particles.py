"""Particles far outside the grid, up to the ends of FP32 and at infinity: they are
reported and left alone, and the others move as if alone. Positions over 2^31
cells away are those whose base cell saturates. Tolerance for the others: four
substeps' node sums of some 64 terms in another order, 4 x 64 x 6e-8 of the
largest velocity (the material is soft: its stress's rounding is far below)."""
import numpy as np
import pytest

from paper_2503_05046_gb300 import scenes

pytestmark = pytest.mark.gpu
FAR = (3e34, -3e34, np.inf, -np.inf, 2.2e7, -2.2e7, 1e4)


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("n", [64, 9000])
def test_far_particles_are_reported_and_left_alone(n, sparse):
    from paper_2503_05046_gb300 import native
    sc = scenes.sand_random(n, 4.0, penetration=-0.02)
    if sparse:
        sc["grid"] = dict(sc["grid"], max_blocks=int(np.prod(np.asarray(sc["grid"]["res"]) // 4)) - 1)
    sc["groups"] = [dict(sc["groups"][0], material=scenes.elastic(1e4, 0.3, 1000.0))]
    m = len(sc["groups"][0]["x"])
    far = np.arange(3 * len(FAR)) * (m // (3 * len(FAR)))
    x = sc["groups"][0]["x"].copy()
    for k, i in enumerate(far):
        x[i, k % 3] = FAR[k // 3]
    near = np.setdiff1d(np.arange(m), far)
    one = dict(sc, groups=[dict(sc["groups"][0], x=sc["groups"][0]["x"][near], v=sc["groups"][0]["v"][near])])
    sim, alone = native.Sim(sc), native.Sim(one)
    try:
        st = sim.get_particles()
        sim.set_particles(x, st["v"], st["C"], st["F"])
        for _ in range(2):
            code, _ = sim.step(n_substeps=2, check=False)
            assert code == native.ERR_OUT_OF_DOMAIN
            alone.step(n_substeps=2)
        got, want = sim.get_particles(), alone.get_particles()
        assert np.array_equal(got["x"][far], x[far]) and np.array_equal(got["v"][far], st["v"][far])
        for key in ("x", "v"):
            err = np.max(np.abs(got[key][near] - want[key]))
            assert err <= 1.6e-5 * np.max(np.abs(want[key])), (key, err)
    finally:
        sim.close()
        alone.close()
