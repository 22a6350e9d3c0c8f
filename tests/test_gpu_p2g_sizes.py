"""P2G at the edges of its launch shapes: one particle, less and more than a
warp's set of 32 and than its three sets of 96, the size from which a warp
takes three sets, dense and block-sparse, each in cell order and in an order
that has nothing to do with the cells any more (the step's sort is as old as
the step). The particles carry no stress (F = I), so a node's v* - h g is the
weighted mean of v + C (x_i - x_p): in FP32 a sum of N terms, each with about
six roundings, is within (N + 6) 6e-8 of the largest term, 1e-5 at the 150
particles that the fullest stencil here sees; masses alike, plus 1e-6 of a
particle's for the absolute error of small weights."""
import numpy as np
import pytest

import oracle as O
from paper_2503_05046_gb300 import scenes
from gpu_helpers import align_grids, oracle_substep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("stale", [False, True])
@pytest.mark.parametrize("n,ppc", [(1, 1.0), (31, 4.0), (33, 1.0), (97, 4.0), (1_000, 0.5), (160_001, 4.0)])
def test_p2g_sizes(n, ppc, stale, sparse):
    from paper_2503_05046_gb300 import native
    sc = scenes.sand_random(n, ppc, penetration=-0.02)  # two cells above the ground: no contact
    if sparse:
        sc["grid"] = dict(sc["grid"], max_blocks=int(np.prod([r // 4 for r in sc["grid"]["res"]])) - 1)
    rng = np.random.default_rng(5)
    sim = native.Sim(sc)
    try:
        solver = native.solver_params()
        st = sim.get_particles()
        if stale:  # sorted once; every particle then takes another one's place
            native.mpm_set_option(sim.ctx, native.OPT_SORT_EVERY, 1000)
            sim.step(n_substeps=1, solver=solver)
            st["x"] = st["x"][rng.permutation(n)]
        st["v"] = rng.uniform(-0.1, 0.1, (n, 3)).astype(np.float32)
        st["C"] = rng.uniform(-5.0, 5.0, (n, 3, 3)).astype(np.float32)
        st["F"] = np.tile(np.eye(3, dtype=np.float32), (n, 1, 1))
        sim.set_particles(st["x"], st["v"], st["C"], st["F"])
        _, _, osim, _, code = oracle_substep(sc, st, sim.bodies(), O.solver())
        assert code == O.OK
        sim.step(n_substeps=1, solver=solver)
        mass_p = np.float32(sc["groups"][0]["vol"]) * np.float32(scenes.SAND["rho"])
        (m, vs, _), (om, ovs, _) = align_grids(sim.grid(), osim.last_grid(), 1e-6 * mass_p)
        assert np.all(np.abs(m - om) <= 1e-5 * om + 1e-6 * mass_p)
        term = 0.1 + 5.0 * 1.5 * sc["grid"]["dx"] * 3 + 9.81 * sc["h"]
        held = om >= 1e-2 * mass_p
        assert np.max(np.abs(vs[held] - ovs[held]), initial=0.0) <= 1e-5 * term
    finally:
        sim.close()
