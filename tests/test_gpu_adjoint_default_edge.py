"""The contact-solve adjoint on both sides of the count from which it is a
cooperative launch by default (512 contacts by one cluster, 513 not), against the
oracle's. The cotangents are a velocity's, as the adjoint of the transfers gives
them: a node's in proportion to its mass. (The iteration stops by the residual in
the inverse preconditioner's norm, in which a cotangent of one on a node of a
billionth of the others' mass outweighs all of them.) Tolerance: the oracle's own
change under FP32 rounding of the problem, and 1e-4 of the largest: eps_r = 1e-6
times the square root of some 4,000 nodes."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import contact_problem
from test_gpu_adjoint import TIGHT, _oracle_with_floor
from test_gpu_solve_small import slab

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("contacts", [512, 513])
def test_adjoint_at_the_default_edge(contacts):
    from paper_2503_05046_gb300 import native
    sc = slab(contacts)
    sim = native.Sim(sc)
    try:
        solver = native.solver_params(**TIGHT)
        st0, bodies = sim.get_particles(), sim.bodies()
        stats = sim.step(n_substeps=1, solver=solver)
        assert stats.contacts_max == contacts and stats.residual_max <= 1e-4
        grid, found = sim.grid(), sim.contacts()
        ids, m, _, v = grid
        prob, R, _ = contact_problem(sc, st0, bodies, grid, found, solver.eps_s, lagged_from_gpu=True)
        vbar = (np.random.default_rng(7).normal(size=v.shape) * (m / np.max(m))[:, None]).astype(np.float32)
        refs, floors = _oracle_with_floor(prob, R, v.astype(np.float64), vbar.astype(np.float64), patterns=2)
        assert refs[3] == O.OK
        vsb, cbar, _, ast, code = sim.contact_adjoint(ids, vbar, eps_r=1e-6, max_iters=5000)
        assert code == native.OK and ast.residual <= 1e-6 and ast.contacts == contacts
        for name, got, ref, f in zip(("dL/dv*", "dL/dv_r", "dL/dmu"), (vsb, cbar[:, :3], cbar[:, 3]), refs, floors):
            err, scale = np.abs(got - ref), np.max(np.abs(ref))
            assert np.all(err <= 1e-4 * scale + 2.0 * f), "%s max err %.3e of %.3e" % (name, err.max(), scale)
    finally:
        sim.close()
