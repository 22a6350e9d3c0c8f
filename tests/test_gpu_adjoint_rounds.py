"""The contact-solve adjoint at the edges of its launches against the oracle's,
as test_gpu_adjoint does: a single contact, one block's last count and the first
over a cluster (16, 17), the cluster's last count and the first of the
cooperative launch (100 of at most 100 and 99), more contacts than a small
cluster has warps, and the cooperative launch asked for."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import contact_problem
from test_gpu_adjoint import TIGHT, _oracle_with_floor
from test_gpu_solve_small import slab

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("contacts,cluster,blocks", [
    (1, 1024, 0), (16, 1024, 0), (17, 1024, 0), (100, 100, 0), (100, 99, 0), (100, 1024, 2), (100, 0, 0)])
def test_adjoint_routes(contacts, cluster, blocks):
    from paper_2503_05046_gb300 import native
    sc = slab(contacts)
    sim = native.Sim(sc)
    try:
        native.mpm_set_option(sim.ctx, native.OPT_CLUSTER_CONTACTS, cluster)
        native.mpm_set_option(sim.ctx, native.OPT_CLUSTER_BLOCKS, blocks)
        solver = native.solver_params(**TIGHT)
        st0, bodies = sim.get_particles(), sim.bodies()
        stats = sim.step(n_substeps=1, solver=solver)
        assert stats.contacts_max == contacts and stats.residual_max <= 1e-4
        grid, found = sim.grid(), sim.contacts()
        ids, _, _, v = grid
        prob, R, _ = contact_problem(sc, st0, bodies, grid, found, solver.eps_s, lagged_from_gpu=True)
        vbar = np.random.default_rng(7).normal(size=v.shape).astype(np.float32)
        refs, floors = _oracle_with_floor(prob, R, v.astype(np.float64), vbar.astype(np.float64))
        assert refs[3] == O.OK
        vsb, cbar, _, ast, code = sim.contact_adjoint(ids, vbar, eps_r=1e-6, max_iters=5000)
        assert code == native.OK and ast.residual <= 1e-6 and ast.contacts == contacts
        for name, got, ref, f in zip(("dL/dv*", "dL/dv_r", "dL/dmu"), (vsb, cbar[:, :3], cbar[:, 3]), refs, floors):
            err, scale = np.abs(got - ref), np.max(np.abs(ref))
            assert np.all(err <= 1e-4 * scale + 2.0 * f), "%s max err %.3e of %.3e" % (name, err.max(), scale)
    finally:
        sim.close()
