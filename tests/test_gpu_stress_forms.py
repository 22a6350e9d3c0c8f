"""The stress of a deformation gradient on both sides of the strain up to which
it is a polynomial of F^T F - I (|M| = 1/4), at tiny strains, under a rotation
and for a reflection, for both materials: particles far from each other, so
that a node's v* is one particle's stress, for a given F (set from outside) and
for the F of a substep before (stress stored by G2P).

Tolerance: M is formed from FP32 differences to 6e-8 of its largest terms
(F - I: up to 2 under a rotation, the strain without one), so the stress is
within (lam + 2 mu) 1e-6 absolutely; one substep turns a stress s into at most
h 4 / dx^2 (V / m) s 1.5 dx of velocity, and the sums add 1e-6 of the largest."""
import numpy as np
import pytest

import oracle as O
from paper_2503_05046_gb300 import scenes
from gpu_helpers import oracle_substep

pytestmark = pytest.mark.gpu


def deformations(rng, n):
    """n gradients R (I + X): |M| from 1e-6 to 0.6, dense around 1/4."""
    F = np.zeros((n, 3, 3))
    for i in range(n):
        X = rng.standard_normal((3, 3))
        X = (X + X.T) / np.linalg.norm(X + X.T)
        s = (10.0 ** rng.uniform(-6, -1), 0.125 * rng.uniform(0.9, 1.1), rng.uniform(0.1, 0.3))[i % 3]
        Q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
        if np.linalg.det(Q) < 0 and i % 7:
            Q[:, 0] *= -1  # (one in seven may stay a reflection)
        F[i] = (Q if i % 2 else np.eye(3)) @ (np.eye(3) + s * X)
    return F.astype(np.float32)


@pytest.mark.parametrize("sand", [False, True])
def test_stress_forms(sand):
    from paper_2503_05046_gb300 import native
    side, dx = 8, 0.01
    n = side ** 3
    rng = np.random.default_rng(3)
    mat = dict(scenes.SAND) if sand else scenes.elastic(1e5, 0.3, 1000.0)
    g = scenes.cube_group(side, 4 * dx, (0.0, 0.0, 0.0), (0.0, 0.0, 0.0), mat, jitter=0.3 * dx, rng=rng)
    g["vol"] = (dx / 2) ** 3
    res = 4 * (side + 4)
    sc = {"name": "apart", "grid": {"dx": dx, "res": (res, res, res), "origin": (-res * dx / 2,) * 3,
                                    "gravity": (0.0, 0.0, 0.0), "bc_layers": 3},
          "groups": [g], "bodies": [], "h": 1e-5, "substeps": 1}
    sim = native.Sim(sc)
    try:
        F = deformations(rng, n)
        sim.set_particles(F=F)
        lame = mat["E"] * mat["nu"] / ((1 + mat["nu"]) * (1 - 2 * mat["nu"])) + mat["E"] / (1 + mat["nu"])
        per_stress = sc["h"] * 4 / dx ** 2 / mat["rho"] * 1.5 * dx
        for _ in range(2):
            st = sim.get_particles()
            _, _, osim, _, code = oracle_substep(sc, st, [], O.solver())
            assert code == O.OK
            sim.step(n_substeps=1, solver=native.solver_params())
            ids, m, vs, _ = sim.grid()
            oids, om, ovs, _ = osim.last_grid()
            both = np.intersect1d(ids, oids)
            a, b = np.searchsorted(ids, both), np.searchsorted(oids, both)
            held = om[b] >= 1e-2 * np.float32(g["vol"]) * np.float32(mat["rho"])
            err = np.max(np.abs(vs[a][held] - ovs[b][held]))
            assert err <= per_stress * lame * 1e-6 * 3 ** 0.5 + 1e-6 * np.max(np.abs(ovs[b][held]))
    finally:
        sim.close()
