"""The default route of a large context's contact solve (1,600 contacts under
160,000 particles) by whether another step is in flight on the device: alone the
cooperative launch, beside another context's step the cluster, which does not
wait for the whole device. A context that is merely alive changes nothing, nor
does one whose own option says otherwise. The solution is the same either way
to the solve's tolerance, and the count of steps in flight returns to zero
after steps, batches and backward passes."""
import time

import numpy as np
import pytest

from paper_2503_05046_gb300 import scenes

pytestmark = pytest.mark.gpu
SUB = 1  # (every bottom particle is in contact in the first substep)


def slab():
    sc = scenes.sand_slab(40, 40, 100)
    sc["bodies"] = sc["bodies"][:1]
    return sc


def run(sim, st):
    """(substeps by cluster, state) of a step from st."""
    sim.set_particles(st["x"], st["v"], st["C"], st["F"])
    stats = sim.step(n_substeps=SUB)
    assert stats.contacts_max == 1600 and stats.residual_max <= 5e-2
    return stats.cluster_substeps, sim.get_particles()


def keep_busy(sim):
    """A step that goes on for tens of milliseconds."""
    sim.step(n_substeps=1000, stats=False, check=False)
    time.sleep(0.002)


def test_route_follows_what_is_in_flight():
    from paper_2503_05046_gb300 import native
    sim, other = native.Sim(slab()), native.Sim(scenes.cube_contact(n_side=20))
    try:
        st = sim.get_particles()
        c0, alone = run(sim, st)
        assert c0 == 0
        keep_busy(other)
        c1, beside = run(sim, st)
        assert c1 == SUB and not other.torch_stream.query()
        other.torch_stream.synchronize()
        native.mpm_synchronize(other.ctx)
        assert run(sim, st)[0] == 0
        scale = np.max(np.abs(alone["v"]))
        assert np.max(np.abs(alone["v"] - beside["v"])) <= 5e-2 * scale
        # an option of its own is kept whatever else runs
        native.mpm_set_option(sim.ctx, native.OPT_CLUSTER_CONTACTS, 1024)
        keep_busy(other)
        assert run(sim, st)[0] == 0
        other.torch_stream.synchronize()
        native.mpm_set_option(sim.ctx, native.OPT_CLUSTER_CONTACTS, 4096)
        assert run(sim, st)[0] == SUB
    finally:
        sim.close()
        other.close()


def test_count_returns_to_zero():
    """After a batch's steps, a step without particles' motion (no substeps), a
    taped rollout and its backward pass, and direct launches, a lone context is
    alone again."""
    from paper_2503_05046_gb300 import native
    sim = native.Sim(slab())
    batch = native.Batch([scenes.batch_scene(i, n_min=2000, n_max=4000) for i in range(3)])
    sc = scenes.cube_contact(n_side=6)
    small = native.Sim(sc)
    try:
        st = sim.get_particles()
        for _ in range(3):
            batch.step(batch.sims[0].scene["h"], 2, native.solver_params())
        batch.synchronize(stats=False)
        assert run(sim, st)[0] == 0
        small.step(n_substeps=0)
        native.mpm_set_option(small.ctx, native.OPT_GRAPHS, 0)
        small.step(n_substeps=1)
        small.tape_begin()
        for _ in range(2):
            small.step(n_substeps=3)
        small.tape_end()
        bar = np.zeros((small.n, 3), np.float32)
        bar[:, 2] = 1.0
        small.backward(x_bar=bar, v_bar=bar, check=False)
        assert run(sim, st)[0] == 0
    finally:
        sim.close()
        small.close()
        batch.close()
