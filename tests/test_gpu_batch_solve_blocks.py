"""The blocks that a batch gives each scene's contact solve by itself, on both
sides of the count from which a scene has one block (1.5 per SM: two blocks,
measured, lose to one beyond it). A solve over a cluster counts in
cluster_substeps, one block's (of more contacts than the shared-memory kernel
takes) does not."""
import pytest

from paper_2503_05046_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beyond", [0, 1])
def test_blocks_by_scene_count(beyond):
    import torch
    from paper_2503_05046_gb300 import native
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sc = scenes.sand_slab(19, 19, 1)
    sc["bodies"] = sc["bodies"][:1]
    batch = native.Batch([sc] * (3 * sms // 2 + beyond))
    try:
        batch.step(sc["h"], 1, native.solver_params())
        _, codes, stats = batch.synchronize()
        assert all(c == 0 for c in codes)
        assert all(s["contacts_max"] == 361 for s in stats)
        assert all(s["cluster_substeps"] == 1 - beyond for s in stats)
    finally:
        batch.close()
