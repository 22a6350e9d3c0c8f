"""The blocks that a batch gives each scene's contact solve by itself, on both
sides of the count from which a scene has one block: 1.5 scenes per SM, three if
one of them has 12,000 particles. A solve over a cluster counts in
cluster_substeps, one block's (of more contacts than the shared-memory kernel
takes) does not."""
import pytest

from paper_2503_05046_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,clustered", [(0, True), (1, False), (33, False), (34, True)])
def test_blocks_by_scene_count_and_size(layers, clustered):
    """228 scenes (layers 0), and 229 of which one has that many layers of 361"""
    import torch
    from paper_2503_05046_gb300 import native
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sc = scenes.sand_slab(19, 19, 1)
    sc["bodies"] = sc["bodies"][:1]
    one = scenes.sand_slab(19, 19, max(layers, 1))
    one["bodies"] = one["bodies"][:1]
    batch = native.Batch([sc] * (3 * sms // 2) + ([one] if layers else []))
    try:
        batch.step(sc["h"], 1, native.solver_params())
        _, codes, stats = batch.synchronize()
        assert all(c == 0 for c in codes)
        assert all(s["contacts_max"] == 361 for s in stats)
        assert all(s["cluster_substeps"] == int(clustered) for s in stats)
    finally:
        batch.close()
