"""The contact solve over several blocks at the edges of its rounds, against
the oracle, per substep as test_gpu_parity does: the counts at which the line
search is split over the blocks (512, 513), at which the cooperative launch takes
over from the cluster (4,096, 4,097; 1,024 from 160,000 particles on) and at which a block's warps go over their
contacts again (128 per block: 512 and 513 with four blocks, 2,048 and 2,049 with
a cluster of sixteen), and one contact more than a warp's eight."""
import pytest

from paper_2503_05046_gb300 import scenes
from test_gpu_parity import native, run_parity  # noqa: F401 (fixture)
from test_gpu_solve_small import slab

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("contacts,cluster", [(321, 1), (512, 1), (513, 1), (1024, 1), (4096, 1), (4097, 0)])
def test_default_route(native, contacts, cluster):  # noqa: F811
    rep = run_parity(native, slab(contacts), n_sub=1)
    assert rep[0][1] == contacts and rep[0][6] == cluster, rep
    assert rep[0][5] == (1 if contacts > 512 else 0), rep


@pytest.mark.parametrize("layers,cluster", [(99, 1), (100, 0)])
def test_default_route_by_particles(native, layers, cluster):  # noqa: F811
    """1,600 contacts under 158,400 and 160,000 particles"""
    sc = scenes.sand_slab(40, 40, layers)
    sc["bodies"] = sc["bodies"][:1]
    sim = native.Sim(sc)
    try:
        stats = sim.step(n_substeps=1)
        assert stats.contacts_max == 1600 and stats.cluster_substeps == cluster
        assert stats.ls_split_substeps == 1 and stats.residual_max <= 5e-2
    finally:
        sim.close()


@pytest.mark.parametrize("blocks", [0, 4])
@pytest.mark.parametrize("contacts", [9, 512, 513, 1500])
def test_cooperative(native, contacts, blocks):  # noqa: F811
    rep = run_parity(native, slab(contacts), n_sub=1,
                     options=((native.OPT_CLUSTER_CONTACTS, 0), (native.OPT_SOLVE_BLOCKS, blocks)))
    assert rep[0][1] == contacts and rep[0][6] == 0, rep
    assert rep[0][5] == (1 if contacts > 512 else 0), rep


@pytest.mark.parametrize("contacts", [2048, 2049])
def test_cluster(native, contacts):  # noqa: F811
    rep = run_parity(native, slab(contacts), n_sub=1, options=((native.OPT_CLUSTER_CONTACTS, 1 << 16),))
    assert rep[0][1] == contacts and rep[0][6] == 1 and rep[0][5] == 1, rep
