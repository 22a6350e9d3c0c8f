"""The one-block contact solve (up to 320 contacts whose nodes fit in shared
memory) at its edges against the oracle, per substep as test_gpu_parity does:
a single contact, the last count it takes and the first it does not, and few
contacts with too many nodes (which go on to the cluster). Several bodies are
in test_gpu_parity's cube cases."""
import numpy as np
import pytest

from paper_2503_05046_gb300 import scenes
from test_gpu_parity import native, run_parity  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def slab(contacts):
    """A sand slab with exactly `contacts` particles in the ground."""
    side = int(np.ceil(np.sqrt(contacts)))
    sc = scenes.sand_slab(side, side, 2)
    x = sc["groups"][0]["x"]
    low = np.argsort(x[:, 2], kind="stable")[:side * side]  # the bottom layer
    x[low[contacts:], 2] += np.float32(1e-4)
    sc["bodies"] = sc["bodies"][:1]
    return sc


@pytest.mark.parametrize("contacts", [1, 31, 319, 320, 321])
def test_contact_counts(native, contacts):  # noqa: F811
    rep = run_parity(native, slab(contacts), n_sub=1)
    assert rep[0][1] == contacts
    assert all(r[6] == 1 and r[5] == 0 for r in rep), rep


def test_few_contacts_many_nodes(native):  # noqa: F811
    """Contacts far from each other: 27 nodes each, more than the table holds."""
    dx, side = 0.01, 14
    sc = scenes.sand_slab(side, side, 1)
    x = sc["groups"][0]["x"]
    x[:, :2] *= np.float32(6.0)  # particles three cells apart
    sc["bodies"] = sc["bodies"][:1]
    res = 4 * int(np.ceil((6.0 * side * 0.5 + 16) / 4))
    sc["grid"] = dict(sc["grid"], res=(res, res, sc["grid"]["res"][2]),
                      origin=(-res * dx / 2, -res * dx / 2, -8 * dx))
    rep = run_parity(native, sc, n_sub=1)
    assert rep[0][1] == side * side and rep[0][6] == 1, rep
