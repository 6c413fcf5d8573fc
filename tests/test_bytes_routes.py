"""Byte layout without a bit layout: short calls of large lattices take a launch per half-sweep and step, longer
ones a resident launch.  Both ways give the same spins, permutation and integer sums."""
import numpy as np
import pytest

import paper_1508_06268_gb300 as rf
from paper_1508_06268_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [(24, 64), (40, 160), (48, 40), (50, 24), (50, 3), (56, 40), (72, 3), (100, 2), (116, 2), (30, 250), (10, 24)]


def make(L, R, kind):
    return rf.Realization(L, inputs.geometric_temps(1.0, 5.0, R), h=1.5, field_kind=kind, field_seed=3, seed=9,
                          layout=rf.LAYOUT_INT8)


def same(a, b):
    x, y = a.get_state(), b.get_state()
    np.testing.assert_array_equal(x["spins"], y["spins"])
    np.testing.assert_array_equal(x["t2r"], y["t2r"])


@pytest.mark.parametrize("L,R", SIZES)
def test_call_by_call_equals_one_call(L, R):
    a, b = make(L, R, rf.FIELD_BIMODAL), make(L, R, rf.FIELD_BIMODAL)
    assert a.plan()[-1] == "b"
    a.run(24, 6, 1)
    for _ in range(4):
        for _ in range(3):
            b.sweep(2)
        b.exchange(1)
    same(a, b)
    p, q = a.observables(), b.observables()
    for k in ("sums", "att", "acc"):
        np.testing.assert_array_equal(p[k], q[k])
    # float field: the decisions of the sweeps (energies are sums in another order)
    a, b = make(L, R, rf.FIELD_GAUSSIAN), make(L, R, rf.FIELD_GAUSSIAN)
    a.sweep(40)
    for _ in range(40):
        b.sweep(1)
    same(a, b)
    a.exchange(0)
    b.exchange(0)
    np.testing.assert_allclose(a.observables()["sums"], b.observables()["sums"], rtol=1e-12)


def test_routes_by_size():
    """Small lattices stay on the resident kernel for every call; the largest with few replicas do not."""
    for L, R, launches in ((10, 24, 1), (24, 40, 1), (116, 2, 4), (72, 3, 4)):
        g = make(L, R, rf.FIELD_GAUSSIAN)
        n0 = g.launch_count
        g.sweep(2)
        assert g.launch_count - n0 == launches
        g.close()
