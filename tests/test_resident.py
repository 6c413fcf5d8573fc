"""The resident sweep kernel (small realizations, many exchange intervals per launch): every launch
shape it is instantiated for, partial replica groups included, against the oracle."""
import numpy as np
import pytest

import oracle
import paper_1508_06268_gb300 as rf
from paper_1508_06268_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [  # L, R, "S,G,NB,threads,r" (m: several items per thread)
    (8, 2, "1,1,1,64,r"), (8, 7, "1,3,1,256,r"), (8, 19, "1,4,2,128,r"), (8, 37, "1,5,4,256,r"),
    (16, 2, "1,1,1,512,r"), (16, 5, "1,2,2,512,r"), (16, 13, "1,3,4,384,r"), (16, 3, "2,1,1,256,r"), (16, 5, "2,2,2,256,r"),
    (32, 3, "2,1,4,512,r"), (32, 2, "4,1,4,256,r"), (32, 3, "8,1,2,256,r"), (32, 3, "1,2,4,512,m"), (32, 5, "2,3,4,512,m"),
    (64, 2, "16,1,4,512,r"), (64, 3, "8,2,4,512,m"), (64, 3, "4,2,4,512,m"),
]


def make(monkeypatch, L, R, plan, **kw):
    monkeypatch.setenv("RFIM_BITS_PLAN", plan)
    g = rf.Realization(L, inputs.geometric_temps(1.0, 5.0, R), **kw)
    monkeypatch.delenv("RFIM_BITS_PLAN")
    if plan[-1] in "rmb":
        assert g.plan().replace(",int8", "") == plan
    else:  # a cluster plan: its group is clipped to R
        assert g.plan()[-1] not in "rmb"
    return g


@pytest.mark.parametrize("L,R,plan", SHAPES)
@pytest.mark.parametrize("layout", [rf.LAYOUT_BITPACK, rf.LAYOUT_INT8])
def test_resident_shapes_bit_exact(L, R, plan, layout, monkeypatch):
    """Bimodal field: spins, permutation, exchange counts and sums equal the oracle's after several
    launches of several intervals, with an odd number of half-sweep pairs between exchanges."""
    if layout == rf.LAYOUT_INT8 and L == 64:
        pytest.skip("one layout is enough at the largest size")
    g = make(monkeypatch, L, R, plan, h=1.5, field_kind=rf.FIELD_BIMODAL, field_seed=3, seed=42, layout=layout)
    o = oracle.Oracle(L, inputs.geometric_temps(1.0, 5.0, R), h=1.5, field_kind=oracle.FIELD_BIMODAL, field_seed=3, seed=42)
    n0 = g.launch_count
    g.run(9, 3, 1)
    assert g.launch_count - n0 == 1
    g.sweep(1)
    g.exchange(0)
    g.run(7, 2, 0)
    o.run(9, 3, 1)
    o.sweep(1)
    o.exchange(0)
    o.run(7, 2, 0)
    st = g.get_state()
    np.testing.assert_array_equal(st["spins"], o.spins())
    np.testing.assert_array_equal(st["t2r"], o.perm()[0])
    np.testing.assert_array_equal(g.observables()["sums"], o.observables())


@pytest.mark.parametrize("L,R,plan,ref", [(8, 6, "1,1,1,64,r", "1,16,1,128"), (16, 5, "1,1,2,256,r", "1,8,1,512"),
                                           (32, 4, "2,1,4,512,r", "2,1,1,256"), (64, 5, "8,1,4,512,m", "4,4,4,512")])
def test_resident_gaussian_equals_cluster_plan(L, R, plan, ref, monkeypatch):
    """Float field: the decisions are those of the one-launch-per-interval kernel (the same float
    operations on the same words), and the fixed-point energies are the same sums."""
    kw = dict(field_kind=rf.FIELD_EXPLICIT, field=inputs.gaussian_field(L, 77), seed=5)
    a = make(monkeypatch, L, R, plan, **kw)
    b = make(monkeypatch, L, R, ref, **kw)
    for g in (a, b):
        g.run(60, 3, 4)
    x, y = a.get_state(), b.get_state()
    np.testing.assert_array_equal(x["spins"], y["spins"])
    np.testing.assert_array_equal(x["t2r"], y["t2r"])
    p, q = a.observables(), b.observables()
    assert p["n_meas"] == q["n_meas"] == 16
    for k in ("sums", "att", "acc"):
        np.testing.assert_array_equal(p[k], q[k])


MULTIHIT = [  # L, R, tile, "S,G,NB,threads,r": slabs of whole tiles and slabs that cut them, partial groups
    (16, 3, 8, "1,2,1,512,r"), (16, 5, 8, "1,3,2,384,r"), (16, 5, 8, "1,4,4,256,r"), (32, 2, 8, "4,1,1,512,r"),
    (32, 3, 8, "4,2,2,512,r"), (32, 3, 8, "2,1,2,512,r"), (32, 3, 8, "2,2,4,512,r"), (32, 2, 16, "4,1,1,512,r"),
    (32, 3, 16, "2,1,2,512,r"), (32, 3, 16, "2,2,4,512,r"), (64, 4, 8, "16,1,2,512,r"), (64, 4, 8, "8,1,4,512,r"),
    (64, 5, 8, "4,2,4,512,m"), (64, 4, 16, "16,1,2,512,r"), (64, 4, 16, "8,1,4,512,r"), (64, 5, 16, "4,3,4,512,m"),
    (64, 4, 32, "16,1,2,512,r"), (64, 4, 32, "8,1,4,512,r"), (64, 5, 32, "4,2,4,512,m"),
]


@pytest.mark.parametrize("L,R,tile,plan", MULTIHIT)
@pytest.mark.parametrize("kind", [rf.FIELD_BIMODAL, rf.FIELD_EXPLICIT])
def test_resident_multihit(L, R, tile, plan, kind, monkeypatch):
    """Multi-hit sweeps of the resident kernel, several intervals per launch: with a bimodal field equal
    to the oracle's; with a float field equal to the cluster kernel's (the same float operations)."""
    mh = 3 if L < 64 else 2
    kw = dict(h=1.5, field_kind=kind, field=inputs.gaussian_field(L, 3) if kind == rf.FIELD_EXPLICIT else None, seed=8)
    monkeypatch.setenv("RFIM_BITS_PLAN", plan)
    g = rf.Realization(L, inputs.geometric_temps(1.0, 5.0, R), **kw)
    g.set_multihit(mh, tile)
    assert g.plan() == plan
    if kind == rf.FIELD_BIMODAL:
        o = oracle.Oracle(L, inputs.geometric_temps(1.0, 5.0, R), **kw)
    else:
        monkeypatch.setenv("RFIM_BITS_PLAN", {16: "1,4,1,512", 32: "2,1,1,256", 64: "4,4,4,512"}[L])
        o = rf.Realization(L, inputs.geometric_temps(1.0, 5.0, R), **kw)
    o.set_multihit(mh, tile)
    n0 = g.launch_count
    for x in (g, o):
        x.run(4, 2, 1)
        x.sweep(1)
        x.exchange(0)
    assert g.launch_count - n0 == 3
    st = g.get_state()
    if kind == rf.FIELD_BIMODAL:
        want = (o.spins(), o.perm()[0], o.observables())
    else:
        assert o.plan() in ("1,4,1,512", "1,3,1,512", "2,1,1,256", "4,4,4,512")
        want = (o.get_state()["spins"], o.get_state()["t2r"], o.observables()["sums"])
    np.testing.assert_array_equal(st["spins"], want[0])
    np.testing.assert_array_equal(st["t2r"], want[1])
    np.testing.assert_array_equal(g.observables()["sums"], want[2])


@pytest.mark.parametrize("L,R,plan", [(8, 7, "1,3,1,256,r"), (16, 13, "1,3,4,384,r"), (16, 5, "2,2,2,256,r"),
                                      (32, 3, "8,1,2,256,r"), (32, 3, "1,2,4,512,m"), (64, 2, "16,1,4,512,r"),
                                      (64, 3, "8,2,4,512,m")])
def test_resident_structure_factor(L, R, plan, monkeypatch):
    """The structure factor measured inside a launch of several intervals, some before measure_from, then
    call by call: integers, the same Fourier sums and the same order as one kernel per measuring
    step, so the sums are the oracle's to its tests' 1e-11 (exact marginals, sums in double)."""
    kw = dict(h=1.5, field_kind=rf.FIELD_BIMODAL, field_seed=3, seed=6)
    g = make(monkeypatch, L, R, plan, **kw)
    o = oracle.Oracle(L, inputs.geometric_temps(1.0, 5.0, R), **kw)
    g.set_measure_xi()
    o.set_measure_xi(True)
    n0 = g.launch_count
    for x in (g, o):
        x.run(12, 2, 2)
        x.exchange(0)
        x.run(6, 2, 100)
        x.run(4, 2, 0)
    assert g.launch_count - n0 == 7  # four launches of intervals, three of Fourier sums
    np.testing.assert_array_equal(g.observables()["sums"], o.observables())
    np.testing.assert_allclose(g.observables()["F"], o.observables_F(), rtol=1e-11, atol=1e-20)


BYTES = [  # L, R, "S,G,4,threads,b": rows of whole blocks, even rows, odd rows; blocks across slabs
    (4, 2, "1,1,4,32,b"), (4, 9, "2,4,4,64,b"), (6, 5, "1,3,4,96,b"), (6, 3, "2,2,4,32,b"), (10, 3, "1,1,4,128,b"),
    (10, 5, "4,2,4,96,b"), (14, 3, "2,2,4,256,b"), (18, 2, "8,1,4,128,b"), (12, 5, "1,2,4,256,b"), (12, 3, "4,2,4,128,b"),
    (20, 3, "2,1,4,512,b"), (28, 2, "8,1,4,448,b"), (24, 3, "1,1,4,512,b"), (24, 5, "4,2,4,512,b"), (40, 2, "4,1,4,512,b"),
    (48, 2, "8,1,4,512,b"), (50, 2, "8,1,4,512,b"), (56, 2, "1,1,4,512,b"), (36, 2, "2,1,4,512,b"),
]


@pytest.mark.parametrize("L,R,plan", BYTES)
@pytest.mark.parametrize("kind", [rf.FIELD_BIMODAL, rf.FIELD_EXPLICIT])
def test_resident_bytes_match_oracle(L, R, plan, kind, monkeypatch):
    """Sizes without a bit layout: bimodal spins, permutation and sums equal the oracle's; with a
    float field one sweep from the same state gives the oracle's spins up to 1e-4 of the sites (the
    device's acceptance test is within a few 2^-23 of the oracle's) and its energies to 1e-9."""
    field = inputs.gaussian_field(L, 9) if kind == rf.FIELD_EXPLICIT else None
    kw = dict(h=1.5, field_kind=kind, field=field, field_seed=3, seed=42)
    g = make(monkeypatch, L, R, plan, layout=rf.LAYOUT_INT8, **kw)
    o = oracle.Oracle(L, inputs.geometric_temps(1.0, 5.0, R), **kw)
    if kind == rf.FIELD_BIMODAL:
        for x in (g, o):
            x.run(6, 3, 1)
            x.sweep(1)
            x.exchange(0)
            x.run(4, 2, 0)
        np.testing.assert_array_equal(g.get_state()["spins"], o.spins())
        np.testing.assert_array_equal(g.get_state()["t2r"], o.perm()[0])
        np.testing.assert_array_equal(g.observables()["sums"], o.observables())
        return
    for x in (g, o):
        x.sweep(1)
    spins = g.get_state()["spins"]
    assert np.mean(spins != o.spins()) <= 1e-4
    o.set_spins(spins)
    for x in (g, o):
        x.exchange(0)
    np.testing.assert_array_equal(g.get_state()["t2r"], o.perm()[0])
    np.testing.assert_allclose(g.observables()["sums"], o.observables(), rtol=1e-9)


@pytest.mark.parametrize("L,R,plan", [(6, 3, "3,1,4,32,b"), (14, 5, "5,2,4,256,b")])
@pytest.mark.parametrize("kind", [rf.FIELD_BIMODAL, rf.FIELD_EXPLICIT])
def test_resident_bytes_slabs_not_a_power_of_two(L, R, plan, kind, monkeypatch):
    """Slab counts that only a named shape has: their records are added one after another."""
    test_resident_bytes_match_oracle(L, R, plan, kind, monkeypatch)
