"""Bounded waits inside the resident launches: one that is given up ends the launch in order (no CTA pushes
or arrives again, none leaves while a push to it is on its way), the error is reported once, and
the realization goes on from a state that is set."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import paper_1508_06268_gb300 as rf
from paper_1508_06268_gb300 import inputs

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SLABS = [  # L, R, "S,G,NB,threads,r" (m: several items per thread, b: bytes), tile (0: plain checkerboard)
    (8, 7, "1,3,1,256,r", 0), (10, 3, "1,1,4,128,b", 0), (16, 5, "1,3,2,384,r", 8),
    (16, 5, "2,2,2,256,r", 0), (32, 3, "8,1,2,256,r", 0), (32, 2, "4,1,4,256,r", 0), (32, 5, "2,3,4,512,m", 0),
    (64, 2, "16,1,4,512,r", 0), (64, 3, "8,2,4,512,m", 0), (14, 5, "5,2,4,256,b", 0), (24, 5, "4,2,4,512,b", 0),
    (28, 2, "8,1,4,448,b", 0), (32, 3, "4,2,2,512,r", 8), (32, 3, "2,2,4,512,r", 16), (64, 4, "8,1,4,512,r", 8),
    (64, 5, "4,2,4,512,m", 32), (64, 4, "16,1,2,512,r", 16),
]


def pair(monkeypatch, L, R, plan, tile):
    kw = dict(h=1.5, field_kind=rf.FIELD_BIMODAL, field_seed=3, seed=42)
    temps = inputs.geometric_temps(1.0, 5.0, R)
    env = monkeypatch or pytest.MonkeyPatch()
    env.setenv("RFIM_BITS_PLAN", plan)
    g = rf.Realization(L, temps, layout=rf.LAYOUT_INT8 if plan[-1] == "b" else rf.LAYOUT_BITPACK, **kw)
    o = oracle.Oracle(L, temps, **kw)
    if tile:
        g.set_multihit(2, tile)
        o.set_multihit(2, tile)
    env.delenv("RFIM_BITS_PLAN")
    assert g.plan() == plan
    return g, o


CHILD = r"""
import ctypes as C, os, sys
import numpy as np
sys.path.insert(0, os.environ["RFIM_ROOT"])
import paper_1508_06268_gb300 as rf
from tests.test_resident_waits import SLABS, pair

assert rf.debug_build()


def timed_out(f):
    try:
        f()
    except rf.RfimError as e:
        return e.code == rf.ETIMEOUT
    return False


for L, R, plan, tile in SLABS:
    g, o = pair(None, L, R, plan, tile)
    S, G = int(plan.split(",")[0]), int(plan.split(",")[1])
    ctas = (R + G - 1) // G * S
    g.run(4, 2, 0)
    o.run(4, 2, 0)
    good = g.get_state()
    assert np.array_equal(good["spins"], o.spins()), plan
    for cta, interval in ((0, 0), (ctas - 1, 1), (S // 2, 2)):
        g.selftest_resident(cta, interval)
        g.run(12, 2, 0)
        g.sweep(3)
        g.exchange(0)
        assert timed_out(g.get_state), (plan, cta, interval)
        g.selftest_resident()
        g.set_state(good["spins"], good["t2r"], good["sweep"], good["xstep"])
    g.run(6, 2, 0)
    o.run(6, 2, 0)
    st = g.get_state()
    assert np.array_equal(st["spins"], o.spins()), plan
    assert np.array_equal(st["t2r"], o.perm()[0]), plan

# a read that reports the error writes nothing of the caller's
g, _ = pair(None, 16, 5, "2,2,2,256,r", 0)
g.selftest_resident(0)
g.run(4, 2, 0)
spins, t2r, E = np.full((5, 4096), 7, np.int8), np.full(5, -7, np.int32), np.full(5, 0.5)
sweep, xstep = C.c_int64(-7), C.c_int64(-7)
rc = rf.load().rfim_get_state(g._h, spins.ctypes.data, t2r.ctypes.data, E.ctypes.data, C.byref(sweep), C.byref(xstep))
assert rc == rf.ETIMEOUT
assert (spins == 7).all() and (t2r == -7).all() and (E == 0.5).all() and sweep.value == xstep.value == -7
print("waits ok")
"""


def test_given_up_wait_ends_in_order():
    """Debug library: one CTA gives up a wait, at once, in a later interval, and in launches that are queued behind
    the failed one.  Its neighbours in the cluster, at every distance, and the other clusters stop too."""
    env = dict(os.environ, RFIM_LIBRARY="debug", RFIM_ROOT=ROOT)
    env.pop("RFIM_BITS_PLAN", None)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0 and "waits ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def test_stops_are_refused_in_the_release_library(monkeypatch):
    g, _ = pair(monkeypatch, 16, 5, "2,2,2,256,r", 0)
    with pytest.raises(rf.RfimError) as e:
        g.selftest_resident(0)
    assert e.value.code == rf.ESTATE


def test_long_intervals_do_not_run_out_of_polls(monkeypatch):
    """The last cluster holds one replica where the other holds twenty, so it waits for almost the whole
    interval: 0.18 ms per sweep, 3.6 s in all."""
    monkeypatch.setenv("RFIM_BITS_PLAN", "4,20,4,512,m")
    g = rf.Realization(64, inputs.geometric_temps(1.0, 5.0, 21), field_kind=rf.FIELD_GAUSSIAN, seed=4)
    assert g.plan() == "4,20,4,512,m"
    g.run(20000, 20000, 0)
    st = g.get_state()
    assert st["sweep"] == 20000 and st["xstep"] == 1
    assert g.observables()["n_meas"] == 1


@pytest.mark.parametrize("mh,tile,every", [(0, 0, 2049), (700, 8, 3)])
def test_intervals_swept_apart_match_oracle(mh, tile, every, monkeypatch):
    """Above 2048 sweeps (multi-hit: passes) per interval the sweeps are a launch of their own."""
    g, o = pair(monkeypatch, 16, 3, "1,1,1,512,r", 0)
    if mh:
        g.set_multihit(mh, tile)
        o.set_multihit(mh, tile)
    n0 = g.launch_count
    g.run(2 * every, every, 0)
    assert g.launch_count - n0 == 4
    o.run(2 * every, every, 0)
    st = g.get_state()
    np.testing.assert_array_equal(st["spins"], o.spins())
    np.testing.assert_array_equal(st["t2r"], o.perm()[0])
    np.testing.assert_array_equal(g.observables()["sums"], o.observables())


@pytest.mark.parametrize("which", [0, 1, 2])
def test_each_wait_expires(which):
    """A wait for what nobody sets ends with the status, one for what is set with success; the context goes on."""
    assert rf.selftest_waits(which, 1000, False) == rf.ETIMEOUT
    assert rf.selftest_waits(which, 1, True) == rf.OK
    assert rf.selftest_waits(which, 1, False) == rf.ETIMEOUT
    assert rf.selftest_waits(which, 0, True) == rf.EINVAL


@pytest.mark.parametrize("L,R,plan", [(16, 5, "2,2,2,256,r"), (24, 5, "4,2,4,512,b")])
def test_interval_numbers_start_again(L, R, plan, monkeypatch):
    """The numbers that energy records carry end at 2^22 - 1; launches before, across and after that line."""
    g, o = pair(monkeypatch, L, R, plan, 0)
    g.selftest_resident(number=(1 << 22) - 12)
    for sweeps in (4, 12, 6, 8):
        g.run(sweeps, 2, 0)
        o.run(sweeps, 2, 0)
    st = g.get_state()
    np.testing.assert_array_equal(st["spins"], o.spins())
    np.testing.assert_array_equal(st["t2r"], o.perm()[0])
    np.testing.assert_array_equal(g.observables()["sums"], o.observables())
    with pytest.raises(rf.RfimError):
        g.selftest_resident(number=(1 << 22) - 1)
