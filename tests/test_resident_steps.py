"""Exchange step numbers past 2^32 on the resident plan: the streams use the low 32 bits, the structure factor
is measured by the whole number, as by one kernel per measuring step."""
import numpy as np
import pytest

import paper_1508_06268_gb300 as rf
from paper_1508_06268_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("xstep,measure_from", [(2**32 - 2, 2), (2**32 + 1, 3), (2**33, 2**33 + 2), (3, -2**63)])
@pytest.mark.parametrize("L,R,plan,ref", [(16, 5, "1,2,2,512,r", "1,4,1,512"), (32, 3, "8,1,2,256,r", "2,1,1,256")])
def test_structure_factor_by_whole_step_number(L, R, plan, ref, xstep, measure_from, monkeypatch):
    """Against the cluster plan: the same integers, and Fourier sums in the same order (1e-11 as in the oracle's
    tests)."""
    got = []
    for p in (plan, ref):
        monkeypatch.setenv("RFIM_BITS_PLAN", p)
        g = rf.Realization(L, inputs.geometric_temps(1.0, 5.0, R), h=1.5, field_kind=rf.FIELD_BIMODAL, seed=6)
        g.set_measure_xi()
        g.set_state(sweep=0, xstep=xstep)
        g.run(12, 2, measure_from)
        got.append((g.plan()[-1] == "r", g.get_state(), g.observables()))
        g.close()
    (res, st, obs), (_, st_ref, obs_ref) = got
    assert res and not got[1][0]
    np.testing.assert_array_equal(st["spins"], st_ref["spins"])
    np.testing.assert_array_equal(st["t2r"], st_ref["t2r"])
    np.testing.assert_array_equal(obs["sums"], obs_ref["sums"])
    np.testing.assert_allclose(obs["F"], obs_ref["F"], rtol=1e-11, atol=1e-20)
    assert (obs["F"] > 0).all()
