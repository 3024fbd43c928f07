"""The rates of a step on lists with interleaved rows against the same step on
plain lists, in the norm that the right-hand sides are held to."""
import numpy as np
import pytest

import oracle
from paper_2107_01276_gb300 import sph
from tests.helpers import MIXED_TOL, by_id, cuda_ok, norm
from tests.test_gpu_step_paths import _row_cases, _sim

pytestmark = pytest.mark.gpu
RATES = ("rho", "beta", "pavg", "drx", "dry", "dpdt", "dudt", "dvdt")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not cuda_ok():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("case", ["first", "levels", "overflow", "walls", "one_lane"])
def test_rates_of_a_step_on_rows_and_on_plain_lists(case):
    """The rates a step ends with (its second evaluation, half a time step
    on): either form's are within MIXED_TOL of the exact ones, in units of
    the largest sum of |terms| of the field, so they are within twice that
    of each other.  The units are the oracle's at the start of the step,
    and the step's changes of u, v and p follow the rates."""
    d = _row_cases()[case]
    pt = d["particles"]
    out = []
    for walk in (3, 4):
        s = _sim(d, sph.SPH_MIXED)
        if "walls" in d:
            s.load(d["walls"], kind=sph.SPH_WALL)
        s.set_tuning(walk=walk)
        t = s.step(1)
        out.append(by_id(s, RATES + ("nnb", "u", "v", "p")))
        s.close()
    oracle.set_walls(d.get("walls"))
    try:
        P = oracle.params(**d["params"])
        ref = oracle.rhs(P, oracle.dt(P, pt["h"]), oracle.make_state(pt))
    finally:
        oracle.set_walls(None)
    a, b = out
    assert np.array_equal(a["nnb"], b["nnb"])
    for f in RATES:
        assert norm(a[f], b[f], ref["s_" + f]) <= 2 * MIXED_TOL, f
    for f, r in (("u", "dudt"), ("v", "dvdt"), ("p", "dpdt")):
        assert np.abs(a[f] - b[f]).max() <= 2 * MIXED_TOL * t * ref["s_" + r].max(), f
