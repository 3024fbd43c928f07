"""Sets whose cell keys need more than 32 bits take the one-block sort, and
the batched build of small sets, at the sizes that narrower keys do."""
import numpy as np
import pytest

from paper_2107_01276_gb300 import sph
from paper_2107_01276_gb300 import workloads as wl
from tests.helpers import by_id, cuda_ok, stream_handle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not cuda_ok():
        pytest.skip("no CUDA device")


def _sim(d, c0):
    P = sph.make_params(d["params"], precision=sph.SPH_MIXED,
                        capacity=len(d["particles"]["x"]), cell_c0=c0)
    s = sph.Simulation(P, stream_handle())
    s.load(d["particles"])
    return s


# cell sides of one level of the same grid: the particles' cells and order
# are the same, the keys 18 and 40 bits wide
WIDE = 2.0 ** -12


@pytest.mark.parametrize("nx", [90, 91, 128])
def test_launches_of_a_build_do_not_depend_on_the_key_width(nx):
    d = wl.taylor_green(nx=nx, jitter=0.1, seed=nx)
    c0 = 3.0 * float(d["particles"]["h"][0])
    out = []
    for k in (1.0, WIDE):
        s = _sim(d, c0 * k)
        s.rhs()
        a = s.info()["launches"]
        s.rhs()
        out.append((s.info()["launches"] - a, by_id(s, ("rho", "dudt", "dpdt", "nnb"))))
        s.close()
    assert out[0][0] == out[1][0]
    for f in ("rho", "dudt", "dpdt", "nnb"):
        assert np.allclose(out[0][1][f], out[1][1][f], rtol=1e-4, atol=1e-4 *
                           np.abs(out[0][1][f]).max()), f


def test_batched_builds_take_wide_keys():
    sets = [wl.taylor_green(nx=nx, jitter=0.1, seed=nx) for nx in (60, 95, 110)]
    out = []
    for k in (1.0, WIDE):
        sims = [_sim(d, 3.0 * float(d["particles"]["h"][0]) * k) for d in sets]
        b = sph.Batch(len(sims), stream_handle())
        b.step(sims)
        n0 = b.launches
        b.step(sims)
        out.append((b.launches - n0, [s.info()["launches"] for s in sims]))
        for s in sims:
            s.close()
        b.close()
    assert out[0] == out[1]
