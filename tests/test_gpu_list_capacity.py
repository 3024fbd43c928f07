"""Neighbour-list storage: builds without a size read-back that run out of
it, and sets loaded into a context whose sizes come from another set."""
import numpy as np
import pytest

from paper_2107_01276_gb300 import sph
from paper_2107_01276_gb300 import workloads as wl
from tests.helpers import by_id, cuda_ok, stream_handle

pytestmark = pytest.mark.gpu
STATE = ["x", "y", "u", "v", "p", "rho"]


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not cuda_ok():
        pytest.skip("no CUDA device")


def _sim(d, precision, **kw):
    P = sph.make_params(d["params"], precision=precision,
                        capacity=len(d["particles"]["x"]), **kw)
    s = sph.Simulation(P, stream_handle())
    s.load(d["particles"])
    if "walls" in d:
        s.load(d["walls"], kind=sph.SPH_WALL)
    return s


def _packed(pt, **scale):
    """The set squeezed along the given axes, h as it was."""
    return dict(pt, **{a: pt[a] * f for a, f in scale.items()})


@pytest.mark.parametrize("case,precision,call", [
    ("small", sph.SPH_MIXED, "step"), ("small", sph.SPH_FP64, "step"),
    ("small", sph.SPH_MIXED, "rhs"), ("rows", sph.SPH_MIXED, "step"),
    ("walls", sph.SPH_MIXED, "step"), ("walls", sph.SPH_FP64, "rhs")])
def test_overflow_without_readback_is_reported_and_left_behind(case, precision, call):
    """The third set has the first one's count and h but at least four times
    its neighbours, so its build runs without a read-back and overflows: the
    call reports it (what the kernels read meanwhile lies inside the lists,
    whose offsets end at the capacity), the packed set then builds, and the
    first set steps as in a fresh context."""
    if case == "walls":
        d = wl.half_plane_walls(nx=60, ny=20, layers=4, dx=0.02, seed=5)
        packed = _packed(d["particles"], y=0.1)
    else:
        d = wl.taylor_green(nx=50 if case == "small" else 220, jitter=0.1, seed=4)
        packed = _packed(d["particles"], x=0.4, y=0.4)

    def advance(s):
        if call == "step":
            s.step(1)
        else:
            s.rhs()
            s.read("dudt")

    sim = _sim(d, precision)
    if case == "walls":
        sim.set_tuning(walls=2)
    for _ in range(2):
        advance(sim)
        sim.load(d["particles"])
    advance(sim)
    sim.load(packed)
    with pytest.raises(sph.SphError) as e:
        advance(sim)
    assert e.value.status == sph.SPH_ECAPACITY and "overflow" in str(e.value)
    sim.load(packed)
    advance(sim)
    assert all(np.isfinite(v).all() for v in by_id(sim, STATE).values())
    sim.load(d["particles"])
    advance(sim)
    ref = _sim(d, precision)
    if case == "walls":
        ref.set_tuning(walls=2)
    advance(ref)
    a, b = by_id(sim, STATE), by_id(ref, STATE)
    sim.close()
    ref.close()
    for f in STATE:
        assert np.array_equal(a[f], b[f]), f
