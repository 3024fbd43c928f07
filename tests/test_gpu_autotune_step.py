"""The autotuner measures what a step runs: the step's lists, and a walk
together with the passes that read its lists."""
import pytest

from paper_2107_01276_gb300 import sph
from paper_2107_01276_gb300 import workloads as wl
from tests.helpers import cuda_ok, stream_handle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not cuda_ok():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("precision", [sph.SPH_FP64, sph.SPH_MIXED])
def test_a_walk_is_timed_with_the_passes_on_its_lists(precision):
    """One candidate of the walks is the form that the cell sizes were
    measured with, so its build and passes take that time again; a walk
    alone is a small part of it."""
    d = wl.taylor_green(nx=300, jitter=0.1, seed=6)
    P = sph.make_params(d["params"], precision=precision, capacity=90000)
    with sph.Simulation(P, stream_handle()) as s:
        s.load(d["particles"])
        s.step(2)
        t = s.autotune()
        s.step(2)
    w = dict(zip((1, 2, 4), t["ms_walk"]))
    assert t["walk"] == min(w, key=w.get)
    assert w[t["walk"]] > 0.6 * min(t["ms_cell"])
