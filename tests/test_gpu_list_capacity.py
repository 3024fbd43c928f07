"""Neighbour-list storage: builds without a size read-back that run out of
it, sets loaded into a context whose sizes come from another set, and the
cells of particles whose positions are lost."""
import numpy as np
import pytest

from paper_2107_01276_gb300 import sph
from paper_2107_01276_gb300 import workloads as wl
from tests.helpers import MIXED_TOL, by_id, cuda_ok, stream_handle

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


@pytest.mark.parametrize("second", ["coarser_h", "denser", "fewer"])
def test_reloaded_context_takes_a_set_whose_rows_overflow(second):
    """A set whose step keeps every own entry in the rows, then one of the
    same count with more own entries a particle than a row holds: with
    larger h, or denser by 1.6 at the same h, or with a tenth fewer
    particles and larger h.  The steps after the second load are a fresh
    context's to the mixed tolerance of the change, once a step."""
    d = wl.taylor_green(nx=230, hdx=1.2, jitter=0.1, seed=8)
    pt = dict(d["particles"])
    if second == "denser":
        pt = _packed(pt, x=0.62)
    else:
        pt["h"] = pt["h"] * (1.55 / 1.2)
        if second == "fewer":
            pt = {k: v[:48100] for k, v in pt.items()}
    sim = _sim(d, sph.SPH_MIXED)
    sim.step(2)
    sim.load(pt)
    ref = _sim(dict(d, particles=pt), sph.SPH_MIXED)
    out = []
    for s in (sim, ref):
        s.step(1)
        one = by_id(s, STATE)
        s.step(3)
        out.append((one, by_id(s, STATE)))
        s.close()
    for a, b, k in zip(*out, (1, 4)):
        for f in ("u", "v", "p"):
            change = np.abs(b[f] - pt[f]).max()
            assert np.abs(a[f] - b[f]).max() <= k * MIXED_TOL * change, f


@pytest.mark.parametrize("walk", [1, 2, 3, 4])
@pytest.mark.parametrize("precision", [sph.SPH_FP64, sph.SPH_MIXED])
def test_nan_positions_leave_the_cells_of_the_others_alone(precision, walk):
    """A NaN pressure makes the positions around it NaN within a step.  In
    the next build they count for cell 0: the walks over a level of two by
    two cells, all of them in reach, still find the other particles, which
    stay finite."""
    d = wl.taylor_green(nx=50, jitter=0.1, seed=4)
    pt = dict(d["particles"], p=d["particles"]["p"].copy())
    pt["p"][1275] = np.nan
    s = _sim(dict(d, particles=pt), precision, cell_c0=0.4)
    s.set_tuning(walk=walk)
    for _ in range(2):
        with pytest.raises(sph.SphError) as e:
            s.step(1)
        assert e.value.status == sph.SPH_ENONFINITE
    got = by_id(s, STATE)
    s.close()
    bad = ~np.isfinite(got["x"])
    assert 1 < bad.sum() < 400
    for f in STATE:
        assert np.isfinite(got[f][pt["y"] < 0.2]).all(), f


@pytest.mark.parametrize("change", ["same", "h", "n"])
def test_a_set_reloaded_with_little_change_keeps_the_list_sizes(change):
    """Small sets reloaded before every step, as they were, with h 4 % larger
    or with one particle fewer: the step takes the launches of the batched
    build every time (a build that reads its size back is not batched)."""
    ds = [wl.taylor_green(nx=nx, jitter=0.1, seed=nx) for nx in (30, 42)]
    sims = [_sim(d, sph.SPH_MIXED) for d in ds]
    per_step = []
    with sph.Batch(2, stream_handle()) as b:
        b.set_graphs(False)
        for k in range(6):
            for s, d in zip(sims, ds):
                pt = d["particles"]
                if k % 2 and change == "h":
                    pt = dict(pt, h=pt["h"] * 1.04)
                if k % 2 and change == "n":
                    pt = {f: v[:-1] for f, v in pt.items()}
                s.load(pt)
            before = b.launches
            b.step(sims)
            per_step.append(b.launches - before)
    for s in sims:
        s.close()
    assert len(set(per_step[2:])) == 1 and per_step[2] == 20
