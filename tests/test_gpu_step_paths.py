"""The sizes at which a step's kernels change their form: the one-block sort
compiled for 1, 4, 8 and 16 items a lane (and the tiled one beyond), cells
longer than the warp that gathers their first particle, and the step's lists
with interleaved rows (from 48000 particles)."""
import numpy as np
import pytest

import oracle
from paper_2107_01276_gb300 import sph
from paper_2107_01276_gb300 import workloads as wl
from tests.helpers import FP64_TOL, MIXED_TOL, by_id, cuda_ok, norm, stream_handle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not cuda_ok():
        pytest.skip("no CUDA device")


def _sim(d, precision, **kw):
    P = sph.make_params(d["params"], precision=precision,
                        capacity=len(d["particles"]["x"]), **kw)
    s = sph.Simulation(P, stream_handle())
    s.load(d["particles"])
    return s


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 4095, 4096, 4097, 8191, 8192,
                               8193, 16383, 16384, 16385])
def test_sort_at_the_edges_of_its_forms(n, wide):
    """Keys equal the oracle's, in ascending order, equal keys in input
    order; wide: keys of more than 32 bits."""
    import torch
    rng = np.random.default_rng(n)
    x, y, h = rng.random(n), rng.random(n), rng.uniform(2e-3, 0.1, n)
    x[n // 2:] = x[:n - n // 2]        # equal keys
    y[n // 2:] = y[:n - n // 2]
    h[n // 2:] = h[:n - n // 2]
    c0 = 3e-6 if wide else 6e-3
    prm = dict(lo=(0.0, 0.0), hi=(1.0, 1.0), periodic=(1, 0))
    P = sph.make_params(prm, capacity=n, cell_c0=c0)
    d = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x, y, h)]
    key = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    perm = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    st = sph.cell_sort_noalloc(P, n, *(t.data_ptr() for t in d), key.data_ptr(),
                               perm.data_ptr(), stream_handle())
    assert st == sph.SPH_OK, sph.last_error()
    torch.cuda.synchronize()
    okey, _ = oracle.cell_keys(oracle.params(**prm), c0, x, y, h)
    order = np.argsort(okey, kind="stable")
    assert np.array_equal(perm.cpu().numpy(), order)
    assert np.array_equal(key.cpu().numpy().view(np.uint64), okey[order])


@pytest.mark.parametrize("precision,tol", [(sph.SPH_FP64, FP64_TOL),
                                           (sph.SPH_MIXED, MIXED_TOL)])
@pytest.mark.parametrize("cell_scale", [1.0, 3.0, 6.0])
def test_cells_longer_than_a_warp(cell_scale, precision, tol):
    """Level-0 cells of up to about 350 particles: their ends and largest h
    come from beyond the warp that holds their first particle."""
    d = wl.perturbed(nx=61, ny=53, h_ratio=1.5, seed=5)
    pt = d["particles"]
    P = oracle.params(**d["params"])
    ref = oracle.rhs(P, oracle.dt(P, pt["h"]), oracle.make_state(pt))
    c0 = cell_scale * 3.0 * float(pt["h"].min())
    s = _sim(d, precision, cell_c0=c0)
    s.rhs()
    got = by_id(s, ["rho", "dpdt", "dudt", "dvdt", "nnb"])
    s.close()
    assert np.array_equal(got["nnb"], ref["nnb"])
    for f in ("rho", "dpdt", "dudt", "dvdt"):
        assert norm(got[f], ref[f], ref["s_" + f]) <= tol, f


def _row_cases():
    return {"below": wl.taylor_green(nx=219, Re=100.0, jitter=0.1, seed=3),
            "first": wl.taylor_green(nx=220, Re=100.0, jitter=0.1, seed=3),
            "levels": wl.perturbed(nx=251, ny=203, h_ratio=6.0, seed=4),
            "overflow": wl.perturbed(nx=250, ny=200, h_ratio=2.0, hdx=1.7, seed=11),
            "walls": wl.half_plane_walls(nx=401, ny=127, layers=4, dx=0.9 / 127, seed=2),
            "one_lane": wl.graded_strip(n_target=330000, ratio=25.0, seed=6)}


@pytest.mark.parametrize("case", ["below", "first", "levels", "overflow", "walls", "one_lane"])
def test_step_with_rows_matches_the_step_with_plain_lists(case):
    """One mixed step whose passes read own entries from the rows (merged
    walk) and one on plain lists (cell-per-chunk walk), from the same state.
    The lists may differ in entries within rounding of the skin radius,
    which add zeros but move the lanes' shares, so each FP32 sum may round
    apart: within MIXED_TOL of the largest change of the step."""
    d = _row_cases()[case]
    out = []
    for walk in (3, 4):
        s = _sim(d, sph.SPH_MIXED)
        if "walls" in d:
            s.load(d["walls"], kind=sph.SPH_WALL)
        s.set_tuning(walk=walk)
        s.step(1)
        out.append(by_id(s, ["x", "y", "u", "v", "p", "rho", "nnb"]))
        s.close()
    a, b = out
    assert np.array_equal(a["nnb"], b["nnb"])
    for f in ("u", "v", "p", "rho"):
        assert np.abs(a[f] - b[f]).max() <= MIXED_TOL * np.abs(a[f]).max(), f
    for f in ("x", "y"):
        assert np.abs(a[f] - b[f]).max() <= 1e-9, f
