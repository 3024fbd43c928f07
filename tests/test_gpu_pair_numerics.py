"""Arithmetic of the pair sums where it could leave its range: separations
whose square is no normal number."""
import numpy as np
import pytest

import oracle
from paper_2107_01276_gb300 import sph
from paper_2107_01276_gb300 import workloads as wl
from tests.helpers import FP64_TOL, by_id, cuda_ok, norm, stream_handle

pytestmark = pytest.mark.gpu
RHS = ("rho", "beta", "pavg", "drx", "dry", "dpdt", "dudt", "dvdt")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not cuda_ok():
        pytest.skip("no CUDA device")


def _close_pair(r):
    """A periodic set without walls, one pair of it r apart on the edge
    x = 0."""
    d = wl.perturbed(nx=24, ny=24, h_ratio=1.0, jitter=0.1, hdx=1.2, seed=12)
    pt = d["particles"]
    pt["x"][0], pt["x"][1] = 0.0, r
    pt["y"][1] = pt["y"][0]
    return d


@pytest.mark.parametrize("r", [1e-153, 1.6e-154, 1.2e-154, 1e-157, 1e-161, 1e-170])
def test_fp64_rates_of_nearly_coincident_particles(r):
    """r^2 normal, subnormal and zero."""
    d = _close_pair(r)
    pt = d["particles"]
    P = sph.make_params(d["params"], precision=sph.SPH_FP64, capacity=len(pt["x"]))
    with sph.Simulation(P, stream_handle()) as s:
        s.load(pt)
        s.rhs()
        got = by_id(s, RHS + ("nnb",))
    OP = oracle.params(**d["params"])
    ref = oracle.rhs(OP, oracle.dt(OP, pt["h"]), oracle.make_state(pt))
    assert np.array_equal(got["nnb"], ref["nnb"])
    for f in RHS:
        assert norm(got[f], ref[f], ref["s_" + f]) <= FP64_TOL, f


@pytest.mark.parametrize("r", [1e-153, 1e-157, 1e-170])
def test_fp64_shift_and_h_of_nearly_coincident_particles(r):
    """sph_adapt whose background asks for the sizes that are there: no
    split, no merge, three shift rounds and the h update."""
    d = _close_pair(r)
    pt = d["particles"]
    n = len(pt["x"])
    g = (np.arange(24) + 0.5) / 24
    X, Y = np.meshgrid(g, g, indexing="xy")
    bg = {"x": X.ravel(), "y": Y.ravel(), "h": np.full(n, 1.2 / 24), "ds": np.full(n, d["dx"])}
    P = sph.make_params(d["params"], precision=sph.SPH_FP64, capacity=n)
    with sph.Simulation(P, stream_handle()) as s:
        s.load(pt)
        s.load(bg, kind=sph.SPH_BACKGROUND)
        z = s.adapt()
        got = by_id(s, ("x", "y", "h", "u", "v", "p", "rho"))
    st = oracle.make_state(pt, cap=n)
    _, o, _ = oracle.adapt(oracle.params(**d["params"]), st, bg=bg)
    assert (z["n_split"], z["n_merged"]) == (o["n_split"], o["n_merged"]) == (0, 0)
    order = np.argsort(st["id"][:n])
    for f in ("x", "y", "h", "u", "v", "p", "rho"):
        ref = st[f][:n][order]
        e = got[f] - ref
        if f in "xy":
            e -= np.round(e)
        scale = pt["h"].max() if f in "xy" else np.abs(ref).max()
        assert np.abs(e).max() <= 1e-11 * scale, f
