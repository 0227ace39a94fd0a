"""The FP64 fit in a field along z steps by closed-form polynomials of the RKN4 map; a field that
points anywhere else takes the stage-by-stage form. Both against the oracle at the parity tolerance
(tests/parity.py) where the closed form could go wrong: both signs of the field and none, curling low
momenta, forward tracks, holes, ragged warps, zero q/p, and every mapping of tracks to lanes."""

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf
import synth
from tests import parity
from tests.test_gpu_parity import TOL64, check, run_gpu, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return tkf.Context(0)


def _tilted(w):
    """The same workload with a field direction the closed form does not take (1e-200 T along x)."""
    f = synth.Field(kind=0, B=(1e-200, 0.0, w.field.B[2]))
    return synth.Workload(w.name, w.geometry, f, w.tracks, w.mass)


@pytest.mark.parametrize("n,bz,pmin,pmax", [(1, 2.0, 0.5, 100.0), (33, -2.0, 0.5, 1.0), (700, 2.0, 0.2, 0.6),
                                            (500, -0.5, 0.1, 50.0), (300, 1e-6, 0.5, 5.0)])
def test_closed_form_steps_match_the_oracle_and_the_stages(ctx, n, bz, pmin, pmax):
    w = synth.barrel_workload(n_events=1, lo=n, hi=n, seed=31 + n, fld=synth.uniform_field(bz), pmin=pmin, pmax=pmax,
                              p_hole=0.1)
    o = run_oracle(w)
    g, s = run_gpu(ctx, w), run_gpu(ctx, _tilted(w))
    check(g, o, TOL64, w=w, tracks=np.arange(n))
    np.testing.assert_array_equal(g["status"], s["status"])
    np.testing.assert_array_equal(g["steps"], s["steps"])


@pytest.mark.parametrize("smoother", [tkf.SMOOTHER_RTS, tkf.SMOOTHER_TWO_FILTER])
def test_without_curvature(ctx, smoother):
    """No field, and q/p = 0 through planes without material: straight lines, no error estimate."""
    w = synth.telescope_workload(65, seed=9)
    geom = synth.telescope_geometry(thickness=0.0)
    w.tracks.seed_par[::2, 4] = 0.0
    for bz in (0.0, 2.0):
        v = synth.Workload(w.name, geom, synth.uniform_field(bz), w.tracks, w.mass)
        opts = tkf.Options(mass=w.mass, smoother=smoother)
        g, s = run_gpu(ctx, v, opts=opts), run_gpu(ctx, _tilted(v), opts=opts)
        np.testing.assert_array_equal(g["status"], s["status"])
        np.testing.assert_array_equal(g["steps"], s["steps"])
        sig = np.sqrt(np.abs(np.stack([s["cov"][:, k] for k in (0, 5, 9, 12, 14)], 1)))
        assert np.nanmax(np.abs(g["par"] - s["par"]) / np.maximum(np.abs(s["par"]), sig)) <= TOL64


@pytest.mark.parametrize("opts", [dict(lanes_per_track=4), dict(max_registers=128), dict(max_registers=64),
                                  dict(tracks_per_warp=3)])
def test_every_mapping_gives_the_same_bits(ctx, opts):
    w = synth.barrel_workload(n_events=1, lo=333, hi=333, seed=5, p_hole=0.1)
    a, b = run_gpu(ctx, w), run_gpu(ctx, w, opts=tkf.Options(mass=w.mass, **opts))
    if opts.get("max_registers"):  # other register caps may fuse the general code's sums differently
        ok, same, stats = parity.compare(b, run_oracle(w), TOL64)
        assert ok.all() and same.all(), stats
        return
    for k in ("par", "cov", "chi2", "status", "steps"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
