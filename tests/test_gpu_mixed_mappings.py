"""The mixed fit computes a track with the same operations whatever the mapping of tracks to lanes, the register cap and
the smoother's output: the results in a uniform field in any direction are the same bits."""

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MAPPINGS = {"255": dict(max_registers=255), "128": dict(max_registers=128), "four lanes": dict(lanes_per_track=4),
            "one warp": dict(block_threads=32, blocks_per_sm=8), "by size": {}, "states": {}}


@pytest.mark.parametrize("B", [(0.3, -0.2, 1.9), (0.0, 2.0, 0.0)])
@pytest.mark.parametrize("smoother", [tkf.SMOOTHER_RTS, tkf.SMOOTHER_TWO_FILTER])
@pytest.mark.parametrize("n", [300, 10_000])
def test_tilted_field(B, smoother, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = tkf.Context(0)
    w = synth.barrel_workload(n_events=1, lo=n, hi=n, seed=33)
    t = w.tracks
    b = tkf.Batch.from_arrays(t.offsets, t.meas, t.sid, t.seed_par, t.seed_cov).to("cuda:0")
    geo = tkf.Geometry.from_table(ctx, w.geometry.table)
    fld = tkf.Field.from_desc(ctx, synth.Field(kind=0, B=B))

    def fit(states=False, **kw):
        r = tkf.fit(ctx, geo, fld, b, tkf.Options(precision=tkf.MIXED, smoother=smoother, mass=w.mass, **kw), states=states)
        torch.cuda.synchronize()
        return {k: getattr(r, k).cpu().numpy() for k in ("par", "cov", "chi2", "ndf", "status", "steps")}

    want = fit(max_registers=64)
    assert (want["status"] == 0).mean() > 0.5
    for name, kw in MAPPINGS.items():
        if smoother == tkf.SMOOTHER_TWO_FILTER and name in ("four lanes", "states"):
            continue  # refused
        got = fit(name == "states", **kw)
        for k in want:
            np.testing.assert_array_equal(got[k], want[k], err_msg=f"{name}: {k}")
