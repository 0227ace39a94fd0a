"""Seed estimation from points without a direction: three equal points, two equal ones, and points above one another
along the field. Status, q/p and covariance are the oracle's (q/p 0, the wide variances), also where an angle is NaN."""

import numpy as np
import pytest

import oracle
import paper_2505_22822_gb300 as tkf
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bz", [2.0, 0.0])
def test_points_without_a_direction(bz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    geom, field = synth.telescope_geometry(n_planes=3), synth.uniform_field(bz)
    # surfaces, then (y, z) on them: equal points, the last two equal, a line along z in one plane, an ordinary track
    tracks = [((0, 0, 0), [(3.0, 2.0)] * 3), ((0, 1, 1), [(3.0, 2.0)] * 3), ((0, 0, 0), [(3.0, 0.0), (3.0, 5.0), (3.0, 9.0)]),
              ((0, 1, 2), [(0.0, 0.0), (1.0, 2.0), (3.0, 4.0)])]
    sid = np.concatenate([s for s, _ in tracks]).astype(np.uint32)
    loc = np.concatenate([p for _, p in tracks])
    meas = np.concatenate([loc, np.tile([1e-4, 0.0, 1e-4], (len(loc), 1))], 1)
    n = len(tracks)
    offsets = np.arange(0, 3 * n + 1, 3).astype(np.uint32)
    ctx = tkf.Context(0)
    b = tkf.Batch.from_arrays(offsets, meas, sid, np.zeros((n, 5)), np.zeros((n, 15))).to("cuda:0")
    r = tkf.estimate_seeds(ctx, tkf.Geometry.from_table(ctx, geom.table), tkf.Field.from_desc(ctx, field), b)
    torch.cuda.synchronize()
    par, cov, status = oracle.estimate_seeds(geom.table, oracle.field_from(field), offsets, meas, sid)
    np.testing.assert_array_equal(r.status.cpu().numpy().view(np.uint32), status)
    np.testing.assert_allclose(r.par.cpu().numpy().T, par, rtol=1e-12, atol=1e-15)
    np.testing.assert_allclose(r.cov.cpu().numpy().T, cov, rtol=1e-12)
