"""Seed angles come from a table-driven arc tangent: directions in and on the borders of every octant,
both senses of turning, arcs from a thousandth of a turn to most of one, steep and flat, and lengths
from microns to kilometres (beyond the FP32 range of the circle's squares), against the oracle."""

import numpy as np
import pytest

import oracle
import paper_2505_22822_gb300 as tkf
import synth
from tests.test_gpu_seed import compare_seeds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = np.finfo(float).eps


@pytest.mark.parametrize("radius", [1e-2, 1e3, 1e6, 1e17])
@pytest.mark.parametrize("cot", [0.0, 1e-3, -1.0, 40.0])
def test_every_octant_and_scale(radius, cot):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # points on a circle of this radius, in planes at the helix's z (u = x, v = y)
    phi, turn, arc = (x.ravel() for x in np.meshgrid(np.arange(16) * np.pi / 8, [-1.0, 1.0], [6e-3, 1.0, 3.0, 5.5]))
    pts, z = [], []
    for part in (0.0, 0.4, 1.0):
        a = part * arc
        pts.append(radius * turn[:, None] * np.stack([np.sin(phi + turn * a) - np.sin(phi), np.cos(phi) - np.cos(phi + turn * a)], 1))
        z.append(radius * a * cot)
    n = len(phi)
    loc, zz = np.stack(pts, 1).reshape(-1, 2), np.stack(z, 1).ravel()
    table = np.zeros((3 * n, 16))
    table[:, 0] = table[:, 4] = table[:, 8] = 1.0
    table[:, 11], table[:, 12], table[:, 13] = zz, 0.3, 93.7
    meas = np.concatenate([loc, np.tile([1e-4, 0.0, 1e-4], (3 * n, 1))], 1)
    sid, offsets = np.arange(3 * n, dtype=np.uint32), np.arange(0, 3 * n + 1, 3).astype(np.uint32)
    field = synth.uniform_field(2.0)
    ctx = tkf.Context(0)
    b = tkf.Batch.from_arrays(offsets, meas, sid, np.zeros((n, 5)), np.zeros((n, 15))).to("cuda:0")
    r = tkf.estimate_seeds(ctx, tkf.Geometry.from_table(ctx, table), tkf.Field.from_desc(ctx, field), b)
    torch.cuda.synchronize()
    got = r.par.cpu().numpy().T, r.cov.cpu().numpy().T, r.status.cpu().numpy().view(np.uint32)
    want = oracle.estimate_seeds(table, oracle.field_from(field), offsets, meas, sid)
    assert np.all(want[2] == 0)
    # one ulp of the coordinates moves the curvature by eps |r| / sagitta, sagitta = R (1 - cos(arc / 2))
    compare_seeds(got, want, 1e-10 + 1e3 * EPS * 2.0 / (1.0 - np.cos(arc / 2)))
