"""The FP64 field-map lookup finds its cell from an FP32 estimate and its radius from a reciprocal
square root: exact nodes, the last cell, both ends of z and points just outside, through the seed
estimation (whose q/p is the mean field at three points) against the oracle."""

import numpy as np
import pytest

import oracle
import paper_2505_22822_gb300 as tkf
import synth
from tests.test_gpu_seed import compare_seeds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

Z_EDGE = 3500.0


def _tracks(offset):
    """Three points a track on planes x = 0, 50 .. 1200 mm, y on the first two off the axis: the third
    at every node radius up to the map's edge, z on nodes, at the edges and `offset` beyond them."""
    sid, loc = [], []
    for last in range(2, 25):
        for z in (0.0, 5.0, -1235.0, Z_EDGE, -Z_EDGE, Z_EDGE + offset, -Z_EDGE - offset, 2.5, np.nextafter(5.0, 0)):
            sid += [0, last // 2, last]
            loc += [(3.0, z - 20.0 * np.sign(z)), (0.0, z - 10.0 * np.sign(z)), (0.0, z)]
    return np.array(sid, np.uint32), np.array(loc)


@pytest.mark.parametrize("offset", [1e-9, 4.0])
def test_lookup_on_nodes_and_at_the_edges(offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = tkf.Context(0)
    geom, field = synth.telescope_geometry(n_planes=25, spacing=50.0), synth.solenoid_map()
    sid, loc = _tracks(offset)
    meas = np.concatenate([loc, np.tile([1e-4, 0.0, 1e-4], (len(loc), 1))], 1)
    offsets = np.arange(0, len(sid) + 1, 3).astype(np.uint32)
    n = len(offsets) - 1
    b = tkf.Batch.from_arrays(offsets, meas, sid, np.zeros((n, 5)), np.zeros((n, 15))).to("cuda:0")
    r = tkf.estimate_seeds(ctx, tkf.Geometry.from_table(ctx, geom.table), tkf.Field.from_desc(ctx, field), b)
    torch.cuda.synchronize()
    got = r.par.cpu().numpy().T, r.cov.cpu().numpy().T, r.status.cpu().numpy().view(np.uint32)
    want = oracle.estimate_seeds(geom.table, oracle.field_from(field), offsets, meas, sid)
    # the three points' sagitta is above 0.5 mm at radii up to 1.2 m: 1e-10 holds in q/p
    compare_seeds(got, want, np.full(n, 1e-10))
