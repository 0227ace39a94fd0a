"""The warps of a block of the mixed fit pass their entries in step, but wait for one another only a while: tracks that
curl for thousands of steps towards a plane they never reach, each in its own warp and at its own entry, take no
longer together than the longest of them, as in blocks of one warp."""

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ENTRIES = 9


def _curling(n):
    """Track i stays on the first plane for 1 + i mod 8 entries, then heads for the last, 400 mm away, on a circle of 83 mm."""
    geom = synth.telescope_geometry(thickness=0.0)
    t = synth.telescope_workload(n, seed=4).tracks
    sid = np.zeros((n, ENTRIES), np.uint32)
    for i in range(n):
        sid[i, 1 + i % 8:] = geom.n - 1
    sid[:, 1:] |= np.uint32(tkf.SID_NO_MEASUREMENT)
    meas = np.repeat(t.meas[t.offsets[:-1].astype(np.int64)], ENTRIES, axis=0)
    seed = t.seed_par.copy()
    seed[:, 4] = 1.0 / 0.05
    offsets = (ENTRIES * np.arange(n + 1)).astype(np.uint32)
    return geom, tkf.Batch.from_arrays(offsets, meas, sid.ravel(), seed, t.seed_cov).to("cuda:0")


@pytest.mark.parametrize("smoother", [tkf.SMOOTHER_RTS, tkf.SMOOTHER_TWO_FILTER])
@pytest.mark.parametrize("threads,registers", [(128, 255), (128, 128), (256, 255)])
def test_warps_wait_a_while(smoother, threads, registers):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = tkf.Context(0)
    geom, b = _curling(threads // 32)
    geo, fld = tkf.Geometry.from_table(ctx, geom.table), tkf.Field.from_desc(ctx, synth.uniform_field(2.0))

    def run(block):
        o = tkf.Options(precision=tkf.MIXED, smoother=smoother, block_threads=block, blocks_per_sm=1, tracks_per_warp=1,
                        max_registers=registers)
        times = []
        for _ in range(4):
            begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            begin.record()
            r = tkf.fit(ctx, geo, fld, b, o)
            end.record()
            torch.cuda.synchronize()
            times.append(begin.elapsed_time(end))
        return min(times), r

    alone, want = run(32)
    together, got = run(threads)
    assert np.all(want.steps.cpu().numpy()[0] >= 10_000) and np.all(want.status.cpu().numpy() != 0)
    for k in ("status", "steps"):
        np.testing.assert_array_equal(getattr(got, k).cpu().numpy(), getattr(want, k).cpu().numpy(), err_msg=k)
    assert together < 1.5 * alone, (together, alone)


def test_a_small_batch_reaches_every_sm():
    """A block takes the shares of its warps at once; 600 tracks in blocks of four warps are spread over the SMs as if
    a warp asked for one track, not handed to five blocks."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = tkf.Context(0)
    w = synth.solenoid_muon_workload(600, seed=35)
    t = w.tracks
    b = tkf.Batch.from_arrays(t.offsets, t.meas, t.sid, t.seed_par, t.seed_cov).to("cuda:0")
    geo, fld = tkf.Geometry.from_table(ctx, w.geometry.table), tkf.Field.from_desc(ctx, w.field)

    def run(**kw):
        o = tkf.Options(precision=tkf.MIXED, mass=w.mass, block_threads=128, blocks_per_sm=4, max_registers=128, **kw)
        times = []
        for _ in range(21):
            begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            begin.record()
            tkf.fit(ctx, geo, fld, b, o)
            end.record()
            torch.cuda.synchronize()
            times.append(begin.elapsed_time(end))
        return sorted(times)[10]

    run()
    spread, default = run(tracks_per_warp=1), run()
    assert default < 1.12 * spread, (default, spread)
