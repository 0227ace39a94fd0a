"""The mixed fit's blocks pass their entries in step, one barrier an entry, up to the longest track of the
block. Every mapping computes a track with the same operations, so the results of blocks of several warps are
those of the kernels that do not wait (64 registers), bit for bit: for blocks that mix lengths, tracks
without measurements or entries, refused and failing tracks, and batches around the edges of a block."""

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HOLE = np.uint32(tkf.SID_NO_MEASUREMENT)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return tkf.Context(0)


def _batch(w):
    """Every 7th track loses all but its first 0 .. 3 entries, every 11th its measurements, every 13th names a
    surface that does not exist, every 17th starts from NaN, every 19th runs along the beam."""
    t, off = w.tracks, w.tracks.offsets.astype(np.int64)
    n = len(off) - 1
    keep = [min(i // 7 % 4, off[i + 1] - off[i]) if i % 7 == 3 else off[i + 1] - off[i] for i in range(n)]
    rows = np.concatenate([np.arange(off[i], off[i] + keep[i]) for i in range(n)])
    offsets = np.concatenate([[0], np.cumsum(keep)]).astype(np.uint32)
    meas, sid = t.meas[rows].copy(), t.sid[rows].copy()
    seed = t.seed_par.copy()
    for i in range(n):
        a, b = offsets[i], offsets[i + 1]
        if i % 11 == 5:
            sid[a:b] |= HOLE
        if i % 13 == 6 and b > a:
            sid[b - 1] = len(w.geometry.table)
        if i % 17 == 8:
            seed[i, 4] = np.nan
        if i % 19 == 9:
            seed[i, 3] = 0.0
    return tkf.Batch.from_arrays(offsets, meas, sid, seed, t.seed_cov).to("cuda:0")


WORKLOADS = {"uniform": lambda n: synth.barrel_workload(n_events=1, lo=n, hi=n, seed=41, pmin=0.2, p_hole=0.1),
             "map": lambda n: synth.solenoid_muon_workload(n, seed=43, p_hole=0.1)}


@pytest.mark.parametrize("field", sorted(WORKLOADS))
@pytest.mark.parametrize("smoother", [tkf.SMOOTHER_RTS, tkf.SMOOTHER_TWO_FILTER])
@pytest.mark.parametrize("n,shape", [(1, (128, 2, 255)), (33, (64, 4, 255)), (127, (128, 4, 128)), (129, (128, 2, 255)),
                                     (300, (256, 1, 255)), (2500, (128, 4, 128)), (2500, (32, 8, 255))])
def test_blocks_in_step(ctx, field, smoother, n, shape):
    w = WORKLOADS[field](n)
    geo, fld, b = tkf.Geometry.from_table(ctx, w.geometry.table), tkf.Field.from_desc(ctx, w.field), _batch(w)
    out = []
    for threads, blocks, regs in (shape, (128, 8, 64)):
        for tpw in (32, 5):
            out.append(tkf.fit(ctx, geo, fld, b, tkf.Options(
                precision=tkf.MIXED, smoother=smoother, mass=w.mass, block_threads=threads, blocks_per_sm=blocks,
                tracks_per_warp=tpw, max_registers=regs)))
    torch.cuda.synchronize()
    if n == 2500:
        status = out[0].status.cpu().numpy().view(np.uint32)
        assert len(np.unique(status)) > 2  # fitted, too few hits, refused
    for r in out[:-1]:
        for k in ("par", "cov", "chi2", "ndf", "status", "steps"):
            np.testing.assert_array_equal(getattr(r, k).cpu().numpy(), getattr(out[-1], k).cpu().numpy(), err_msg=k)


@pytest.mark.parametrize("per_sm,extra", [(56, 0), (56, 1), (1024, 0), (1024, 1)])
def test_the_size_without_tuning(ctx, per_sm, extra):
    """Four lanes a track up to 56 tracks an SM; the full register file up to 4 waves, 128 registers beyond."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    w = synth.telescope_workload(n, seed=22)
    t = w.tracks
    b = tkf.Batch.from_arrays(t.offsets, t.meas, t.sid, t.seed_par, t.seed_cov).to("cuda:0")
    geo, fld = tkf.Geometry.from_table(ctx, w.geometry.table), tkf.Field.from_desc(ctx, w.field)
    a = tkf.fit(ctx, geo, fld, b, tkf.Options(precision=tkf.MIXED, mass=w.mass))
    f = tkf.fit(ctx, geo, fld, b, tkf.Options(precision=tkf.MIXED, mass=w.mass, block_threads=128, blocks_per_sm=8,
                                              max_registers=64))
    torch.cuda.synchronize()
    for k in ("par", "cov", "chi2", "ndf", "status", "steps"):
        np.testing.assert_array_equal(getattr(a, k).cpu().numpy(), getattr(f, k).cpu().numpy(), err_msg=k)
