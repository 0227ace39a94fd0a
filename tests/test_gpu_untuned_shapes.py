"""The launch shape without tuning depends on the batch's size: on both sides of every line the results
are those of one fixed shape, bit for bit (mixed and FP64 in a field along z; every mapping computes a
track with the same operations)."""

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = tkf.Context(0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = synth.telescope_workload(10 * 256 * sms // 4 + 100, seed=21)  # beyond 1.75 waves
    t = w.tracks
    b = tkf.Batch.from_arrays(t.offsets, t.meas, t.sid, t.seed_par, t.seed_cov).to("cuda:0")
    return ctx, sms, tkf.Geometry.from_table(ctx, w.geometry.table), tkf.Field.from_desc(ctx, w.field), b, w.mass


def _first(b, n):
    m = int(b.offsets[n])
    return tkf.Batch(b.offsets[:n + 1].contiguous(), *(x[:m].contiguous() for x in (b.loc0, b.loc1, b.v00, b.v01, b.v11, b.sid)),
                     b.seed_par[:, :n].contiguous(), b.seed_cov[:, :n].contiguous())


@pytest.mark.parametrize("precision", [tkf.FP64, tkf.MIXED])
@pytest.mark.parametrize("smoother", [tkf.SMOOTHER_RTS, tkf.SMOOTHER_TWO_FILTER])
@pytest.mark.parametrize("per_sm,extra", [(0, 1), (1, 0), (1, 1), (4, 1), (80, 0), (80, 1), (256, -31), (448, 0), (448, 1)])
def test_both_sides_of_every_line(case, precision, smoother, per_sm, extra):
    ctx, sms, geo, fld, b, mass = case
    b = _first(b, per_sm * sms + extra)
    fixed = tkf.Options(precision=precision, smoother=smoother, mass=mass, block_threads=128, blocks_per_sm=2)
    a = tkf.fit(ctx, geo, fld, b, tkf.Options(precision=precision, smoother=smoother, mass=mass))
    f = tkf.fit(ctx, geo, fld, b, fixed)
    torch.cuda.synchronize()
    for k in ("par", "cov", "chi2", "ndf", "status", "steps"):
        np.testing.assert_array_equal(getattr(a, k).cpu().numpy(), getattr(f, k).cpu().numpy(), err_msg=k)


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 8191, 8192, 8193, 9216])
def test_ordering_by_one_block_or_many(case, n):
    """Up to 8,192 tracks one block orders the batch; every track is fitted once on both sides of that."""
    ctx, _, geo, fld, b, mass = case
    opts = tkf.Options(precision=tkf.MIXED, mass=mass)
    a, f = tkf.fit(ctx, geo, fld, _first(b, n), opts), tkf.fit(ctx, geo, fld, _first(b, 10_000), opts)
    torch.cuda.synchronize()
    for k in ("par", "cov", "chi2", "ndf", "status", "steps"):
        np.testing.assert_array_equal(getattr(a, k).cpu().numpy(), getattr(f, k)[..., :n].cpu().numpy(), err_msg=k)
