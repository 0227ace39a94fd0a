"""The lines of the launch shape by size: four lanes a track up to 56 tracks an SM (RTS), and for the mixed fit the full
register file up to 1,024 tracks an SM, 128 registers beyond. On both sides of each, in both precisions and with both
smoothers, the results are those of one fixed shape, bit for bit, and so are those of the allocation-free fit, which
keeps the two-filter smoother at the full register file."""

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
    w = synth.telescope_workload(1024 * sms + 1, seed=23)
    t = w.tracks
    b = tkf.Batch.from_arrays(t.offsets, t.meas, t.sid, t.seed_par, t.seed_cov).to("cuda:0")
    return ctx, sms, tkf.Geometry.from_table(ctx, w.geometry.table), tkf.Field.from_desc(ctx, w.field), b, w.mass


@pytest.mark.parametrize("precision", [tkf.FP64, tkf.MIXED])
@pytest.mark.parametrize("smoother", [tkf.SMOOTHER_RTS, tkf.SMOOTHER_TWO_FILTER])
@pytest.mark.parametrize("per_sm,extra", [(56, 0), (56, 1), (1024, 0), (1024, 1)])
def test_both_sides(case, precision, smoother, per_sm, extra):
    ctx, sms, geo, fld, b, mass = case
    n = per_sm * sms + extra
    m = int(b.offsets[n])
    b = tkf.Batch(b.offsets[:n + 1].contiguous(), *(x[:m].contiguous() for x in (b.loc0, b.loc1, b.v00, b.v01, b.v11, b.sid)),
                  b.seed_par[:, :n].contiguous(), b.seed_cov[:, :n].contiguous())
    opts = tkf.Options(precision=precision, smoother=smoother, mass=mass)
    fixed = tkf.Options(precision=precision, smoother=smoother, mass=mass, block_threads=128, blocks_per_sm=2)
    want, sized = tkf.fit(ctx, geo, fld, b, fixed), tkf.fit(ctx, geo, fld, b, opts)
    free = tkf.fit_noalloc(ctx, geo, fld, b, tkf.alloc_outputs(n, b.offsets.device), opts)
    torch.cuda.synchronize()
    assert (want.status == 0).all()
    for name, got in (("sized", sized), ("allocation-free", free)):
        for k in ("par", "cov", "chi2", "ndf", "status", "steps"):
            np.testing.assert_array_equal(getattr(got, k).cpu().numpy(), getattr(want, k).cpu().numpy(), err_msg=f"{name}: {k}")
