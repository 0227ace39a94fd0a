"""A large mixed call of track finding predicts its branches with the block's queue, in step; a small one tries
module after module. Every branch is predicted with the same operations: the candidates of a seed list repeated
until it takes the queue are those of the list on its own, bit for bit, with beams of one to eight, seeds on
missing surfaces, seeds off the detector and short entry limits among them."""

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf
import synth
from tests.test_gpu_ckf import _seeds, gpu_find

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("workload,beam,max_entries", [("pions", 3, 24), ("pions", 1, 5), ("map", 8, 24)])
def test_queue_finds_the_same_candidates(workload, beam, max_entries):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = tkf.Context(0)
    w = (synth.barrel_workload(n_events=1, lo=2900, hi=2900, seed=37, pmin=0.2) if workload == "pions"
         else synth.solenoid_muon_workload(1000, seed=13))
    mc = synth.measurement_container(w.tracks, w.geometry.n)
    sid, par, cov, _ = _seeds(w)
    sid, par = sid.copy(), par.copy()
    n = len(sid)
    sid[7::50] = w.geometry.n  # no such surface
    par[11::60, 0] += 5e3  # far off the module
    par[13::70, 4] *= 40.0  # stopped by the material, or curling
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = 8 * 128 * sms // (n * beam) + 2  # beyond two waves of up to four blocks an SM
    kw = dict(precision=tkf.MIXED, beam=beam, max_entries=max_entries)
    small = gpu_find(ctx, w, mc, sid, par, cov, **kw)
    large = gpu_find(ctx, w, mc, np.tile(sid, copies), np.tile(par, (copies, 1)), np.tile(cov, (copies, 1)), **kw)
    assert 0 < (small["n_entries"] == 0).sum() < n
    for k in small:
        for c in range(copies):
            np.testing.assert_array_equal(large[k][c * n:(c + 1) * n], small[k], err_msg=k)
