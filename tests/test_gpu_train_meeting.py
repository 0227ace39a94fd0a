"""The CTAs of a training batch that is no cluster meet by a counter, whose wait is bounded. With a limit of no polls at all
the first meeting fails: the call returns as usual, with NaN parameters and NaN losses; the next call, with the
library's own limit, trains. The limit is an argument of the library's internal function, called by a few lines of
C++ compiled here."""

import ctypes
import os
import subprocess

import pytest

import paper_2505_22822_gb300 as tkf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALL = r"""
#include "tkf_internal.cuh"
extern "C" size_t scratch_bytes(uint32_t batch) { return tkf::mlp_train_scratch_bytes(batch); }
extern "C" int train(const float* rec, uint32_t n, uint32_t batch, uint32_t epochs, float* p, float* mom, uint32_t* t,
                     float* loss, void* scratch, uint32_t polls) {
  return int(tkf::mlp_train(rec, n, batch, epochs, 2e-3f, 0.9f, 0.999f, 1e-8f, p, mom, t, loss, scratch, nullptr, polls));
}
"""


def test_a_meeting_that_fails_is_seen(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    here = os.path.dirname(os.path.abspath(tkf.__file__))
    tkf.lib()
    (tmp_path / "call.cu").write_text(CALL)
    so = os.path.join(here, "_build", "libtkf.so")
    subprocess.check_call([tkf._nvcc(), *tkf.NVCC_FLAGS, "-shared", "-cudart", "shared", "-I", os.path.join(here, "csrc"), "-I",
                           os.path.join(os.path.dirname(here), "include"), "-o", str(tmp_path / "call.so"),
                           str(tmp_path / "call.cu"), so, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(so)])
    call = ctypes.CDLL(str(tmp_path / "call.so"))
    call.scratch_bytes.restype = ctypes.c_size_t
    batch, batches, epochs = 1200, 4, 3  # ten CTAs: no cluster
    ctx = tkf.Context(0)
    rec = torch.randn(batch * batches, 13, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    scratch = torch.empty(call.scratch_bytes(batch), dtype=torch.uint8, device="cuda")

    def train(polls):
        p = torch.empty(tkf.MLP_PARAMS, device="cuda")
        tkf.mlp_init(ctx, p, 3)
        mom, loss = torch.zeros(2, tkf.MLP_PARAMS, device="cuda"), torch.zeros(epochs, device="cuda")
        t = ctypes.c_uint32(0)
        torch.cuda.synchronize()
        rc = call.train(ctypes.c_void_p(rec.data_ptr()), batch * batches, batch,
                        epochs, *(ctypes.c_void_p(x.data_ptr()) for x in (p, mom)), ctypes.byref(t),
                        *(ctypes.c_void_p(x.data_ptr()) for x in (loss, scratch)), ctypes.c_uint32(polls))
        torch.cuda.synchronize()
        assert rc == 0 and t.value == batches * epochs
        return p, loss

    p, loss = train(0)
    assert torch.isnan(p).all() and torch.isnan(loss).all()
    p, loss = train(1 << 22)
    assert torch.isfinite(p).all() and torch.isfinite(loss).all()
    want = torch.empty_like(p)
    tkf.mlp_init(ctx, want, 3)
    tkf.mlp_train(ctx, rec, want, torch.zeros(2, tkf.MLP_PARAMS, device="cuda"), 0, batch=batch, epochs=epochs, lr=2e-3)
    assert torch.equal(p, want)
