"""Training on a device that cannot hold a batch's CTAs together: where no cluster can be placed the steps run as a
cooperative launch, where that is refused too, step by step, with the same parameters, losses and step count. The refusals
come from a fake of the two CUDA calls, loaded before the CUDA runtime in a process of its own."""

import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
#include <string.h>
#include <driver_types.h>
static int refuse(const cudaLaunchConfig_t* c) {
  const char* what = getenv("FAKE_REFUSE");
  for (unsigned i = 0; what && i < c->numAttrs; ++i) {
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return 1;
    if (c->attrs[i].id == cudaLaunchAttributeCooperative && !strcmp(what, "all")) return 1;
  }
  return 0;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
  typedef cudaError_t (*Fn)(int*, const void*, const cudaLaunchConfig_t*);
  if (getenv("FAKE_REFUSE") && strcmp(getenv("FAKE_REFUSE"), "launch")) {
    *n = 0;
    return cudaSuccess;
  }
  return ((Fn)dlsym(RTLD_NEXT, "cudaOccupancyMaxActiveClusters"))(n, f, c);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  typedef cudaError_t (*Fn)(const cudaLaunchConfig_t*, const void*, void**);
  if (refuse(c)) return cudaErrorCooperativeLaunchTooLarge;
  return ((Fn)dlsym(RTLD_NEXT, "cudaLaunchKernelExC"))(c, f, args);
}
"""

TRAIN = """
import sys
import numpy as np
import torch
import paper_2505_22822_gb300 as tkf
batch, out = int(sys.argv[1]), sys.argv[2]
ctx = tkf.Context(0)
g = torch.Generator(device="cuda").manual_seed(7)
rec = torch.randn(batch * 300, 13, generator=g, device="cuda")
p = torch.empty(tkf.MLP_PARAMS, device="cuda")
tkf.mlp_init(ctx, p, 3)
mom = torch.zeros(2, tkf.MLP_PARAMS, device="cuda")
loss, t = tkf.mlp_train(ctx, rec, p, mom, 5, batch=batch, epochs=2, lr=2e-3)
np.savez(out, p=p.cpu().numpy(), mom=mom.cpu().numpy(), loss=loss.cpu().numpy(), t=t)
"""


@pytest.mark.parametrize("batch", [100, 1024])
def test_refused_launches(tmp_path, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(tkf.__file__)))
    (tmp_path / "fake.c").write_text(FAKE)
    cuda = os.path.dirname(os.path.dirname(tkf._nvcc()))
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"), "-o", str(tmp_path / "fake.so"),
                           str(tmp_path / "fake.c"), "-ldl"])

    def train(refuse):
        out = str(tmp_path / f"{refuse}.npz")
        env = dict(os.environ, LD_PRELOAD=str(tmp_path / "fake.so"), PYTHONPATH=root)
        env.pop("FAKE_REFUSE", None)
        if refuse:
            env["FAKE_REFUSE"] = refuse
        subprocess.run([sys.executable, "-c", TRAIN, str(batch), out], env=env, cwd=root, check=True, timeout=300)
        return np.load(out)

    want = train(None)
    assert want["t"] == 5 + 600
    # no cluster can be placed; the cluster's launch is refused; every joint launch is refused
    for refuse in ("clusters", "launch", "all"):
        got = train(refuse)
        for k in ("t", "p", "mom", "loss"):
            np.testing.assert_array_equal(got[k], want[k], err_msg=f"{refuse}: {k}")
