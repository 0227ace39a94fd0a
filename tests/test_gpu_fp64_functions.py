"""The reciprocal, root, logarithm and arc tangent that stand for CUDA's on the FP64 path (tkf_fp64.cuh), over the ranges
they are called with and at the borders of their tables, octants and fallbacks, against long double: the bounds that
their comments state, in units in the last place of the exact result."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALL = r"""
#include "tkf_fp64.cuh"
__global__ void run(int f, const double* x, const double* y, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = f == 0 ? tkf::rcp_nr(x[i]) : f == 1 ? tkf::rsqrt_nr(x[i]) : f == 2 ? tkf::log_nr(x[i]) : tkf::atan2_nr(y[i], x[i]);
}
extern "C" int call(int f, const double* x, const double* y, double* out, int n) {
  run<<<(n + 255) / 256, 256>>>(f, x, y, out, n);
  return int(cudaDeviceSynchronize());
}
"""
L = np.longdouble


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(L).nmant < 63:
        pytest.skip("long double is no wider than double here")
    d = tmp_path_factory.mktemp("fp64")
    (d / "call.cu").write_text(CALL)
    here = os.path.dirname(os.path.abspath(tkf.__file__))
    subprocess.check_call([tkf._nvcc(), *tkf.NVCC_FLAGS, "-shared", "-cudart", "shared", "-I", os.path.join(here, "csrc"),
                           "-o", str(d / "call.so"), str(d / "call.cu")])
    lib = ctypes.CDLL(str(d / "call.so"))

    def run(f, x, y=None):
        x = torch.from_numpy(np.ascontiguousarray(x, np.float64)).cuda()
        y = torch.from_numpy(np.ascontiguousarray(y, np.float64)).cuda() if y is not None else x
        out = torch.empty_like(x)
        torch.cuda.synchronize()
        assert lib.call(f, *(ctypes.c_void_p(t.data_ptr()) for t in (x, y, out)), x.numel()) == 0
        return out.cpu().numpy()

    return run


def ulps(got, exact):
    """|got - exact| in units in the last place of the exact value."""
    unit = np.spacing(np.abs(exact).astype(np.float64))
    return np.abs((got.astype(L) - exact) / unit.astype(L)).astype(np.float64)


def with_neighbours(x):
    return np.concatenate([x, np.nextafter(x, np.inf), np.nextafter(x, -np.inf)])


def magnitudes(rng, n, lo, hi):
    """n values with exponents in [lo, hi] and random mantissas, and the powers of two with their neighbours"""
    return np.concatenate([np.ldexp(rng.uniform(1, 2, n), rng.integers(lo, hi + 1, n)), with_neighbours(np.ldexp(1.0, np.arange(lo, hi + 1)))])


def test_reciprocal_and_root(call):
    rng = np.random.default_rng(1)
    x = magnitudes(rng, 2_000_000, -960, 960)
    for s in (x, -x):
        e = ulps(call(0, s), 1 / s.astype(L))
        assert e.max() <= 1.0, e.max()
    # the product x y is rounded once before the remainder (half a unit), the result once more
    e = ulps(call(1, x), 1 / np.sqrt(x.astype(L)))
    assert e.max() <= 1.1, e.max()


def test_logarithm(call):
    rng = np.random.default_rng(2)
    cells = with_neighbours(1 + np.arange(128) / 128)  # the table's cells, in every octave of the callers' range
    x = np.concatenate([np.exp(rng.uniform(-40, 40, 3_000_000)), np.ldexp(cells[:, None], np.arange(-58, 58)).ravel(),
                        1 + rng.uniform(-1e-3, 1e-3, 100_000)])
    exact = np.log(x.astype(L))
    got = call(2, x)
    large = np.abs(exact) >= 4
    assert ulps(got, exact)[large & (np.abs(exact) <= 40)].max() <= 1.2
    assert np.abs(got - exact)[~large].astype(np.float64).max() <= 2.0 ** -50
    # beyond the normal numbers CUDA's log
    odd = call(2, np.array([0.0, -0.0, 5e-324, np.inf, -1.0, np.nan]))
    np.testing.assert_array_equal(odd, [-np.inf, -np.inf, np.log(5e-324), np.inf, np.nan, np.nan])


def test_arc_tangent(call):
    rng = np.random.default_rng(3)
    a = rng.uniform(-np.pi, np.pi, 2_000_000)
    r = 10.0 ** rng.uniform(-12, 12, a.size)
    x, y = [r * np.cos(a)], [r * np.sin(a)]
    t = with_neighbours(np.arange(1, 33) / 32)  # cell centres and borders, the diagonal
    for sx in (1.0, -1.0):
        for sy in (1.0, -1.0):
            x += [np.full(t.shape, sx), sx * t]
            y += [sy * t, np.full(t.shape, sy)]
    tiny = 10.0 ** rng.uniform(-35, 35, (2, 200_000)) * rng.choice([-1, 1], (2, 200_000))  # across the fallback's limits
    x, y = np.concatenate(x + [tiny[0]]), np.concatenate(y + [tiny[1]])
    # CUDA's own atan2 beyond the limits: 2 units
    own = (np.maximum(np.abs(x), np.abs(y)) > 1.001e-30) & (np.abs(x) < 0.999e30) & (np.abs(y) < 0.999e30)
    e = ulps(call(3, x, y), np.arctan2(y.astype(L), x.astype(L)))
    assert e[own].max() <= 1.9, e[own].max()
    assert e.max() <= 2.0, e.max()
    z = np.array([0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan])
    x, y = (v.ravel() for v in np.meshgrid(z, z))
    got, want = call(3, x, y), np.arctan2(y, x)
    np.testing.assert_allclose(got, want, rtol=4e-16)
    np.testing.assert_array_equal(np.signbit(got[~np.isnan(got)]), np.signbit(want[~np.isnan(want)]))
