"""The FP64 step's 1 / x, |F| and 1 / |F| (pair_tile.cuh: recip_density, norm_of) against quotients and
roots in numpy's long double (64 or more bits), in a kernel of the test's own that includes the header.

Bounds, in half-ulps (2^-53 relative), from the steps' own roundings: 1 / x rounds once (1; the cube of
the approximation's error, about 2^-60, and the roundings of e + e^2 stay below 0.1), 1 / |F| takes half
of the rounding of F2 y besides (1.5), |F| = F2 / |F| one more (2.5)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2412_14859_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pair_tile.cuh"
__global__ void k(const double* x, double* r, double* n, double* in, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  r[i] = cgevap::recip_density(x[i]);
  n[i] = in[i] = 0.0;
  if (x[i] > 0.0) cgevap::norm_of(x[i], n[i], in[i]);
}
extern "C" __attribute__((visibility("default"))) int evaluate(const double* x, double* r, double* n, double* in, int count) {
  k<<<(count + 255) / 256, 256>>>(x, r, n, in, count);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64")
    (d / "k.cu").write_text(SOURCE)
    subprocess.check_call([build.NVCC] + build.ARCH + build.FLAGS + ["-I", build.SRC, "-shared", "-cudart", "shared",
                          str(d / "k.cu"), "-o", str(d / "k.so")])
    lib = ctypes.CDLL(str(d / "k.so"))

    def call(x):
        t = torch.from_numpy(np.ascontiguousarray(x, np.float64)).cuda()
        out = [torch.empty_like(t) for _ in range(3)]
        torch.cuda.synchronize()
        p = [ctypes.c_void_p(v.data_ptr()) for v in [t] + out]
        assert lib.evaluate(*p, ctypes.c_int(t.numel())) == 0
        return [v.cpu().numpy() for v in out]
    return call


def half_ulps(got, want):
    return float(np.max(np.abs(got.astype(np.longdouble) - want) / np.abs(want)) * np.longdouble(2.0) ** 53)


def mantissas(n, seed):
    """n values over [1, 2): evenly spread, with the ends and the places next to them."""
    g = np.random.default_rng(seed)
    m = 1.0 + (np.arange(n) + g.random(n)) / n
    ends = [1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0), 1.5, np.sqrt(2.0), 4.0 / 3.0]
    return np.concatenate([np.minimum(m, np.nextafter(2.0, 1.0)), ends])


def test_reciprocal(evaluate):
    x = np.concatenate([mantissas(1 << 17, 1) * 2.0 ** e for e in (-4, -1, 0, 1, 7)] +
                       [mantissas(64, 2) * np.ldexp(1.0, e) for e in range(-1022, 1022, 11)] +
                       [np.ldexp([1.0, np.nextafter(2.0, 1.0)], e) for e in (-1022, 1021)] + [[2.0 ** 1022]])
    for v in (x, -x):
        assert half_ulps(evaluate(v)[0], 1 / v.astype(np.longdouble)) <= 1.1


def test_reciprocal_where_it_or_its_argument_is_subnormal(evaluate):
    x = np.array([6e-309, 1e-308, 2.2e-308, np.nextafter(2.0 ** -1022, 0), 2.0 ** 1022, np.nextafter(2.0 ** 1022, np.inf),
                  4.6e307, 1e308, np.finfo(np.float64).max, 0.0, np.inf])
    with np.errstate(divide="ignore"):
        want = 1.0 / x
    assert np.array_equal(evaluate(x)[0], want)
    assert np.array_equal(evaluate(-x)[0], -want)
    assert np.isnan(evaluate(np.array([np.nan]))[0]).all()


def test_norm_and_its_reciprocal(evaluate):
    edge = np.array([1e-280, 1e280])
    x = np.concatenate([mantissas(1 << 17, 3) * 2.0 ** e for e in (-60, -9, -2, -1, 0, 1)] +
                       [mantissas(64, 4) * np.ldexp(1.0, e) for e in range(-1020, 1020, 11)] +
                       [edge, np.nextafter(edge, 0.0), np.nextafter(edge, np.inf)])
    _, n, inv = evaluate(x)
    root = np.sqrt(x.astype(np.longdouble))
    assert half_ulps(inv, 1 / root) <= 1.6
    assert half_ulps(n, root) <= 2.6
