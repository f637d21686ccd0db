"""The split path's BF16 slices (tc_slices.cuh, compiled here for the host) against FP64 residuals, bit for bit."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2512_01055_gb300 import build

SRC = """
#include "%s"
extern "C" void slices(const double *x, long long n, int S, uint32_t *out) {
  for (long long e = 0; e < n; ++e) {
    tc::Slicer a = tc::slicer(x[e]);
    for (int p = 0; p < S; ++p) out[p * n + e] = tc::next_slice(a, p);
  }
}
"""
N = 1 << 20


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("slices")
    src, so = d / "slices.cpp", d / "libslices.so"
    src.write_text(SRC % os.path.join(build.CSRC, "tc_slices.cuh"))
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def slices(lib, x, s):
    out = np.empty((s, x.size), np.uint32)
    lib.slices(ctypes.c_void_p(x.ctypes.data), ctypes.c_longlong(x.size), s, ctypes.c_void_p(out.ctypes.data))
    return (out << 16).view(np.float32).astype(np.float64)


def by_fp64_residuals(x, s):
    out = np.empty((s, x.size))
    r = x.copy()
    for p in range(s):
        m, e = np.frexp(r)
        out[p] = np.ldexp(np.rint(m * 256.0), e - 8)               # 8 significant bits, half to even
        r = r - out[p]                                             # exact
    return out


def values(kind):
    g = np.random.default_rng(7)
    x = g.standard_normal(N) * 0.05
    if kind == "grid":                                             # short significands, so residuals end early
        return np.round(x * 2.0 ** 20) * 2.0 ** -20
    if kind == "near midways":                                     # a few bits, then half a last place, then little or nothing
        hi = g.integers(128, 256, N) * 2.0
        k = g.integers(9, 44, N)
        low = g.integers(-2, 3, N) * 2.0 ** -k
        return np.ldexp(np.where(g.random(N) < 0.5, hi + 1.0, hi) + low, g.integers(-60, 10, N)) * g.choice([-1.0, 1.0], N)
    if kind == "late midways":                                     # the same at the third and fourth slice
        k = g.integers(16, 50, N)
        mid = 2.0 ** -k * (1 + g.integers(0, 2, N) * 2.0 ** -8.0)
        return (1.0 + g.integers(0, 128, N) / 128.0 + mid + 2.0 ** -52 * g.integers(-16, 17, N)) * g.choice([-1.0, 1.0], N)
    if kind == "wide":
        return x * np.exp2(g.uniform(-60, 60, N))
    return x


@pytest.mark.parametrize("s", [2, 3, 4])
@pytest.mark.parametrize("kind", ["normal", "grid", "near midways", "late midways", "wide"])
def test_slices_equal_those_of_fp64_residuals(lib, kind, s):
    x = values(kind)
    assert np.array_equal(slices(lib, x, s), by_fp64_residuals(x, s))


def test_special_values(lib):
    x = np.array([0.0, -0.0, 1.0, -1.0, 3.0e38, np.inf, -np.inf, np.nan])
    got = slices(lib, x, 4)
    assert np.array_equal(got[:, :5].sum(0), by_fp64_residuals(x[:5], 4).sum(0))
    assert not np.isfinite(got[:, 5:].sum(0)).any()
