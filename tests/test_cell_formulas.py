"""The rearranged float64 formulas of the cell kernels (csrc/step_cell.cuh)
and the grouped MRT collision (csrc/mrt.cuh), compiled for the host, against
the pointwise physics they replace.  Inputs are of order one and every output
is a sum of at most about a hundred products of a few of them, so the two
orders of summation agree within 100 rounding errors of order-one terms:
1e-13 in float64 and 100 eps = 1.2e-5 in float32."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def hc(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("hc") / "libhc.so"
    subprocess.check_call([nvcc, "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                           "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                           "-I", os.path.join(os.path.dirname(HERE), "include"),
                           "-shared", os.path.join(HERE, "host_cell.cu"), "-o", str(out)])
    return ctypes.CDLL(str(out))


def P(a):
    return ctypes.c_void_p(a.ctypes.data)


def params(rng):
    return np.array([rng.uniform(0.05, 0.2), rng.uniform(0.01, 0.05), rng.uniform(2.5, 3.1),
                     rng.uniform(0.2, 0.5), rng.uniform(-1, 1), rng.uniform(0.6, 2)])


@pytest.mark.parametrize("iso", [0, 1], ids=["standard", "isotropic"])
@pytest.mark.parametrize("d3", [0, 1], ids=["d2q9", "d3q19"])
def test_cell_formulas_match_the_pointwise_physics(hc, d3, iso):
    rng = np.random.default_rng(7)
    cell, ref = np.zeros(19), np.zeros(19)
    for _ in range(200):
        p, x = params(rng), rng.uniform(-1, 1, 42)
        hc.hc_compare(d3, iso, P(p), P(x), P(cell), P(ref))
        assert np.abs(cell - ref).max() < 1e-13 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("f32,tol", [(0, 1e-13), (1, 1.2e-5)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("d3", [0, 1], ids=["d2q9", "d3q19"])
def test_grouped_mrt_matches_the_dense_transform(hc, d3, f32, tol):
    rng = np.random.default_rng(8)
    q = 19 if d3 else 9
    out, ref = np.zeros(q), np.zeros(q)
    for k in range(200):
        p = params(rng)
        g = rng.uniform(-0.03, 0.03, q).astype(np.float32).astype(np.float64)
        F = rng.uniform(-0.1, 0.1, 3).astype(np.float32).astype(np.float64)
        if not d3:
            F[2] = 0.0
        rates = np.full(q, 1.0 / p[5]) if k % 2 else rng.uniform(0.1, 1.9, q)
        hc.hc_mrt(d3, f32, P(p), P(g), P(F), P(rates), P(out), P(ref))
        assert np.abs(out - ref).max() < tol


def test_integer_conversions_match_the_hardware(hc):
    """All exponents, ties, infinities, NaN and both signs."""
    hc.hc_convert.restype = ctypes.c_long
    rng = np.random.default_rng(9)
    n = 400000
    f = rng.integers(0, 1 << 32, n, dtype=np.uint32)
    d = rng.integers(0, 1 << 64, n, dtype=np.uint64)
    # half of the doubles in the float range, a quarter of those on a tie
    e = rng.integers(890, 1160, n // 2, dtype=np.uint64) << np.uint64(52)
    d[: n // 2] = (d[: n // 2] & np.uint64(0x800FFFFFFFFFFFFF)) | e
    t = n // 8
    d[:t] = (d[:t] & np.uint64(0xFFFFFFFFE0000000)) | np.uint64(0x10000000)
    f[:8] = [0, 0x80000000, 1, 0x7F800000, 0xFF800000, 0x7FC00000, 0x00800000, 0x7F7FFFFF]
    d[-6:] = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028235677973366e38]).view(np.uint64)
    assert hc.hc_convert(P(f), P(d), ctypes.c_long(n)) == 0
