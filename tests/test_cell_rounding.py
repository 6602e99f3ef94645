"""Rounding of pointwise formulas, compiled for the host: in the float64 cell
kernels (csrc/step_cell.cuh) Q meets its increment in one rounding and a
uniform field has no Laplacian; the coefficients of the grouped MRT collision
(csrc/mrt.cuh) are rounded once, and its velocity is divided by the density
without an approximate reciprocal."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
LD = np.longdouble
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def hr(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("hr") / "libhr.so"
    subprocess.check_call([nvcc, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-ftz=true",
                           "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                           "-I", os.path.join(os.path.dirname(HERE), "include"),
                           "-shared", os.path.join(HERE, "host_round.cu"), "-o", str(out)])
    return ctypes.CDLL(str(out))


def P(a):
    return ctypes.c_void_p(a.ctypes.data)


def full(q):
    return np.array([[q[0], q[1], q[2]], [q[1], q[3], q[4]], [q[2], q[4], -q[0] - q[3]]], dtype=LD)


def increment(p, q, h, d, u, g, dim):
    """R of Eq. 1, its trace projected out, in extended precision; grad = d/2."""
    xi, Gamma = LD(p[4]), LD(p[3])
    G = g.astype(LD) / 2
    Q, Qt = full(q), full(q) + np.eye(3, dtype=LD) / 3
    D, W = (G + G.T) / 2, (G - G.T) / 2
    M = xi * D + W
    S = M @ Qt + Qt @ M.T - 2 * xi * Qt * (Q * G).sum()
    R = S + Gamma * full(h)
    for a in range(dim):
        R = R - LD(u[a]) * full(d[a].astype(LD) / 2)
    R = R - np.eye(3, dtype=LD) * np.trace(R) / 3
    return np.array([R[0, 0], R[0, 1], R[0, 2], R[1, 1], R[1, 2]])


@pytest.mark.parametrize("d3", [0, 1], ids=["d2q9", "d3q19"])
def test_the_increment_is_added_in_one_rounding(hr, d3):
    """|r - (base + R)| is half a unit of r for the sum, and less than 100
    roundings of terms below 1e-3 for R itself (velocity gradients, u and H
    below 1e-4, Q below one half, differences of Q below 0.1, |xi| below 1)."""
    if LD(1) + LD(EPS) / 8 == LD(1):
        pytest.skip("no extended precision")
    rng = np.random.default_rng(11)
    dim = 3 if d3 else 2
    small = 1e-4
    for _ in range(300):
        p = np.array([0.1, 0.02, 2.7, rng.uniform(0.2, 0.5), rng.uniform(-1, 1), 1.0])
        q, base = rng.uniform(-0.5, 0.5, 5), rng.uniform(0.5, 1.0, 5)
        h, u = rng.uniform(-small, small, 5), rng.uniform(-small, small, 3)
        d, g = np.zeros((3, 5)), np.zeros((3, 3))
        d[:dim] = rng.uniform(-0.1, 0.1, (dim, 5))
        g[:dim, :dim] = rng.uniform(-small, small, (dim, dim))
        u[dim:] = 0.0
        r = np.zeros(5)
        hr.hr_rhs(d3, P(p), P(q), P(h), P(d), P(u), P(g), P(base), P(r))
        exact = base.astype(LD) + increment(p, q, h, d, u, g, dim)
        bound = np.spacing(np.abs(r)) / 2 + 100 * EPS * 10 * small
        assert (np.abs(r - exact) <= bound).all()


@pytest.mark.parametrize("iso", [0, 1], ids=["standard", "isotropic"])
@pytest.mark.parametrize("d3", [0, 1], ids=["d2q9", "d3q19"])
def test_a_uniform_field_has_no_laplacian(hr, d3, iso):
    """With s the exact weighted sum of equal neighbours, H does not depend
    on K, bit for bit."""
    weights = {(0, 0): 4, (0, 1): 5, (1, 0): 6, (1, 1): 12}[(d3, iso)]
    rng = np.random.default_rng(12)
    for _ in range(100):
        q = np.round(rng.uniform(-0.5, 0.5, 5) * 2**40) / 2**40
        s = weights * q
        h = [np.zeros(5), np.zeros(5)]
        for k, K in enumerate((0.0, rng.uniform(0.01, 0.05))):
            p = np.array([0.1, K, 2.7, 0.34, 0.8, 1.5])
            hr.hr_field(d3, iso, P(p), P(q), P(s), P(h[k]))
        assert np.array_equal(h[0], h[1])


@pytest.mark.parametrize("d3", [0, 1], ids=["d2q9", "d3q19"])
def test_mrt_coefficients_are_rounded_once(hr, d3):
    hr.hr_mrt_coef.restype, hr.hr_mrt_coef.argtypes = ctypes.c_float, [ctypes.c_int, ctypes.c_float,
                                                                       ctypes.c_int]
    hr.hr_mrt_norm.restype = ctypes.c_double
    conserved = (0, 3, 5, 7) if d3 else (0, 3, 5)
    rng = np.random.default_rng(13)
    for rate in rng.uniform(0.05, 1.95, 200).astype(np.float32):
        for k in range(19 if d3 else 9):
            if k not in conserved:
                exact = float(rate) / hr.hr_mrt_norm(d3, k)
                got = np.float32(hr.hr_mrt_coef(d3, rate, k))
                assert abs(float(got) - exact) <= 0.5000001 * float(np.spacing(np.abs(got)))


@pytest.mark.gpu
@pytest.mark.parametrize("d3", [0, 1], ids=["d2q9", "d3q19"])
def test_velocity_is_divided_by_the_density_exactly(hr, d3):
    """J = 1, so u is 1/rho, correctly rounded."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(14)
    rho0 = torch.from_numpy(rng.uniform(-0.3, 0.7, 100000).astype(np.float32)).cuda()
    rho, ux = torch.empty_like(rho0), torch.empty_like(rho0)
    torch.cuda.synchronize()
    assert hr.hr_velocity(d3, rho0.numel(), *(ctypes.c_void_p(t.data_ptr())
                                              for t in (rho0, rho, ux))) == 0
    rho, ux = rho.cpu().numpy(), ux.cpu().numpy()
    assert np.array_equal(ux, np.float32(1) / rho)
