"""The sweep kernels' own arithmetic (csrc/aw_math.cuh): the reciprocal against
the rounded quotient, the limb sums against integer arithmetic, and the
predictor that uses them against the oracle at the edges of its tiles and far
from unit scales.

Tolerances: the reciprocal's last operation rounds y (1 + e + e^2) with a
relative error of 2^-53 (half an ulp) plus below 2^-59 of the truncated series
and of the rounding of e + e^2: one ulp covers it.  Limb sums are integers:
equal.  The predictor: the parity contract's 1e-12 of each variable's largest
magnitude."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.pyoracle import Oracle  # noqa: E402
from paper_1408_3719_gb300 import build as B  # noqa: E402
from paper_1408_3719_gb300 import workloads as W  # noqa: E402

SRC = r"""
#include "aw_math.cuh"
__global__ void k_rcp(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = aw::rcp3(x[i]);
}
__global__ void k_limbs(const double* x, const int* E, float4* f, double* j, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    f[i] = aw::limbs18(x[i], E[i]);
    j[i] = aw::join18(f[i].x, f[i].y, f[i].z) * aw::limb_unit(E[i]);
  }
}
extern "C" int rcp(const double* x, double* y, int n) {
  k_rcp<<<(n + 127) / 128, 128>>>(x, y, n);
  return cudaDeviceSynchronize();
}
extern "C" int limbs(const double* x, const int* E, float4* f, double* j, int n) {
  k_limbs<<<(n + 127) / 128, 128>>>(x, E, f, j, n);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("arith")
    (d / "t.cu").write_text(SRC)
    subprocess.check_call([B._nvcc(), *B.ARCH, "-std=c++17", "-I", B.CSRC, "-shared", "-Xcompiler", "-fPIC", "-o",
                           str(d / "t.so"), str(d / "t.cu")])
    return C.CDLL(os.path.join(str(d), "t.so"))


def _p(t):
    return C.c_void_p(t.data_ptr())


def test_reciprocal(lib):
    rng = np.random.default_rng(1)
    x = np.ldexp(rng.uniform(1.0, 2.0, 200000), rng.integers(-1020, 1020, 200000)) * rng.choice([-1.0, 1.0], 200000)
    x[:4] = 1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0), 3.0
    xd, y = torch.tensor(x, device="cuda"), torch.empty(x.size, dtype=torch.float64, device="cuda")
    assert lib.rcp(_p(xd), _p(y), x.size) == 0
    y, r = y.cpu().numpy(), 1.0 / x
    assert (np.abs(y - r) <= np.spacing(np.abs(r))).all()


def test_limbs(lib):
    rng = np.random.default_rng(2)
    n = 50000
    E = rng.integers(128, 2000, n).astype(np.int32)
    below = rng.integers(0, 70, n)  # exponents below the group's largest
    x = np.ldexp(rng.uniform(1.0, 2.0, n), E - 1023 - below) * rng.choice([-1.0, 1.0], n)
    x[:3] = 0.0, -0.0, np.ldexp(2.0 - 2.0 ** -52, int(E[2]) - 1023)
    xd, Ed = torch.tensor(x, device="cuda"), torch.tensor(E, device="cuda")
    f = torch.empty((n, 4), dtype=torch.float32, device="cuda")
    j = torch.empty(n, dtype=torch.float64, device="cuda")
    assert lib.limbs(_p(xd), _p(Ed), _p(f), _p(j), n) == 0
    f, j = f.cpu().numpy(), j.cpu().numpy()
    for i in range(n):
        m, ex = np.frexp(abs(x[i]))
        num = int(m * 2 ** 53)  # |x| = num 2^(ex - 53); unit 2^(E - 1076)
        sh = int(ex) - 53 - (int(E[i]) - 1076)
        q = num << sh if sh >= 0 else (num + (1 << (-sh - 1))) >> -sh  # half away from zero
        q = -q if x[i] < 0 else q
        l2, l1, l0 = (int(v) for v in f[i, :3])
        assert (l2 << 36) + (l1 << 18) + l0 == q, i
        assert abs(l2) <= 2 ** 18 and 0 <= l1 < 2 ** 18 and 0 <= l0 < 2 ** 18
        assert abs(j[i] - x[i]) <= np.ldexp(1.0, int(E[i]) - 1077), i


@pytest.mark.parametrize("order,n", [(1, 5), (1, 37), (2, 7), (2, 25), (3, 9), (3, 19)])
@pytest.mark.parametrize("rho,vel", [(1.0, 1.0), (1e-7, 1e4), (3e5, 1e-6)])
def test_predictor_tiles_and_scales(lib, order, n, rho, vel):
    """2 n^2 elements: fewer than one block's, an odd number of blocks, more
    than the resident blocks; densities and velocities scaled by rho and vel
    (the times scale by 1 / vel, so that the tick steps stay the same)."""
    from paper_1408_3719_gb300 import aleweno
    mesh, Q = W.vortex(n)
    Q = Q * np.array([rho, rho * vel, rho * vel, rho * vel * vel])
    g, o = aleweno.Solver(order_M=order, t_end=1.0 / vel), Oracle(order_M=order, t_end=1.0 / vel)
    for s in (g, o):
        s.load_mesh(mesh)
        s.load_state(Q)
    eg, eo = g.get_elem(), o.get_elem()
    assert np.array_equal(eg["dt"], eo["dt"])
    d = np.abs(eg["qhat"] - eo["qhat"]).max(axis=(0, 1))
    assert (d <= 1e-12 * np.abs(eo["qhat"]).max(axis=(0, 1))).all(), d
    g.close()
