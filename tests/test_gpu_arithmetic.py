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
    const double v = i & 1 ? aw::join18<true>(f[i].x, f[i].y, f[i].z) : aw::join18<false>(f[i].x, f[i].y, f[i].z);
    j[i] = v * aw::limb_unit(E[i]);
  }
}
__global__ void k_roots(const double* x, double* s, double* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    s[i] = aw::sqrt5(x[i]);
    r[i] = aw::rsqrt5(x[i]);
  }
}
// one dot product of `len` terms per thread, as the least-squares sums take it
__global__ void k_dot(const double* a, const double* b, int len, long long* hh, long long* hl, float2* f, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  long long h = 0, l = 0;
  for (int k = 0; k < len; ++k)
    aw::dot28(h, l, aw::limbs28(aw::fixed_point<57>(a[i * len + k], 1022)),
              aw::limbs28(aw::fixed_point<57>(b[i * len + k], 1022)));
  hh[i] = h;
  hl[i] = l;
  const aw::F2 g = aw::f2_of_dot(h, l);
  f[i] = make_float2(g.h, g.l);
}
__global__ void k_int(const long long* q, double* x, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = aw::int_to_double(q[i]);
}
extern "C" int from_int(const long long* q, double* x, int n) {
  k_int<<<(n + 127) / 128, 128>>>(q, x, n);
  return cudaDeviceSynchronize();
}
extern "C" int roots(const double* x, double* s, double* r, int n) {
  k_roots<<<(n + 127) / 128, 128>>>(x, s, r, n);
  return cudaDeviceSynchronize();
}
extern "C" int dot(const double* a, const double* b, int len, long long* hh, long long* hl, float2* f, int n) {
  k_dot<<<(n + 127) / 128, 128>>>(a, b, len, hh, hl, f, n);
  return cudaDeviceSynchronize();
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


def test_roots(lib):
    """sqrt and its reciprocal from series truncated below 2^-60 with at most
    three roundings of half an ulp on small terms or halved: one ulp; zero and
    subnormal arguments of the square root give 0, negative ones NaN."""
    rng = np.random.default_rng(3)
    x = np.ldexp(rng.uniform(1.0, 2.0, 200000), rng.integers(-1020, 1020, 200000))
    x[:6] = 1.0, 4.0, np.nextafter(4.0, 5.0), 0.0, 1e-310, -1.0
    xd = torch.tensor(x, device="cuda")
    s, r = torch.empty_like(xd), torch.empty_like(xd)
    assert lib.roots(_p(xd), _p(s), _p(r), x.size) == 0
    s, r = s.cpu().numpy(), r.cpu().numpy()
    assert s[3] == 0.0 and s[4] == 0.0 and np.isnan(s[5])
    k = np.r_[0:3, 6:x.size]
    assert (np.abs(s[k] - np.sqrt(x[k])) <= np.spacing(np.sqrt(x[k]))).all()
    ref = (1.0 / np.sqrt(x[k].astype(np.longdouble))).astype(np.float64)
    assert (np.abs(r[k] - ref) <= 1.5 * np.spacing(ref)).all()


@pytest.mark.parametrize("length", [1, 11, 19])
def test_integer_dot(lib, length):
    """hh 2^28 + hl equals the product sum but for the low limbs' products,
    which are below 2^54 each; the pair of floats carries 46 bits of it."""
    rng = np.random.default_rng(4)
    n = 3000
    a, b = (np.ldexp(rng.uniform(-0.5, 0.5, (n, length)), -rng.integers(0, 30, (n, length))) for _ in range(2))
    ad, bd = torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda")
    hh, hl = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
    f = torch.empty((n, 2), dtype=torch.float32, device="cuda")
    assert lib.dot(_p(ad), _p(bd), length, _p(hh), _p(hl), _p(f), n) == 0
    hh, hl, f = hh.cpu().numpy(), hl.cpu().numpy(), f.cpu().numpy().astype(np.float64)
    half_up = lambda v: int(np.floor(abs(v) * 2.0 ** 57 + 0.5)) * (1 if v >= 0 else -1)  # noqa: E731
    for i in range(n):
        exact = sum(half_up(x) * half_up(y) for x, y in zip(a[i], b[i]))
        got = (int(hh[i]) << 56) + (int(hl[i]) << 28)
        assert abs(got - exact) <= length << 54, i
        v = got / 2.0 ** 56
        assert abs(f[i, 0] + f[i, 1] - v) <= abs(v) * 2.0 ** -46 + 2.0 ** -20, i


def test_int_to_double(lib):
    """The nearest double, ties to even."""
    rng = np.random.default_rng(5)
    q = rng.integers(-2 ** 62, 2 ** 62, 100000) >> rng.integers(0, 62, 100000)
    q[:10] = 0, 1, -1, 2 ** 53 - 1, 2 ** 53 + 1, -2 ** 53 - 3, 2 ** 62 - 1, -2 ** 62, 2 ** 54 - 1, 2 ** 61 + 2 ** 8
    qd, x = torch.tensor(q, device="cuda"), torch.empty(q.size, dtype=torch.float64, device="cuda")
    assert lib.from_int(_p(qd), _p(x), q.size) == 0
    for a, b in zip(q.tolist(), x.cpu().tolist()):
        assert b == float(a), a


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
