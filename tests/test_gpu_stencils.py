"""Reconstruction from badly conditioned stencils: elements pressed down to a
fraction of their height, whose stencils have condition numbers kappa up to 8 10^9 in
the element's frame, where a factorisation of the normal equations in less than
about 2 log2(kappa) bits is no preconditioner.

The averages are those of one polynomial of the scheme's degree per variable, so
that every stencil's least-squares fit is that polynomial, whatever the nonlinear
weights are, and the nodal values of w_h (the predictor's dofs at tau = 0) are known
without any solver.

Tolerance, per element.  With the columns of a stencil's matrix A divided by
their largest entries c_l, sigma its smallest singular value, m its rows and z
the scaled solution, rows and data that are off by 16 u (u = 2^-53: averages,
positions, products) and a solver whose backward error is of that size too move z
by at most 32 u sqrt(m) (q + sum |z|) / sigma, q the largest average; the
basis functions are at most 1 on the element, so a nodal value moves by that
times sum 1 / c_l; the transformation to characteristic fields and back, whose
factors are of order one here, doubles it.  The weights mix the stencils, so the
element's bound is its worst stencil's, and 16 u of the average are added."""
import numpy as np
import pytest

from oracle.pyoracle import Oracle
from paper_1408_3719_gb300 import workloads as W

MON = [(1, 0), (0, 1), (2, 0), (1, 1), (0, 2), (3, 0), (2, 1), (1, 2), (0, 3)]
U = 2.0 ** -53


def _averages(x, y, n):
    """Averages of the monomials over triangles with corners x, y [k, 3]."""
    s, t, w = W._duffy_rule(4)
    lam = np.stack([1.0 - s - t, s, t])
    px, py = x @ lam, y @ lam
    return np.stack([((px ** a * py ** b) * w).sum(1) for a, b in MON[:n]], axis=1)


def _bounds(o, mesh, M, Q, elems):
    """Tolerance of the nodal values of each element, and the largest kappa."""
    X, n = W._corner_coords(mesh), 9 if M == 3 else 5
    ref = np.array([[0.0, 1.0, 0.0]]) - 1.0 / 3.0, np.array([[0.0, 0.0, 1.0]]) - 1.0 / 3.0
    mbar, tol, kmax = _averages(*ref, n), np.zeros(len(elems)), 0.0
    for k, i in enumerate(elems):
        Ji = np.linalg.inv(np.stack([X[i, 1] - X[i, 0], X[i, 2] - X[i, 0]], axis=1))
        for s in o.stencils(i)[0]:
            if s.min() < 0 or len(set(s.tolist())) < len(s):
                continue  # a dropped sector
            R = (X[s[1:]] - X[i, 0]) @ Ji.T - 1.0 / 3.0
            A, b = _averages(R[:, :, 0], R[:, :, 1], n) - mbar, Q[s[1:]] - Q[i]
            c = np.abs(A).max(0)
            sv = np.linalg.svd(A / c, compute_uv=False)
            z = np.linalg.lstsq(A / c, b, rcond=None)[0]
            grow = 64.0 * np.sqrt(len(b)) * (np.abs(Q[s]).max() + np.abs(z).sum(0).max()) / sv[-1] * (1.0 / c).sum()
            tol[k] = max(tol[k], U * (16.0 * np.abs(Q[i]).max() + grow))
            kmax = max(kmax, sv[0] / sv[-1])
    return tol, kmax


def pressed(M, height):
    """(mesh, averages, exact nodal values, pressed elements): a square mesh with
    some elements, no two of them near each other, pressed along one height."""
    mesh = W.shock_tube_mesh(16, 16, 1.0, 1.0, jitter=0.1)
    tri, taken, elems = mesh["tri"], np.zeros(len(mesh["xy"]), bool), []
    for i in range(len(tri)):
        if taken[tri[i]].any():
            continue
        for k in range(3):
            a, b, c = (mesh["xy"][tri[i, (k + q) % 3]] for q in (1, 2, 0))
            n = tri[i, k]
            if min(c.min(), 1.0 - c.max()) < 1e-9:
                continue  # a boundary node stays
            t = b - a
            xy = mesh["xy"].copy()
            xy[n] += (height - 1.0) * (c - a - t * np.dot(c - a, t) / np.dot(t, t))
            if (W._signed_areas(xy, tri) > 0).all():
                mesh["xy"] = xy
                ring = np.unique(tri[np.isin(tri, tri[i]).any(1)])
                taken[np.unique(tri[np.isin(tri, ring).any(1)])] = True
                elems.append(i)
                break

    mon = [(a, b) for a in range(M + 1) for b in range(M + 1 - a) if a + b > 0]
    co = np.random.default_rng(3).uniform(-0.6, 0.6, (4, len(mon))) / len(mon)

    def fun(x, y):  # another polynomial in each variable
        p = [sum(c * (x - 0.5) ** a * (y - 0.5) ** b for c, (a, b) in zip(row, mon)) for row in co]
        return np.stack(p, axis=-1) + np.array([1.0, 0.3, 0.1, 2.5])

    return mesh, fun, elems


CASES = [(2, 1 / 30), (2, 1 / 1000), (2, 1 / 3000), (3, 1 / 30), (3, 1 / 100), (3, 1 / 300)]


def _check(solver, M, height):
    """Errors of the pressed elements' nodal values in units of their bounds."""
    mesh, fun, elems = pressed(M, height)
    Q = W.cell_average(mesh, fun, W._duffy_rule(4))
    o = Oracle(order_M=M, t_end=1.0)
    o.load_mesh(mesh)
    tol, kappa = _bounds(o, mesh, M, Q, elems)
    assert kappa > 10.0 / height
    solver.load_mesh(mesh)
    solver.load_state(Q)
    X, lat = W._corner_coords(mesh)[elems], np.array([(i / M, j / M) for j in range(M + 1) for i in range(M + 1 - j)])
    pts = X[:, None, 0] + lat[:, :1] * (X[:, None, 1] - X[:, None, 0]) + lat[:, 1:] * (X[:, None, 2] - X[:, None, 0])
    w = solver.get_elem()["qhat"][elems, : len(lat)]
    return np.abs(w - fun(pts[..., 0], pts[..., 1])).max((1, 2)) / tol


@pytest.mark.parametrize("M,height", CASES)
def test_oracle_reproduces_the_polynomial(M, height):
    """The oracle's orthogonal factorisation keeps the bound."""
    r = _check(Oracle(order_M=M, t_end=1.0), M, height)
    assert (r <= 1.0).all(), r.max()


@pytest.mark.gpu
@pytest.mark.parametrize("M,height", CASES)
def test_gpu_reproduces_the_polynomial(M, height):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1408_3719_gb300 import aleweno
    s = aleweno.Solver(order_M=M, t_end=1.0)
    r = _check(s, M, height)
    s.close()
    assert (r <= 1.0).all(), r.max()
