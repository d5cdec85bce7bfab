"""A differentiated run takes plain FP64 kernels of its own; that is a property of
its calls, not of how the state came in.  Everything is compared bit for bit, but
for the gradients, whose scatters are atomics (1e-12 of the largest, as for
different checkpoint intervals)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.adjoint_fd import _dJ, _mask, wavy_vortex  # noqa: E402


def _solver(mesh, order):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1408_3719_gb300 import aleweno
    s = aleweno.Solver(order_M=order, t_end=1.0)
    s.load_mesh(mesh)
    return s


def _equal(a, b):
    ea, eb = a.get_elem(), b.get_elem()
    for k in ea:
        assert np.array_equal(ea[k], eb[k]), k
    for x, y in zip(a.get_nodes(), b.get_nodes()):
        assert np.array_equal(x, y)


def _copy(a, b):
    b.set_nodes(*a.get_nodes())
    b.set_elem(a.get_elem())


@pytest.mark.parametrize("order", [1, 2, 3])
def test_both_loaders_give_the_same_run(order):
    mesh, Q = wavy_vortex(14)
    a, b = _solver(mesh, order), _solver(mesh, order)
    a.load_state(Q)
    b.load_state_xy(Q, mesh["xy"])
    _equal(a, b)
    for s in (a, b):
        s.enqueue(9)
        s.sync()
    _equal(a, b)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("first", ["load_state_xy", "adjoint_forward", "adjoint"])
def test_restored_run_goes_on_as_the_uninterrupted_one(order, first):
    mesh, Q = wavy_vortex(14)
    a, b = _solver(mesh, order), _solver(mesh, order)
    a.load_state_xy(Q, mesh["xy"])
    if first == "load_state_xy":
        a.enqueue(5)
        a.sync()
    else:
        a.adjoint_forward(5, 2)
    if first == "adjoint":
        e = a.get_elem()
        a.adjoint(*_dJ(e["Q"], e["X"], _mask(mesh)))
    _copy(a, b)
    for s in (a, b):
        s.enqueue(6)
        s.sync()
    _equal(a, b)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("loader", ["load_state_xy", "adjoint_load_state"])
def test_adjoint_does_not_depend_on_the_loader(order, loader):
    mesh, Q = wavy_vortex(14)
    a, b = _solver(mesh, order), _solver(mesh, order)
    a.load_state(Q)
    getattr(b, loader)(Q, mesh["xy"])
    g = []
    for s in (a, b):
        s.adjoint_forward(7, 3)
        e = s.get_elem()
        g.append(s.adjoint(*_dJ(e["Q"], e["X"], _mask(mesh))))
    _equal(a, b)
    for x, y in zip(*g):
        assert np.abs(x - y).max() <= 1e-12 * np.abs(x).max()


@pytest.mark.parametrize("option", [dict(flux="osher"), dict(gts=True), dict(t_switch=0.1, cfl_start=0.1)])
def test_adjoint_load_state_refuses_what_the_adjoint_does_not_cover(option):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1408_3719_gb300 import aleweno
    mesh, Q = wavy_vortex(8)
    s, ref = (aleweno.Solver(order_M=2, t_end=1.0, **option) for _ in range(2))
    for x in (s, ref):
        x.load_mesh(mesh)
        x.load_state(Q)
    with pytest.raises(aleweno.AwError) as e:
        s.adjoint_load_state(Q, mesh["xy"])
    assert "INVALID_ARG" in str(e.value)
    for x in (s, ref):  # the loaded state is as it was
        x.enqueue(5)
        x.sync()
    _equal(s, ref)
