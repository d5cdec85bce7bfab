"""Loading a state checks and spreads it on the device.  A refused state names
its first bad element (a bad average before an inverted element) and leaves the
loaded one as it is: the arrays stay equal, and so do the sweeps after it, bit
for bit.  The two loaders agree: whole numbers, averages and corners equal, the
dofs within 2e-12 of the largest (each is held within 1e-12 of the oracle)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1408_3719_gb300 import workloads as W  # noqa: E402


def _setup(order, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1408_3719_gb300 import aleweno
    mesh = W.vortex_grid_mesh(n, jitter=0.1)
    Q = W.cell_average(mesh, lambda x, y: W.vortex_state(x, y, 1.4, mesh["period"]), W._duffy_rule(8))
    s = aleweno.Solver(order_M=order, t_end=1.0)
    s.load_mesh(mesh)
    return aleweno, mesh, np.ascontiguousarray(Q), s


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("order,n", [(1, 12), (3, 12), (2, 40)])
def test_refused_states_leave_the_old_one(order, n, device):
    aw, mesh, Q, s = _setup(order, n)
    ref = aw.Solver(order_M=order, t_end=1.0)
    ref.load_mesh(mesh)
    put = (lambda a: torch.tensor(a, device="cuda")) if device else (lambda a: a)
    for x in (s, ref):
        x.load_state(put(Q))
        x.enqueue(3)
        x.sync()
    before, ne = s.get_elem(), len(Q)
    low, nan = Q.copy(), Q.copy()
    low[[ne - 1, ne // 2], 0] = -1.0, -1.0
    nan[0, 3] = np.nan
    xy = mesh["xy"].copy()
    a, b, c = mesh["tri"][ne - 1]
    xy[[a, b]] = xy[[b, a]]
    for q, p, el in ((low, None, ne // 2), (nan, None, 0), (low, xy, ne // 2), (Q, xy, None)):
        with pytest.raises(aw.AwError) as e:
            s.load_state(put(q)) if p is None else s.load_state_xy(put(q), put(p))
        if el is not None:
            assert f"element {el} is not physical" in str(e.value)
        else:
            assert "is not counter-clockwise" in str(e.value)
    after = s.get_elem()
    for k in before:
        assert np.array_equal(before[k], after[k]), k
    for x in (s, ref):
        x.enqueue(5)
        x.sync()
    eg, er = s.get_elem(), ref.get_elem()
    for k in er:
        assert np.array_equal(eg[k], er[k]), k


@pytest.mark.parametrize("order", [1, 2, 3])
def test_both_loaders_agree(order):
    _, mesh, Q, s = _setup(order, 20)
    s.load_state(Q)
    a = s.get_elem()
    s.load_state_xy(Q, mesh["xy"])
    b = s.get_elem()
    for k in a:
        if k == "qhat":
            assert np.abs(a[k] - b[k]).max() <= 2e-12 * np.abs(b[k]).max()
        else:
            assert np.array_equal(a[k], b[k]), k
