"""The ways a run can be issued: graphs of four sweeps against single ones, contexts
in two threads, and launches large enough for the predictor with integer
conversions.  Runs of the same library are compared bit for bit; the dofs with the
oracle by the parity contract (1e-12 of each variable's largest magnitude)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.pyoracle import Oracle  # noqa: E402
from paper_1408_3719_gb300 import workloads as W  # noqa: E402


def _solver(mesh, Q, **opt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1408_3719_gb300 import aleweno
    s = aleweno.Solver(t_end=1.0, **opt)
    s.load_mesh(mesh)
    s.load_state(Q)
    return s


def _equal(ea, eb):
    for k in ea:
        assert np.array_equal(ea[k], eb[k]), k


@pytest.mark.parametrize("rest", [0, 1, 2, 3])
@pytest.mark.parametrize("order,opt", [(1, {}), (2, {}), (3, {}), (2, dict(gts=True)), (2, dict(flux="osher")),
                                       (1, dict(t_switch=0.02, cfl_start=0.2))])
def test_runs_of_sweeps_equal_single_sweeps(order, opt, rest):
    mesh, Q = W.vortex(12)
    a, b, n = _solver(mesh, Q, order_M=order, **opt), _solver(mesh, Q, order_M=order, **opt), 12 + rest
    a.enqueue(n)
    total = a.sync()
    assert total == sum(b.sweep() for _ in range(n))
    _equal(a.get_elem(), b.get_elem())
    for x, y in zip(a.get_nodes(), b.get_nodes()):
        assert np.array_equal(x, y)
    assert a.diag() == b.diag()


def test_contexts_in_two_threads():
    """Two meshes, orders and streams at once, several times: the results of one
    after the other."""
    def run(order, n, out, times):
        try:
            mesh, Q = W.vortex(n)
            s = _solver(mesh, Q, order_M=order)
            for _ in range(times):
                s.load_state(Q)
                s.enqueue(30)
                s.sync()
                out.append(s.get_elem())
            s.close()
        except Exception as e:  # seen by the main thread
            out.append(e)

    alone, both = ([], []), ([], [])
    jobs = ((3, 16), (2, 40))
    for job, out in zip(jobs, alone):
        run(*job, out, 1)
    threads = [threading.Thread(target=run, args=(*job, out, 6)) for job, out in zip(jobs, both)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ref, got in zip(alone, both):
        assert len(got) == 6, got
        for e in got:
            _equal(ref[0], e)


@pytest.mark.parametrize("order,per_block", [(1, 10), (2, 2), (3, 1)])
@pytest.mark.parametrize("wide", [0, 1])
def test_predictor_over_more_than_two_grids(order, per_block, wide):
    """More elements than two grids of four blocks per SM hold (two of twice the
    size with wide blocks)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    need = 8 * torch.cuda.get_device_properties(0).multi_processor_count * per_block
    n = int(np.sqrt(need / 2)) + 2
    mesh, Q = W.vortex(n)
    g, o = _solver(mesh, Q, order_M=order), Oracle(order_M=order, t_end=1.0)
    assert g.n_tris > need
    if wide:
        g.set_tiles(pred_wide=1)
        g.load_state(Q)
    o.load_mesh(mesh)
    o.load_state(Q)
    eg, eo = g.get_elem(), o.get_elem()
    assert np.array_equal(eg["dt"], eo["dt"])
    d = np.abs(eg["qhat"] - eo["qhat"]).max(axis=(0, 1))
    assert (d <= 1e-12 * np.abs(eo["qhat"]).max(axis=(0, 1))).all(), d
