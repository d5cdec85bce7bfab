"""Reconstruction on badly conditioned stencils against the oracle.

The mesh is a vortex torus whose node columns are drawn together towards a few
lines, so that neighbouring elements differ in width by up to 1 / squeeze and
the least-squares matrices' condition numbers kappa grow with it (the GPU's
factorisation in pairs of floats with integer residuals has to hold there as
the oracle's orthogonal one does).  Tolerance: both sides' coefficients are
off by at most about kappa 2^-53 of the data; with kappa up to 10^3 / squeeze
(10^2..2 10^3 on the plain meshes), and the limiter's weights at most eight times
as sensitive, 8 10^3 2^-53 / squeeze of the largest magnitude, which is
10^-12 / squeeze rounded up."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.pyoracle import Oracle  # noqa: E402
from paper_1408_3719_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("squeeze", [0.3, 0.03])
def test_preprocessing_on_squeezed_columns(order, squeeze):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1408_3719_gb300 import aleweno
    mesh = W.vortex_grid_mesh(14, jitter=0.1)
    L = mesh["period"][0]
    x = mesh["xy"][:, 0] / L * 2.0 * np.pi
    mesh["xy"][:, 0] = L / (2.0 * np.pi) * (x - (1.0 - squeeze) / 3.0 * np.sin(3.0 * x))  # slope squeeze at three lines
    if not (W._signed_areas(mesh["xy"], mesh["tri"], mesh["shift"], mesh["period"]) > 0).all():
        pytest.fail("the squeezed mesh has an inverted element")
    Q = W.cell_average(mesh, lambda x, y: W.vortex_state(x, y, 1.4, mesh["period"]), W._duffy_rule(8))
    g, o = aleweno.Solver(order_M=order, t_end=1.0), Oracle(order_M=order, t_end=1.0)
    for s in (g, o):
        s.load_mesh(mesh)
        s.load_state(Q)
    eg, eo = g.get_elem(), o.get_elem()
    assert np.array_equal(eg["dt"], eo["dt"])
    assert np.abs(eg["qhat"] - eo["qhat"]).max() <= 1e-12 / squeeze * np.abs(eo["qhat"]).max()
    g.close()
