"""The nonlinear weights with an epsilon whose reciprocal is beyond FP64's
range (a subnormal one, which the parameters accept): a component that is
uniform to the bit has all its smoothness indicators 0, hence 0 / epsilon = 0
and the linear weights, as in the oracle."""
import numpy as np
import pytest

from paper_2102_01366_gb300 import gks
from paper_2102_01366_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 1e-11  # normwise, FP64: some hundred operations on O(1) values, as the parity tests


@pytest.fixture(scope="module")
def cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2102_01366_gb300 import _build
    _build.build()
    gks.lib()
    return torch


def _state(nc):
    """Rough density and energy, momenta uniform to the bit."""
    rng = np.random.default_rng(71)
    W = np.zeros((5, nc))
    W[0] = 1.0 + 0.1 * rng.uniform(-1, 1, nc)
    W[1] = 0.25
    W[4] = 2.5 + 0.1 * rng.uniform(-1, 1, nc)
    dW = np.zeros((15, nc))
    dW[:3], dW[12:] = [0.1 * rng.uniform(-1, 1, (3, nc)) for _ in range(2)]
    return W, dW


# 1e-300: the last decade whose reciprocal is a number; below 5.6e-309 it is not
@pytest.mark.parametrize("eps", [1e-8, 1e-300, 1e-310, 5e-324])
@pytest.mark.parametrize("order", [2, 3])
def test_uniform_components_keep_their_reconstruction(cuda, oracle_mod, eps, order):
    mesh = I.box_mesh((3, 3, 2), jitter=0.1, seed=70)
    W, dW = _state(len(mesh["tet"]))
    kw = dict(weno=1, order=order, cfl=0.4, eps_weno=eps)
    om, p = oracle_mod.Mesh(mesh), oracle_mod.params(**kw)
    poly_o, _, fb_o = om.reconstruct(p, W, dW)
    assert np.isfinite(poly_o).all() and not fb_o.any()
    s = gks.State(gks.Mesh(mesh), gks.params(precision=0, **kw))
    s.init(W, dW)
    poly, _, fb = [x.cpu().numpy() for x in s.debug_reconstruct()]
    np.testing.assert_array_equal(fb, fb_o)
    for q in range(5):
        assert np.abs(poly[:, q] - poly_o[:, q]).max() <= TOL * np.abs(poly_o).max(), q
    # the step's first face records: the reconstruction as the flux sees it
    dt = om.timestep(p, W)
    got, ref = s.debug_face_records(dt, 1).cpu().numpy(), om.face_records(p, W, dW, dt, 1)
    assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()
