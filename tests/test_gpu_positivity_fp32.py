"""The positivity check's shortcut (a bound over the largest offsets clears a
cell without looking at its Gauss points) in FP32 bulk, with FP32 and with
FP64 operators: some cells cleared, some looked at, some falling back."""
import numpy as np
import pytest

from paper_2102_01366_gb300 import gks
from paper_2102_01366_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# FP32 bulk's tolerance of a reconstruction against the oracle (normwise, as
# the parity tests); the pressure adds five such terms, so that a point within
# ten of it of zero may fall either way
TOL = 2e-5
# R at a point in FP32: ten terms of its size, each rounded
ROUND = 10 * 2.0 ** -24


@pytest.fixture(scope="module")
def cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2102_01366_gb300 import _build
    _build.build()
    gks.lib()
    return torch


def _smallest(g, poly):
    """Each cell's smallest density and pressure over its 12 face Gauss points
    for the reconstruction poly [nc, 5, 10], FP64."""
    top, geo = g.topology(), g.geometry()
    left = top["csr_sign"] > 0
    gp = np.where(left[..., None, None], geo["gp_l"][top["csr_face"]], geo["gp_r"][top["csr_face"]])
    x, y, z = np.moveaxis(gp.reshape(g.nc, 12, 3), 2, 0)
    basis = np.stack([np.ones_like(x), x, y, z, x * x, x * y, x * z, y * y, y * z, z * z], axis=1)
    v = np.einsum("cqk,ckp->cqp", poly, basis)
    p = 0.4 * (v[:, 4] - 0.5 * (v[:, 1:4] ** 2).sum(1) / v[:, 0])
    return v[:, 0].min(1), np.where(v[:, 0] > 0, p, -np.inf).min(1)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("dims", [(3, 3, 3), (7, 5, 5)])
@pytest.mark.parametrize("weno, order", [(0, 3), (1, 3), (1, 2)])
def test_positivity_fallback_flags_fp32(cuda, oracle_mod, dims, weno, order, precision):
    mesh = I.box_mesh(dims, jitter=0.1, seed=91)
    rng = np.random.default_rng(92)
    nc = len(mesh["tet"])
    rho, p = 1.0 + 0.1 * rng.uniform(-1, 1, nc), 1.0 + 0.1 * rng.uniform(-1, 1, nc)
    u = np.array([[0.3], [-0.2], [0.1]]) + 0.1 * rng.uniform(-1, 1, (3, nc))
    W = np.concatenate([rho[None], rho * u, (p / 0.4 + 0.5 * rho * (u * u).sum(0))[None]])
    W[:, rng.permutation(nc)[:nc // 12]] *= 0.02  # near-vacuum cells: the polynomials around them undershoot
    dW = 0.1 * rng.uniform(-1, 1, (15, nc))
    kw = dict(weno=weno, order=order, cfl=0.4)
    om, g = oracle_mod.Mesh(mesh), gks.Mesh(mesh)
    _, _, fb_o = om.reconstruct(oracle_mod.params(**kw), W, dW)
    assert 0 < fb_o.astype(bool).sum() < nc
    # every cell's reconstruction before the check: that of a state so far from
    # vacuum that none falls back (a constant changes no slope and no weight)
    shift = np.zeros((5, 1))
    shift[0], shift[4] = 100.0, 1000.0
    s64 = gks.State(g, gks.params(precision=0, **kw))
    s64.init(W + shift, dW)
    poly64, _, fb64 = [a.cpu().numpy() for a in s64.debug_reconstruct()]
    assert not fb64.any()
    poly64[:, :, 0] -= shift[:, 0]
    rho64, p64 = _smallest(g, poly64)
    near = np.minimum(np.abs(rho64), np.abs(p64)) < 10 * TOL * np.abs(W).max()
    bad = (rho64 <= 0) | (p64 <= 0)
    np.testing.assert_array_equal(fb_o[~near], bad[~near])  # the same check in the oracle
    s = gks.State(g, gks.params(precision=precision, **kw))
    s.init(W, dW)
    poly, _, fb = [a.cpu().numpy() for a in s.debug_reconstruct()]
    assert near.sum() < 0.02 * nc
    np.testing.assert_array_equal(fb[~near], bad[~near])
    # no cell keeps a reconstruction that is not positive at its points
    rho_min, p_min = [a[fb == 0] for a in _smallest(g, poly)]
    assert rho_min.min() > -ROUND * np.abs(W).max() and p_min.min() > -5 * ROUND * np.abs(W).max()
