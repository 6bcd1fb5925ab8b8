"""Sizes and values at which the hot kernels change their path or leave lanes
idle: ragged blocks of faces and cells, several cases in one warp, cells that
the positivity bound clears beside cells that are checked point by point, and
the integer conversions between FP64 and FP32 over their whole range."""
import numpy as np
import pytest

from paper_2102_01366_gb300 import gks
from paper_2102_01366_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# normwise against the oracle (FP64: some hundred operations on O(1) values
# and differences of the time step's inverse; FP32: 2^-24 times the same)
TOL = {0: 1e-11, 1: 2e-5}


@pytest.fixture(scope="module")
def cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2102_01366_gb300 import _build
    _build.build()
    gks.lib()
    return torch


def _rough_state(mesh, amp, seed):
    """Seeded cell averages around (1, 0.3, -0.2, 0.1, p = 1) with gradients
    of the same size over a cell's width."""
    rng = np.random.default_rng(seed)
    nc = len(mesh["tet"])
    rho = 1.0 + amp * rng.uniform(-1, 1, nc)
    u = np.array([[0.3], [-0.2], [0.1]]) + amp * rng.uniform(-1, 1, (3, nc))
    p = 1.0 + amp * rng.uniform(-1, 1, nc)
    W = np.concatenate([rho[None], rho * u, (p / 0.4 + 0.5 * rho * (u * u).sum(0))[None]])
    return np.ascontiguousarray(W), rng.uniform(-1, 1, (15, nc)) * amp


# faces of a periodic box of n hexahedra: 12 n.  FP64 takes blocks of 21 faces
# where these leave the fullest of 152 SMs fewer warps than blocks of 32 do
# (warps: 2 against 3; 4 against 3; 4 against 6; 6 against 6)
@pytest.mark.parametrize("viscous", [0, 1])
@pytest.mark.parametrize("dims, warps", [((3, 2, 2), (2, 3)), ((7, 7, 7), (4, 3)), ((8, 8, 8), (4, 6)),
                                         ((10, 9, 8), (6, 6))])
def test_fp64_flux_blocks(cuda, oracle_mod, dims, warps, viscous):
    mesh = I.box_mesh(dims, jitter=0.1, seed=61)
    nf = 12 * dims[0] * dims[1] * dims[2]
    assert tuple(-(-(-(-nf // f)) // 152) * w for f, w in ((21, 2), (32, 3))) == warps
    W, dW = _rough_state(mesh, 0.05, 62)
    kw = dict(weno=1, cfl=0.4, viscous=viscous, mu=1e-3 * viscous)
    g, o, p = gks.Mesh(mesh), oracle_mod.Mesh(mesh), oracle_mod.params(**kw)
    assert g.nf == nf
    s = gks.State(g, gks.params(precision=0, **kw))
    s.init(W, dW)
    dt = o.timestep(p, W)
    for stage, groups in ((1, (0, 5, 10, 25, 40)), (2, (0, 5, 20))):
        got = s.debug_face_records(dt, stage).cpu().numpy()
        ref = o.face_records(p, W, dW, dt, stage)
        for a, b in zip(groups, groups[1:]):
            assert np.abs(got[:, a:b] - ref[:, a:b]).max() <= TOL[0] * np.abs(ref[:, a:b]).max(), (stage, a)


# FP32: blocks of 32 faces, stage 1's records stored as one stretch, stage 2's
# copied ahead; a box of a x b x c hexahedra open on all sides has 12 abc +
# 2 (ab + bc + ca) faces, the last block here 18, 2, 30 and 16 of them.
# Groups that nearly vanish are held to 1e-3 of the state, as the parity tests do
@pytest.mark.parametrize("viscous", [0, 1])
@pytest.mark.parametrize("flux_blocks", [2, 3])
@pytest.mark.parametrize("dims, nf", [((1, 1, 1), 18), ((2, 1, 1), 34), ((3, 2, 1), 94), ((3, 2, 2), 176)])
def test_fp32_flux_ragged_blocks(cuda, oracle_mod, dims, nf, flux_blocks, viscous):
    mesh = I.box_mesh(dims, jitter=0.0, seed=0, periodic=(False, False, False))
    W, dW = _rough_state(mesh, 0.05, 69)
    kw = dict(weno=1, cfl=0.4, viscous=viscous, mu=1e-3 * viscous)
    g, o, p = gks.Mesh(mesh), oracle_mod.Mesh(mesh), oracle_mod.params(**kw)
    assert g.nf == nf
    s = gks.State(g, gks.params(precision=1, **kw))
    s.set_variant(0, flux_blocks, 1)
    s.init(W, dW)
    dt = o.timestep(p, W)
    for stage, groups in ((1, (0, 5, 10, 25, 40)), (2, (0, 5, 20))):
        got = s.debug_face_records(dt, stage).cpu().numpy()
        ref = o.face_records(p, W, dW, dt, stage)
        floor = 1e-3 * g.geometry()["farea"].max() / 3.0 * np.abs(W).max()
        for a, b in zip(groups, groups[1:]):
            scale = max(np.abs(ref[:, a:b]).max(), floor)
            assert np.abs(got[:, a:b] - ref[:, a:b]).max() <= TOL[1] * scale, (stage, a)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shapes", [[(1, 1, 1)] * 7, [(2, 1, 1), (1, 1, 1), (3, 2, 1), (1, 1, 1), (1, 1, 1)],
                                    [(2, 1, 1), (1, 1, 1), (1, 1, 1), (2, 1, 1), (1, 1, 1)]])
def test_small_cases_sharing_a_warp(cuda, oracle_mod, precision, shapes):
    """Each case's time step is the minimum over its own cells only.  A batch
    with a case that loses its positivity (in the oracle: no number) is
    refused."""
    meshes = [I.box_mesh(sh, (1.0, 1.0, 1.0), (False, False, False), 0.0, 0) for sh in shapes]
    states = [I.riemann_x_state(m, left=(1.0, 0.2, 1.0 + 0.3 * k), right=(0.5, 0.2, 0.6), x0=0.45)
              for k, m in enumerate(meshes)]
    g = gks.Mesh(I.batch_mesh(meshes))
    s = gks.State(g, gks.params(weno=1, cfl=0.4, precision=precision))
    s.init(*[np.concatenate([st[i] for st in states], axis=1) for i in (0, 1)])
    s.step(3)
    p = oracle_mod.params(weno=1, cfl=0.4)
    runs = [oracle_mod.Mesh(m).run(p, *st, nsteps=3) for m, st in zip(meshes, states)]
    if not all(np.isfinite(r[0]).all() for r in runs):
        with pytest.raises(gks.GksError, match="non-positive"):
            s.sync()
        return
    s.sync()
    Wg = s.get()[0].cpu().numpy()
    tg, _ = s.case_times()
    for k, (Wo, _, to, _) in enumerate(runs):
        c0, c1 = g.case_first[k], g.case_first[k + 1]
        assert abs(tg[k] - to) <= TOL[precision] * to
        for q in range(5):
            assert np.abs(Wg[q, c0:c1] - Wo[q]).max() <= TOL[precision] * max(np.abs(Wo[q]).max(), 1e-300), (k, q)


@pytest.mark.parametrize("dims", [(3, 3, 3), (5, 4, 3), (7, 5, 5)])
@pytest.mark.parametrize("weno, order", [(0, 3), (1, 3), (1, 2)])
def test_positivity_fallback_flags(cuda, oracle_mod, dims, weno, order):
    """Cells the bound clears, cells whose points are checked and pass, and
    cells that fall back, mixed in a block of cells."""
    mesh = I.box_mesh(dims, jitter=0.1, seed=63)
    W, dW = _rough_state(mesh, 0.1, 64)
    rng = np.random.default_rng(65)
    for c in rng.permutation(W.shape[1])[:W.shape[1] // 12]:
        W[:, c] *= 0.02  # near-vacuum cells: the polynomials of their neighbours undershoot
    kw = dict(weno=weno, order=order, cfl=0.4)
    s = gks.State(gks.Mesh(mesh), gks.params(precision=0, **kw))
    s.init(W, dW)
    poly, _, fb = [x.cpu().numpy() for x in s.debug_reconstruct()]
    poly_o, _, fb_o = oracle_mod.Mesh(mesh).reconstruct(oracle_mod.params(**kw), W, dW)
    assert 0 < fb_o.astype(bool).sum() < fb_o.size
    np.testing.assert_array_equal(fb, fb_o)
    for q in range(5):
        assert np.abs(poly[:, q] - poly_o[:, q]).max() <= TOL[0] * np.abs(poly_o[:, q]).max()


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 3, 3), (11, 1, 1), (7, 5, 4)])
def test_slopes_pass_against_recomputed_slopes(cuda, precision, dims):
    mesh = I.box_mesh(dims, jitter=0.0, seed=0, periodic=(False, False, False))
    W, dW = _rough_state(mesh, 0.05, 66)
    out = []
    for sp in (0, 1):
        s = gks.State(gks.Mesh(mesh), gks.params(precision=precision, weno=1, cfl=0.4))
        s.set_variant(0, 3, sp)
        s.init(W, dW)
        s.step(2, 1e-3)
        s.sync()
        out.append([x.cpu().numpy() for x in s.get()])
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= TOL[min(precision, 1)] * np.abs(a).max()


@pytest.mark.parametrize("order", [0, 1, 2])
@pytest.mark.parametrize("dims", [(1, 1, 1), (7, 3, 2)])
def test_state_in_and_out(cuda, dims, order):
    """FP64 averages come back as they went in; the gradients as the nearest
    FP32 values: ties, values below FP32's range and above it, and zeros of
    either sign among them."""
    mesh = I.box_mesh(dims, periodic=(False, False, False))
    W, _ = _rough_state(mesh, 0.1, 67)
    rng = np.random.default_rng(68)
    dW = rng.uniform(-1, 1, (15, W.shape[1])) * 10.0 ** rng.uniform(-50, 37, (15, W.shape[1]))
    special = np.array([0.0, -0.0, 1e-46, -1e-45, 1.1754943e-38, 1.1754942e-38, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24,
                        1.0 + 2.0 ** -24 + 2.0 ** -50, 3.4028234663852886e38, 3.4028235677973366e38, -1e39, 5e-324,
                        2.0 ** -149 * 1.5, -2.0 ** -150])
    dW[:, :6] = rng.permuted(np.tile(special, (6, 1)).T, axis=0)
    s = gks.State(gks.Mesh(mesh), gks.params(precision=1, weno=1))
    if order:
        s.set_cell_order(order)
    s.init(W, dW)
    Wg, dWg = [x.cpu().numpy() for x in s.get()]
    np.testing.assert_array_equal(Wg, W)
    with np.errstate(over="ignore", under="ignore"):
        ref = dW.astype(np.float32).astype(np.float64)
    np.testing.assert_array_equal(dWg, ref)
    np.testing.assert_array_equal(np.signbit(dWg), np.signbit(ref))
