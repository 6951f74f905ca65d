"""GPU parity of the shadow adjoint over the share of restricted steps: all,
some and none of a march's steps cut at step_max (only steps shorter than it
carry a derivative back), marches of one step, and step counts at the limit.
Same bars as the adjoint's parity test: 1e-3 of the largest entry on points
whose fp32 march takes the fp64 path (fp32 rounding of t and h, amplified by
up to ~1e3 in k dd / (t - y)).

Grids with infinities (no seed near) and NaN, forward and backward, against the
oracle.  And the forward march's bound, which leaves out penumbra terms that
cannot lower the visibility, against a march that evaluates every term: the
same bits."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_shadow import BMIN, _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("smax, steps, k", [(1.0, 256, 4.0), (2.5, 64, 2.0), (8.0, 64, 8.0), (4.0, 2, 2.0)])
def test_backward_over_step_limits(smax, steps, k):
    import torch
    nf = 64
    rt, grid, pos, nrm, tg, tp, tn = _setup(nf, 64, k)
    L, h = np.array([0.4, 1.0, 0.3]), 1.0 / nf
    cfg = dict(k=k, steps=steps, step_max=smax * h, eps=h)
    vis_o = oracle.shadow(grid, nf, BMIN, 1.0, pos, nrm, L, **cfg)
    kw = dict(k=k, steps=steps, step_max_vox=smax, eps_vox=1.0, sdf=tg)
    vis_g = rt.shadow(tp, tn, L, **kw).cpu().numpy().ravel()
    w = np.random.default_rng(1).normal(size=vis_o.size) * (np.abs(vis_g - vis_o) <= 1e-5)
    gs_o, gl_o = oracle.shadow_grad(grid, nf, BMIN, 1.0, pos, nrm, L, dvis=w, **cfg)
    dsdf, dl = torch.zeros(nf ** 3, device=rt.device), torch.zeros(3, device=rt.device)
    rt.shadow_backward(tp, tn, L, torch.tensor(w, dtype=torch.float32, device=rt.device), dsdf, dl, **kw)
    scale = max(np.max(np.abs(gs_o)), 1e-30)
    assert np.max(np.abs(dsdf.cpu().numpy() - gs_o)) / scale <= 1e-3
    assert np.max(np.abs(dl.cpu().numpy() - gl_o)) / max(np.max(np.abs(gl_o)), 1e-30) <= 1e-3


def _holes(grid, kind):
    """The grid with texels that are not finite: all, the far side, or a block
    that some marches cross and others start in."""
    g = grid.copy()
    nf = g.shape[0]
    if kind == "inf everywhere":
        g[:] = np.inf
    elif kind == "nan everywhere":
        g[:] = np.nan
    elif kind == "inf far":
        g[nf // 2:] = np.inf
    else:
        q = nf // 4
        g[q:2 * q, :, q:3 * q] = np.inf if kind == "inf block" else np.nan
    return g


@pytest.mark.parametrize("kind", ["inf everywhere", "nan everywhere", "inf far", "inf block", "nan block"])
@pytest.mark.parametrize("smax, light", [(2.5, (0.4, 1.0, 0.3)), (1.0, (0.2, 0.5, -0.6)), (8.0, (-0.5, 0.6, 0.4))])
def test_march_and_adjoint_over_grids_that_are_not_finite(kind, smax, light):
    # +inf and NaN take the same way through both sides' comparisons: a sample
    # that is not finite never sets the visibility, is a step of step_max, and
    # gives the adjoint of a later step 0 times its taps, which is NaN
    import torch
    nf, k = 64, 4.0
    rt, grid, pos, nrm, _, tp, tn = _setup(nf, 64, k)
    grid = _holes(grid, kind)
    tg = torch.tensor(grid.reshape(-1), device=rt.device)
    L, h = np.array(light), 1.0 / nf
    cfg = dict(k=k, steps=64, step_max=smax * h, eps=h)
    vis_o, info = oracle.shadow(grid, nf, BMIN, 1.0, pos, nrm, L, info=True, **cfg)
    kw = dict(k=k, steps=64, step_max_vox=smax, eps_vox=1.0, sdf=tg)
    vis_g = rt.shadow(tp, tn, L, **kw).cpu().numpy().ravel()
    d = np.abs(vis_g - vis_o)
    assert np.isfinite(vis_g).all()
    assert (d > 1e-4).mean() < 0.01 and np.median(d) < 1e-6
    if kind.endswith("everywhere"):
        assert (vis_g == 1).all()
    w = np.random.default_rng(1).normal(size=vis_o.size) * (d <= 1e-5)

    def gradients(w):
        with np.errstate(invalid="ignore"):
            gs, gl = oracle.shadow_grad(grid, nf, BMIN, 1.0, pos, nrm, L, dvis=w, **cfg)
        dsdf, dl = torch.zeros(nf ** 3, device=rt.device), torch.zeros(3, device=rt.device)
        rt.shadow_backward(tp, tn, L, torch.tensor(w, dtype=torch.float32, device=rt.device), dsdf, dl, **kw)
        return gs, gl, dsdf.cpu().numpy(), dl.cpu().numpy()

    gs_o, gl_o, gs_g, gl_g = gradients(w)
    assert np.array_equal(np.isfinite(gs_g), np.isfinite(gs_o))
    assert np.array_equal(np.isfinite(gl_g), np.isfinite(gl_o))
    ok = np.isfinite(gs_o)
    scale = max(np.max(np.abs(gs_o[ok]), initial=0.0), 1e-30)
    assert np.max(np.abs(gs_g[ok] - gs_o[ok]), initial=0.0) / scale <= 1e-3
    # the points whose own march met finite samples only: no NaN reaches these
    finite = np.array([np.isfinite(oracle.shadow_grad(grid, nf, BMIN, 1.0, pos.reshape(-1, 3)[i:i + 1],
                                                      nrm.reshape(-1, 3)[i:i + 1], L, dvis=np.ones(1), **cfg)[1]).all()
                       for i in range(0, vis_o.size, 16)])
    pick = np.zeros(vis_o.size)
    pick[::16] = finite
    gs_o, gl_o, gs_g, gl_g = gradients(w * pick)
    assert np.isfinite(gs_g).all() and np.isfinite(gl_g).all()
    assert np.max(np.abs(gs_g - gs_o)) / max(np.max(np.abs(gs_o)), 1e-30) <= 1e-3
    assert np.max(np.abs(gl_g - gl_o)) / max(np.max(np.abs(gl_o)), 1e-30) <= 1e-3


@pytest.mark.parametrize("smax, steps, k", [(1.0, 256, 2.0), (2.5, 64, 4.0), (4.0, 64, 8.0), (1.0, 256, 16.0),
                                            (8.0, 200, 0.5)])
@pytest.mark.parametrize("light", [(0.4, 1.0, 0.3), (0.7, 0.35, -0.2)])
def test_the_bound_on_penumbra_terms_keeps_every_bit(smax, steps, k, light):
    # The bound gives way to the exact term where the squares it compares are
    # below 1e-30.  A scene scaled by 2^-47 is all below it (no sample above
    # 0.1 of the extent: (0.1 x 2^-47)^2 = 5e-31), so that its march evaluates
    # every term; and a scale by a power of two changes no bit of any quotient,
    # root or comparison (the smallest square, y^2 >= (eps^2 / (2 0.1 extent))^2,
    # is 7e-35 there: nothing underflows).
    import torch
    from paper_2210_04449_gb300 import RTSDF
    nf, ratio = 64, 2.0 ** -47
    rt, grid, pos, nrm, _, tp, tn = _setup(nf, 128, k)
    grid = torch.tensor(np.minimum(grid, 0.1).reshape(-1), device=rt.device)
    kw = dict(k=k, steps=steps, step_max_vox=smax, eps_vox=1.0)
    vis = rt.shadow(tp, tn, light, sdf=grid, **kw)
    small = RTSDF(nf // 2, extent=ratio)
    every = small.shadow(tp * ratio, tn, light, sdf=grid * ratio, **kw)
    assert ((vis > 0) & (vis < 1)).float().mean() > 0.002   # points in the penumbra (fewest at k = 16: 0.4 %)
    assert torch.equal(vis, every)
