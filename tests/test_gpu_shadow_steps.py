"""GPU parity of the shadow adjoint over the share of restricted steps: all,
some and none of a march's steps cut at step_max (only steps shorter than it
carry a derivative back), marches of one step, and step counts at the limit.
Same bars as the adjoint's parity test: 1e-3 of the largest entry on points
whose fp32 march takes the fp64 path (fp32 rounding of t and h, amplified by
up to ~1e3 in k dd / (t - y))."""
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
