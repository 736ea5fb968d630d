"""An infinite optical depth in the leaf optimiser (a density that overflows):
with exponential transmittance the compensated sum makes it NaN, which has to
reach the loss and the gradient of every leaf the ray crosses, however many
lie behind; with linear transmittance the ray ends there."""
import numpy as np
import pytest

import paper_2207_05009_gb300 as plo
from tests.trees import uniform_tree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", [0, 5, 31, 32, 40])
@pytest.mark.parametrize("trans", [plo.TRANS_EXP, plo.TRANS_LINEAR])
def test_infinite_density(cuda_available, trans, at):
    import torch
    tree = uniform_tree(5, 0.001, np.full((3, 4), 0.1), sh_degree=1)
    ray = torch.tensor([[-0.2, -0.15, -0.1, 1.0, 0.95, 0.9]], device="cuda")
    leaf, _, count = plo.trace(plo.Tree(tree), ray, 128)
    crossed = leaf[0, :int(count[0])].cpu().numpy()
    crossed = crossed[crossed >= 0]
    assert len(crossed) > 64  # three turns of 32
    opt = plo.OctOpt(tree, 2.0, max_rays=1, transmittance=trans)
    target = torch.full((1, 3), 0.5, device="cuda"), torch.full((1,), 0.5, device="cuda")
    loss = opt.grad(ray, *target)
    assert bool(torch.isfinite(loss).all())
    assert (opt.read(plo.OCTOPT_GRAD_SIGMA)[crossed] != 0).all()
    s = np.full(tree.n_leaves, 0.001, np.float32)
    s[crossed[at]] = np.inf
    opt.write(plo.OCTOPT_SIGMA, s)
    loss = opt.grad(ray, *target)
    gs, gk = opt.read(plo.OCTOPT_GRAD_SIGMA), opt.read(plo.OCTOPT_GRAD_SH)
    if trans == plo.TRANS_EXP:
        assert bool(torch.isnan(loss[0]))
        assert np.isnan(gs[crossed]).all() and np.isnan(gk[crossed]).all()
    else:
        assert bool(torch.isfinite(loss[0]))
        assert (gs[crossed[at + 1:]] == 0).all() and (gk[crossed[at + 1:]] == 0).all()
        assert np.isfinite(gs[crossed[:at]]).all() and np.isfinite(gk[crossed]).all()
    others = np.setdiff1d(np.arange(tree.n_leaves), crossed)
    assert np.isfinite(gs[others]).all() and np.isfinite(gk[others]).all()
