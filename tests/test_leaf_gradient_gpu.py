"""The leaf optimiser's gradient kernel on rays that cross more leaves than a
warp takes at a time (32), dense and thin enough that some saturate and some
do not, for every SH degree, against the FP64 oracle."""
import numpy as np
import pytest

import paper_2207_05009_gb300 as plo
import plogen
from oracle import octopt as ooct
from tests.test_octopt_gpu import _close, _dev
from tests.trees import uniform_tree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("trans,name", [(plo.TRANS_EXP, "exp"), (plo.TRANS_LINEAR, "linear")])
@pytest.mark.parametrize("deg,thick", [(0, 0.3), (1, 1.0), (2, 0.3), (3, 4.0), (4, 1.0)])
def test_many_leaves_per_ray(cuda_available, trans, name, deg, thick):
    rng = np.random.default_rng(70 + deg)
    tree = uniform_tree(5, 1.0, np.zeros((3, (deg + 1) ** 2)), sh_degree=deg)
    n, l_max = 97, 2.0
    s = (rng.uniform(0.2, 1.0, tree.n_leaves) * thick).astype(np.float32)
    s[rng.random(tree.n_leaves) < 0.1] = -0.5
    k = rng.normal(0.0, 0.8, (tree.n_leaves, 3, tree.K)).astype(np.float32)
    init = plogen.HostTree(tree.depth, deg, tree.child, np.maximum(s, 0.0), k)
    rays = plogen.rays_sphere(n, seed=71)
    C_gt, a_gt = rng.uniform(0, l_max, (n, 3)).astype(np.float32), rng.uniform(0, 1, n).astype(np.float32)
    opt = plo.OctOpt(init, l_max, max_rays=n, loss=plo.LOSS_PAPER, transmittance=trans, tv_sigma=0.03, tv_sh=0.01)
    opt.write(plo.OCTOPT_SIGMA, s)
    opt.grad(*_dev(__import__("torch"), rays, C_gt, a_gt))
    opt.check()
    _, ds, dk, ex = ooct.loss_and_grads(tree, s.astype(np.float64), k.reshape(tree.n_leaves, -1).astype(np.float64),
                                        rays, C_gt.astype(np.float64), a_gt.astype(np.float64), l_max, name, "paper",
                                        0.03, 0.01)
    assert ex["segs"][0].shape[1] > 64  # leaves of the longest ray
    _close("d/ds", opt.read(plo.OCTOPT_GRAD_SIGMA), ds, 3e-3, 3e-4)
    _close("d/dk", opt.read(plo.OCTOPT_GRAD_SH).reshape(tree.n_leaves, -1), dk, 3e-3, 3e-4)
