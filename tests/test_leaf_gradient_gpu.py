"""The leaf optimiser's gradient kernel on rays that cross more leaves than a
warp takes at a time (32), dense and thin enough that some saturate and some
do not, for every SH degree, against the FP64 oracle."""
import numpy as np
import pytest

import paper_2207_05009_gb300 as plo
import plogen
from oracle import octopt as ooct
from tests.test_octopt_gpu import _close, _dev
from tests.trees import random_tree, uniform_tree

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


@pytest.mark.parametrize("tv_sigma,tv_sh", [(0.0, 0.0), (0.03, 0.0), (0.0, 0.01), (0.03, 0.01)])
def test_total_variation_beside_the_trace(cuda_available, tv_sigma, tv_sh):
    """The TV gradients start the leaves' gradients on a stream of their own
    while the rays are traced: with either weight zero, with no rays, called
    twice, and captured in a graph, against the FP64 oracle."""
    import torch
    rng = np.random.default_rng(80)
    tree = random_tree(4, rng, sh_degree=1, p_split=0.5, p_empty=0.2)
    n, l_max = 300, 2.0
    s = rng.uniform(0.5, 3.0, tree.n_leaves).astype(np.float32)
    k = rng.normal(0.0, 0.8, (tree.n_leaves, 3, tree.K)).astype(np.float32)
    rays = plogen.rays_sphere(n, seed=81)
    C_gt, a_gt = rng.uniform(0, l_max, (n, 3)).astype(np.float32), rng.uniform(0, 1, n).astype(np.float32)
    opt = plo.OctOpt(plogen.HostTree(tree.depth, 1, tree.child, s, k), l_max, max_rays=n, tv_sigma=tv_sigma,
                     tv_sh=tv_sh)
    batch = _dev(torch, rays, C_gt, a_gt)
    args = (tree, s.astype(np.float64), k.reshape(tree.n_leaves, -1).astype(np.float64))
    _, ds, dk, _ = ooct.loss_and_grads(*args, rays, C_gt.astype(np.float64), a_gt.astype(np.float64), l_max, "exp",
                                       "paper", tv_sigma, tv_sh)
    _, ds0, dk0, _ = ooct.loss_and_grads(*args, rays, C_gt.astype(np.float64), a_gt.astype(np.float64), l_max, "exp",
                                         "paper", 0.0, 0.0)

    def check(ws, wk, what):
        _close(what, opt.read(plo.OCTOPT_GRAD_SIGMA), ws, 3e-3, 3e-4)
        _close(what, opt.read(plo.OCTOPT_GRAD_SH).reshape(tree.n_leaves, -1), wk, 3e-3, 3e-4)

    for _ in range(2):
        opt.grad(*batch)
        check(ds, dk, "rays")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        opt.grad(*batch)
    opt.grad(*[x[:0] for x in batch])
    if tv_sigma or tv_sh:
        check(ds - ds0, dk - dk0, "no rays")
    else:
        assert not opt.read(plo.OCTOPT_GRAD_SIGMA).any() and not opt.read(plo.OCTOPT_GRAD_SH).any()
    for _ in range(2):
        graph.replay()
        check(ds, dk, "graph")
    opt.check()
