"""The render walk where its fixed-point parameters and its emission queue can
go wrong, against the FP64 oracle: rays (nearly) parallel to an axis,
directions of any length, every tree depth, and leaves that all emit (the
per-warp queue then fills faster than rays finish)."""
import numpy as np
import pytest

import oracle
import paper_2207_05009_gb300 as plo
import plogen
from tests.parity import RTOL_FP32, assert_radiance_close
from tests.trees import random_tree

pytestmark = pytest.mark.gpu


def _render(tree, rays, layout=plo.LAYOUT_OCTREE, **kw):
    import torch
    t = plo.Tree(tree, plo.PREC_FP32, layout)
    rgb, T, _ = plo.render(t, torch.from_numpy(rays).cuda(), plo.RenderParams(**kw))
    torch.cuda.synchronize()
    t.check()
    return rgb.cpu().numpy(), T.cpu().numpy()


@pytest.mark.parametrize("layout", [plo.LAYOUT_OCTREE, plo.LAYOUT_BRICKS])
@pytest.mark.parametrize("depth", [1, 3, 7, 11, 16])
def test_flat_and_unnormalised_directions(cuda_available, depth, layout):
    rng = np.random.default_rng(depth)
    tree = random_tree(depth, rng, sh_degree=1) if depth <= 3 else plogen.luminaire_tree(
        plogen.LUMINAIRE_D6.with_(depth=min(depth, 7), sh_degree=1))
    if depth > 7:  # the same tree under a path of first children: cells of 2^-depth
        extra = depth - 7
        child = np.where(tree.child >= 0, tree.child + extra, tree.child)
        top = np.full((extra, 8), -1, np.int32)
        top[:, 0] = np.arange(1, extra + 1)
        tree.child, tree.depth = np.concatenate([top, child]).astype(np.int32), depth
    size = 0.5 ** max(0, depth - 7)
    n = 3000
    o = rng.uniform(-1.5, 2.5, (n, 3)) * size
    d = rng.uniform(0, 1, (n, 3)) * size - o
    flat = rng.random((n, 3)) < 0.4
    flat[flat.all(1)] = False
    d = np.where(flat, d * 10.0 ** rng.uniform(-30, -1, (n, 3)), d)
    d[rng.random((n, 3)) < 0.1] = 0.0
    d[(d == 0).all(1)] = 1.0
    d *= 10.0 ** rng.uniform(-3, 3, (n, 1)) / np.abs(d).max(1, keepdims=True)
    inside = flat & (rng.random((n, 3)) < 0.8)
    o = np.where(inside, rng.uniform(0, 1, (n, 3)) * size, o)
    rays = np.concatenate([o, d], 1).astype(np.float32)
    rgb, T = _render(tree, rays, layout)
    ref = oracle.render(tree, rays)
    assert (ref["T"] < 1).mean() > 0.05
    assert_radiance_close(rgb, T, ref, RTOL_FP32, what=f"depth {depth}")


@pytest.mark.parametrize("act", [plo.ACT_RELU, plo.ACT_SIGMOID])
@pytest.mark.parametrize("n", [1, 31, 33, 5000])
def test_every_leaf_emits(cuda_available, n, act):
    tree = plogen.luminaire_tree(plogen.LUMINAIRE_D6.with_(emissive_fraction=1.0 if act == plo.ACT_RELU else 0.5,
                                                           sigma_log10=(-2.0, 0.5)))
    if act == plo.ACT_SIGMOID:
        tree.sh *= 1e-4
    rays = plogen.rays_sphere(n, seed=40 + n)
    rgb, T = _render(tree, rays, activation=act, l_max=3.0)
    ref = oracle.render(tree, rays, activation=oracle.SIGMOID if act == plo.ACT_SIGMOID else oracle.RELU, l_max=3.0)
    assert_radiance_close(rgb, T, ref, RTOL_FP32, what=f"{n} rays")


def test_wavefront_sizes_and_the_work_counter(cuda_available):
    """Each ray's arithmetic is its own, so a prefix of a wavefront gives the
    same bits whatever the launch: one ray, fewer than a warp, spread out over
    the SMs or not, with the work counter, without it because the allocation
    failed, or captured in a graph."""
    import torch
    t = plo.Tree(plogen.luminaire_tree(plogen.LUMINAIRE_D6))
    rays = torch.from_numpy(plogen.rays_sphere(3 << 17, seed=50)).cuda()
    n = rays.shape[0]
    rgb, T, _ = plo.render(t, rays)
    torch.cuda.synchronize()
    for m in (1, 31, 33, 2432, 2433, 77823, 77824, n - 1):
        r, tr, _ = plo.render(t, rays[:m])
        assert torch.equal(r, rgb[:m]) and torch.equal(tr, T[:m]), m
    try:
        plo.debug_fail_alloc_after(0)
        r, tr, _ = plo.render(t, rays)
    finally:
        plo.debug_fail_alloc_after(-1)
    assert torch.equal(r, rgb) and torch.equal(tr, T)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        r, tr, _ = plo.render(t, rays)
    for _ in range(2):
        r.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(r, rgb) and torch.equal(tr, T)
    t.check()


def test_batch_with_few_rays_per_warp(cuda_available):
    """The claims of a batch shrink with its rays: a handful to 60,000 rays
    over three trees equal the trees' own renders bit for bit."""
    import torch
    trees = [plo.Tree(plogen.luminaire_tree(plogen.LUMINAIRE_D6.with_(seed=s)), prec)
             for s, prec in ((1, plo.PREC_FP32), (2, plo.PREC_FP16), (3, plo.PREC_BF16))]
    for counts in ((1, 0, 2), (33, 5000, 1), (20000, 20001, 19999)):
        offs = np.concatenate([[0], np.cumsum(counts)])
        n = int(offs[-1])
        rays = torch.from_numpy(plogen.rays_sphere(n, seed=60 + n)).cuda()
        rgb, T = torch.full((n, 3), -1.0, device="cuda"), torch.full((n,), -1.0, device="cuda")
        plo.Batch(trees, offs).render(rays, rgb, T)
        for t, a, b in zip(trees, offs[:-1], offs[1:]):
            if b > a:
                r, tr, _ = plo.render(t, rays[a:b])
                assert torch.equal(rgb[a:b], r) and torch.equal(T[a:b], tr), (counts, a)
