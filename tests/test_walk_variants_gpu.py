"""The walk's variants that no other test reaches: brick trees in a batch, and
the sphere proxy on rays (nearly) parallel to an axis and of any length."""
import numpy as np
import pytest

import oracle
import paper_2207_05009_gb300 as plo
import plogen
from tests.parity import RTOL_FP32, assert_radiance_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [(1, 33, 2), (70_001, 1_000, 250_037)])
def test_bricks_in_a_batch(cuda_available, counts):
    """Brick trees of both brick sizes beside an octree, with different depths,
    degrees and precisions: each tree's own render bit for bit."""
    import torch
    forms = [(dict(), plo.PREC_FP32, plo.LAYOUT_BRICKS, 2),
             (dict(depth=7, sh_degree=3, seed=5), plo.PREC_FP16, plo.LAYOUT_BRICKS, 3),
             (dict(depth=5, sh_degree=1, seed=6), plo.PREC_BF16, plo.LAYOUT_OCTREE, 0)]
    trees = [plo.Tree(plogen.luminaire_tree(plogen.LUMINAIRE_D6.with_(**kw)), prec, layout, log)
             for kw, prec, layout, log in forms]
    offs = np.concatenate([[0], np.cumsum(counts)])
    n = int(offs[-1])
    rays = torch.from_numpy(plogen.rays_sphere(n, seed=97)).cuda()
    rgb, T = torch.full((n, 3), -1.0, device="cuda"), torch.full((n,), -1.0, device="cuda")
    status = torch.full((n,), -9, dtype=torch.int32, device="cuda")
    plo.Batch(trees, offs).render(rays, rgb, T, status)
    for t, a, b in zip(trees, offs[:-1], offs[1:]):
        want, wantT, _ = plo.render(t, rays[a:b])
        assert torch.equal(rgb[a:b], want) and torch.equal(T[a:b], wantT)
    assert not bool(status.any())


@pytest.mark.parametrize("layout", [plo.LAYOUT_OCTREE, plo.LAYOUT_BRICKS])
@pytest.mark.parametrize("sphere", [(0.5, 0.5, 0.5, 0.4), (0.62, 0.45, 0.5, 0.55)])
def test_sphere_proxy_and_flat_directions(cuda_available, sphere, layout):
    import torch
    rng = np.random.default_rng(98)
    tree = plogen.luminaire_tree(plogen.LUMINAIRE_D6.with_(depth=7, sh_degree=1))
    n = 6000
    o = rng.uniform(-1.5, 2.5, (n, 3))
    d = rng.uniform(0, 1, (n, 3)) - o
    flat = rng.random((n, 3)) < 0.4
    flat[flat.all(1)] = False
    d = np.where(flat, d * 10.0 ** rng.uniform(-30, -1, (n, 3)), d)
    d[rng.random((n, 3)) < 0.1] = 0.0
    d[(d == 0).all(1)] = 1.0
    d *= 10.0 ** rng.uniform(-3, 3, (n, 1)) / np.abs(d).max(1, keepdims=True)
    o = np.where(flat & (rng.random((n, 3)) < 0.8), rng.uniform(0, 1, (n, 3)), o)
    rays = np.concatenate([o, d], 1).astype(np.float32)
    t = plo.Tree(tree, plo.PREC_FP32, layout)
    rgb, T, _ = plo.render(t, torch.from_numpy(rays).cuda(), plo.RenderParams(sphere=sphere))
    torch.cuda.synchronize()
    t.check()
    ref = oracle.render(tree, rays, sphere=tuple(float(np.float32(v)) for v in sphere))
    box = oracle.render(tree, rays)
    assert (np.abs(box["T"] - ref["T"]) > 1e-6).mean() > 0.02 and (ref["T"] < 1).mean() > 0.05
    assert_radiance_close(rgb.cpu().numpy(), T.cpu().numpy(), ref, RTOL_FP32, what=f"sphere {sphere}")
