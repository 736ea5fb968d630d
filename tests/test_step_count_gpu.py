"""A ray's step count is the number of cells that the trace reports: the walk's
empty steps behind a plane that its rounded position hides do not count."""
import contextlib

import numpy as np
import pytest

import paper_2207_05009_gb300 as plo
import plogen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [7, 16])
def test_a_cap_of_the_traced_cells_is_not_reached(cuda_available, depth):
    import torch
    tree = plogen.luminaire_tree(plogen.LUMINAIRE_D6.with_(depth=7, sh_degree=1))
    extra = depth - 7
    if extra:  # the same tree under a path of first children: cells of 2^-16
        child = np.where(tree.child >= 0, tree.child + extra, tree.child)
        top = np.full((extra, 8), -1, np.int32)
        top[:, 0] = np.arange(1, extra + 1)
        tree.child, tree.depth = np.concatenate([top, child]).astype(np.int32), depth
    rays = plogen.rays_sphere(200_000, seed=61)
    rays[:, :3] *= 0.5 ** extra
    rays[:, 3:] *= 0.5 ** extra
    t = plo.Tree(tree)
    rays = torch.from_numpy(rays).cuda()
    _, _, count = plo.trace(t, rays, 512)
    want, wantT, _ = plo.render(t, rays)
    torch.cuda.synchronize()
    t.check()
    assert int(count.max()) < 512 and len(torch.unique(count)) > 20
    for c in torch.unique(count[count > 0]).tolist():
        mine = torch.nonzero(count == c).squeeze(1)
        status = torch.zeros(len(mine), dtype=torch.int32, device="cuda")
        # a ray whose step count reaches the cap is reported, so one more
        rgb, T, _ = plo.render(t, rays[mine].contiguous(), plo.RenderParams(max_steps=c + 1), status=status)
        torch.cuda.synchronize()
        t.check()
        assert not bool(status.any())
        assert torch.equal(rgb, want[mine]) and torch.equal(T, wantT[mine])
        # and one that reaches it is, as before
        plo.render(t, rays[mine].contiguous(), plo.RenderParams(max_steps=c), status=status)
        torch.cuda.synchronize()
        saturated = wantT[mine] <= 0
        assert bool(((status == plo.RAY_STEP_LIMIT) | saturated).all())
        with pytest.raises(plo.PloError) if not bool(saturated.all()) else contextlib.nullcontext():
            t.check()
