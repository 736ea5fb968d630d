"""The scratch pool of a device's trees: one bound for all of them, and nothing
held where another allocation of the library finds no memory."""
import pytest

import paper_2207_05009_gb300 as plo
import plogen

pytestmark = pytest.mark.gpu


def _used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def _trees(n):
    host = plogen.luminaire_tree(plogen.LUMINAIRE_D6)
    return [plo.Tree(host) for _ in range(n)]


def test_the_bound_is_for_all_trees_together(cuda_available):
    import torch
    rays = torch.from_numpy(plogen.rays_sphere(9 << 20, seed=90))  # 2 x 94 MB of buffers a call
    first, *others = _trees(5)
    plo.render_host(first, rays)
    for t in others:
        plo.render_host(t, rays[:1000])
    before = _used()
    for t in others:
        plo.render_host(t, rays)
    assert _used() - before <= 64 << 20  # what a pool rounds up to
    for t in (first, *others[:-1]):  # the last tree keeps the pool usable
        t.free()
    rgb, T = plo.render_host(others[-1], rays[:400_000])
    want, wantT, _ = plo.render(others[-1], rays[:400_000].cuda())
    torch.cuda.synchronize()
    assert torch.equal(rgb, want.cpu()) and torch.equal(T, wantT.cpu())


def test_a_failed_allocation_takes_what_the_pool_keeps(cuda_available):
    import torch
    rays = torch.from_numpy(plogen.rays_sphere(2 << 20, seed=91))
    tree, = _trees(1)
    net = plo.Mlp(l_max=1.0)
    n = 1 << 20
    batch = rays[:n].cuda(), torch.zeros(n, 3, device="cuda"), torch.zeros(n, device="cuda")
    jitter = torch.empty(1, device="cuda")  # not reached
    plo.render_host(tree, rays)
    held = _used()
    # a workspace of 2^28 samples: 137 GB a layer
    loss = torch.empty(1, device="cuda")
    with pytest.raises(plo.PloError) as ei:
        plo._check(plo.mlp_lib().plo_mlp_train_step(net.handle, *(plo._ptr(b) for b in batch), n, 256,
                                                    plo._ptr(jitter), plo._ptr(loss), None))
    assert ei.value.status == -3
    assert held - _used() >= 64 << 20
    rgb, T = plo.render_host(tree, rays)
    assert bool(torch.isfinite(rgb).all())
