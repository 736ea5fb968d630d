"""Renders while another thread captures a graph in the global mode, which
forbids unsafe calls (allocations among them) in every thread."""
import threading

import pytest

import paper_2207_05009_gb300 as plo
import plogen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1000, 3 << 17, (1 << 20) - 1])
def test_renders_beside_a_capture(cuda_available, n):
    """The first call on a tree that needs scratch (from 3 * 2^17 rays on) and
    further ones, on two trees, from a thread that does not capture."""
    import torch
    trees = [plo.Tree(plogen.luminaire_tree(plogen.LUMINAIRE_D6)) for _ in range(2)]
    rays = torch.from_numpy(plogen.rays_sphere(n, seed=95)).cuda()
    small = rays[:1000].clone()
    for t in trees:
        plo.render(t, small)
    rgb, T = torch.empty((1000, 3), device="cuda"), torch.empty(1000, device="cuda")
    out = [(torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda")) for _ in range(3)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    failed = []

    def calls():
        try:
            for t, (c, a) in zip((*trees, trees[0]), out):
                plo.render(t, rays, rgb=c, T=a, stream=stream)
        except plo.PloError as e:
            failed.append(e)

    graph = torch.cuda.CUDAGraph()
    thread = threading.Thread(target=calls)
    with torch.cuda.graph(graph, capture_error_mode="global"):
        plo.render(trees[0], small, rgb=rgb, T=T)
        thread.start()
        thread.join()
    assert not failed
    stream.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    want, wantT, _ = plo.render(trees[0], rays)
    torch.cuda.synchronize()
    for c, a in out:
        assert torch.equal(c, want) and torch.equal(a, wantT)
    assert torch.equal(rgb, want[:1000]) and torch.equal(T, wantT[:1000])
