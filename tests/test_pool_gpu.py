"""The scratch pool of a tree: kept between calls up to its bound, given back
with the tree, shared safely by threads and streams."""
import threading

import pytest

import paper_2207_05009_gb300 as plo
import plogen

pytestmark = pytest.mark.gpu


def _used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_pool_is_bounded_and_given_back(cuda_available):
    import torch
    host = plogen.luminaire_tree(plogen.LUMINAIRE_D6)
    rays = torch.from_numpy(plogen.rays_sphere(9 << 20, seed=90))  # 4 chunks: 2 x 94 MB of buffers
    tree = plo.Tree(host)
    plo.render_host(tree, rays[:1000])  # kernels loaded, streams made
    plo.render_host(tree, rays)
    tree.free()
    before = _used()
    for _ in range(3):
        tree = plo.Tree(host)
        for _ in range(2):
            plo.render_host(tree, rays)
        # 128 MB and what a pool rounds up to (32 MB blocks)
        assert _used() - before <= (128 + 64) << 20
        tree.free()
        assert _used() - before <= 4 << 20


def test_threads_and_streams_share_a_tree(cuda_available):
    import torch
    tree = plo.Tree(plogen.luminaire_tree(plogen.LUMINAIRE_D6))
    sizes = (1000, 400_000, 1_100_000, 600_000)
    rays = [torch.from_numpy(plogen.rays_sphere(n, seed=91 + i)).cuda() for i, n in enumerate(sizes)]
    want = [plo.render(tree, r)[:2] for r in rays]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        stream = torch.cuda.Stream()
        for _ in range(5):
            with torch.cuda.stream(stream):
                rgb, T, _ = plo.render(tree, rays[i], stream=stream)
                hr, hT = plo.render_host(tree, rays[i].cpu(), stream=stream)
            stream.synchronize()
            if not (torch.equal(rgb, want[i][0]) and torch.equal(T, want[i][1]) and
                    torch.equal(hr, want[i][0].cpu()) and torch.equal(hT, want[i][1].cpu())):
                bad.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    tree.check()


def test_pool_is_made_while_another_thread_captures(cuda_available):
    """The first call on a tree that needs scratch, from one thread, while
    another is capturing a render of the same tree."""
    import torch
    tree = plo.Tree(plogen.luminaire_tree(plogen.LUMINAIRE_D6))
    rays = torch.from_numpy(plogen.rays_sphere(500_000, seed=95)).cuda()
    small = rays[:1000].clone()
    plo.render(tree, small)
    torch.cuda.synchronize()
    rgb, T = torch.empty((1000, 3), device="cuda"), torch.empty(1000, device="cuda")
    big, bigT = torch.empty((500_000, 3), device="cuda"), torch.empty(500_000, device="cuda")
    stream = torch.cuda.Stream()

    def first_call():
        plo.render(tree, rays, rgb=big, T=bigT, stream=stream)
        stream.synchronize()

    graph = torch.cuda.CUDAGraph()
    thread = threading.Thread(target=first_call)
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        plo.render(tree, small, rgb=rgb, T=T)
        thread.start()
        thread.join()
    graph.replay()
    torch.cuda.synchronize()
    want, wantT, _ = plo.render(tree, rays)
    torch.cuda.synchronize()
    assert torch.equal(big, want) and torch.equal(bigT, wantT)
    assert torch.equal(rgb, want[:1000]) and torch.equal(T, wantT[:1000])
