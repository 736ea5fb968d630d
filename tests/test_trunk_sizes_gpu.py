"""The layer-fused trunk at the edges of its tiles (a pair of CTAs takes 256
rows, 128 each, two tiles in flight): bit for bit the layer-by-layer GEMM."""
import numpy as np
import pytest

import paper_2207_05009_gb300 as plo
from tests.test_mlp_gpu import random_params, unflatten

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256, 257, 76 * 256, 76 * 256 + 1, 152 * 256 + 129, 153 * 256])
def test_trunk_equals_layer_by_layer_gemm(cuda_available, n):
    import torch
    flat = random_params(9)
    net = plo.Mlp(l_max=8.0)
    net.set_params(flat)
    net.forward(torch.from_numpy(np.random.default_rng(n).random((n, 3)).astype(np.float32)).cuda())
    h = net.activation(0, n)
    Ws, bs = unflatten(flat)
    for l in range(8):
        W = np.zeros((256, h.shape[1]), np.float32)
        W[:, :Ws[l].shape[1]] = Ws[l]
        h, err = plo.gemm_bf16(h.contiguous(), torch.from_numpy(W).cuda().to(torch.bfloat16), 0,
                               bias=torch.from_numpy(bs[l].astype(np.float32)).cuda())
        assert torch.equal(h, net.activation(l + 1, n)), l
    net.check()


@pytest.mark.parametrize("n", [1, 3, 4, 126, 127, 128, 130, 257, 76 * 256 + 131])
def test_head_rows_reach_any_buffer(cuda_available, n):
    """The linear head, the trunk's ninth job: bit for bit the single-layer
    GEMM on the eighth layer's output, in a 16-byte aligned buffer (written by
    the kernel, the last rows of a count that is not a multiple of four apart)
    and in one that is not; no value next to the rows changes."""
    import torch
    flat = random_params(9)
    net = plo.Mlp(l_max=8.0)
    net.set_params(flat)
    x = torch.from_numpy(np.random.default_rng(n).random((n, 3)).astype(np.float32)).cuda()
    net.forward(x)
    Ws, bs = unflatten(flat)
    W, b = np.zeros((64, 256), np.float32), np.zeros(64, np.float32)
    W[:49], b[:49] = Ws[8], bs[8]
    want, err = plo.gemm_bf16(net.activation(8, n), torch.from_numpy(W).cuda().to(torch.bfloat16), 1,
                              bias=torch.from_numpy(b).cuda())
    for off in (0, 4, 1):
        buf = torch.full((n * 49 + 64,), -7.0, device="cuda")
        plo._check(plo.mlp_lib().plo_mlp_forward(net._h, plo._ptr(x), n, plo._ptr(buf[off:]), None))
        torch.cuda.synchronize()
        assert torch.equal(buf[off:off + n * 49].view(n, 49), want[:, :49]), off
        assert bool((buf[:off] == -7.0).all()) and bool((buf[off + n * 49:] == -7.0).all()), off
    net.check()
