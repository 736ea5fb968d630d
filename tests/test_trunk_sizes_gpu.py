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
