"""The weight-gradient kernel where its tensor-core sums are moved into FP32
registers (every 256 rows): fewer, exactly as many, and more rows than that,
in every weight shape of the network, against float64."""
import pytest

import paper_2207_05009_gb300 as plo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_out,n_in", [(256, 256), (64, 256), (256, 64), (64, 64)])
def test_weight_gradient_row_counts(cuda_available, n_out, n_in):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n_out + n_in)
    for blocks in (1, 3, 4, 5, 8, 9, 152 * 4 + 1, 1500):
        M = 64 * blocks
        dZ = torch.randn(M, n_out, device="cuda", generator=g).to(torch.bfloat16)
        H = torch.randn(M, n_in, device="cuda", generator=g).to(torch.bfloat16)
        dW, err = plo.wgrad_bf16(dZ, H, torch.full((n_out, n_in), 0.5, device="cuda"))
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        ref = dZ.double().t() @ H.double() + 0.5
        # products are exact in FP32; at most 272 FP32 additions of one ulp
        # (2^-23) of the sum of magnitudes each lie between two flushes, whose
        # errors average out far below this bound
        bound = (dZ.double().abs().t() @ H.double().abs() + 0.5) * 272 * 2.0 ** -23
        assert bool(((dW.double() - ref).abs() <= bound).all()), blocks
