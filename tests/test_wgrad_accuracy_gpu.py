"""The weight-gradient kernel's accuracy over long sums, where the tensor
core's truncation is biased: operands of one sign, and the bias gradients
beside the weights', against float64."""
import pytest

import paper_2207_05009_gb300 as plo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_out,n_in", [(256, 256), (64, 256), (256, 64), (64, 64)])
def test_sums_of_one_sign(cuda_available, n_out, n_in):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n_out + 3 * n_in)
    M = 1 << 21
    dZ = (0.5 + 0.5 * torch.rand(M, n_out, device="cuda", generator=g)).to(torch.bfloat16)
    H = (0.5 + 0.5 * torch.rand(M, n_in, device="cuda", generator=g)).to(torch.bfloat16)
    db = torch.zeros(n_out, device="cuda")
    dW, err = plo.wgrad_bf16(dZ, H, torch.zeros(n_out, n_in, device="cuda"), db=db)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref = sum(z.double().t() @ h.double() for z, h in zip(dZ.split(1 << 18), H.split(1 << 18)))
    refb = dZ.sum(0, dtype=torch.float64)
    # Relative to a sum of one sign.  Between two flushes 16 instructions each
    # align 16 products and the accumulator to the largest and cut them off at
    # one ulp (2^-23), and the accumulator is half full on average: 17 * 16 / 2
    # ulps.  Then one FP32 rounding (2^-24) per flush and per CTA, of which a
    # sum has at most 2^21 / 256 / 76 + 1 and 304.  (Without the flushes up to
    # 1,700 instructions follow each other, all cut off downwards: 1.3e-4 with
    # 256 x 256, 5.7e-5 with two of its halves.)
    bound = 17 * 16 / 2 * 2.0 ** -23 + ((1 << 21) // 256 // 76 + 1 + 304) * 2.0 ** -24
    assert bound < 4.2e-5
    assert float(((dW.double() - ref) / ref).abs().max()) <= bound
    assert float(((db.double() - refb) / refb).abs().max()) <= bound
