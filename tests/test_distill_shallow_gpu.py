"""Distillation into trees with fewer voxels than samples per voxel (depth 1
and 2): one voxel's samples then set the size of the network's workspace."""
import numpy as np
import pytest

import paper_2207_05009_gb300 as plo
from oracle import mlp as omlp
from tests.test_mlp_gpu import bf16, random_params, unflatten

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth,samples", [(1, 129), (1, 256), (2, 129), (2, 256)])
def test_more_samples_than_voxels(cuda_available, depth, samples):
    import torch
    seed, flat = 99, random_params(7, scale=0.6)

    def network():
        net = plo.Mlp(l_max=5.0, jitter_seed=seed)
        net.set_params(flat)
        return net

    got = network().distill(depth, samples=samples, sigma_thresh=0.0).export()
    # a workspace made by a larger call first
    net = network()
    net.forward(torch.rand(1024, 3, device="cuda"))
    again = net.distill(depth, samples=samples, sigma_thresh=0.0).export()
    for a, b in ((got.child, again.child), (got.sigma, again.sigma), (got.sh, again.sh)):
        np.testing.assert_array_equal(a, b)
    # threshold 0 keeps every voxel; the leaves are in Morton order
    G = 1 << depth
    idx = np.arange(G ** 3)
    ijk = np.stack([idx % G, (idx // G) % G, idx // (G * G)], 1)
    codes = np.array(omlp.morton_code(ijk, depth), dtype=np.int64)
    ijk = ijk[np.argsort(codes)]
    assert got.n_leaves == G ** 3
    Ws, bs = unflatten(flat)
    jit = omlp.distill_jitter(seed, np.sort(codes), samples)
    raw, _ = omlp.forward([bf16(w) for w in Ws], bs,
                          omlp.positional_encoding(((ijk[:, None, :] + jit) / G).reshape(-1, 3)))
    raw = raw.reshape(G ** 3, samples, -1)
    sig, sh = np.maximum(raw[..., 0], 0).mean(1), raw[..., 1:].mean(1)
    # the network's bf16 precision (threshold 0 keeps voxels of any density,
    # so the densities are held to 3% of the largest, as the coefficients are)
    np.testing.assert_allclose(got.sigma, sig, rtol=0, atol=3e-2 * float(np.abs(sig).max()))
    np.testing.assert_allclose(got.sh.reshape(G ** 3, -1), sh, rtol=0, atol=3e-2 * float(np.abs(sh).max()))
