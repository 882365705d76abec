"""The fused MLP kernels at the edges of their tiles: rows just below, at and
above 128-row tiles and tile pairs, frames that change inside a warp's rows and
inside a tile (the shared time encoding), against the one-GEMM-per-layer path
(same operands, same MMA order: bit-identical offsets, dZ and encoding gradient;
weight gradients equal up to summation order)."""
import numpy as np
import pytest
import torch

from paper_2505_05356_gb300 import mlp, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,B", [(1, 1), (127, 1), (128, 1), (129, 1), (256, 1), (257, 1),
                                 (5, 40), (33, 7), (100, 64)])
def test_fused_equals_layerwise_at_tile_edges(N, B):
    rng = np.random.default_rng(N * 100 + B)
    theta = torch.as_tensor(scenes.init_mlp_params(3, head_std=0.05), device="cuda")
    theta += 0.01 * torch.as_tensor(rng.standard_normal(theta.numel()).astype(np.float32),
                                    device="cuda")
    means = torch.as_tensor(rng.uniform(-2, 4, (N, 3)).astype(np.float32), device="cuda")
    times = list(np.linspace(0, 1, B).astype(np.float32))
    dd = torch.as_tensor(rng.standard_normal((B, N, 3)).astype(np.float32), device="cuda")
    net = mlp.DeformationMLP(N, B, 0.2)

    def run():
        d = net.forward(theta, means, times).clone()
        g, m = net.backward(theta, means, times, dd)
        keep = [net.export("enc").clone(), net.export("d_enc").clone()]
        keep += [net.export(w, l).clone() for w in ("H", "dZ") for l in range(8)]
        return d, g.clone(), m.clone(), keep

    mlp.debug_inject(2)
    try:
        ref = run()
    finally:
        mlp.debug_inject(0)
    got = run()
    net.check()
    assert torch.equal(got[0], ref[0])
    for a, b in zip(got[3], ref[3]):
        assert torch.equal(a, b)
    assert torch.equal(net.infer(theta, means, times), ref[0])
    # sums of at most B N rows of equal terms in another order: a few roundings each
    for a, b in ((got[1], ref[1]), (got[2], ref[2])):
        assert float((a - b).double().norm()) <= 1e-5 * float(b.double().norm())
