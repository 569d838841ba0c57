"""The training loss of the seed network over batches of one tile, several and a ragged last one.

The loss is a sum over the whole batch of positive terms.  Each output carries FP32 rounding
of independent sign (a few 1e-7, which the sum over the batch averages out) and the kernels'
silu a relative error of at most a few units in the last place; the sum itself is in FP64.
The bound is 5e-7 for batches that average (half of the 1e-6 that FP32 additions of the
warps' sums into one word exceeded), and 2e-6 where a few samples stand for themselves."""
import numpy as np
import pytest

from oracle import mlp as ref_mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 65, 2047, 8192, 16384])
def test_loss_matches_fp64_reference(batch):
    import torch
    import paper_2210_08024_gb300 as P
    P.build()
    from paper_2210_08024_gb300 import tc
    g = np.random.default_rng(21)
    theta = g.normal(0.0, 0.2, ref_mlp.n_params()).astype(np.float32)
    parts = ref_mlp.unflatten(theta)
    th = ref_mlp.flatten([ref_mlp.bf16_round(p) if i % 2 == 0 else p for i, p in enumerate(parts)])
    net = tc.SeedNet(1)
    net.set_params(theta)
    net.set_norm(np.zeros(ref_mlp.N_IN), np.ones(ref_mlp.N_IN))
    for k in range(4):
        x = g.normal(0, 1, (batch, ref_mlp.N_IN)).astype(np.float32)
        y = g.normal(0, 1, (batch, 3)).astype(np.float32)
        _, loss = net.grad(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), (1.0, 2.0, 0.5))
        ref = ref_mlp.loss(th, x.astype(np.float64), y.astype(np.float64), (1.0, 2.0, 0.5))
        assert abs(float(loss.item()) - ref) <= (5e-7 if batch >= 2047 else 2e-6) * ref, (batch, k)
    net.close()
