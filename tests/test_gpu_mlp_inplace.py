"""Results of the seed network's calls that lie in their own inputs (an output over the features, a
gradient over the batch) equal, bit for bit, those in buffers of their own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def net():
    import paper_2210_08024_gb300 as P
    P.build()
    from paper_2210_08024_gb300 import tc
    n = tc.SeedNet(3)
    yield tc, n
    n.close()


def _batch(B):
    import torch
    g = np.random.default_rng(B)
    return (torch.from_numpy(g.normal(0, 1, (B, 13)).astype(np.float32)).cuda(),
            torch.from_numpy(g.normal(0, 1, (B, 3)).astype(np.float32)).cuda())


@pytest.mark.parametrize("B,offset", [(4000, 0), (40000, 0), (40000, 13 * 64 + 1)])
def test_predict_over_the_features(net, B, offset):
    import torch
    tc, n = net
    X, _ = _batch(B)
    want = n.predict(X)
    flat = torch.cat([X.reshape(-1), torch.zeros(offset, device="cuda")])
    out = flat[offset: offset + 3 * B]
    assert tc.lib.tc_mlp_predict(n.h, flat.data_ptr(), B, out.data_ptr(), None) == 0
    torch.cuda.synchronize()
    assert torch.equal(out.reshape(B, 3), want)


@pytest.mark.parametrize("over", ["X", "Y"])
def test_gradient_over_the_batch(net, over):
    import torch
    tc, n = net
    B = 64  # one block: its sums have one order
    P = n.n_params()
    X, Y = _batch(B)
    want, loss = n.grad(X, Y)
    X1, Y1 = (torch.cat([v.reshape(-1), torch.zeros(P, device="cuda")]) for v in (X, Y))
    grad, loss1 = (X1 if over == "X" else Y1)[:P], torch.zeros(1, device="cuda")
    assert tc.lib.tc_mlp_grad(n.h, X1.data_ptr(), Y1.data_ptr(), B, None, grad.data_ptr(), loss1.data_ptr(), None) == 0
    torch.cuda.synchronize()
    assert torch.equal(grad, want) and torch.equal(loss1, loss)
