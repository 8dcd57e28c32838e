"""The training gradient at the sizes where its tiles of 32 rows, its one-tile-per-block path and its
vector reductions begin and end, against FP64 sums of the same rounded forward."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,offset", [(1, 0), (31, 0), (32, 1), (33, 0), (1000, 3), (9728, 0), (9729, 0), (20000, 1)])
def test_loss_grad(n, offset):
    import torch

    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis, learned
    gen = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(n + 7, 22, generator=gen, device="cuda")
    T = 3 * torch.randn(n + 7, 5, generator=gen, device="cuda")
    idx = torch.randperm(n + 7, generator=gen, device="cuda")[:n].to(torch.int32)
    p = torch.from_numpy(learned.init_params(n)).cuda()
    buf = torch.full((agis.MLP_N_PARAMS + 8,), 7.0, device="cuda")
    grad = buf[offset:offset + agis.MLP_N_PARAMS]     # not 16-byte aligned for offset != 0
    loss = torch.empty(1, device="cuda")
    agis.mlp_loss_grad(p, X, T, grad, loss, idx=idx)
    torch.cuda.synchronize()
    bf = lambda x: x.to(torch.bfloat16).double()  # noqa: E731
    W, at = [], 0
    for s in ((64, 22), (64,), (64, 64), (64,), (5, 64), (5,)):
        m = int(np.prod(s))
        v = p[at:at + m].reshape(s)
        W.append(bf(v) if len(s) == 2 else v.double())
        at += m
    x, t = bf(X[idx.long()]), T[idx.long()].double()
    h1 = bf((x @ W[0].T + W[1]).relu().float())
    h2 = bf((h1 @ W[2].T + W[3]).relu().float())
    e = h2 @ W[4].T + W[5] - t
    dy = 2 * e / n
    d2 = (dy @ W[4]) * (h2 > 0)
    d1 = (d2 @ W[2]) * (h1 > 0)
    ref = torch.cat([v.reshape(-1) for v in (d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0))])
    # FP32 sums of up to 20,000 products: sqrt(n) 2^-24 of their size, and a hidden unit whose sum lies
    # within an ulp of a BF16 rounding boundary may round the other way (2^-8 of one of n x 128 units)
    assert (grad.double() - ref).norm() <= 2e-5 * ref.norm()
    assert abs(float(loss) - float(e.square().sum() / n)) <= 2e-5 * float(e.square().sum() / n)
    assert torch.all(buf[:offset] == 7.0) and torch.all(buf[offset + agis.MLP_N_PARAMS:] == 7.0)
