"""The learned terminator with BF16 operands on the tensor cores, against the
same network in FP64 with the operands rounded to BF16 where the kernels round
them: ragged batches around the 16 and 32 samples of a warp and of a block,
many blocks, and buffers that are only 4-byte aligned.

Tolerances: FP32 sums of 128 terms are good to 1e-6; now and then that moves a
value across a rounding boundary of BF16, which changes one operand by 2^-8 and
y by at most 2^-8 |w3| ~ 4e-4 (five of them: 2e-3), a gradient entry's sample by
2^-8 of it (2e-3 of the norm where there is one sample, and less with more).
"""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0
    return chi0


def _reference(p, x, t):
    import torch
    low = lambda a: a.float().bfloat16().double()  # noqa: E731
    p, x, t = (torch.from_numpy(a.astype(np.float32)).double() for a in (p, x, t))
    cut = np.cumsum([0, 640, 128, 16384, 128, 256, 2])
    w1, b1, w2, b2, w3, b3 = (p[a:b] for a, b in zip(cut, cut[1:]))
    w1, w2, w3 = low(w1.reshape(128, 5)), low(w2.reshape(128, 128)), low(w3.reshape(2, 128))
    h1 = torch.tanh(low(x) @ w1.T + b1)
    h2 = torch.tanh(low(h1) @ w2.T + b2)
    y = low(h2) @ w3.T + b3
    dy = (y - t) / len(x)
    d2 = (low(dy) @ w3) * (1.0 - h2 * h2)
    d1 = (low(d2) @ w2) * (1.0 - h1 * h1)
    g = torch.cat([(low(d1).T @ low(x)).flatten(), d1.sum(0), (low(d2).T @ low(h1)).flatten(), d2.sum(0),
                   (low(dy).T @ low(h2)).flatten(), dy.sum(0)])
    return y.numpy(), 0.5 * float(((y - t) ** 2).sum()) / len(x), g.numpy()


@pytest.mark.parametrize("B", [1, 15, 16, 17, 31, 33, 129, 60001])
@pytest.mark.parametrize("shift", [0, 1])
def test_bf16_network(lib, B, shift):
    import torch
    rng = np.random.default_rng(B)
    p = omlp.init_params(B) + 0.02 * rng.standard_normal(omlp.n_params())
    x = rng.standard_normal((B, 5))
    t = 0.3 * rng.standard_normal((B, 2))
    y_ref, l_ref, g_ref = _reference(p, x, t)

    def buf(n):   # n floats `shift` words behind a 16-byte boundary, guard words after them
        return torch.full((n + 8,), 7.0, device="cuda")[shift:]

    def put(a):
        b = buf(a.size)
        b[:a.size] = torch.from_numpy(a.astype(np.float32).ravel()).cuda()
        return b[:a.size]

    P, X, T = put(p), put(x).view(B, 5), put(t).view(B, 2)
    yb = buf(2 * B)
    lib.mlp_predict(P, X, yb[:2 * B].view(B, 2), bf16=True)
    assert bool((yb[2 * B:] == 7.0).all())
    assert np.abs(yb[:2 * B].view(B, 2).cpu().numpy() - y_ref).max() < 2e-3
    if B > 5000:
        return
    gb, n = buf(omlp.n_params()), lib.mlp_workspace_floats(B)
    wb, loss = buf(n), torch.zeros(1, device="cuda")
    lib.mlp_loss_grad(P, X, T, gb[:omlp.n_params()], loss, wb[:n], bf16=True)
    assert bool((gb[omlp.n_params():] == 7.0).all()) and bool((wb[n:] == 7.0).all())
    assert abs(loss.item() - l_ref) < 2e-3 * l_ref
    g = gb[:omlp.n_params()].cpu().numpy()
    assert np.linalg.norm(g - g_ref) < 2e-3 * np.linalg.norm(g_ref)
