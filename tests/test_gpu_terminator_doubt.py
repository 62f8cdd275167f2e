"""BF16 prediction on the tensor cores against the chain of FP32 multiply-adds whose
roundings it has to reproduce, for networks whose partial sums are large against
the weights (biases far above them) or against the result (sums that rise and
fall), beside trained-like ones.  The chains are followed in FP64, rounded to FP32
after each step; both weights of the last layer are 1, so that one rounding of an
operand taken the other way moves the output by 2^-9 of it.

tanhf may round either way within its two ulp (1.2e-7) of a boundary of BF16: samples with such a value in the first layer are left out, one in the second
adds the distance of the two neighbours to the tolerance of its sample, which
otherwise is that of 128 additions in FP32 of operands below 1, 2e-5.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 80000


def _networks():
    rng = np.random.default_rng(17)
    fall = np.where(np.arange(128) < 64, 1.0, -1.0)
    yield "bias", 0.005 * rng.standard_normal((128, 128)), 0.6 * np.sign(rng.standard_normal(128))
    yield "large bias", 0.02 * rng.standard_normal((128, 128)), 1.1 * np.sign(rng.standard_normal(128))
    yield "down from a bias", -0.147 * rng.uniform(size=(128, 128)), 8.0 + 0.2 * rng.standard_normal(128)
    yield "rise and fall", 0.1 * rng.uniform(size=(128, 128)) * fall, np.zeros(128)
    yield "initial", rng.uniform(-1, 1, (128, 128)) / np.sqrt(128), 0.1 * rng.standard_normal(128)
    yield "trained", 0.3 * rng.standard_normal((128, 128)), 0.3 * rng.standard_normal(128)


@pytest.mark.parametrize("name,w2,b2", list(_networks()), ids=[n[0] for n in _networks()])
def test_roundings_of_the_chain(name, w2, b2):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0 as lib
    rng = np.random.default_rng(5)
    up = name in ("rise and fall", "down from a bias")   # there every output of the first layer is near 1
    w1 = rng.standard_normal((128, 5)) * (0.2 if up else 1.0)
    b1 = 1.5 + 0.2 * rng.uniform(size=128) if up else 0.3 * rng.standard_normal(128)
    p = np.concatenate([w1.ravel(), b1, w2.ravel(), b2, np.ones(256), np.zeros(2)]).astype(np.float32)
    P = torch.from_numpy(p).cuda()
    X = torch.from_numpy(rng.uniform(-1, 1, (N, 5)).astype(np.float32)).cuda().bfloat16().float()
    dev = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()  # noqa: E731

    def chain(bias, x, w):
        z = dev(bias).double().expand(len(x), 128)
        for k in range(w.shape[1]):
            z = (z + x[:, k:k + 1].double() * dev(w).bfloat16().double()[:, k]).float().double()
        return z

    def neighbours(h):
        return [(h + d).float().bfloat16().double() for d in (-1.2e-7, 1.2e-7)]

    h1 = torch.tanh(chain(b1, X, w1))
    near = neighbours(h1)
    sure = (near[0] == near[1]).all(1)
    assert int(sure.sum()) > N // 2
    X, h1 = X[sure].contiguous(), near[0][sure]
    z = chain(b2, h1, w2)
    h2 = torch.tanh(z)
    near = neighbours(h2)
    ref = h2.float().bfloat16().double().sum(1)
    tol = 2e-5 + (near[1] - near[0]).sum(1)
    Y = torch.empty(len(X), 2, device="cuda")
    lib.mlp_predict(P, X, Y, bf16=True)
    off = (Y.double() - ref[:, None]).abs() > tol[:, None]
    assert int(off.sum()) == 0, int(off.any(1).sum())
