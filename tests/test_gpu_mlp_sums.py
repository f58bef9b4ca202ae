"""The sums over samples of the cost model's gradient and loss.

Gradient: no less precise than FP64 sums of exact products.  A network whose activations are
whole numbers (zero W1 and W2, b1 = c, b2 in equal pairs under w3 = +1, -1, so that y = 0) and
targets that make dL/dy whole: every term of a sum is then a whole number, and the magnitudes
of the terms sum to less than 2**53, so FP64 sums are exact in any order and the gradient has
to be the exact sum rounded to FP32.  The terms cancel down to their last bits, which sums of
48 bits lose.

Loss: its FP64 sum runs in an order that the number of samples fixes, on any GPU: parts of
about 38 samples (at most 152), batches of 16 samples within a part, each of the 16 in a
chain of its own, then the parts in eight interleaved chains."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2504_21450_gb300 import vlasov

from test_gpu_costmodel import stream, workspace

pytestmark = pytest.mark.gpu


def gradient(p, x, t):
    import torch
    vlasov.load(build_if_missing=True)
    n = t.size
    P, X, T = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in (p, x, t))
    buf, ws, nbytes = workspace(n)
    grad, loss = torch.zeros_like(P), torch.zeros(1, dtype=torch.float64, device="cuda")
    vlasov.vl_mlp_gradient(P.data_ptr(), X.data_ptr(), T.data_ptr(), n, ws, nbytes, grad.data_ptr(),
                           loss.data_ptr(), stream())
    return grad.cpu().numpy(), float(loss.item())


def cancelling(n, bits, shift, rng):
    """n whole numbers of `bits` bits times up to 2**shift that cancel but for four small ones, the
    positive ones first."""
    a = rng.integers(2 ** (bits - 1), 2 ** bits, n // 2 - 2) | 1
    a = a << rng.integers(0, shift + 1, a.size)
    return np.concatenate([a, [1, 2, 4, 8], -a])


# c: bits of the activations
@pytest.mark.parametrize("n, bits, shift, c", [(16, 24, 0, 24), (32, 24, 22, 1), (64, 23, 0, 23), (64, 20, 5, 21),
                                               (256, 23, 0, 21), (1024, 22, 0, 20)])
def test_gradient_is_as_precise_as_fp64(n, bits, shift, c):
    rng = np.random.default_rng(112)
    dy = cancelling(n, bits, shift, rng)
    assert np.array_equal(dy.astype(np.float32).astype(np.int64), dy)
    c1 = rng.integers(2 ** (c - 1), 2 ** c, omlp.NH)
    c2 = np.repeat(rng.integers(2 ** (c - 1), 2 ** c, omlp.NH // 2), 2)
    w3 = np.tile([1, -1], omlp.NH // 2)
    zero = np.zeros
    p = omlp.pack(zero((omlp.NH, omlp.NIN)), c1, zero((omlp.NH, omlp.NH)), c2, w3, 0.0)
    t = -dy.astype(np.float64) * (n / 2)  # dL/dy = 2 (0 - t) / n
    x = rng.integers(-4, 5, (n, omlp.NIN))
    assert np.abs(dy).sum() * 2 ** c < 2 ** 53
    s = int(dy.sum())
    assert s != 0 and abs(s) < 2 ** bits
    want = omlp.pack(zero((omlp.NH, omlp.NIN)), zero(omlp.NH), np.outer(w3, c1) * s, w3 * s, c2 * s, s)
    np.testing.assert_array_equal(gradient(p, x, t)[0], want.astype(np.float32))


@pytest.mark.parametrize("n", [1, 16, 40, 300, 1000, 5696, 7001])
def test_order_of_the_loss(n):
    rng = np.random.default_rng(113)
    t = rng.normal(size=n).astype(np.float32)
    _, loss = gradient(np.zeros(omlp.NPARAM), np.zeros((n, omlp.NIN)), t)  # y = 0
    most = max(1, min(152, (vlasov.vl_mlp_workspace_bytes(n) - 256 - (4 * omlp.NPARAM + 255) // 256 * 256)
                      // (8 * (omlp.NPARAM + 1))))
    per = -(-n // most)
    sq = t.astype(np.float64) ** 2  # exact
    parts = []
    for a in range(0, n, per):
        chains = [0.0] * 16
        for s in range(a, min(a + per, n)):
            chains[(s - a) % 16] += sq[s]
        e = 0.0
        for v in chains:
            e += v
        parts.append(e)
    total = parts[0]
    if len(parts) > 1:
        sums = [0.0] * 8
        for i, e in enumerate(parts):
            sums[i % 8] += e
        total = sums[0]
        for v in sums[1:]:
            total += v
    assert loss == total / n
