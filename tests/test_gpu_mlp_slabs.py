"""The cost model's gradient at the edges of its batches (16 samples) and parts (one CTA, one
part, several parts, more samples than a part per SM): FP64 sums over the oracle's
activations in the same tolerance as the other gradient tests, and the same result twice,
with a loss pointer that is only 4-byte aligned as well."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2504_21450_gb300 import vlasov

from test_gpu_costmodel import mlp_case, stream, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 15, 16, 17, 38, 39, 77, 1000, 6001])
def test_gradient(n):
    import torch
    vlasov.load(build_if_missing=True)
    P, X, T, p, x, t = mlp_case(n, seed=11)
    buf, ws, nbytes = workspace(n)
    want, want_loss = omlp.gradient(p, x, t), omlp.loss(p, x, t)
    out = []
    for shift in (0, 4, 0):
        grad = torch.full_like(P, 7.0)
        room = torch.zeros(32, dtype=torch.uint8, device="cuda")
        vlasov.vl_mlp_gradient(P.data_ptr(), X.data_ptr(), T.data_ptr(), n, ws, nbytes, grad.data_ptr(),
                               room.data_ptr() + shift, stream())
        loss = float(room.cpu()[shift:shift + 8].clone().view(torch.float64)[0])
        assert loss == pytest.approx(want_loss, rel=1e-5)
        out.append((grad.cpu().numpy(), loss))
    np.testing.assert_allclose(out[0][0], want, rtol=0, atol=1e-5 * np.abs(want).max())
    for g, loss in out[1:]:
        np.testing.assert_array_equal(g, out[0][0])
        assert loss == out[0][1]
