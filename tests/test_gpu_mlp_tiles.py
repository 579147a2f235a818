"""Training and inference tiles of the learned-guess MLP (csrc/kt_mlp.cu) at batch sizes
around the tile (64 samples) and beyond one launch's blocks (512 tiles), on rows that are only
4-byte aligned, against the FP64 reference on the same BF16 weights and inputs; the same call
twice gives the same bits."""
import numpy as np
import pytest

from oracle import mlp_ref as R
from test_gpu_zlearned_guess import _close, _data, _ref_params, _split

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_04941_gb300 import build, kt as ktm
    build.build()
    return ktm


def _odd(a):
    import torch
    t = torch.empty(a.size + 1, dtype=torch.float32, device="cuda")[1:].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("B,nin,nout", [(1, 4, 1), (15, 16, 16), (63, 6, 3), (64, 13, 11), (65, 13, 11), (1000, 5, 2),
                                        (32768 + 130, 13, 11)])
def test_batch_sizes(kt, B, nin, nout):
    mlp = kt.Mlp(nin, nout, seed=B)
    X, Tg = _data(B, nin, nout, B)
    Xd, Td = _odd(X), _odd(Tg)
    g, loss = mlp.gradients(Xd, Td)
    g2, loss2 = mlp.gradients(Xd, Td)
    assert np.array_equal(g, g2) and loss == loss2
    P = _ref_params(kt, mlp)
    Xr = R.bf16_round(X[:, :].astype(np.float64))
    lref, gref = R.loss_and_grads(P, Xr, Tg.astype(np.float64))
    assert abs(loss - lref) <= 1e-2 * lref
    for l, ((gW, gb), (rW, rb)) in enumerate(zip(_split(kt, g), gref)):
        assert _close(gW, rW), (l, "W")
        assert _close(gb, rb), (l, "b")
    out = mlp.forward(Xd).cpu().numpy()
    ref, _ = R.forward(P, Xr)
    assert _close(out[:, :nout], ref[:, :nout], rel=1e-2) and np.all(out[:, nout:] == 0.0)
