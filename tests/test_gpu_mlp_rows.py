"""Batch inference of the learned-guess MLP (csrc/kt_mlp.cu infer) across its launch shapes: a row's
outputs are the same bits whatever batch it is in."""
import pytest

from test_gpu_mlp_tiles import kt  # noqa: F401

pytestmark = pytest.mark.gpu


def test_rows_do_not_depend_on_the_batch(kt):  # noqa: F811
    import torch
    mlp = kt.Mlp(13, 11, seed=3)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    line = 2 * sm * 64                      # rows of the largest launch of four-warp blocks
    X = torch.randn(4 * line + 77, 16, device="cuda")
    want = torch.cat([mlp.forward(X[i:i + 1000].contiguous()) for i in range(0, X.shape[0], 1000)])
    for n in (1, 64, 65, line, line + 1, 2 * line, 2 * line + 1, X.shape[0]):
        got = mlp.forward(X[:n].contiguous())
        assert torch.equal(got, want[:n]), n
