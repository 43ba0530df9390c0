"""The predictor's kernels at the largest sample count that they accept, 2^31 - 1, whose last tile
and chunk end beyond the 32-bit signed range: outputs of the last samples as for those samples
alone, and the loss of equal samples.

Tolerance of the loss: a thread adds up the terms of 2^31 / (128 x 152) = 110377 chunks in FP32, an
error of at most 110377 x 2^-24 = 0.7 %; 2 % for all sums of a block.
"""
import numpy as np
import pytest

from paper_2603_28710_gb300 import learned

pytestmark = pytest.mark.gpu
N = 2 ** 31 - 1


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


def test_largest_sample_count():
    import torch
    p = learned.init_params(3) + np.random.default_rng(3).normal(0, 0.1, 4545).astype(np.float32)
    tr = learned.Trainer(p)
    x = torch.zeros((N, 4), device="cuda")
    y0 = float(tr.forward(x[:1])[0])
    target = torch.zeros(N, device="cuda")
    loss = float(tr.grad(x, target)[0])
    assert abs(loss - y0 * y0) <= 0.02 * y0 * y0
    del target
    x[-200:] = torch.randn((200, 4), device="cuda")
    tail = tr.forward(x[-200:].clone())
    y = tr.forward(x)
    assert torch.equal(y[-200:], tail) and bool((y[:-200] == y0).all())
    del x, y
    torch.cuda.empty_cache()
