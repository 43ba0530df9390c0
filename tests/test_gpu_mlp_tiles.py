"""The MLP gradient kernel (hidden-layer products on the tensor cores from three-term BF16
splits) at the edges of its chunks of 128 samples and of its rounds over the SMs, against the
FP64 oracle.

Tolerance: every gradient entry is a sum of n terms of FP32 accuracy; the entries of one
parameter block are compared in the 2-norm, 2e-6 of it (32 units of 2^-24: forward chains of
at most 64 + 64 products, the sum over a chunk, and one addition per block).
"""
import numpy as np
import pytest

from oracle import mlp as OM
from paper_2603_28710_gb300 import learned

pytestmark = pytest.mark.gpu
BLOCKS = {"W1": slice(0, 256), "b1": slice(256, 320), "W2": slice(320, 4416), "b2": slice(4416, 4480),
          "w3": slice(4480, 4544), "b3": slice(4544, 4545)}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 128, 129, 152 * 128, 152 * 128 + 1, 50001])
def test_gradient_blocks(n):
    import torch
    rng = np.random.default_rng(n)
    p = learned.init_params(n % 97) + rng.normal(0, 0.1, 4545).astype(np.float32)
    x = rng.normal(0, 1, (n, 4)).astype(np.float32)
    t = (x @ rng.normal(0, 1, 4) + 3.0).astype(np.float32)  # errors of one sign: no cancellation
    tr = learned.Trainer(p)
    loss = float(tr.grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()).item())
    g = tr.g.cpu().numpy().astype(np.float64)
    lo, go = OM.loss_and_grad(OM.bf16_round(p), x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - lo) < 2e-6 * lo
    for name, s in BLOCKS.items():
        assert np.linalg.norm(g[s] - go[s]) < 2e-6 * np.linalg.norm(go[s]), name
