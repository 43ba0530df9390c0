"""Accuracy of the predictor's inference kernel against a plain FP32 evaluation of the same network.

The hidden layer's activations enter the tensor cores as three BF16 terms.  Tolerance: 8 times the
root mean square and the largest error of the FP32 evaluation (numpy), on the same samples: the
kernel rounds as often, but its tensor-core sums truncate 12 times per output where FP32 sums round
to nearest (a bias of half a unit per addition, 12 / 2 units against sqrt(64 / 12) of them), and its
tanh may be off by 2 units.  A kernel that loses the third term, or feeds it from the wrong lanes,
is outside of it: emulated with two terms, the errors are 11 to 17 times the FP32 ones (checked on
the CPU).
"""
import numpy as np
import pytest

from oracle import mlp as OM
from paper_2603_28710_gb300 import learned

F = np.float32


def network(seed, n):
    rng = np.random.default_rng(seed)
    p = learned.init_params(seed) + rng.normal(0, 0.1, 4545).astype(F)
    x = rng.normal(0, 1, (n, 4)).astype(F)
    q = OM.bf16_round(p)
    return p, x, [np.asarray(t, F) for t in OM.unpack(q)], OM.forward(q.astype(np.float64), x)[0]


def spread(y, ref):
    e = y.astype(np.float64) - ref
    return np.sqrt(np.mean(e ** 2)), np.abs(e).max()


def evaluate(x, weights, terms=None):
    """FP32 evaluation; with `terms`, the first activations as that many BF16 terms."""
    W1, b1, W2, b2, w3, b3 = weights
    h = np.tanh(x @ W1.T + b1)
    if terms is None:
        z = h @ W2.T
    else:
        r, z = h.astype(np.float64), 0.0
        for _ in range(terms):
            t = OM.bf16_round(r.astype(F)).astype(np.float64)
            z, r = z + t @ W2.T.astype(np.float64), r - t
        z = np.asarray(z, F)
    return np.tanh(z + b2) @ w3 + b3


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_two_terms_are_outside_the_tolerance(seed):
    _, x, weights, ref = network(seed, 4096)
    plain = spread(evaluate(x, weights), ref)
    three, two = spread(evaluate(x, weights, 3), ref), spread(evaluate(x, weights, 2), ref)
    assert all(t <= 8 * f for t, f in zip(three, plain))
    assert all(t > 8 * f for t, f in zip(two, plain))


@pytest.mark.gpu
@pytest.mark.parametrize("seed,n", [(1, 4096), (2, 4097), (3, 100003)])
def test_inference(seed, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()
    p, x, weights, ref = network(seed, n)
    y = learned.Trainer(p).forward(torch.from_numpy(x).cuda()).cpu().numpy().reshape(-1)
    plain, got = spread(evaluate(x, weights), ref), spread(y, ref)
    assert all(g <= 8 * f for g, f in zip(got, plain)), (got, plain)
