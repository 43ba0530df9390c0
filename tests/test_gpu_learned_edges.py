"""The predictor's inference kernel at the edges of its tiles of 16 samples and of its grid, and
its inputs for stored levels of any magnitude (the reciprocal of the level spread has a short
form between 2^-100 and 2^100).

Tolerances.  Inference: an activation carries at most 8 rounding errors of 2^-24 (products and
sum of the first layer, tanh), a hidden sum 12 tensor-core additions with truncation (24 of
them) and the splits, an output sum 64; each of them scaled by the absolute weights that
follow, 128 x 2^-24 x sum |w3| (1 + sum |W2|) in all.  Inputs: one FP32 rounding of a value that
is exact to 1e-12, 2^-24 of it; targets two (the estimate in FP64 is exact to 1e-9).
"""
import numpy as np
import pytest

from oracle import mlp as OM
from paper_2603_28710_gb300 import adg, learned

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 152 * 7 * 64, 152 * 7 * 64 + 1, 200003])
def test_inference(n):
    import torch
    rng = np.random.default_rng(n)
    p = learned.init_params(n % 89) + rng.normal(0, 0.1, 4545).astype(np.float32)
    x = rng.normal(0, 1, (n, 4)).astype(np.float32)
    y = learned.Trainer(p).forward(torch.from_numpy(x).cuda()).cpu().numpy().reshape(-1)
    q = OM.bf16_round(p).astype(np.float64)
    w1, b1, w2, b2 = q[:256].reshape(64, 4), q[256:320], q[320:4416].reshape(64, 64), q[4416:4480]
    ref = np.tanh(np.tanh(x.astype(np.float64) @ w1.T + b1) @ w2.T + b2) @ q[4480:4544] + q[4544]
    tol = 128 * 2.0 ** -24 * np.sum(np.abs(q[4480:4544]) * (1 + np.abs(w2).sum(1)))
    assert y.shape == (n,) and np.all(np.abs(y - ref) < tol)


@pytest.mark.parametrize("scale", [1e-290, 2.0 ** -101, 2.0 ** -90, 1.0, 2.0 ** 90, 2.0 ** 101, 1e290])
def test_inputs_of_any_magnitude(scale):
    import torch
    rng = np.random.default_rng(3)
    s = adg.Solver(n_elem=(8, 8), degree=2, P=(2, 2), max_delay=0, flux="at_trace", at_np=2,
                   rk="ck45", cfl=0.1)
    rec = s.set_trace_log(None, 0)
    L = (rng.choice([-1.0, 1.0], rec) * scale) * (1 + 1e-3 * rng.uniform(-1, 1, (50, rec)))
    L[:, ::7] = L[0, ::7]                         # constant levels: no sample
    picks = np.stack([rng.integers(0, rec, 300), rng.integers(6, 10, 300), rng.integers(0, 5, 300),
                      rng.integers(1, 5, 300)], 1).astype(np.int32)
    x = torch.empty((300, 4), dtype=torch.float32, device="cuda")
    t, ok = torch.empty(300, device="cuda"), torch.empty(300, dtype=torch.int32, device="cuda")
    s.learned_samples(torch.from_numpy(L).cuda(), 50, torch.from_numpy(picks).cuda(), x, t, ok)
    x, t, ok = x.cpu().numpy(), t.cpu().numpy(), ok.cpu().numpy()
    cs = adg.host_rk("ck45")[2]
    LL = L.astype(np.longdouble)
    for i, (c, st, m, k) in enumerate(picks):
        if c % 7 == 0:
            assert ok[i] == 0 and not x[i].any()
            continue
        a = [LL[(st - k - l) * 5, c] for l in range(3)]
        km = np.longdouble(k + cs[m])
        d0, d1 = a[0] - a[1], a[1] - a[2]
        e3 = (km + 1) * (km + 2) / 2 * a[0] - km * (km + 2) * a[1] + km * (km + 1) / 2 * a[2]
        est, sp = e3 - a[0] - km * d0, abs(d0) + abs(d1)
        assert ok[i] == 1
        np.testing.assert_allclose(x[i], np.array([d0 / sp, d1 / sp, k / 8, cs[m]], np.float64),
                                   rtol=6.1e-8, atol=0)
        np.testing.assert_allclose(t[i], float((LL[st * 5 + m, c] - e3) / est), rtol=1.3e-7, atol=1e-7)
