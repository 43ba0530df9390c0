"""The trace section of a checkpoint: the same order, [direction][side][variable][element][face
node], in every arithmetic, whatever order the operator keeps on the device, and about as fast to
save or restore in FP32 as in FP32 pairs, whose section is twice as long (factor 2 for noise).

Tolerance of the values: FP32 interpolation of FP32 values, (2 N + 1) 2^-24 sum |weights| max |w|.
"""
import statistics
import time

import numpy as np
import pytest

import oracle as O
from paper_2603_28710_gb300 import adg
from paper_2603_28710_gb300.inputs import random_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


def traces_of(u, dim, n_elem, N):
    """[d][side][v][e][j] in FP64 from u [v][e][node]."""
    x, _ = O.gauss(N)
    l = [np.array([O.lagrange(x, a, y) for a in range(N)]) for y in (-1.0, 1.0)]
    w = u.reshape((dim + 2, u.shape[1]) + (N,) * dim)
    out = [[np.tensordot(w, l[side], ([1 + dim - d], [0])).reshape(dim + 2, u.shape[1], -1)
            for side in range(2)] for d in range(dim)]
    return np.array(out)


@pytest.mark.parametrize("path", ["split", "element"])
@pytest.mark.parametrize("precision", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("dim,n_elem,degree", [(2, (7, 5), 3), (3, (3, 4, 5), 2)])
def test_order(dim, n_elem, degree, precision, path):
    N = degree + 1
    s = adg.Solver(dim=dim, n_elem=n_elem, degree=degree, dt=1e-3, precision=precision, kernel_path=path)
    u = random_state(s.shape, dim, seed=9)
    s.set_state(u)
    buf = s.checkpoint()
    ref = traces_of(u, dim, n_elem, N)
    kind = {"fp64": np.float64, "fp32": np.float32, "df64": np.float32}[precision]
    per = 2 if precision == "df64" else 1
    section = buf[len(buf) - ref.size * per * np.dtype(kind).itemsize:].copy().view(kind)
    t = section.reshape(ref.shape + (per,)).astype(np.float64).sum(-1)
    x, _ = O.gauss(N)
    tol = (2 * N + 1) * 2.0 ** -24 * sum(abs(O.lagrange(x, a, 1.0)) for a in range(N)) * np.abs(u).max()
    assert np.abs(t - ref).max() <= tol
    # restored into a fresh handle and saved again: the same bytes
    r = adg.Solver(dim=dim, n_elem=n_elem, degree=degree, dt=1e-3, precision=precision, kernel_path=path)
    r.restore(buf)
    assert np.array_equal(r.checkpoint(), buf)
    s.close()
    r.close()


def test_time():
    def seconds(precision):
        s = adg.Solver(dim=3, n_elem=(48,) * 3, degree=3, lo=(0.0,) * 3, hi=(1.0,) * 3, dt=1e-3,
                       precision=precision)
        s.init_tgv(0.1)
        buf = s.checkpoint()
        t = []
        for _ in range(5):
            t0 = time.perf_counter()
            s._chk(s._L.adg_checkpoint_save(s._h, adg._np_ptr(buf), buf.size))
            t1 = time.perf_counter()
            s.restore(buf)
            t.append((t1 - t0, time.perf_counter() - t1))
        s.close()
        return [statistics.median(c) for c in zip(*t)]
    pairs, single = seconds("df64"), seconds("fp32")
    print("save, restore: pairs %.3f %.3f s, FP32 %.3f %.3f s" % (*pairs, *single))
    assert single[0] <= 2 * pairs[0] and single[1] <= 2 * pairs[1]
