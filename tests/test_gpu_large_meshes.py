"""Meshes whose face traces pass 2^31 values (their degrees of freedom do not): a state that
repeats along z with the period of a small mesh gives that mesh's results, bit for bit, in every
copy.  Covers the three arithmetics, the right-hand side and steps on the split and element path.
"""
import numpy as np
import pytest

from paper_2603_28710_gb300 import adg
from paper_2603_28710_gb300.inputs import random_state

pytestmark = pytest.mark.gpu

SMALL, COPIES, DEGREE = (264, 264, 4), 66, 1   # 18.4 M elements: 2.2e9 trace values, 0.74e9 DoF


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


def pair(n_elem, copies, degree, **kw):
    """Solvers of a mesh and of `copies` of it along z, with elements of the same size."""
    out = []
    for c in (1, copies):
        n = n_elem[:2] + (n_elem[2] * c,)
        out.append(adg.Solver(dim=3, n_elem=n, degree=degree, lo=(0.0,) * 3,
                              hi=(float(n[0]), float(n[1]), float(n[2])), dt=1e-3, **kw))
    return out


def same_in_every_copy(big, small, copies):
    """big [v][copies * e][node] against small [v][e][node], one variable at a time."""
    return all(bool((b.reshape(copies, -1) == s.reshape(1, -1)).all()) for b, s in zip(big, small))


@pytest.mark.parametrize("precision,path", [("fp64", "split"), ("fp64", "element"), ("fp32", "split"),
                                            ("fp32", "element"), ("df64", "split")])
def test_traces_beyond_2_31_values(precision, path):
    import torch
    small, big = pair(SMALL, COPIES, DEGREE, precision=precision, kernel_path=path)
    assert 2 * 3 * 5 * 4 * SMALL[0] * SMALL[1] * SMALL[2] * COPIES >= 2 ** 31 > big.n_dof
    u = torch.from_numpy(random_state(small.shape, 3, seed=5)).cuda()
    U = u.repeat(1, COPIES, 1)
    for step in (False, True):
        if step:
            small.set_state(u)
            big.set_state(U)
            small.step(1)
            big.step(1)
            k, K = small.get_state(torch.empty_like(u)), big.get_state(U)
        else:
            k, K = small.rhs(u, torch.empty_like(u)), big.rhs(U, torch.empty_like(U))
        assert bool(torch.isfinite(k).all()) and same_in_every_copy(K, k, COPIES)
        del K
    small.close()
    big.close()
    del U
    torch.cuda.empty_cache()
