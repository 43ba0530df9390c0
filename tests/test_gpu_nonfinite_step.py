"""A time step that is not finite is visible in the FP64 operator's state: also of a uniform gas,
whose right-hand side is rounding noise, a step with it leaves no variable finite at any node.  In
FP32 and FP32 pairs adg_check_finite reports it.
"""
import numpy as np
import pytest

from paper_2603_28710_gb300 import adg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


def uniform(shape):
    u = np.ones(shape)
    u[1], u[2], u[-1] = 0.5, -0.25, 2.5
    return u


@pytest.mark.parametrize("path", ["split", "element", "fused"])
@pytest.mark.parametrize("dim,n_elem,degree", [(2, (6, 5), 2), (2, (4, 4), 4), (3, (3, 2, 2), 3)])
@pytest.mark.parametrize("step", [{"dt": np.inf}, {"cfl": np.inf}])
def test_infinite_time_step(step, dim, n_elem, degree, path):
    s = adg.Solver(dim=dim, n_elem=n_elem, degree=degree, rk="ck45", kernel_path=path, **step)
    s.set_state(uniform(s.shape))
    s.step(1)
    assert not s.check_finite()
    assert not np.isfinite(s.get_state()).any()
    s.close()


def test_infinite_time_step_in_a_batch():
    b = adg.Batch([dict(n_elem=(4, 4), degree=3, P=(1, 1)), dict(n_elem=(3, 5), degree=2, P=(1, 1))],
                  flux="sync", rk="ck45", dt=np.inf, precision="fp64")
    for i, shape in enumerate([(4, 16, 16), (4, 15, 9)]):
        b.set_state(i, uniform(shape))
    b.step(1)
    for i in range(2):
        assert not np.isfinite(b.get_state(i)).any()


@pytest.mark.parametrize("path", ["split", "element", "fused"])
@pytest.mark.parametrize("precision", ["df64", "fp32"])
@pytest.mark.parametrize("rk", ["ck45", "rk33"])
@pytest.mark.parametrize("step", [{"dt": np.inf}, {"cfl": np.inf}])
def test_the_check_sees_it_in_the_other_arithmetics(step, rk, precision, path):
    s = adg.Solver(n_elem=(6, 5), degree=2, rk=rk, precision=precision, kernel_path=path, **step)
    s.init_vortex()
    assert s.check_finite()
    s.step(1)
    assert not s.check_finite()
    s.close()
