"""adg_rhs_noalloc at its scratch limit: the largest mesh whose traces, face fluxes and 8960
bytes of tables fit into 32 MiB is accepted and gives the handle's right-hand side, one element
more is refused.  Tolerance 1e-12, that of the operator's parity tests.
"""
import pytest

from paper_2603_28710_gb300 import adg
from paper_2603_28710_gb300.inputs import random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,ne,per", [(2, 87358, 384), (3, 23295, 1440)])
def test_limit(dim, ne, per):
    import torch
    from paper_2603_28710_gb300 import build
    build.build()
    assert 8960 + per * ne <= 32 << 20 < 8960 + per * (ne + 1)
    n_elem, lo, hi = (ne,) + (1,) * (dim - 1), (0.0,) * dim, (float(ne),) + (1.0,) * (dim - 1)
    s = adg.Solver(dim=dim, n_elem=n_elem, degree=1, lo=lo, hi=hi, dt=1e-3)
    u = torch.from_numpy(random_state(s.shape, dim, seed=1)).cuda()
    ref, k = torch.empty_like(u), torch.full_like(u, float("nan"))
    s.rhs(u, ref)
    adg.rhs_noalloc(dim, n_elem, 1, u, k, lo=lo, hi=hi)
    torch.cuda.synchronize()
    assert float((k - ref).norm() / ref.norm()) < 1e-12
    v = torch.zeros((dim + 2) * (ne + 1) * 2 ** dim, dtype=torch.float64, device="cuda")
    with pytest.raises(adg.AdgError, match="scratch"):
        adg.rhs_noalloc(dim, (ne + 1,) + (1,) * (dim - 1), 1, v, torch.empty_like(v), lo=lo, hi=hi)
