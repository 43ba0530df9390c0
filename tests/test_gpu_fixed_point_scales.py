"""Accuracy of the FP64 operator (csrc/fixline.cuh) at every node where the magnitudes within an
element or the element's side lengths differ by many orders: the error of a node's derivative is
bounded by the terms of the lines through that node, not by the largest value in its element.

With density 1 the density row of the operator is linear in the momenta (the dissipation of the
face flux vanishes), so its exact value is a sum over each line of nodes, taken here in extended
precision.  Tolerance, against S = sum of the absolute terms of the node's own lines: a trace
rounds N products and N sums, a line N + 2 of each, the directions add up: 4 (N + 2) eps S in the
worst case, and 2 eps S in the root mean square (that many independent roundings of at most half
a unit in partial sums below S, with sqrt(4 (N + 2) / 12) <= 2).  Paths and batches: equal bits.
"""
import numpy as np
import pytest

import oracle as O
from paper_2603_28710_gb300 import adg

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


def tables(N):
    """Sweep rows Q[i][a], traces l(-1), l(+1) and weights in extended precision, from the FP64
    nodes and weights that the library uses."""
    x, w = (np.asarray(t).astype(LD) for t in adg.host_gauss(N))
    lam = np.array([1 / np.prod([x[j] - x[k] for k in range(N) if k != j]) for j in range(N)], LD)
    D = np.zeros((N, N), LD)
    for a in range(N):
        for i in range(N):
            if i != a:
                D[a, i] = lam[i] / lam[a] / (x[a] - x[i])
        D[a, a] = -D[a].sum()
    at = [(lam / (y - x)) / (lam / (y - x)).sum() for y in (LD(-1), LD(1))]
    return (w[:, None] * D / w[None, :]).T, at[0], at[1], w


def density_row(m, dim, n_elem, N, h):
    """(d rho / dt, S) for density 1 and momenta m [dim][elements z.. x][nodes z.. x]."""
    Q, lm, lp, w = tables(N)
    k, S = np.zeros(m.shape[1:], LD), np.zeros(m.shape[1:], LD)
    for d in range(dim):
        ea, na = dim - 1 - d, 2 * dim - 1 - d
        f = np.moveaxis(m[d].astype(LD), na, -1)
        for absolute, out in ((False, k), (True, S)):
            op = np.abs if absolute else (lambda t: t)
            v = op(f)
            up, dn = (v * op(lp)).sum(-1), (v * op(lm)).sum(-1)  # traces at the two ends
            hi = (up + np.roll(dn, -1, ea)) / 2                    # numerical flux on the +d face
            lo = np.roll(hi, 1, ea)
            r = (v[..., None, :] * op(Q)).sum(-1)
            r = r + (op(lm / w) * lo[..., None] if absolute else (lm / w) * lo[..., None])
            r = r + (op(lp / w) * hi[..., None] if absolute else -(lp / w) * hi[..., None])
            out += 2 / LD(h[d]) * np.moveaxis(r, -1, na)
    return k, S


def state(kind, dim, n_elem, N, seed):
    """Density 1, momenta by kind, and an energy above the kinetic one."""
    rng = np.random.default_rng(seed)
    shape = tuple(n_elem[::-1]) + (N,) * dim
    m = rng.uniform(0.5, 1.0, (dim,) + shape) * rng.choice([-1.0, 1.0], (dim,) + shape)
    c = 1e-7
    if kind == "corner":        # one large node per element
        m *= c
        m[(Ellipsis,) + (0,) * dim] /= c
    elif kind == "row":         # flow along x, one small row of nodes in every element
        m[1:] = 0.0
        m[(Ellipsis, N // 2, slice(None))] *= c
    elif kind == "zero row":
        m[1:] = 0.0
        m[(Ellipsis, N // 2, slice(None))] = 0.0
    elif kind == "spread":      # eight orders from node to node
        m *= 10.0 ** rng.uniform(-8, 0, m.shape)
    elif kind == "along":       # flow along the long side only
        m[1:] = 0.0
    elif kind == "across":      # weak flow along the long side, strong across it
        m[0] *= c
    u = np.zeros((dim + 2,) + shape)
    u[0], u[1:1 + dim], u[dim + 1] = 1.0, m, 10.0
    return u, m


CASES = [("corner", 1.0), ("row", 1.0), ("zero row", 1.0), ("spread", 1.0), ("along", 100.0), ("along", 1e6),
         ("across", 1e3)]
MESHES = [(2, (3, 4), N) for N in range(2, 9)] + [(3, (3, 2, 2), N) for N in range(2, 7)]


@pytest.mark.parametrize("kind,aspect", CASES)
@pytest.mark.parametrize("dim,n_elem,N", MESHES)
def test_error_of_every_node(kind, aspect, dim, n_elem, N):
    hi = tuple(n / (1.0 if d == 0 else aspect) for d, n in enumerate(n_elem))
    s = adg.Solver(dim=dim, n_elem=n_elem, degree=N - 1, lo=(0.0,) * dim, hi=hi, dt=1e-3)
    u, m = state(kind, dim, n_elem, N, 7 * N + dim)
    k = s.rhs(u.reshape(s.shape))[0].reshape(m.shape[1:])
    s.close()
    ref, S = density_row(m, dim, n_elem, N, [hi[d] / n_elem[d] for d in range(dim)])
    err = np.abs(k - ref)
    assert np.all(k[S == 0] == 0.0)
    e = (err[S > 0] / (EPS * S[S > 0])).astype(float)
    assert e.max() <= 4 * (N + 2), e.max()
    assert np.sqrt(np.mean(e ** 2)) <= 2, np.sqrt(np.mean(e ** 2))


@pytest.mark.parametrize("kind", ["spread", "zero row", "mid"])
@pytest.mark.parametrize("dim,n_elem,N", [(2, (6, 5), 3), (2, (5, 4), 5), (2, (4, 4), 8), (3, (4, 3, 2), 3),
                                          (3, (2, 3, 2), 4)])
def test_paths_agree(kind, dim, n_elem, N):
    # split, element and fused path and a batch: the same bits, also where lines of one element
    # take the FP64 chain (mid: at odd N the middle node exceeds its lines by more than 2^5)
    u, m = state("spread" if kind == "mid" else kind, dim, n_elem, N, 11 * N + dim)
    if kind == "mid":
        u[1:1 + dim] *= 1e-9
        u[(slice(1, 1 + dim), Ellipsis) + (N // 2,) * dim] = 0.5
    out = {}
    kw = dict(n_elem=n_elem, degree=N - 1, P=(1,) * dim)
    for path in ("split", "element", "fused"):
        s = adg.Solver(dim=dim, lo=(0.0,) * dim, hi=(1.0, 0.1, 3.0)[:dim], dt=1e-5, rk="ck45", flux="sync",
                       kernel_path=path, **kw)
        s.set_state(u.reshape(s.shape))
        s.step(2)
        out[path] = s.get_state()
        s.close()
    assert np.isfinite(out["split"]).all()
    assert np.array_equal(out["split"], out["element"])
    assert np.array_equal(out["split"], out["fused"])
