"""The FP64 operator's fixed-point contractions (csrc/fixline.cuh) at the edges of their range:
element counts around the tile sizes, fields of very different magnitude, exact zeros,
magnitudes that need the FP64 chain, and non-finite values.

Tolerance: S = sum_d (2/h_d) Lambda max|F_d| bounds the terms an operator evaluation sums per
element and variable (F_d over the element and its face neighbours, whose fluxes enter through
the faces); each of the two evaluations rounds about 2d (p+1) + 2d of them, in its own order,
plus the pointwise and face fluxes: 256 eps S, as for the other operator comparisons.
"""
import numpy as np
import pytest

import oracle as O
from paper_2603_28710_gb300 import adg
from paper_2603_28710_gb300.inputs import random_state

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build
    build.build()


def sum_scale(u, dim, degree, n_elem, h):
    """[var][elem]: S with the maximum over the element and its face neighbours, from the
    fluxes and from the dissipation terms lambda |w| of the face flux."""
    n = degree + 1
    x, w = O.gauss(n)
    lam = max(sum(abs(w[a] * O.lagrange_deriv(x, i, x[a]) / w[i]) for a in range(n))
              + abs(O.lagrange(x, i, 1.0) / w[i]) + abs(O.lagrange(x, i, -1.0) / w[i])
              for i in range(n))
    amp = sum(abs(O.lagrange(x, a, 1.0)) for a in range(n))  # trace amplification
    vel = u[1:1 + dim] / u[0]
    kin = (u[1:1 + dim] * vel).sum(0)
    p = 0.4 * (np.abs(u[dim + 1]) + 0.5 * kin)
    speed = np.sqrt((vel ** 2).sum(0) + 1.4 * p / u[0])
    S = np.zeros(u.shape[:2])
    for d in range(dim):
        F = np.abs(u * vel[d])
        F[1 + d] += p
        F[dim + 1] += np.abs(p * vel[d])
        F = amp ** 2 * (F + speed.max() * np.abs(u)).max(axis=2)  # [var][elem]
        g = F.reshape((dim + 2,) + tuple(n_elem[::-1]))
        near = g.copy()
        for ax in range(1, dim + 1):
            near = np.maximum(near, np.maximum(np.roll(g, 1, ax), np.roll(g, -1, ax)))
        S += 2.0 / h[d] * lam * near.reshape(S.shape)
    return S


def solver(dim, n_elem, p, **kw):
    return adg.Solver(dim=dim, n_elem=n_elem, degree=p, lo=(0.0,) * dim, hi=(1.0, 2.0, 3.0)[:dim],
                      dt=1e-3, **kw)


def oracle(dim, n_elem, p):
    return O.Oracle(dim=dim, n_elem=n_elem, degree=p, lo=(0.0,) * dim, hi=(1.0, 2.0, 3.0)[:dim], dt=1e-3)


SHAPES = [(2, (1, 1), 4), (2, (5, 1), 4), (2, (3, 2), 4), (2, (11, 1), 3), (2, (33, 1), 1), (2, (7, 3), 2),
          (2, (4, 1), 6), (2, (3, 1), 7), (3, (1, 1, 1), 3), (3, (3, 1, 1), 3), (3, (5, 1, 1), 2),
          (3, (17, 1, 1), 1), (3, (1, 2, 1), 4), (3, (1, 1, 2), 5)]


@pytest.mark.parametrize("exponent", [0, -8, -150])
@pytest.mark.parametrize("dim,n_elem,p", SHAPES)
def test_magnitudes(dim, n_elem, p, exponent):
    # momenta of relative size 10^exponent beside O(1) density and energy, one of them exactly
    # zero (of both signs)
    s, o = solver(dim, n_elem, p), oracle(dim, n_elem, p)
    u = random_state(s.shape, dim, seed=300 + p)
    u[1] *= 10.0 ** exponent
    u[2] = np.where(u[2] > 0, 0.0, -0.0)
    kg, ko = s.rhs(u), o.rhs(u)
    h = [(1.0, 2.0, 3.0)[d] / n_elem[d] for d in range(dim)]
    bound = 256 * EPS * sum_scale(u, dim, p, n_elem, h)[:, :, None]
    assert (np.abs(kg - ko) <= bound).all(), (np.abs(kg - ko) / bound).max()
    s.close()


@pytest.mark.parametrize("dim,n_elem,p", [(2, (5, 3), 4), (2, (9, 1), 2), (3, (3, 2, 1), 3)])
def test_beyond_the_exponent_range(dim, n_elem, p):
    # uniform energy of 1e306 with varying density: the momentum fluxes exceed the fixed-point
    # range, so the elements take the FP64 chain.  Compared: density and momentum (the energy
    # row is beyond FP64: the signal speed of 1e153 times the rounding of an energy trace)
    s, o = solver(dim, n_elem, p), oracle(dim, n_elem, p)
    u = random_state(s.shape, dim, seed=400 + p)
    u[1:1 + dim] = 0.0
    u[dim + 1] = 1e306
    kg, ko = s.rhs(u)[:1 + dim], o.rhs(u)[:1 + dim]
    assert np.isfinite(kg).all()
    h = [(1.0, 2.0, 3.0)[d] / n_elem[d] for d in range(dim)]
    n = p + 1
    x, w = O.gauss(n)
    lam = max(sum(abs(w[a] * O.lagrange_deriv(x, i, x[a]) / w[i]) for a in range(n))
              + abs(O.lagrange(x, i, 1.0) / w[i]) + abs(O.lagrange(x, i, -1.0) / w[i]) for i in range(n))
    size = np.array([1.0 * np.sqrt(1.4 * 0.4e306)] + [0.4e306] * dim)  # |F| by variable
    S = sum(2.0 / h[d] for d in range(dim)) * lam * size
    err = np.abs(kg - ko).max(axis=(1, 2))
    assert (err <= 4 * 256 * EPS * S).all(), err / (EPS * S)
    s.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("dim,n_elem,p", [(2, (5, 4), 4), (2, (7, 3), 2), (3, (3, 3, 3), 3)])
def test_nonfinite_values_spread_along_lines(dim, n_elem, p, bad):
    # a non-finite density at one node makes every variable non-finite on the lines of nodes
    # through it, in its element and (through the faces) its neighbours, and nowhere else
    s = solver(dim, n_elem, p)
    N = p + 1
    u = random_state(s.shape, dim, seed=500 + p)
    clean = s.rhs(u)
    full = (dim + 2,) + tuple(n_elem[::-1]) + (N,) * dim
    ec, nc = [n // 2 for n in n_elem], [0, 1, 1][:dim]  # element and node (x, y, z)
    v = u.copy().reshape(full)
    v[(0,) + tuple(ec[::-1]) + tuple(nc[::-1])] = bad
    k = s.rhs(v.reshape(u.shape)).reshape(full)
    hit = np.zeros(full[1:], bool)
    for d in range(dim):
        for step in (-1, 0, 1):
            e = list(ec)
            e[d] = (e[d] + step) % n_elem[d]
            idx = list(e[::-1]) + list(nc[::-1])
            idx[2 * dim - 1 - d] = slice(None)
            hit[tuple(idx)] = True
    if np.isnan(bad):
        assert not np.isfinite(k[:, hit]).any()
    assert np.isfinite(k[:, ~hit]).all()
    h = [(1.0, 2.0, 3.0)[d] / n_elem[d] for d in range(dim)]
    bound = 256 * EPS * sum_scale(u, dim, p, n_elem, h)[:, :, None]
    far = np.abs(k.reshape(u.shape) - clean) <= bound
    assert far.reshape(full)[:, ~hit].all()
    s.close()


@pytest.mark.parametrize("exponent", [-290, -200, -37, 0, 37, 200, 290])
@pytest.mark.parametrize("dim,n_elem,p", [(2, (5, 3), 3), (3, (3, 2, 2), 2)])
def test_signal_speeds_of_any_magnitude(dim, n_elem, p, exponent):
    # a gas at rest with energies of 10^exponent: the face flux's square root (an FP32 seed on
    # the scaled argument) over the exponent range, the momentum fluxes and the dissipation of
    # the density with it
    s, o = solver(dim, n_elem, p), oracle(dim, n_elem, p)
    u = random_state(s.shape, dim, seed=600 + p)
    u[1:1 + dim] = 0.0
    u[dim + 1] *= 10.0 ** exponent
    kg, ko = s.rhs(u), o.rhs(u)
    h = [(1.0, 2.0, 3.0)[d] / n_elem[d] for d in range(dim)]
    with np.errstate(over="ignore"):
        bound = 256 * EPS * sum_scale(u, dim, p, n_elem, h)[:, :, None]
    rows = slice(0, 1 + dim if exponent >= 200 else dim + 2)  # (energy row: 1e290 * 1e145)
    assert (np.abs(kg - ko) <= bound)[rows].all(), (np.abs(kg - ko) / bound)[rows].max()
    s.close()
