"""Edges of the fixed-point operator and recurrence: zero links, values outside the exponent
windows, sources beside one another, components far below their site's largest.

Operator: per site against the numpy oracle in extended precision, in units of 2^-53 m(x),
m(x) = |psi(x)| + |kappa| sum over the eight hops of |U|_max |psi(neighbour)| (largest components).
A component of out(x) is psi's own and six products per hop, so it is at most 6 m; rounding the
sum and the result to FP64 each cost half a unit of 2^-53 of that, and the fixed-point sum and the
links' factor e^(+-mu) less than two units together: 8 units bound the difference.
"""
import numpy as np
import pytest
import torch

from oracle import dirac
from paper_1604_08057_gb300 import binding, inputs

pytestmark = pytest.mark.gpu
MU, M_W = 0.4, -1.3


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def T(a):
    return torch.tensor(a, device="cuda")


def local_magnitude(u, psi):
    kappa = abs(dirac.kappa_of(M_W))
    p, a = np.abs(psi).max(axis=(-1, -2)), np.abs(u).max(axis=(-1, -2))
    m = p.copy()
    for nu in range(4):
        ax, f = 3 - nu, np.exp(MU) if nu == 3 else 1.0
        m = m + kappa * f * (a[..., nu] * np.roll(p, -1, ax) + np.roll(a[..., nu] * p, 1, ax))
    return m


def check_operator(u, psi):
    ul, pl = u.astype(np.clongdouble), psi.astype(np.clongdouble)
    m = local_magnitude(u, psi)
    for dagger in (False, True):
        got = binding.apply_H(T(u), MU, M_W, T(psi), dagger=dagger).cpu().numpy()
        want = (dirac.apply_h_dagger if dagger else dirac.apply_h)(ul, pl, MU, M_W)
        err = np.abs(got - want).max(axis=(-1, -2)).astype(np.float64)
        assert np.all(err <= 8 * 2.0 ** -53 * m), (dagger, float((err / np.where(m > 0, m, 1)).max() * 2.0 ** 53))


def ragged(rng, psi, lo, hi):
    return psi * 2.0 ** rng.integers(lo, hi, size=psi.shape[:4], endpoint=True)[..., None, None]


# magnitudes from 2^-60 to 2^60 from site to site, links far from unitary, and half of them zero
@pytest.mark.parametrize("dims", [(1, 2, 3, 2), (3, 5, 2, 4), (6, 4, 5, 7)])
@pytest.mark.parametrize("links", ["su3", "ragged", "zeros"])
def test_operator_against_extended_precision(dims, links):
    rng = np.random.default_rng(41)
    u = inputs.su3_links(dims, 0.3, rng)
    psi = inputs.gaussian_spinors(dims, 1, rng)[0]
    if links == "ragged":
        u = u * 2.0 ** rng.integers(-20, 20, size=u.shape[:5])[..., None, None]
    if links == "zeros":
        u = u * rng.integers(0, 2, size=u.shape[:5])[..., None, None]
    if links != "su3":
        psi = ragged(rng, psi, -60, 60)
    check_operator(u, psi)
