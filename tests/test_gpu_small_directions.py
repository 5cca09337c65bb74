"""Theorem-1 calls along directions far smaller than the links, zero on most of them.

dx is of the direction's size, and the k-step map's own rounding floor at these points (the oracle
with b perturbed by 2^-53, relative 2-norm) is at most 5e-12: the bar is 1e-10, that of the other
Theorem-1 tests, at every size of the direction.  The oracle forms dH psi along links as
(psi - kappa hops) - psi, so it is given the direction at order one and its dH is scaled by the
power of two.
"""
import numpy as np
import pytest
import torch

from oracle import dirac, tsl
from paper_1604_08057_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("dims,k,rebiorth", [((3, 5, 2, 4), 40, 10), ((4, 3, 3, 3), 40, 1)])
@pytest.mark.parametrize("scale", [2.0 ** -33, 2.0 ** -60])
@pytest.mark.parametrize("links,mu_dir", [(True, 0.0), (True, 0.7), (False, 0.7)])
def test_small_direction_matches_the_oracle(monkeypatch, dims, k, rebiorth, scale, links, mu_dir):
    rng = np.random.default_rng(75)
    u = inputs.su3_links(dims, 0.3, rng)
    b = inputs.gaussian_spinors(dims, 1, rng)[0]
    e = None
    if links:
        e = np.zeros_like(u)
        for nu, at in ((1, (0, 1, 0, 1)), (3, (2, 0, 1, 0))):
            e[at + (nu,)] = scale * (rng.standard_normal((3, 3)) + 1j * rng.standard_normal((3, 3)))
    t = lambda a: None if a is None else torch.tensor(a, device="cuda")   # noqa: E731
    dx, x = binding.tsl_sign_jvp(t(u), 0.3, -1.0, t(b), k, t(e), scale * mu_dir, rebiorth=rebiorth)
    for name in ("apply_dh", "apply_dh_dagger"):
        full = getattr(dirac, name)
        monkeypatch.setattr(dirac, name, lambda u_, e_, psi, mu, m_w, m, full=full: scale * full(
            u_, None if e_ is None else e_ / scale, psi, mu, m_w, m / scale))
    want, xo, _ = tsl.block_tsl(u, b, 0.3, -1.0, k, e, scale * mu_dir, rebiorth=rebiorth)
    assert rel(x.cpu().numpy(), xo) <= 1e-10
    assert rel(dx.cpu().numpy(), want) <= 1e-10
