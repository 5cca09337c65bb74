"""The FP64 operator's fixed-point arithmetic at the edges of its exponent windows and tiles.

Per site, out(x) is compared with the numpy oracle in units of the local magnitude
m(x) = |psi(x)| + |kappa| sum over the eight hops of |U|_max |psi(neighbour)|: the oracle rounds
some 30 times per component and the fixed-point sum once per hop below 2^-53 of m, so 64 rounding
units of m (7.1e-15) bound their difference, for every dynamic range from site to site.
"""
import numpy as np
import pytest
import torch

from oracle import dirac
from paper_1604_08057_gb300 import binding, inputs

pytestmark = pytest.mark.gpu
UNIT = 64 * 2.0 ** -53


def local_magnitude(u, psi, mu, m_w):
    kappa = abs(1.0 / (2.0 * m_w + 8.0))
    p = np.abs(psi).max(axis=(-1, -2))
    a = np.abs(u).max(axis=(-1, -2))
    m = p.copy()
    for nu in range(4):
        ax = 3 - nu
        f = np.exp(abs(mu)) if nu == 3 else 1.0
        m = m + 12 * kappa * f * a[..., nu] * np.roll(p, -1, ax)
        m = m + 12 * kappa * f * np.roll(a[..., nu] * p, 1, ax)
    return m


def fields(kind, dims, n, rng):
    psi = inputs.gaussian_spinors(dims, n, rng)
    if kind == "point":
        keep = psi[:, 0, 0, 0, 0].copy()
        psi[:] = 0.0
        psi[:, 0, 0, 0, 0] = keep
    elif kind == "ragged":       # magnitudes spread over 2^-60 .. 2^60 from site to site, in the window
        psi *= 2.0 ** rng.integers(-60, 30, size=psi.shape[:5])[..., None, None]
    elif kind == "huge":         # above the window: FP64
        psi *= 1e200
    elif kind == "tiny":         # below the window: FP64
        psi *= 1e-280
    elif kind == "mixed":        # both forms meet on neighbouring sites
        psi[:, ::2] *= 1e30
    return psi


@pytest.mark.parametrize("dims,nsrc", [((1, 2, 3, 2), 1), ((3, 5, 2, 4), 3), ((5, 3, 3, 3), 2), ((4, 4, 4, 4), 5),
                                       ((6, 8, 10, 12), 4)])
@pytest.mark.parametrize("kind", ["gauss", "point", "ragged", "huge", "tiny", "mixed"])
def test_operator_per_site(dims, nsrc, kind):
    rng = np.random.default_rng(11)
    u = inputs.su3_links(dims, 0.3, rng)
    if kind == "ragged":         # links far from unitary
        u = u * 2.0 ** rng.integers(-20, 20, size=u.shape[:5])[..., None, None]
    psi = fields(kind, dims, nsrc, rng)
    ut, pt = torch.tensor(u, device="cuda"), torch.tensor(psi, device="cuda")
    for dagger in (False, True):
        got = binding.apply_H(ut, 0.4, -1.3, pt, dagger=dagger).cpu().numpy()
        for s in range(nsrc):
            want = (dirac.apply_h_dagger if dagger else dirac.apply_h)(u, psi[s], 0.4, -1.3)
            m = local_magnitude(u, psi[s], 0.4, -1.3)
            err = np.abs(got[s] - want).max(axis=(-1, -2))
            assert np.all(err <= UNIT * m), (kind, dagger, float((err / np.where(m > 0, m, 1)).max()))


def test_non_finite_values_reach_the_same_sites():
    rng = np.random.default_rng(5)
    dims = (3, 4, 3, 5)
    u = inputs.su3_links(dims, 0.3, rng)
    psi = inputs.gaussian_spinors(dims, 1, rng)[0]
    psi[1, 2, 3, 0, 1, 2] = np.nan
    psi[4, 0, 0, 2, 0, 0] = np.inf
    want = dirac.apply_h(u, psi, 0.2, -1.0)
    got = binding.apply_H(torch.tensor(u, device="cuda"), 0.2, -1.0, torch.tensor(psi, device="cuda")).cpu().numpy()
    bad = ~np.isfinite(want).all(axis=(-1, -2))
    assert np.array_equal(bad, ~np.isfinite(got).all(axis=(-1, -2))) and bad.any()
    assert np.abs(got[~bad] - want[~bad]).max() <= 1e-13
