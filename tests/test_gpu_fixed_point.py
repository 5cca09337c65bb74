"""The FP64 operator's fixed-point arithmetic at the edges of its exponent windows and tiles.

Per site, out(x) is compared with the numpy oracle in units of the local magnitude
m(x) = |psi(x)| + |kappa| sum over the eight hops of |U|_max |psi(neighbour)|: the oracle rounds
some 30 times per component and the fixed-point sum once per hop below 2^-53 of m, so 64 rounding
units of m (7.1e-15) bound their difference, for every dynamic range from site to site.
"""
import numpy as np
import pytest
import torch

from oracle import dirac, vjp
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


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("dims,k,rebiorth,passes", [((1, 3, 2, 5), 20, 1, 2), ((5, 3, 4, 7), 45, 10, 1),
                                                    ((4, 6, 3, 3), 70, 1, 2)])
def test_recurrence_and_force_from_a_point_source(dims, k, rebiorth, passes):
    """b and xbar on one site each: the Krylov vectors start with most sites zero and decay over many
    binary orders.  m_w = -1, rounding floors of the map ~1e-14: the bars of the parity tests."""
    rng = np.random.default_rng(21)
    u = inputs.su3_links(dims, 0.3, rng)
    b = inputs.gaussian_spinors(dims, 1, rng)[0]
    xbar = inputs.gaussian_spinors(dims, 1, rng)[0]
    for f, at in ((b, (0, 0, 0, 0)), (xbar, tuple(n - 1 for n in b.shape[:4]))):
        keep = f[at].copy()
        f[...] = 0.0
        f[at] = keep
    du_o, dmu_o, fwd = vjp.tsl_vjp(u, b, 0.2, -1.0, k, xbar, rebiorth=rebiorth, passes=passes)
    t = lambda a: torch.tensor(a, device="cuda")   # noqa: E731
    du, dmu, x = binding.tsl_sign_vjp(t(u), 0.2, -1.0, t(b), k, t(xbar), rebiorth=rebiorth, passes=passes)
    assert rel(x.cpu().numpy(), fwd.x) <= 1e-11
    assert rel(du.cpu().numpy(), du_o) <= 1e-9 and abs(dmu - dmu_o) <= 1e-9 * abs(dmu_o)


@pytest.mark.parametrize("dims,nsrc", [((3, 5, 2, 4), 1), ((6, 4, 5, 4), 3)])
def test_powers_of_two_pass_through_exactly(dims, nsrc):
    """Scaling the source or the cotangent by a power of two shifts exponents and nothing else."""
    rng = np.random.default_rng(3)
    t = lambda a: torch.tensor(a, device="cuda")   # noqa: E731
    u, b = t(inputs.su3_links(dims, 0.3, rng)), t(inputs.gaussian_spinors(dims, nsrc, rng))
    xbar = t(inputs.gaussian_spinors(dims, nsrc, rng))
    du, dmu, x = binding.tsl_sign_vjp(u, 0.3, -1.0, b, 25, xbar, rebiorth=10, passes=1)
    for sb, sx in ((2.0 ** 90, 1.0), (2.0 ** -130, 1.0), (1.0, 2.0 ** -80), (1.0, 2.0 ** 150)):
        du2, dmu2, x2 = binding.tsl_sign_vjp(u, 0.3, -1.0, sb * b, 25, sx * xbar, rebiorth=10, passes=1)
        assert torch.equal(x2, sb * x)
        assert torch.equal(du2, (sb * sx) * du) and dmu2 == sb * sx * dmu
