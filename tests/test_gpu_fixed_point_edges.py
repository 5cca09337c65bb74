"""Edges of the fixed-point operator (zero links, values outside the exponent windows, products at
the ends of FP64's range, components far below their site's largest), and what the calls around it
have to keep: values that small in b and xbar, sources that do not depend on one another.

Operator: per site against the numpy oracle in extended precision, in units of 2^-53 m(x),
m(x) = |psi(x)| + |kappa| sum over the eight hops of |U|_max |psi(neighbour)| (largest components).
A component of out(x) is psi's own and six products per hop, so it is at most 6 m; rounding the
sum and the result to FP64 each cost half a unit of 2^-53 of that, and the fixed-point sum and the
links' factor e^(+-mu) less than two units together: 8 units bound the difference.
"""
import numpy as np
import pytest
import torch

from oracle import dirac, nested, overlap, tsl, vjp
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


def check_operator(u, psi, units=8):
    ul, pl = u.astype(np.clongdouble), psi.astype(np.clongdouble)
    m = local_magnitude(u, psi)
    for dagger in (False, True):
        got = binding.apply_H(T(u), MU, M_W, T(psi), dagger=dagger).cpu().numpy()
        want = (dirac.apply_h_dagger if dagger else dirac.apply_h)(ul, pl, MU, M_W)
        err = np.abs(got - want).max(axis=(-1, -2)).astype(np.float64)
        assert np.all(err <= units * 2.0 ** -53 * m), (dagger, float((err / np.where(m > 0, m, 1)).max() * 2.0 ** 53))


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


def tails(rng, dims):
    """A Gaussian field whose last planes fall to 1e-260 and to the smallest subnormal."""
    f = inputs.gaussian_spinors(dims, 1, rng)[0]
    f[-1] *= 1e-260
    f[0, -1] = 5e-324
    return f


# b (and the cotangent) down to subnormals on some sites, a link of 1e-290.  x and the gradients are
# the oracle's to the bars of the parity tests at m_w = -1
@pytest.mark.parametrize("rebiorth,passes", [(1, 2), (10, 1)])
def test_sites_and_links_below_the_window(rebiorth, passes):
    dims, k = (3, 4, 3, 5), 30
    rng = np.random.default_rng(43)
    u = inputs.su3_links(dims, 0.3, rng)
    u[2, 1, 0, 1, 2] *= 1e-290
    b, xbar = tails(rng, dims), tails(rng, dims)
    opts = dict(rebiorth=rebiorth, passes=passes)
    du_o, dmu_o, f = vjp.tsl_vjp(u, b, 0.2, -1.0, k, xbar, **opts)
    assert rel(binding.tsl_sign(T(u), 0.2, -1.0, T(b), k, **opts).cpu().numpy(), f.x) <= 1e-11
    du, dmu, x = binding.tsl_sign_vjp(T(u), 0.2, -1.0, T(b), k, T(xbar), **opts)
    assert rel(x.cpu().numpy(), f.x) <= 1e-11
    assert rel(du.cpu().numpy(), du_o) <= 1e-9 and abs(dmu - dmu_o) <= 1e-9 * abs(dmu_o)
    dx_o, x_o, _ = tsl.block_tsl(u, b, 0.2, -1.0, k, None, 0.7, **opts)
    dx, xj = binding.tsl_sign_jvp(T(u), 0.2, -1.0, T(b), k, None, 0.7, **opts)
    assert rel(dx.cpu().numpy(), dx_o) <= 1e-10 and rel(xj.cpu().numpy(), x_o) <= 1e-10
    want, _, _ = nested.nested_tsl(u, b, 0.2, -1.0, k, 15, **opts)
    binding.nested_sign(15, **opts)
    try:
        xn = binding.tsl_sign(T(u), 0.2, -1.0, T(b), k, **opts)
    finally:
        binding.nested_sign(0, **opts)
    assert rel(xn.cpu().numpy(), want) <= 1e-10
    eps = binding.tsl_eps(T(u), 0.2, -1.0, T(b), k, **opts)
    assert abs(eps - tsl.eps_a(u, b, 0.2, -1.0, k, **opts)) <= 1e-6 * eps
    do = binding.overlap_apply(T(u), 0.2, -1.0, T(b), k, **opts)
    assert rel(do.cpu().numpy(), overlap.apply_dov(u, b, 0.2, -1.0, k, **opts)) <= 1e-10


def test_operator_below_the_window():
    """The same values through the operator: at the sites that meet them FP64 sums of up to 6 m with
    some ten roundings each, 64 units of m."""
    rng = np.random.default_rng(44)
    dims = (3, 4, 3, 5)
    u = inputs.su3_links(dims, 0.3, rng)
    u[2, 1, 0, 1, 2] *= 1e-290
    psi = tails(rng, dims)
    psi[0, -1] = 1e-280     # (a subnormal site's sums round to the subnormals' own unit)
    check_operator(u, psi, 64)


# V times the sources on either side of the number of warps that fill the GPU
@pytest.mark.parametrize("dims,nsrc", [((8, 8, 8, 8), 4), ((6, 6, 6, 6), 8), ((6, 8, 4, 6), 9)])
def test_a_source_does_not_depend_on_those_beside_it(dims, nsrc):
    rng = np.random.default_rng(45)
    k, opts = 40, dict(rebiorth=20, passes=1)
    u, b = T(inputs.su3_links(dims, 0.25, rng)), T(inputs.gaussian_spinors(dims, nsrc, rng))
    binding.nested_sign(20, **opts)
    try:
        x = binding.tsl_sign(u, 0.2, -1.0, b, k, **opts)
        co = [binding.tsl_coefficients(k, s, **opts) for s in range(nsrc)]
        for s in (0, 1, nsrc - 1):
            assert torch.equal(binding.tsl_sign(u, 0.2, -1.0, b[s], k, **opts), x[s]), s
            for one, all_ in zip(binding.tsl_coefficients(k, 0, **opts), co[s]):
                assert np.array_equal(one, all_), s
    finally:
        binding.nested_sign(0, **opts)


@pytest.mark.parametrize("dims,nsrc", [((1, 2, 3, 2), 1), ((3, 5, 2, 4), 3), ((5, 3, 3, 3), 5)])
def test_operator_returns_its_own_term_as_it_is(dims, nsrc):
    """Without links H is gamma5: bit for bit, components of 2^-100 of their site's largest among them."""
    rng = np.random.default_rng(46)
    psi = inputs.gaussian_spinors(dims, nsrc, rng)
    psi *= 2.0 ** rng.integers(-100, 0, size=psi.shape, endpoint=True)
    u = np.zeros(inputs.lattice_shape(dims) + (4, 3, 3), dtype=np.complex128)
    for dagger in (False, True):
        got = binding.apply_H(T(u), MU, M_W, T(psi), dagger=dagger).cpu().numpy()
        for s in range(nsrc):
            assert np.array_equal(got[s], dirac.apply_gamma5(psi[s]))


@pytest.mark.parametrize("field,link", [(2.0 ** -700, 2.0 ** -300), (2.0 ** -800, 2.0 ** -200), (2.0 ** 700, 2.0 ** 400)])
def test_operator_products_at_the_ends_of_the_range(field, link):
    """One colour of one site, diagonal links: products below 2^-1000 are still normal numbers, and
    where they overflow the other colours stay zero."""
    rng = np.random.default_rng(48)
    dims = (3, 4, 3, 5)
    u = np.zeros(inputs.lattice_shape(dims) + (4, 3, 3), dtype=np.complex128)
    i = np.arange(3)
    u[..., i, i] = link * np.exp(0.3j * rng.standard_normal(u.shape[:5] + (3,)))
    psi = np.zeros(inputs.lattice_shape(dims) + (4, 3), dtype=np.complex128)
    psi[2, 1, 2, 1, :, 1] = field * (1.0 + 0.5j)
    if field < 1.0:
        return check_operator(u, psi, 64)   # FP64 sums
    got = binding.apply_H(T(u), MU, M_W, T(psi)).cpu().numpy()
    assert np.array_equal(got[..., ::2], np.zeros_like(got[..., ::2]))
    assert not np.isfinite(got[..., 1]).all()


@pytest.mark.parametrize("nsrc", [1, 3, 16])
def test_operator_shapes(nsrc):
    """The FP64 operator has six launch shapes beside its rule; the variant numbers above them start
    again (and are not timed again), and every shape gives the same bits."""
    rng = np.random.default_rng(49)
    dims = (6, 4, 5, 7)
    u, psi = T(inputs.su3_links(dims, 0.3, rng)), T(inputs.gaussian_spinors(dims, nsrc, rng))
    want = binding.apply_H(u, MU, M_W, psi)
    rep = binding.autotune(u, MU, M_W, nsrc=nsrc)
    us = rep["apply_us"]
    assert min(us) > 0.0 and all(us[v] == us[(v - 1) % 6 + 1] for v in range(7, len(us)))
    try:
        for v in range(len(us)):
            binding.set_stencil_variants(v, 0)
            assert torch.equal(binding.apply_H(u, MU, M_W, psi), want), v
    finally:
        binding.set_stencil_variants(0, 0)
