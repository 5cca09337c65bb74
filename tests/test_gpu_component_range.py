"""sgn(H) b, its gradient and Theorem 1 where one colour is 2^-60 of the others.

Diagonal links keep the three colours apart, so each colour's part of x, dx and dU is a sum of
products of its own components and has FP64's relative accuracy whatever the others' size.  The
rounding floors of the map here (the oracle with b perturbed by 2^-53, per colour) are 4e-15 for x,
6e-14 for dU; the bars are those of the other parity tests at m_w = -1: 1e-11, 1e-9, and 1e-10 for dx.
"""
import numpy as np
import pytest
import torch

from oracle import tsl, vjp
from paper_1604_08057_gb300 import binding, inputs

pytestmark = pytest.mark.gpu
DIMS, MU, M_W, K = (3, 4, 2, 5), 0.2, -1.0, 20


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def data():
    rng = np.random.default_rng(31)
    shape = inputs.lattice_shape(DIMS) + (4, 3)
    u = np.zeros(shape + (3,), dtype=np.complex128)
    e = np.zeros_like(u)
    i = np.arange(3)
    u[..., i, i] = np.exp(0.3j * rng.standard_normal(shape))
    b = inputs.gaussian_spinors(DIMS, 1, rng)[0]
    xbar = inputs.gaussian_spinors(DIMS, 1, rng)[0]
    e[..., i, i] = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    b[..., 1] *= 2.0 ** -60
    xbar[..., 1] *= 2.0 ** -60
    return u, b, xbar, e


@pytest.mark.parametrize("rebiorth,passes", [(1, 2), (10, 1)])
def test_each_colour_keeps_its_digits(rebiorth, passes):
    u, b, xbar, e = data()
    t = lambda a: torch.tensor(a, device="cuda")   # noqa: E731
    opts = dict(rebiorth=rebiorth, passes=passes)
    du_o, dmu_o, f = vjp.tsl_vjp(u, b, MU, M_W, K, xbar, **opts)
    dx_o, xb_o, _ = tsl.block_tsl(u, b, MU, M_W, K, e, 0.7, **opts)
    x = binding.tsl_sign(t(u), MU, M_W, t(b), K, **opts).cpu().numpy()
    du, dmu, xv = binding.tsl_sign_vjp(t(u), MU, M_W, t(b), K, t(xbar), **opts)
    dx, xj = binding.tsl_sign_jvp(t(u), MU, M_W, t(b), K, t(e), 0.7, **opts)
    du, xv, dx, xj = (a.cpu().numpy() for a in (du, xv, dx, xj))
    assert abs(dmu - dmu_o) <= 1e-9 * abs(dmu_o)
    for c in range(3):
        assert rel(x[..., c], f.x[..., c]) <= 1e-11 and rel(xv[..., c], f.x[..., c]) <= 1e-11, c
        assert rel(dx[..., c], dx_o[..., c]) <= 1e-10 and rel(xj[..., c], xb_o[..., c]) <= 1e-10, c
        for d in range(3):
            assert rel(du[..., c, d], du_o[..., c, d]) <= 1e-9, (c, d)
