"""Outer-product and gauge force kernels in emulated FP64 (paired arithmetic)
and FP32 against the native FP64 kernels, on lattices with partial blocks of 32
links, extents of 2 (both neighbours the same site) and of 4 (straight lines).

Tolerances relative to the largest component: 2e-13 in emulated FP64 (unit
roundoff 2^-47 over some hundred chained operations), 2e-5 in FP32, those of
the force parity tests.
"""
import numpy as np
import pytest

from paper_1805_03560_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LATTICES = [(2, 2, 2, 2), (4, 2, 2, 6), (2, 6, 4, 8), (4, 6, 10, 14), (20, 14, 6, 10)]


@pytest.fixture(scope="module")
def H():
    from paper_1805_03560_gb300 import hmc
    return hmc


@pytest.fixture(scope="module")
def ctx(H):
    return H.Context(0)


def _force(ctx, H, L, U, phi, fp, n):
    F = ctx.new_algebra(L)
    F.data.fill_(0.25)  # forces add to what is there
    ctx.force_pf(L, U, phi, 0.13, F, coeff=0.7, b=[1.0 / (i + 1) for i in range(n + 1)],
                 alpha=0.0, force_prec=fp)
    return ctx.unpack_algebra(L, F).cpu().numpy() - 0.25


@pytest.mark.parametrize("fmt", [18, 12])
@pytest.mark.parametrize("n", [1, 5])
@pytest.mark.parametrize("L", LATTICES)
def test_outer_product_force(ctx, H, L, n, fmt):
    U = ctx.pack_gauge(L, I.gauge_links(L, 0.3, 1), 0, fmt)
    phi = ctx.pack_spinor(L, I.gaussian_half(L, 2), 0)
    want = _force(ctx, H, L, U, phi, H.F64, n)
    for fp, tol in ((H.F64E, 2e-13), (H.F32, 2e-5)):
        if fp == H.F32 and fmt == 12:
            continue  # needs F32 links or an 18-real copy
        got = _force(ctx, H, L, U, phi, fp, n)
        assert np.abs(got - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("fmt", [18, 12])
@pytest.mark.parametrize("L", LATTICES + [(4, 4, 6, 8)])
def test_gauge_force(ctx, H, L, fmt):
    Uc = I.gauge_links(L, 0.3, 1)
    k = 2 if min(L) >= 4 else 0
    res = {}
    for prec in (H.F64, H.F64E, H.F32):
        F = ctx.new_algebra(L)
        F.data.fill_(0.25)
        ctx.force_hopexp(L, ctx.pack_gauge(L, Uc, prec, fmt), 5.6, 0.156, k, F=F, coeff=0.7,
                         want_action=False)
        res[prec] = ctx.unpack_algebra(L, F).cpu().numpy() - 0.25
    want = res[H.F64]
    assert np.abs(res[H.F64E] - want).max() <= 2e-13 * np.abs(want).max()
    assert np.abs(res[H.F32] - want).max() <= 2e-5 * np.abs(want).max()


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (4, 6, 10, 14)])
def test_force_with_exact_zeros(ctx, H, L):
    """Links with zero entries and a source with zero components (values the
    bitwise F64 -> F64E conversion leaves to the FP64 conversions)."""
    U = ctx.pack_gauge(L, I.integer_links(L), 0, 18)
    phi = I.gaussian_half(L, 2)
    phi[::2, 1] = 0.0
    phi = ctx.pack_spinor(L, phi, 0)
    want = _force(ctx, H, L, U, phi, H.F64, 3)
    got = _force(ctx, H, L, U, phi, H.F64E, 3)
    assert np.abs(got - want).max() <= 2e-13 * np.abs(want).max()
