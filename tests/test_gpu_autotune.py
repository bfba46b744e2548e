"""The autotuner (hemi-Dslash variant -2): it times variants where there is a
choice, on lattices above those of the one-thread-per-direction kernel, and
launches nothing besides where there is none."""
import numpy as np
import pytest

from paper_1805_03560_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SMALL, LARGE = (4, 4, 8, 16), (32, 16, 16, 16)


@pytest.fixture(scope="module")
def H():
    from paper_1805_03560_gb300 import hmc
    return hmc


def _np(t):
    return t.cpu().numpy()


def _launches(ctx, f):
    n = ctx.launches()
    f()
    return ctx.launches() - n


@pytest.mark.parametrize("prec,fmt", [(0, 18), (1, 12), (1, 18), (3, 18), (3, 12)])
def test_nothing_is_timed_on_small_lattices(H, prec, fmt):
    """One launch per hemi-Dslash, and a solve launches what it launches with
    the default."""
    L = SMALL
    links = I.gauge_links(L, 0.3, 1)
    psi = I.gaussian_half(L, 3)
    n, xs = [], []
    for v in (-1, -2):
        ctx = H.Context(0)
        ctx.set_dslash_variant(v)
        U = ctx.pack_gauge(L, links, prec, fmt)
        src, out = ctx.pack_spinor(L, psi, prec), ctx.new_spinor(L, prec)
        assert _launches(ctx, lambda: ctx.dslash(L, U, out, src, 0)) == 1
        if prec != 3:
            Uh = ctx.pack_gauge(L, links, 0, 18)
            x, b = ctx.new_spinor(L, 0), ctx.pack_spinor(L, psi, 0)
            n.append(_launches(ctx, lambda: ctx.cg_solve(
                L, Uh, x, b, 0.12, 1e-8, U_lo=U if prec else None, inner_prec=prec)))
            xs.append(_np(ctx.unpack_spinor(L, x)))
    if prec != 3:
        assert n[0] == n[1] and np.array_equal(xs[0], xs[1])


@pytest.mark.parametrize("prec,fmt", [(0, 18), (1, 12), (1, 18), (3, 12)])
def test_large_lattices_are_tuned_to_the_same_bits(H, prec, fmt):
    """The first launch of a class times the variants (four launches each), the
    next ones do not; the outputs are those of the default variant."""
    L = LARGE
    links = I.gauge_links(L, 0.3, 1)
    psi = I.gaussian_half(L, 3)
    ctx = H.Context(0)
    U = ctx.pack_gauge(L, links, prec, fmt)
    src, want, got = ctx.pack_spinor(L, psi, prec), ctx.new_spinor(L, prec), ctx.new_spinor(L, prec)
    for dagger in (False, True):
        ctx.set_dslash_variant(-1)
        ctx.dslash(L, U, want, src, 0, dagger)
        ctx.set_dslash_variant(-2)
        # at least plain and paired loads, each with and without tiles
        assert _launches(ctx, lambda: ctx.dslash(L, U, got, src, 0, dagger)) >= 4 * 4 + 1
        assert np.array_equal(_np(ctx.unpack_spinor(L, got)), _np(ctx.unpack_spinor(L, want)))
        got.data.fill_(0xFF)
        assert _launches(ctx, lambda: ctx.dslash(L, U, got, src, 0, dagger)) == 1
        assert np.array_equal(_np(ctx.unpack_spinor(L, got)), _np(ctx.unpack_spinor(L, want)))


def test_one_kernel_is_not_timed(H):
    """Emulated FP64 with 18-real links: one kernel for every variant."""
    L = LARGE
    ctx = H.Context(0)
    ctx.set_dslash_variant(-2)
    U = ctx.pack_gauge(L, I.gauge_links(L, 0.3, 1), 3, 18)
    src, out = ctx.pack_spinor(L, I.gaussian_half(L, 3), 3), ctx.new_spinor(L, 3)
    assert _launches(ctx, lambda: ctx.dslash(L, U, out, src, 0)) == 1


def test_solve_on_a_large_lattice_is_tuned_to_the_same_bits(H):
    L = LARGE
    links = I.gauge_links(L, 0.3, 1)
    psi = I.gaussian_half(L, 3)
    xs, n = [], []
    for v in (-1, -2):
        ctx = H.Context(0)
        ctx.set_dslash_variant(v)
        Uh, Ul = ctx.pack_gauge(L, links, 0, 18), ctx.pack_gauge(L, links, 1, 12)
        x, b = ctx.new_spinor(L, 0), ctx.pack_spinor(L, psi, 0)
        n.append(_launches(ctx, lambda: ctx.cg_solve(L, Uh, x, b, 0.12, 1e-10, U_lo=Ul,
                                                     inner_prec=1)))
        xs.append(_np(ctx.unpack_spinor(L, x)))
    assert n[1] > n[0] and np.array_equal(xs[0], xs[1])
