"""One-thread-per-direction hemi-Dslash (the default on small lattices) against
the one-thread-per-site kernel (variant 0).

Both apply the same hops; the sums over the four directions associate
differently, so results agree to the rounding of eight summed hops: within the
tolerances of the parity tests of each precision, relative to the field's
largest component.
"""
import numpy as np
import pytest

from paper_1805_03560_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {0: 1e-14, 1: 1e-6, 3: 2e-13}


@pytest.fixture(scope="module")
def H():
    from paper_1805_03560_gb300 import hmc
    return hmc


@pytest.fixture(scope="module")
def ctx(H):
    return H.Context(0)


def _np(t):
    return t.cpu().numpy()


# extents of 2 (both neighbours the same site), partial blocks of 32 sites
# (Vh = 8, 24, 48, 1680, 8400), one block (32) and whole blocks (96, 4096)
LATTICES = [(2, 2, 2, 2), (2, 2, 6, 2), (4, 2, 2, 6), (4, 4, 2, 2), (4, 6, 10, 14),
            (20, 14, 6, 10), (6, 4, 4, 2), (16, 8, 8, 8)]


@pytest.mark.parametrize("prec,fmt", [(0, 18), (0, 12), (1, 18), (1, 12), (3, 18), (3, 12)])
@pytest.mark.parametrize("L", LATTICES)
def test_split_matches_site_kernel(ctx, H, L, prec, fmt):
    U = ctx.pack_gauge(L, I.gauge_links(L, 0.3, 1), prec, fmt)
    src = ctx.pack_spinor(L, I.gaussian_half(L, 3), prec)
    res = {}
    for v in (-1, 0):
        ctx.set_dslash_variant(v)
        r = []
        for dagger in (False, True):
            for p in (0, 1):
                out = ctx.new_spinor(L, prec)
                out.data.fill_(0xFF)  # NaN pattern: an unwritten site would show
                ctx.dslash(L, U, out, src, p, dagger)
                r.append(_np(ctx.unpack_spinor(L, out)))
            out = ctx.new_spinor(L, prec)
            out.data.fill_(0xFF)
            ctx.mhat(L, U, out, src, 0.156, dagger)
            r.append(_np(ctx.unpack_spinor(L, out)))
        res[v] = r
    ctx.set_dslash_variant(-1)
    for a, b in zip(res[-1], res[0]):
        assert np.abs(a - b).max() <= TOL[prec] * np.abs(b).max()


@pytest.mark.parametrize("inner", [0, 1])
@pytest.mark.parametrize("L", [(2, 2, 2, 2), (4, 2, 2, 6), (20, 14, 6, 10), (16, 8, 8, 8)])
def test_split_solves(ctx, H, L, inner):
    """A solve with the fused update on partial blocks reaches its tolerance
    (checked with the one-thread-per-site operator) with and without the graph."""
    U = I.gauge_links(L, 0.3, 1)
    Uh = ctx.pack_gauge(L, U, 0, 18)
    Ul = ctx.pack_gauge(L, U, 1, 12) if inner else None
    b = I.gaussian_half(L, 2)
    src = ctx.pack_spinor(L, b, 0)
    xs = []
    for graph in (True, False):
        ctx.set_cg_graph(graph)
        x = ctx.new_spinor(L, 0)
        r = ctx.cg_solve(L, Uh, x, src, 0.12, 1e-11, U_lo=Ul, inner_prec=inner,
                         reliable_delta=1e-5)
        assert r["status"] == 0
        xs.append(_np(ctx.unpack_spinor(L, x)))
    ctx.set_cg_graph(True)
    assert np.array_equal(xs[0], xs[1])
    ctx.set_dslash_variant(0)
    t, o = ctx.new_spinor(L, 0), ctx.new_spinor(L, 0)
    ctx.mhat(L, Uh, t, x, 0.12)
    ctx.mhat(L, Uh, o, t, 0.12, True)
    ctx.set_dslash_variant(-1)
    res = b - _np(ctx.unpack_spinor(L, o))
    assert np.linalg.norm(res) <= 1.1e-11 * np.linalg.norm(b)
