"""The one-thread-per-site hemi-Dslash kernels (variants 0 and 2), the
production kernels of large lattices, against the oracle on lattices whose last
block is partial and on degenerate ones, and inside solves there: the reduction
block, the fused update and the partial sums at the tail.

Small lattices run the one-thread-per-direction kernel by default, so these ask
for the variants.  Emulated FP64 with 18-real links shares its paired arithmetic
with that kernel; here it is compared with the oracle."""
import numpy as np
import pytest

from paper_1805_03560_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# relative to the largest component: sums of eight hops in each precision
TOL = {0: 1e-14, 1: 1e-6, 3: 2e-13}
VARIANTS = [0, 2]
CLASSES = [(0, 18), (0, 12), (1, 18), (1, 12), (3, 18), (3, 12)]


@pytest.fixture(scope="module")
def H():
    from paper_1805_03560_gb300 import hmc
    return hmc


@pytest.fixture(scope="module", params=VARIANTS)
def ctx(H, request):
    c = H.Context(0)
    c.set_dslash_variant(request.param)
    return c


def _np(t):
    return t.cpu().numpy()


def _hop(ctx, L, U, src, prec, p, dagger):
    out = ctx.new_spinor(L, prec)
    out.data.fill_(0xFF)  # NaN pattern: an unwritten site would show
    ctx.dslash(L, U, out, src, p, dagger)
    return _np(ctx.unpack_spinor(L, out))


@pytest.mark.parametrize("prec,fmt", CLASSES)
def test_integer_fields_bit_exact(orc, ctx, H, prec, fmt):
    """Signed-permutation links and small-integer spinors: every product and
    sum is exact.  Vh = 720: five blocks and a partial one."""
    L = (4, 6, 6, 10)
    U = I.integer_links(L, 5)
    Ud = ctx.pack_gauge(L, U, prec, fmt)
    for p in (0, 1):
        psi = I.integer_half(L, 6 + p)
        src = ctx.pack_spinor(L, psi, prec)
        for dagger in (False, True):
            assert np.array_equal(_hop(ctx, L, Ud, src, prec, p, dagger),
                                  orc.hop_eo(L, U, p, psi, dagger=dagger)), (p, dagger)


@pytest.mark.parametrize("prec,fmt", CLASSES)
@pytest.mark.parametrize("L", [(2, 2, 2, 2), (2, 4, 2, 2), (6, 2, 4, 8), (4, 6, 6, 10)])
def test_random_fields(orc, ctx, H, L, prec, fmt):
    """Extents of 2 (both neighbours the same site), fewer sites than a block,
    a partial last block."""
    Ud = ctx.pack_gauge(L, I.gauge_links(L, 0.3, 1), prec, fmt)
    Uq = _np(ctx.unpack_gauge(L, Ud))  # the rounded links the GPU uses
    src = ctx.pack_spinor(L, I.gaussian_half(L, 10), prec)
    psi = _np(ctx.unpack_spinor(L, src))
    for p in (0, 1):
        for dagger in (False, True):
            want = orc.hop_eo(L, Uq, p, psi, dagger=dagger)
            got = _hop(ctx, L, Ud, src, prec, p, dagger)
            assert np.abs(got - want).max() <= TOL[prec] * np.abs(want).max(), (p, dagger)


@pytest.mark.parametrize("inner,fmt", [(0, 18), (1, 12), (1, 18)])
@pytest.mark.parametrize("L", [(2, 2, 2, 2), (4, 6, 6, 10), (20, 14, 6, 10)])
def test_solves(orc, ctx, H, L, inner, fmt):
    """A solve reaches its tolerance (checked with the oracle) and gives the
    same bits as one graph and launch by launch.  Vh = 8, 720, 8400."""
    U = I.gauge_links(L, 0.3, 1)
    kappa, tol = 0.12, 1e-11
    Uh = ctx.pack_gauge(L, U, 0, 18)
    Ul = ctx.pack_gauge(L, U, 1, fmt) if inner else None
    b = I.gaussian_half(L, 2)
    src = ctx.pack_spinor(L, b, 0)
    xs = []
    for graph in (True, False):
        ctx.set_cg_graph(graph)
        x = ctx.new_spinor(L, 0)
        r = ctx.cg_solve(L, Uh, x, src, kappa, tol, U_lo=Ul, inner_prec=inner,
                         reliable_delta=1e-5)
        assert r["status"] == 0
        xs.append(_np(ctx.unpack_spinor(L, x)))
    ctx.set_cg_graph(True)
    assert np.array_equal(xs[0], xs[1])
    res = b - orc.mdagm(L, U, kappa, xs[0])
    assert np.linalg.norm(res) <= 1.1 * tol * np.linalg.norm(b)
