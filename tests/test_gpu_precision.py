"""Figures that hold over the whole range of the number format, through the public calls."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def msh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1210_5246_gb300 import msh as m
    m.load()
    return m


@pytest.mark.parametrize("rho,P", [(1e-250, 1e-100), (1e300, 1e50), (3e-160, 7e-100), (1.7, 0.3), (1e-5, 1e5),
                                   (1e120, 1e-90), (2e-308, 3e99)])
def test_fp64_cfl_step_over_the_range(msh, rho, P):
    """CFL step of a uniform gas at rest, cfl dx / sqrt(3 P / rho), also where P rho under- or
    overflows.  Bound: the root of the quotient within 1 ulp, sqrt(3) and the product with it
    and the last quotient half an ulp each (the cell width is a power of two)."""
    n, cfl = 32, 0.5
    W = np.zeros((10, 1, 1, n))
    W[0] = rho
    W[4] = W[7] = W[9] = P
    g = msh.Grid((n,), (0.0,), (1.0,), ((1, 1),), cfl, msh.FP64)
    g.set_state(W, msh.PRIMITIVE)
    _, dt, ok = g.reduce_layers(0, n)
    g.close()
    want = np.longdouble(cfl) / n / np.sqrt(np.longdouble(3) * np.longdouble(P) / np.longdouble(rho))
    assert ok and abs(np.longdouble(dt) - want) <= 3 * 2.0 ** -52 * want


@pytest.mark.parametrize("n,tiling", [((96, 70), (4, 8)), ((96, 70), (16, 16)), ((40, 30, 20), (8, 0)), ((40, 30, 20), (16, 5)),
                                      ((500,), (8, 1))])
def test_fp32_totals_beyond_the_fp32_range(msh, n, tiling):
    """Totals of a uniform FP32 state with a field (zz stress, in 3D the density) that is
    representable in every cell and summed over a thread's, but not over a warp's: the totals are
    FP64 sums (a thread's FP32 sum of at most 20 equal cells rounds by 20 2^-24 at most)."""
    nd = len(n)
    big = 1e38 if nd == 1 else 1e37
    W = np.zeros((10,) + (1,) * (3 - nd) + n[::-1])
    W[0] = W[4] = W[7] = 1.0
    W[9] = 1.0
    W[9 if nd < 3 else 0] = big
    g = msh.Grid(n, (0.0,) * nd, (1.0,) * nd, ((0, 0),) * nd, 0.3, msh.FP32)
    g.set_tiling(*tiling)
    g.set_state(W.astype(np.float32), msh.PRIMITIVE)
    g.run(max_steps=2)
    tot, ok, _ = g.diagnostics()
    U = g.get_state().astype(np.float64)
    g.close()
    want = U.reshape(10, -1).sum(axis=1)
    assert ok and np.isfinite(tot).all()
    assert (np.abs(tot - want) <= 20 * 2.0 ** -24 * np.abs(U).reshape(10, -1).sum(axis=1)).all()
