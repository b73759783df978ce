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
