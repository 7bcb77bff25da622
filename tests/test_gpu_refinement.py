"""The mixed form's refinement of X q in slices of up to 64 sites."""
import numpy as np
import pytest

from oracle import dyson_oracle as O
from paper_1102_3137_gb300 import dyson as D
from paper_1102_3137_gb300 import inputs as I
from parity_util import OPEN, plan_for, wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1102_3137_gb300 import build
    build.build()
    D.load()


def interface_mask(L, p):
    """True on the interface layers, natural order."""
    mask = np.zeros(L[::-1], bool)
    mask[O.dd_partition(L, p)[2]] = True
    return mask.ravel()


def stencil(L, t, z, x):
    """H x and sum |H||x| per site in extended precision."""
    x = x.astype(np.clongdouble).reshape(L[::-1])
    y = z.astype(np.clongdouble).reshape(x.shape) * x
    s = np.abs(y)
    for d in range(x.ndim):
        lo = tuple(slice(None, -1) if a == d else slice(None) for a in range(x.ndim))
        hi = tuple(slice(1, None) if a == d else slice(None) for a in range(x.ndim))
        y[lo] += t * x[hi]
        y[hi] += t * x[lo]
        s[lo] += abs(t) * np.abs(x[hi])
        s[hi] += abs(t) * np.abs(x[lo])
    return y.ravel(), s.ravel()


# widths 16, 32 (rows on and off chip), 48, 64; 4 x 4 slices of a thin 3D slab
@pytest.mark.parametrize("L,p", [((40, 33), 2), ((96, 65), 2), ((600, 65), 2), ((30, 97), 2), ((33, 129), 2),
                                 ((9, 4, 9), 2)])
@pytest.mark.parametrize("eta", [0.0, 0.2])
def test_refinement_reaches_binary64_rounding(L, p, eta):
    """u = X q solves (H u)_B = 0 on the subdomains.  With no tolerance to stop at, the
    refinement ends at the rounding of its residual: per real part six fused
    multiply-adds, each off by 2^-53 of sum |H||u| at most, and u's own rounding, once
    more, so 7 sqrt(2) 2^-53 of it."""
    w = wl(L, p, 4, K=2)
    omega, V, sigma, _ = I.make_inputs(w, axis="real" if eta else "matsubara")
    pl = plan_for(w, D.DYSON_MIXED, eta=eta, refine_tol=1e-30, refine_max=8)
    rng = np.random.default_rng(3)
    q = rng.normal(size=(2, w.N)) + 1j * rng.normal(size=(2, w.N))
    u = np.zeros_like(q)
    D.dyson_xmatvec(pl.handle, 2, omega, V, sigma, q, u)
    sub = ~interface_mask(w.L, p)
    for k in range(2):
        y, s = stencil(w.L, w.t, O.axis_diagonal(omega[k], w.mu, V, sigma[k], eta), u[k])
        assert np.max(np.abs(y[sub])) <= 10 * 2.0 ** -53 * np.max(s[sub])
    pl.close()
