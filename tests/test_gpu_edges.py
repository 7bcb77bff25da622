"""The strip, slab and Lanczos kernels at the edges of their tiles, rules and splits,
against the oracle through the C ABI.  Tolerances are those of the same quantities in the
other parity tests (FP64 / mixed): diag(B^-1) 1e-12 / 1e-10, B^-1 q 1e-12 / 1e-5, X q
1e-11 / 1e-9, a truncated run step by step 1e-10 / 1e-6."""
import numpy as np
import pytest

from oracle import dyson_oracle as O
from paper_1102_3137_gb300 import dyson as D
from paper_1102_3137_gb300 import inputs as I
from parity_util import OPEN, TOL_FP64, TOL_MIXED, oracle_parts, plan_for, relerr, stepwise_check, wl

pytestmark = pytest.mark.gpu

# Lines of one, two and three slices (no chain, one chain, one step each); the width
# classes 4, 16, 17 (20 padded), 32, 33 (36 padded), 64 at small and odd numbers of
# slices; the layer inverse on chip (160) and by 64 x 64 tiles (161); rows in the scratch
# at W = 64; narrow strips with lines past the preconditioner's limit.
STRIPS = [((1, 9), 2), ((2, 14), 3), ((3, 33), 2), ((5, 35), 2), ((6, 65), 2), ((7, 67), 2), ((4, 129), 2),
          ((160, 17), 2), ((161, 33), 2), ((260, 129), 2), ((1030, 9), 2)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1102_3137_gb300 import build
    build.build()
    D.load()


@pytest.mark.parametrize("L,p", STRIPS)
@pytest.mark.parametrize("precision,tol", [(D.DYSON_FP64, (1e-12, 1e-12, 1e-11)), (D.DYSON_MIXED, (1e-10, 1e-5, 1e-9))])
def test_strips(L, p, precision, tol):
    w = wl(L, p, 4, K=2)
    omega, V, sigma, _ = I.make_inputs(w)
    pl = plan_for(w, precision)
    dB = np.zeros((2, w.N), complex)
    D.dyson_subdomain_diag(pl.handle, 2, omega, V, sigma, dB)
    rng = np.random.default_rng(5)
    q = rng.normal(size=(2, w.N)) + 1j * rng.normal(size=(2, w.N))
    wv, u = np.zeros_like(q), np.zeros_like(q)
    D.dyson_subdomain_solve(pl.handle, 2, omega, V, sigma, q, wv)
    D.dyson_xmatvec(pl.handle, 2, omega, V, sigma, q, u)
    for k in range(2):
        subs, X = oracle_parts(w, omega[k], V, sigma[k])
        mask = subs.diagB != 0
        assert relerr(dB[k][mask], subs.diagB[mask]) < tol[0]
        for got, ref, bound in ((wv[k], subs.solve(q[k]), tol[1]), (u[k], X(q[k]), tol[2])):
            assert np.max(np.abs(got - ref)) <= bound * np.max(np.abs(ref))


@pytest.mark.parametrize("L,p", [((4, 16, 17), 2), ((3, 17, 9), 2)])     # W = 128; 68, no whole tiles
@pytest.mark.parametrize("precision,tol", [(D.DYSON_FP64, 1e-12), (D.DYSON_MIXED, 1e-10)])
def test_wide_factor_cluster_sizes(L, p, precision, tol):
    """1, 40 and 100 frequencies of two slabs take clusters of 8 to 1 CTAs a unit; the split
    of the tiles does not change the arithmetic, so a frequency's bits are the same."""
    w = wl(L, p, 4, K=100)
    omega, V, sigma, _ = I.make_inputs(w)
    pl = plan_for(w, precision)
    out = {}
    for K in (1, 40, 100):
        out[K] = np.zeros((K, w.N), complex)
        D.dyson_subdomain_diag(pl.handle, K, omega[:K], V, sigma[:K], out[K])
    assert np.array_equal(out[1], out[100][:1]) and np.array_equal(out[40], out[100][:40])
    for k in (0, 99):
        subs = O.Subdomains(w.L, OPEN, w.t, O.dyson_diagonal(omega[k], w.mu, V, sigma[k]), p)
        mask = subs.diagB != 0
        assert relerr(out[100][k][mask], subs.diagB[mask]) < tol


# mixed: strips of one (20 sites: fewer than a warp each), two and four CTAs; FP64: two; k = 9
# and 4 end inside and at the end of a group of basis vectors
@pytest.mark.parametrize("L,p,k", [((5, 9), 2, 4), ((256, 33), 2, 9), ((300, 65), 2, 4)])
@pytest.mark.parametrize("precision,tol", [(D.DYSON_FP64, TOL_FP64), (D.DYSON_MIXED, TOL_MIXED)])
def test_lanczos_step_splits(L, p, k, precision, tol):
    w = wl(L, p, k, K=2, seed=7)
    omega, V, sigma, q1 = I.make_inputs(w)
    pl = plan_for(w, precision)
    out = pl.solve(omega, V, sigma, q1)
    info = pl.info(w.K)
    for f in range(w.K):
        subs, X = oracle_parts(w, omega[f], V, sigma[f])
        assert stepwise_check(w, pl, f, subs, X, q1, out[f], info, tol) == k
