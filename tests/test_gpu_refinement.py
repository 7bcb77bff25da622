"""The mixed form's refinement of X q in slices of up to 64 sites."""
import numpy as np
import pytest

from oracle import dyson_oracle as O
from paper_1102_3137_gb300 import dyson as D
from paper_1102_3137_gb300 import inputs as I
from parity_util import OPEN, TOL_FP64, TOL_MIXED, plan_for, wl

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


def local_X(w, omega_k, V, sigma_k):
    """q -> X q = H^-1 [0; q_C - E^T w_B] with w = B^-1 q, without the cancellation of
    Eq. 8: accurate relative to max |u| also where u lies 30 decades below q."""
    z = O.dyson_diagonal(omega_k, w.mu, V, sigma_k)
    subs, full = O.Subdomains(w.L, OPEN, w.t, z, w.p), O.FullLattice(w.L, OPEN, w.t, z)
    mask = interface_mask(w.L, w.p)

    def X(q):
        r = q - O.apply_H(w.L, OPEN, w.t, w.mu, V, sigma_k, omega_k, subs.solve(q))
        return full.solve(np.where(mask, r, 0))

    return subs, X


def vector(kind, w, rng):
    x, y = np.arange(w.N) % w.L[0], np.arange(w.N) // w.L[0]
    if kind[0] == "site":                      # a point source; its interface right-hand side is ~1e-29
        return ((x == kind[1]) & (y == kind[2])).astype(complex)
    if kind[0] == "gauss":                     # tails of 1e-30 and less in the far strips
        return np.exp(-((x - kind[1]) ** 2 + (y - kind[2]) ** 2) / 18.0).astype(complex)
    return kind[1] * (rng.normal(size=w.N) + 1j * rng.normal(size=w.N))


@pytest.mark.parametrize("precision,tol", [(D.DYSON_FP64, 1e-11), (D.DYSON_MIXED, 1e-9)])
@pytest.mark.parametrize("kind", [("site", 64, 8), ("site", 4, 15), ("gauss", 40, 50), ("dense", 1e-20), ("dense", 1e20)])
def test_xmatvec_of_small_and_local_vectors(kind, precision, tol):
    """The trap workload's lowest frequencies on 128^2, p = 4; the bounds are those of
    dense vectors of norm ~1 in the other parity tests."""
    w = wl((128, 128), 4, 4, K=2, beta=20.0)
    omega, V, sigma, _ = I.make_inputs(w)
    q = vector(kind, w, np.random.default_rng(5))
    pl = plan_for(w, precision)
    qs = np.stack([q, q])
    u = np.zeros_like(qs)
    D.dyson_xmatvec(pl.handle, 2, omega, V, sigma, qs, u)
    for k in range(2):
        ref = local_X(w, omega[k], V, sigma[k])[1](q)
        assert np.all(np.isfinite(u[k]))
        assert np.max(np.abs(u[k] - ref)) <= tol * np.max(np.abs(ref))
    pl.close()


@pytest.mark.parametrize("size", [1e-100, 1e100])
def test_mixed_xmatvec_of_any_size(size):
    w = wl((64, 65), 2, 4, K=1)
    omega, V, sigma, _ = I.make_inputs(w)
    q = vector(("dense", size), w, np.random.default_rng(7))[None]
    pl = plan_for(w, D.DYSON_MIXED)
    u = np.zeros_like(q)
    D.dyson_xmatvec(pl.handle, 1, omega, V, sigma, q, u)
    ref = local_X(w, omega[0], V, sigma[0])[1](q[0])
    assert np.max(np.abs(u[0] - ref)) <= 1e-9 * np.max(np.abs(ref))
    pl.close()


@pytest.mark.parametrize("L,p", [((40, 33), 2), ((64, 129), 2)])     # W = 16 and 64
def test_xmatvec_of_a_vector_on_one_strip(L, p):
    """q is zero, or 1e-25 and 1e-35 of the rest, on the second strip."""
    w = wl(L, p, 4, K=3)
    omega, V, sigma, _ = I.make_inputs(w)
    rng = np.random.default_rng(6)
    q = rng.normal(size=w.N) + 1j * rng.normal(size=w.N)
    y = np.arange(w.N) // w.L[0]
    qs = np.stack([np.where(y > w.L[1] // 2, f, 1.0) * q for f in (0.0, 1e-25, 1e-35)])
    pl = plan_for(w, D.DYSON_MIXED)
    u = np.zeros_like(qs)
    D.dyson_xmatvec(pl.handle, 3, omega, V, sigma, qs, u)
    for k in range(3):
        ref = local_X(w, omega[k], V, sigma[k])[1](qs[k])
        assert np.max(np.abs(u[k] - ref)) <= 1e-9 * np.max(np.abs(ref))
    pl.close()


@pytest.mark.parametrize("precision,tol", [(D.DYSON_FP64, TOL_FP64), (D.DYSON_MIXED, TOL_MIXED)])
@pytest.mark.parametrize("site", [(64, 8), (64, 28)])
def test_solve_from_a_unit_start_vector(site, precision, tol):
    """The rank-4 sum is nearly zero on interface sites away from the start vector, so the
    error is taken relative to the largest diagonal entry."""
    w = wl((128, 128), 4, 4, K=2, beta=20.0)
    omega, V, sigma, _ = I.make_inputs(w)
    q1 = np.zeros(w.N)
    q1[site[0] + w.L[0] * site[1]] = 1.0
    pl = plan_for(w, precision)
    out = pl.solve(omega, V, sigma, q1)
    for k in range(2):
        subs, X = local_X(w, omega[k], V, sigma[k])
        acc, al = O.cs_lanczos(X, q1, w.k)[:2]
        assert pl.info(2)["steps"][k] == len(al) == w.k
        ref = subs.diagB + acc
        assert np.max(np.abs(out[k] - ref)) <= tol * np.max(np.abs(ref))
    pl.close()


@pytest.mark.parametrize("L,p", [((64, 65), 2), ((4, 16, 17), 2)])   # strips; slabs with slices of 128 sites
def test_xmatvec_reads_small_vectors_in_binary64(L, p):
    """q and 2^-100 q (exact, ~1e-30): the same X q times 2^-100 to the stopping tolerance of
    the refinement, 1e-13, in both, times the lattice's condition (|H^-1| <= 1 / w_0 = 3.2,
    |H| < 12) with room for two of them."""
    w = wl(L, p, 4, K=2)
    omega, V, sigma, _ = I.make_inputs(w)
    rng = np.random.default_rng(8)
    q = rng.normal(size=(2, w.N)) + 1j * rng.normal(size=(2, w.N))
    pl = plan_for(w, D.DYSON_MIXED)
    u, us = np.zeros_like(q), np.zeros_like(q)
    D.dyson_xmatvec(pl.handle, 2, omega, V, sigma, q, u)
    D.dyson_xmatvec(pl.handle, 2, omega, V, sigma, q * 2.0 ** -100, us)
    assert np.max(np.abs(us * 2.0 ** 100 - u)) <= 2 * 40 * 1e-13 * np.max(np.abs(u))
    pl.close()


def test_nan_frequency_costs_no_iterations():
    """A NaN in Sigma makes the interface right-hand side of its frequency NaN: X q counts as
    zero there, without interface iterations, and the other frequencies keep their bits."""
    w = wl((40, 33), 2, 4, K=3)
    omega, V, sigma, q1 = I.make_inputs(w)
    pl = plan_for(w, D.DYSON_MIXED)
    clean = pl.solve(omega, V, sigma, q1)
    bad = sigma.copy()
    bad[1, 500] = np.nan
    out = pl.solve(omega, V, bad, q1)
    info = pl.info(3)
    assert info["iters"][1] == 0 and info["steps"][1] == 1
    for k in (0, 2):
        assert np.array_equal(out[k], clean[k])
    assert np.isnan(out[1, 500])
    pl.close()


@pytest.mark.parametrize("L,p", [((6, 527), 16), ((6, 1039), 16)])   # W = 32, 64
@pytest.mark.parametrize("precision,tol", [(D.DYSON_FP64, 1e-11), (D.DYSON_MIXED, 1e-9)])
def test_sixteen_strips(L, p, precision, tol):
    """The largest cluster, 16 CTAs with up to an SM's shared memory each."""
    w = wl(L, p, 4, K=2, trap=1e-5)
    omega, V, sigma, _ = I.make_inputs(w)
    rng = np.random.default_rng(9)
    q = rng.normal(size=(2, w.N)) + 1j * rng.normal(size=(2, w.N))
    pl = plan_for(w, precision)
    u = np.zeros_like(q)
    D.dyson_xmatvec(pl.handle, 2, omega, V, sigma, q, u)
    for k in range(2):
        ref = local_X(w, omega[k], V, sigma[k])[1](q[k])
        assert np.max(np.abs(u[k] - ref)) <= tol * np.max(np.abs(ref))
    pl.close()


def test_infinite_interface_entry_is_not_answered_with_zero():
    w = wl((40, 33), 2, 4, K=1)              # the interface line is y = 16
    omega, V, sigma, _ = I.make_inputs(w)
    q = np.ones((1, w.N), complex)
    q[0, 5 + 40 * 16] = np.inf
    pl = plan_for(w, D.DYSON_MIXED, krylov_maxit=50)
    u = np.zeros_like(q)
    D.dyson_xmatvec(pl.handle, 1, omega, V, sigma, q, u)
    assert not np.any(np.isfinite(u))
    pl.close()
