"""QML_FP64 where the pixels' noise differs by orders of magnitude inside a 512-wide
block of the digit products (n >= 256): Cholesky and its solves do not depend on
the scale of rows and columns, and the products with block inverses must not
either.

Bounds.  A solve with C = D S D, cond(S) about 10, has a relative error of at most
about n cond(S) 2^-53 = 1e-12, whatever D.  Against the oracle (float64 too): the
tolerances the same calls have with even noise."""
import numpy as np
import pytest

import parity as P
from oracle import qml
from paper_2605_21149_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_21149_gb300 import api as A
    from paper_2605_21149_gb300 import build
    build.build()
    return A


def td(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device="cuda").t().contiguous().t()


def correlated(n, g):
    B = g.normal(size=(n, n))
    S = B @ B.T / n + 0.5 * np.eye(n)
    d = np.sqrt(np.diag(S))
    return S / d[:, None] / d[None, :]


def t_workload(n, lmax, seed):
    th, ph, _ = synth.healpix_ring_centres(16)
    return synth.make_workload("T", 16, lmax, True, False, 0.0, ("TT",), 7, seed,
                               geometry=(th[500:500 + n], ph[500:500 + n]))


@pytest.mark.parametrize("nmaps", [8, 9, 40])
@pytest.mark.parametrize("n,bits", [(300, 13), (513, 13), (1100, 13), (1100, 200)])
def test_loglike_scaled_pixels(api, n, bits, nmaps):
    """Noise D S D and maps D x, D powers of two in 2^+-bits, no signal: chi^2 of S
    and x, ln|C| shifted by 2 ln|D|.  (8 maps: solved on the float64 pipe.)"""
    g = np.random.default_rng(n + nmaps)
    S = correlated(n, g)
    x = np.linalg.cholesky(S) @ g.normal(size=(n, nmaps))
    e = g.integers(-bits, bits + 1, size=n)
    wl = t_workload(n, 6, 3)
    wl.cl_fid[:] = 0.0
    out = []
    for ex in (np.zeros(n, int), e):
        wl.N = lambda: np.ldexp(S, ex[:, None] + ex[None, :])
        prob = api.Problem.from_workload(wl)
        r = api.loglike(prob, torch.zeros(6 * (wl.lmax + 1), dtype=torch.float64, device="cuda"),
                        td(np.ldexp(x, ex[:, None])))
        out.append([P.to_np(v) for v in r])
    (l0, c0, d0), (l1, c1, d1) = out
    assert np.abs(c1 - c0).max() <= 1e-12 * c0.max()
    assert abs(float(d1) - float(d0) - 2 * np.log(2.0) * e.sum()) <= 1e-12 * max(
        abs(float(d1)), 2 * np.log(2.0) * np.abs(e).sum())
    ref = (np.linalg.solve(np.linalg.cholesky(S), x) ** 2).sum(axis=0)
    assert np.abs(c1 - ref).max() <= 1e-12 * ref.max()


@pytest.mark.parametrize("basis", [0, 1])
@pytest.mark.parametrize("spread", [1e2, 1e6])
def test_fisher_estimate_uneven_noise(api, spread, basis):
    """Correlated noise whose standard deviation runs over `spread` from about the
    signal's up, in no order; a tenth of the pixels has the lowest."""
    g = np.random.default_rng(8)
    n = 700
    wl = t_workload(n, 11, 4)
    Y, _, _, maps = P.oracle_maps(wl, 12)
    sig = np.sqrt(np.diag(qml.total_cov(Y, wl.cl_fid, wl.comps, wl.lmin, wl.lmax, 0 * wl.N())).mean())
    d = sig * spread ** np.clip(g.uniform(-0.1, 1.0, size=n), 0.0, None)
    N = correlated(n, g) * d[:, None] * d[None, :]
    wl.N = lambda: N
    maps = maps + np.linalg.cholesky(N) @ g.normal(size=(n, 12))
    ref = qml.qml_for(wl, Y, maps=maps)
    prob = api.Problem.from_workload(wl, basis=basis)
    F, plan = api.fisher(prob)
    est = plan.estimate(td(maps))
    plan.free()
    assert P.rel_max(F, ref["F"]) <= 1e-11
    assert P.rel_max(est["y"], ref["y"]) <= 1e-11
    assert P.rel_max(est["b"], ref["b"]) <= 1e-11
    rl, rc, rd = qml.loglike(qml.total_cov(Y, wl.cl_fid, wl.comps, wl.lmin, wl.lmax, N), maps)
    lnl, chi2, ld = (P.to_np(v) for v in api.loglike(
        prob, torch.as_tensor(wl.cl_fid.reshape(-1), device="cuda"), td(maps)))
    assert np.abs(chi2 - rc).max() <= 1e-11 * rc.max()
    assert np.abs(lnl - rl).max() <= 1e-11 * np.abs(rl).max()


@pytest.mark.parametrize("nmaps", [8, 12])
def test_batch_uneven_noise(api, nmaps):
    """Likelihood scan, inner matrices of order 495 on digit products, maps on both
    sides of the few-columns form; every map's chi^2 against the oracle."""
    g = np.random.default_rng(5)
    masks, taus, rs = synth.batch_workload(nside=8, lmax=12, rank=30, ngrid=4)
    wl = masks[0]
    Y, _, _, maps = P.oracle_maps(wl, nmaps)
    n = len(maps)
    sig = np.sqrt(np.diag(qml.total_cov(Y, wl.cl_fid, wl.comps, wl.lmin, wl.lmax, 0 * wl.N())))
    d = sig * 1e4 ** g.uniform(0.0, 1.0, size=n)
    N = correlated(n, g) * d[:, None] * d[None, :]
    wl.N = lambda: N
    maps = maps + np.linalg.cholesky(N) @ g.normal(size=(n, nmaps))
    cl = synth.batch_item_spectra(12, taus[:6], rs[:6])
    lnl, chi2, ld = (P.to_np(v) for v in api.loglike_batch(
        [(api.Problem.from_workload(wl), td(maps))], np.zeros(6, int),
        torch.as_tensor(cl, device="cuda")))
    for i in range(6):
        rl, rc, rd = qml.loglike(qml.total_cov(Y, cl[i], wl.comps, wl.lmin, wl.lmax, N), maps)
        assert np.abs(chi2[i, :nmaps] - rc).max() <= 1e-10 * rc.max()
        assert np.abs(chi2[i, :nmaps] - rc).max() <= 1e-10 * np.abs(rc).min()
        assert abs(ld[i] - rd) <= 1e-10 * abs(rd)


@pytest.mark.parametrize("n", [300, 700])
def test_maps_with_zeros_and_nonfinite_pixels(api, n):
    """Pixels that are 0 in every map, a map of zeros, and maps with an infinity or a
    NaN, which spoil their own results and no others."""
    g = np.random.default_rng(n)
    S = correlated(n, g)
    x = np.linalg.cholesky(S) @ g.normal(size=(n, 14))
    x[5:n:7] = 0.0
    x[:, 3] = 0.0
    wl = t_workload(n, 6, 3)
    wl.cl_fid[:] = 0.0
    wl.N = lambda: S
    prob = api.Problem.from_workload(wl)
    cl = torch.zeros(6 * (wl.lmax + 1), dtype=torch.float64, device="cuda")
    ref = (np.linalg.solve(np.linalg.cholesky(S), x) ** 2).sum(axis=0)
    bad = x.copy()
    bad[n // 3, 8], bad[n - 2, 11], bad[0, 12] = np.nan, np.inf, -np.inf
    for m in (x, bad):
        lnl, chi2, ld = (P.to_np(v) for v in api.loglike(prob, cl, td(m)))
        ok = np.isfinite(m).all(axis=0)
        assert np.abs(chi2 - ref)[ok].max() <= 1e-12 * ref.max()
        assert chi2[3] == 0.0 and not np.isfinite(chi2[~ok]).any()
    chi2 = P.to_np(api.loglike(prob, cl, td(0.0 * x))[1])
    assert (chi2 == 0.0).all()


@pytest.mark.parametrize("n", [100, 300, 700])
def test_pixels_over_most_of_the_exponent_range(api, n):
    """Standard deviations between 2^-480 and 2^480 (covariances to 2^+-960)."""
    g = np.random.default_rng(n)
    S = correlated(n, g)
    x = np.linalg.cholesky(S) @ g.normal(size=(n, 10))
    e = g.integers(-480, 481, size=n)
    wl = t_workload(n, 6, 3)
    wl.cl_fid[:] = 0.0
    wl.N = lambda: np.ldexp(S, e[:, None] + e[None, :])
    lnl, chi2, ld = (P.to_np(v) for v in api.loglike(
        api.Problem.from_workload(wl), torch.zeros(6 * (wl.lmax + 1), dtype=torch.float64,
                                                   device="cuda"), td(np.ldexp(x, e[:, None]))))
    ref = (np.linalg.solve(np.linalg.cholesky(S), x) ** 2).sum(axis=0)
    assert np.abs(chi2 - ref).max() <= 1e-12 * ref.max()


@pytest.mark.parametrize("tnoise", [1.0, 1e4, 1e6])
def test_fields_of_different_noise(api, tnoise):
    """TQU with T noise far above that of Q and U, in a block that holds pixels of
    both: entries of F down to 1e-6 of their diagonal's, one by one (TOL of each: on
    the float64 pipe 7e-12)."""
    wl = synth.workload(1, "small")
    assert len(wl.theta_T) % 512 != 0
    N = wl.N()
    s = np.ones(len(N))
    s[:len(wl.theta_T)] = tnoise
    N = N * s[:, None] * s[None, :]
    wl.N = lambda: N
    Y, _, _, maps = P.oracle_maps(wl, 12)
    ref = qml.qml_for(wl, Y, maps=maps)
    F, plan = api.fisher(api.Problem.from_workload(wl))
    est = plan.estimate(td(maps))
    plan.free()
    F, Fr = P.to_np(F), ref["F"]
    big = np.abs(Fr) >= 1e-6 * np.sqrt(np.outer(np.diag(Fr), np.diag(Fr)))
    assert (np.abs(F - Fr) / np.abs(Fr))[big].max() <= P.TOL
    for a in range(len(Fr)):
        assert P.rel_max(est["y"][a], ref["y"][a]) <= P.TOL
