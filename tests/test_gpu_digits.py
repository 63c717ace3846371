"""8-bit digit products (csrc/ozaki.cu) where they can go wrong: K beyond one
int32 piece, digits that all agree in sign, rows with an infinity or a NaN, and
QML_FP64 problems at the order where it changes to 55-bit digits.

Bounds.  48 bits: an operand's rounding is at most 2^-49 of its row's maximum
2^e (2 K 2^-49 over the sum), the dropped levels 8 and beyond at most 5.1 K
2^(14-64) (levels of 5, 4, ... products of digits up to 2^7), and level 6 past
2^24 loses no more than those: below 2^-45 K 2^(e+f) in all."""
import numpy as np
import pytest

import parity as P
from oracle import harmonic, qml
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


@pytest.mark.parametrize("m,n,k", [(129, 131, 15361), (128, 64, 16), (1, 1, 40000)])
def test_equal_digits_long_k(api, m, n, k):
    """Every element (2^48 - 1) 2^-48 or the value whose digits are all 127: the
    level sums are as large as they can be."""
    lo = sum(127.0 * 256.0 ** i for i in range(5))
    for v in (1.0 - 2.0 ** -48, (127.0 * 256.0 ** 5 + lo) * 2.0 ** -48):
        A = np.full((m, k), v)
        B = np.full((k, n), v)
        C = api.gemm(td(A), td(B), precision=1).cpu().numpy()
        ref = float(k) * v * v
        e = np.frexp(v)[1]
        assert np.abs(C - ref).max() <= k * 2.0 ** (2 * e - 45) + 2.0 ** -52 * ref
        assert (C == C[0, 0]).all()


def test_nonfinite_rows_poison_their_outputs_only(api):
    rng = np.random.default_rng(3)
    A, B = rng.normal(size=(300, 200)), rng.normal(size=(200, 150))
    A[7, 11], A[260, 199], B[5, 149] = np.inf, np.nan, -np.inf
    C0 = rng.normal(size=(300, 150))
    Cd = td(C0)
    api.gemm(td(A), td(B), Cd, alpha=-1.0, beta=1.0, precision=1)
    C = Cd.cpu().numpy()
    bad = np.zeros((300, 150), dtype=bool)
    bad[[7, 260], :] = True
    bad[:, 149] = True
    assert np.isnan(C[bad]).all()
    A[7, 11] = A[260, 199] = B[5, 149] = 0.0
    ref = C0 - A @ B
    assert np.abs(C - ref)[~bad].max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("m,n", [(1, 1), (128, 64), (127, 65), (129, 128), (300, 200), (520, 33)])
@pytest.mark.parametrize("k", [16, 130, 1100])
def test_narrow_tiles_equal_wide(api, m, n, k):
    """Products of few tiles take half-width ones: the same bits as the same
    entries of a product of 81 whole tiles, for every alpha and beta form."""
    rng = np.random.default_rng(m + n + k)
    A, B, C0 = rng.normal(size=(1100, k)), rng.normal(size=(k, 1100)), rng.normal(size=(1100, 1100))
    for alpha, beta in ((1.0, 0.0), (-1.0, 1.0), (0.3, -0.7)):
        W, Nw = td(C0), td(C0[:m, :n])
        api.gemm(td(A), td(B), W, alpha=alpha, beta=beta, precision=1)
        api.gemm(td(A[:m]), td(B[:, :n]), Nw, alpha=alpha, beta=beta, precision=1)
        assert torch.equal(W[:m, :n], Nw)
    if m == 300:  # X^T X, lower: the upper triangle stays
        W, Nw = td(np.zeros((1700, 1700))), td(C0[:m, :m])
        X = rng.normal(size=(k, 1700))
        api.gemm(td(X), td(X), W, transA=True, lower=True, precision=1)
        api.gemm(td(X[:, :m]), td(X[:, :m]), Nw, transA=True, lower=True, precision=1)
        W, Nw = W.cpu().numpy(), Nw.cpu().numpy()
        assert np.array_equal(np.tril(W[:m, :m]), np.tril(Nw))
        assert np.array_equal(np.triu(Nw, 1), np.triu(C0[:m, :m], 1))


@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("m,n,k", [(130, 70, 24576), (130, 70, 24577), (33, 129, 49153)])
def test_k_in_pieces(api, m, n, k, ta, tb):
    """K past the digits kept at a time: each piece adds to C (bound as above, with
    a rounding of C for each)."""
    rng = np.random.default_rng(k + m)
    A, B, C0 = rng.uniform(-1, 1, (m, k)), rng.uniform(-1, 1, (k, n)), rng.normal(size=(m, n))
    Cd = td(C0)
    api.gemm(td(A.T if ta else A), td(B.T if tb else B), Cd, transA=ta, transB=tb, alpha=-1.0,
             beta=0.5, precision=1)
    C = Cd.cpu().numpy()
    bound = k * 2.0 ** -45 + 8 * 2.0 ** -52 * np.abs(C).max()
    assert np.abs(C - (0.5 * C0 - A @ B)).max() <= bound
    if m == 130 and ta != tb:
        Gd = td(A.T if ta else A)
        G = api.gemm(Gd, Gd, transA=ta, transB=tb, lower=True, precision=1).cpu().numpy()
        ref = np.tril(A @ A.T)
        assert np.abs(np.tril(G) - ref).max() <= k * 2.0 ** -45 + 8 * 2.0 ** -52 * np.abs(ref).max()


@pytest.mark.parametrize("n", [255, 256, 257, 511, 513])
@pytest.mark.parametrize("basis", [0, 1])
def test_fp64_order_where_digits_start(api, n, basis):
    """T maps on n pixels, float64: F, b, y and lnL against the oracle, at
    float64 rounding times the covariance's condition (about 1e4)."""
    th, ph, _ = synth.healpix_ring_centres(8)
    wl = synth.make_workload("T", 8, 11, True, False, 0.0, ("TT",), 7, 40 + n,
                             geometry=(th[100:100 + n], ph[100:100 + n]))
    Y, alm, noise, maps = P.oracle_maps(wl, 3)
    ref = qml.qml_for(wl, Y, maps=maps)
    prob = api.Problem.from_workload(wl, basis=basis)
    F, plan = api.fisher(prob)
    est = plan.estimate(td(maps))
    plan.free()
    assert P.rel_max(F, ref["F"]) <= 1e-11
    assert P.rel_max(est["b"], ref["b"]) <= 1e-11
    assert P.rel_max(est["y"], ref["y"]) <= 1e-11
    C = qml.total_cov(Y, wl.cl_fid, wl.comps, wl.lmin, wl.lmax, wl.N())
    lnl, chi2, ld = qml.loglike(C, maps)
    g = api.loglike(prob, torch.as_tensor(wl.cl_fid.reshape(-1), device="cuda"), td(maps))
    assert P.rel_max(g[0], lnl) <= 1e-12
    assert abs(float(P.to_np(g[2])) - ld) <= 1e-12 * abs(ld)


@pytest.mark.parametrize("beta", [0.0, 1.0])
@pytest.mark.parametrize("m,n", [(128, 64), (300, 200), (1700, 1500)])
def test_rows_and_columns_of_any_size(api, m, n, beta):
    """Rows and columns scaled by powers of two whose sums leave the normal range
    one with another but not with those of the same index: a product is the
    unscaled one times the power, down to subnormal results, 0 and infinity.
    (128, 64) takes the half-width tiles, (1700, 1500) the whole ones."""
    rng = np.random.default_rng(m)
    k = 130
    A, B = rng.uniform(0.5, 1, (m, k)), rng.uniform(0.5, 1, (k, n))
    C0 = rng.normal(size=(m, n))
    r, c = np.zeros(m, int), np.zeros(n, int)
    r[3::37], r[11::41], r[20::53] = -600, 600, -530
    c[5::29], c[14::31], c[23::43] = -600, 600, -530
    with np.errstate(over="ignore", under="ignore"):
        ref = beta * C0 + np.ldexp(A @ B, r[:, None] + c[None, :])
        Cd = td(C0)
        api.gemm(td(np.ldexp(A, r[:, None])), td(np.ldexp(B, c[None, :])), Cd, beta=beta,
                 precision=1)
        C = Cd.cpu().numpy()
        inf = np.isinf(ref)
        assert inf.any() and (C[inf] == ref[inf]).all()
        # 48 bits: 2^-45 K against sums of at least K / 4; a rounding of C, and
        # one in the last place of a subnormal result
        err = np.abs(C[~inf] - ref[~inf])
        assert (err <= 2.0 ** -43 * np.abs(ref - beta * C0)[~inf] + 2.0 ** -51 * np.abs(ref[~inf])
                + 2.0 ** -1073).all()


@pytest.mark.parametrize("m,n,lower", [(2500, 2500, True), (1300, 2300, False)])
def test_work_order_bands_same_bits(api, m, n, lower):
    """Tiles taken in bands of one row, of an odd few, of more rows than there are."""
    rng = np.random.default_rng(m)
    A = td(rng.normal(size=(m, 70)))
    B = A if lower else td(rng.normal(size=(n, 70)))
    outs = []
    try:
        for band in (1, 3, 8, 4096):
            api.tune_set("ozaki_band", band)
            C = td(np.ones((m, n)))
            api.gemm(A, B, C, transB=True, alpha=-1.0, beta=1.0, lower=lower, precision=1)
            outs.append(C)
    finally:
        api.tune_set("ozaki_band", 8)
    assert all(torch.equal(outs[0], C) for C in outs[1:])
    ref = 1.0 - (A @ B.t()).cpu().numpy()
    got = outs[0].cpu().numpy()
    sel = np.tril(np.ones((m, n), bool)) if lower else np.ones((m, n), bool)
    assert np.abs(got - ref)[sel].max() <= 1e-12 * np.abs(ref).max()
    assert (got[~sel] == 1.0).all()


@pytest.mark.parametrize("nslices,bits", [(1, 24), (4, 24), (5, 48), (9, 55), (10, 55)])
def test_nslices_forms(api, nslices, bits):
    """Every digit count that nslices asks for, through a Fisher matrix and estimates.
    A product's error is about sqrt(K) 2^-bits of its row's and column's maxima; C
    passes it on with its condition number (and the float64 parts add 1e-11)."""
    th, ph, _ = synth.healpix_ring_centres(8)
    n = 560
    wl = synth.make_workload("T", 8, 11, True, False, 0.0, ("TT",), 7, 50,
                             geometry=(th[100:100 + n], ph[100:100 + n]))
    Y, alm, noise, maps = P.oracle_maps(wl, 10)
    ref = qml.qml_for(wl, Y, maps=maps)
    cond = np.linalg.cond(qml.total_cov(Y, wl.cl_fid, wl.comps, wl.lmin, wl.lmax, wl.N()))
    tol = 4 * cond * np.sqrt(n) * 2.0 ** -bits + 1e-11
    prob = api.Problem.from_workload(wl, precision=1, nslices=nslices)
    F, plan = api.fisher(prob)
    est = plan.estimate(td(maps))
    plan.free()
    assert P.rel_max(F, ref["F"]) <= tol
    assert P.rel_max(est["y"], ref["y"]) <= tol


@pytest.mark.parametrize("call", ["fisher", "estimate", "loglike", "cross", "batch"])
def test_fp64_calls_report_a_timeout(api, call):
    """QML_FP64 calls with digit products report a wait that runs out as the split
    ones do, and run normally afterwards."""
    th, ph, _ = synth.healpix_ring_centres(8)
    wl = synth.make_workload("T", 8, 9, True, False, 0.0, ("TT",), 7, 51,
                             geometry=(th[100:700], ph[100:700]))
    maps = td(P.oracle_maps(wl, 10)[3])
    prob = api.Problem.from_workload(wl)
    cl = torch.as_tensor(wl.cl_fid.reshape(-1), device="cuda")
    F0, plan = api.fisher(prob)
    run = {"fisher": lambda: api.fisher(prob, keep_plan=False),
           "estimate": lambda: plan.estimate(maps),
           "loglike": lambda: api.loglike(prob, cl, maps),
           "cross": lambda: api.cross(plan, plan, maps, maps),
           "batch": lambda: api.loglike_batch([(prob, maps)], np.zeros(2, int), cl.repeat(2, 1))}
    api.tune_set("test_wait_timeout", 1)
    try:
        with pytest.raises(api.QMLError) as ei:
            run[call]()
    finally:
        api.tune_set("test_wait_timeout", 0)
    assert ei.value.status == 5, str(ei.value)
    run[call]()
    plan.free()
    F1, p1 = api.fisher(prob)
    p1.free()
    assert torch.equal(F0, F1)
