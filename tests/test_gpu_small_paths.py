"""The kernels that small problems and small products take, at the sizes where
they can go wrong: the one-CTA eigensolver up to its largest order, the quadratic
estimate's lane groups, 64-wide Cholesky blocks whose diagonals leave the range
of their factor's fast form, products with the whole K range on chip, triangular
solves with a few columns, and the emulator's fused training and input passes.

Bounds.  A product of K terms in float64: K 2^-53 sum |a||b| at most.  Solves and
factors of well-conditioned matrices: the tolerances the same calls have at other
sizes.  Powers of two scale exactly, so a scaled matrix has the unscaled one's
bound.  The first Adam step moves every weight by the learning rate times the
sign of its gradient: two orders of summation give the same step unless a gradient
is at the level of float32 rounding (fewer than one in a hundred)."""
import numpy as np
import pytest
import scipy.linalg as sla

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


def spd(n, seed):
    g = np.random.default_rng(seed)
    B = g.normal(size=(n, n))
    return B @ B.T / n + np.eye(n)


@pytest.mark.parametrize("na", [1, 2, 3, 4, 31, 32, 61, 62, 63, 64])
def test_small_eigensolver_orders(api, na):
    """F^-1/2 q and F^-1 q of na multipoles (full sky, no beam) against LAPACK on
    the same F and q."""
    th, ph, _ = synth.healpix_ring_centres(8)
    wl = synth.make_workload("T", 8, na + 1, True, False, 0.0, ("TT",), 5, 60 + na,
                             geometry=(th, ph))
    wl.transfer_T[:] = 1.0
    _, _, _, maps = P.oracle_maps(wl, 2)
    F, plan = api.fisher(api.Problem.from_workload(wl))
    est = plan.estimate(td(maps))
    plan.free()
    Fh, q = P.to_np(F), P.to_np(est["q_conv"])
    w, V = np.linalg.eigh(Fh)
    assert w[0] > 1e-12 * w[-1]  # no eigenvalue is cut
    dcr = (V / np.sqrt(w)) @ (V.T @ q)
    dec = (V / w) @ (V.T @ q)
    assert P.cl_decorr_error(est["cl_decorr"], dcr) <= P.decorr_tol(Fh)
    assert P.cl_deconv_error(est["cl_deconv"], dec, Fh) <= P.decorr_tol(Fh)


@pytest.mark.parametrize("nsims", [1, 5, 33])
@pytest.mark.parametrize("comp", ["T", "QU", "TQU"])
def test_quadratic_estimate_lane_groups(api, comp, nsims):
    spec = {"T": ("TT",), "QU": ("EE", "BB", "EB"),
            "TQU": ("TT", "EE", "BB", "TE", "TB", "EB")}[comp]
    wl = synth.make_workload(comp, 4, 9, "T" in comp, "Q" in comp, 20.0, spec, 6, 70 + len(comp))
    Y, _, _, maps = P.oracle_maps(wl, nsims)
    ref = qml.qml_for(wl, Y, maps=maps)
    F, plan = api.fisher(api.Problem.from_workload(wl))
    est = plan.estimate(td(maps))
    plan.free()
    assert P.rel_max(F, ref["F"]) <= P.TOL
    assert P.rel_max(est["y"], ref["y"]) <= P.TOL


@pytest.mark.parametrize("exps", [(0, 0), (600, 600), (-600, -600), (-600, 600), (-511, 512)])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 63, 64, 65, 130])
def test_potrf_block_ranges(api, n, exps):
    """A = D S D with D powers of two, so that diagonals lie between 2^exps[0] and
    2^exps[1]: L = D chol(S)."""
    S = spd(n, n)
    d = 2.0 ** np.random.default_rng(n).integers(exps[0] // 2, exps[1] // 2 + 1, size=n)
    ref = np.linalg.cholesky(S)
    At = td(S * d[:, None] * d[None, :])
    ld = float(P.to_np(api.potrf(At)))
    L = np.tril(At.cpu().numpy()) / d[:, None]
    assert np.abs(L - ref).max() <= 1e-12 * np.abs(ref).max()
    ldr = 2 * np.log(np.diag(ref)).sum() + 2 * np.log(d).sum()
    assert abs(ld - ldr) <= 1e-12 * max(1.0, np.abs(np.log(d)).sum())


@pytest.mark.parametrize("col", [0, 7, 8, 39, 63, 64, 99])
def test_potrf_refuses_at_any_column(api, col):
    S = spd(100, 5)
    S[col, col] = -1.0
    with pytest.raises(api.QMLError):
        api.potrf(td(S))


@pytest.mark.parametrize("lower", [False, True])
@pytest.mark.parametrize("transB", [False, True])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (15, 17, 3), (16, 16, 16), (130, 130, 255),
                                   (33, 33, 256), (64, 49, 64)])
def test_gemm_whole_k_on_chip(api, m, n, k, transB, lower):
    """The tuning table names the kernel (code 10); every product form it takes."""
    if lower:
        n = m
    g = np.random.default_rng(m * n + k)
    A, B, C0 = g.normal(size=(m, k)), g.normal(size=(k, n)), g.normal(size=(m, n))
    api.tune_load(f"dgemm:0,{int(transB)},{int(lower)},{m},{n},{k},0 10\n")
    Ct = td(C0)
    api.gemm(td(A), td(B.T) if transB else td(B), Ct, transB=transB, alpha=-0.5, beta=2.0,
             lower=lower)
    got = Ct.cpu().numpy()
    ref = -0.5 * (A @ B) + 2.0 * C0
    bound = (k + 4) * 2.0 ** -53 * (0.5 * np.abs(A) @ np.abs(B) + 2.0 * np.abs(C0)) * 2
    sel = np.tril(np.ones((m, n), dtype=bool)) if lower else np.ones((m, n), dtype=bool)
    assert (np.abs(got - ref) <= bound)[sel].all()


@pytest.mark.parametrize("nrhs", [1, 2, 4, 5, 8, 9])
@pytest.mark.parametrize("n", [1, 65, 513, 1100])
def test_trsm_few_columns(api, n, nrhs):
    L = np.linalg.cholesky(spd(n, n))
    B = np.random.default_rng(nrhs).normal(size=(n, nrhs))
    X = api.trsm(td(L), td(B), precision=1).cpu().numpy()
    ref = sla.solve_triangular(L, B, lower=True)
    assert np.abs(X - ref).max() <= 1e-9 * np.abs(ref).max()


@pytest.mark.parametrize("n,batch", [(16, 16), (17, 32), (100, 112), (500, 512)])
@pytest.mark.parametrize("width,depth", [(16, 1), (64, 2), (256, 4)])
def test_emu_fused_step_matches_layerwise(api, width, depth, n, batch):
    """One epoch of one batch: fused up to 512 rows, layer by layer at 528 (the
    added rows are padding)."""
    g = np.random.default_rng(n)
    th = g.uniform(-1, 1, size=(n, 3))
    y = -(th ** 2).sum(axis=1) + np.sin(5 * th[:, 0]) * th[:, 1]
    got = []
    for b in (batch, 528):
        emu = api.Emulator(-np.ones(3), np.ones(3), width=width, depth=depth, seed=2)
        start = [emu.params(h) for h in (0, 1)]
        fl = emu.train(th, y, epochs=1, batch=b, lr=1e-3)
        got.append((start, fl, [emu.params(h) for h in (0, 1)]))
        emu.free()
    (s0, l0, p0), (s1, l1, p1) = got
    for h in (0, 1):
        assert (s0[h] == s1[h]).all()
        assert (p0[h] != s0[h]).any()
        assert np.mean(np.abs(p0[h] - p1[h]) > 1e-6) <= 0.01
        assert abs(l0[h] - l1[h]) <= 1e-2 * abs(l1[h])


@pytest.mark.parametrize("ndim", [1, 5, 8])
@pytest.mark.parametrize("npts", [1, 127, 129, 1000])
def test_emu_first_layer_inputs(api, ndim, npts):
    """Points normalised and widened by one pass (first layer on tcgen05) against
    the WMMA first layer; points outside the training box among them."""
    g = np.random.default_rng(ndim)
    th = g.uniform(-1, 1, size=(600, ndim))
    y = -(th ** 2).sum(axis=1) + np.sin(3 * th[:, 0])
    emu = api.Emulator(-np.ones(ndim), np.ones(ndim), width=64, depth=2, seed=4)
    emu.train(th, y, epochs=4, batch=64)
    test = g.uniform(-1.1, 1.1, size=(npts, ndim))
    try:
        pa, fa = emu.predict(test, tol=0.05)
        api.tune_set("emu_tc0", 0)
        pb, fb = emu.predict(test, tol=0.05)
    finally:
        api.tune_set("emu_tc0", 1)
    emu.free()
    assert np.isfinite(pa).all() and np.abs(pa - pb).max() <= 5e-3
    out = (np.abs(test) > 1).any(axis=1)
    assert (fa[out] == 1).all() and (fb[out] == 1).all()
    assert np.mean(fa == fb) >= 0.99


@pytest.mark.parametrize("form", ["ldl", "general", "float-float"])
def test_potrf_rows_agree_between_warps(api, form):
    """Rows 16-39 and 40-63 of a block equal in its first 16 columns: a panel's
    rows fall to three warps, each with the pivot block factored for itself, and
    equal rows must come out with equal bits.  'general': diagonals outside
    the range of the fast form."""
    g = np.random.default_rng(11)
    B = g.normal(size=(64, 64))
    S = B @ B.T / 64
    S[40:, :16] = S[16:40, :16]
    S[:16, 40:] = S[40:, :16].T
    S += 8.0 * np.eye(64)
    if form == "general":
        S *= 2.0 ** -600
    At = td(S)
    ref = np.linalg.cholesky(S)
    if form == "float-float":
        api.tune_set("split_diag_df", 1)
    try:
        for _ in range(200):
            W = At.clone()
            api.potrf(W, precision=int(form == "float-float"))
            L = W.cpu().numpy()
            assert np.array_equal(L[16:40, :16], L[40:, :16])
    finally:
        api.tune_set("split_diag_df", 0)
    assert np.abs(np.tril(L) - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("transB", [False, True])
@pytest.mark.parametrize("m,n", [(1, 1048560), (1, 1048561), (1, 1048576), (3, 1048577)])
def test_gemm_more_columns_than_a_grid(api, m, n, transB):
    """16-wide tiles would put more CTAs along the columns than a launch takes: the
    autotuner, the built-in choice, and a tuning table that names them (codes 10 and
    11)."""
    g = np.random.default_rng(n)
    A, B = g.normal(size=(m, 3)), g.normal(size=(3, n))
    ref = A @ B
    bound = 8 * 2.0 ** -53 * (np.abs(A) @ np.abs(B))
    Bd = td(B.T) if transB else td(B)
    key = f"dgemm:0,{int(transB)},0,{m},{n},3,0"
    try:
        for text in ("dgemm_autotune 0\n", "dgemm_autotune 1\n", key + " 10\n", key + " 11\n"):
            api.tune_load(text)
            C = api.gemm(td(A), Bd, transB=transB).cpu().numpy()
            assert (np.abs(C - ref) <= bound).all()
    finally:
        api.tune_set("dgemm_autotune", 1)


def test_potrf_column_by_reciprocal(api):
    """First column of a block, L_i0 = (a_i0 (1 / d)) sqrt(d), for pivots d of many
    mantissas and exponents: four roundings, each at most 0.51 units."""
    g = np.random.default_rng(17)
    for e in (-500, -40, -1, 0, 1, 30, 500):
        for d in np.ldexp(np.concatenate([[0.5, np.nextafter(1.0, 0.0), 0.75],
                                          g.uniform(0.5, 1.0, size=37)]), e):
            A = np.diag(np.full(64, 64.0 * d))
            A[0, 0] = d
            A[1:, 0] = d * g.uniform(-1.0, 1.0, size=63)
            W = td(A)
            api.potrf(W)
            L = W.cpu().numpy()[:, 0].astype(np.longdouble)
            dl = np.longdouble(d)
            ref = A[:, 0].astype(np.longdouble) / np.sqrt(dl)
            assert (np.abs(L - ref)[1:] <= 4 * 0.51 * 2.0 ** -52 * np.abs(ref)[1:]).all()
            assert abs(L[0] - np.sqrt(dl)) <= 0.51 * 2.0 ** -52 * np.sqrt(dl)
