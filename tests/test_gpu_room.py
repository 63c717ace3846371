"""Memory that a call can do without: the tuning keys test_room (scan workers beyond
four) and test_digit_room make it count as not available, and the call gives the
same answer without it."""
import ctypes

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


def with_room(api, nbytes, fn, key="test_room"):
    api.tune_set(key, nbytes)
    try:
        return fn()
    finally:
        api.tune_set(key, 0)


def with_digit_room(api, nbytes, fn):
    return with_room(api, nbytes, fn, "test_digit_room")


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("items", [5, 20])
def test_scan_without_more_workers(api, items, graphs):
    """Eight workers, or the four that are always there: an item's result does not
    depend on its worker.  (2.5 MB: an extra worker's inner matrix would fit, the
    rest of its scratch would not.)"""
    masks, taus, rs = synth.batch_workload(nside=8, lmax=12, rank=30, ngrid=5)
    wls = masks[:2]
    probs = []
    for j, wl in enumerate(wls):
        probs.append((api.Problem.from_workload(wl, precision=1),
                      td(P.oracle_maps(wl, 2, seed_purpose=20 + j)[3])))
    cl = torch.as_tensor(synth.batch_item_spectra(12, taus[:items], rs[:items]), device="cuda")
    im = np.arange(items) % 2
    run = lambda: [P.to_np(v) for v in api.loglike_batch(probs, im, cl)]
    api.tune_set("batch_graphs", graphs)
    try:
        full = run()
        for nbytes in (1, 2_500_000):
            part = with_room(api, nbytes, run)
            assert all(np.array_equal(a, b) for a, b in zip(full, part))
    finally:
        api.tune_set("batch_graphs", 1)


def peak_pool_bytes(fn):
    """Highest use of the device's default memory pool while fn runs, above what was
    in use before."""
    cu = ctypes.CDLL("libcuda.so.1")
    pool, v = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    used_now, used_high = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH
    torch.cuda.synchronize()
    assert cu.cuMemPoolSetAttribute(pool, used_high, ctypes.byref(v)) == 0
    assert cu.cuMemPoolGetAttribute(pool, used_now, ctypes.byref(v)) == 0
    before = v.value
    fn()
    torch.cuda.synchronize()
    assert cu.cuMemPoolGetAttribute(pool, used_high, ctypes.byref(v)) == 0
    return v.value - before


@pytest.mark.parametrize("precision", [0, 1])
def test_scan_masks_share_digit_buffers(api, precision):
    """Each further mask of a scan adds its own matrices and no digits."""
    masks, taus, rs = synth.batch_workload(nside=8, lmax=12, rank=30, ngrid=4)
    wl = masks[0]
    prob = api.Problem.from_workload(wl, precision=precision)
    maps = td(P.oracle_maps(wl, 2, seed_purpose=20)[3])
    cl = torch.as_tensor(synth.batch_item_spectra(12, taus[:4], rs[:4]), device="cuda")
    n, k = prob.n, prob.k
    one, four = (peak_pool_bytes(lambda: api.loglike_batch([(prob, maps)] * nm, np.arange(4) % nm, cl))
                 for nm in (1, 4))
    own = 8 * (n * k + n * n + 64 * (n + 64) + k * k + 3 * n + 3 * k) + (1 << 20)
    assert four - one <= 3 * own


@pytest.mark.parametrize("nbytes", [1, 2_200_000, 40_000_000])
@pytest.mark.parametrize("basis", [0, 1])
def test_fp64_without_room_for_digits(api, basis, nbytes):
    """QML_FP64 on a device without room for digits (or for some of them): the
    float64 pipe, in every call that would use them, with plans of either kind."""
    th, ph, _ = synth.healpix_ring_centres(16)
    wl = synth.make_workload("T", 16, 17, True, False, 0.0, ("TT",), 7, 9,
                             geometry=(th[300:900], ph[300:900]))
    Y, _, _, maps = P.oracle_maps(wl, 11)
    ref = qml.qml_for(wl, Y, maps=maps)
    rl, rc, rd = qml.loglike(qml.total_cov(Y, wl.cl_fid, wl.comps, wl.lmin, wl.lmax, wl.N()), maps)
    prob = api.Problem.from_workload(wl, basis=basis)
    cl = torch.as_tensor(wl.cl_fid.reshape(-1), device="cuda")
    d = td(maps)
    Ff, full = api.fisher(prob)
    Fs, small = with_digit_room(api, nbytes, lambda: api.fisher(prob))
    for F in (Ff, Fs):
        assert P.rel_max(F, ref["F"]) <= P.TOL
    for plan in (full, small):
        for room in (0, nbytes):
            est = with_digit_room(api, room, lambda: plan.estimate(d))
            assert P.rel_max(est["y"], ref["y"]) <= P.TOL
    x = with_digit_room(api, nbytes, lambda: api.cross(full, small, d, d))
    assert P.rel_max(x["q"], ref["y"]) <= P.TOL and P.rel_max(x["Wx"], ref["F"]) <= P.TOL
    full.free()
    small.free()
    lnl, chi2, ld = (P.to_np(v) for v in with_digit_room(api, nbytes, lambda: api.loglike(prob, cl, d)))
    assert np.abs(lnl - rl).max() <= P.TOL * np.abs(rl).max()
    assert np.abs(chi2 - rc).max() <= P.TOL * rc.max()
    lnl, chi2, ld = (P.to_np(v) for v in with_digit_room(
        api, nbytes, lambda: api.loglike_batch([(prob, d)], np.zeros(6, int), cl.repeat(6, 1))))
    assert np.abs(chi2 - rc).max() <= P.TOL * rc.max()
    assert np.abs(ld - rd).max() <= P.TOL * abs(rd)


@pytest.mark.parametrize("width,depth,n,batch", [(64, 2, 300, 64), (256, 4, 1000, 512), (16, 1, 50, 16)])
def test_training_without_second_activations(api, width, depth, n, batch):
    """Both heads in fused steps, or head by head without the memory for them."""
    g = np.random.default_rng(n)
    th = g.uniform(-1, 1, size=(n, 3))
    y = -(th ** 2).sum(axis=1) + np.sin(5 * th[:, 0]) * th[:, 1]

    def train():
        emu = api.Emulator(-np.ones(3), np.ones(3), width=width, depth=depth, seed=3)
        loss = emu.train(th, y, epochs=3, batch=batch, lr=1e-3)
        out = [emu.params(h) for h in (0, 1)]
        emu.free()
        return np.array(loss), *out

    full, part = train(), with_room(api, 1, train)
    assert all(np.array_equal(a, b) for a, b in zip(full, part))
