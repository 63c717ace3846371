"""Performance cases: the calls a user of this library makes, over their real range of sizes.

Kinds of case
  solve      qml_fisher + qml_estimate: Fisher matrix, then spectra of a set of maps
  estimate   qml_estimate alone, many maps through one plan that the program keeps
  lnl        pix_loglike: one likelihood evaluation
  scan       pix_loglike_batch: a parameter scan over one or several masks
  predict    emu_predict: likelihood-emulator inference
  train      emu_create + emu_train: fitting the emulator

Inputs: HEALPix pixel centres outside a Galactic cut, Gaussian beam and pixel window, a dense
noise covariance sigma^2 I + G G^T, spectra templates with seeded parameters, and maps drawn from
the model.  Precision 0 is QML_FP64, 1 is QML_SPLIT_BF16.
"""
import math

import numpy as np
import torch

from paper_2605_21149_gb300 import api, synth

DEV = "cuda"
F64 = torch.float64
SPECS = {"T": ("TT",), "QU": ("EE", "BB", "EB"), "TQU": ("TT", "EE", "BB", "TE", "TB", "EB")}
PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))  # TT EE BB TE TB EB
MAX_FLOPS = 2.6e13   # of a drawn split-precision case (the largest listed one)
MAX_FLOPS64 = 9.0e11  # of a drawn float64 case


def _solve(name, fields, nside, lmax, cut, prec, maps, rank, basis=0, lsig=0, dl=0):
    return {"name": name, "kind": "solve", "fields": fields, "nside": nside, "lmax": lmax,
            "cut": cut, "precision": prec, "maps": maps, "rank": rank, "basis": basis,
            "lsig": lsig, "dl": dl}


def listed():
    return [
        # smallest call: one likelihood of a temperature-only low-resolution mask, as a sampler
        # makes it thousands of times; latency and launches
        {"name": "lnl_t8_f64", "kind": "lnl", "fields": "T", "nside": 8, "lmax": 16, "cut": 20.0,
         "precision": 0, "maps": 1, "rank": 10},
        # the small temperature-only analysis, ten simulations
        _solve("solve_t8_f64", "T", 8, 16, 20.0, 0, 10, 10),
        # a quick full-polarisation analysis at Nside 8, binned by two multipoles
        _solve("solve_tqu8_f64", "TQU", 8, 15, 20.0, 0, 100, 40, dl=2),
        # the headline analysis: TQU Nside 16, l = 2..47, 100 simulations, float64
        _solve("solve_tqu16_f64", "TQU", 16, 47, 20.0, 0, 100, 200),
        # the same analysis with split precision
        _solve("solve_tqu16_split", "TQU", 16, 47, 20.0, 1, 100, 200),
        # the largest analysis: QU Nside 32, l = 2..95, f_sky 0.7, split precision
        _solve("solve_qu32_split", "QU", 32, 95, 17.457603123722095, 1, 2, 200),
        # many pixels, few modes: the automatic basis rule picks the harmonic basis; the signal
        # band is wider than the window (multipole switching)
        _solve("solve_t16_harm_f64", "T", 16, 32, 0.0, 0, 25, 10, basis=2, lsig=40),
        # Monte-Carlo: 1000 simulations through a plan the program already has
        {"name": "estimate_qu16_f64", "kind": "estimate", "fields": "QU", "nside": 16, "lmax": 32,
         "cut": 10.0, "precision": 0, "maps": 1000, "rank": 10},
        # a piece of the (tau, r) scan over three masks, split precision for the per-mask products
        {"name": "scan_tqu16_split", "kind": "scan", "fields": "TQU", "nside": 16, "lmax": 47,
         "cuts": "30.0,17.5,5.7", "precision": 1, "maps": 1, "rank": 200, "items": 9},
        # exact likelihood labels for the emulator: many evaluations of a small mask, float64
        {"name": "scan_tqu8_f64", "kind": "scan", "fields": "TQU", "nside": 8, "lmax": 15,
         "cuts": "17.5", "precision": 0, "maps": 1, "rank": 40, "items": 256},
        # emulator inference over a chain's worth of points
        {"name": "predict_1m", "kind": "predict", "dim": 4, "width": 256, "depth": 4,
         "points": 1 << 20, "labels": 2048},
        # fitting the emulator: two epochs over the label set at the usual batch
        {"name": "train_8k", "kind": "train", "dim": 4, "width": 256, "depth": 4, "labels": 8192,
         "batch": 64, "epochs": 2},
    ]


# ------------------------------------------------------------------- sizes --
def _npix(nside, cut):
    z = synth.healpix_ring_centres(nside)[2]
    return len(synth.galactic_cut(z, cut))


def _dims(fields, nside, lmax, cut, lmin=2):
    """n (map rows), nc (components), k (modes of the window)."""
    nf = {"T": 1, "QU": 2, "TQU": 3}[fields]
    return nf * _npix(nside, cut), nf, nf * ((lmax + 1) ** 2 - lmin ** 2)


def _mid(rng, a, b):
    """An integer of [a, b], uniform in its logarithm."""
    return max(a, min(b, int(round(math.exp(rng.uniform(math.log(a), math.log(b + 0.49)))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "estimate", "lnl", "scan", "predict", "train"])
    if kind == "predict":
        return {"kind": kind, "dim": rng.randint(2, 6), "width": rng.choice([64, 128, 192, 256]),
                "depth": rng.randint(2, 4), "points": _mid(rng, 100, 1 << 20), "labels": 2048}
    if kind == "train":
        return {"kind": kind, "dim": rng.randint(2, 6), "width": rng.choice([64, 128, 192, 256]),
                "depth": rng.randint(2, 4), "labels": _mid(rng, 700, 8192),
                "batch": 16 * _mid(rng, 2, 16), "epochs": rng.randint(1, 2)}
    while True:
        prec = rng.randint(0, 1)
        fields = rng.choice(["T", "QU", "TQU"])
        nside = _mid(rng, 6, 32 if prec and kind in ("solve", "lnl") else 16)
        lmax = rng.randint(nside, (5 if fields != "T" else 4) * nside // 2)
        cut = rng.uniform(0.0, 20.0)
        n, nc, k = _dims(fields, nside, lmax, cut)
        case = {"kind": kind, "fields": fields, "nside": nside, "lmax": lmax,
                "precision": prec, "maps": _mid(rng, 1, 300), "rank": rng.choice([10, 40, 200])}
        if kind == "scan":
            cuts = [round(rng.uniform(2.0, 30.0), 2) for _ in range(rng.randint(1, 3))]
            case |= {"cuts": ",".join(str(c) for c in cuts), "maps": rng.randint(1, 8),
                     "items": _mid(rng, 1, 200)}
        else:
            case["cut"] = round(cut, 2)
        if kind == "solve":
            case |= {"basis": rng.randint(0, 2), "lsig": rng.choice([0, 0, lmax + 5]),
                     "dl": rng.choice([0, 0, 2, 3])}
        if kind == "estimate":
            case["maps"] = _mid(rng, 1, 1000)
        nl = lmax - 1
        if len(SPECS[fields]) * nl > 600:
            continue
        if kind in ("solve", "estimate") and (k > 1.2 * n or n < 100):
            continue  # more modes than the mask constrains: not an analysis anyone runs
        # what stays in float64 (float64 cases, the inner matrices of the harmonic basis and of a
        # scan) is bounded by the float64 rate
        w = work(case)["flops"]
        f64 = not prec or kind == "scan" or (kind == "solve" and case["basis"] != 0)
        if w > (MAX_FLOPS64 if f64 else MAX_FLOPS):
            continue
        return case


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _harmonics(theta, phi, lmin, lmax, fields, transfer):
    """The real harmonic matrix (rows T, Q, U pixels; columns component-major, l, then m = 0,
    cos 1, sin 1, ...) with the transfer folded in, in float64: Wigner d^l_{m s}, s = 0 and +-2,
    by the three-term recurrence in l from its closed form at l = max(m, |s|)."""
    dev = theta.device
    npx = theta.numel()
    has_t, has_p = "T" in fields, "QU" in fields
    nc = (1 if has_t else 0) + (2 if has_p else 0)
    k0 = (lmax + 1) ** 2 - lmin ** 2
    Y = torch.zeros((nc * k0, nc * npx), dtype=F64, device=dev)  # transposed: one row per mode
    m = torch.arange(lmax + 1, dtype=F64, device=dev)[None, :]
    x = torch.cos(theta)[:, None]
    ch, sh = torch.cos(theta / 2)[:, None], torch.sin(theta / 2)[:, None]
    ang = phi[:, None] * m
    cosm, sinm = torch.cos(ang), torch.sin(ang)
    spins = ((0,) if has_t else ()) + ((2, -2) if has_p else ())
    lg = lambda v: torch.lgamma(v + 1)
    start, prev, cur = {}, {}, {}
    for s in spins:
        l0 = torch.clamp(m, min=float(abs(s)))
        a, b = (l0 + abs(s)), (l0 - abs(s))
        hi = torch.where(m >= abs(s), m, torch.full_like(m, float(abs(s))))
        if s == 0:
            nrm = torch.exp(0.5 * (lg(2 * m) - 2 * lg(m)))
            d0 = torch.where(m % 2 == 0, 1.0, -1.0) * nrm * (ch * sh) ** m
        else:
            # m >= 2: (-1)^(m-s) sqrt((2m)!/((m+s)!(m-s)!)) c^(m+s) s^(m-s)
            ms = torch.clamp(m, min=2.0)
            big = torch.where((ms - s) % 2 == 0, 1.0, -1.0) * torch.exp(
                0.5 * (lg(2 * ms) - lg(ms + s) - lg(ms - s))) * ch ** (ms + s) * sh ** (ms - s)
            mm = torch.clamp(m, max=2.0)
            n2 = torch.exp(0.5 * (math.lgamma(5) - lg(2 + mm) - lg(2 - mm)))
            if s == 2:
                small = n2 * ch ** (2 + mm) * sh ** (2 - mm)
            else:
                small = torch.where(mm % 2 == 0, 1.0, -1.0) * n2 * ch ** (2 - mm) * sh ** (2 + mm)
            d0 = torch.where(m >= 2, big, small)
        start[s], cur[s], prev[s] = d0, torch.zeros_like(d0), torch.zeros_like(d0)
    l0 = {s: torch.clamp(m, min=float(abs(s))) for s in spins}
    c_e = k0 if has_t else 0
    c_b = c_e + k0
    q0 = npx if has_t else 0
    for l in range(0, lmax + 1):
        for s in spins:
            # from l - 1 to l; start at l = l0
            j = l - 1.0
            if l >= 1:
                den = j * torch.sqrt(torch.clamp((l * l - m * m) * (l * l - s * s), min=0.0))
                num = ((2 * j + 1) * (j * (j + 1) * x - m * s) * cur[s]
                       - (j + 1) * math.sqrt(max(j * j - s * s, 0.0))
                       * torch.sqrt(torch.clamp(j * j - m * m, min=0.0)) * prev[s])
                if j == 0:  # s = 0, m = 0: P_1 = x P_0
                    nxt = torch.where(m == 0, x * cur[s], torch.zeros_like(num))
                else:
                    nxt = torch.where(l > l0[s], num / torch.where(den == 0, 1.0, den), 0.0)
            else:
                nxt = torch.zeros_like(cur[s])
            nxt = torch.where(l0[s] == l, start[s], nxt)
            prev[s], cur[s] = cur[s], nxt
        if l < lmin:
            continue
        off = l * l - lmin * lmin
        t = float(transfer[l]) * math.sqrt((2 * l + 1) / (4 * math.pi))
        wt = torch.full((l + 1,), math.sqrt(2.0) * t, dtype=F64, device=dev)
        wt[0] = t
        ic = torch.cat([torch.zeros(1, dtype=torch.long, device=dev),
                        2 * torch.arange(1, l + 1, device=dev) - 1]) + off
        isn = 2 * torch.arange(1, l + 1, device=dev) + off
        C, S = cosm[:, :l + 1], sinm[:, :l + 1]
        if has_t:
            lam = cur[0][:, :l + 1] * wt
            Y[ic, :npx] = (lam * C).t()
            Y[isn, :npx] = (lam * S)[:, 1:].t()
        if has_p:
            f1 = -0.5 * (cur[-2][:, :l + 1] + cur[2][:, :l + 1]) * wt
            f2 = 0.5 * (cur[-2][:, :l + 1] - cur[2][:, :l + 1]) * wt
            re_e, im_e, re_b, im_b = f1 * C, f1 * S, -f2 * S, f2 * C
            Q, U = slice(q0, q0 + npx), slice(q0 + npx, q0 + 2 * npx)
            Y[c_e + ic, Q], Y[c_e + ic, U] = re_e.t(), re_b.t()
            Y[c_b + ic, Q], Y[c_b + ic, U] = -re_b.t(), re_e.t()
            Y[c_e + isn, Q], Y[c_e + isn, U] = im_e[:, 1:].t(), im_b[:, 1:].t()
            Y[c_b + isn, Q], Y[c_b + isn, U] = -im_b[:, 1:].t(), im_e[:, 1:].t()
    return Y.t()


def _lambda(cl, comps, lmin, lmax):
    """Spectrum block of every multipole, (nl, nc, nc)."""
    nc = len(comps)
    lam = np.zeros((lmax - lmin + 1, nc, nc))
    for s, (a, b) in enumerate(PAIRS):
        if a in comps and b in comps:
            i, j = comps.index(a), comps.index(b)
            lam[:, i, j] = lam[:, j, i] = cl[s, lmin:lmax + 1]
    return lam


def _per_mode(lam, lmin, lmax, dev):
    """(nl, ...) rows repeated over the 2l + 1 modes of each l."""
    rep = torch.as_tensor([2 * l + 1 for l in range(lmin, lmax + 1)], device=dev)
    return torch.repeat_interleave(torch.as_tensor(lam, dtype=F64, device=dev), rep, dim=0)


def _comps(fields):
    return {"T": (0,), "QU": (1, 2), "TQU": (0, 1, 2)}[fields]


def _geometry(case, cut):
    nside = case["nside"]
    theta, phi, z = synth.healpix_ring_centres(nside)
    keep = synth.galactic_cut(z, cut)
    return (torch.as_tensor(theta[keep], dtype=F64, device=DEV),
            torch.as_tensor(phi[keep], dtype=F64, device=DEV))


def _mask(case, cut, seed, cl, want_maps):
    """Geometry, transfer, noise covariance and (from the model) maps of one mask."""
    fields, lsig = case["fields"], case.get("lsig") or case["lmax"]
    theta, phi = _geometry(case, cut)
    nf = len(_comps(fields))
    n = nf * theta.numel()
    tr = torch.as_tensor(synth.transfer(lsig, case["nside"]), dtype=F64, device=DEV)
    g = _gen(seed)
    G = torch.randn((n, case["rank"]), generator=g, dtype=F64, device=DEV) / math.sqrt(case["rank"])
    N = G @ G.t()
    N.diagonal().add_(1.0)
    out = {"theta": theta, "phi": phi, "transfer": tr, "N": N, "n": n}
    if want_maps:
        # d = Y a + noise, a ~ N(0, Lambda) at the fiducial spectra, noise ~ N(0, N)
        nm = case["maps"]
        comps = _comps(fields)
        lam = _lambda(cl, comps, 2, lsig)
        w, v = np.linalg.eigh(lam)
        root = _per_mode(v * np.sqrt(np.clip(w, 0.0, None))[:, None, :], 2, lsig, DEV)
        z = torch.randn((root.shape[0], nf, nm), generator=g, dtype=F64, device=DEV)
        a = (root @ z).transpose(0, 1).reshape(nf * root.shape[0], nm)
        Y = _harmonics(theta, phi, 2, lsig, fields, synth.transfer(lsig, case["nside"]))
        d = Y @ a
        d += torch.randn((n, nm), generator=g, dtype=F64, device=DEV)
        d += G @ torch.randn((case["rank"], nm), generator=g, dtype=F64, device=DEV)
        out["maps"] = d.t().contiguous().t()  # column-major, as the library takes it
    return out


def _spectra(lmax, seed):
    r = np.random.default_rng(seed)
    return synth.spectra(lmax, tau=r.uniform(0.04, 0.08), r=r.uniform(0.0, 0.05),
                         a_ee=r.uniform(0.9, 1.1), a_tt=r.uniform(0.9, 1.1))


def _edges(case):
    dl, lmax = case.get("dl") or 0, case["lmax"]
    if not dl:
        return None
    e = list(range(2, lmax + 1, dl)) + [lmax + 1]
    return e


def _problem(case, mk, cl):
    f = case["fields"]
    kw = {}
    if "T" in f:
        kw |= {"theta_T": mk["theta"], "phi_T": mk["phi"], "transfer_T": mk["transfer"]}
    if "QU" in f:
        kw |= {"theta_P": mk["theta"], "phi_P": mk["phi"], "transfer_P": mk["transfer"]}
    return api.Problem(2, case["lmax"], spec=SPECS[f],
                       cl_fid=torch.as_tensor(cl.reshape(-1), dtype=F64, device=DEV), N=mk["N"],
                       precision=case["precision"], bin_edges=_edges(case),
                       lsig=(2, case["lsig"]) if case.get("lsig") else None,
                       basis=case.get("basis", 0), **kw)


def _scan_spectra(case, seed):
    r = np.random.default_rng(seed + 17)
    return np.stack([synth.spectra(case["lmax"], tau=r.uniform(0.03, 0.09), r=r.uniform(0.0, 0.1))
                     for _ in range(case["items"])])


def _item_mask(case):
    nm = len(case["cuts"].split(","))
    return np.arange(case["items"]) % nm


def _labels(case, seed):
    """Training points and labels: a likelihood-like ridge with curvature and a product term."""
    r = np.random.default_rng(seed)
    d, n = case["dim"], case["labels"]
    th = r.uniform(-1.0, 1.0, size=(n, d))
    curv = 30.0 / (1.0 + np.arange(d))
    y = (-0.5 * (th ** 2 * curv).sum(axis=1) + np.sin(2.0 * th[:, 0]) * th[:, -1]
         + 0.3 * np.cos(3.0 * th.sum(axis=1)))
    return th, y


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("predict", "train"):
        th, y = _labels(case, seed)
        d = case["dim"]
        th_d = torch.as_tensor(th, dtype=F64, device=DEV).t().contiguous().t()
        y_d = torch.as_tensor(y, dtype=F64, device=DEV)
        st = {"case": case, "theta": th_d, "lnl": y_d, "lo": -np.ones(d), "hi": np.ones(d),
              "seed": 1 + seed % 1000}
        if kind == "predict":
            emu = api.Emulator(st["lo"], st["hi"], width=case["width"], depth=case["depth"],
                               seed=st["seed"])
            emu.train(th_d, y_d, epochs=1, batch=64)
            st["emu"] = emu
            pts = torch.rand((d, case["points"]), generator=_gen(seed + 5), dtype=F64, device=DEV)
            st["points"] = (2.1 * pts - 1.05).t()
        return st
    if kind == "scan":
        cl0 = _spectra(case["lmax"], seed)
        masks = []
        for j, c in enumerate(case["cuts"].split(",")):
            mk = _mask(case, float(c), seed + 101 * j, cl0, True)
            masks.append((_problem(case, mk, cl0), mk["maps"]))
        return {"case": case, "masks": masks, "item_mask": _item_mask(case).astype(np.int32),
                "cl": torch.as_tensor(_scan_spectra(case, seed), dtype=F64, device=DEV)}
    cl = _spectra(case.get("lsig") or case["lmax"], seed)
    mk = _mask(case, case["cut"], seed, cl, True)
    st = {"case": case, "maps": mk["maps"], "prob": _problem(case, mk, cl)}
    if kind == "lnl":
        st["cl"] = torch.as_tensor(cl.reshape(-1), dtype=F64, device=DEV)
    if kind == "estimate":
        st["plan"] = api.fisher(st["prob"])[1]
    return st


# --------------------------------------------------------------------- run --
def run(state):
    kind = state["case"]["kind"]
    if kind == "solve":
        F, plan = api.fisher(state["prob"])
        est = plan.estimate(state["maps"])
        plan.free()
        return {"F": F, **est}
    if kind == "estimate":
        return state["plan"].estimate(state["maps"])
    if kind == "lnl":
        lnl, chi2, logdet = api.loglike(state["prob"], state["cl"], state["maps"])
        return {"lnL": lnl, "chi2": chi2, "logdet": logdet}
    if kind == "scan":
        lnl, chi2, logdet = api.loglike_batch(state["masks"], state["item_mask"], state["cl"])
        return {"lnL": lnl, "chi2": chi2, "logdet": logdet}
    if kind == "predict":
        out, flags = state["emu"].predict(state["points"])
        return {"lnL": out, "flags": flags}
    c = state["case"]
    emu = api.Emulator(state["lo"], state["hi"], width=c["width"], depth=c["depth"],
                       seed=state["seed"])
    loss = emu.train(state["theta"], state["lnl"], epochs=c["epochs"], batch=c["batch"])
    coef, sigma = emu.baseline()
    res = {"loss": np.array(loss), "head0": emu.params(0), "head1": emu.params(1), "coef": coef,
           "sigma": sigma}
    emu.free()
    return res


# -------------------------------------------------------------------- work --
def _net_macs(case):
    w = case["width"]
    return case["dim"] * w + (case["depth"] - 1) * w * w + w


def work(case):
    kind = case["kind"]
    if kind == "predict":
        n = case["points"]
        return {"bytes": n * (8 * case["dim"] + 8 + 4), "flops": 2 * 2 * n * _net_macs(case)}
    if kind == "train":
        n, e = case["labels"], case["epochs"]
        params = 2 * _net_macs(case)
        return {"bytes": n * 8 * (case["dim"] + 1) + 4 * params,
                "flops": 2 * 3 * 2 * (n - n // 8) * e * _net_macs(case)}
    if kind == "scan":
        flops = nbytes = 0
        cuts = [float(c) for c in case["cuts"].split(",")]
        for j, c in enumerate(cuts):
            n, nc, k = _dims(case["fields"], case["nside"], case["lmax"], c)
            items = len(range(j, case["items"], len(cuts)))
            # mask: factor of N, U = L^-1 Y, M = U^T U; item: factor of the inner matrix
            flops += n ** 3 // 3 + n * n * k + n * k * k + items * (k ** 3 // 3)
            nbytes += 4 * n * n + 8 * n * case["maps"] + 16 * n
        nbytes += case["items"] * 8 * (6 * (case["lmax"] + 1) + 2 * case["maps"] + 1)
        return {"bytes": nbytes, "flops": flops}
    n, nc, k = _dims(case["fields"], case["nside"], case["lmax"], case["cut"])
    ks = k if not case.get("lsig") else nc * ((case["lsig"] + 1) ** 2 - 4)
    s = case["maps"]
    if kind == "lnl":
        return {"bytes": 4 * n * n + 8 * n * (s + 2) + 8 * (2 * s + 1),
                "flops": n * n * k + n ** 3 // 3 + n * n * s}
    nl = case["lmax"] - 1
    nb = nl if not case.get("dl") else -(-nl // case["dl"])
    na = len(SPECS[case["fields"]]) * nb
    est = {"bytes": 8 * s * (n + 4 * na) + 8 * na, "flops": s * (n * n + 2 * n * k + 4 * na * na)}
    if kind == "estimate":
        # the plan's factors are read once: L (lower), X
        est["bytes"] += 4 * n * n + 8 * n * k
        return est
    pixel = n * n * ks + n ** 3 // 3 + n * n * k + n * k * k
    harm = n ** 3 // 3 + n * n * (ks - k) + n * n * k + n * k * k + 7 * k ** 3 // 3
    basis = case.get("basis", 0)
    fl = pixel if basis == 0 else harm if basis == 1 else min(pixel, harm)
    return {"bytes": 4 * n * n + 16 * n + 8 * na * na + est["bytes"], "flops": fl + est["flops"]}


# ------------------------------------------------------------------- exact --
def _covariance(Y, cl, comps, lmin, lmax, N=None):
    """Y Lambda Y^T (+ N), Lambda block-diagonal over the modes."""
    k0 = (lmax + 1) ** 2 - lmin ** 2
    lam = _per_mode(_lambda(cl, comps, lmin, lmax), lmin, lmax, Y.device)
    YL = torch.zeros_like(Y)
    for b in range(len(comps)):
        for a in range(len(comps)):
            YL[:, b * k0:(b + 1) * k0] += Y[:, a * k0:(a + 1) * k0] * lam[:, a, b][None, :]
    C = YL @ Y.t()
    C = 0.5 * (C + C.t())
    return C if N is None else C + N


def _pairs(spec, comps):
    a, b = PAIRS[spec]
    i, j = comps.index(a), comps.index(b)
    return [(i, i)] if i == j else [(i, j), (j, i)]


def _exact_solve(case, seed, with_f):
    comps, lmax = _comps(case["fields"]), case["lmax"]
    lsig = case.get("lsig") or lmax
    cl = _spectra(lsig, seed)
    mk = _mask(case, case["cut"], seed, cl, True)
    tr = synth.transfer(lsig, case["nside"])
    N = mk["N"]
    if lsig > lmax:  # the fiducial signal above the window is fixed, part of the noise
        Yo = _harmonics(mk["theta"], mk["phi"], lmax + 1, lsig, case["fields"], tr)
        N = N + _covariance(Yo, cl, comps, lmax + 1, lsig)
    Y = _harmonics(mk["theta"], mk["phi"], 2, lmax, case["fields"], tr)
    L = torch.linalg.cholesky(_covariance(Y, cl, comps, 2, lmax, N))
    X = torch.linalg.solve_triangular(L, Y, upper=False)
    W = X.t() @ X
    Z = torch.linalg.solve_triangular(L.t(), X, upper=True)
    ZNZ = Z.t() @ (N @ Z)
    w = X.t() @ torch.linalg.solve_triangular(L, mk["maps"], upper=False)
    k0, nc = (lmax + 1) ** 2 - 4, len(comps)
    edges = _edges(case) or list(range(2, lmax + 2))
    nb = len(edges) - 1
    B = torch.zeros((nb, k0), dtype=F64, device=DEV)
    for i in range(nb):
        B[i, edges[i] ** 2 - 4:edges[i + 1] ** 2 - 4] = 1.0
    spec = [synth.SPEC_INDEX[s] for s in SPECS[case["fields"]]]
    W4 = W.reshape(nc, k0, nc, k0)
    ns = len(spec)
    F = torch.zeros((ns * nb, ns * nb), dtype=F64, device=DEV)
    bias = torch.zeros(ns * nb, dtype=F64, device=DEV)
    y = torch.zeros((ns * nb, w.shape[1]), dtype=F64, device=DEV)
    seen = {}
    for a, sa in enumerate(spec):
        ra = slice(a * nb, (a + 1) * nb)
        for u, v in _pairs(sa, comps):
            bias[ra] += 0.5 * (B @ torch.diagonal(ZNZ[v * k0:(v + 1) * k0, u * k0:(u + 1) * k0]))
            y[ra] += 0.5 * (B @ (w[u * k0:(u + 1) * k0] * w[v * k0:(v + 1) * k0]))
        for b, sb in enumerate(spec):
            for u, v in _pairs(sa, comps):
                for u2, v2 in _pairs(sb, comps):
                    key = (v, u2, v2, u)
                    if key not in seen:
                        seen[key] = B @ (W4[v, :, u2, :] * W4[v2, :, u, :].t()) @ B.t()
                    F[ra, b * nb:(b + 1) * nb] += 0.5 * seen[key]
    q = y - bias[:, None]
    Fn = F.cpu().numpy()
    xi, V = np.linalg.eigh(0.5 * (Fn + Fn.T))
    keep = xi >= 1e-12 * xi.max()
    half = (V * np.where(keep, 1.0 / np.sqrt(np.where(keep, xi, 1.0)), 0.0)) @ V.T
    qn = q.cpu().numpy()
    dec = np.linalg.solve(Fn, qn)
    est = {"y": y, "cl_deconv": torch.as_tensor(dec), "cl_decorr": torch.as_tensor(half @ qn),
           "q_conv": q, "b": bias}
    return {"F": F, **est} if with_f else est


def _lnl(C, d):
    L = torch.linalg.cholesky(C)
    ld = 2.0 * torch.log(torch.diagonal(L)).sum()
    x = torch.linalg.solve_triangular(L, d, upper=False)
    chi2 = (x * x).sum(dim=0)
    return -0.5 * (chi2 + ld), chi2, ld


def _exact_flops(case):
    """Operations of the plain evaluation below (a scan's items each factor their own C)."""
    if case["kind"] != "scan":
        return 4 * work(case)["flops"]
    total, cuts = 0, [float(c) for c in case["cuts"].split(",")]
    for j, c in enumerate(cuts):
        n, nc, k = _dims(case["fields"], case["nside"], case["lmax"], c)
        total += len(range(j, case["items"], len(cuts))) * (2 * n * n * k + n ** 3 // 3)
    return total


def exact(case, seed):
    kind = case["kind"]
    if kind in ("predict", "train"):
        return None  # the weights come from the library's own training
    if _exact_flops(case) > 1.0e13:
        return None  # over twenty seconds in plain float64
    comps, lmax = _comps(case["fields"]), case["lmax"]
    if kind == "solve":
        return _exact_solve(case, seed, True)
    if kind == "estimate":
        return _exact_solve(case, seed, False)
    tr = synth.transfer(lmax, case["nside"])
    if kind == "lnl":
        cl = _spectra(lmax, seed)
        mk = _mask(case, case["cut"], seed, cl, True)
        Y = _harmonics(mk["theta"], mk["phi"], 2, lmax, case["fields"], tr)
        lnl, chi2, ld = _lnl(_covariance(Y, cl, comps, 2, lmax, mk["N"]), mk["maps"])
        return {"lnL": lnl, "chi2": chi2, "logdet": ld}
    cl0, cls = _spectra(lmax, seed), _scan_spectra(case, seed)
    im, nm = _item_mask(case), case["maps"]
    lnl = torch.zeros((case["items"], nm), dtype=F64)
    chi2, ld = torch.zeros_like(lnl), torch.zeros(case["items"], dtype=F64)
    for j, c in enumerate(case["cuts"].split(",")):
        mk = _mask(case, float(c), seed + 101 * j, cl0, True)
        Y = _harmonics(mk["theta"], mk["phi"], 2, lmax, case["fields"], tr)
        for i in np.nonzero(im == j)[0]:
            a, b, e = _lnl(_covariance(Y, cls[i], comps, 2, lmax, mk["N"]), mk["maps"])
            lnl[i], chi2[i], ld[i] = a.cpu(), b.cpu(), e.cpu()
    return {"lnL": lnl, "chi2": chi2, "logdet": ld}
