"""The work whose speed is measured: what a user of libchi0 has it do.

Each case is one pass through the public entry points (paper_1902_03837_gb300.chi0)
on seeded synthetic crystals of the kinds that the tests and the benchmark use:
cubic cells, Gamma-centred k grids, k-centred plane-wave spheres, orthonormal
time-reversal-symmetric states.  Coefficients, plans and output buffers are in
place before the pass, as in a program that goes over q points, frequencies or
new coefficients on one geometry.

FP64 results come back as the library writes them.  The mixed form is good to
about 1e-6, so its complex128 buffers are handed on in single precision, as a
program that stores them would do.
"""
import functools
import math

import numpy as np
import torch

from paper_1902_03837_gb300 import chi0 as lib

HA_EV = 27.211386245988
ETA = 0.1 / HA_EV

# Cost (rough operations) up to which exact() is evaluated: some ten seconds of FP64
EXACT_MAX = 6e12


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _response(name, form, k, nocc, nb, a, r, fft, ng, nw, axis="imag", metal=False, bg=0.0, q=(1, 0, 0)):
    """rho, chi0 and eps~^-1 of one q point.  form: fp64 or mixed; r: sphere
    radius in units of 2 pi / a; axis: imag (i w on [0, 100] eV), static
    (w = 0 with eta) or real (w on (0, 40] eV with eta); metal: Fermi-Dirac
    occupations at 0.05 eV for 2 nocc electrons; bg: extrapolar energy (eV)
    of the Bruneval-Gonze correction, 0 for none."""
    return {"name": name, "kind": "response", "form": form, "k1": k[0], "k2": k[1], "k3": k[2], "nocc": nocc,
            "nb": nb, "a": a, "r": r, "f1": fft[0], "f2": fft[1], "f3": fft[2], "ng": ng, "nw": nw, "axis": axis,
            "metal": metal, "bg": bg, "q1": q[0], "q2": q[1], "q3": q[2]}


def listed():
    return [
        # a smoke-test-sized crystal: launches and host set-up count
        _response("tiny-fp64", "fp64", (2, 2, 2), 3, 8, 6.0, 1.93, (16, 16, 16), 9, 2),
        # the plain FP64 workload of the repository: one q point, static screening
        _response("plain-fp64", "fp64", (4, 4, 4), 8, 32, 10.0, 4.1458, (24, 24, 24), 59, 1, axis="static"),
        # a metal in the FP64 form, ragged sizes, a grid without factors of four
        _response("metal-fp64-odd", "fp64", (4, 3, 2), 10, 28, 9.0, 3.4, (21, 25, 18), 137, 3, metal=True,
                  q=(1, 1, 0)),
        # the precision workload (16 + 184 bands, about 2000 plane waves, N_G = 1000, 32
        # frequencies) on a 6x6x6 grid, so that several problems fit the card
        _response("precision-mixed", "mixed", (6, 6, 6), 16, 200, 10.0, 7.8184, (48, 48, 48), 1000, 32),
        # one problem of the batching workload, taken by itself: a metal with few transitions per G
        _response("metal-mixed", "mixed", (4, 4, 4), 16, 64, 11.0, 6.6, (30, 30, 30), 431, 16, metal=True,
                  q=(0, 1, 0)),
        # eps~^-1 on the real axis, as full-frequency GW wants it
        _response("real-axis-mixed", "mixed", (4, 4, 4), 16, 100, 10.0, 6.0, (40, 40, 40), 400, 24, axis="real"),
        # the paper's band-sum correction
        _response("extrapolar-mixed", "mixed", (4, 4, 4), 12, 80, 10.0, 5.2, (36, 36, 36), 220, 16, bg=40.0,
                  q=(0, 0, 1)),
        # several metals at several q points in one captured batch
        {"name": "batch-mixed", "kind": "batch", "form": "mixed", "nsys": 3, "nq": 3, "kn": 4, "nocc": 12, "nb": 40,
         "a": 10.0, "r": 5.3, "over": 1.5, "ng": 330, "nw": 12, "nstreams": 4},
        # plasmon-pole model and self-energy kernel of a window of four bands
        {"name": "ppa-sigma-mixed", "kind": "gw", "form": "mixed", "k1": 4, "k2": 4, "k3": 4, "nocc": 12, "nb": 64,
         "a": 10.0, "r": 4.6, "f1": 30, "f2": 30, "f3": 30, "ng": 300, "nf": 48, "nqp": 4},
        # the Dyson step alone on chi0 that the caller holds
        {"name": "dyson-fp64", "kind": "dyson", "ng": 300, "nw": 12},
        # one training step of the learned terminator at its minibatch
        {"name": "terminator-train", "kind": "train", "batch": 4096, "bf16": True},
        # its prediction for every entry of chi0 at N_G = 250 and 16 frequencies
        {"name": "terminator-predict", "kind": "predict", "rows": 1000000, "bf16": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fft_size(rng, r, ng):
    """From the smallest alias-free grid to the grid that holds the density."""
    lo = 2 * int(r + 1) + int((3.0 * ng / (4.0 * math.pi)) ** (1.0 / 3.0) + 1.5) + 3
    return rng.randint(lo, max(lo, 4 * int(r + 1) + 1))


def _draw_response(rng):
    form = rng.choice(["fp64", "mixed", "mixed"])
    axis = rng.choice(["imag", "imag", "imag", "static" if form == "fp64" else "real"])
    metal = axis != "real" and rng.random() < 0.4
    k = tuple(rng.randint(2, 4) for _ in range(3))
    if form == "fp64":
        ng, nw, r = _log_int(rng, 9, 160), 1 if axis == "static" else rng.randint(1, 4), rng.uniform(2.4, 4.2)
        nocc = rng.randint(3, 10)
        nb = nocc + rng.randint(4, 24)
    else:
        ng, nw, r = _log_int(rng, 60, 900), _log_int(rng, 4, 32), rng.uniform(3.5, 7.5)
        nocc = rng.randint(4, 16)
        nb = nocc + _log_int(rng, 16, 120)
    bg = 40.0 if form == "mixed" and axis == "imag" and not metal and ng <= 300 and rng.random() < 0.3 else 0.0
    fft = [_fft_size(rng, r, ng) for _ in range(3)]
    if bg:  # alias free for the difference set G - G' too
        h = int((3.0 * ng / (4.0 * math.pi)) ** (1.0 / 3.0) + 1.5) + 1
        fft = [max(f, 2 * int(r + 1) + 2 * h + 1) for f in fft]
    axis_q = rng.randrange(3)
    q = [rng.randint(1, k[d] - 1) if d == axis_q or rng.random() < 0.3 else 0 for d in range(3)]
    return _response("", form, k, nocc, nb, round(rng.uniform(8.0, 14.0), 2), round(r, 4), fft, ng, nw, axis, metal,
                     bg, q)


def draw(rng):
    kind = rng.choice(["response"] * 6 + ["batch", "gw", "dyson", "dyson", "train", "predict"])
    if kind == "response":
        case = _draw_response(rng)
        del case["name"]
        return case
    if kind == "batch":
        return {"kind": "batch", "form": "mixed", "nsys": rng.randint(1, 4), "nq": rng.randint(1, 3),
                "kn": rng.randint(2, 4), "nocc": rng.randint(6, 14), "nb": rng.randint(28, 48),
                "a": round(rng.uniform(8.0, 14.0), 2), "r": round(rng.uniform(4.0, 6.0), 4),
                "over": round(rng.uniform(1.0, 1.6), 2), "ng": _log_int(rng, 100, 450), "nw": rng.randint(4, 16),
                "nstreams": rng.randint(1, 4)}
    if kind == "gw":
        r, ng = round(rng.uniform(3.5, 5.5), 4), _log_int(rng, 80, 400)
        f = [_fft_size(rng, r, ng) for _ in range(3)]
        return {"kind": "gw", "form": rng.choice(["mixed", "mixed", "fp64"] if ng < 200 else ["mixed"]),
                "k1": rng.randint(2, 4), "k2": rng.randint(2, 4), "k3": rng.randint(2, 4), "nocc": rng.randint(6, 12),
                "nb": rng.randint(24, 64), "a": round(rng.uniform(8.0, 14.0), 2), "r": r, "f1": f[0], "f2": f[1],
                "f3": f[2], "ng": ng, "nf": rng.randint(6, 48), "nqp": rng.randint(2, 8)}
    if kind == "dyson":
        ng = _log_int(rng, 20, 900)
        return {"kind": "dyson", "ng": ng, "nw": max(1, min(32, _log_int(rng, 1, 32), int(2e9 / ng ** 3)))}
    if kind == "train":
        return {"kind": "train", "batch": _log_int(rng, 200, 16384), "bf16": rng.random() < 0.7}
    return {"kind": "predict", "rows": _log_int(rng, 5000, 2000000), "bf16": rng.random() < 0.7}


# ---------------------------------------------------------------------------
# synthetic crystals
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=8)
def _geometry(k1, k2, k3, r):
    """Spheres |k + G| < r of every k, and the time-reversal partner of each k
    with the places of the partner's plane waves: c_k'(G) = conj c_k(-G - G1)."""
    kg = np.array([k1, k2, k3])
    kint = np.stack(np.meshgrid(np.arange(k1), np.arange(k2), np.arange(k3), indexing="ij"), -1).reshape(-1, 3)
    m = int(r) + 2
    box = np.stack(np.meshgrid(*[np.arange(-m, m + 1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    spheres = [box[((box + ki / kg) ** 2).sum(1) < r * r] for ki in kint]
    npw = np.array([len(s) for s in spheres])
    gvec = np.zeros((len(kint), npw.max(), 3), np.int32)
    for i, s in enumerate(spheres):
        gvec[i, : len(s)] = s
    pint = (-kint) % kg
    partner = (pint[:, 0] * k2 + pint[:, 1]) * k3 + pint[:, 2]
    side = 2 * m + 3
    code = lambda g: ((g[:, 0] + m + 1) * side + g[:, 1] + m + 1) * side + g[:, 2] + m + 1  # noqa: E731
    place = np.zeros((len(kint), npw.max()), np.int64)  # of partner[i]'s plane waves in k's sphere
    for i, s in enumerate(spheres):
        g1 = (kint[i] + pint[i]) // kg
        c = code(s)
        order = np.argsort(c)
        t = spheres[partner[i]]
        place[i, : len(t)] = order[np.searchsorted(c[order], code(-t - g1))]
    return npw, gvec, partner, place


def _coefficients(k, r, nb, dtype, seed):
    """[nk][nb][npw_max]: Gaussian draws, orthonormalised at each k (Cholesky
    factor of the overlap), partners by conjugation, self-partners in the
    coordinates in which time reversal holds."""
    npw, gvec, partner, place = _geometry(*k, r)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nk = len(npw)
    reps = np.nonzero(partner >= np.arange(nk))[0]
    n = torch.from_numpy(npw).cuda()
    pl = torch.from_numpy(place).cuda()
    mask = torch.arange(gvec.shape[1], device="cuda")[None] < n[:, None]
    c = torch.randn(len(reps), nb, gvec.shape[1], dtype=dtype, device="cuda", generator=gen)
    c *= mask[reps][:, None]
    own = [i for i, ik in enumerate(reps) if partner[ik] == ik]
    for i in own:
        p = pl[reps[i]]
        c[i] = (c[i] + c[i][:, p].conj()) * mask[reps[i]]
    low = torch.linalg.cholesky(c @ c.mH)
    c = torch.linalg.solve_triangular(low, c, upper=False)
    out = torch.empty(nk, nb, gvec.shape[1], dtype=dtype, device="cuda")
    out[reps] = c
    for i, ik in enumerate(reps):
        if partner[ik] != ik:
            out[partner[ik]] = c[i][:, pl[ik]].conj() * mask[partner[ik]]
    return npw, gvec, out


def _energies(case_k, nocc, nb, metal, seed):
    """Energies (Ha) and occupations, equal at k and -k."""
    partner = _geometry_partner(*case_k)
    rng = np.random.default_rng(seed)
    nk = len(partner)
    if metal:
        e = np.sort(rng.uniform(-10.0, 30.0, (nk, nb)), 1)
    else:
        e = np.concatenate([np.sort(rng.uniform(-10.0, 0.0, (nk, nocc)), 1),
                            np.sort(rng.uniform(1.1, 30.0, (nk, nb - nocc)), 1)], 1)
    e = e[np.minimum(partner, np.arange(nk))] / HA_EV
    if not metal:
        return e, np.broadcast_to((np.arange(nb) < nocc).astype(float), (nk, nb)).copy()
    kt = 0.05 / HA_EV
    fermi = lambda mu: 1.0 / (np.exp(np.clip((e - mu) / kt, -700, 700)) + 1.0)  # noqa: E731
    lo, hi = e.min() - 1.0, e.max() + 1.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if fermi(mid).sum() / nk < nocc else (lo, mid)
    return e, fermi(0.5 * (lo + hi))


def _geometry_partner(k1, k2, k3):
    kint = np.stack(np.meshgrid(np.arange(k1), np.arange(k2), np.arange(k3), indexing="ij"), -1).reshape(-1, 3)
    p = (-kint) % np.array([k1, k2, k3])
    return (p[:, 0] * k2 + p[:, 1]) * k3 + p[:, 2]


def _frequencies(axis, nw):
    if axis == "static":
        return np.zeros(1, complex)
    if axis == "real":
        return np.linspace(40.0 / nw, 40.0, nw) / HA_EV + 0j
    x, _ = np.polynomial.legendre.leggauss(nw)
    return 1j * (50.0 * x + 50.0) / HA_EV


def _system(case, seed, dtype, omega, eta, q_frac):
    """A context with its states and energies set, and the arrays behind it."""
    k = (case["k1"], case["k2"], case["k3"])
    npw, gvec, coef = _coefficients(k, case["r"], case["nb"], dtype, seed)
    eps, occ = _energies(k, case["nocc"], case["nb"], case["metal"], seed)
    ctx = lib.Chi0(a=case["a"], kgrid=k, nbands=case["nb"], npw_max=int(npw.max()),
                   fft=(case["f1"], case["f2"], case["f3"]), ng=case["ng"], q_frac=q_frac, omega=omega, eta=eta,
                   precision=lib.CHI0_FP64 if case["form"] == "fp64" else lib.CHI0_MIXED_BF16X3,
                   occ_drop_tol=1e-12, stream=torch.cuda.current_stream().cuda_stream)
    gdev = torch.from_numpy(gvec).cuda()
    for ik, n in enumerate(npw):
        ctx.set_wavefunctions(ik, gdev[ik, :n].contiguous(), coef[ik, :, :n].contiguous())
    ctx.set_energies(eps, occ)
    ctx.synchronize()
    return ctx


def _dtype(case):
    return torch.complex128 if case["form"] == "fp64" else torch.complex64


def _batch_parts(case):
    """The systems of a batch: cells, spheres, response sets and frequency
    counts that differ from system to system, nq q points each."""
    kn = case["kn"]
    grid = [(i, j, l) for i in range(kn) for j in range(kn) for l in range(kn) if i + j + l]
    for s in range(case["nsys"]):
        r = case["r"] * (1.0 - 0.09 * s)
        ng = max(20, int(case["ng"] * (1.0 - 0.23 * s)))
        lo = 2 * int(r + 1) + int((3.0 * ng / (4.0 * math.pi)) ** (1.0 / 3.0) + 1.5) + 3
        f = max(lo, int(case["over"] * lo))
        yield {"form": case["form"], "k1": kn, "k2": kn, "k3": kn, "nocc": case["nocc"], "nb": case["nb"],
               "a": case["a"] + 0.7 * s, "r": r, "f1": f, "f2": f, "f3": f, "ng": ng,
               "nw": max(2, case["nw"] - 3 * s), "metal": True,
               "qs": [grid[(5 * s + 3 * j) % len(grid)] for j in range(min(case["nq"], len(grid)))]}


# ---------------------------------------------------------------------------
# preparation and the pass
# ---------------------------------------------------------------------------

def _q_frac(case):
    return [(case["q1"] / case["k1"], case["q2"] / case["k2"], case["q3"] / case["k3"])]


def _screening(ng, nw, seed):
    """chi0 of nw imaginary frequencies (Hermitian, negative semidefinite, of
    the size an insulator has) and the Coulomb factors of its G set."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    m = int((3.0 * ng / (4.0 * math.pi)) ** (1.0 / 3.0)) + 3
    g = np.stack(np.meshgrid(*[np.arange(-m, m + 1)] * 3, indexing="ij"), -1).reshape(-1, 3) + [0.25, 0.0, 0.0]
    qg = np.sort(np.sqrt((g ** 2).sum(1)))[:ng] * (2.0 * math.pi / 10.0)
    v = np.sqrt(4.0 * math.pi) / qg
    size = torch.from_numpy(qg / (1.0 + qg * qg)).cuda()
    b = torch.randn(ng, 2 * ng, dtype=torch.complex128, device="cuda", generator=gen) * size[:, None]
    d = torch.rand(2 * ng, dtype=torch.float64, device="cuda", generator=gen) + 0.1
    nu = torch.from_numpy(_frequencies("imag", nw).imag.copy()).cuda()
    w = 2.0 * d[None] / (d[None] ** 2 + nu[:, None] ** 2) * (0.02 / ng)
    chi = torch.stack([-((b * wi) @ b.mH) for wi in w])
    return 0.5 * (chi + chi.mH).contiguous(), v


def _model_screening(ng, seed):
    """eps~^-1 at w = 0 and at i (1 Ha) of such a chi0."""
    chi, v = _screening(ng, 2, seed)
    vd = torch.from_numpy(v).cuda()
    chi = torch.stack([chi[0], 0.5 * chi[0] + 0.3 * chi[1]])
    e = torch.eye(ng, dtype=torch.complex128, device="cuda") - vd[:, None] * chi * vd[None, :]
    return torch.linalg.inv(e).contiguous()


def _network(seed, rows):
    """Parameters as training starts from, and features and targets as the
    truncated chi0 gives them."""
    rng = np.random.default_rng(seed)
    i, h, o = 5, 128, 2
    parts = [rng.uniform(-1, 1, (h, i)) / math.sqrt(i), 0.1 * rng.standard_normal(h),
             rng.uniform(-1, 1, (h, h)) / math.sqrt(h), 0.1 * rng.standard_normal(h),
             rng.uniform(-1, 1, (o, h)) / math.sqrt(h), 0.1 * rng.standard_normal(o)]
    p = torch.from_numpy(np.concatenate([a.ravel() for a in parts]).astype(np.float32)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand(rows, 5, device="cuda", generator=gen)
    x[:, 3:] = 0.1 * torch.randn(rows, 2, device="cuda", generator=gen)
    t = 0.3 * torch.randn(rows, 2, device="cuda", generator=gen)
    return p, x.contiguous(), t


def prepare(case, seed):
    kind = case["kind"]
    out = functools.partial(torch.empty, dtype=torch.complex128, device="cuda")
    if kind == "response":
        omega = _frequencies(case["axis"], case["nw"])
        ctx = _system(case, seed, _dtype(case), omega, 0.0 if case["axis"] == "imag" else ETA, _q_frac(case))
        if case["bg"]:
            ctx.set_bg_terminator(case["bg"] / HA_EV)
        n = (len(omega), case["ng"], case["ng"])
        return {"case": case, "ctx": ctx, "chi": out(n), "eps": out(n)}
    if kind == "batch":
        ctxs, iqs, chis, epss = [], [], [], []
        for s, part in enumerate(_batch_parts(case)):
            qs = [tuple(v / case["kn"] for v in q) for q in part["qs"]]
            ctx = _system(part, seed + 1000 * s, _dtype(case), _frequencies("imag", part["nw"]), 0.0, qs)
            for iq in range(len(qs)):
                ctxs.append(ctx)
                iqs.append(iq)
                chis.append(out((part["nw"], part["ng"], part["ng"])))
                epss.append(out((part["nw"], part["ng"], part["ng"])))
        batch = lib.Batch(ctxs, iqs, eps_out=epss, nstreams=case["nstreams"], chi_out=chis)
        return {"case": case, "batch": batch, "chi": chis, "eps": epss}
    if kind == "gw":
        ctx = _system(dict(case, metal=False), seed, _dtype(case), [0j], ETA, [(1.0 / case["k1"], 0.0, 0.0)])
        ctx.compute_rho(0)
        ctx.synchronize()
        ng, nk = case["ng"], ctx.nk
        return {"case": case, "ctx": ctx, "e": _model_screening(ng, seed), "wt": out((ng, ng)), "R": out((ng, ng)),
                "model": out((case["nf"], ng, ng)), "freqs": _frequencies("real", case["nf"]),
                "I": out((case["nf"], nk, case["nb"], case["nqp"], case["nqp"]))}
    if kind == "dyson":
        chi, v = _screening(case["ng"], case["nw"], seed)
        return {"case": case, "chi": chi, "v": v, "out": torch.empty_like(chi)}
    if kind == "train":
        p, x, t = _network(seed, case["batch"])
        z = torch.zeros_like
        return {"case": case, "p": p, "x": x, "t": t, "g": z(p), "m": z(p), "v": z(p), "step": 0,
                "loss": torch.zeros(1, device="cuda"),
                "work": torch.empty(lib.mlp_workspace_floats(case["batch"]), device="cuda")}
    p, x, _ = _network(seed, case["rows"])
    return {"case": case, "p": p, "x": x, "y": torch.empty(case["rows"], 2, device="cuda")}


def _given(case, *tensors):
    """Results as the program keeps them (mixed form: single precision)."""
    return [t if case["form"] == "fp64" else t.to(torch.complex64) for t in tensors]


def run(state):
    case = state["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "response":
        ctx = state["ctx"]
        ctx.compute_rho(0)
        ctx.build_invert(0, state["eps"], state["chi"])
        return _given(case, state["chi"], state["eps"])
    if kind == "batch":
        state["batch"].run(stream)
        return _given(case, *state["chi"], *state["eps"])
    if kind == "gw":
        e = state["e"]
        lib.ppa_fit(e[0], e[1], 1.0, state["wt"], state["R"], stream=stream)
        lib.ppa_eval(state["wt"], state["R"], state["freqs"], ETA, state["model"], stream=stream)
        lo = case["nocc"] - case["nqp"] // 2
        state["ctx"].build_sigma_i(0, lo, lo + case["nqp"], state["model"], state["I"])
        return [state["wt"], state["R"], state["model"]] + _given(case, state["I"])
    if kind == "dyson":
        return lib.invert_eps_noalloc(state["chi"], state["v"], state["out"], stream=stream)
    if kind == "train":
        state["step"] += 1
        lib.mlp_loss_grad(state["p"], state["x"], state["t"], state["g"], state["loss"], state["work"],
                          bf16=case["bf16"], stream=stream)
        lib.mlp_adam(state["p"], state["g"], state["m"], state["v"], 2e-3, state["step"], stream=stream)
        return {k: state[k] for k in ("loss", "g", "p", "m", "v")}
    lib.mlp_predict(state["p"], state["x"], state["y"], bf16=case["bf16"], stream=stream)
    return state["y"]


# ---------------------------------------------------------------------------
# work of one pass
# ---------------------------------------------------------------------------

def _transitions(case, seed=0):
    """(weighted transitions, states) of a response case; 0/1 occupations or
    about as many pairs as a metal of 2 nocc electrons has."""
    nk = case["k1"] * case["k2"] * case["k3"]
    return nk * case["nocc"] * ((case["nb"] if case.get("bg") else case["nb"] - case["nocc"])), nk * case["nb"]


def _smallest_grid(case):
    """Points of the smallest alias-free real-space grid of rho."""
    n = 2 * int(case["r"]) + int((3.0 * case["ng"] / (4.0 * math.pi)) ** (1.0 / 3.0)) + 2
    return n ** 3


def _rho_flops(case, nt, states):
    """Transforms of the states, products and transforms of the pairs."""
    n = _smallest_grid(case)
    return (nt + states) * 5.0 * n * math.log2(n) + 6.0 * n * nt


def _response_work(case, ng, nw):
    nt, states = _transitions(case)
    c = 16 if case["form"] == "fp64" else 8
    npw = 4.0 / 3.0 * math.pi * case["r"] ** 3
    # a real frequency's chi0 has no symmetry: every entry, and a general inverse
    half = 1.0 if case.get("axis") == "real" else 0.5
    flops = _rho_flops(case, nt, states) + 8.0 * half * ng * (ng + 1) * nt * nw + 8.0 * half * ng ** 3 * nw
    return {"bytes": states * npw * c + 2 * 16.0 * ng * ng * nw, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "response":
        return _response_work(case, case["ng"], case["nw"])
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for part in _batch_parts(case):
            one = _response_work(part, part["ng"], part["nw"])
            total = {k: total[k] + one[k] * len(part["qs"]) for k in total}
        return total
    if kind == "gw":
        ng, nf, nqp = case["ng"], case["nf"], case["nqp"]
        states = case["k1"] * case["k2"] * case["k3"] * case["nb"]
        nt = states * nqp
        # W^delta is Hermitian, so I is Hermitian in (a, b)
        flops = _rho_flops(case, nt, states) + nf * (20.0 * ng * ng + 8.0 * ng * ng * nt + 4.0 * ng * nt * nqp)
        return {"bytes": 16.0 * (ng * ng * (4 + nf) + nf * nt * nqp), "flops": flops}
    if kind == "dyson":
        n = float(case["ng"])
        return {"bytes": 32.0 * n * n * case["nw"], "flops": 4.0 * n ** 3 * case["nw"]}
    if kind == "train":
        macs = 5 * 128 + 128 * 128 + 128 * 2
        return {"bytes": 28.0 * case["batch"] + 4 * 8.0 * 17538, "flops": 6.0 * macs * case["batch"]}
    return {"bytes": 28.0 * case["rows"] + 4 * 17538.0, "flops": 2.0 * 17280 * case["rows"]}


# ---------------------------------------------------------------------------
# the same results in 64 bits, by plain transforms and products
# ---------------------------------------------------------------------------

def _response_set(k, q, ng):
    """The ng vectors of smallest |q + G|, ties by (x, y, z), exactly."""
    scale = math.lcm(*k)
    lq = np.array([q[d] * (scale // k[d]) for d in range(3)])
    m = int((3.0 * ng / (4.0 * math.pi)) ** (1.0 / 3.0)) + 3
    g = np.stack(np.meshgrid(*[np.arange(-m, m + 1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    n2 = ((lq + scale * g) ** 2).sum(1)
    return g[np.lexsort((g[:, 2], g[:, 1], g[:, 0], n2))[:ng]]


class _Exact:
    """rho in 64 bits: products of the states on an alias-free grid and their
    transforms, one k point at a time."""

    def __init__(self, case, seed, q):
        self.k = (case["k1"], case["k2"], case["k3"])
        self.npw, self.gvec, coef = _coefficients(self.k, case["r"], case["nb"], _dtype(case), seed)
        self.coef = coef.to(torch.complex128)
        self.eps, self.occ = _energies(self.k, case["nocc"], case["nb"], case["metal"], seed)
        self.G = _response_set(self.k, q, case["ng"])
        self.q, self.nk = q, len(self.npw)
        spread = int((self.G.max(0) - self.G.min(0)).max())
        self.n = 2 * int(np.abs(self.gvec).max()) + max(spread, int(np.abs(self.G).max()) + 1) + 1
        self.pref = 2.0 / (self.nk * case["a"] ** 3)

    def pair(self, ik):
        """k - q = k' + G0."""
        i, rest = divmod(ik, self.k[1] * self.k[2])
        j, l = divmod(rest, self.k[2])
        src = np.array([i, j, l]) - np.array(self.q)
        kk = np.array(self.k)
        rep = src % kk
        return int((rep[0] * kk[1] + rep[1]) * kk[2] + rep[2]), (src - rep) // kk

    def states(self, ik, lo, hi):
        n, N = self.npw[ik], self.n
        g = torch.from_numpy(self.gvec[ik, :n].astype(np.int64) % N).cuda()
        box = torch.zeros(hi - lo, N, N, N, dtype=torch.complex128, device="cuda")
        box[:, g[:, 0], g[:, 1], g[:, 2]] = self.coef[ik, lo:hi, :n]
        return torch.fft.ifftn(box, dim=(1, 2, 3)) * N ** 3

    def gather(self, f, h):
        t = torch.fft.ifftn(f, dim=(-3, -2, -1))
        h = torch.from_numpy(h % self.n).cuda()
        return t[..., h[:, 0], h[:, 1], h[:, 2]]

    def rho(self, ik, n0, n1, m0, m1):
        """[n][m][G] of k point ik."""
        kp, g0 = self.pair(ik)
        un, um = self.states(ik, n0, n1), self.states(kp, m0, m1)
        step = max(1, int(4e8 / (16 * (m1 - m0) * self.n ** 3)))
        return torch.cat([self.gather(un[s:s + step, None].conj() * um[None], self.G - g0)
                          for s in range(0, n1 - n0, step)])


def _factor(w, eta, d):
    """Two-pole frequency factor of pole energies d."""
    if w.real == 0.0:
        return (2.0 * d / (d * d + (w.imag + eta) ** 2)).to(torch.complex128)
    z = w + 1j * eta
    return 1.0 / (z + d) - 1.0 / (z - d)


def _exact_cost(case, ng, nw):
    nt, states = _transitions(case)
    if case["metal"]:
        nt *= 2
    n = (2 * int(case["r"] + 1) + 2 * int((3.0 * ng / (4.0 * math.pi)) ** (1.0 / 3.0) + 1.5)) ** 3
    return (nt + states) * n * 5.0 * math.log2(n) + 8.0 * ng * ng * nt * nw + 30.0 * ng ** 3 * nw


def _exact_response(case, seed, q, omega, eta):
    x = _Exact(case, seed, q)
    ng = case["ng"]
    occ, eps = torch.from_numpy(x.occ).cuda(), torch.from_numpy(x.eps).cuda()
    mmax = int(np.nonzero((x.occ > 1e-12).any(0))[0].max()) + 1
    ebar = case.get("bg", 0.0) / HA_EV
    chi = torch.zeros(len(omega), ng, ng, dtype=torch.complex128, device="cuda")
    diff = None
    if ebar:
        dv = (x.G[:, None] - x.G[None]).reshape(-1, 3)
        diff, where = np.unique(dv, axis=0, return_inverse=True)
        where = torch.from_numpy(where.reshape(-1)).cuda()
        P = torch.zeros(len(omega), len(diff), dtype=torch.complex128, device="cuda")
    for ik in range(x.nk):
        kp, _ = x.pair(ik)
        df = occ[kp][None, :mmax] - occ[ik][:, None]
        d = eps[kp][None, :mmax] - eps[ik][:, None]
        keep = df > 1e-12
        if ebar:
            keep = torch.ones_like(keep)
        used = torch.nonzero(keep.any(1)).flatten()
        if not len(used):
            continue
        n0 = int(used.min())
        R = x.rho(ik, n0, case["nb"], 0, mmax)[keep[n0:]]
        for iw, w in enumerate(omega):
            f = x.pref * torch.where(df > 1e-12, df * _factor(w, eta, d), 0.0)
            if ebar:
                f = f - x.pref * (occ[kp][:mmax] * _factor(w, eta, eps[kp][:mmax] - ebar))[None]
            chi[iw] += (R * f[n0:][keep[n0:]][:, None]).T @ R.conj()
        if ebar:
            u = x.states(ik, 0, mmax)
            dens = torch.cat([x.gather((u[m:m + 1].abs() ** 2).to(torch.complex128), diff) for m in range(mmax)])
            for iw, w in enumerate(omega):
                P[iw] += ((x.pref * occ[ik][:mmax] * _factor(w, eta, eps[ik][:mmax] - ebar))[:, None] * dens).sum(0)
    if ebar:
        chi += P[:, where].reshape(chi.shape)
    qg = np.sqrt((((x.G + np.array(q) / np.array(x.k)) * (2.0 * math.pi / case["a"])) ** 2).sum(1))
    v = torch.from_numpy(np.sqrt(4.0 * math.pi) / qg).cuda()
    return chi, torch.linalg.inv(torch.eye(ng, dtype=torch.complex128, device="cuda") - v[:, None] * chi * v[None])


def _exact_gw(case, seed):
    ng, nqp, nf = case["ng"], case["nqp"], case["nf"]
    x = _Exact(dict(case, metal=False), seed, (1, 0, 0))
    e = _model_screening(ng, seed)
    eye = torch.eye(ng, dtype=torch.complex128, device="cuda")
    x0, xp = e[0] - eye, e[1] - eye
    w2 = xp / (x0 - xp)
    pole = w2.real > 0
    wt = torch.where(pole, torch.sqrt(w2), 0.0)
    R = torch.where(pole, -0.5 * x0 * wt, x0)
    model = []
    for w in _frequencies("real", nf):
        a = complex(w) + 1j * ETA
        model.append(torch.where(pole, R * (1.0 / (a - wt) - 1.0 / (a + wt)), x0) + eye)
    model = torch.stack(model)
    qg = np.sqrt((((x.G + np.array([1.0 / x.k[0], 0.0, 0.0])) * (2.0 * math.pi / case["a"])) ** 2).sum(1))
    v = torch.from_numpy(np.sqrt(4.0 * math.pi) / qg).cuda()
    lo = case["nocc"] - nqp // 2
    I = torch.empty(nf, x.nk, case["nb"], nqp, nqp, dtype=torch.complex128, device="cuda")
    for ik in range(x.nk):
        r = x.rho(ik, lo, lo + nqp, 0, case["nb"]).transpose(0, 1)      # [m][a][G]
        for f in range(nf):
            W = v[:, None] * model[f] * v[None]
            Wd = 0.5 * (W + W.T).imag - 0.5j * (W - W.T).real
            I[f, ik] = -0.5 * x.pref * ((r @ Wd) @ r.conj().transpose(1, 2))
    return [wt, R, model, I]


def _exact_network(case, seed, rows):
    p, x, t = _network(seed, rows)
    low = (lambda a: a.float().bfloat16().double()) if case["bf16"] else (lambda a: a)
    p64, x, t = p.double(), x.double(), t.double()
    cut = np.cumsum([0, 640, 128, 16384, 128, 256, 2])
    w1, b1, w2, b2, w3, b3 = (p64[a:b] for a, b in zip(cut, cut[1:]))
    w1, w2, w3 = w1.reshape(128, 5), w2.reshape(128, 128), w3.reshape(2, 128)
    xr = low(x)
    h1 = torch.tanh(xr @ low(w1).T + b1)
    h2 = torch.tanh(low(h1) @ low(w2).T + b2)
    y = low(h2) @ low(w3).T + b3
    if case["kind"] == "predict":
        return y
    dy = (y - t) / rows
    loss = 0.5 * ((y - t) ** 2).sum() / rows
    d2 = (low(dy) @ low(w3)) * (1.0 - h2 * h2)
    d1 = (low(d2) @ low(w2)) * (1.0 - h1 * h1)
    g = torch.cat([(low(d1).T @ xr).flatten(), d1.sum(0), (low(d2).T @ low(h1)).flatten(), d2.sum(0),
                   (low(dy).T @ low(h2)).flatten(), dy.sum(0)])
    new = p64 - 2e-3 * g / (g.abs() + 1e-8)
    return {"loss": loss.reshape(1), "g": g, "p": new, "m": 0.1 * g, "v": 0.001 * g * g}


def exact(case, seed):
    kind = case["kind"]
    if kind == "response":
        omega = _frequencies(case["axis"], case["nw"])
        half = 1 if case["axis"] != "real" else 2
        if _exact_cost(case, case["ng"], half * len(omega)) > EXACT_MAX:
            return None
        return list(_exact_response(case, seed, (case["q1"], case["q2"], case["q3"]), omega,
                                    0.0 if case["axis"] == "imag" else ETA))
    if kind == "batch":
        parts = list(_batch_parts(case))
        if sum(_exact_cost(p, p["ng"], p["nw"]) * len(p["qs"]) for p in parts) > EXACT_MAX:
            return None
        got = [_exact_response(p, seed + 1000 * s, q, _frequencies("imag", p["nw"]), 0.0)
               for s, p in enumerate(parts) for q in p["qs"]]
        return [c for c, _ in got] + [e for _, e in got]
    if kind == "gw":
        return _exact_gw(case, seed)
    if kind == "dyson":
        chi, v = _screening(case["ng"], case["nw"], seed)
        vd = torch.from_numpy(v).cuda()
        eye = torch.eye(case["ng"], dtype=torch.complex128, device="cuda")
        return torch.stack([torch.linalg.inv(eye - vd[:, None] * c * vd[None]) for c in chi])
    return _exact_network(case, seed, case["batch"] if kind == "train" else case["rows"])
