"""The workloads this library is timed on, through its public entry points.

Every case is one call a fit, a toy study or a generator makes: an NLL and
gradient pass (the whole work of a minimiser's step), over one sample, over a
batch of toys or over the categories of a simultaneous fit; a batch of
pseudo-experiments; a CLs scan.  Sizes are those of the repository's benchmark
and tests, from the smallest fit request (1e3 events) to the largest (1e7).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1706_01420_gb300 import api, synth

# ---- the cases -------------------------------------------------------------

F64 = torch.float64
T_HI = 15.0
T_LO = {"1d": 0.3, "4d": 0.0, "tagged": 0.0, "phis": 0.0}
COLS = {"1d": ("t",), "4d": ("t", "ck", "cl", "phi"), "tagged": ("t", "q"), "phis": ("t", "ck", "cl", "phi", "q")}
TRUTH = {
    "1d": list(synth.TRUTH_1D.values()),
    "4d": list(synth.TRUTH_4D.values()),
    "tagged": list(synth.TRUTH_TAGGED.values()),
    # the 4D parameters, DG, Dm, phi_s, omega, C_SP and the tag selector
    "phis": list(synth.TRUTH_4D.values()) + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0],
}
# Example 2's simultaneous fit: six m(KK) bins times two flavours
CSP_BINS = (0.96, 0.93, 0.88, 0.90, 0.95, 0.97)
TRUTH_JOINT = [0.66, 0.52, 0.25, 3.2, 3.1, 0.085, 17.77, 0.8,
               0.02, 0.035, 0.05, 0.06, 0.04, 0.03, 1.2, 0.7, 0.2, -0.3, -0.8, -1.3]


def listed() -> list[dict]:
    def grad(name, model, n, weighted=False, cached=False):
        return {"name": name, "kind": "grad", "model": model, "n": n, "weighted": weighted, "cached": cached}

    return [
        # the decay-time fit of 1e5 events: one minimiser step
        grad("time_1e5", "1d", 100_000),
        # the smallest request of the fit server (weighted, 1e3 events): latency
        grad("angtime_w_1e3", "4d", 1_000, weighted=True),
        # the headline sample of the benchmark
        grad("angtime_1e6", "4d", 1_000_000),
        # the server's largest request, weighted
        grad("angtime_w_1e7", "4d", 10_000_000, weighted=True),
        # one pass over a batch of uneven toys (each at its own parameters)
        {"name": "angtime_toys", "kind": "toys", "model": "4d", "toys": 512, "mean": 20_000, "weighted": False},
        # the flavour-tagged decay-time fit; a size that is no multiple of anything
        grad("tagged_1e6", "tagged", 999_983),
        # the time-dependent angular fit with tagging
        grad("phis_1e6", "phis", 1_000_000),
        # Example 2's twelve categories at its small sample
        {"name": "phis_joint_1e4", "kind": "joint", "n": 10_000},
        # pseudo-experiments of the 4D model, a batch for a toy study ...
        {"name": "toygen_batch", "kind": "toygen", "model": "4d", "toys": 512, "mean": 20_000},
        # ... and one sample of Example 5's size
        {"name": "toygen_one", "kind": "toygen", "model": "4d", "toys": 1, "mean": 133_725},
        # one category of Example 2's 1e7-event sample, in sub-samples
        {"name": "phis_toygen", "kind": "toygen", "model": "phis", "toys": 102, "mean": 8_170},
        # Example 4: CLs of 10 000 bins from 10 000 toys per hypothesis
        {"name": "cls", "kind": "cls", "bins": 10_000, "toys": 10_000},
    ]


def draw(rng) -> dict:
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["grad", "grad", "grad", "toys", "joint", "toygen", "toygen", "cls"])
    if kind == "grad":
        model = rng.choice(["1d", "4d", "4d", "tagged", "phis"])
        n = log(1e3, {"1d": 2e6, "4d": 1e7, "tagged": 2e6, "phis": 1e6}[model])
        return {"kind": kind, "model": model, "n": n, "weighted": rng.random() < 0.5,
                "cached": model in ("4d", "phis") and rng.random() < 0.25}
    if kind == "toys":
        return {"kind": kind, "model": rng.choice(["1d", "4d", "4d"]), "toys": log(16, 512), "mean": log(1e3, 2e4),
                "weighted": rng.random() < 0.5}
    if kind == "joint":
        return {"kind": kind, "n": log(1e4, 1e6)}
    if kind == "toygen":
        model = rng.choice(["1d", "4d", "tagged", "phis"])
        toys = log(1, 512) if model in ("1d", "4d") else log(1, 100)
        most = 2e4 if model in ("1d", "4d") else 8e3
        if toys < 8 and model == "4d":
            most = 1.4e5
        return {"kind": kind, "model": model, "toys": toys, "mean": log(1e3, most)}
    return {"kind": kind, "bins": log(500, 1e4), "toys": log(1e3, 1e4)}


# ---- inputs ----------------------------------------------------------------

def _model(name):
    return {"1d": api.model_1d, "4d": api.model_4d, "tagged": api.model_tagged, "phis": api.model_phis}[name](
        T_LO[name], T_HI)


def _theta(name, seed, rows=1):
    """Parameters a fit visits: the truth, every non-zero one a per cent or so off."""
    rng = np.random.default_rng(seed + 17)
    th = np.tile(np.array(TRUTH[name]), (rows, 1))
    th *= 1.0 + 0.01 * rng.uniform(-1.0, 1.0, th.shape)
    return th


def _events(name, n, seed, weighted, dev, f_b=0.1):
    """The recipe of synth.py, drawn on the GPU: an exponential with a Gaussian
    resolution over a flat background, uniform angles, tags +-1, weights N(1, 0.2)."""
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def uni(k, lo, hi):
        return torch.empty(k, dtype=F64, device=dev).uniform_(lo, hi, generator=g)

    lo, hi = T_LO[name], T_HI
    k = n + n // 2 + 1024
    sig = torch.empty(k, dtype=F64, device=dev).exponential_(0.66, generator=g)
    sig += 0.045 * torch.empty(k, dtype=F64, device=dev).normal_(generator=g)
    sig = sig[(sig >= lo) & (sig <= hi)][:n]
    ev = {"t": torch.where(uni(n, 0.0, 1.0) < f_b, uni(n, lo, hi), sig)}
    if "ck" in COLS[name]:
        ev["ck"], ev["cl"] = uni(n, -1.0, 1.0), uni(n, -1.0, 1.0)
        ev["phi"] = uni(n, -math.pi, math.pi)
    if "q" in COLS[name]:
        ev["q"] = torch.where(uni(n, 0.0, 1.0) < 0.5, 1.0, -1.0).to(F64)
    if weighted:
        ev["w"] = torch.empty(n, dtype=F64, device=dev).normal_(1.0, 0.2, generator=g)
    return ev


def _sizes(case, seed):
    """Per-toy counts: Poisson around the mean, a tenth of each background.  A
    generator's counts are the case's own (its columns have one length)."""
    n_sig, n_bkg = synth.toy_sizes(case["toys"], case["mean"], 0.1, seed if case["kind"] == "toys" else case["mean"])
    return n_sig, n_bkg, np.concatenate([[0], np.cumsum(n_sig + n_bkg)]).astype(np.int64)


def _joint_map():
    jmap, value = [], []
    for b in range(6):
        for q in (1.0, -1.0):
            jmap.append([0, -1, -1, -1, 1, 2, 3, 4, 8 + b, 14 + b, 5, 6, 7, -1, -1, -1])
            value.append([0, 0.045, 0.0, 0.0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0.0, CSP_BINS[b], q])
    return jmap, value


def _joint_theta(seed):
    rng = np.random.default_rng(seed + 17)
    return np.array(TRUTH_JOINT) * (1.0 + 0.01 * rng.uniform(-1.0, 1.0, 20))


def _joint_events(case, seed, dev):
    per = case["n"] // 12
    ev = _events("phis", 12 * per, seed, False, dev, f_b=0.0)
    ev["q"] = torch.tensor([1.0, -1.0] * 6, dtype=F64, device=dev).repeat_interleave(per)
    return ev, np.arange(13, dtype=np.int64) * per


def _cls_inputs(case, seed, dev):
    """Example 4's shapes: a smeared Gaussian peak over exp(0.001 m), about 70
    signal and 5000 background events, and data drawn from their sum."""
    rng = np.random.default_rng(seed)
    n = case["bins"]
    lo, hi = 5179.0, 5379.0
    c = lo + (np.arange(n) + 0.5) * ((hi - lo) / n)
    m0, width = 5279.6 + rng.uniform(-5.0, 5.0), math.hypot(5.0, 8.0) * rng.uniform(0.9, 1.1)
    sig = np.exp(-0.5 * ((c - m0) / width) ** 2)
    bkg = np.exp(0.001 * c)
    s, b = sig / sig.sum() * 70.0 * rng.uniform(0.8, 1.2), bkg / bkg.sum() * 5000.0 * rng.uniform(0.9, 1.1)
    data = rng.poisson(b + s * (seed % 2)).astype(np.int32)
    return [torch.tensor(x, device=dev) for x in (s, b, data)]


def prepare(case: dict, seed: int) -> dict:
    dev = torch.device("cuda")
    kind = case["kind"]
    st = {"kind": kind, "seed": seed}
    if kind == "cls":
        st["s"], st["b"], st["data"] = _cls_inputs(case, seed, dev)
        st["toys"] = case["toys"]
        return st
    if kind == "joint":
        st["m"] = api.model_phis(0.0, T_HI)
        st["joint"] = api.Joint(*_joint_map())
        st["ev"], seg = _joint_events(case, seed, dev)
        st["seg"] = torch.tensor(seg, device=dev)
        st["theta"] = torch.tensor(_joint_theta(seed)[None, :], device=dev)
        return st
    st["m"] = _model(case["model"])
    if kind == "grad":
        st["ev"] = _events(case["model"], case["n"], seed, case["weighted"], dev)
        if case["cached"]:      # kept by a fit for all its passes over these events
            st["ev"]["fk"] = api.ipa_angular_basis(st["m"], st["ev"])
        st["theta"] = torch.tensor(_theta(case["model"], seed)[0], device=dev)
        return st
    n_sig, n_bkg, off = _sizes(case, seed)
    if kind == "toys":
        st["ev"] = _events(case["model"], int(off[-1]), seed, case["weighted"], dev)
        st["seg"] = torch.tensor(off, device=dev)
        st["theta"] = torch.tensor(_theta(case["model"], seed, case["toys"]), device=dev)
        return st
    st["theta"] = torch.tensor(_theta(case["model"], seed)[0], device=dev)
    st["n_sig"], st["n_bkg"], st["off"] = (torch.tensor(x, device=dev) for x in (n_sig, n_bkg, off[:-1].copy()))
    st["out"] = {k: torch.empty(int(off[-1]), dtype=F64, device=dev) for k in COLS[case["model"]]}
    return st


def run(st: dict):
    kind = st["kind"]
    if kind == "grad":
        return api.ipa_nll_grad(st["m"], st["ev"], st["theta"])
    if kind == "toys":
        return api.ipa_nll_grad_segmented(st["m"], st["ev"], st["seg"], st["theta"])
    if kind == "joint":
        return api.ipa_nll_grad_joint(st["m"], st["ev"], st["seg"], st["joint"], st["theta"])
    if kind == "toygen":
        return api.ipa_toygen(st["m"], st["theta"], st["seed"], st["n_sig"], st["n_bkg"], st["off"], st["out"])
    return api.ipa_cls(st["s"], st["b"], st["data"], st["toys"], st["seed"], with_x=True)


# FP64 operations per event of the formulas (an elementary function counted as
# 20, a Faddeeva function as 200 for the fifth of the events near the peak), and
# of one candidate of a generator (its Philox blocks counted as 100 each).
FLOPS = {"1d": 80, "4d": 220, "tagged": 250, "phis": 450}
CANDIDATES = {"1d": 12, "4d": 50, "tagged": 12, "phis": 12}     # per accepted event, about
FLOPS_CANDIDATE = {"1d": 160, "4d": 190, "tagged": 400, "phis": 800}


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "cls":
        draws = 2 * case["bins"] * case["toys"]
        return {"bytes": 20 * case["bins"] + 16 * case["toys"], "flops": 110 * draws}
    if kind == "joint":
        return {"bytes": 40 * case["n"], "flops": FLOPS["phis"] * case["n"]}
    model = case["model"]
    if kind == "toygen":
        n = case["toys"] * case["mean"]
        return {"bytes": 8 * len(COLS[model]) * n, "flops": CANDIDATES[model] * FLOPS_CANDIDATE[model] * n}
    n = case["n"] if kind == "grad" else case["toys"] * case["mean"]
    cols = len(COLS[model]) + case["weighted"] + (7 if case.get("cached") else 0)
    return {"bytes": 8 * cols * n, "flops": FLOPS[model] * n}


# ---- the same values in 64 bits from plain torch ---------------------------

@functools.lru_cache(maxsize=None)
def _weideman(n=64):
    """Coefficients of Weideman's rational approximation of w(z) (1994), N = n."""
    m = 4 * n
    ell = math.sqrt(n / math.sqrt(2.0))
    th = np.arange(-m + 1, m) * (math.pi / m)
    t = ell * np.tan(0.5 * th)
    f = np.concatenate([[0.0], np.exp(-t * t) * (ell * ell + t * t)])
    a = np.real(np.fft.fft(np.fft.fftshift(f))) / (2 * m)
    return ell, a[1:n + 1].copy()


class _Faddeeva(torch.autograd.Function):
    """w(z) = exp(-z^2) erfc(-iz) for Im z >= 0, with w' = -2 z w + 2i / sqrt(pi)."""

    @staticmethod
    def forward(ctx, z):
        ell, a = _weideman()
        d = ell - 1j * z
        x = (ell + 1j * z) / d
        p = torch.zeros_like(z)
        for c in a[::-1]:
            p = p * x + float(c)
        w = 2.0 * p / (d * d) + (1.0 / math.sqrt(math.pi)) / d
        ctx.save_for_backward(z, w)
        return w

    @staticmethod
    def backward(ctx, g):
        z, w = ctx.saved_tensors
        return g * torch.conj(-2.0 * z * w + 2.0j / math.sqrt(math.pi))


SQRT2 = math.sqrt(2.0)


def _conv(tau, gam, sig):
    """exp(-gam u) convolved with a unit Gaussian of width sig, at tau."""
    z = (gam * sig * sig - tau) / (SQRT2 * sig)
    return 0.5 * torch.exp(-gam * tau + 0.5 * (gam * sig) ** 2) * torch.special.erfc(z)


def _conv_c(tau, gam, dm, sig):
    """The same for the complex rate gam - i dm, through the Faddeeva function."""
    a = (gam * sig * sig - tau) / (SQRT2 * sig)
    beta = (dm * sig / SQRT2).expand_as(a)
    gx = torch.exp(-0.5 * (tau / sig) ** 2)
    neg = a < 0
    w = _Faddeeva.apply(torch.complex(torch.where(neg, -beta, beta), torch.abs(a)))
    mag = torch.exp(-gam * tau + 0.5 * (gam - dm) * (gam + dm) * sig * sig)
    ph = dm * tau - gam * dm * sig * sig
    re = torch.where(neg, mag * torch.cos(ph) - 0.5 * gx * w.real, 0.5 * gx * w.real)
    im = torch.where(neg, mag * torch.sin(ph) - 0.5 * gx * w.imag, 0.5 * gx * w.imag)
    return re, im


def _norm(gam, sig, mu, lo, hi):
    def anti(t):
        return (0.5 * torch.special.erfc(-(t - mu) / (SQRT2 * sig)) - _conv(t - mu, gam, sig)) / gam
    return anti(hi) - anti(lo)


def _norm_c_imag(gam, dm, sig, mu, lo, hi):
    def anti(t):
        re, im = _conv_c(t - mu, gam, dm, sig)
        re = 0.5 * torch.special.erfc(-(t - mu) / (SQRT2 * sig)) - re
        return (re * dm - im * gam) / (gam * gam + dm * dm)     # Im of (Phi - g) / (gam - i dm)
    return anti(hi) - anti(lo)


def _basis(ev):
    sk, sl = torch.sqrt(1.0 - ev["ck"] ** 2), torch.sqrt(1.0 - ev["cl"] ** 2)
    ck, cl, cp, sp = ev["ck"], ev["cl"], torch.cos(ev["phi"]), torch.sin(ev["phi"])
    r6, r3 = 2.0 / math.sqrt(6.0), 2.0 / math.sqrt(3.0)
    return [(ck * sl) ** 2, 0.5 * sk ** 2 * (1.0 - (sl * cp) ** 2), 0.5 * sk ** 2 * (1.0 - (sl * sp) ** 2),
            (sk * sl) ** 2 * sp * cp, SQRT2 * sk * ck * sl * cl * cp, -SQRT2 * sk * ck * sl * cl * sp, sl ** 2 / 3.0,
            r6 * sk * sl * cl * cp, -r6 * sk * sl * cl * sp, r3 * ck * sl ** 2]


BASIS_MAX = [1.0, 0.5, 0.5, 0.5, SQRT2 / 4, SQRT2 / 4, 1 / 3, 1 / math.sqrt(6.0), 1 / math.sqrt(6.0),
             2 / math.sqrt(3.0)]
I_OMEGA = 16.0 * math.pi / 9.0


def _bilinears(p):
    """Magnitude and phase of the ten products of transversity amplitudes."""
    x0, xe, dpa, dpe, f, ds = p[4:10]
    xa, s = 1.0 - x0 - xe, 1.0 - f
    r0, ra, re, rf = torch.sqrt(s * x0), torch.sqrt(s * xa), torch.sqrt(s * xe), torch.sqrt(f)
    zero = torch.zeros_like(x0)
    return [(r0 * r0, zero), (ra * ra, zero), (re * re, zero), (ra * re, dpe - dpa), (r0 * ra, dpa), (r0 * re, dpe),
            (rf * rf, zero), (rf * ra, dpa - ds), (rf * re, dpe - ds), (rf * r0, -ds)]


# per term: "r" or "i" (real or imaginary part) and the CP eigenvalues of its two amplitudes
PARTS = ["r", "r", "r", "i", "r", "i", "r", "r", "i", "r"]
ETA = [(1, 1), (1, 1), (-1, -1), (1, -1), (1, 1), (1, -1), (-1, -1), (-1, 1), (-1, -1), (-1, 1)]


def _rate_phis(ev, p):
    """The time-dependent angular rate of the event's tag."""
    gam, sig, mu, dg, dm, phi, om, csp = p[0], p[1], p[2], p[10], p[11], p[12], p[13], p[14]
    tau = ev["t"] - mu
    gl, gh = _conv(tau, gam + 0.5 * dg, sig), _conv(tau, gam - 0.5 * dg, sig)
    cr, ci = _conv_c(tau, gam, dm, sig)
    d = 1.0 - 2.0 * om
    cr, ci = ev["q"] * d * cr, ev["q"] * d * ci
    c, s = torch.cos(phi), torch.sin(phi)
    rate = 0.0
    for k, (f, (m, psi)) in enumerate(zip(_basis(ev), _bilinears(p))):
        e1, e2 = ETA[k]
        re, im = m * torch.cos(psi), m * torch.sin(psi)
        if e1 == e2:
            term = (re if PARTS[k] == "r" else im) * (0.5 * (1 + e2 * c) * gl + 0.5 * (1 - e2 * c) * gh + e2 * s * ci)
        else:
            odd = e2 * (0.5 * s * (gl - gh) - c * ci)
            term = cr * re + odd * im if PARTS[k] == "r" else cr * im - odd * re
        rate = rate + f * term * (csp if k >= 7 else 1.0)
    return rate


def _pdf(name, ev, p):
    """P of every event; p: the parameters, each broadcasting against the columns."""
    lo = torch.full_like(p[0], T_LO[name])
    hi = torch.full_like(p[0], T_HI)
    gam, sig, mu, fb = p[:4]
    span = T_HI - T_LO[name]
    if name in ("1d", "4d"):
        pdf = _conv(ev["t"] - mu, gam, sig) / _norm(gam, sig, mu, lo, hi)
        vol = span
        if name == "4d":
            amp = sum(f * m * (torch.cos(psi) if PARTS[k] == "r" else torch.sin(psi))
                      for k, (f, (m, psi)) in enumerate(zip(_basis(ev), _bilinears(p))))
            pdf, vol = pdf * amp / I_OMEGA, vol * 8.0 * math.pi
        return (1.0 - fb) * pdf + fb / vol
    dg, dm = (p[4], p[5]) if name == "tagged" else (p[10], p[11])
    phi, om = (p[6], p[7]) if name == "tagged" else (p[12], p[13])
    c, s, d = torch.cos(phi), torch.sin(phi), 1.0 - 2.0 * om
    il, ih = _norm(gam + 0.5 * dg, sig, mu, lo, hi), _norm(gam - 0.5 * dg, sig, mu, lo, hi)
    if name == "tagged":
        tau = ev["t"] - mu
        rate = (0.5 * (1 - c) * _conv(tau, gam - 0.5 * dg, sig) + 0.5 * (1 + c) * _conv(tau, gam + 0.5 * dg, sig)
                + ev["q"] * d * s * _conv_c(tau, gam, dm, sig)[1])
        return (1.0 - fb) * rate / ((1 - c) * ih + (1 + c) * il) + fb / (2.0 * span)
    b = _bilinears(p)
    even, odd = b[0][0] + b[1][0], b[2][0] + b[6][0]
    norm = I_OMEGA * (even * ((1 + c) * il + (1 - c) * ih) + odd * ((1 - c) * il + (1 + c) * ih))
    one = torch.sign(p[15])
    part = 0.5 * norm + one * I_OMEGA * d * s * (even - odd) * _norm_c_imag(gam, dm, sig, mu, lo, hi)
    both = one == 0
    vol = 2.0 * span * 8.0 * math.pi * torch.where(both, 1.0, 0.5).to(F64)
    return (1.0 - fb) * _rate_phis(ev, p) / torch.where(both, norm, part) + fb / vol


def _nll_grad(name, ev, w, theta):
    """[NLL, gradient] of each row: columns and weights (rows, events), theta (rows, parameters)."""
    th = theta.clone().requires_grad_(True)
    nll = -(w * torch.log(_pdf(name, ev, [th[:, j:j + 1] for j in range(th.shape[1])]))).sum(1)
    g, = torch.autograd.grad(nll.sum(), th)
    return torch.cat([nll.detach()[:, None], g], 1)


def _rows(name, ev, off, theta):
    """[NLL, gradient] of every segment, a few rows at a time."""
    dev = ev["t"].device
    out = []
    length = np.diff(off)
    i = 0
    while i < len(length):
        j = i + 1
        while j < len(length) and (j + 1 - i) * int(length[i:j + 1].max()) <= 1 << 20:
            j += 1
        most = max(1, int(length[i:j].max()))
        at = torch.arange(most, device=dev)[None, :]
        lo = torch.tensor(off[i:j], device=dev)[:, None]
        inside = at < torch.tensor(length[i:j], device=dev)[:, None]
        idx = torch.where(inside, lo + at, lo.clamp(max=int(off[-1]) - 1))
        cols = {k: v[idx] for k, v in ev.items() if k in COLS[name]}
        w = inside.to(F64) * (ev["w"][idx] if "w" in ev else 1.0)
        out.append(_nll_grad(name, cols, w, theta[i:j]))
        i = j
    return torch.cat(out)


M32 = 0xFFFFFFFF


def _philox(idx, toy, call, seed):
    """Philox-4x32-10 (Salmon et al. 2011) at counters (idx lo, idx hi, toy, call); words as int64."""
    c0, c1 = idx & M32, idx >> 32
    c2, c3 = (torch.as_tensor(x, device=idx.device).expand_as(idx) for x in (toy, call))
    k0, k1 = seed & M32, seed >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57           # modulo 2^64
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _uni(hi, lo):
    return (((((hi << 32) | lo) >> 11) & ((1 << 53) - 1)) + 1).to(F64) * 2.0 ** -53


def _toy(name, p, seed, toy, n_sig, n_bkg, dev):
    """One pseudo-experiment: accept-reject over counted candidates, then the background."""
    lo, span = T_LO[name], T_HI - T_LO[name]
    pt = [torch.tensor(float(v), dtype=F64, device=dev) for v in p]
    gam, sig, mu = p[:3]

    def most(x, t):
        return min(1.0, math.exp(-x * (t - mu) + 0.5 * (x * sig) ** 2))

    def angles(b, d):
        return {"ck": 2.0 * _uni(b[0], b[1]) - 1.0, "cl": 2.0 * _uni(b[2], b[3]) - 1.0,
                "phi": math.pi * (2.0 * _uni(d[0], d[1]) - 1.0)}

    def tag(u):
        return torch.where(u <= 0.5, 1.0, -1.0).to(F64)

    if name in ("4d", "phis"):
        mag = [float(m) for m, _ in _bilinears(pt)]
    if name == "phis":
        ang = sum(x * m * (abs(p[14]) if k >= 7 else 1.0) for k, (x, m) in enumerate(zip(BASIS_MAX, mag)))
        wid = span / 64
        edge = [lo + i * wid for i in range(64)]
        bound = [(most(gam + 0.5 * p[10], e) + most(gam - 0.5 * p[10], e) + 2 * most(gam, e)) * ang for e in edge]
        cum = torch.tensor(np.cumsum(bound), dtype=F64, device=dev)
        bound, edge = torch.tensor(bound, dtype=F64, device=dev), torch.tensor(edge, dtype=F64, device=dev)
    kept, got, j0, chunk = [], 0, 0, int(min(1 << 23, max(1 << 16, 30 * n_sig)))
    while got < n_sig:
        j = torch.arange(j0, j0 + chunk, device=dev)
        a = _philox(j, toy, 0, seed)
        if name in ("1d", "4d"):
            ev = {"t": lo + _uni(a[0], a[1]) * span}
            keep = _uni(a[2], a[3]) * most(gam, lo) < _conv(ev["t"] - mu, pt[0], pt[1])
            if name == "4d":
                j, ev = j[keep], {"t": ev["t"][keep]}
                d = _philox(j, toy, 2, seed)
                ev.update(angles(_philox(j, toy, 1, seed), d))
                h = [m * (torch.cos(psi) if PARTS[k] == "r" else torch.sin(psi))
                     for k, (m, psi) in enumerate(_bilinears(pt))]
                top = sum(abs(float(x)) * b for x, b in zip(h, BASIS_MAX))
                keep = _uni(d[2], d[3]) * top < sum(x * f for x, f in zip(h, _basis(ev)))
        elif name == "tagged":
            ev = {"t": lo + _uni(a[0], a[1]) * span, "q": tag(_uni(*_philox(j, toy, 1, seed)[:2]))}
            c, s, d = math.cos(p[6]), math.sin(p[6]), 1.0 - 2.0 * p[7]
            gh, gl = gam - 0.5 * p[4], gam + 0.5 * p[4]
            top = 0.5 * (1 - c) * most(gh, lo) + 0.5 * (1 + c) * most(gl, lo) + abs(d * s) * most(gam, lo)
            tau = ev["t"] - mu
            rate = (0.5 * (1 - c) * _conv(tau, pt[0] - 0.5 * pt[4], pt[1])
                    + 0.5 * (1 + c) * _conv(tau, pt[0] + 0.5 * pt[4], pt[1])
                    + ev["q"] * d * s * _conv_c(tau, pt[0], pt[5], pt[1])[1])
            keep = _uni(a[2], a[3]) * top < rate
        else:
            d = _philox(j, toy, 2, seed)
            i = torch.searchsorted(cum, _uni(a[0], a[1]) * cum[-1])
            u = _uni(*_philox(j, toy, 3, seed)[:2])
            ev = {"t": torch.clamp(edge[i] + _uni(d[2], d[3]) * wid, max=T_HI), **angles(_philox(j, toy, 1, seed), d),
                  "q": tag(u) if p[15] == 0 else torch.full_like(u, math.copysign(1.0, p[15]))}
            keep = _uni(a[2], a[3]) * bound[i] < _rate_phis(ev, pt)
        kept.append({k: v[keep] for k, v in ev.items()})
        got += kept[-1]["t"].numel()
        j0 += chunk
    out = {k: torch.cat([e[k] for e in kept])[:n_sig] for k in COLS[name]}
    i = torch.arange(n_bkg, device=dev)
    a, b = _philox(i, toy, 4, seed), _philox(i, toy, 5, seed)
    bkg = {"t": lo + _uni(a[0], a[1]) * span}
    if "ck" in out:
        bkg.update({"ck": 2.0 * _uni(a[2], a[3]) - 1.0, "cl": 2.0 * _uni(b[0], b[1]) - 1.0,
                    "phi": math.pi * (2.0 * _uni(b[2], b[3]) - 1.0)})
    if name == "tagged":
        bkg["q"] = tag(_uni(a[2], a[3]))
    if name == "phis":
        bkg["q"] = tag(_uni(*_philox(i, toy, 6, seed)[:2]))
    return {k: torch.cat([out[k], bkg[k]]) for k in out}


def _counts(lam, hyp, toys, seed):
    """(toys, bins) Poisson counts of means below 400, by inversion."""
    n = lam.numel()
    i = torch.arange(n, device=lam.device)[None, :].expand(len(toys), n)
    k = torch.tensor(toys, device=lam.device)[:, None].expand(len(toys), n)
    a = _philox(i, k, 8 + (hyp << 16), seed)
    u = _uni(a[0], a[1])
    prob = torch.exp(-lam)
    cum, out, m = prob.clone(), torch.zeros_like(u), 0
    while True:
        more = u > cum
        if not bool(more.any()) or m > 200:
            return out
        out += more
        m += 1
        prob = prob * lam / m
        cum = cum + prob


def exact(case: dict, seed: int):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind = case["kind"]
    if kind == "cls":
        s, b, data = _cls_inputs(case, seed, dev)
        w = torch.log1p(s / b)
        x = [[], []]
        step = max(1, (1 << 23) // case["bins"])
        for hyp, lam in enumerate((b, s + b)):
            for k in range(0, case["toys"], step):
                x[hyp].append(_counts(lam, hyp, list(range(k, min(k + step, case["toys"]))), seed) @ w)
        xb, xsb, xo = torch.cat(x[0]), torch.cat(x[1]), (data.to(F64) * w).sum()
        nb, nsb = int((xb <= xo).sum()), int((xsb <= xo).sum())
        cl = [nb / case["toys"], nsb / case["toys"], nsb / nb if nb else math.nan]
        cl = torch.tensor(cl, dtype=F64, device=dev)
        return {"cl_b": cl[0], "cl_sb": cl[1], "cl_s": cl[2], "counts": torch.tensor([nb, nsb], device=dev),
                "x_b": xb, "x_sb": xsb, "x_obs": xo}
    if kind == "joint":
        ev, off = _joint_events(case, seed, dev)
        jmap, value = _joint_map()
        th = _joint_theta(seed)
        cat = [[th[j] if j >= 0 else v for j, v in zip(*row)] for row in zip(jmap, value)]
        r = _rows("phis", ev, off, torch.tensor(cat, dtype=F64, device=dev))
        out = torch.zeros(1, 21, dtype=F64, device=dev)
        out[0, 0] = r[:, 0].sum()
        for c, row in enumerate(jmap):
            for k, j in enumerate(row):
                if j >= 0:
                    out[0, 1 + j] += r[c, 1 + k]
        return out
    name = case["model"]
    if kind == "grad":
        ev = _events(name, case["n"], seed, case["weighted"], dev)
        off = np.unique(np.concatenate([np.arange(0, case["n"], 1 << 20), [case["n"]]]))
        th = torch.tensor(_theta(name, seed), device=dev).expand(len(off) - 1, -1)
        r = _rows(name, ev, off, th).sum(0)
        if name == "phis":
            r[16] = 0.0     # the tag selector is no parameter of the rate
        return r
    n_sig, n_bkg, off = _sizes(case, seed)
    if kind == "toys":
        ev = _events(name, int(off[-1]), seed, case["weighted"], dev)
        return _rows(name, ev, off, torch.tensor(_theta(name, seed, case["toys"]), device=dev))
    p = _theta(name, seed)[0]
    toys = [_toy(name, p, seed, k, int(n_sig[k]), int(n_bkg[k]), dev) for k in range(case["toys"])]
    return {c: torch.cat([t[c] for t in toys]) for c in COLS[name]}
