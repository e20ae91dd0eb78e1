"""Inputs at the edges of the event loops' fixed-point formats and scales, against the
oracle, for all models that share them.

Tolerances: the NLL within 1e-14 of sum |w log P| and each gradient component within
5e-13 of the sum of |terms| (the reciprocal's 6e-14 and the fixed-point units, with
cancellation among the terms of a component by a factor of a few), unless a test says
otherwise."""
import numpy as np
import pytest

from paper_1706_01420_gb300 import synth

pytestmark = pytest.mark.gpu

TH4 = [0.66, 0.045, 0.0, 0.1, 0.52, 0.25, 3.2, 3.1, 0.04, 0.3]
TRUTH = {"1d": TH4[:4], "4d": TH4, "tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3],
         "phis": TH4 + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}
KINDS = list(TRUTH)


@pytest.fixture(scope="module")
def env(oracle):
    from tests import gpu_common as G
    G.need_gpu()
    import torch
    from paper_1706_01420_gb300 import api
    return oracle, G, torch, api


def columns(kind, n, seed, weighted=False):
    if kind == "1d":
        cols = {"t": synth.events_1d(n, seed, t_lo=0.0)}
        if weighted:
            cols["w"] = synth.weights(n, seed + 1)
        return cols
    return {"4d": synth.events_4d, "tagged": synth.events_tagged,
            "phis": synth.events_phis}[kind](n, seed, weighted=weighted)


def oracle_model(O, kind, lo, hi):
    return O.Model("tag" if kind == "tagged" else kind, lo, hi)


def gradients(env, kind, lo, hi, cols, th, cached=None):
    """The call with one warp per tile and with a team per tile: the same bits."""
    _, G, torch, api = env
    m = getattr(api, "model_" + kind)(lo, hi)
    n = len(cols["t"])
    ev = G.to_dev(cols)
    if cached is not None:
        ev["fk"] = cached
    theta = torch.tensor(np.asarray(th), device="cuda")
    got = {}
    try:
        for warps in (1, 2):
            api.ipa_launch_config_set(m, n, {"warps_per_block": warps, "warps_per_sm": 0, "tiles_per_take": 1},
                                      cached=cached is not None)
            got[warps] = api.ipa_nll_grad(m, ev, theta).cpu().numpy()
    finally:
        api.ipa_launch_config_set(m, n, {"warps_per_block": 1, "warps_per_sm": 0, "tiles_per_take": 1},
                                  cached=cached is not None)
    assert np.array_equal(got[1], got[2], equal_nan=True), (got[1], got[2])
    return got[1]


def check(env, kind, lo, hi, cols, th):
    O = env[0]
    got = gradients(env, kind, lo, hi, cols, th)
    m = oracle_model(O, kind, lo, hi)
    f, g = O.nll_grad(m, cols, th)
    logl, terms = O.nll_grad_terms(m, cols, th)
    assert abs(got[0] - f) <= 1e-14 * np.abs(logl).sum(), (got[0], f)
    assert np.all(np.abs(got[1:] - g) <= 5e-13 * np.abs(terms).sum(1)), (got[1:], g)


def by_the_plain_loop(env, kind, lo, hi, cols, th):
    """The same gradient from the FP64 loop, which the oracle tests cover elsewhere (a range
    under the peak has a normalisation that cancels in FP64, the oracle's and the library's
    differently, so there the two paths of the library are compared).  4D and phi_s: as fits
    of fewer than 64 events, which take it; 1D and tagged: with weights of 2^-500, whose scale
    is out of the integers' range and which multiply every sum exactly."""
    _, G, torch, api = env
    m = getattr(api, "model_" + kind)(lo, hi)
    n = len(cols["t"])
    if kind in ("1d", "tagged"):
        w = cols.get("w", np.ones(n))
        return np.ldexp(gradients(env, kind, lo, hi, {**cols, "w": np.ldexp(w, -500)}, th), 500)
    off = np.append(np.arange(0, n, 60), n)
    out = api.ipa_nll_grad_segmented(m, G.to_dev(cols), torch.tensor(off, device="cuda"),
                                     torch.tensor(np.tile(th, (len(off) - 1, 1)), device="cuda"))
    return out.cpu().numpy().sum(0)


def check_paths(env, kind, lo, hi, cols, th, rtol):
    fast, plain = gradients(env, kind, lo, hi, cols, th), by_the_plain_loop(env, kind, lo, hi, cols, th)
    logl, terms = env[0].nll_grad_terms(oracle_model(env[0], kind, lo, hi), cols, th)
    scale = np.abs(terms).sum(1)
    assert np.isfinite(plain).all() and np.isfinite(scale).all()
    assert abs(fast[0] - plain[0]) <= 1e-13 * np.abs(logl).sum(), (fast, plain)
    assert np.all(np.abs(fast[1:] - plain[1:]) <= rtol * scale), (fast, plain)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kind", KINDS)
def test_gaussian_just_below_a_power_of_two(env, kind, weighted):
    """tau^2 / (2 sigma^2) within a few last places of 1, 2, .., 32, on both sides of the peak
    (times on a grid meet these: 0.18 is 4 sigma)."""
    x = np.sqrt(2.0 * 2.0 ** np.arange(6.0)) * TRUTH[kind][1]
    steps = np.arange(-24, 25)
    t = (x[:, None] + steps * np.spacing(x)[:, None]).ravel()
    cols = columns(kind, 2 * t.size, 5, weighted)
    cols["t"] = np.concatenate([t, -t])
    check(env, kind, -0.5, 15.0, cols, TRUTH[kind])


@pytest.mark.parametrize("kind", KINDS)
def test_weighted_log_just_below_a_power_of_two(env, kind):
    """Weighted events with P = 2^e (1 - 2^-k), k = 32 .. 40, placed by bisection in t."""
    O = env[0]
    th = np.array(TRUTH[kind])
    m = oracle_model(O, kind, 0.0, 15.0)
    cols = columns(kind, 400, 7, weighted=True)
    one = {k: v[200:201].copy() for k, v in cols.items()}

    def density(t):
        one["t"][0] = t
        return float(O.pdf(m, one, th)[0])
    p = np.array([density(t) for t in np.linspace(0.35, 4.0, 400)])
    e = np.floor(np.log2(p))
    for i in np.nonzero(e[1:] != e[:-1])[0][:3]:
        edge = 2.0 ** max(e[i], e[i + 1])
        for k in (32, 33, 36, 40):
            goal = edge * (1.0 - 2.0 ** -k)
            lo, hi = np.linspace(0.35, 4.0, 400)[i:i + 2]
            for _ in range(80):
                mid = 0.5 * (lo + hi)
                if (density(mid) < goal) == (p[i] < goal):
                    lo = mid
                else:
                    hi = mid
            assert abs(density(lo) / edge - (1.0 - 2.0 ** -k)) < 2.0 ** -45
            cols["t"][200], cols["w"][200] = lo, 1.7
            check(env, kind, 0.0, 15.0, cols, th)


OUTSIDE = [("1d", 3, 1.5), ("1d", 3, -0.1), ("1d", 1, -0.045), ("1d", 0, -0.1), ("1d", 0, np.nan),
           ("tagged", 3, np.nan), ("tagged", 6, np.nan), ("tagged", 0, np.nan)]


@pytest.mark.parametrize("kind, index, value", OUTSIDE)
@pytest.mark.parametrize("n", [3000, 700_000])
def test_no_scale_outside_the_domain(env, kind, index, value, n):
    """Parameters for which the integers' scale is out of range leave the tile to the plain
    loop in either form: NaN throughout, as from the NLL alone (the larger call takes single
    warps in the built-in geometry, and has NaN in every component too)."""
    _, G, torch, api = env
    th = np.array(TRUTH[kind])
    th[index] = value
    cols = columns(kind, n, 9)
    if n == 3000:
        got = gradients(env, kind, 0.0, 15.0, cols, th)
    else:
        m = getattr(api, "model_" + kind)(0.0, 15.0)
        got = api.ipa_nll_grad(m, G.to_dev(cols), torch.tensor(th, device="cuda")).cpu().numpy()
    assert np.isnan(got).all(), got


def test_fit_of_one_parameter_from_outside_the_domain(env):
    _, G, torch, api = env
    n = 700_000
    start = np.array(TRUTH["1d"])
    start[3] = 1.5
    params = [api.Param(float(v), fixed=True) for v in start[:3]] + [api.Param(1.5, -1.0, 2.0, 0.01)]
    off = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    r = api.ipa_fit_batch(api.model_1d(0.0, 15.0), G.to_dev(columns("1d", n, 9)), off, params,
                          torch.tensor(start[None, :], device="cuda"), max_iter=50, tol=1e-8)
    assert int(r["status"].cpu()[0]) == 3                 # IPA_FIT_BAD_PDF


@pytest.mark.parametrize("kind", ["1d", "tagged"])
@pytest.mark.parametrize("sigmas", [20.0, 24.0, 26.0])
def test_no_scale_far_below_the_peak(env, kind, sigmas):
    """A range that ends 24 sigma and more below mu: cs is beyond the integers' scale, and both
    calls take the plain loop (a tile that was left out gave nothing): 5e-13 of the sum of |terms|;
    20 sigma is within it, at the next test's tolerance."""
    th = np.array(TRUTH[kind])
    cols = columns(kind, 3000, 13)
    hi = -sigmas * th[1]
    cols["t"] = np.random.default_rng(3).uniform(hi - 3.0 * th[1], hi, 3000)
    check_paths(env, kind, hi - 3.0 * th[1], hi, cols, th, 1e-9 if sigmas == 20.0 else 5e-13)


@pytest.mark.parametrize("kind", ["1d", "tagged"])
@pytest.mark.parametrize("sigma", [0.0313, 0.045, 0.0624])
@pytest.mark.parametrize("f_b", [0.0, 0.1, 0.99])
@pytest.mark.parametrize("below", [6.0, 8.0, 10.0, 14.0, 16.0, 18.0, 20.0, 22.0])
def test_gaussian_sums_below_the_peak(env, kind, sigma, f_b, below):
    """Ranges of 3.5 sigma that end `below` sigma under mu.  The integers' unit against the
    pieces of a component, which cancel to sigma / (|tau| Gamma sigma) of themselves, and again
    in sigma: 1e3 times (|tau| / sigma)^2 units of 2^-49, below 1e-9 of the sum of |terms| for
    |tau| = 26 sigma."""
    th = np.array(TRUTH[kind])
    th[1], th[3] = sigma, f_b
    hi, lo = -below * sigma, -(below + 3.5) * sigma
    cols = columns(kind, 1500, 17)
    cols["t"] = np.random.default_rng(5).uniform(lo, hi, 1500)
    check_paths(env, kind, lo, hi, cols, th, 1e-9)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("miss", [0.0, 1e-13, 1e-4])
@pytest.mark.parametrize("kind", KINDS)
def test_signal_terms_all_small(env, kind, miss, weighted):
    """f_b = 1 - miss and a range 9 to 14 sigma under the peak: P is all background, every
    signal term is 1e-4 and less of what the sums' unit is set for, and the derivative in f_b is
    made of them.  1e-9 of the sum of |terms|, as above."""
    th = np.array(TRUTH[kind])
    th[3] = 1.0 - miss
    cols = columns(kind, 700, 19, weighted)
    for lo, hi in ((-12.0, -9.0), (-14.0, -11.0)):
        lo, hi = lo * th[1], hi * th[1]
        cols["t"] = np.random.default_rng(9).uniform(lo, hi, 700)
        check_paths(env, kind, lo, hi, cols, th, 1e-9)


@pytest.mark.parametrize("kind", KINDS)
def test_subnormal_weights(env, kind):
    """Weights of 2^-1030: the terms and partial sums are subnormal and keep 44 bits at unit size;
    the constants that multiply them take up to 2^14 of that: 1e-8 of the sum of |terms|."""
    O, G, torch, api = env
    th = np.array(TRUTH[kind])
    cols = columns(kind, 512, 23)
    unit = gradients(env, kind, 0.0, 15.0, cols, th)
    cols["w"] = np.full(512, 2.0 ** -1030)
    tiny = gradients(env, kind, 0.0, 15.0, cols, th)
    _, terms = O.nll_grad_terms(oracle_model(O, kind, 0.0, 15.0), {k: v for k, v in cols.items() if k != "w"}, th)
    scale = np.abs(terms).sum(1)
    assert np.all(np.abs(np.ldexp(np.ldexp(tiny[1:], 1000), 30) - unit[1:]) <= 1e-8 * scale), (tiny, unit)


def test_cached_columns_add_up_within_their_range(env):
    """Columns of one sign with the coefficients, up to 1.7 each: A' is up to twice eight times its
    largest coefficient.  Late events with background, where P stays positive whatever A' is.
    The whole call, without the odd events, and those alone (fewer than 64: the plain loop)."""
    O, G, torch, api = env
    th = np.array([0.66, 0.045, 0.0, 0.5, 0.3045, 0.3433, 0.439, 1.896, 0.2397, 0.1279])
    h = O.amplitude_coeffs(th)
    IT = O.time_norm(*th[:3], 0.0, 15.0)
    largest = np.abs(h).max() * (1.0 - th[3]) / (IT * O.I_OMEGA) / 2.0
    th[3] = 1.0 - (1.0 - th[3]) * 2.0 ** np.ceil(np.log2(largest)) * 0.98 / largest / 2.0
    m = api.model_4d(0.0, 15.0)
    cols = columns("4d", 200, 29)
    cols["t"][160:] = 14.5
    ev = G.to_dev(cols)
    fk = api.ipa_angular_basis(m, ev)
    for size in (1.2, 1.45, 1.55, 1.7):
        fk[:, 160:] = torch.tensor(size * np.sign(h), device="cuda")[:, None]

        def part(a, b):
            return gradients(env, "4d", 0.0, 15.0, {k: np.ascontiguousarray(v[a:b]) for k, v in cols.items()}, th,
                             cached=fk[:, a:b].contiguous())
        whole, most, few = part(0, 200), part(0, 160), part(160, 200)
        P = (1.0 - th[3]) * O.time_conv(14.5, *th[:2]) / IT * size * np.abs(h).sum() / O.I_OMEGA + th[3] / m_volume(O)
        assert abs(few[0] + 40.0 * np.log(P)) <= 1e-12 * 40.0 * abs(np.log(P))
        logl, terms = O.nll_grad_terms(O.Model("4d", 0.0, 15.0), {k: v[:160] for k, v in cols.items()}, th)
        scale = 2.0 * np.append(np.abs(logl).sum(), np.abs(terms).sum(1)) + np.abs(few)
        assert np.all(np.abs(whole - most - few) <= 1e-12 * scale), (size, whole, most + few)


def m_volume(O):
    return O.Model("4d", 0.0, 15.0).volume
