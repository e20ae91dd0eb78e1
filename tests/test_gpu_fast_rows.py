"""The fixed-point rows of the 4D likelihood (complete rows of 32 events of a
tile) and their hand-over to the plain loop, against the oracle:

* event counts around a row, a group of four rows, a tile and several tiles;
* every unit of time and scale of weights (the fixed-point sums follow the
  segment's typical r T and the tile's largest weight), with and without
  background, and no signal at all (no fixed-point coefficients);
* a tile in which some r T exceeds the sums' range (A near zero, no background)
  and tiles with events beyond the fitted range (their exponential leaves the
  fixed-point range), both at full accuracy;
* a column of ones gives the bits of no column at all.

Tolerance: each gradient component within 2e-13 of the sum of the absolute
values of the pieces it is built from (the reciprocal's 6e-14, E2's |argument|
2^-53 with arguments up to 50, and the fixed-point units of 2^-48 of a typical
term), the NLL within 1e-14 of sum |w log P|.
"""
import numpy as np
import pytest

from paper_1706_01420_gb300 import synth

pytestmark = pytest.mark.gpu

TH4 = np.array([0.66, 0.045, 0.0, 0.1, 0.52, 0.25, 3.2, 3.1, 0.04, 0.3])
LO, HI = 0.3, 15.0


@pytest.fixture(scope="module")
def env(oracle):
    from tests import gpu_common as G
    G.need_gpu()
    import torch
    from paper_1706_01420_gb300 import api

    def grad(ev, th, lo, hi):
        return api.ipa_nll_grad(api.model_4d(lo, hi), G.to_dev(ev), torch.tensor(th, device="cuda")).cpu().numpy()
    return oracle, G, grad


def compare(env, ev, th, ts=1.0):
    O, G, grad = env
    m = O.Model("4d", LO * ts, HI * ts)
    got = grad(ev, th, LO * ts, HI * ts)
    f, g = O.nll_grad(m, ev, th)
    logl, _ = O.nll_grad_terms(m, ev, th)
    assert abs(got[0] - f) <= 1e-14 * np.abs(logl).sum()
    assert np.all(np.abs(got[1:] - g) <= 2e-13 * G.grad_scale(O, m, ev, th)), (got[1:], g)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n", [31, 32, 33, 127, 128, 129, 160, 511, 512, 513, 545, 16384 + 33])
def test_event_counts(env, n, weighted):
    compare(env, synth.events_4d(n, 41, weighted=weighted), TH4)


@pytest.mark.parametrize("f_b", [0.0, 0.1, 0.999, 1.0])
@pytest.mark.parametrize("ws", [None, 1.0, 1e-30, -3e12])
@pytest.mark.parametrize("ts", [1e-12, 1.0, 1e9])
def test_units_and_weight_scales(env, ts, ws, f_b):
    ev = synth.events_4d(700, 43, weighted=ws is not None)
    ev["t"] = ev["t"] * ts
    if ws is not None:
        ev["w"] = ev["w"] * ws
    th = TH4.copy()
    th[0] /= ts
    th[1:3] *= ts
    th[3] = f_b
    compare(env, ev, th, ts)


def test_handover_to_the_plain_loop(env):
    ev = synth.events_4d(1100, 47)
    th = TH4.copy()
    th[3:6] = 0.0, 1.0 - 2e-6, 1e-6                       # A near cos^2 thK sin^2 thmu, no background
    ev["ck"] = np.where(np.abs(ev["ck"]) < 0.1, 0.1, ev["ck"])
    compare(env, ev, th)
    ev["ck"][700] = 2.0 ** -13                            # r T 2^17 times the typical one: its tile is redone
    compare(env, ev, th)
    ev = synth.events_4d(1100, 53)
    ev["t"][[5, 600]] = 40.0, 16.5                        # beyond t_hi
    compare(env, ev, TH4)


def test_unit_weights_are_no_weights(env):
    _, _, grad = env
    ev = synth.events_4d(1500, 59)
    ev["ck"][77] = 1.0
    assert np.array_equal(grad(ev, TH4, LO, HI), grad({**ev, "w": np.ones(1500)}, TH4, LO, HI))


@pytest.mark.parametrize("ts", [1e-12, 1.0, 1e9])
@pytest.mark.parametrize("kind", ["tagged", "phis"])
def test_time_functions_and_their_range(env, kind, ts):
    """The tagged and phi_s models' exponentials and phase are linear in t in fixed
    point over the fitted range, in any unit of time; events beyond it take the
    general functions.  Tolerance: 5e-13 of the sum of |terms| (the terms of one
    component can cancel among themselves by a factor of a few)."""
    O, G, _ = env
    import torch
    from paper_1706_01420_gb300 import api
    th = np.array({"tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3],
                   "phis": list(TH4) + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}[kind])
    first = 4 if kind == "tagged" else 10                 # DG, Dm
    ev = {"tagged": synth.events_tagged, "phis": synth.events_phis}[kind](700, 61)
    ev["t"][[3, 40, 600]] = 17.0, 40.0, 16.0              # beyond t_hi = 15 and beyond 16, the power of two above
    ev["t"] = ev["t"] * ts
    th[[0, first, first + 1]] /= ts
    th[1:3] *= ts
    got = api.ipa_nll_grad(getattr(api, "model_" + kind)(0.0, HI * ts), G.to_dev(ev),
                                       torch.tensor(th, device="cuda")).cpu().numpy()
    m = O.Model("tag" if kind == "tagged" else "phis", 0.0, HI * ts)
    f, g = O.nll_grad(m, ev, th)
    logl, terms = O.nll_grad_terms(m, ev, th)
    assert abs(got[0] - f) <= 1e-14 * np.abs(logl).sum()
    assert np.all(np.abs(got[1:] - g) <= 5e-13 * np.abs(terms).sum(1)), (got[1:], g)


@pytest.mark.parametrize("ws", [None, 1e-30, -3e12])
@pytest.mark.parametrize("kind", ["tagged", "phis"])
def test_time_models_weight_scales_and_handover(env, kind, ws):
    """The tagged and phi_s models' integer sums follow the scale of the weights; a
    warp's rows with a factor beyond the sums' range (phi_s: all angular products
    near zero and no background) are redone.  Tolerance as above."""
    O, G, _ = env
    import torch
    from paper_1706_01420_gb300 import api
    th = np.array({"tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3],
                   "phis": list(TH4) + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}[kind])
    th[3] = 0.0
    ev = {"tagged": synth.events_tagged, "phis": synth.events_phis}[kind](1100, 67, weighted=ws is not None)
    if ws is not None:
        ev["w"] = ev["w"] * ws
        ev["w"][[9, 300]] = 0.0, ws
    if kind == "phis":
        ev["ck"][5] = ev["cl"][5] = 1.0 - 2.0 ** -16
        ev["ck"][600] = 1.0 - 2.0 ** -18                  # the FP64 basis
    got = api.ipa_nll_grad(getattr(api, "model_" + kind)(0.0, HI), G.to_dev(ev),
                           torch.tensor(th, device="cuda")).cpu().numpy()
    m = O.Model("tag" if kind == "tagged" else "phis", 0.0, HI)
    f, g = O.nll_grad(m, ev, th)
    logl, terms = O.nll_grad_terms(m, ev, th)
    assert abs(got[0] - f) <= 1e-14 * np.abs(logl).sum()
    assert np.all(np.abs(got[1:] - g) <= 5e-13 * np.abs(terms).sum(1)), (got[1:], g)


@pytest.mark.parametrize("redo", [False, True])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kind", ["1d", "4d", "tagged"])
def test_one_warp_or_a_team_per_tile(env, kind, weighted, redo):
    """A tile's four quarters taken by one warp or by the four of a team give the
    same bits, on the fixed-point path and where a tile is redone (P below the Newton
    reciprocal's range); the values against the oracle (tolerance as above)."""
    O, G, _ = env
    import torch
    from paper_1706_01420_gb300 import api
    th = np.array({"1d": TH4[:4], "4d": TH4, "tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3]}[kind])
    th[3] = 0.0 if redo else th[3]
    m = getattr(api, "model_" + kind)(-2.0, HI)
    mo = O.Model("tag" if kind == "tagged" else kind, -2.0, HI)
    theta = torch.tensor(th, device="cuda")
    for n in (1, 63, 64, 129, 385, 512, 545, 1537):
        if kind == "1d":
            cols = {"t": synth.events_1d(n, 71, t_lo=0.0)}
            if weighted:
                cols["w"] = synth.weights(n, 73)
        else:
            cols = {"4d": synth.events_4d, "tagged": synth.events_tagged}[kind](n, 71, weighted=weighted)
        if redo:
            cols["t"][n // 2] = -1.1                      # 24 sigma before the edge: P near 1e-130
        ev = G.to_dev(cols)
        got = {}
        try:
            for warps in (1, 2):
                api.ipa_launch_config_set(m, n, {"warps_per_block": warps, "warps_per_sm": 0, "tiles_per_take": 1})
                got[warps] = api.ipa_nll_grad(m, ev, theta).cpu().numpy()
        finally:
            api.ipa_launch_config_set(m, n, {"warps_per_block": 1, "warps_per_sm": 0, "tiles_per_take": 1})
        assert np.array_equal(got[1], got[2]), n
        f, g = O.nll_grad(mo, cols, th)
        logl, terms = O.nll_grad_terms(mo, cols, th)
        assert abs(got[1][0] - f) <= 1e-14 * np.abs(logl).sum(), n
        assert np.all(np.abs(got[1][1:] - g) <= 5e-13 * np.abs(terms).sum(1)), n


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kind", ["4d", "phis"])
def test_cached_basis_rows(env, kind, weighted):
    """The cached basis on the fixed-point path: one warp or a team per tile give the
    same bits, the values are the oracle's (tolerance as above), and basis values
    beyond the path's range (1.75) go by the plain loop, as they are."""
    O, G, _ = env
    import torch
    from paper_1706_01420_gb300 import api
    th = np.array({"4d": TH4, "phis": list(TH4) + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}[kind])
    m = getattr(api, "model_" + kind)(0.0, HI)
    theta = torch.tensor(th, device="cuda")
    mo = O.Model(kind, 0.0, HI)
    for n in (63, 64, 545, 1537):
        cols = {"4d": synth.events_4d, "phis": synth.events_phis}[kind](n, 79, weighted=weighted)
        ev = G.to_dev(cols)
        ev["fk"] = api.ipa_angular_basis(m, ev)
        got = {}
        try:
            for warps in (1, 2):
                api.ipa_launch_config_set(m, n, {"warps_per_block": warps, "warps_per_sm": 0, "tiles_per_take": 1},
                                          cached=True)
                got[warps] = api.ipa_nll_grad(m, ev, theta).cpu().numpy()
        finally:
            api.ipa_launch_config_set(m, n, {"warps_per_block": 1, "warps_per_sm": 0, "tiles_per_take": 1}, cached=True)
        assert np.array_equal(got[1], got[2]), n
        f, g = O.nll_grad(mo, cols, th)
        logl, terms = O.nll_grad_terms(mo, cols, th)
        assert abs(got[1][0] - f) <= 1e-14 * np.abs(logl).sum(), n
        assert np.all(np.abs(got[1][1:] - g) <= 5e-13 * np.abs(terms).sum(1)), n
        # without background P is proportional to the basis: scaling it by 8 shifts the NLL by
        # -sum w ln 8 and leaves the gradient as it is
        th0 = th.copy()
        th0[3] = 0.0
        t0 = torch.tensor(th0, device="cuda")
        ref = api.ipa_nll_grad(m, ev, t0).cpu().numpy()
        ev["fk"] = ev["fk"] * 8.0
        big = api.ipa_nll_grad(m, ev, t0).cpu().numpy()
        _, terms = O.nll_grad_terms(mo, cols, th0)
        w = cols["w"] if weighted else np.ones(n)
        labs = np.abs(O.nll_grad_terms(mo, cols, th0)[0]).sum() + np.abs(w).sum() * np.log(8.0)
        assert abs(big[0] - (ref[0] - w.sum() * np.log(8.0))) <= 2e-14 * labs, n
        keep = np.arange(len(th0)) != 3                   # (the derivative in f_b scales with the basis)
        assert np.all(np.abs(big[1:] - ref[1:])[keep] <= 5e-13 * np.abs(terms).sum(1)[keep]), n


@pytest.mark.parametrize("kind", ["1d", "4d", "tagged", "phis"])
def test_weights_of_changing_scale_over_a_tile(env, kind):
    """The integer sums' scale follows the largest weight so far: weights that are zero
    for a quarter of a tile, then grow by 2^40 over it, then fall again.  One warp
    and a team per tile give the same bits; values as above."""
    O, G, _ = env
    import torch
    from paper_1706_01420_gb300 import api
    th = np.array({"1d": TH4[:4], "4d": TH4, "tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3],
                   "phis": list(TH4) + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}[kind])
    m = getattr(api, "model_" + kind)(0.0, HI)
    mo = O.Model("tag" if kind == "tagged" else kind, 0.0, HI)
    theta = torch.tensor(th, device="cuda")
    n = 1100
    if kind == "1d":
        cols = {"t": synth.events_1d(n, 83, t_lo=0.0)}
    else:
        cols = {"4d": synth.events_4d, "tagged": synth.events_tagged, "phis": synth.events_phis}[kind](n, 83)
    i = np.arange(n)
    cols["w"] = np.where(i < 128, 0.0, np.where(i < 512, 2.0 ** ((i - 512) / 10.0), 2.0 ** (-(i - 512) / 20.0)))
    ev = G.to_dev(cols)
    got = {}
    try:
        for warps in (1, 2):
            api.ipa_launch_config_set(m, n, {"warps_per_block": warps, "warps_per_sm": 0, "tiles_per_take": 1})
            got[warps] = api.ipa_nll_grad(m, ev, theta).cpu().numpy()
    finally:
        api.ipa_launch_config_set(m, n, {"warps_per_block": 1, "warps_per_sm": 0, "tiles_per_take": 1})
    assert np.array_equal(got[1], got[2])
    f, g = O.nll_grad(mo, cols, th)
    logl, terms = O.nll_grad_terms(mo, cols, th)
    assert abs(got[1][0] - f) <= 1e-14 * np.abs(logl).sum()
    assert np.all(np.abs(got[1][1:] - g) <= 5e-13 * np.abs(terms).sum(1))


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kind", ["4d", "phis"])
@pytest.mark.parametrize("bad", [(1.5, 0.2, 0.1), (0.1, -1.5, 0.1), (0.2, 0.1, np.nan), (np.nan, 0.1, 0.2),
                                 (0.2, np.inf, 0.1), (3.0, 3.0, 0.4), (-3.0, 2.0, 1.4)])
def test_angles_outside_their_domain(env, kind, weighted, bad):
    """One event whose angles lie outside the domain (|cos| > 1, not a number): the values
    are those of the plain loop, which takes a call of fewer than 64 events, NaN or not.
    With both |cos| > 1 the basis values are finite and up to 72; at late t with background
    P stays positive.  Tolerance: 5e-13 of the sum of |terms| for each of the three calls."""
    O, G, _ = env
    import torch
    from paper_1706_01420_gb300 import api
    th = np.array({"4d": TH4, "phis": list(TH4) + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}[kind])
    th[3] = 0.5
    m = getattr(api, "model_" + kind)(0.0, HI)
    cols = {"4d": synth.events_4d, "phis": synth.events_phis}[kind](200, 89, weighted=weighted)
    cols["t"][170] = 14.5
    cols["ck"][170], cols["cl"][170], cols["phi"][170] = bad

    def grad(a, b):
        ev = G.to_dev({k: np.ascontiguousarray(v[a:b]) for k, v in cols.items()})
        return api.ipa_nll_grad(m, ev, torch.tensor(th, device="cuda")).cpu().numpy()
    whole, most, few = grad(0, 200), grad(0, 160), grad(160, 200)
    assert np.isfinite(most).all()
    assert np.array_equal(np.isnan(whole), np.isnan(few)), (whole, few)
    assert np.isnan(few[0]) == (max(abs(bad[0]), abs(bad[1])) != 3.0)
    logl, terms = O.nll_grad_terms(O.Model(kind, 0.0, HI), {k: v[:160] for k, v in cols.items()}, th)
    scale = 2.0 * np.append(np.abs(logl).sum(), np.abs(terms).sum(1)) + np.abs(few)
    ok = ~np.isnan(few)
    assert np.all(np.abs(whole - most - few)[ok] <= 1e-12 * scale[ok]), (whole, most + few)
