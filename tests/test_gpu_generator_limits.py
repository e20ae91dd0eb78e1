"""The generators where the work is cut differently: envelopes that accept one candidate in
a thousand to one in a million (tickets of many units), buffers far larger than the events,
and calls of few events per toy.  The events are those of a warp per toy without a
workspace, bit for bit, and the rest of the buffer stays as it was."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COLS = {"1d": ("t",), "4d": ("t", "ck", "cl", "phi"), "tagged": ("t", "q"), "phis": ("t", "ck", "cl", "phi", "q")}
TH4 = [0.66, 0.045, 0.0, 0.1, 0.52, 0.25, 3.2, 3.1, 0.04, 0.3]
THETA = {"1d": TH4[:4], "4d": TH4, "tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3],
         "phis": TH4 + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}


@pytest.fixture(scope="module")
def api():
    from tests import gpu_common as G
    G.need_gpu()
    from paper_1706_01420_gb300 import api
    return api


def generate(api, kind, hi, seed, n_sig, n_bkg, room=0):
    m = getattr(api, "model_" + kind)(0.0, hi)
    n_sig, n_bkg = np.asarray(n_sig, np.int64), np.asarray(n_bkg, np.int64)
    off = np.concatenate([[0], np.cumsum(n_sig + n_bkg)]).astype(np.int64)
    out = {k: torch.full((int(off[-1]) + room,), -7.0, dtype=torch.float64, device="cuda") for k in COLS[kind]}
    dev = [torch.tensor(a, device="cuda") for a in (n_sig, n_bkg, off[:-1].copy())]
    api.ipa_toygen(m, torch.tensor(THETA[kind], dtype=torch.float64, device="cuda"), seed, *dev, out)
    torch.cuda.synchronize()
    assert all(bool((v[int(off[-1]):] == -7.0).all()) for v in out.values())
    return {k: v[:int(off[-1])].cpu().numpy() for k, v in out.items()}


def without_workspace(api, *args, **kw):
    from paper_1706_01420_gb300 import _capi as C
    old = api.ipa_fault_inject(C.IPA_FAULT_ALLOC)
    try:
        return generate(api, *args, **kw)
    finally:
        api.ipa_fault_inject(old)


def same(a, b):
    return all(np.array_equal(a[k], b[k]) for k in a)


@pytest.mark.parametrize("kind, hi", [("1d", 3e4), ("1d", 1e6), ("tagged", 3e4), ("4d", 3e3), ("4d", 3e4)])
def test_tickets_of_many_units(api, kind, hi):
    n_sig = [40, 0, 3, 17] if hi < 1e5 else [2, 1]
    n_bkg = [2, 700, 0, 1][:len(n_sig)]
    generate(api, kind, 15.0, 3, [1], [0])               # the library's scratch is in place
    a = generate(api, kind, hi, 41, n_sig, n_bkg)
    assert all(np.isfinite(v).all() for v in a.values())
    assert same(a, without_workspace(api, kind, hi, 41, n_sig, n_bkg))


@pytest.mark.parametrize("kind", list(COLS))
def test_buffers_larger_than_the_events(api, kind):
    """The workspace follows the events, not the buffers alone: the same events in 3e7 of room,
    and a batch of many toys in buffers of its own size."""
    generate(api, kind, 15.0, 3, [1], [0])
    n_sig, n_bkg = [900, 0, 20000], [5, 1000, 0]
    a = generate(api, kind, 15.0, 43, n_sig, n_bkg, room=30_000_000)
    assert same(a, generate(api, kind, 15.0, 43, n_sig, n_bkg))
    rng = np.random.default_rng(3)
    n_sig = rng.integers(0, 4000, 3000)
    n_bkg = rng.integers(0, 40, 3000)
    assert same(generate(api, kind, 15.0, 47, n_sig, n_bkg), without_workspace(api, kind, 15.0, 47, n_sig, n_bkg))


@pytest.mark.parametrize("toys, most", [(1, 1), (1, 130), (1, 450), (3, 460), (600, 90), (700, 3), (3000, 60), (6000, 40)])
def test_few_events_per_toy(api, toys, most):
    """1D calls of few events: a block per toy, by the room of the buffers, a warp where there are
    more toys than warps; the events are those of the tickets, which the same call takes in
    buffers of ample room, and the oracle's."""
    from oracle import ipa_oracle as O
    rng = np.random.default_rng(toys + most)
    n_sig, n_bkg = rng.integers(0, most + 1, toys), rng.integers(0, most // 8 + 1, toys)
    n_sig[0], n_bkg[0] = most, most // 9
    generate(api, "1d", 15.0, 3, [1], [0])
    a = generate(api, "1d", 15.0, (3 << 34) + 5, n_sig, n_bkg)
    assert same(a, generate(api, "1d", 15.0, (3 << 34) + 5, n_sig, n_bkg, room=1000 * toys + 1))
    ref = O.toy_one(O.Model("1d", 0.0, 15.0), np.array(THETA["1d"]), (3 << 34) + 5, 0, most, most // 9)
    assert np.array_equal(a["t"][:most + most // 9], ref["t"])


@pytest.mark.parametrize("sigma", [np.nan, -1.0])
def test_few_events_and_bad_parameters(api, sigma):
    m = api.model_1d(0.0, 15.0)
    th = torch.tensor([0.66, sigma, 0.0, 0.1], dtype=torch.float64, device="cuda")
    got = {}
    i64 = lambda v: torch.tensor([v], dtype=torch.int64, device="cuda")
    for room in (70, 5000):
        t = torch.full((room,), -7.0, dtype=torch.float64, device="cuda")
        api.ipa_toygen(m, th, 9, i64(60), i64(10), i64(0), {"t": t})
        got[room] = t.cpu().numpy()
    assert np.array_equal(got[70], got[5000][:70], equal_nan=True)
    assert np.all(got[5000][70:] == -7.0) and np.isfinite(got[70][60:]).all()
