"""The generators over many blocks: a toy cut into chunks (many blocks, one
look-back) gives the events of one block walking it alone, bit for bit, and
the oracle's, at the edges of chunks, for ragged and empty toys, for envelopes
that accept too little to be cut, and under stream capture."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COLS = {"1d": ("t",), "4d": ("t", "ck", "cl", "phi"), "tagged": ("t", "q"), "phis": ("t", "ck", "cl", "phi", "q")}
TH4 = [0.66, 0.045, 0.0, 0.1, 0.52, 0.25, 3.2, 3.1, 0.04, 0.3]
THETA = {"1d": TH4[:4], "4d": TH4, "tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3],
         "phis": TH4 + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}
T_LO = {"1d": 0.3, "4d": 0.0, "tagged": 0.0, "phis": 0.0}


def _generate(model, theta, seed, n_sig, n_bkg, stream=None):
    from paper_1706_01420_gb300 import api
    dev = torch.device("cuda")
    m = {"1d": api.model_1d, "4d": api.model_4d, "tagged": api.model_tagged, "phis": api.model_phis}[model](T_LO[model], 15.0)
    n_sig, n_bkg = np.asarray(n_sig, np.int64), np.asarray(n_bkg, np.int64)
    off = np.concatenate([[0], np.cumsum(n_sig + n_bkg)]).astype(np.int64)
    d = lambda a: torch.tensor(a, device=dev)
    out = {k: torch.full((int(off[-1]) + 3,), -7.0, dtype=torch.float64, device=dev) for k in COLS[model]}
    api.ipa_toygen(m, d(np.asarray(theta)), seed, d(n_sig), d(n_bkg), d(off[:-1].copy()), out, stream=stream)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


def _alone(model, theta, seed, n_sig, n_bkg):
    """The same call without a workspace: one block per toy."""
    from paper_1706_01420_gb300 import _capi as C
    from paper_1706_01420_gb300 import api
    old = api.ipa_fault_inject(C.IPA_FAULT_ALLOC)
    try:
        return _generate(model, theta, seed, n_sig, n_bkg)
    finally:
        api.ipa_fault_inject(old)


def _same(a, b):
    return all(np.array_equal(a[k], b[k], equal_nan=True) for k in a)


@pytest.mark.parametrize("model", ["1d", "4d", "tagged", "phis"])
def test_chunks_equal_one_block(model):
    n_sig = [0, 1, 2, 79, 83, 350, 900, 0, 20011, 5, 60000]
    n_bkg = [0, 0, 3, 2047, 2048, 2049, 1, 4100, 0, 7, 33]
    _generate(model, THETA[model], 3, [1], [0])          # the library's scratch is in place
    a = _generate(model, THETA[model], (5 << 40) + 11, n_sig, n_bkg)
    assert _same(a, _alone(model, THETA[model], (5 << 40) + 11, n_sig, n_bkg))
    assert all(np.all(v[-3:] == -7.0) for v in a.values())
    assert all(np.isfinite(v).all() for v in a.values())


@pytest.mark.parametrize("model", ["1d", "4d", "tagged", "phis"])
def test_chunks_equal_the_oracle(model):
    from oracle import ipa_oracle as O
    from oracle import phis, tagged
    kind = "tag" if model == "tagged" else model
    n_sig, n_bkg = [600, 0, 2500], [5, 3, 0]
    for change in ({}, {0: 1.4, 1: 0.15}, {1: 0.012, 2: 0.03}):
        th = np.array(THETA[model])
        for i, v in change.items():
            th[i] = v
        a = _generate(model, th, 77, n_sig, n_bkg)
        m = O.Model(kind, T_LO[model], 15.0)
        toy = {"tagged": tagged.toy_one, "phis": phis.toy_one}.get(model, O.toy_one)
        at = 0
        for k in range(3):
            ref = toy(m, th, 77, k, n_sig[k], n_bkg[k])
            n = n_sig[k] + n_bkg[k]
            assert all(np.array_equal(a[c][at:at + n], ref[c]) for c in COLS[model]), (model, change, k)
            at += n


def test_tickets_of_several_units():
    """Enough work for larger tickets (four units of candidates each)."""
    rng = np.random.default_rng(5)
    n_sig = rng.integers(15000, 35000, 320)
    n_sig[[3, 100]] = 0, 1
    n_bkg = rng.integers(0, 1500, 320)
    _generate("4d", THETA["4d"], 3, [1], [0])
    assert _same(_generate("4d", THETA["4d"], 21, n_sig, n_bkg), _alone("4d", THETA["4d"], 21, n_sig, n_bkg))


def test_low_acceptance_and_bad_parameters():
    _generate("4d", THETA["4d"], 3, [1], [0])
    steep = np.array(THETA["4d"])
    steep[0] = 9.0                                       # a chunk accepts about five events: not cut
    assert _same(_generate("4d", steep, 9, [700, 3], [1, 0]), _alone("4d", steep, 9, [700, 3], [1, 0]))
    bad = np.array(THETA["4d"])
    bad[1] = -1.0                                        # a finite envelope: events, as from one block
    assert _same(_generate("4d", bad, 9, [50, 9000], [4, 4]), _alone("4d", bad, 9, [50, 9000], [4, 4]))
    from oracle import ipa_oracle as O
    ref = O.toy_one(O.Model("4d", 0.0, 15.0), bad, 9, 0, 50, 4)
    a = _generate("4d", bad, 9, [50], [4])
    assert all(np.array_equal(a[k][:54], ref[k]) for k in COLS["4d"])
    bad[1] = np.nan
    a = _generate("4d", bad, 9, [50, 9000], [4, 4])
    assert np.isnan(a["t"][:50]).all() and np.isfinite(a["t"][50:54]).all() and np.isnan(a["phi"][54:9054]).all()


def test_under_stream_capture():
    from paper_1706_01420_gb300 import api
    dev = torch.device("cuda")
    n = 30000
    m = api.model_4d(0.0, 15.0)
    out = {k: torch.zeros(n, dtype=torch.float64, device=dev) for k in COLS["4d"]}
    th = torch.tensor(THETA["4d"], dtype=torch.float64, device=dev)
    i64 = lambda v: torch.tensor([v], dtype=torch.int64, device=dev)
    ns, nb, off = i64(n - 100), i64(100), i64(0)
    api.ipa_toygen(m, th, 5, ns, nb, off, out)
    torch.cuda.synchronize()
    ref = {k: v.clone() for k, v in out.items()}
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            api.ipa_toygen(m, th, 5, ns, nb, off, out, stream=s)
    for _ in range(2):
        for v in out.values():
            v.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(out[k], ref[k]) for k in out)


FIRST_CAPTURED = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_1706_01420_gb300 import api, synth
dev = torch.device("cuda")
th = torch.tensor([0.66, 0.045, 0.0, 0.1, 0.52, 0.25, 3.2, 3.1, 0.04, 0.3], dtype=torch.float64, device=dev)
m = api.model_4d(0.0, 15.0)
ev = {k: torch.tensor(v, device=dev) for k, v in synth.events_4d(1000, 1).items()}
api.ipa_nll_grad(m, ev, th)
n = 30000
out = {k: torch.zeros(n, dtype=torch.float64, device=dev) for k in ("t", "ck", "cl", "phi")}
i64 = lambda v: torch.tensor([v], dtype=torch.int64, device=dev)
ns, nb, off = i64(n - 100), i64(100), i64(0)
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
s = torch.cuda.Stream()
with torch.cuda.stream(s):
    with torch.cuda.graph(g, stream=s):
        api.ipa_toygen(m, th, 5, ns, nb, off, out, stream=s)
g.replay()
torch.cuda.synchronize()
a = {k: v.clone() for k, v in out.items()}
api.ipa_toygen(m, th, 5, ns, nb, off, out)
torch.cuda.synchronize()
assert all(torch.equal(a[k], out[k]) for k in out) and a["t"].min() > 0
print("captured first")
"""


def test_first_call_of_a_process_under_stream_capture():
    """After a likelihood call (which sizes the scratch) the generator's first call may be captured."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FIRST_CAPTURED, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured first" in r.stdout, r.stderr[-2000:]
