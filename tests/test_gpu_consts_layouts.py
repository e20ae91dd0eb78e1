"""The parameter records of many fits, a block per fit (up to 1024) or a thread
per fit (beyond): both layouts give the same bits, so the results of the first
1024 fits do not change when one more is added to the call."""
import numpy as np
import pytest

from paper_1706_01420_gb300 import synth

pytestmark = pytest.mark.gpu

TH4 = [0.66, 0.045, 0.0, 0.1, 0.52, 0.25, 3.2, 3.1, 0.04, 0.3]
MODELS = {"1d": TH4[:4], "4d": TH4, "tagged": [0.66, 0.045, 0.0, 0.1, 0.085, 17.77, 0.8, 0.3],
          "phis": TH4 + [0.085, 17.77, 0.8, 0.3, 0.8, 0.0]}


@pytest.mark.parametrize("kind", list(MODELS))
def test_block_and_thread_layouts_agree(kind):
    from tests import gpu_common as G
    G.need_gpu()
    import torch
    from paper_1706_01420_gb300 import api
    n_seg, per = 1025, 3
    n = n_seg * per
    cols = {"1d": lambda: {"t": synth.events_1d(n, 3, t_lo=0.0)}, "4d": lambda: synth.events_4d(n, 3),
            "tagged": lambda: synth.events_tagged(n, 3), "phis": lambda: synth.events_phis(n, 3)}[kind]()
    ev = G.to_dev(cols)
    m = getattr(api, "model_" + kind)(0.0, 15.0)
    rng = np.random.default_rng(7)
    th = np.tile(MODELS[kind], (n_seg, 1)) * (1.0 + 0.02 * rng.uniform(-1, 1, (n_seg, len(MODELS[kind]))))
    th[5, 1] = -1.0                                       # outside the domain
    th = torch.tensor(th, device="cuda")
    off = torch.arange(n_seg + 1, device="cuda", dtype=torch.int64) * per
    thread = api.ipa_nll_grad_segmented(m, ev, off, th).cpu().numpy()
    block = api.ipa_nll_grad_segmented(m, {k: v[:n - per] for k, v in ev.items()}, off[:-1].clone(),
                                       th[:-1].clone()).cpu().numpy()
    assert np.array_equal(thread[:-1], block, equal_nan=True)


@pytest.mark.parametrize("kind, cached", [("1d", False), ("4d", False), ("4d", True), ("tagged", False), ("phis", False),
                                          ("phis", True)])
def test_layouts_agree_on_the_fixed_point_rows(kind, cached):
    """The same with 70 and 129 events per fit, which read every field of the records that the
    fixed-point rows use (fewer than 64 take the plain loop), and with the cached basis."""
    from tests import gpu_common as G
    G.need_gpu()
    import torch
    from paper_1706_01420_gb300 import api
    n_seg = 1025
    sizes = np.where(np.arange(n_seg) % 3 == 0, 129, 70)
    n = int(sizes.sum())
    cols = {"1d": lambda: {"t": synth.events_1d(n, 5, t_lo=0.0)}, "4d": lambda: synth.events_4d(n, 5),
            "tagged": lambda: synth.events_tagged(n, 5), "phis": lambda: synth.events_phis(n, 5)}[kind]()
    ev = G.to_dev(cols)
    m = getattr(api, "model_" + kind)(0.0, 15.0)
    rng = np.random.default_rng(11)
    th = np.tile(MODELS[kind], (n_seg, 1)) * (1.0 + 0.02 * rng.uniform(-1, 1, (n_seg, len(MODELS[kind]))))
    th = torch.tensor(th, device="cuda")
    off = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]), device="cuda")
    last = int(sizes[:-1].sum())
    few = {k: v[:last] for k, v in ev.items()}
    if cached:
        ev["fk"], few["fk"] = api.ipa_angular_basis(m, ev), api.ipa_angular_basis(m, few)
    thread = api.ipa_nll_grad_segmented(m, ev, off, th).cpu().numpy()
    block = api.ipa_nll_grad_segmented(m, few, off[:-1].clone(), th[:-1].clone()).cpu().numpy()
    assert np.isfinite(block).all() and np.array_equal(thread[:-1], block)
