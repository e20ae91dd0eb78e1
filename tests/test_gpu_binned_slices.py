"""The CLs kernel over slices of bins and the Poisson threshold tables, at the
edges of their ranges: one bin, a slice less and more than full, a toy block
less and more than full, tables of one entry (tiny means), long tables, means
split into pieces, bins without background.  Counts equal the oracle's; X within
1e-12 relative (sums of a few hundred terms in another order: below 1e-13)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bins,n_toys", [(1, 40), (63, 5), (64, 128), (65, 129), (300, 127), (1000, 300)])
def test_slices_match_oracle(n_bins, n_toys):
    import torch

    from oracle import binned as B
    from paper_1706_01420_gb300 import api
    rng = np.random.default_rng(n_bins)
    s, b = rng.exponential(0.3, n_bins), rng.exponential(2.0, n_bins) + 0.01
    if n_bins > 64:
        b[3], b[40], b[63], b[5], b[6] = 30.0, 500.0, 390.0, 1e-17, 1e-9
        s[5] = s[6] = 1e-9
    d = rng.poisson(b + s).astype(np.int32)
    cl, counts, (xb, xsb, xo) = B.cls(s, b, d, n_toys, 9)
    r = api.ipa_cls(*(torch.tensor(x, device="cuda") for x in (s, b, d)), n_toys, 9, with_x=True)
    assert tuple(r["counts"].cpu().numpy()) == counts
    np.testing.assert_array_equal([float(r["cl_b"]), float(r["cl_sb"]), float(r["cl_s"])], cl)
    np.testing.assert_allclose(r["x_b"].cpu().numpy(), xb, rtol=1e-12)
    np.testing.assert_allclose(r["x_sb"].cpu().numpy(), xsb, rtol=1e-12)
    np.testing.assert_allclose(float(r["x_obs"]), xo, rtol=1e-12)


def test_bin_without_background_counts_only_its_events():
    import torch

    from oracle import binned as B
    from paper_1706_01420_gb300 import api
    s, b = np.full(70, 0.02), np.full(70, 1.5)
    b[[0, 65]] = 0.0
    d = np.ones(70, dtype=np.int32)
    d[[0, 65]] = 0
    r = api.ipa_cls(*(torch.tensor(x, device="cuda") for x in (s, b, d)), 200, 4, with_x=True)
    x_sb, x_b = r["x_sb"].cpu().numpy(), r["x_b"].cpu().numpy()
    assert np.isfinite(x_b).all() and np.isfinite(float(r["x_obs"]))
    for k in range(200):
        n = B.generate_binned_fast(s + b, 4, k, 1)
        assert np.isfinite(x_sb[k]) == (n[0] == 0 and n[65] == 0)


def test_tables_where_memory_is_short():
    """Tables of 256 bytes a bin do not fit, those of the entries alone do: the same counts."""
    from tests import gpu_common as G
    G.need_gpu()
    import torch
    from paper_1706_01420_gb300 import api
    n = 30_000_000
    lam = torch.rand(n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3)) * 0.6
    ref = api.ipa_binned_generate(lam, 11, 1)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    try:
        ballast = torch.empty(free - (6 << 30), dtype=torch.uint8, device="cuda")
    except torch.cuda.OutOfMemoryError:
        pytest.skip("the card's free memory cannot be held")
    try:
        got = api.ipa_binned_generate(lam, 11, 1)
        assert torch.equal(got, ref)
    finally:
        del ballast
        torch.cuda.empty_cache()
