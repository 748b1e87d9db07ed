"""Relabelling, spanning and largest cluster where their kernels change path:
run ends, values that fill a warp and hand over to another, the size limit of
the spanning test's shared-memory set. Integers: equality, no tolerance."""
import numpy as np
import pytest
import torch

import paper_1603_08357_gb300 as ccl
from ccl_testutil import DEV
from oracle import stats

pytestmark = pytest.mark.gpu


def _labels(n, pattern, seed):
    """Canonical labels of n sites (label = smallest site with that label)."""
    rng = np.random.default_rng(seed)
    if pattern == "giant":              # one cluster on nine sites of ten
        raw = np.where(rng.random(n) < 0.9, 0, 1 + np.arange(n))
    elif pattern == "stripes":          # the value that fills the warps changes every 40 sites
        raw = (np.arange(n) // 40) % 7
    elif pattern == "pairs":            # two equal giants (a tie) and singles
        raw = np.where(np.arange(n) % 3 < 2, np.arange(n) % 3, 3 + np.arange(n))
    else:                               # all singles
        raw = np.arange(n)
    order = np.unique(raw, return_index=True, return_inverse=True)
    return order[1][order[2]].astype(np.int32)


@pytest.mark.parametrize("n", [1, 31, 127, 129, 1024, 8191, 8193, 200_003])
@pytest.mark.parametrize("pattern", ["giant", "stripes", "pairs", "singles"])
def test_relabel_and_largest(ctx, n, pattern):
    lab = _labels(n, pattern, n)
    d = torch.from_numpy(lab).to(DEV)
    seq, sizes = torch.full((n,), -1, dtype=torch.int32, device=DEV), torch.full((n,), -1, dtype=torch.int32, device=DEV)
    count, big = torch.zeros(1, dtype=torch.int32, device=DEV), torch.zeros(2, dtype=torch.int32, device=DEV)
    assert ccl.ccl_relabel(ctx, n, d, seq, count, sizes) == ccl.CCL_OK
    assert ccl.ccl_largest_cluster(ctx, n, d, big) == ccl.CCL_OK
    assert ccl.ccl_sync(ctx) == ccl.CCL_OK
    want_seq, want_sizes = stats.sequential(lab)
    assert int(count) == want_sizes.size
    assert np.array_equal(seq.cpu().numpy(), want_seq)
    assert np.array_equal(sizes.cpu().numpy()[:want_sizes.size], want_sizes)
    assert tuple(big.tolist()) == tuple(stats.largest_cluster(lab))


@pytest.mark.parametrize("n_top", [1, 33, 4096, 8192, 8193])
@pytest.mark.parametrize("spans", [False, True])
def test_spanning_set_limit(ctx, n_top, spans):
    n = 40_000
    lab = np.arange(n, dtype=np.int32)                  # singles ...
    top, bottom = np.arange(n_top, dtype=np.int32), np.arange(n - 9000, n, dtype=np.int32)
    if spans:                                           # ... but for two clusters from top to bottom
        lab[bottom[5000]] = top[-1]
        lab[bottom[17]] = top[n_top // 2]
    res = torch.zeros(1, dtype=torch.int32, device=DEV)
    args = [torch.from_numpy(a).to(DEV) for a in (lab, top, bottom)]
    assert ccl.ccl_spanning(ctx, n, args[0], args[1], n_top, args[2], bottom.size, res) == ccl.CCL_OK
    assert ccl.ccl_sync(ctx) == ccl.CCL_OK
    assert int(res) == (int(min(top[-1], top[n_top // 2])) if spans else -1)


def test_relabel_needs_a_count_per_block_only():
    """Scratch of 4 bytes per 8192 sites: a context whose scratch is that large (from
    the largest cluster of 100 sites, 416 bytes) relabels 104 blocks under capture,
    where nothing can be allocated."""
    n = 104 * 8192 - 5
    lab = _labels(n, "pairs", 3)
    c = ccl.ccl_context_create(0)
    s = torch.cuda.Stream()
    d = torch.from_numpy(lab).to(DEV)
    seq, sizes = (torch.full((n,), -1, dtype=torch.int32, device=DEV) for _ in range(2))
    count, big = (torch.zeros(k, dtype=torch.int32, device=DEV) for k in (1, 2))
    torch.cuda.synchronize()
    assert ccl.ccl_largest_cluster(c, 100, d, big, s) == ccl.CCL_OK
    assert ccl.ccl_relabel(c, 100, d, seq, count, sizes, s) == ccl.CCL_OK        # (loads the kernels)
    assert ccl.ccl_sync(c, s) == ccl.CCL_OK
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        assert ccl.ccl_relabel(c, n, d, seq, count, sizes, s) == ccl.CCL_OK
    want_seq, want_sizes = stats.sequential(lab)
    for _ in range(2):
        seq.fill_(-1)
        sizes.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert int(count) == want_sizes.size
        assert np.array_equal(seq.cpu().numpy(), want_seq)
        assert np.array_equal(sizes.cpu().numpy()[:want_sizes.size], want_sizes)
    ccl.ccl_context_destroy(c)


@pytest.mark.parametrize("n_top", [1, 1023, 1025, 8192])
@pytest.mark.parametrize("n_bottom", [1, 8193, 16384, 16385, 70_000])
def test_spanning_scattered_sites(ctx, n_top, n_bottom):
    """Sites anywhere, some twice, some out of range (skipped and latched), on both
    sides of the one-launch path's limits and of a CTA's share of them."""
    n = 300_000
    rng = np.random.default_rng(n_top + n_bottom)
    for spans in (False, True):
        lab = np.arange(n, dtype=np.int32)
        top, bottom = rng.integers(0, n // 2, n_top), rng.integers(n // 2, n, n_bottom)
        if spans:
            lab[bottom[-1]] = top[-1]
            lab[bottom[n_bottom // 2]] = top[n_top // 3]
        for bad in (False, True):
            t, b = top, bottom
            if bad:
                t, b = np.append(t[2:], [n, -1]), np.append(b[1:], n + 7)
            t_in, b_in = t[(t >= 0) & (t < n)], b[b < n]
            common = set(lab[t_in].tolist()) & set(lab[b_in].tolist())
            res = torch.zeros(1, dtype=torch.int32, device=DEV)
            args = [torch.from_numpy(a.astype(np.int32)).to(DEV) for a in (lab, t, b)]
            assert ccl.ccl_spanning(ctx, n, args[0], args[1], t.size, args[2], b.size, res) == ccl.CCL_OK
            assert ccl.ccl_sync(ctx) == (ccl.CCL_ERR_INDEX_OUT_OF_RANGE if bad else ccl.CCL_OK)
            assert int(res) == (min(common) if common else -1)
