"""Corrupt row pointers: reported by ccl_sync, never followed. The labels of such
a call are only promised to be sites; the context labels correctly afterwards."""
import numpy as np
import pytest
import torch

import lattices as L
import oracle
import paper_1603_08357_gb300 as ccl
from ccl_testutil import DEV, gpu_label, gpu_label_batched

pytestmark = pytest.mark.gpu


def _rows(n, degrees, seed, p=0.5):
    rng = np.random.default_rng(seed)
    rp = np.concatenate([[0], np.cumsum(degrees)]).astype(np.int32)
    col = rng.integers(0, n, int(rp[-1])).astype(np.int32)
    return L.Lattice("random", n, int(rp[-1]), rp, col, L.pack_bits(rng.random(int(rp[-1])) < p), p, seed)


@pytest.mark.parametrize("degree", [3, 4, 6, 5, 0])
@pytest.mark.parametrize("first", [2**31 - 1 - 60, 2**31 - 1 - 2000, -70])
def test_row_pointers_around_the_type_limit(ctx, degree, first):
    """The 128 rows of one warp moved to the end of int32 (past it they wrap) or
    below zero, in steps that are rows of one degree (0: mixed), between valid
    tile boundaries."""
    n = 4096
    deg = np.full(n, degree) if degree else np.random.default_rng(1).integers(0, 9, n)
    lat = _rows(n, deg, 5)
    rp = lat.row_ptr.astype(np.int64)
    s = 1024 + 128
    rp[s:s + 129] += first - rp[s]
    wrapped = rp.astype(np.uint32).view(np.int32)
    bad = L.Lattice("random", n, lat.nnz, wrapped, lat.col_idx, lat.open_bits, 0.5, 0)
    got = gpu_label(ctx, bad, expect_status=ccl.CCL_ERR_INDEX_OUT_OF_RANGE)
    assert got.min() >= 0 and got.max() < n
    assert np.array_equal(gpu_label(ctx, lat), oracle.uf_label(lat))


def _overfull(n, nnz):
    """Rows that alternate between all entries and none backwards: every other row
    reads the whole list of open bonds to site 0, far more pairs than entries."""
    rp = np.where(np.arange(n + 1) % 2, nnz, 0).astype(np.int32)
    rp[-1] = nnz
    return L.Lattice("random", n, nnz, rp, np.zeros(nnz, np.int32), L.pack_bits(np.ones(nnz, bool)), 1.0, 0)


def _batch(lats):
    so = np.concatenate([[0], np.cumsum([x.n for x in lats])])
    eo = np.concatenate([[0], np.cumsum([x.nnz for x in lats])])
    bits = L.pack_bits(np.concatenate([L.unpack_bits(x.open_bits, x.nnz) for x in lats]))
    rp, ci = (np.concatenate(a).astype(np.int32) for a in ([x.row_ptr for x in lats], [x.col_idx for x in lats]))
    return L.Batch(so, eo, rp, ci, bits, [{"kind": "random"}] * len(lats))


@pytest.mark.parametrize("sites", [1024, 3000])
@pytest.mark.parametrize("far", [0, 1])
def test_overfull_rows_in_a_batch(sites, far):
    """Pairs of the corrupt instance run over the queue slots of its neighbours,
    whose sites are fewer: beside small instances (pairs set aside) and with the
    in-order hand-out (slots)."""
    c = ccl.ccl_context_create(0)
    try:
        if far:
            assert ccl.ccl_set_option(c, ccl.CCL_OPT_REFILL, 0) == ccl.CCL_OK
        good = [_rows(n, np.full(n, 3), n) for n in (40, 2000, 7, 300)]
        b = _batch([good[0], _overfull(sites, 4000), good[1], _overfull(sites, 4000), good[2], good[3]])
        for _ in range(3):
            dev = [torch.from_numpy(a).to(DEV) for a in (b.row_ptr, b.col_idx, b.open_bits.view(np.int32))]
            out = torch.zeros(b.n_total, dtype=torch.int32, device=DEV)
            assert ccl.ccl_label_batched(c, b.k, b.site_off, b.ent_off, *dev, out) == ccl.CCL_OK
            assert ccl.ccl_sync(c) == ccl.CCL_ERR_INDEX_OUT_OF_RANGE
            got = out.cpu().numpy()
            for k in range(b.k):
                lab = got[b.site_off[k]:b.site_off[k + 1]]
                assert lab.min() >= 0 and lab.max() < lab.size
        ok = _batch(good)
        got = gpu_label_batched(c, ok)
        for k, x in enumerate(good):
            assert np.array_equal(got[ok.site_off[k]:ok.site_off[k + 1]], oracle.uf_label(x))
    finally:
        ccl.ccl_context_destroy(c)


def test_overfull_batch_after_a_larger_single_call():
    """The workspace's pairs grown by a single instance, the pairs' instance numbers
    (only batches have them) not: a corrupt batch stays inside both."""
    c = ccl.ccl_context_create(0)
    try:
        big = L.triangle(1200, 0.4, 3)
        assert np.array_equal(gpu_label(c, big), oracle.uf_label(big))
        good = _rows(300, np.full(300, 3), 2)
        b = _batch([_overfull(1024, 4000), good, _overfull(3000, 4000)])
        dev = [torch.from_numpy(a).to(DEV) for a in (b.row_ptr, b.col_idx, b.open_bits.view(np.int32))]
        out = torch.zeros(b.n_total, dtype=torch.int32, device=DEV)
        assert ccl.ccl_label_batched(c, b.k, b.site_off, b.ent_off, *dev, out) == ccl.CCL_OK
        assert ccl.ccl_sync(c) == ccl.CCL_ERR_INDEX_OUT_OF_RANGE
        assert np.array_equal(gpu_label(c, big), oracle.uf_label(big))
    finally:
        ccl.ccl_context_destroy(c)
