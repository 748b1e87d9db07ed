"""Corrupt row pointers: reported by ccl_sync, never followed. The labels of such
a call are only promised to be sites; the context labels correctly afterwards."""
import numpy as np
import pytest
import torch

import lattices as L
import oracle
import paper_1603_08357_gb300 as ccl
from ccl_testutil import gpu_label

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
