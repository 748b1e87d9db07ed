"""Paths that only very large calls take: the dense list above 2^28 sites (a key no
longer holds the site and its place) and batches whose labels span more than 2^32
sites (step (iii) carries addresses). The inputs' labels are known in closed form,
except for lattices at both ends of the batch, which the oracle labels."""
import numpy as np
import pytest
import torch

import lattices as L
import oracle
import paper_1603_08357_gb300 as ccl
from ccl_testutil import DEV

pytestmark = pytest.mark.gpu


def _pack(st):
    w = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], dtype=torch.uint8, device=DEV)
    return (st.view(-1, 8) * w).sum(1, dtype=torch.uint8).view(torch.int32)


@pytest.mark.parametrize("n", [(1 << 28) + 32, (1 << 28) + 12_345_696])
def test_dense_list_above_2_28_sites(n):
    """Blocks of 1000 sites, every site joined to the one before or, where that slot
    is closed, to the one before that."""
    c = ccl.ccl_context_create(0)
    i = torch.arange(n, dtype=torch.int32, device=DEV)
    at = i % 1000
    nn = torch.empty(2 * n, dtype=torch.int32, device=DEV)
    nn[:n] = torch.where(at > 0, i - 1, -1)
    nn[n:] = torch.where(at > 1, i - 2, -1)
    bits = torch.full((2 * n // 32,), -1, dtype=torch.int32, device=DEV)
    bits[:n // 32] = _pack(((i % 7 != 3) | (at < 2)).to(torch.uint8))
    want = i - at
    out = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    assert ccl.ccl_label_dense(c, n, 2, nn, bits, out) == ccl.CCL_OK
    assert ccl.ccl_sync(c) == ccl.CCL_OK
    assert bool((out == want).all())
    out.fill_(-1)
    assert ccl.ccl_label_dense_random(c, n, 2, nn, 5, 1.0, out) == ccl.CCL_OK
    assert ccl.ccl_sync(c) == ccl.CCL_OK
    assert bool((out == want).all())
    ccl.ccl_context_destroy(c)


def test_batch_of_labels_more_than_2_32_apart():
    c = ccl.ccl_context_create(0)
    ends = [L.square(2500, 0.5, 3), L.triangle(2500, L.PC_TRIANGLE, 4)]
    most = 2**31 - 4097                                 # isolated sites in between
    ns = [ends[0].n, most, most, ends[1].n]
    so = np.concatenate([[0], np.cumsum(ns, dtype=np.int64)])
    assert so[-1] > 1 << 32
    eo = np.array([0, ends[0].nnz, ends[0].nnz, ends[0].nnz, ends[0].nnz + ends[1].nnz], np.int64)
    rp = torch.zeros(int(so[-1]) + 4, dtype=torch.int32, device=DEV)
    rp[:ns[0] + 1] = torch.from_numpy(ends[0].row_ptr).to(DEV)
    rp[int(so[3]) + 3:] = torch.from_numpy(ends[1].row_ptr).to(DEV)
    ci = torch.from_numpy(np.concatenate([x.col_idx for x in ends])).to(DEV)
    bits = L.pack_bits(np.concatenate([L.unpack_bits(x.open_bits, x.nnz) for x in ends]))
    out = torch.full((int(so[-1]),), -1, dtype=torch.int32, device=DEV)
    assert ccl.ccl_label_batched(c, 4, so, eo, rp, ci, torch.from_numpy(bits.view(np.int32)).to(DEV), out) == ccl.CCL_OK
    assert ccl.ccl_sync(c) == ccl.CCL_OK
    assert ccl.ccl_get_stats(c).reduce_window == 512
    for k, x in ((0, ends[0]), (3, ends[1])):
        assert np.array_equal(out[int(so[k]):int(so[k + 1])].cpu().numpy(), oracle.uf_label(x)), k
    for k in (1, 2):
        for lo in range(0, most, 1 << 28):
            part = out[int(so[k]) + lo:int(so[k]) + min(lo + (1 << 28), most)]
            assert bool((part == torch.arange(lo, lo + part.numel(), dtype=torch.int32, device=DEV)).all())
    ccl.ccl_context_destroy(c)
    del rp, ci, out
    torch.cuda.empty_cache()
