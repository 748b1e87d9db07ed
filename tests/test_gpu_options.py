"""Options and tuning where the library has a choice of its own: it can be read,
written back and had again, and tuning on one input does not take it away."""
import numpy as np
import pytest
import torch

import lattices as L
import oracle
import paper_1603_08357_gb300 as ccl
from ccl_testutil import DEV, gpu_label, gpu_label_batched, to_dev

pytestmark = pytest.mark.gpu

OPTIONS = [getattr(ccl, f"CCL_OPT_{n}") for n in (
    "PRE_ANALYSIS", "BLOCK_THREADS", "CTAS_PER_SM", "LINK_MODE", "REFILL", "ANALYSIS_ORDER", "ITER_CAP",
    "REDUCE_WINDOW", "ANALYSIS_GROUP", "ANALYSIS_PARK")]


@pytest.fixture
def fresh():
    c = ccl.ccl_context_create(0)
    yield c
    ccl.ccl_context_destroy(c)


def test_step_ii_by_sample_can_be_read_and_set(fresh):
    opt = ccl.CCL_OPT_PRE_ANALYSIS
    assert ccl.ccl_get_option(fresh, opt) == -1
    for v, reads in ((1, 1), (0, 0), (-1, -1), (5, 1), (-1, -1)):
        assert ccl.ccl_set_option(fresh, opt, v) == ccl.CCL_OK
        assert ccl.ccl_get_option(fresh, opt) == reads


@pytest.mark.parametrize("opt", OPTIONS)
def test_writing_back_what_was_read_changes_nothing(fresh, opt):
    v = ccl.ccl_get_option(fresh, opt)
    assert ccl.ccl_set_option(fresh, opt, v) == ccl.CCL_OK
    assert ccl.ccl_get_option(fresh, opt) == v


def test_statistics_tell_how_step_ii_ran(fresh):
    """By sample (-1), also where it walks (honeycomb at 1.5 p_c, long chains)."""
    lats = [L.honeycomb(750, p, 3) for p in (L.PC_HONEYCOMB, 1.5 * L.PC_HONEYCOMB)]
    for setting in (-1, 0, 1, -1):
        assert ccl.ccl_set_option(fresh, ccl.CCL_OPT_PRE_ANALYSIS, setting) == ccl.CCL_OK
        for lat in lats:
            assert np.array_equal(gpu_label(fresh, lat), oracle.uf_label(lat))
            assert ccl.ccl_get_stats(fresh).pre_analysis == setting


def _supercritical():
    return L.honeycomb(750, 1.5 * L.PC_HONEYCOMB, 3)       # 1,125,000 sites of degree 3: size class 20 * 1024 + 3


def test_tuning_at_the_threshold_keeps_the_sample_for_other_sizes(fresh):
    lat = L.triangle(256, L.PC_TRIANGLE, 3)
    rp, ci, bits = to_dev(lat)
    out = torch.empty(lat.n, dtype=torch.int32, device=DEV)
    st, _ = ccl.ccl_autotune(fresh, lat.n, lat.nnz, rp, ci, bits, out)
    assert st == ccl.CCL_OK
    assert ccl.ccl_get_option(fresh, ccl.CCL_OPT_PRE_ANALYSIS) == -1
    other = _supercritical()
    assert np.array_equal(gpu_label(fresh, other), oracle.uf_label(other))
    assert ccl.ccl_get_stats(fresh).pre_analysis == -1


def test_tune_cache_keeps_the_sample(tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    path.write_text(f"{20 * 1024 + 3} 256 0 -1 0 1 1 0 -1 -1\n")
    monkeypatch.setenv("CCL_TUNE_CACHE", str(path))
    c = ccl.ccl_context_create(0)
    try:
        other = _supercritical()
        assert np.array_equal(gpu_label(c, other), oracle.uf_label(other))
        assert ccl.ccl_get_stats(c).pre_analysis == -1
    finally:
        ccl.ccl_context_destroy(c)


def test_link_mode_as_set_or_by_window(fresh):
    """0 and 1 as set; -1 (the default) by window in the slots of one large instance,
    0 elsewhere."""
    small, large = L.square(200, 0.5, 4), L.square(3700, 0.5, 4)
    opt = ccl.CCL_OPT_LINK_MODE
    assert ccl.ccl_get_option(fresh, opt) == -1
    for setting in (-1, 0, 1, -1):
        assert ccl.ccl_set_option(fresh, opt, setting) == ccl.CCL_OK
        assert ccl.ccl_get_option(fresh, opt) == setting
        for lat, by_window in ((small, 0), (large, -1)):
            assert np.array_equal(gpu_label(fresh, lat), oracle.uf_label(lat))
            assert ccl.ccl_get_stats(fresh).link_mode == (setting if setting >= 0 else by_window)


def test_small_calls_walk_step_ii(fresh):
    """Up to 2^18 sites, single and batched, step (ii) left to the library runs."""
    for side, ran in ((512, 1), (513, -1)):
        lat = L.square(side, 0.65, 2)
        assert np.array_equal(gpu_label(fresh, lat), oracle.uf_label(lat))
        assert ccl.ccl_get_stats(fresh).pre_analysis == ran
        b = L.make_batch([dict(kind="square", L=side // 2, p=0.65, seed=k) for k in range(4 if ran == 1 else 5)])
        assert np.array_equal(gpu_label_batched(fresh, b), oracle.uf_label_batched(b))
        assert ccl.ccl_get_stats(fresh).pre_analysis == ran
