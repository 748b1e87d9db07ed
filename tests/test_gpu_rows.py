"""Step (i)'s row scan against the oracle where its variants meet: rows of one
degree (3, 4 and 6 have their own code), mixed rows, rows past the register
path, chunk groups that end at 128 sites, and every alignment of an instance's
entries inside a batch. Labels are integers: equality, no tolerance."""
import ctypes

import numpy as np
import pytest
import torch

import lattices as L
import oracle
import paper_1603_08357_gb300 as ccl
from ccl_testutil import DEV, gpu_label, gpu_label_batched

pytestmark = pytest.mark.gpu


def _graph(n, degrees, p, seed):
    """Rows of the given degrees with uniform random columns (repeats and
    self-loops included) and Bernoulli(p) entry bits."""
    rng = np.random.default_rng(seed)
    rp = np.concatenate([[0], np.cumsum(degrees)]).astype(np.int32)
    nnz = int(rp[-1])
    near = rng.random(nnz) < 0.5          # half of the columns close by: chains inside a chunk
    row = np.repeat(np.arange(n), degrees)
    col = np.where(near, np.clip(row - rng.integers(0, 40, nnz), 0, n - 1), rng.integers(0, n, nnz)).astype(np.int32)
    return L.Lattice("random", n, nnz, rp, col, L.pack_bits(rng.random(nnz) < p), p, seed)


@pytest.mark.parametrize("degree", [1, 2, 3, 4, 5, 6, 8, 9])
@pytest.mark.parametrize("n", [127, 128, 129, 1024, 1151, 4000])
def test_one_degree(ctx, degree, n):
    for p in (0.0, 0.3, 1.0):
        lat = _graph(n, np.full(n, degree), p, 100 * degree + n)
        assert np.array_equal(gpu_label(ctx, lat), oracle.uf_label(lat))
        assert ccl.ccl_get_stats(ctx).residual_pairs == oracle.steps_label(lat)["n_residual"]


@pytest.mark.parametrize("top", [1, 3, 7, 8, 12])
def test_mixed_degrees(ctx, top):
    for n in (128, 1000, 5000):
        deg = np.random.default_rng(n + top).integers(0, top + 1, n)
        lat = _graph(n, deg, 0.6, n)
        assert np.array_equal(gpu_label(ctx, lat), oracle.uf_label(lat))


def test_batch_alignments(ctx):
    """Instances of odd entry counts one after another: entries, bits, row
    pointers and labels of later instances start at every offset of 16 bytes."""
    lats = [_graph(n, np.full(n, d), 0.45, 7 * n + d) for d in (3, 4, 6, 5) for n in (129, 1025, 641, 2047)]
    so = np.concatenate([[0], np.cumsum([x.n for x in lats])])
    eo = np.concatenate([[0], np.cumsum([x.nnz for x in lats])])
    bits = L.pack_bits(np.concatenate([L.unpack_bits(x.open_bits, x.nnz) for x in lats]))
    dev = [torch.from_numpy(np.concatenate(a)).to(DEV) for a in ([x.row_ptr for x in lats], [x.col_idx for x in lats])]
    out = torch.full((int(so[-1]),), -1, dtype=torch.int32, device=DEV)
    assert ccl.ccl_label_batched(ctx, len(lats), so, eo, *dev, torch.from_numpy(bits.view(np.int32)).to(DEV), out) == ccl.CCL_OK
    assert ccl.ccl_sync(ctx) == ccl.CCL_OK
    got = out.cpu().numpy()
    for k, x in enumerate(lats):
        assert np.array_equal(got[so[k]:so[k + 1]], oracle.uf_label(x)), k


@pytest.mark.parametrize("degree", [3, 4, 5, 6])
@pytest.mark.parametrize("value", [-1, 4000, 2**28 + 5, 2**31 - 1])
def test_column_out_of_range_is_reported(ctx, degree, value):
    lat = _graph(4000, np.full(4000, degree), 1.0, degree)
    lat.col_idx[1234 * degree + 1] = value
    rp, ci = torch.from_numpy(lat.row_ptr).to(DEV), torch.from_numpy(lat.col_idx).to(DEV)
    out = torch.empty(lat.n, dtype=torch.int32, device=DEV)
    assert ccl.ccl_label(ctx, lat.n, lat.nnz, rp, ci, torch.from_numpy(lat.open_bits.view(np.int32)).to(DEV), out) == ccl.CCL_OK
    assert ccl.ccl_sync(ctx) == ccl.CCL_ERR_INDEX_OUT_OF_RANGE
    assert int(out.min()) >= 0 and int(out.max()) < lat.n


def test_bands_in_rounds(ctx):
    """A batch large enough for step (i) to hand its tiles out in rounds of
    bands (64 tiles per CTA at least): every label and the pair count."""
    specs = [s for s in L.batched_mix_specs(64, seed=12) if s["kind"] != "cayley" or s["shells"] > 3]
    b = L.make_batch(specs)
    assert b.n_total > 64 * 1024 * 2 * 160, "too few tiles for the rounds"
    got = gpu_label_batched(ctx, b)
    want, _ = oracle.uf_label_batched_threads(b)
    assert np.array_equal(got, want[:b.n_total])
    st = ccl.ccl_get_stats(ctx)
    assert np.array_equal(gpu_label_batched(ctx, b), got)          # again: the ticket starts over
    assert ccl.ccl_get_stats(ctx).residual_pairs == st.residual_pairs > 0


def _ladder(rungs, seed):
    """Two paths joined by rungs, numbered at random along the paths: every
    label chain is long, and every rung but the first closes a cycle."""
    rng = np.random.default_rng(seed)
    num = rng.permutation(2 * rungs) if seed else np.arange(2 * rungs)
    a, b = num[:rungs], num[rungs:]
    u = np.concatenate([a[:-1], b[:-1], a])
    v = np.concatenate([a[1:], b[1:], b])
    rows, cols = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.argsort(rows, kind="stable")
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=2 * rungs))]).astype(np.int32)
    nnz = rows.size
    return L.Lattice("random", 2 * rungs, nnz, rp, cols[order].astype(np.int32), L.pack_bits(np.ones(nnz, bool)), 1.0, seed)


@pytest.mark.parametrize("rungs", [1, 2, 31, 33, 64, 65, 1000, 20_000])
@pytest.mark.parametrize("link", [0, 1])
def test_long_chains(rungs, link):
    """Pairs that are set aside again and again, at the edges of the list."""
    c = ccl.ccl_context_create(0)
    try:
        assert ccl.ccl_set_option(c, ccl.CCL_OPT_LINK_MODE, link) == ccl.CCL_OK
        for seed in (0, 1, 2):
            lat = _ladder(rungs, seed)
            assert np.array_equal(gpu_label(c, lat), oracle.uf_label(lat))
    finally:
        ccl.ccl_context_destroy(c)


def test_far_pairs_beyond_l2(ctx):
    """Windows that take link mode 1 by themselves (few pairs, far ends) next to
    windows that do not: a randomly numbered tree, and the same sites with a
    lattice in the second half, both beyond L2."""
    tree = L.cayley(3, 23, 0.6, 3, perm_seed=7)
    sq = L.square(4000, 0.55, 5)
    both = L.Lattice("random", tree.n + sq.n, tree.nnz + sq.nnz,
                     np.concatenate([tree.row_ptr, sq.row_ptr[1:] + tree.nnz]).astype(np.int32),
                     np.concatenate([tree.col_idx, sq.col_idx + tree.n]).astype(np.int32),
                     L.pack_bits(np.concatenate([L.unpack_bits(tree.open_bits, tree.nnz), L.unpack_bits(sq.open_bits, sq.nnz)])), 0.5, 1)
    for lat in (tree, both):
        assert np.array_equal(gpu_label(ctx, lat), oracle.uf_label(lat))


@pytest.mark.parametrize("L_cells", [16, 200, 400])
def test_small_call_in_a_users_graph(ctx, L_cells):
    """A call captured into a user's graph: the programmatic chain of small
    calls (16 and 200 cells) and the ordinary launches (400), replayed on inputs
    rewritten in place."""
    a, b = (L.honeycomb(L_cells, p, seed) for p, seed in ((0.6527, 3), (0.75, 4)))
    rp, ci, bits = (torch.from_numpy(x).to(DEV) for x in (a.row_ptr, a.col_idx, a.open_bits.view(np.int32)))
    out = torch.full((a.n,), -7, dtype=torch.int32, device=DEV)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert ccl.ccl_label(ctx, a.n, a.nnz, rp, ci, bits, out, s) == ccl.CCL_OK    # sizes the workspace
    assert ccl.ccl_sync(ctx, s) == ccl.CCL_OK
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        assert ccl.ccl_label(ctx, a.n, a.nnz, rp, ci, bits, out, s) == ccl.CCL_OK
    for x in (a, b, a):
        out.fill_(-7)
        bits.copy_(torch.from_numpy(x.open_bits.view(np.int32)))
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), oracle.uf_label(x))


@pytest.mark.parametrize("n_cells", [1, 3, 13, 14, 100, 300])
def test_sampled_analysis(n_cells):
    """Step (ii) left to the library: inputs it walks (few roots), leaves alone
    (many) and batches of both, from fewer sites than it samples."""
    c = ccl.ccl_context_create(0)
    lats = [L.honeycomb(n_cells, p, 5) for p in (0.0, 0.5, 0.8, 0.95, 1.0)] if n_cells > 2 else \
        [_graph(k, np.full(k, 2), 0.9, k) for k in (1, 2, 31, 33, 384)]
    for x in lats:
        assert np.array_equal(gpu_label(c, x), oracle.uf_label(x))
    so = np.concatenate([[0], np.cumsum([x.n for x in lats])])
    eo = np.concatenate([[0], np.cumsum([x.nnz for x in lats])])
    bits = L.pack_bits(np.concatenate([L.unpack_bits(x.open_bits, x.nnz) for x in lats]))
    dev = [torch.from_numpy(np.concatenate(a)).to(DEV) for a in ([x.row_ptr for x in lats], [x.col_idx for x in lats])]
    out = torch.full((int(so[-1]),), -1, dtype=torch.int32, device=DEV)
    assert ccl.ccl_label_batched(c, len(lats), so, eo, *dev, torch.from_numpy(bits.view(np.int32)).to(DEV), out) == ccl.CCL_OK
    assert ccl.ccl_sync(c) == ccl.CCL_OK
    got = out.cpu().numpy()
    for k, x in enumerate(lats):
        assert np.array_equal(got[so[k]:so[k + 1]], oracle.uf_label(x)), k
    ccl.ccl_context_destroy(c)


def test_rounds_start_from_empty_band_records():
    """A launch in rounds clears the ticket and every band's record with it: a band
    that a CTA took but never began (it gave up waiting) counts no pairs. Read off
    the captured call, whose graph is not run."""
    class Memset(ctypes.Structure):
        _fields_ = [("dst", ctypes.c_uint64), ("pitch", ctypes.c_size_t), ("value", ctypes.c_uint),
                    ("element", ctypes.c_uint), ("width", ctypes.c_size_t), ("height", ctypes.c_size_t)]

    ctx = ccl.ccl_context_create(0)
    n = 12_000_000                              # isolated sites, enough tiles for the rounds
    so, eo = np.array([0, n, 2 * n], np.int64), np.zeros(3, np.int64)
    rp = torch.zeros(2 * n + 2, dtype=torch.int32, device=DEV)
    out = torch.empty(2 * n, dtype=torch.int32, device=DEV)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert ccl.ccl_label_batched(ctx, 2, so, eo, rp, None, None, out, s) == ccl.CCL_OK
    assert ccl.ccl_sync(ctx, s) == ccl.CCL_OK
    drv = ctypes.CDLL("libcuda.so.1")
    h, graph, count = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert drv.cuStreamBeginCapture_v2(h, 2) == 0
    assert ccl.ccl_label_batched(ctx, 2, so, eo, rp, None, None, out, s) == ccl.CCL_OK
    assert drv.cuStreamEndCapture(h, ctypes.byref(graph)) == 0
    assert drv.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes, kind, cleared = (ctypes.c_void_p * count.value)(), ctypes.c_int(), []
    assert drv.cuGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    for node in nodes:
        assert drv.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 2:                     # a memset
            m = Memset()
            assert drv.cuGraphMemsetNodeGetParams(ctypes.c_void_p(node), ctypes.byref(m)) == 0
            assert m.value == 0
            cleared.append(m.element * m.width * m.height)
    assert drv.cuGraphDestroy(graph) == 0
    # a ticket and at least eleven rounds of a 16-byte record per SM
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert len(cleared) == 1 and cleared[0] >= 16 * (1 + 11 * sms)
    ccl.ccl_context_destroy(ctx)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("mixed", [False, True])
def test_full_stage(shift, mixed):
    """Tiles whose 7168 entries fill a stage: rows of seven, or mixed rows whose last
    ones are empty (a row's scan reads past the last entry there), with the
    columns `shift` entries off their alignment (an instance of that many before)."""
    n = 3 * 1024
    deg = np.full(n, 7)
    if mixed:
        rng = np.random.default_rng(shift)
        deg = np.concatenate([np.concatenate([rng.permutation([6, 8] * 448), np.full(112, 8), np.zeros(16, np.int64)])
                              for _ in range(3)])
        assert deg.size == n and deg[:1024].sum() == 7168
    lats = [_graph(shift + 1, np.r_[0, np.ones(shift, np.int64)], 0.5, 1), _graph(n, deg, 0.4, 9 + shift)]
    so, eo = (np.concatenate([[0], np.cumsum([getattr(x, f) for x in lats])]) for f in ("n", "nnz"))
    bits = L.pack_bits(np.concatenate([L.unpack_bits(x.open_bits, x.nnz) for x in lats]))
    rp, ci = (np.concatenate(a).astype(np.int32) for a in ([x.row_ptr for x in lats], [x.col_idx for x in lats]))
    c = ccl.ccl_context_create(0)
    got = gpu_label_batched(c, L.Batch(so, eo, rp, ci, bits, [{"kind": "random"}] * 2))
    for k, x in enumerate(lats):
        assert np.array_equal(got[so[k]:so[k + 1]], oracle.uf_label(x)), k
    assert np.array_equal(gpu_label(c, lats[1]), oracle.uf_label(lats[1]))
    ccl.ccl_context_destroy(c)


@pytest.mark.parametrize("degree", [7, 9, 15, 16, 17, 31, 32, 33, 40, 41, 65])
def test_long_rows_in_blocks(ctx, degree):
    """Rows scanned in blocks of eight, around the blocks' ends and the 32 entries of
    the residual mask: in a stage (few rows) and too many for it, alone and mixed
    with short rows, with bits from memory and drawn."""
    for n, mixed in ((70, False), (1300, False), (1300, True)):
        rng = np.random.default_rng(degree + n)
        deg = np.where(rng.random(n) < 0.7, rng.integers(0, 4, n), degree) if mixed else np.full(n, degree)
        for p in (0.05, 0.5, 1.0):
            lat = _graph(n, deg, p, degree + n)
            assert np.array_equal(gpu_label(ctx, lat), oracle.uf_label(lat))
            assert ccl.ccl_get_stats(ctx).residual_pairs == oracle.steps_label(lat)["n_residual"]
        rp, ci = torch.from_numpy(lat.row_ptr).to(DEV), torch.from_numpy(lat.col_idx).to(DEV)
        out = torch.full((n,), -1, dtype=torch.int32, device=DEV)
        assert ccl.ccl_label_random(ctx, n, lat.nnz, rp, ci, 99, 0.2, out) == ccl.CCL_OK
        assert ccl.ccl_sync(ctx) == ccl.CCL_OK
        drawn = L.Lattice("random", n, lat.nnz, lat.row_ptr, lat.col_idx, oracle.keyed_bits(lat, 99, 0.2), 0.2, 0)
        assert np.array_equal(out.cpu().numpy(), oracle.uf_label(drawn))


@pytest.mark.parametrize("link", [-1, 0, 1])
def test_deep_windows(link):
    """Calls of more than 2^21 sites whose sample finds long chains (honeycomb from
    1.4 p_c on) drain their windows in slots; the choice is made anew by each call."""
    c = ccl.ccl_context_create(0)
    try:
        assert ccl.ccl_set_option(c, ccl.CCL_OPT_LINK_MODE, link) == ccl.CCL_OK
        lats = [L.honeycomb(1030, r * L.PC_HONEYCOMB, 5) for r in (1.5, 1.0, 1.42)]
        assert lats[0].n > 1 << 21
        for graphs in (1, 0):
            assert ccl.ccl_set_option(c, ccl.CCL_OPT_USE_GRAPHS, graphs) == ccl.CCL_OK
            for lat in lats:
                assert np.array_equal(gpu_label(c, lat), oracle.uf_label(lat))
    finally:
        ccl.ccl_context_destroy(c)


@pytest.mark.parametrize("before", [False, True])
def test_batch_in_a_users_graph(before):
    """A batched call captured into a user's graph, with and without an uncaptured
    call before it: replays label its own instances after the context has labelled
    other and larger batches, and those are labelled as ever."""
    c = ccl.ccl_context_create(0)
    a = L.make_batch([dict(kind="triangle", L=n, p=0.4, seed=n) for n in (30, 47, 128)])
    others = [L.make_batch([dict(kind="square", L=5 + k % 9, p=0.5, seed=k) for k in range(K)]) for K in (3, 300)]
    rp, ci, bits = (torch.from_numpy(x).to(DEV) for x in (a.row_ptr, a.col_idx, a.open_bits.view(np.int32)))
    out = torch.full((a.n_total,), -7, dtype=torch.int32, device=DEV)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert ccl.ccl_reserve(c, 0, 4 * a.nnz_total, 0) == ccl.CCL_OK
    if before:
        assert ccl.ccl_label_batched(c, a.k, a.site_off, a.ent_off, rp, ci, bits, out, s) == ccl.CCL_OK
        assert ccl.ccl_sync(c, s) == ccl.CCL_OK
    else:                                       # (loads the kernels)
        assert np.array_equal(gpu_label_batched(c, others[0]), oracle.uf_label_batched(others[0]))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        assert ccl.ccl_label_batched(c, a.k, a.site_off, a.ent_off, rp, ci, bits, out, s) == ccl.CCL_OK
    want = oracle.uf_label_batched(a)
    for graphs in (0, 1):
        assert ccl.ccl_set_option(c, ccl.CCL_OPT_USE_GRAPHS, graphs) == ccl.CCL_OK
        for b in others:
            assert np.array_equal(gpu_label_batched(c, b), oracle.uf_label_batched(b))
            out.fill_(-7)
            g.replay()
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), want)
    del g
    ccl.ccl_context_destroy(c)
