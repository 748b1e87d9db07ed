"""Performance cases of the cluster-labelling library: what its users have it do.

Each case is one call sequence through the public entry points on one seeded
percolation input; sizes and open probabilities come from the benchmark's
configurations (honeycomb 256^2, triangle 4096^2 and 16384^2, a randomly
numbered Bethe lattice of 24 shells, the batched mix, the request stream), the
threshold sweeps and the tests. Inputs are made on the GPU from the seed alone.

A case has a "form" (which calls it makes) and describes its graph:
  kind    honeycomb | triangle | square | cubic | cayley
  L       lattice size (honeycomb: L x L cells; cubic: L^3 sites)
  z, shells   Cayley tree (randomly numbered)
  ratio   open probability over the lattice's threshold p_c
"""
import math
import random
import types

import numpy as np
import torch

import paper_1603_08357_gb300 as ccl
from paper_1603_08357_gb300 import percolation

PC = {"honeycomb": 1 - 2 * math.sin(math.pi / 18), "triangle": 2 * math.sin(math.pi / 18), "square": 0.5,
      "cubic": 0.2488126}
DEGREE = {"honeycomb": 3, "triangle": 6, "square": 4, "cubic": 6}


def listed():
    return [
        # one small system in a loop: a latency-bound call, as in equilibration runs and in the smallest requests
        dict(name="label_honeycomb_64", form="label", kind="honeycomb", L=64, ratio=1.0),
        # the small benchmark system: everything fits L2
        dict(name="label_honeycomb_256", form="label", kind="honeycomb", L=256, ratio=1.0),
        # the ordinary single system of a percolation study
        dict(name="label_triangle_4096", form="label", kind="triangle", L=4096, ratio=1.0),
        # an irregular graph: a Bethe lattice stored in random order, neighbours anywhere in memory
        dict(name="label_bethe_24", form="label", kind="cayley", z=3, shells=24, ratio=1.0),
        # the largest single system, far beyond L2
        dict(name="label_triangle_16384", form="label", kind="triangle", L=16384, ratio=1.0),
        # a Monte-Carlo ensemble of uneven systems around p_c in one call
        dict(name="batched_mix_1024", form="batched", K=1024, lo=64, hi=1024, shells=16, spread=0.05),
        # many small requests gathered into one call
        dict(name="batched_small_256", form="batched", K=256, lo=12, hi=128, shells=11, spread=0.0),
        # one realisation of a threshold sweep: bonds drawn on the device, spanning test, largest cluster
        dict(name="realise_triangle_1023", form="realise", kind="triangle", L=1023, ratio=1.0),
        # the same at the largest size of the sweeps, above the threshold
        dict(name="realise_honeycomb_2896", form="realise", kind="honeycomb", L=2896, ratio=1.25),
        # the strided neighbour list in place of CSR, three dimensions, below the threshold
        dict(name="dense_cubic_200", form="dense", kind="cubic", L=200, ratio=0.75, extra=0),
        # cluster numbers and sizes of a labelled system
        dict(name="relabel_triangle_4096", form="relabel", kind="triangle", L=4096, ratio=0.9),
        # the request loop: mixed requests in pinned host memory, all in flight at once, labels back on the host
        dict(name="served_32", form="served", K=32, lo=32, hi=1000, shells=16, spread=0.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _lattice(rng, lo, hi, kinds=("honeycomb", "triangle", "square", "cubic", "cayley")):
    kind, n = rng.choice(kinds), _log(rng, lo, hi)
    ratio = round(rng.choice([rng.uniform(0.95, 1.05), rng.uniform(0.5, 1.5)]), 4)
    if kind == "cayley":
        z = rng.randint(3, 6)
        shells = 2
        while _cayley_starts(z, shells + 1)[-1] <= n:
            shells += 1
        return dict(kind=kind, z=z, shells=shells, ratio=ratio)
    side = {"honeycomb": math.sqrt(n / 2), "cubic": n ** (1 / 3)}.get(kind, math.sqrt(n))
    return dict(kind=kind, L=max(3, round(side)), ratio=min(ratio, 1.5))


def draw(rng):
    form = rng.choice(["label", "label", "label", "batched", "batched", "realise", "dense", "relabel", "host", "served"])
    if form == "label":
        return dict(form=form, **_lattice(rng, 5e3, 1e8))
    if form == "batched":
        lo = round(_log(rng, 12, 200))
        hi = round(_log(rng, lo + 20, 1024))
        most = max(16, min(2048, int(4e8 / (hi * hi))))
        return dict(form=form, K=round(_log(rng, 8, most)), lo=lo, hi=hi, shells=rng.randint(9, 16),
                    spread=rng.choice([0.0, 0.05]))
    if form == "served":
        return dict(form=form, K=rng.randint(8, 48), lo=32, hi=round(_log(rng, 100, 1000)), shells=rng.randint(9, 16), spread=0.0)
    if form == "dense":
        return dict(form=form, extra=rng.randint(0, 2), **_lattice(rng, 1e4, 1.7e7, tuple(DEGREE)))
    if form == "realise":
        return dict(form=form, **_lattice(rng, 5e4, 1.7e7, ("triangle", "honeycomb")))
    return dict(form=form, **_lattice(rng, 1e4, 1.7e7 if form == "relabel" else 2e6, ("triangle", "honeycomb", "square")))


# ---------------------------------------------------------------------------
# inputs: CSR entries (rows in site order) and the open state of each entry


def _cayley_starts(z, shells):
    """First site of every shell in centre-first numbering, then the site count."""
    starts, size = [0, 1], z
    for _ in range(shells):
        starts.append(starts[-1] + size)
        size *= z - 1
    return starts


def _pick(mask, a, b):
    return torch.where(mask, a, b).int()


def _lattice_rows(kind, L, p, g, open_y, dev):
    """(columns [n, degree], open states, mask of the entries present or None)."""
    i32 = torch.int32
    if kind == "cubic":
        n, step, wrap = L ** 3, [1, L, L * L], [L, L, L]
        i = torch.arange(n, dtype=i32, device=dev)
        at = [i % L, (i // L) % L, i // (L * L)]
        on = [torch.rand(n, generator=g, device=dev) < p for _ in range(3)]
        up = [i + _pick(at[a] == wrap[a] - 1, step[a] * (1 - L), step[a]) for a in range(3)]
        dn = [i + _pick(at[a] == 0, step[a] * (L - 1), -step[a]) for a in range(3)]
        return torch.stack(up + dn, 1), torch.stack(on + [on[a][dn[a].long()] for a in range(3)], 1), None
    i = torch.arange(L * L, dtype=i32, device=dev)        # cell numbers, row by row
    x, y = i % L, i // L
    xp, xm = _pick(x == L - 1, 1 - L, 1), _pick(x == 0, L - 1, -1)
    yp, ym = _pick(y == L - 1, L * (1 - L), L), _pick(y == 0, L * (L - 1), -L)
    bonds = 2 if kind == "square" else 3
    on = [torch.rand(L * L, generator=g, device=dev) < p for _ in range(bonds)]
    no_up, no_dn = (y == L - 1, y == 0) if open_y else (None, None)
    all_in = torch.ones_like(y, dtype=torch.bool)
    if kind == "honeycomb":
        a, b = 2 * i, 2 * i + 1
        lt, dn, rt, up = i + xm, i + ym, i + xp, i + yp
        col = torch.stack([b, 2 * lt + 1, 2 * dn + 1, a, 2 * rt, 2 * up], 1)
        st = torch.stack([on[0], on[1], on[2], on[0], on[1][rt.long()], on[2][up.long()]], 1)
        here = torch.stack([all_in, all_in, ~no_dn, all_in, all_in, ~no_up], 1) if open_y else None
        shape = (2 * L * L, 3)
        return col.view(shape), st.view(shape), here.view(shape) if open_y else None
    nb = [i + xp, i + yp, i + xm, i + ym] if kind == "square" else [i + xp, i + yp, i + xp + yp, i + xm, i + ym, i + xm + ym]
    col = torch.stack(nb, 1)
    st = torch.stack(on + [on[k][nb[bonds + k].long()] for k in range(bonds)], 1)
    here = None
    if open_y:
        here = torch.stack([all_in] + [~no_up] * (bonds - 1) + [all_in] + [~no_dn] * (bonds - 1), 1)
    return col, st, here


def _cayley_rows(z, shells, p, g, dev):
    """(row degrees, columns, open states) of a randomly numbered Cayley tree."""
    starts = _cayley_starts(z, shells)
    n, inner = starts[-1], starts[-2]
    perm = torch.randperm(n, generator=g, device=dev, dtype=torch.int32)
    on = torch.rand(n, generator=g, device=dev) < p       # bond of each site to its parent
    deg = torch.empty(n, dtype=torch.int32, device=dev)
    at = perm.long()
    deg[at[:inner]] = z
    deg[at[inner:]] = 1
    first = torch.cumsum(deg, 0, dtype=torch.int64) - deg
    nnz = int(deg.sum())
    col = torch.empty(nnz, dtype=torch.int32, device=dev)
    st = torch.empty(nnz, dtype=torch.bool, device=dev)
    par = torch.cat([torch.zeros(starts[2] - 1, dtype=torch.int64, device=dev)] +
                    [starts[k - 1] + torch.arange(starts[k + 1] - starts[k], device=dev) // (z - 1)
                     for k in range(2, shells + 1)])        # parents of sites 1 .. n-1
    slot = first[at[1:]]
    col[slot], st[slot] = perm[par], on[1:]
    kid = torch.arange(inner, device=dev)
    child0 = 1 + torch.cat([kid[:1], z + (kid[1:] - 1) * (z - 1)])      # first child of each inner site
    for c in range(z):
        who = kid if c < z - 1 else kid[:1]               # the centre has one child more
        child = child0[: who.numel()] + c
        slot = first[at[: who.numel()]] + c + (who > 0)
        col[slot], st[slot] = perm[child], on[child]
    return deg, col, st


def _graph(case, g, dev, open_y=False):
    """(n, row degrees or the one degree, columns, open states)."""
    if case["kind"] == "cayley":
        deg, col, st = _cayley_rows(case["z"], case["shells"], case["ratio"] / (case["z"] - 1), g, dev)
        return deg.numel(), deg, col, st
    col, st, here = _lattice_rows(case["kind"], case["L"], case["ratio"] * PC[case["kind"]], g, open_y, dev)
    n, d = col.shape
    if here is None:
        return n, d, col.reshape(-1), st.reshape(-1)
    return n, here.sum(1, dtype=torch.int32), col[here], st[here]


def _row_ptr(n, deg, dev):
    if isinstance(deg, int):
        return torch.arange(n + 1, dtype=torch.int32, device=dev) * deg
    rp = torch.zeros(n + 1, dtype=torch.int32, device=dev)
    rp[1:] = torch.cumsum(deg, 0)
    return rp


def _pack(st):
    """Open states as bit words, entry e at word e >> 5, bit e & 31."""
    words = max(1, (st.numel() + 31) // 32)
    b = torch.zeros(words * 32, dtype=torch.uint8, device=st.device)
    b[: st.numel()] = st
    w = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], dtype=torch.uint8, device=st.device)
    return (b.view(-1, 8) * w).sum(1, dtype=torch.uint8).view(torch.int32)


def _batch_specs(case):
    """The instances of a batch: sizes and kinds follow from the case alone."""
    r, specs = random.Random(4 + case["K"]), []
    for _ in range(case["K"]):
        kind = r.choice(["honeycomb", "triangle", "cayley"])
        if kind == "cayley":
            z = r.randint(3, 6)
            most = 8
            while most < case["shells"] and _cayley_starts(z, most + 1)[-1] <= 2 * case["hi"] ** 2:
                most += 1
            while most > 3 and _cayley_starts(z, most)[-1] > 2 * case["hi"] ** 2:
                most -= 1
            s, pc = dict(kind=kind, z=z, shells=r.randint(min(8, most), most)), 1 / (z - 1)
        else:
            s, pc = dict(kind=kind, L=r.randint(case["lo"], case["hi"])), PC[kind]
        specs.append(dict(s, ratio=1 + r.uniform(-case["spread"], case["spread"]) / pc))
    return specs


def _sites(spec):
    if spec["kind"] == "cayley":
        return _cayley_starts(spec["z"], spec["shells"])[-1]
    return spec["L"] ** 3 if spec["kind"] == "cubic" else spec["L"] ** 2 * (2 if spec["kind"] == "honeycomb" else 1)


def _entries(spec):
    return 2 * (_sites(spec) - 1) if spec["kind"] == "cayley" else _sites(spec) * DEGREE[spec["kind"]]


def _generator(seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    return torch.Generator(device=dev).manual_seed(seed), dev


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _server():
    """The process's request loop, as a serving program keeps it."""
    if "server" not in _kept:
        _kept["server"] = ccl.ccl_server_create(torch.cuda.current_device())
    return _kept["server"]


_kept = {}


def prepare(case, seed):
    g, dev = _generator(seed)
    form = case["form"]
    s = types.SimpleNamespace(form=form, ctx=ccl.default_context(dev.index))
    if form in ("batched", "served"):
        parts = [_graph(sp, g, dev) for sp in _batch_specs(case)]
    if form == "served":
        s.server = _server()
        s.labels = torch.empty(sum(q[0] for q in parts), dtype=torch.int32, pin_memory=True)
        outs = torch.split(s.labels, [q[0] for q in parts])
        s.requests = [(q[0], q[2].numel(), _pinned(_row_ptr(q[0], q[1], dev)), _pinned(q[2]), _pinned(_pack(q[3])), out)
                      for q, out in zip(parts, outs)]
        return s
    if form == "batched":
        s.K = len(parts)
        s.site_off = np.concatenate([[0], np.cumsum([q[0] for q in parts])]).astype(np.int64)
        s.ent_off = np.concatenate([[0], np.cumsum([q[2].numel() for q in parts])]).astype(np.int64)
        s.rp = torch.cat([_row_ptr(q[0], q[1], dev) for q in parts])
        s.ci = torch.cat([q[2] for q in parts])
        s.bits = _pack(torch.cat([q[3] for q in parts]))
        s.labels = torch.empty(int(s.site_off[-1]), dtype=torch.int32, device=dev)
        return s
    s.n, deg, col, st = _graph(case, g, dev, open_y=form == "realise")
    s.nnz = col.numel()
    s.labels = torch.empty(s.n, dtype=torch.int32, device=dev)
    if form == "dense":
        s.width = deg + case["extra"]
        none = torch.full((s.n, case["extra"]), -1, dtype=torch.int32, device=dev)
        s.nn = torch.cat([col.view(s.n, deg), none], 1).t().contiguous()
        s.bits = _pack(torch.cat([st.view(s.n, deg), none > 0], 1).t().reshape(-1))
        return s
    rp = _row_ptr(s.n, deg, dev)
    if form == "realise":
        lat = types.SimpleNamespace(n=s.n, nnz=s.nnz, row_ptr=rp.cpu().numpy(), col_idx=col.cpu().numpy())
        s.sampler = percolation.Sampler(s.ctx, lat, *percolation.boundary_rows(case["kind"], case["L"]))
        s.p, s.seed = case["ratio"] * PC[case["kind"]], seed
        s.span = torch.empty(1, dtype=torch.int32, device=dev)
        s.largest = torch.empty(2, dtype=torch.int32, device=dev)
        return s
    s.rp, s.ci, s.bits = rp, col, _pack(st)
    if form == "host":
        for name in ("rp", "ci", "bits", "labels"):
            setattr(s, name, _pinned(getattr(s, name)))
    if form == "relabel":
        ccl.check(ccl.ccl_label(s.ctx, s.n, s.nnz, s.rp, s.ci, s.bits, s.labels), "ccl_label")
        ccl.check(ccl.ccl_sync(s.ctx), "ccl_sync")
        del s.rp, s.ci, s.bits
        s.seq = torch.empty_like(s.labels)
        s.sizes = torch.zeros_like(s.labels)              # only one value per cluster is written
        s.count = torch.empty(1, dtype=torch.int32, device=dev)
    return s


def run(s):
    if s.form == "label":
        ccl.check(ccl.ccl_label(s.ctx, s.n, s.nnz, s.rp, s.ci, s.bits, s.labels), "ccl_label")
    elif s.form == "batched":
        ccl.check(ccl.ccl_label_batched(s.ctx, s.K, s.site_off, s.ent_off, s.rp, s.ci, s.bits, s.labels), "ccl_label_batched")
    elif s.form == "dense":
        ccl.check(ccl.ccl_label_dense(s.ctx, s.n, s.width, s.nn, s.bits, s.labels), "ccl_label_dense")
    elif s.form == "realise":
        s.sampler.realise(s.seed, s.p, s.span.data_ptr(), s.largest.data_ptr())
        return s.sampler.labels, s.span, s.largest
    elif s.form == "relabel":
        ccl.check(ccl.ccl_relabel(s.ctx, s.n, s.labels, s.seq, s.count, s.sizes), "ccl_relabel")
        return s.seq, s.count, s.sizes
    elif s.form == "served":
        tickets = []
        for n, nnz, rp, ci, bits, _ in s.requests:
            status, ticket = ccl.ccl_server_submit_nocopy(s.server, n, nnz, rp, ci, bits)
            ccl.check(status, "ccl_server_submit_nocopy")
            tickets.append(ticket)
        for ticket, r in zip(tickets, s.requests):
            ccl.check(ccl.ccl_server_wait(s.server, ticket, r[-1]), "ccl_server_wait")
    else:
        ccl.check(ccl.ccl_label_host(s.ctx, s.n, s.nnz, s.rp, s.ci, s.bits, s.labels), "ccl_label_host")
    return s.labels


def work(case):
    """Inputs read once and outputs written once; no floating-point operations."""
    if case["form"] in ("batched", "served"):
        specs = _batch_specs(case)
        n, nnz, k = sum(map(_sites, specs)), sum(map(_entries, specs)), len(specs)
    else:
        n, nnz, k = _sites(case), _entries(case), 1
    if case["form"] == "relabel":
        return {"bytes": 8 * n, "flops": 0}
    if case["form"] == "dense":
        slots = nnz + case["extra"] * n
        return {"bytes": 4 * slots + slots // 8 + 4 * n, "flops": 0}
    bits = 0 if case["form"] == "realise" else nnz // 8
    return {"bytes": 4 * (n + k) + 4 * nnz + bits + 4 * n, "flops": 0}


# ---------------------------------------------------------------------------
# the same outputs by plain torch, in 64-bit integers


def _components(n, u, v):
    """Smallest site of every site's component under the edges u[k] - v[k]."""
    lab = torch.arange(n, device=u.device)
    while True:
        a, b = lab[u], lab[v]
        if bool((a == b).all()):
            return lab
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        lab.scatter_reduce_(0, hi, lo, "amin")
        while True:
            up = lab[lab]
            if bool((up == lab).all()):
                break
            lab = up


def _drawn_open(u, v, seed, p):
    """Open states of the bonds {u, v} as the library draws them: SplitMix64 output u * 2^32 + v (u < v) of `seed`."""
    def shr(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)

    def word(c):
        return c - (1 << 64) if c >= 1 << 63 else c

    z = word(seed % (1 << 64)) + ((u << 32) + v + 1) * word(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * word(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * word(0x94D049BB133111EB)
    z = z ^ shr(z, 31)
    return shr(z, 11) < math.ceil(p * 2.0 ** 53)


def exact(case, seed):
    g, dev = _generator(seed)
    specs = _batch_specs(case) if case["form"] in ("batched", "served") else [case]
    if sum(map(_sites, specs)) > 6e7:
        return None                                       # many seconds in plain torch
    out = []
    for sp in specs:
        n, deg, col, st = _graph(sp, g, dev, open_y=case["form"] == "realise")
        row = torch.arange(n, device=dev).repeat_interleave(deg)
        col = col.long()
        if case["form"] == "realise":
            st = _drawn_open(torch.minimum(row, col), torch.maximum(row, col), seed, case["ratio"] * PC[case["kind"]])
        keep = st & (col < row)
        out.append(_components(n, row[keep], col[keep]))
    lab = torch.cat(out)
    if case["form"] == "realise":
        top, bottom = (torch.from_numpy(t).to(dev).long() for t in percolation_rows(case["kind"], case["L"]))
        both = torch.tensor(sorted(set(lab[top].tolist()) & set(lab[bottom].tolist()))[:1] or [-1])
        sizes = torch.bincount(lab)
        return lab, both, torch.tensor([int(sizes.max()), int(sizes.argmax())])
    if case["form"] == "relabel":
        roots, seq, sizes = torch.unique(lab, return_inverse=True, return_counts=True)
        tail = torch.zeros(lab.numel() - roots.numel(), dtype=sizes.dtype, device=dev)
        return seq, torch.tensor([roots.numel()]), torch.cat([sizes, tail])
    return lab


def percolation_rows(kind, L):
    """First and last row of sites of an open lattice."""
    per = 2 * L if kind == "honeycomb" else L
    return np.arange(per), np.arange((L - 1) * per, L * per)
