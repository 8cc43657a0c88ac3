"""What the speed of this library is measured on: the calls its users make.

A case is one call (or the few calls that belong together) through the Python
binding `paper_1111_7171_gb300.passjoin`.  The string sets have the shapes of
`paper_1111_7171_gb300/synth.py` (short: names, medium: titles, long: near-
duplicate documents, short2k: the small uniform set), drawn here on the GPU so that a
million strings take milliseconds.  A case's sizes give its strings; the seed
spells them with another permutation of the alphabet and puts them in another
order, which leaves every edit distance, and so the number of pairs, as it is.

Kinds of call
  step      strings in device memory -> segment index of one threshold -> self
            join, pairs left in device memory: deduplicating a set once.
  resident  self join of an index that is kept, tuned and recorded as a CUDA
            graph: the same set joined again and again.
  rs        R x S join of two host sets, pairs back on the host.
  query     one batch of host queries against a resident index, one threshold.
  multi     one batch whose queries carry their own thresholds.
  plan      the same through a query plan (one CUDA graph launch per batch).
  noalloc   a device batch answered without any allocation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1111_7171_gb300 import passjoin as pj

ALPHA26 = b"abcdefghijklmnopqrstuvwxyz"
ALPHA27 = b"abcdefghijklmnopqrstuvwxyz "
ALPHA40 = b"abcdefghijklmnopqrstuvwxyz0123456789 .,-"

# lengths: ("uniform", lo, hi) or ("normal", mean, deviation); clip: shortest
# and longest string; near: share of the strings that are edited copies;
# copies: how many edited copies a string has; edits: most edits of a copy
# (None: the threshold)
SHAPES = {
    "short2k": dict(alphabet=ALPHA26, zipf=0.0, lengths=("uniform", 8, 20), clip=(1, 64), near=0.2, copies=(1, 1),
                    edits=3),
    "short": dict(alphabet=ALPHA27, zipf=1.1, lengths=("normal", 15, 4), clip=(5, 40), near=0.24, copies=(1, 7),
                  edits=None),
    "medium": dict(alphabet=ALPHA40, zipf=1.0, lengths=("normal", 100, 30), clip=(20, 300), near=0.18, copies=(1, 4),
                   edits=None),
    "long": dict(alphabet=ALPHA40, zipf=1.0, lengths=("normal", 1000, 200), clip=(400, 2000), near=0.10,
                 copies=(1, 1), edits=None),
}


def listed():
    return [
        # one person types one name: a lookup in the resident set, eager call
        dict(name="query-1", kind="query", shape="short", n=1_000_000, tau=2, queries=1),
        # a serving batch of mixed thresholds, replayed through a plan
        dict(name="plan-64", kind="plan", shape="short", n=1_000_000, tau=4, queries=64),
        # a large serving batch of mixed thresholds, eager
        dict(name="multi-4096", kind="multi", shape="short", n=1_000_000, tau=4, queries=4096),
        # a caller that owns its memory: device batch, no allocation, odd size
        dict(name="noalloc-777", kind="noalloc", shape="short", n=400_000, tau=3, queries=777),
        # the smallest set the tests and the benchmark join
        dict(name="step-short2k-t2", kind="step", shape="short2k", n=2_000, tau=2, tune=False),
        # names, the usual threshold, odd size
        dict(name="step-short-417k-t2", kind="step", shape="short", n=417_283, tau=2, tune=False),
        # names, the headline: a million strings at the largest threshold
        dict(name="step-short-1m-t4", kind="step", shape="short", n=1_000_000, tau=4, tune=True),
        # titles, odd size, library defaults
        dict(name="step-medium-61k-t4", kind="step", shape="medium", n=61_459, tau=4, tune=False),
        # titles, full size, the benchmark's options
        dict(name="step-medium-500k-t8", kind="step", shape="medium", n=500_000, tau=8, tune=True),
        # documents, full size, the largest threshold
        dict(name="step-long-100k-t32", kind="step", shape="long", n=100_000, tau=32, tune=False),
        # documents joined again and again on one index
        dict(name="resident-long-100k-t16", kind="resident", shape="long", n=100_000, tau=16),
        # two host sets matched once, end to end
        dict(name="rs-short-50k-300k-t2", kind="rs", shape="short", n=300_007, tau=2, queries=50_021),
    ]


def _size(rng, lo, hi):
    """A size between lo and hi, even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "resident", "rs", "query", "multi", "plan", "noalloc"])
    if kind in ("step", "resident"):
        shape = rng.choice(["short", "medium", "long"])
        n = _size(rng, 2_000, {"short": 1_000_000, "medium": 500_000, "long": 100_000}[shape])
        tau = {"short": rng.randint(1, 4), "medium": rng.randint(2, 8), "long": rng.randint(8, 32)}[shape]
        if kind == "step":
            return dict(kind=kind, shape=shape, n=n, tau=tau, tune=rng.random() < 0.5)
        return dict(kind=kind, shape=shape, n=n, tau=tau)
    tau = rng.randint(1, 4)
    n = _size(rng, 10_000, 1_000_000)
    if kind == "rs":
        return dict(kind=kind, shape="short", n=min(n, 500_000), tau=min(tau, 3), queries=_size(rng, 1_000, 100_000))
    return dict(kind=kind, shape="short", n=n, tau=tau, queries=_size(rng, 1, 4096))


# ---------------------------------------------------------------- inputs --

def _lengths(shape, n, gen):
    kind, a, b = shape["lengths"]
    lo, hi = shape["clip"]
    if kind == "uniform":
        return torch.randint(a, b + 1, (n,), generator=gen, device="cuda")
    x = torch.randn(n, generator=gen, device="cuda", dtype=torch.float32) * b + a
    return x.round().clamp(lo, hi).long()


def _chars(shape, rows, cols, gen):
    """rows x cols characters of the shape's distribution (inverse CDF over
    a 2^16-entry table)."""
    alpha = np.frombuffer(shape["alphabet"], dtype=np.uint8)
    w = np.arange(1, len(alpha) + 1, dtype=np.float64) ** -shape["zipf"]
    cdf = np.cumsum(w / w.sum())
    grid = (np.arange(1 << 16) + 0.5) / (1 << 16)
    table = torch.from_numpy(alpha[np.minimum(np.searchsorted(cdf, grid, side="right"), len(alpha) - 1)]).cuda()
    u = torch.randint(0, 1 << 16, (rows, cols), generator=gen, device="cuda", dtype=torch.int32)
    return table[u]


def _edit(shape, rows, lens, edits, gen):
    """Applies edits[k] random insertions, deletions and substitutions to the
    first lens[k] characters of row k (in a copy)."""
    lo, hi = shape["clip"]
    m, width = rows.shape
    col = torch.arange(width, device="cuda", dtype=torch.int32)[None, :]
    lens = lens.clone()
    for step in range(int(edits.max()) if m else 0):
        on = edits > step
        kind = torch.randint(0, 3, (m,), generator=gen, device="cuda")
        u = torch.rand(m, generator=gen, device="cuda")
        c = _chars(shape, m, 1, gen)
        kind = torch.where((kind == 0) & (lens >= hi) | (kind == 1) & (lens <= lo), torch.full_like(kind, 2), kind)
        ins, dele = on & (kind == 0), on & (kind == 1)
        put = on & (kind != 1)
        at = torch.minimum((u * (lens + ins.long()).float()).long(), torch.clamp(lens - 1 + ins.long(), min=0))
        at = at.to(torch.int32)[:, None]
        src = col - (ins[:, None] & (col > at)).to(torch.int32) + (dele[:, None] & (col >= at)).to(torch.int32)
        rows = torch.gather(rows, 1, src.clamp_(0, width - 1).long())
        rows = torch.where(put[:, None] & (col == at), c, rows)
        lens = lens + ins.long() - dele.long()
    return rows, lens


def _pack(rows, lens):
    """(bytes, offsets) of the first lens[k] characters of every row."""
    off = torch.zeros(len(lens) + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    keep = torch.arange(rows.shape[1], device="cuda")[None, :] < lens[:, None]
    return rows[keep].contiguous(), off


def _matrix(shape, n, tau, gen):
    """n strings of a shape as a character matrix and lengths: fresh strings
    and edited copies of some of them."""
    width = shape["clip"][1] + 1 if shape["lengths"][0] == "normal" else shape["lengths"][2] + (shape["edits"] or tau)
    lo, hi = shape["copies"]
    n_copy = int(shape["near"] * n)
    n_base = max(1, int(round(n_copy / ((lo + hi) / 2)))) if n_copy else 0
    fresh = n - n_copy
    lens = _lengths(shape, fresh, gen)
    rows = _chars(shape, fresh, width, gen)
    if n_copy:
        pick = torch.randint(0, min(n_base, fresh), (n_copy,), generator=gen, device="cuda")
        edits = torch.randint(1, (shape["edits"] or max(1, tau)) + 1, (n_copy,), generator=gen, device="cuda")
        crows, clens = _edit(shape, rows[pick], lens[pick], edits, gen)
        rows, lens = torch.cat([rows, crows]), torch.cat([lens, clens])
    return rows, lens


def _respell(gen):
    """A permutation of the byte values that keeps the shapes' alphabets."""
    table = torch.arange(256, device="cuda", dtype=torch.uint8)
    for part in (ALPHA27, bytes(c for c in ALPHA40 if c not in ALPHA27)):
        codes = torch.tensor(list(part), device="cuda")
        table[codes] = codes[torch.randperm(len(part), generator=gen, device="cuda")].to(torch.uint8)
    return table


def _queries(rows, lens, count, taus, gen):
    """Queries against an index of short strings: a quarter fresh short
    strings, a quarter fresh titles (of at most 200 characters), half indexed
    strings with 1..tau edits."""
    short, title = SHAPES["short"], dict(SHAPES["medium"], clip=(5, 200))
    width = 201
    kind = torch.randint(0, 4, (count,), generator=gen, device="cuda")
    kind[0] = 2  # a batch of one looks up a misspelt name
    out = torch.zeros(count, width, dtype=torch.uint8, device="cuda")
    a = short["clip"][1] + 1
    out[:, :a] = _chars(short, count, a, gen)
    qlens = _lengths(short, count, gen)
    titles, tlens = _chars(title, count, width, gen), _lengths(title, count, gen)
    pick = torch.randint(0, len(lens), (count,), generator=gen, device="cuda")
    u = torch.rand(count, generator=gen, device="cuda")
    edits = torch.minimum(1 + (u * taus.float()).long(), taus)
    near, nlens = _edit(short, rows[pick], lens[pick], edits, gen)
    wide = torch.zeros_like(out)
    wide[:, :near.shape[1]] = near
    out = torch.where((kind == 1)[:, None], titles, torch.where((kind >= 2)[:, None], wide, out))
    qlens = torch.where(kind == 1, tlens, torch.where(kind >= 2, nlens, qlens))
    return out, qlens


def _host(packed):
    b, off = packed
    return b.cpu().numpy(), off.cpu().numpy().astype(np.uint64)


def _draw(case, gen):
    """The case's strings and queries before they are spelt and ordered."""
    rows, lens = _matrix(SHAPES[case["shape"]], case["n"], case["tau"], gen)
    if "queries" not in case:
        return rows, lens, None, None, None
    count = case["queries"]
    if case["kind"] in ("multi", "plan"):
        taus = torch.randint(1, case["tau"] + 1, (count,), generator=gen, device="cuda")
    else:
        taus = torch.full((count,), case["tau"], device="cuda")
    if case["kind"] == "rs":  # another set of the same source: half of it edited copies
        short = SHAPES["short"]
        half = count // 2
        pick = torch.randint(0, len(lens), (half,), generator=gen, device="cuda")
        edits = torch.randint(1, case["tau"] + 1, (half,), generator=gen, device="cuda")
        crows, clens = _edit(short, rows[pick], lens[pick], edits, gen)
        frows, flens = _matrix(short, count - half, case["tau"], gen)
        return rows, lens, torch.cat([frows, crows]), torch.cat([flens, clens]), taus
    qrows, qlens = _queries(rows, lens, count, taus, gen)
    return rows, lens, qrows, qlens, taus


def _inputs(case, seed):
    """The case's strings as (rows, lengths), its queries likewise (or None)
    and their thresholds."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(case["n"] + 64 * case["tau"] + case.get("queries", 0))
    rows, lens, qrows, qlens, taus = _draw(case, gen)
    gen.manual_seed(1_000_003 * int(seed) + 17)
    table = _respell(gen)
    order = torch.randperm(len(lens), generator=gen, device="cuda")
    rows, lens = table[rows[order].int()], lens[order]
    if qrows is not None:
        order = torch.randperm(len(qlens), generator=gen, device="cuda")
        qrows, qlens, taus = table[qrows[order].int()], qlens[order], taus[order]
    return rows, lens, qrows, qlens, taus


def prepare(case, seed):
    rows, lens, qrows, qlens, taus = _inputs(case, seed)
    kind, tau = case["kind"], case["tau"]
    state = dict(kind=kind, tau=tau)
    strings = _pack(rows, lens)
    del rows
    if kind == "step":
        state.update(strings=strings, tune=bool(case["tune"]))
    elif kind == "resident":
        state["index"] = pj.pj_build_index(strings, tau, results_on_device=True, lazy_partitions=True, autotune=True,
                                           graph_joins=True)
    elif kind == "rs":
        state.update(S=_host(strings), R=_host(_pack(qrows, qlens)))
    else:
        state["index"] = pj.pj_build_index(strings, tau)
        queries = _pack(qrows, qlens)
        if kind == "noalloc":
            state.update(batch=queries, cap=1 << 20,
                         out=torch.empty(3 << 20, dtype=torch.int32, device="cuda"))
        else:
            state["batch"] = _host(queries)
        state["taus"] = taus.cpu().numpy().astype(np.uint8)
        if kind == "plan":
            state["plan"] = pj.Plan(state["index"], max_queries=max(64, case["queries"]), max_bytes=1 << 20)
    return state


def _device_pairs(result):
    """The pairs of a device result as an (n, 3) int32 tensor that keeps the
    result alive."""
    if result.count == 0:
        return torch.empty((0, 3), dtype=torch.int32, device="cuda")
    pairs = result.tensor().view(torch.int32).view(-1, 3)
    pairs.result = result
    return pairs


def _host_pairs(result):
    return result.pairs.view(np.uint32).reshape(-1, 3)


def run(state):
    kind, tau = state["kind"], state["tau"]
    if kind == "step":
        index = pj.pj_build_index(state["strings"], tau, results_on_device=True, lazy_partitions=True,
                                  autotune=state["tune"])
        pairs = _device_pairs(pj.pj_self_join(index, tau))
        if pairs.numel():
            pairs.index = index  # a result is released before its index
        return pairs
    if kind == "resident":
        return _device_pairs(pj.pj_self_join(state["index"], tau))
    if kind == "rs":
        return _host_pairs(pj.pj_join(state["R"], state["S"], tau))
    if kind == "query":
        return _host_pairs(pj.pj_query(state["index"], state["batch"], tau))
    if kind == "multi":
        return _host_pairs(pj.pj_query_multi(state["index"], state["batch"], state["taus"]))
    if kind == "plan":
        return _host_pairs(state["plan"].query(state["batch"], state["taus"]))
    n = pj.pj_query_noalloc(state["index"], state["batch"], tau, state["out"], state["cap"])
    return state["out"][:3 * n].view(-1, 3)


# ------------------------------------------------------------------ work --

# similar pairs that are neither copies of one string nor of each other, per
# n^2, by threshold (counted on the shapes; the other shapes have none)
_CHANCE = {("short", 1): 1.3e-7, ("short", 2): 1.4e-6, ("short", 3): 1.8e-5, ("short", 4): 1.24e-4}


def work(case):
    """Bytes of one pass: the strings, their offsets and, for a batch, its
    queries read once (a resident index is read only where its strings are
    joined), 12 bytes written per similar pair.  The arithmetic is on
    integers: no floating point operations."""
    shape = SHAPES[case["shape"]]
    mean = shape["lengths"][1] if shape["lengths"][0] == "normal" else sum(shape["lengths"][1:]) / 2
    n, count = case["n"], case.get("queries", 0)
    chance = _CHANCE.get((case["shape"], case["tau"]), 0.0)
    if case["kind"] in ("step", "resident"):
        near = shape["near"] * n * (1 + shape["copies"][1] / 4)
        return {"bytes": n * (mean + 8) + 12 * (near + chance * n * n), "flops": 0}
    qmean = 15 if case["kind"] == "rs" else 36
    pairs = 0.5 * count * 3 + 2 * chance * count * n
    indexed = n * (mean + 8) if case["kind"] == "rs" else 0
    return {"bytes": indexed + count * (qmean + 9) + 12 * pairs, "flops": 0}


# ----------------------------------------------------------------- exact --

def _distances(a, la, b, lb):
    """Edit distances of row pairs, plain Wagner-Fischer over all cells."""
    m = int(lb.max())
    row = torch.arange(m + 1, device="cuda", dtype=torch.int64)[:, None].repeat(1, len(la))
    res = torch.where(la == 0, lb, torch.zeros_like(lb))
    lbi = lb[None, :]
    for i in range(1, int(la.max()) + 1):
        left = torch.full_like(la, i)
        diag = row[0].clone()
        row[0] = left
        ca = a[:, i - 1]
        for j in range(1, m + 1):
            up = row[j].clone()
            left = torch.minimum(torch.minimum(up, left) + 1, diag + (ca != b[:, j - 1]).long())
            diag = up
            row[j] = left
        res = torch.where(la == i, torch.gather(row, 0, lbi)[0], res)
    return res


def exact(case, seed):
    """Definition 1 by brute force where it is quick: every pair whose
    lengths differ by at most its threshold, all DP cells."""
    n, count = case["n"], case.get("queries", case["n"])
    if case["shape"] not in ("short", "short2k") or n * count > 100_000_000:
        return None
    rows, lens, qrows, qlens, taus = _inputs(case, seed)
    self_join = qrows is None
    if self_join:
        qrows, qlens, taus = rows, lens, torch.full_like(lens, case["tau"])
    order = torch.argsort(lens, stable=True)
    cum = torch.zeros(1 << 12, dtype=torch.int64, device="cuda")  # strings of length < l
    cum[1:] = torch.cumsum(torch.bincount(lens, minlength=(1 << 12) - 1), 0)
    out = []
    width = rows.shape[1] + 8  # longer queries are similar to nothing
    q_all = torch.arange(count, device="cuda")
    lo = cum[torch.clamp(qlens - taus, min=0)]
    hi = cum[qlens + taus + 1]
    room = 1 << 21
    at = 0
    while at < count:
        c = torch.cumsum(hi[at:] - lo[at:], 0)
        stop = at + max(1, int((c <= room).sum()))
        q = q_all[at:stop]
        k = hi[q] - lo[q]
        qq = torch.repeat_interleave(q, k)
        first = torch.cumsum(k, 0) - k
        x = order[lo[qq] + torch.arange(len(qq), device="cuda") - torch.repeat_interleave(first, k)]
        if self_join:
            later = x > qq
            qq, x = qq[later], x[later]
        at = stop
        if not len(qq):
            continue
        d = _distances(qrows[qq][:, :width], torch.clamp(qlens[qq], max=width), rows[x], lens[x])
        ok = (d <= taus[qq]) & (qlens[qq] <= width)
        out.append(torch.stack([qq[ok], x[ok], d[ok]], 1))
    pairs = torch.cat(out) if out else torch.zeros((0, 3), dtype=torch.int64, device="cuda")
    key = pairs[:, 0] * n + pairs[:, 1]
    return pairs[torch.argsort(key)]
