"""The calls by which this library's speed is measured.

Five kinds of work, each through the public entry points of
``paper_2305_18663_gb300``:

- ``sweep``: an MCMC phase's sweeps from a given assignment
  (``sbp_set_assignment``, then ``sbp_nodal_sweep`` with its statistics read
  back, as the convergence test needs them), the labels and degrees read
  back at the end;
- ``merge``: a merge phase from a given assignment (``sbp_merge_blocks``);
- ``score``: a new graph from host edge arrays and the blockmodel of a given
  assignment (``sbp_load_graph``, ``sbp_build_blockmodel``, read-back);
- ``partition``: a full golden-ratio search of a new graph from host edge
  arrays (``sbp_load_graph``, ``sbp_partition``);
- ``batch``: many loaded graphs partitioned by one call
  (``sbp_partition_batch``).

Graphs are directed degree-corrected SBM graphs with the laws of this
repository's workloads (``synth/dcsbm.py``), drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

import paper_2305_18663_gb300 as P

# degree laws and planted structures of the workloads: a 1k graph with equal
# blocks, the 200k graph (weak structure), the 1M graph, the batch's graphs
LAWS = {
    "plain_1k": dict(gamma=2.5, kmax=100, ratio=5.0, lognormal=False),
    "plain_200k": dict(gamma=2.1, kmax=2000, ratio=2.0, lognormal=True),
    "dcsbm_1m": dict(gamma=2.1, kmax=2000, ratio=3.0, lognormal=True),
    "batch": dict(gamma=2.5, kmax=100, ratio=4.0, lognormal=False),
}


def _sweep(name, n, e, law, planted, B, frac, sweeps=3, dense_max_B=4096, dl_fp32=1):
    return {"name": name, "kind": "sweep", "n": n, "e": e, "law": law, "planted": planted, "B": B, "frac": frac,
            "sweeps": sweeps, "dense_max_B": dense_max_B, "dl_fp32": dl_fp32}


def listed():
    return [
        # the smallest graph, at its planted block count: launches and host
        # round trips are all there is
        _sweep("sweep_1k", 1_000, 10_000, "plain_1k", 8, 8, 0.3),
        # an ordinary graph late in its search, when few vertices still
        # move: most sweeps of a run are such
        _sweep("sweep_20k_late", 20_011, 320_176, "batch", 71, 71, 0.02),
        # the 200k graph with every Delta DL evaluated exactly (dl_fp32 = 0)
        _sweep("sweep_200k_exact", 200_000, 4_000_000, "plain_200k", 100, 100, 0.3, dl_fp32=0),
        # ... in the middle of its search, at the largest dense blockmodel
        _sweep("sweep_200k_b4096", 200_000, 4_000_000, "plain_200k", 100, 4096, 0.3),
        # ... early in its search, on sparse rows rebuilt by sorting
        _sweep("sweep_200k_b65536", 200_000, 4_000_000, "plain_200k", 100, 65_536, 0.3),
        # the 1M graph on sparse rows: the benchmark's configuration
        _sweep("sweep_1m", 1_000_000, 20_000_000, "dcsbm_1m", 316, 316, 0.3, dense_max_B=1),
        # the first merge phase of a search: one block per vertex, halved
        {"name": "merge_200k", "kind": "merge", "n": 200_000, "e": 4_000_000, "law": "plain_200k", "planted": 100,
         "B": 200_000, "merges": 100_000, "dense_max_B": 4096},
        # a merge phase on a dense blockmodel
        {"name": "merge_20k_b2999", "kind": "merge", "n": 20_011, "e": 320_176, "law": "batch", "planted": 71,
         "B": 2_999, "merges": 1_499, "dense_max_B": 4096},
        # a new graph and the description length of a partition it came with
        {"name": "score_200k", "kind": "score", "n": 200_000, "e": 4_000_000, "law": "plain_200k", "planted": 100,
         "B": 100, "dense_max_B": 4096},
        # full runs of the two plain configurations
        {"name": "partition_1k", "kind": "partition", "n": 1_000, "e": 10_000, "law": "plain_1k", "planted": 8},
        {"name": "partition_200k", "kind": "partition", "n": 200_000, "e": 4_000_000, "law": "plain_200k",
         "planted": 100},
        # a batch of small uneven graphs
        {"name": "batch_32", "kind": "batch", "count": 32, "n_lo": 500, "n_hi": 5_000, "sizes": 0},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "merge", "score", "partition", "batch"])
    if kind == "batch":
        lo = _log_uniform(rng, 500, 1_500)
        return {"kind": kind, "count": rng.randint(8, 32), "n_lo": lo, "n_hi": lo + _log_uniform(rng, 100, 3_000),
                "sizes": rng.randint(1, 10 ** 6)}
    n = _log_uniform(rng, 500, {"sweep": 700_000, "merge": 200_000, "score": 200_000, "partition": 100_000}[kind])
    e = int(n * rng.uniform(8.0, 20.0))
    law = rng.choice(sorted(LAWS))
    if n < 5_000 and LAWS[law]["kmax"] > 100:
        law = "batch"  # the heavy tails need room
    planted = max(2, int(round(math.sqrt(n) * rng.uniform(0.2, 0.5))))
    c = {"kind": kind, "n": n, "e": e, "law": law, "planted": planted}
    if kind == "partition":
        return c
    # the whole range of a search, the planted count most often
    B = planted if rng.random() < 0.5 else _log_uniform(rng, 2, min(n, 4_096 if kind == "score" else 70_000))
    if kind == "score":
        return dict(c, B=B, dense_max_B=4096)
    if kind == "merge":
        return dict(c, B=max(B, 4), merges=max(1, int(max(B, 4) * rng.uniform(0.1, 0.5))), dense_max_B=4096)
    return dict(c, B=B, frac=rng.choice([0.3, 0.1, 0.02]), sweeps=rng.randint(1, 3),
                dense_max_B=rng.choice([4096, 4096, 1]), dl_fp32=rng.choice([1, 1, 1, 0]))


# ---------------------------------------------------------------------------
# inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _power_law(gen, n, gamma, kmax):
    p = torch.arange(1, kmax + 1, dtype=torch.float64, device="cuda").pow(-gamma)
    cdf = (p / p.sum()).cumsum(0)
    x = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    return (torch.searchsorted(cdf, x).clamp_(max=kmax - 1) + 1).double()


def _pick(gen, cdf, count):
    """count positions drawn in proportion to the increments of cdf"""
    x = torch.rand(count, generator=gen, device="cuda", dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(cdf, x, right=True).clamp_(max=cdf.numel() - 1)


def _graph(gen, n, e, planted, law):
    """(src, dst, labels): distinct edges without self-loops, int32 on the GPU"""
    law = LAWS[law]
    dev = "cuda"
    if law["lognormal"]:
        w = torch.randn(planted, generator=gen, device=dev, dtype=torch.float64).exp()
        lab = _pick(gen, w.cumsum(0), n)
        lab[:planted] = torch.arange(planted, device=dev)
        lab = lab[torch.randperm(n, generator=gen, device=dev)]
    else:
        lab = torch.randperm(n, generator=gen, device=dev) % planted
    out_cdf = _power_law(gen, n, law["gamma"], law["kmax"]).cumsum(0)
    th_in = _power_law(gen, n, law["gamma"], law["kmax"])
    order = torch.argsort(lab, stable=True)
    in_cdf = th_in[order].cumsum(0)
    size = torch.bincount(lab, minlength=planted)
    last = size.cumsum(0)
    hi = in_cdf[last - 1]
    lo = hi - torch.zeros(planted, dtype=torch.float64, device=dev).index_add_(0, lab, th_in)
    keys = torch.empty(0, dtype=torch.int64, device=dev)
    for _ in range(50):
        need = e - keys.numel()
        if need <= 0:
            break
        count = need + need // 8 + 16
        s = _pick(gen, out_cdf, count)
        intra = torch.rand(count, generator=gen, device=dev) < law["ratio"] / (1.0 + law["ratio"])
        x = torch.rand(count, generator=gen, device=dev, dtype=torch.float64)
        sb = lab[s]
        y = torch.where(intra, lo[sb] + x * (hi[sb] - lo[sb]), x * in_cdf[-1])
        d = order[torch.searchsorted(in_cdf, y, right=True).clamp_(max=n - 1)]
        keys = torch.unique(torch.cat([keys, (s * n + d)[s != d]]))
    keys = keys[torch.randperm(keys.numel(), generator=gen, device=dev)[:e]]
    return (keys // n).int(), (keys % n).int(), lab.int()


def _labels(gen, case, lab):
    """the planted labels spread over B blocks, a share of them redrawn"""
    n, B, planted = case["n"], case["B"], case["planted"]
    dev = "cuda"
    if B == n:
        return torch.arange(n, dtype=torch.int32, device=dev)
    if B <= planted:
        b = lab.long() % B
    else:  # each planted block split into about B / planted blocks
        per = B // planted
        b = lab.long() * per + torch.randint(0, per, (n,), generator=gen, device=dev)
    frac = case.get("frac", 0.0)
    m = torch.rand(n, generator=gen, device=dev) < frac
    b = torch.where(m, torch.randint(0, B, (n,), generator=gen, device=dev), b)
    return b.int()


def _inputs(case, seed):
    """what the case's calls take, before any of them"""
    gen = _generator(seed)
    if case["kind"] == "batch":
        rng = np.random.default_rng(case["sizes"])  # the seed draws the graphs, not their sizes
        ns = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"])).astype(int)
        deg = rng.uniform(8.0, 32.0, case["count"])
        return [(int(n), *_graph(gen, int(n), int(n * d), max(1, int(round(math.sqrt(n) / 2))), "batch")[:2])
                for n, d in zip(ns, deg)]
    src, dst, lab = _graph(gen, case["n"], case["e"], case["planted"], case["law"])
    return src, dst, _labels(gen, case, lab) if "B" in case else None


def _params(case):
    keys = ("dense_max_B", "dl_fp32")
    return P.Params.default(seed=1, **{k: case[k] for k in keys if k in case})


def prepare(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "batch":
        return {"case": case, "graphs": [P.Graph(n, s, d) for n, s, d in x]}
    src, dst, b = x
    st = {"case": case, "b": b, "params": _params(case)}
    if kind in ("score", "partition"):
        # a graph read from a file: edge arrays in host memory
        st["src"], st["dst"] = src.cpu().numpy(), dst.cpu().numpy()
        return st
    st["graph"] = P.Graph(case["n"], src, dst)
    st["model"] = P.Model(st["graph"], case["B"], b, st["params"])
    st["labels"] = torch.empty_like(b)
    return st


# ---------------------------------------------------------------------------
# the calls

def run(st):
    return {"sweep": _run_sweep, "merge": _run_merge, "score": _run_score, "partition": _run_partition,
            "batch": _run_batch}[st["case"]["kind"]](st)


def _run_sweep(st):
    case, m = st["case"], st["model"].h
    P.sbp_set_assignment(m, case["B"], st["b"])
    stats = [P.sbp_nodal_sweep(m, i, 0, case["n"]) for i in range(case["sweeps"])]
    P.sbp_get_assignment(m, st["labels"])
    dout, din = st["model"].degrees()
    return {"labels": st["labels"], "dout": dout, "din": din, "dl": np.array([s.dl_after for s in stats]),
            "counts": np.array([(s.n_proposed, s.n_moves, s.n_accepted) for s in stats])}


def _run_merge(st):
    case, m = st["case"], st["model"].h
    P.sbp_set_assignment(m, case["B"], st["b"])
    B, rounds = P.sbp_merge_blocks(m, 0, case["merges"])
    P.sbp_get_assignment(m, st["labels"])
    dout, din = st["model"].degrees()
    return {"labels": st["labels"], "dout": dout, "din": din, "dl": P.sbp_get_dl(m), "B": B, "rounds": rounds}


def _run_score(st):
    case = st["case"]
    g = P.Graph(case["n"], st["src"], st["dst"])
    m = P.Model(g, case["B"], st["b"], st["params"])
    dout, din = m.degrees()
    out = {"dl": m.dl(), "dout": dout, "din": din, "M": m.dense()}
    m.close()
    g.close()
    return out


def _run_partition(st):
    g = P.Graph(st["case"]["n"], st["src"], st["dst"])
    b, B, dl, sweeps = g.partition(st["params"])
    g.close()
    return {"labels": b, "B": B, "dl": dl, "sweeps": sweeps}


def _run_batch(st):
    res = P.partition_batch(st["graphs"])
    return {"labels": np.concatenate([r[0] for r in res]), "B": np.array([r[1] for r in res]),
            "dl": np.array([r[2] for r in res]), "sweeps": np.array([r[3] for r in res])}


def work(case):
    """Bytes of the inputs read once and the outputs written once; a sweep
    reads the rows (ids and offsets, both directions) and the labels, and
    writes the labels."""
    if case["kind"] == "batch":
        n = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])  # mean of the log-uniform law
        return {"bytes": case["count"] * n * (8 * 20 + 4), "flops": 0}
    n, e = case["n"], case["e"]
    if case["kind"] == "sweep":
        return {"bytes": case["sweeps"] * (8 * e + 8 * n + 8 * n), "flops": 0}
    return {"bytes": 8 * e + 8 * n, "flops": 0}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the method's definition (torch and numpy)

_M32 = np.uint64(0xFFFFFFFF)


def _mulhi(a, b):
    """high words of the 128-bit products of uint64 values"""
    s = np.uint64(32)
    al, ah, bl, bh = a & _M32, a >> s, b & _M32, b >> s
    x = al * bl
    y = ah * bl + (x >> s)
    z = al * bh + (y & _M32)
    return ah * bh + (y >> s) + (z >> s)


def _philox(c0, c1, c2, k1, seed=1):
    """Philox4x64-10 words for counters (c0, c1[i], c2, 0), key (seed, k1)"""
    c1 = np.asarray(c1, np.uint64)
    c = [np.full_like(c1, c0), c1, np.full_like(c1, c2), np.zeros_like(c1)]
    k = [np.full(1, seed, np.uint64), np.full(1, k1, np.uint64)]
    m0, m1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    for _ in range(10):
        c = [_mulhi(m1, c[2]) ^ c[1] ^ k[0], m1 * c[2], _mulhi(m0, c[0]) ^ c[3] ^ k[1], m0 * c[0]]
        k = [k[0] + np.uint64(0x9E3779B97F4A7C15), k[1] + np.uint64(0xBB67AE8584CAA73B)]
    return c


def _below(words, n):
    """integers in [0, n) from Philox words; n a tensor"""
    return torch.from_numpy(_mulhi(words, n.cpu().numpy().astype(np.uint64)).astype(np.int64)).cuda()


def _f(x):
    x = x.double()
    return torch.special.xlogy(x, x)


class _Counts:
    """the blockmodel of an assignment: its nonzeros in row and column order"""

    def __init__(self, src, dst, b, B):
        r, c = b[src], b[dst]
        self.B, self.E, self.N = B, src.numel(), b.numel()
        self.key, self.val = torch.unique(r * B + c, return_counts=True)
        self.row, self.col = self.key // B, self.key % B
        self.dout, self.din = torch.bincount(r, minlength=B), torch.bincount(c, minlength=B)
        self.d = self.dout + self.din
        tk, order = torch.sort(self.col * B + self.row)
        self.tkey, self.tval, self.trow = tk, self.val[order], tk % B
        self.cum, self.tcum = self.val.cumsum(0), self.tval.cumsum(0)
        self.row0, self.col0 = self.dout.cumsum(0) - self.dout, self.din.cumsum(0) - self.din

    def at(self, r, c):
        k = r * self.B + c
        i = torch.searchsorted(self.key, k).clamp_(max=self.key.numel() - 1)
        return torch.where(self.key[i] == k, self.val[i], torch.zeros_like(k))

    def in_row(self, u, t):
        i = torch.searchsorted(self.cum, self.row0[u] + t, right=True)
        return self.col[i.clamp_(max=self.key.numel() - 1)]

    def in_col(self, u, t):
        i = torch.searchsorted(self.tcum, self.col0[u] + t, right=True)
        return self.trow[i.clamp_(max=self.key.numel() - 1)]

    def far(self, u, t):
        """the block at position t of row u, then column u"""
        return torch.where(t < self.dout[u], self.in_row(u, t), self.in_col(u, t - self.dout[u]))

    def before(self, u, r):
        """weight of row u before column r, and of column u before row r"""
        z = torch.zeros(1, dtype=torch.int64, device="cuda")
        a = torch.cat([z, self.cum])[torch.searchsorted(self.key, u * self.B + r)] - self.row0[u]
        c = torch.cat([z, self.tcum])[torch.searchsorted(self.tkey, u * self.B + r)] - self.col0[u]
        return a, c

    def dl(self):
        L = float(_f(self.val).sum() - _f(self.dout).sum() - _f(self.din).sum())
        x = self.B * self.B / self.E
        return self.E * ((1 + x) * math.log1p(x) - x * math.log(x)) + self.N * math.log(self.B) - L


def _sweep64(src, dst, rows, b, B, sweep_id):
    """one sweep: the new labels and its counters"""
    n = b.numel()
    M = _Counts(src, dst, b, B)
    at, k, kout, kin, first, nbr = rows
    live = torch.nonzero(k > 0).flatten()
    w0, w1, w2, _ = _philox(sweep_id, live.cpu().numpy(), 0, 0)
    u = b[nbr[first[live] + _below(w0, k[live])]]
    y = _below(w1, M.d[u] + B)
    s = torch.where(y < B, y, M.far(u, (y - B).clamp_(min=0)))
    moves = s != b[live]
    v, s = live[moves], s[moves]
    r, m = b[v], v.numel()
    slot = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    slot[v] = torch.arange(m, device="cuda")
    # each mover's counts of edges to and from its neighbours' blocks
    keep = (slot[at] >= 0) & (nbr != at)
    out = torch.arange(at.numel(), device="cuda") - first[at] < kout[at]
    ent, inv = torch.unique((slot[at] * B + b[nbr])[keep], return_inverse=True)
    ko = torch.bincount(inv[out[keep]], minlength=ent.numel())
    ki = torch.bincount(inv[~out[keep]], minlength=ent.numel())
    loops = torch.zeros(m, dtype=torch.int64, device="cuda")
    sl = (slot[at] >= 0) & (nbr == at) & out
    loops.index_add_(0, slot[at][sl], torch.ones_like(at[sl]))
    q, t = ent // B, ent % B
    zero = torch.zeros(m, dtype=torch.int64, device="cuda")
    own = {}
    for name, blk in (("r", r), ("s", s)):
        h = t == blk[q]
        own[name] = (zero.index_add(0, q[h], ko[h]), zero.index_add(0, q[h], ki[h]))
    h = (t != r[q]) & (t != s[q])
    q, t, ko, ki = q[h], t[h], ko[h], ki[h]
    rt, st_, tr, ts = M.at(r[q], t), M.at(s[q], t), M.at(t, r[q]), M.at(t, s[q])
    zd = torch.zeros(m, dtype=torch.float64, device="cuda")
    dL = zd.index_add(0, q, _f(rt - ko) - _f(rt) + _f(st_ + ko) - _f(st_) + _f(tr - ki) - _f(tr) + _f(ts + ki) - _f(ts))
    c, den = (ko + ki).double(), (M.d[t] + B).double()
    pf = zd.index_add(0, q, c * (ts + st_ + 1).double() / den)
    pb = zd.index_add(0, q, c * (tr - ki + rt - ko + 1).double() / den)
    (kor, kir), (kos, kis) = own["r"], own["s"]
    cr, cs, Ko, Ki, K = kor + kir, kos + kis, kout[v], kin[v], k[v]
    rr, ss, rs, sr = M.at(r, r), M.at(s, s), M.at(r, s), M.at(s, r)
    for x, d in ((rr, -(cr + loops)), (ss, cs + loops), (rs, kir - kos), (sr, kor - kis)):
        dL += _f(x + d) - _f(x)
    for x, d in ((M.dout[r], -Ko), (M.dout[s], Ko), (M.din[r], -Ki), (M.din[s], Ki)):
        dL -= _f(x + d) - _f(x)
    dr, ds = M.d[r], M.d[s]
    pf += (cr + 2 * loops).double() * (rs + sr + 1).double() / (dr + B).double()
    pf += cs.double() * (2 * ss + 1).double() / (ds + B).double()
    pb += cr.double() * (2 * (rr - cr - loops) + 1).double() / (dr - K + B).double()
    pb += (cs + 2 * loops).double() * (sr + kor - kis + rs + kir - kos + 1).double() / (ds + K + B).double()
    uni = torch.from_numpy((w2 >> np.uint64(11)).astype(np.float64) * 2.0 ** -53).cuda()[moves]
    yes = uni.log() < 3.0 * dL + pb.log() - pf.log()
    b = b.clone()
    b[v[yes]] = s[yes]
    return b, (live.numel(), m, int(yes.sum()))


def _rows(src, dst, n):
    """every vertex's edge ends, its out-row and then its in-row, each
    ascending by neighbour"""
    one = torch.ones_like(src)
    at = torch.cat([src, dst])
    side = torch.cat([one * 0, one])
    nbr = torch.cat([dst, src])
    order = torch.argsort((at * 2 + side) * n + nbr)
    kout, kin = torch.bincount(src, minlength=n), torch.bincount(dst, minlength=n)
    k = kout + kin
    return at[order], k, kout, kin, k.cumsum(0) - k, nbr[order]


def _merge_round(M, round_id, x=10):
    """best proposal of every block and its Delta DL"""
    B = M.B
    r = torch.arange(B, device="cuda")
    best = torch.full((B,), -1, dtype=torch.int64, device="cuda")
    best_d = torch.zeros(B, dtype=torch.float64, device="cuda")
    best_k = torch.full((B,), 2 ** 62, dtype=torch.int64, device="cuda")

    def g(a, c):  # f(a + c) - f(a) - f(c)
        return _f(a + c) - _f(a) - _f(c)

    for i in range(x):
        w0, w1, _, _ = _philox(round_id, np.arange(B, dtype=np.uint64), i, 1)
        has = M.d > 0
        u = torch.where(has, M.far(r, _below(w0, M.d.clamp(min=1))), r)
        ur, ru = M.at(u, r), M.at(r, u)
        y = _below(w1, torch.where(has, B - 1 + M.d[u] - ur - ru, torch.full_like(r, B - 1)))
        t = (y - (B - 1)).clamp_(min=0)
        roww = M.dout[u] - ur
        pre_r, pre_c = M.before(u, r)
        tc = t - roww
        by_row = M.in_row(u, torch.where(t >= pre_r, t + ur, t))
        by_col = M.in_col(u, torch.where(tc >= pre_c, tc + ru, tc).clamp_(min=0))
        s = torch.where(y < B - 1, y + (y >= r).long(), torch.where(t < roww, by_row, by_col))
        acc = torch.zeros(B, dtype=torch.float64, device="cuda")
        h = (M.col != M.row) & (M.col != s[M.row])
        a, c, val = M.row[h], M.col[h], M.val[h]
        acc.index_add_(0, a, g(M.at(s[a], c), val))
        h = (M.col != M.row) & (M.row != s[M.col])
        a, c, val = M.row[h], M.col[h], M.val[h]
        acc.index_add_(0, c, g(M.at(a, s[c]), val))
        rr, rs, sr, ss = M.at(r, r), M.at(r, s), M.at(s, r), M.at(s, s)
        acc += _f(rr + rs + sr + ss) - _f(rr) - _f(rs) - _f(sr) - _f(ss)
        acc -= g(M.dout[s], M.dout[r]) + g(M.din[s], M.din[r])
        key = torch.floor(-acc * 2.0 ** 20 + 0.5).long()
        less = key < best_k
        best, best_d, best_k = torch.where(less, s, best), torch.where(less, -acc, best_d), torch.where(less, key, best_k)
    return best.cpu().numpy(), best_k.cpu().numpy()


def _merge64(src, dst, b, B, merges):
    rounds = 0
    while merges > 0 and B >= 2:
        s, key = _merge_round(_Counts(src, dst, b, B), rounds)
        rounds += 1
        parent = list(range(B))

        def find(x):
            while parent[x] != x:
                parent[x] = parent[parent[x]]
                x = parent[x]
            return x

        done = 0
        for r in np.lexsort((np.arange(B), key)):
            if done == merges:
                break
            a, c = find(int(r)), find(int(s[r]))
            if a != c:
                parent[a] = c
                done += 1
        root = np.array([find(c) for c in range(B)])
        _, first, inv = np.unique(root, return_index=True, return_inverse=True)
        rank = np.empty(first.size, np.int64)
        rank[np.argsort(first)] = np.arange(first.size)
        b = torch.from_numpy(rank[inv]).cuda()[b]
        B = first.size
        merges -= done
        if done == 0:
            break
    return b, B, rounds


def exact(case, seed):
    if case["kind"] in ("partition", "batch"):
        return None  # hundreds of sweeps and merge rounds: minutes
    B = case["B"]
    src, dst, b = (x.long() for x in _inputs(case, seed))
    if case["kind"] == "score":
        M = _Counts(src, dst, b, B)
        dense = torch.bincount(b[src] * B + b[dst], minlength=B * B)
        return {"dl": M.dl(), "dout": M.dout.int(), "din": M.din.int(), "M": dense.reshape(B, B).int()}
    if case["kind"] == "merge":
        b, B, rounds = _merge64(src, dst, b, B, case["merges"])
        M = _Counts(src, dst, b, B)
        return {"labels": b.int(), "dout": M.dout.int(), "din": M.din.int(), "dl": M.dl(), "B": B, "rounds": rounds}
    rows = _rows(src, dst, case["n"])
    dl, counts = [], []
    for i in range(case["sweeps"]):
        b, c = _sweep64(src, dst, rows, b, B, i)
        counts.append(c)
        M = _Counts(src, dst, b, B)
        dl.append(M.dl())
    return {"labels": b.int(), "dout": M.dout.int(), "din": M.din.int(), "dl": np.array(dl),
            "counts": np.array(counts)}
