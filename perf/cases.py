"""The calls whose speed matters to a user of this framework, as cases a harness can time.

Each case is one pass through the public entry points on inputs of the shape that the
path meets in earnest: planted protein families and unrelated singletons, lengths
log-normal around a median, 30% substitutions drawn by BLOSUM62 and 5% indels inside a
family (the recipe of this repository's benchmark sets, drawn on the GPU so that a set of
10^5 proteins takes a fraction of a second).
"""
import math

import numpy as np
import torch

from paper_2009_14467_gb300 import pastis as P
from paper_2009_14467_gb300 import prefilter as F
from paper_2009_14467_gb300 import serve as S

LETTERS = "ARNDCQEGHILKMFPSTWYVBZX*"

# BLOSUM62 in LETTERS order (Henikoff & Henikoff 1992), an argument of every call that scores residues
BLOSUM62 = np.array([int(v) for v in """
 4 -1 -2 -2  0 -1 -1  0 -2 -1 -1 -1 -1 -2 -1  1  0 -3 -2  0 -2 -1  0 -4
-1  5  0 -2 -3  1  0 -2  0 -3 -2  2 -1 -3 -2 -1 -1 -3 -2 -3 -1  0 -1 -4
-2  0  6  1 -3  0  0  0  1 -3 -3  0 -2 -3 -2  1  0 -4 -2 -3  3  0 -1 -4
-2 -2  1  6 -3  0  2 -1 -1 -3 -4 -1 -3 -3 -1  0 -1 -4 -3 -3  4  1 -1 -4
 0 -3 -3 -3  9 -3 -4 -3 -3 -1 -1 -3 -1 -2 -3 -1 -1 -2 -2 -1 -3 -3 -2 -4
-1  1  0  0 -3  5  2 -2  0 -3 -2  1  0 -3 -1  0 -1 -2 -1 -2  0  3 -1 -4
-1  0  0  2 -4  2  5 -2  0 -3 -3  1 -2 -3 -1  0 -1 -3 -2 -2  1  4 -1 -4
 0 -2  0 -1 -3 -2 -2  6 -2 -4 -4 -2 -3 -3 -2  0 -2 -2 -3 -3 -1 -2 -1 -4
-2  0  1 -1 -3  0  0 -2  8 -3 -3 -1 -2 -1 -2 -1 -2 -2  2 -3  0  0 -1 -4
-1 -3 -3 -3 -1 -3 -3 -4 -3  4  2 -3  1  0 -3 -2 -1 -3 -1  3 -3 -3 -1 -4
-1 -2 -3 -4 -1 -2 -3 -4 -3  2  4 -2  2  0 -3 -2 -1 -2 -1  1 -4 -3 -1 -4
-1  2  0 -1 -3  1  1 -2 -1 -3 -2  5 -1 -3 -1  0 -1 -3 -2 -2  0  1 -1 -4
-1 -1 -2 -3 -1  0 -2 -3 -2  1  2 -1  5  0 -2 -1 -1 -1 -1  1 -3 -1 -1 -4
-2 -3 -3 -3 -2 -3 -3 -3 -1  0  0 -3  0  6 -4 -2 -2  1  3 -1 -3 -3 -1 -4
-1 -2 -2 -1 -3 -1 -1 -2 -2 -3 -3 -1 -2 -4  7 -1 -1 -4 -3 -2 -2 -1 -2 -4
 1 -1  1  0 -1  0  0  0 -1 -2 -2  0 -1 -2 -1  4  1 -3 -2 -2  0  0  0 -4
 0 -1  0 -1 -1 -1 -1 -2 -2 -1 -1 -1 -1 -2 -1  1  5 -2 -2  0 -1 -1  0 -4
-3 -3 -4 -4 -2 -2 -3 -2 -2 -3 -2 -3 -1  1 -4 -3 -2 11  2 -3 -4 -3 -2 -4
-2 -2 -2 -3 -2 -1 -2 -3  2 -1 -1 -2 -1  3 -3 -2 -2  2  7 -1 -3 -2 -1 -4
 0 -3 -3 -3 -1 -2 -2 -3 -3  3  1 -2  1 -1 -2 -2  0 -3 -1  4 -3 -2 -1 -4
-2 -1  3  4 -3  0  1 -1  0 -3 -4  0 -3 -3 -2  0 -1 -4 -3 -3  4  1 -1 -4
-1  0  0  1 -3  3  4 -2  0 -3 -3  1 -1 -3 -1  0 -1 -3 -2 -2  1  4 -1 -4
 0 -1 -1 -1 -2 -1 -1 -1 -1 -1 -1 -1 -1 -1 -2  0  0 -2 -1 -1 -1 -1 -1 -4
-4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4  1
""".split()], np.int8).reshape(24, 24)
BACKGROUND = np.array([0.074, 0.052, 0.045, 0.054, 0.025, 0.034, 0.054, 0.074, 0.026, 0.068,
                       0.099, 0.058, 0.025, 0.047, 0.039, 0.057, 0.051, 0.013, 0.032, 0.073])

MODES = {"sw": P.SW, "sw_filtered": P.SW_FILTERED, "sw_score": P.SW_SCORE, "xd": P.XD, "xd_filtered": P.XD_FILTERED}

# Share of all pairs that are candidates at a median length of 300, by substitutes per k-mer:
# random pairs that share a 6-mer by chance (family pairs come on top, about 20 a sequence).
DENSITY = {0: 0.005, 10: 0.045, 25: 0.1}
DEV = "cuda:0"


def listed():
    return [
        # an all-vs-all search of a small set, the whole path in one call: many short kernels
        # and host round trips, the smallest thing a user runs
        dict(name="path_1k", kind="path", n=1000, lo=50, hi=1000, median=300, subs=0, mode="sw_filtered"),
        # the benchmark's job at a size one pass holds: 25 substitute k-mers, Smith-Waterman
        # of every candidate for the filter
        dict(name="path_5k_subs25", kind="path", n=5000, lo=50, hi=1000, median=300, subs=25, mode="sw_filtered"),
        # encode and the k-mer matrix of a benchmark-sized set
        dict(name="kmers_100k", kind="kmers", n=100000, lo=50, hi=1000, median=300, k=6),
        # candidate discovery with 25 substitute k-mers, S and A S built anew, as for a new set
        dict(name="overlap_subs25_20k", kind="overlap", n=20000, lo=50, hi=1000, median=300, subs=25, rows=1.0,
             min_shared=1),
        # candidate discovery with exact k-mers: one row block of a large set
        dict(name="overlap_exact_200k", kind="overlap", n=200000, lo=50, hi=2000, median=300, subs=0, rows=0.125,
             min_shared=1),
        # Smith-Waterman for the filter on substitute candidates, nearly all of them random
        # pairs: the dominant stage of the benchmark
        dict(name="sw_filtered_1m", kind="align", n=20000, lo=50, hi=1000, median=300, subs=25, mode="sw_filtered",
             pairs=1000000),
        # full Smith-Waterman records of family-rich candidates of long proteins
        dict(name="sw_long_100k", kind="align", n=8000, lo=50, hi=2000, median=800, subs=0, mode="sw",
             pairs=100000),
        # x-drop for the filter on exact candidates of a large set: the 1M configuration's alignment
        dict(name="xd_filtered_2m", kind="align", n=200000, lo=50, hi=2000, median=300, subs=0, mode="xd_filtered",
             pairs=2000000),
        # full x-drop records, family-rich
        dict(name="xd_300k", kind="align", n=20000, lo=50, hi=1000, median=300, subs=0, mode="xd", pairs=300000),
        # a small serving request against a resident database: encode, query k-mers,
        # candidates, alignment replayed from a plan, filter; latency is what counts
        dict(name="serve_16", kind="serve", n=100000, lo=50, hi=2000, median=300, queries=16),
        # the learned prefilter applied to a block of candidates: features, logits, selection
        dict(name="prefilter_apply_1m", kind="apply", n=20000, lo=50, hi=1000, median=300, subs=25, pairs=1000000),
        # one training step of the prefilter at the driver's batch size
        dict(name="prefilter_train_64k", kind="train", batch=65536),
    ]


def _mean_length(case):
    return min(case["median"] * math.exp(0.18), 0.75 * case["hi"])


def _expected_candidates(case, rows=1.0):
    """Candidates of the first `rows` of the set's rows, roughly."""
    n, d = case["n"], min(0.8, DENSITY[case.get("subs", 0)] * (_mean_length(case) / 355) ** 2)
    return int((1 - (1 - rows) ** 2) * (n * n / 2 * d + 20 * n))


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    """A case of the same kinds, with sizes spread over the range the listed ones span."""
    kind = rng.choice(["path", "path", "kmers", "overlap", "overlap", "align", "align", "align", "align", "serve",
                       "apply", "train"])
    c = dict(kind=kind, lo=50, hi=rng.choice([1000, 2000]), median=rng.choice([150, 300, 500]))
    if kind == "path":
        c["subs"] = rng.choice([0, 10, 25])
        c["n"] = _log(rng, 100, 3000 if c["subs"] else 8000)
        c["mode"] = rng.choice(["sw", "sw_filtered", "xd", "xd_filtered"])
        c["median"] = rng.choice([150, 300])
    elif kind == "kmers":
        c["n"] = _log(rng, 300, 60000)
        c["k"] = rng.choice([4, 5, 6, 6])
    elif kind == "overlap":
        c["subs"] = rng.choice([0, 10, 25])
        c["n"] = _log(rng, 500, 8000 if c["subs"] else 120000)
        c["rows"] = rng.choice([1.0, 0.5]) if c["n"] <= 8000 else 0.125
        c["min_shared"] = rng.choice([1, 1, 2, 4])
    elif kind == "align":
        c["subs"] = rng.choice([0, 25])
        c["n"] = _log(rng, 1000, 10000)
        c["mode"] = rng.choice(["sw", "sw_filtered", "sw_score", "xd", "xd_filtered"])
        c["pairs"] = min(_log(rng, 300, 60000 if c["mode"] == "sw" else 300000), _expected_candidates(c) // 2)
    elif kind == "serve":
        c["n"] = _log(rng, 2000, 60000)
        c["queries"] = _log(rng, 1, 500)
    elif kind == "apply":
        c["subs"], c["n"] = 25, _log(rng, 1000, 10000)
        c["pairs"] = min(_log(rng, 1000, 600000), _expected_candidates(c) // 2)
    else:
        c = dict(kind=kind, batch=_log(rng, 1000, 60000))
    return c


# ---- inputs -----------------------------------------------------------------------------
def _proteins(n, lo, hi, median, seed):
    """n proteins as letters (uint8, device) with offsets (int64, device): 80% in n/10
    families of Zipf sizes, the rest singletons, shuffled."""
    rng = np.random.default_rng([seed, n, lo, hi, median])
    g = torch.Generator(device=DEV).manual_seed(int(rng.integers(1 << 62)))
    n_fam, members = max(1, n // 10), int(round(0.8 * n))
    w = np.arange(1, 201, dtype=np.float64) ** -1.5
    sizes = rng.choice(np.arange(1, 201), n_fam, p=w / w.sum())
    fam = rng.choice(n_fam, members, p=sizes / sizes.sum())
    n_root = n_fam + n - members
    root_len = np.clip(np.rint(np.exp(rng.normal(np.log(median), 0.6, n_root))), lo, hi).astype(np.int64)
    order = rng.permutation(n)
    root_of = torch.from_numpy(np.concatenate([fam, np.arange(n_fam, n_root)])[order]).to(DEV)
    rlen = torch.from_numpy(root_len).to(DEV)
    rstart = torch.cumsum(rlen, 0) - rlen
    # letters drawn from tables of 4,096 entries: the background, and the replacements of each residue
    bg = torch.from_numpy(_table(BACKGROUND)).to(DEV)
    sub_p = BACKGROUND[None, :] * 2.0 ** (BLOSUM62[:20, :20].astype(np.float64) / 2.0)
    np.fill_diagonal(sub_p, 0.0)
    sub = torch.from_numpy(np.stack([_table(p / p.sum()) for p in sub_p])).to(DEV).reshape(-1)

    def pick(count):
        return torch.randint(4096, (count,), device=DEV, generator=g)

    def chance(count):
        return torch.rand(count, device=DEV, generator=g)

    def geometric(count):                      # lengths of mean 3
        u = chance(count).clamp_min(1e-7)
        return 1 + torch.floor(torch.log(u) / math.log(2.0 / 3.0)).long()

    roots = bg[pick(int(rlen.sum()))]
    ln = rlen[root_of]
    start = torch.cumsum(ln, 0) - ln
    seq = torch.repeat_interleave(torch.arange(n, device=DEV), ln)
    total = seq.numel()
    res = roots[torch.arange(total, device=DEV) + (rstart[root_of] - start)[seq]]
    member = (root_of < n_fam)[seq]
    hit = member & (chance(total) < 0.30)
    res = torch.where(hit, sub[res * 4096 + pick(total)], res)
    # indel events at 0.05/3 per position, half deletions, half insertions
    u = chance(total)
    rate = 0.05 / 3
    dele = torch.nonzero(member & (u < rate / 2)).reshape(-1)
    mark = torch.zeros(total + 1, dtype=torch.int32, device=DEV)
    end = torch.minimum(dele + geometric(dele.numel()), (start + ln)[seq[dele]])
    one = torch.ones(dele.numel(), dtype=torch.int32, device=DEV)
    mark.index_add_(0, dele, one)
    mark.index_add_(0, end, -one)
    copies = (torch.cumsum(mark[:-1], 0) == 0).long()
    ins = torch.nonzero(member & (u >= rate / 2) & (u < rate)).reshape(-1)
    copies[ins] += geometric(ins.numel())
    src = torch.repeat_interleave(torch.arange(total, device=DEV), copies)
    first = torch.ones(src.numel(), dtype=torch.bool, device=DEV)
    first[1:] = src[1:] != src[:-1]
    res = torch.where(first, res[src], bg[pick(src.numel())])
    # each sequence cut to hi residues
    ln = torch.zeros(n, dtype=torch.int64, device=DEV).index_add_(0, seq, copies)
    start = torch.cumsum(ln, 0) - ln
    seq = seq[src]
    res = res[torch.arange(res.numel(), device=DEV) - start[seq] < hi]
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    offsets[1:] = torch.cumsum(ln.clamp_max(hi), 0)
    letters = torch.from_numpy(np.frombuffer(LETTERS.encode(), np.uint8).copy()).to(DEV)
    return letters[res], offsets


def _table(p, size=4096):
    """size draws whose shares are p (largest remainders)."""
    c = np.floor(p * size).astype(np.int64)
    c[np.argsort(c - p * size, kind="stable")[:size - int(c.sum())]] += 1
    return np.repeat(np.arange(len(p)), c)


def _params(case):
    return P.Params(matrix=BLOSUM62, k=case.get("k", 6), m_subs=case.get("subs", 0),
                    min_shared=case.get("min_shared", 1), mode=MODES[case.get("mode", "sw_filtered")])


def _candidates(codes, offsets, params, pairs):
    """The first `pairs` candidates of the set, in the order the product gives them (from
    the first again where a set has fewer)."""
    ctx = P.Context(0)
    n = offsets.numel() - 1
    A = P.build_kmers(ctx, codes, offsets, params.k)
    rows = min(n, max(64, int(1.5 * pairs / (n * DENSITY[params.m_subs] + 20))))
    cands = P.overlap_spgemm(ctx, A, params, rows=(0, rows))
    while cands.shape[0] < pairs and rows < n:
        rows = min(n, 2 * rows)
        cands = P.overlap_spgemm(ctx, A, params, rows=(0, rows))
    ctx.close()
    return cands.repeat(-(-pairs // cands.shape[0]), 1)[:pairs].contiguous()


def _records(count):
    """A program's own buffer for `count` records, zero where none is written."""
    return torch.zeros((count, P.REC_BYTES), dtype=torch.uint8, device=DEV)


def _keep(buffer, records):
    """Takes a call's records into the program's buffer."""
    if records.shape[0] > buffer.shape[0]:
        raise RuntimeError(f"{records.shape[0]} records for a buffer of {buffer.shape[0]}")
    buffer[:records.shape[0]].copy_(records)
    return buffer


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _prepare_train(case, seed)
    s = dict(kind=kind, params=_params(case))
    n_q = case.get("queries", 0)
    letters, offsets = _proteins(case["n"] + n_q, case["lo"], case["hi"], case["median"], seed)
    s["ctx"] = ctx = P.Context(0)
    # buffers that a program keeps for results whose size a call decides
    room = 20000 + 3 * _expected_candidates(case, case.get("rows", 1.0)) + 60 * case["n"]
    room = min(room, case["n"] * (case["n"] - 1) // 2)
    if kind == "path":
        s.update(letters=letters, offsets=offsets, out=[_records(room) for _ in range(3)])
    elif kind == "kmers":
        n, k = case["n"], s["params"].k
        cap = n * case["hi"] if n < 5000 else int(1.6 * case["median"] * n)
        A = P.kmat_alloc(n, cap, k, DEV)
        for t in (A.row_code, A.row_pos, A.col_seq, A.col_pos):
            t.zero_()
        s.update(letters=letters, offsets=offsets, A=A, codes=torch.zeros(cap, dtype=torch.uint8, device=DEV))
    elif kind == "overlap":
        s["A"] = P.build_kmers(ctx, P.encode(ctx, letters), offsets, s["params"].k)
        s["rows"] = (0, max(1, int(case["n"] * case["rows"])))
        s["out"] = _records(room)
    elif kind in ("align", "apply"):
        codes = P.encode(ctx, letters)
        s.update(codes=codes, offsets=offsets, pairs=_candidates(codes, offsets, s["params"], case["pairs"]))
        if kind == "apply":
            s["out"] = _records(case["pairs"])
            s["net"] = F.MLP(DEV, seed=seed % (1 << 31))
            # a threshold that keeps 7% of the candidates, as a calibrated one does
            x = F.features(ctx, codes, offsets, s["pairs"], s["params"])
            z = _mlp64(s["net"], x.double())[2]
            s["threshold"] = float(torch.sort(z).values[int(0.93 * (z.numel() - 1))])
    else:                                        # serve: the last sequences are the request's
        s["params"] = P.Params(matrix=BLOSUM62, mode=P.XD_FILTERED)
        cut = int(offsets[case["n"]])
        s["db_codes"] = P.encode(ctx, letters[:cut].contiguous())
        s["db_offsets"] = offsets[:case["n"] + 1].contiguous()
        s["DB"] = P.build_kmers(ctx, s["db_codes"], s["db_offsets"], 6)
        s["letters"] = letters[cut:].cpu().numpy()
        s["offsets"] = (offsets[case["n"]:] - cut).cpu().numpy()
        # the serving loop's plan capacities
        s["plan"] = P.AlignPlan(ctx, s["db_codes"], s["db_offsets"], s["params"], 4096, 4 << 20, 1 << 20, 2000)
        s["out"] = [_records(20000 + 3 * n_q * case["n"] // 50 + 200 * n_q) for _ in range(3)]
    return s


def _prepare_train(case, seed):
    """A network in mid-training and a batch of features with the labels' share of positives."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["batch"]

    def normal(*shape):
        return torch.randn(*shape, device=DEV, generator=g)

    net = F.MLP(DEV, seed=seed % (1 << 31))
    for b in (net.b1, net.b2, net.b3):
        b.copy_(0.05 * normal(b.numel()))
    # the values of pair features: counts, seed diagonals, log lengths, seed scores
    ln = torch.log(300.0 * torch.exp(0.6 * normal(n, 2)).clamp(1 / 6, 10 / 3))
    diag = 0.5 * normal(n, 2)
    score = 0.75 + 0.2 * normal(n, 2)
    two = (torch.rand(n, device=DEV, generator=g) < 0.3).float()
    count = torch.exp(normal(n).abs())
    mn, mx = ln.amin(1), ln.amax(1)
    x = torch.stack([torch.log1p(count), diag[:, 0], diag[:, 1], (diag[:, 0] - diag[:, 1]).abs(), ln[:, 0], ln[:, 1],
                     mn, mx, torch.exp(mn - mx), score[:, 0], two * score[:, 1], score[:, 0] + two * score[:, 1],
                     count / torch.exp(mn), two, torch.zeros_like(two), torch.zeros_like(two)], 1).bfloat16()
    y = (torch.rand(n, device=DEV, generator=g) < 0.02 + 0.2 * (score[:, 0] > 1.0)).float()
    net.adam_m.copy_(1e-4 * normal(F.NPARAM))
    net.adam_v.copy_((1e-3 * (1.0 + normal(F.NPARAM).abs())) ** 2)
    net.step = 100
    live = [net.w1, net.b1, net.w2, net.b2, net.w3, net.b3, net.w1b, net.w2b, net.w3b, net.adam_m, net.adam_v]
    return dict(kind="train", ctx=P.Context(0), net=net, x=x.contiguous(), y=y.contiguous(), live=live,
                saved=[t.clone() for t in live], loss=torch.zeros(1, device=DEV), lr=2e-3, pos_weight=4.0)


# ---- one pass -----------------------------------------------------------------------------
def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "path":
        ctx.forget()                             # a new set: S and A S are built with it
        r = P.run(ctx, s["letters"], s["offsets"], s["params"])
        return [_keep(b, r[name]) for b, name in zip(s["out"], ("cands", "alns", "edges"))]
    if kind == "kmers":
        n = s["letters"].numel()
        P.encode(ctx, s["letters"], out=s["codes"])
        A = P.build_kmers(ctx, s["codes"][:n], s["offsets"], s["params"].k, s["A"])
        return [s["codes"], A.row_ptr, A.row_code, A.row_pos, A.col_ptr, A.col_seq, A.col_pos, A.nnz]
    if kind == "overlap":
        ctx.forget()
        return _keep(s["out"], P.overlap_spgemm(ctx, s["A"], s["params"], rows=s["rows"]))
    if kind == "align":
        return P.align_pairs(ctx, s["codes"], s["offsets"], s["pairs"], s["params"])
    if kind == "apply":
        x = F.features(ctx, s["codes"], s["offsets"], s["pairs"], s["params"])
        z = F.forward(ctx, s["net"], x)
        return [x, z, _keep(s["out"], F.select(ctx, s["pairs"], z, s["threshold"]))]
    if kind == "train":
        net = s["net"]
        torch._foreach_copy_(s["live"], s["saved"])      # every pass is the same step
        net.step = 100
        F.train_step(ctx, net, s["x"], s["y"], s["lr"], s["pos_weight"], s["loss"])
        return [s["loss"], net.grad, net.w1, net.b1, net.w2, net.b2, net.w3, net.b3, net.adam_m, net.adam_v]
    # serve: what the serving loop does with one request
    letters = torch.from_numpy(s["letters"]).to(DEV, non_blocking=True)
    offsets = torch.from_numpy(s["offsets"]).to(DEV, non_blocking=True)
    codes = P.encode(ctx, letters)
    Q = P.build_kmers(ctx, codes, offsets, 6)
    cands = S.query_overlap(ctx, Q, s["DB"], s["params"])
    if s["plan"].fits(s["offsets"], cands.shape[0]):
        alns = s["plan"].run(codes, s["offsets"], cands)
    else:
        alns = S.align_pairs_qt(ctx, codes, offsets, s["db_codes"], s["db_offsets"], cands, s["params"])
    edges = S.filter_edges_qt(ctx, offsets, s["db_offsets"], cands, alns, s["params"])
    s["edges"] = P.to_records(edges, P.EDGE_DTYPE)       # what the requester gets
    return [_keep(b, t) for b, t in zip(s["out"], (cands, alns, edges))]


# ---- what a pass cannot do without ------------------------------------------------------------
def work(case):
    """Bytes: each input read and each output written once.  flops: the integer operations of
    the alignments (11 a cell: E 3, F 3, H 4, the running best 1), or the network's products."""
    kind = case["kind"]
    if kind == "train":
        b = case["batch"]
        return {"bytes": b * (16 * 2 + 4) + 12 * F.NPARAM * 4, "flops": 6 * b * (16 * 256 + 256 * 256 + 256)}
    ln = _mean_length(case)
    res = case["n"] * ln
    kmat = res * 12 + 8 * case["n"] + 4 * 24 ** case.get("k", 6)
    per_pair = {"sw": ln * ln, "sw_filtered": ln * ln, "sw_score": ln * ln, "xd": 14000.0, "xd_filtered": 14000.0}
    if kind == "kmers":
        return {"bytes": 3 * res + kmat, "flops": 0}
    if kind == "serve":
        q = case["queries"]
        cands = q * case["n"] * DENSITY[0]
        return {"bytes": q * ln * 14 + cands * 60, "flops": 11 * 14000.0 * cands}
    if kind == "overlap":
        rows, cands = case["rows"], _expected_candidates(case, case["rows"])
        return {"bytes": res * 12 + res * rows * case["subs"] * 12 + cands * 20, "flops": 0}
    if kind == "path":
        cands = _expected_candidates(case)
        return {"bytes": 2 * res + cands * 45, "flops": 11 * per_pair[case["mode"]] * cands}
    if kind == "align":
        return {"bytes": res + case["pairs"] * 40, "flops": 11 * per_pair[case["mode"]] * case["pairs"]}
    return {"bytes": case["pairs"] * (20 + 32 + 4) + 0.07 * 20 * case["pairs"],
            "flops": 2 * case["pairs"] * (16 * 256 + 256 * 256 + 256)}


# ---- the computed numbers in 64 bits ------------------------------------------------------------
def _mlp64(net, x):
    """Hidden activations and logits in float64 from the weights the network computes with."""
    h1 = torch.relu(x @ net.w1b.double() + net.b1.double())
    h2 = torch.relu(h1 @ net.w2b.double() + net.b2.double())
    return h1, h2, h2 @ net.w3b.double() + net.b3.double()


def _features64(s):
    c = s["pairs"].contiguous().view(torch.int32).reshape(-1, 5)
    i, j, count = c[:, 0].long(), c[:, 1].long(), c[:, 2].double()
    pos = s["pairs"].contiguous().view(torch.int16).reshape(-1, 10)[:, 6:].long() & 0xFFFF
    off = s["offsets"]
    lq, lt = (off[i + 1] - off[i]).double(), (off[j + 1] - off[j]).double()
    two = pos[:, 1] != 0xFFFF
    d0 = (pos[:, 0] - pos[:, 2]).double()
    d1 = torch.where(two, (pos[:, 1] - pos[:, 3]).double(), d0)
    mat = torch.from_numpy(BLOSUM62.astype(np.float64)).to(DEV)
    sc = []
    for t in (0, 1):
        v = torch.zeros_like(lq)
        for x in range(s["params"].k):
            a = off[i] + torch.where(two, pos[:, t], 0) + x if t else off[i] + pos[:, 0] + x
            b = off[j] + torch.where(two, pos[:, 2 + t], 0) + x if t else off[j] + pos[:, 2] + x
            v = v + mat[s["codes"][a].long(), s["codes"][b].long()]
        sc.append(torch.where(two, v, 0.0) if t else v)
    mn, mx = torch.minimum(lq, lt), torch.maximum(lq, lt)
    z = torch.zeros_like(lq)
    return torch.stack([torch.log1p(count), d0 / 256, d1 / 256, (d0 - d1).abs() / 256, torch.log(lq + 1),
                        torch.log(lt + 1), torch.log(mn + 1), torch.log(mx + 1), mn / mx.clamp_min(1), sc[0] / 32,
                        sc[1] / 32, (sc[0] + sc[1]) / 32, count / mn.clamp_min(1), two.double(), z, z], 1)


def exact(case, seed):
    if case["kind"] == "apply":
        s = prepare(case, seed)
        x = _features64(s)
        return [x, _mlp64(s["net"], x)[2], None]
    if case["kind"] != "train":
        return None                              # records and codes: whole numbers
    s = prepare(case, seed)
    net, x, y = s["net"], s["x"].double(), s["y"].double()
    h1, h2, z = _mlp64(net, x)
    w = torch.where(y > 0.5, s["pos_weight"], 1.0)
    loss = (w * (torch.nn.functional.softplus(z) - y * z)).mean().reshape(1)
    dz = w * (torch.sigmoid(z) - y) / y.numel()
    dh2 = dz[:, None] * net.w3b.double() * (h2 > 0)
    dh1 = (dh2 @ net.w2b.double().T) * (h1 > 0)
    grads = [x.T @ dh1, dh1.sum(0), h1.T @ dh2, dh2.sum(0), h2.T @ dz, dz.sum().reshape(1)]
    g = torch.cat([v.reshape(-1) for v in grads])
    b1, b2 = 0.9, 0.999
    m = b1 * net.adam_m.double() + (1 - b1) * g
    v = b2 * net.adam_v.double() + (1 - b2) * g * g
    step = net.step + 1
    upd = s["lr"] * (m / (1 - b1 ** step)) / (torch.sqrt(v / (1 - b2 ** step)) + 1e-8)
    out, o = [], 0
    for p in (net.w1, net.b1, net.w2, net.b2, net.w3, net.b3):
        out.append(p.double() - upd[o:o + p.numel()].view(p.shape))
        o += p.numel()
    return [loss, g] + out + [m, v]
