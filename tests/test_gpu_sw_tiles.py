"""GPU Smith-Waterman records against the oracle at the edges of pass 1's tiles: rows that
just fill or overflow a group of 8, 16 or 32 lanes and a stripe, runs of one query that
fill a grab or leave halves and groups empty, and best scores tied inside and across
lanes (two-letter sequences).  Whole numbers, so equality."""
import numpy as np
import pytest
import torch

import synth
from oracle import oracle as O

pytestmark = pytest.mark.gpu

MAT = synth.blosum62()
FIELDS = ("score", "qb", "qe", "tb", "te", "ident", "cols", "passes")


def _check(ps, cands, mode, layout=None, **kw):
    import paper_2009_14467_gb300 as P
    ctx = P.Context(0)
    ctx.set_sw_layout(layout)
    codes = O.encode(ps.ascii)
    params = P.Params(matrix=MAT, mode=mode, **kw)
    got = P.to_records(P.align_pairs(ctx, torch.from_numpy(codes).cuda(), torch.from_numpy(ps.offsets).cuda(),
                                     torch.from_numpy(cands.view(np.uint8).reshape(-1, 20)).cuda(), params),
                       P.ALN_DTYPE)
    ctx.close()
    want, _ = O.align_pairs(codes, ps.offsets, cands, MAT, params.gap_open, params.gap_extend, mode, params.xdrop,
                            params.k, params.ani_min_pct, params.cov_min_pct)
    for f in FIELDS:
        bad = np.flatnonzero(got[f] != want[f])
        assert bad.size == 0, f"{f} differs at {bad[:5]}: {got[bad[:3]]} vs {want[bad[:3]]}"


def _seqs(lengths, letters, seed):
    rng = np.random.default_rng(seed)
    return ["".join(rng.choice(list(letters), size=n)) for n in lengths]


def _cands(i, j):
    c = np.zeros(len(i), O.CAND_DTYPE)
    c["i"], c["j"], c["count"] = i, j, 1
    return c


@pytest.mark.parametrize("letters", ["ACDEFGHIKLMNPQRSTVWY", "AW"])
@pytest.mark.parametrize("m", [1, 2, 15, 16, 17, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2049])
def test_rows_at_tile_edges(m, letters):
    targets = [0, 1, 7, 8, 9, 31, 33, 90, 200, 333]
    ps = synth.from_strings(_seqs([m] + targets, letters, m))
    n = len(targets)
    _check(ps, _cands([0] * n, 1 + np.arange(n)), 0)


@pytest.mark.parametrize("count", [1, 2, 3, 5, 17, 33, 64, 513])
@pytest.mark.parametrize("m", [40, 200, 300, 600])
def test_runs_of_one_query(m, count):
    rng = np.random.default_rng(m * 1000 + count)
    ps = synth.from_strings(_seqs([m] + list(rng.integers(1, 120, 40)), "ACDEFGHIKLMNPQRSTVWY", m + count))
    _check(ps, _cands([0] * count, 1 + rng.integers(0, 40, count)), 3, cov_min_pct=5)


@pytest.mark.parametrize("o,e", [(0, 0), (2, 1), (11, 1)])
@pytest.mark.parametrize("extra", [0, 1, 2])
def test_tied_scores(o, e, extra):
    rng = np.random.default_rng(o + extra)
    lengths = [60, 130, 250, 400, 700, 1100] + list(rng.integers(20, 300, 14))
    ps = synth.from_strings(_seqs(lengths, "AG", 10 * o + extra))
    i, j = np.triu_indices(len(lengths), 1)
    _check(ps, _cands(i, j), 0, layout=np.full(64, extra, np.uint8), gap_open=o, gap_extend=e)


@pytest.mark.parametrize("gap", [0, 1, 3, 6, 7, 8, 20, 31, 33, 45, 62, 66, 90, 130, 200])
@pytest.mark.parametrize("o,e", [(11, 1), (5, 2), (12, 0)])
def test_bands_of_gapped_homologs(gap, o, e):
    """Relatives with one long gap on either side (narrow to very wide bands of the reverse
    pass, every ring of the banded third pass and its fall-backs), at 5% to 60%
    substitutions, paths of a few to 700 rows that start and end anywhere."""
    rng = np.random.default_rng(1000 * gap + 10 * o + e)
    letters = np.array(list("ACDEFGHIKLMNPQRSTVWY"))
    strings = []
    for n in (23, 24, 25, 33, 64, 150, 400, 700):
        base = rng.choice(letters, size=n)
        strings.append("".join(base))
        for p_sub in (0.05, 0.3, 0.6):
            x = base.copy()
            hit = rng.random(n) < p_sub
            x[hit] = rng.choice(letters, size=int(hit.sum()))
            cut = int(rng.integers(0, n + 1))
            x = np.concatenate([x[:cut], rng.choice(letters, size=gap), x[cut:]])
            flank = rng.choice(letters, size=int(rng.integers(0, 60)))
            strings.append("".join(np.concatenate([flank, x])))
    ps = synth.from_strings(strings)
    i = np.repeat(np.arange(0, 32, 4), 3)
    j = i + np.tile([1, 2, 3], 8)
    far = [(a, b) for a in range(0, 32, 4) for b in range(a + 4, 32, 9)]
    ii = np.concatenate([i, j, [a for a, _ in far]])
    jj = np.concatenate([j, i, [b for _, b in far]])
    _check(ps, _cands(ii, jj), 0, gap_open=o, gap_extend=e)
    _check(ps, _cands(ii, jj), 3, gap_open=o, gap_extend=e)
