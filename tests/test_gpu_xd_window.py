"""The x-drop's window against the oracle, for every lane setting and both modes: ranges that
end where single rows fall below the limit, ranges about as wide as the window, and paths
that leave the window on either side and come back.  Records and the number of cells computed,
so that a row kept alive for one antidiagonal too long shows.  Whole numbers, so equality."""
import numpy as np
import pytest
import torch

import synth
from oracle import oracle as O

pytestmark = pytest.mark.gpu

MAT = synth.blosum62()
LETTERS = np.array(list("ACDEFGHIKLMNPQRSTVWY"))


def _check(strings, pairs, seeds, **kw):
    import paper_2009_14467_gb300 as P
    ps = synth.from_strings(strings)
    codes = O.encode(ps.ascii)
    c = np.zeros(len(pairs), O.CAND_DTYPE)
    c["i"], c["j"], c["count"] = pairs[:, 0], pairs[:, 1], 1
    c["qpos"][:, 0], c["tpos"][:, 0] = seeds[:, 0], seeds[:, 1]
    c["qpos"][:, 1] = c["tpos"][:, 1] = 0xFFFF
    dev = [torch.from_numpy(x).cuda() for x in (codes, ps.offsets, c.view(np.uint8).reshape(-1, 20))]
    ctx = P.Context(0)
    for mode in (P.XD_FILTERED, P.XD):
        params = P.Params(matrix=MAT, mode=mode, **kw)
        want, wcells = O.align_pairs(codes, ps.offsets, c, MAT, params.gap_open, params.gap_extend, mode, params.xdrop,
                                     params.k, params.ani_min_pct, params.cov_min_pct)
        for per_warp in (0, 1, 2, 4):
            ctx.set_xd_layout(per_warp)
            cells = torch.zeros(1, dtype=torch.int64, device="cuda")
            got = P.to_records(P.align_pairs(ctx, *dev, params, cells), P.ALN_DTYPE)
            assert got.tobytes() == want.tobytes(), (mode, per_warp)
            assert int(cells.item()) == wcells, (mode, per_warp)
    ctx.close()


def _random(rng, n):
    return "".join(rng.choice(LETTERS, size=n))


@pytest.mark.parametrize("X", [20, 49, 55])
def test_ends_of_the_range(X):
    """Unrelated sequences of every length around the range's width, aligned from their first
    residues: the range's ends meet the limit and the sequences' ends in every order."""
    rng = np.random.default_rng(X)
    strings = [_random(rng, n) for n in range(6, 76)]
    i, j = np.meshgrid(np.arange(len(strings)), np.arange(len(strings)), indexing="ij")
    pairs = np.stack([i.ravel(), j.ravel()], 1)[(i != j).ravel()]
    _check(strings, pairs, np.zeros((len(pairs), 2), np.int64), xdrop=X)


@pytest.mark.parametrize("o,e,X", [(11, 1, x) for x in range(57, 69)] + [(5, 2, x) for x in (97, 103, 109, 115)])
def test_range_about_as_wide_as_the_window(o, e, X):
    """At a best score of 0 the range takes in the gaps of up to (X - o) / e + 1 residues
    either way: 95 to 117 diagonals here, and the window holds 128 in steps of a lane."""
    rng = np.random.default_rng(100 * o + X)
    strings = [_random(rng, int(n)) for n in rng.integers(150, 600, 24)]
    pairs = np.array([(a, b) for a in range(24) for b in range(24) if a != b][::3])
    lens = np.array([len(s) for s in strings])
    seeds = (rng.random((len(pairs), 2)) * (lens[pairs] - 6)).astype(np.int64)
    _check(strings, pairs, seeds, gap_open=o, gap_extend=e, xdrop=X)


@pytest.mark.parametrize("gap", [9, 17, 30])
@pytest.mark.parametrize("X", [49, 60])
def test_paths_past_both_edges_of_the_window(gap, X):
    """Relatives whose path drifts by a gap every 60 residues, 12 in one direction and then 12 in
    the other, extended to both sides from a seed in the middle and from either end."""
    rng = np.random.default_rng(1000 * gap + X)
    strings, pairs, seeds = [], [], []
    for first in (0, 1):
        for p_sub in (0.0, 0.1):
            base = rng.choice(LETTERS, size=60 * 25)
            two, starts = [[], []], []
            for x in range(25):
                if x % 12 == 0:
                    starts.append(tuple(sum(map(len, t)) for t in two))
                piece = base[60 * x:60 * x + 60]
                other = piece.copy()
                hit = rng.random(60) < p_sub
                other[hit] = rng.choice(LETTERS, size=int(hit.sum()))
                two[0].append(piece)
                two[1].append(other)
                if x < 24:
                    two[first if x < 12 else 1 - first].append(rng.choice(LETTERS, size=gap))
            n = len(strings)
            strings += ["".join(np.concatenate(t)) for t in two]
            for a, b in starts:
                pairs += [(n, n + 1), (n + 1, n)]
                seeds += [(a, b), (b, a)]
    _check(strings, np.array(pairs), np.array(seeds), xdrop=X)
