"""Pass 1 of Smith-Waterman on short runs of one query, where the last grab of a run leaves
halves of a group, or whole groups, without a pair.

With 17 or 18 targets a query of 60 or 120 residues takes groups of 16 lanes, two pairs each:
the last grab holds one pair or two, in the same registers, so 18 targets take the time of 17
however many columns the empty halves run on.  The bound allows 10% for the noise of two
runs and the targets' lengths, whose means over 600,000 draws differ by less than 0.2%."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
MAT = synth.blosum62()


def _pass1_ms(ctx, P, m, run, n_queries=33000, n_targets=2000):
    rng = np.random.default_rng(m)
    lens = np.concatenate([np.full(n_queries, m), rng.integers(200, 401, n_targets)])
    offs = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=offs[1:])
    codes = torch.from_numpy(rng.integers(0, 20, int(offs[-1]), dtype=np.uint8)).cuda()
    c = np.zeros(n_queries * run, P.CAND_DTYPE)
    c["i"] = np.repeat(np.arange(n_queries), run)
    c["j"] = n_queries + rng.integers(0, n_targets, len(c))
    c["count"] = 1
    pairs = torch.from_numpy(c.view(np.uint8).reshape(-1, 20)).cuda()
    offsets, params = torch.from_numpy(offs).cuda(), P.Params(matrix=MAT, mode=P.SW_SCORE)
    best = float("inf")
    for _ in range(4):
        ctx.profile(True)
        P.align_pairs(ctx, codes, offsets, pairs, params)
        best = min(best, ctx.profile_read()["sw_pass1"][1])
        ctx.profile(False)
    return best


@pytest.mark.parametrize("m", [60, 120])
def test_a_pair_in_an_empty_half_is_free(m):
    import paper_2009_14467_gb300 as P
    ctx = P.Context(0)
    t17, t18 = _pass1_ms(ctx, P, m, 17), _pass1_ms(ctx, P, m, 18)
    ctx.close()
    assert t18 <= 1.1 * t17
