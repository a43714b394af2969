"""Smith-Waterman where the device has room for the buffers a call needs but not for the
optional bands of passes 2 and 3 beside them: the call goes through on the rectangles, with the
same records, wherever between the two the room lies.

The rest of the device is held by one allocation while a call runs.  What a call needs is the
workspace of the score-only mode, which takes the same buffers but the bands."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
MAT = synth.blosum62()
SLACK = 64 << 20                     # rounding of a dozen allocations, and the call's output


def _set(P, n_pairs, q_len, seed):
    rng = np.random.default_rng(seed)
    lens = np.concatenate([np.full(8, q_len), rng.integers(10, 61, 500)])
    offs = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=offs[1:])
    c = np.zeros(n_pairs, P.CAND_DTYPE)
    c["i"] = np.sort(rng.integers(0, 8, n_pairs))
    c["j"] = 8 + rng.integers(0, 500, n_pairs)
    c["count"] = 1
    return (torch.from_numpy(rng.integers(0, 20, int(offs[-1]), dtype=np.uint8)).cuda(),
            torch.from_numpy(offs).cuda(), torch.from_numpy(c.view(np.uint8).reshape(-1, 20)).cuda())


def _with_room(room, call):
    """The call's result with `room` bytes of the device free."""
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - room, dtype=torch.uint8, device="cuda")
    try:
        return call()
    finally:
        torch.cuda.synchronize()
        del hog
        torch.cuda.empty_cache()


def test_bands_never_take_the_room_of_a_needed_buffer():
    import paper_2009_14467_gb300 as P
    codes, offs, pairs = _set(P, 400_000, 1000, 1)
    need, full = P.Params(matrix=MAT, mode=P.SW_SCORE), P.Params(matrix=MAT, mode=P.SW)
    ctx = P.Context(0)
    P.align_pairs(ctx, codes, offs, pairs, need)
    needed = ctx.workspace_bytes
    want = P.align_pairs(ctx, codes, offs, pairs, full).cpu()
    bands = ctx.workspace_bytes - needed
    ctx.close()
    assert bands > 2 * SLACK
    for part in (0.1, 0.4, 0.7, 1.1):
        ctx = P.Context(0)
        got = _with_room(needed + SLACK + int(part * bands), lambda: P.align_pairs(ctx, codes, offs, pairs, full).cpu())
        ctx.close()
        assert torch.equal(got, want), part


def test_bands_of_an_earlier_call_make_room():
    import paper_2009_14467_gb300 as P
    codes, offs, pairs = _set(P, 400_000, 1000, 2)
    big = _set(P, 1000, 3000, 3)
    need, full = P.Params(matrix=MAT, mode=P.SW_SCORE), P.Params(matrix=MAT, mode=P.SW)
    ctx = P.Context(0)
    want = P.align_pairs(ctx, *big, need).cpu()
    ctx.close()
    ctx = P.Context(0)
    P.align_pairs(ctx, codes, offs, pairs, full)
    # the stripe buffers of 3,000 columns are 350 MB and the ones they replace 130 MB
    got = _with_room(128 << 20, lambda: P.align_pairs(ctx, *big, need).cpu())
    ctx.close()
    assert torch.equal(got, want)
