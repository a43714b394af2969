"""Column pointers of k = 6 on both sides of as many k-mers as there are codes (191 M, some
400,000 proteins): right, and without a jump in their time.

The pointers are formed by tiles of codes or by a search per code.  The work grows by a thirteenth
from 186 to 200 M residues; the bound leaves half as much again, where the searches take nearly four
times as long as the tiles at this size."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# residues per 10,000 in the order ARNDCQEGHILKMFPSTWYV (background frequencies of proteins)
FREQ = [780, 512, 448, 536, 192, 426, 629, 737, 219, 514, 901, 574, 224, 385, 520, 711, 584, 132, 321, 644]


def _residues(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    edges = torch.cumsum(torch.tensor(FREQ, device="cuda", dtype=torch.float32), 0)
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    for s in range(0, n, 1 << 25):
        m = min(1 << 25, n - s)
        u = torch.rand(m, generator=g, device="cuda") * edges[-1]
        out[s:s + m] = torch.searchsorted(edges, u).clamp_(max=19).to(torch.uint8)
    return out


def test_no_jump_where_kmers_outnumber_codes():
    import paper_2009_14467_gb300 as P
    ctx = P.Context(0)
    length, ms = 500, {}
    for n_seqs in (372_000, 400_000):
        codes = _residues(n_seqs * length, n_seqs)
        offsets = torch.arange(0, n_seqs * length + 1, length, device="cuda", dtype=torch.int64)
        for _ in range(3):
            ctx.profile(True)
            A = P.build_kmers(ctx, codes, offsets, 6)
            t = ctx.profile_read()["col_ptr"][1]
            ms[n_seqs] = min(ms.get(n_seqs, t), t)
            ctx.profile(False)
        n = torch.bincount(A.row_code[:A.nnz], minlength=24 ** 6)
        assert int(A.col_ptr[0]) == 0 and n.numel() == 24 ** 6
        assert torch.equal(A.col_ptr[1:].long(), torch.cumsum(n, 0))
        del A, n, codes, offsets
        torch.cuda.empty_cache()
    ctx.close()
    assert ms[400_000] <= 1.5 * ms[372_000]
