"""GPU k-mer matrices against the oracle at the edges of the kernels that build them: the
windows' tiles (4,096 positions, up to 1,024 sequences each before offsets are read from
memory), the radix sort's tiles (2,048 items) and the column pointers' (8,192 codes from
k = 5 on, one search per code below).
Whole numbers, so equality."""
import numpy as np
import pytest
import torch

import synth
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _check(strings, k):
    import paper_2009_14467_gb300 as P
    ctx = P.Context(0)
    ps = synth.from_strings(strings)
    codes = O.encode(ps.ascii)
    A = P.build_kmers(ctx, torch.from_numpy(codes).cuda(), torch.from_numpy(ps.offsets).cuda(), k)
    rp, code, pos = O.kmers(codes, ps.offsets, k)
    assert A.nnz == len(code)
    assert (A.row_ptr.cpu().numpy() == rp).all()
    assert (A.row_code[:A.nnz].cpu().numpy().view(np.uint32) == code).all()
    assert (A.row_pos[:A.nnz].cpu().numpy().view(np.uint16) == pos).all()
    # the posting lists from the rows: entries by code, then sequence
    seq = np.repeat(np.arange(ps.n), np.diff(rp))
    order = np.lexsort((seq, code))
    cp = np.searchsorted(code[order], np.arange(24 ** k + 1))
    assert (A.col_ptr.cpu().numpy().view(np.uint32) == cp).all()
    assert (A.col_seq[:A.nnz].cpu().numpy() == seq[order]).all()
    assert (A.col_pos[:A.nnz].cpu().numpy().view(np.uint16) == pos[order]).all()
    ctx.close()


def _strings(lengths, seed, letters="ACDEFGHIKLMNPQRSTVWY"):
    rng = np.random.default_rng(seed)
    return ["".join(rng.choice(list(letters), size=n)) for n in lengths]


@pytest.mark.parametrize("k", [1, 2, 4, 5])
def test_thousands_of_tiny_sequences(k):
    rng = np.random.default_rng(k)
    _check(_strings(rng.integers(0, 4, 9000), k), k)


@pytest.mark.parametrize("total", [1, 2, 2047, 2048, 2049, 4095, 4096, 4097, 8191, 8193, 20000])
def test_tile_edges(total):
    _check(_strings([total], total), 3)
    _check(_strings([total // 3, 0, total - total // 3, 5], total), 3)
    _check(_strings([total], total), 5)


@pytest.mark.parametrize("letters", ["A", "*", "A*", "ACDEFGHIKLMNPQRSTVWYBZX*"])
def test_codes_at_the_ends_of_the_range(letters):
    _check(_strings([700, 3, 0, 1200], 5, letters), 4)
    _check(_strings([700, 3, 0, 1200], 6, letters), 3)
    _check(_strings([700, 3, 0, 1200], 7, letters), 5)


@pytest.mark.parametrize("k,m", [(1, 10), (2, 25), (3, 7), (3, 60), (6, 25)])
def test_substitute_candidates_where_few_or_all_codes_are_present(k, m):
    """A S keeps the substitutes that A holds: candidates equal the oracle's where that is
    nearly every code (short k) and nearly none (k = 6 on a small set)."""
    import paper_2009_14467_gb300 as P
    mat = synth.blosum62()
    ctx = P.Context(0)
    rng = np.random.default_rng(10 * k + m)
    ps = synth.from_strings(_strings(list(rng.integers(0, 40 if k < 3 else 300, 30)), k + m,
                                     "ACDEFGHIKLMNPQRSTVWYBZX*"))
    codes = O.encode(ps.ascii)
    params = P.Params(matrix=mat, k=k, m_subs=m)
    A = P.build_kmers(ctx, torch.from_numpy(codes).cuda(), torch.from_numpy(ps.offsets).cuda(), k)
    got = P.to_records(P.overlap_spgemm(ctx, A, params), P.CAND_DTYPE)
    rp, code, pos = O.kmers(codes, ps.offsets, k)
    want = O.candidates(rp, code, pos, k, m, mat, 1)
    assert got.tobytes() == want.tobytes()
    ctx.close()
