"""GPU candidates against the oracle where a row changes its form: every number of products
around the sizes of the sorted rows (256 to 4,096 words, a table above), rows whose products
all meet one column, and counts below min_shared.  Whole numbers, so equality."""
import numpy as np
import pytest
import torch

import synth
from oracle import oracle as O

pytestmark = pytest.mark.gpu

LETTERS = list("ACDEFGHIKLMNPQRSTVWYBZX*")


def _check(strings, k, m=0, min_shared=1):
    import paper_2009_14467_gb300 as P
    mat = synth.blosum62()
    ctx = P.Context(0)
    ps = synth.from_strings(strings)
    codes = O.encode(ps.ascii)
    params = P.Params(matrix=mat, k=k, m_subs=m, min_shared=min_shared)
    A = P.build_kmers(ctx, torch.from_numpy(codes).cuda(), torch.from_numpy(ps.offsets).cuda(), k)
    got = P.to_records(P.overlap_spgemm(ctx, A, params), P.CAND_DTYPE)
    rp, code, pos = O.kmers(codes, ps.offsets, k)
    assert got.tobytes() == O.candidates(rp, code, pos, k, m, mat, min_shared).tobytes()
    ctx.close()


@pytest.mark.parametrize("n,windows,min_shared", [(4200, 1, 1), (1400, 3, 3), (700, 6, 7)])
def test_every_number_of_products(n, windows, min_shared):
    # row i meets the n - 1 - i sequences after it in each of its windows
    _check(["ACDEFGHIK"[:windows + 2]] * n, 3, 0, min_shared)


@pytest.mark.parametrize("windows", [255, 256, 257, 4095, 4096, 4097])
def test_products_of_one_column(windows):
    rng = np.random.default_rng(windows)
    a = "".join(rng.choice(LETTERS, size=windows + 3))
    while len({a[x:x + 4] for x in range(windows)}) < windows:      # distinct windows, so one entry each
        a = "".join(rng.choice(LETTERS, size=windows + 40))
        seen, b = set(), a[:3]
        for c in a[3:]:
            if b[-3:] + c not in seen:
                seen.add(b[-3:] + c)
                b += c
        a = b[:windows + 3]
    _check([a, a], 4)


@pytest.mark.parametrize("k,m,min_shared", [(2, 3, 1), (3, 7, 2), (4, 25, 1), (4, 25, 3)])
def test_rows_of_both_orientations(k, m, min_shared):
    rng = np.random.default_rng(100 * k + m + min_shared)
    strings = ["".join(rng.choice(LETTERS[:20], size=n)) for n in rng.integers(k, 400, 300)]
    _check(strings + strings[:20], k, m, min_shared)
