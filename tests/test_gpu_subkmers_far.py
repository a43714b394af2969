"""GPU rows of S against the oracle at the furthest cuts: with a matrix of four times BLOSUM62,
k = 3 and m = 128 some roots' m-th k-mer lies 64 or more from the nearest replacements and the
call is refused; without those roots it equals the oracle's.  Whole numbers, so equality."""
import numpy as np
import pytest
import torch

import synth
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale,k,m,furthest", [(4, 3, 128, 60), (5, 3, 64, 60), (4, 2, 128, 60)])
def test_cuts_up_to_the_limit(scale, k, m, furthest):
    import paper_2009_14467_gb300 as P
    mat = np.clip(synth.blosum62().astype(np.int32) * scale, -64, 63).astype(np.int8)
    rng = np.random.default_rng(10 * scale + k)
    roots = np.unique(rng.choice(24 ** k, size=min(1500, 24 ** k), replace=False).astype(np.uint32))
    want_c, want_d = O.subkmers(roots, k, m, mat)
    m32 = mat.astype(np.int32)
    least = (np.diag(m32)[:, None] - m32).min(axis=1)
    digits = (roots[:, None].astype(np.int64) // 24 ** np.arange(k)) % 24
    cut = want_d[:, 1:].max(axis=1) - least[digits].sum(axis=1)
    near = cut < 64
    assert 0 < near.sum() < len(roots) and cut[near].max() >= furthest

    def call(r):
        return P.substitute_kmers(ctx, torch.from_numpy(r.view(np.int32).copy()).cuda(),
                                  P.Params(matrix=mat, k=k, m_subs=m))

    ctx = P.Context(0)
    with pytest.raises(P.PastisError) as e:
        call(roots)
    assert e.value.status == 8
    gc, gd = call(roots[near])
    ctx.close()
    assert (gc.cpu().numpy().view(np.uint32) == want_c[near]).all()
    assert (gd.cpu().numpy() == want_d[near]).all()
