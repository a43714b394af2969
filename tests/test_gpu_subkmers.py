"""GPU rows of S against the oracle where the kernel changes its form: cuts beyond the
distances counted in registers, CTA widths, and partly filled CTAs.  Whole numbers, so
equality."""
import numpy as np
import pytest
import torch

import synth
from oracle import oracle as O

pytestmark = pytest.mark.gpu

MAT = synth.blosum62()


def _check(roots, k, m, mat):
    import paper_2009_14467_gb300 as P
    ctx = P.Context(0)
    want_c, want_d = O.subkmers(roots, k, m, mat)
    # distances count from the nearest replacement of every position; a root whose m-th
    # k-mer lies 64 or more from there is refused
    m32 = mat.astype(np.int32)
    least = (np.diag(m32)[:, None] - m32).min(axis=1)
    digits = (roots[:, None].astype(np.int64) // 24 ** np.arange(k)) % 24
    if (want_d[:, 1:].max(axis=1) - least[digits].sum(axis=1) >= 64).any():
        with pytest.raises(P.PastisError) as e:
            P.substitute_kmers(ctx, torch.from_numpy(roots.view(np.int32).copy()).cuda(),
                               P.Params(matrix=mat, k=k, m_subs=m))
        assert e.value.status == 8
        ctx.close()
        return
    gc, gd = P.substitute_kmers(ctx, torch.from_numpy(roots.view(np.int32).copy()).cuda(),
                                P.Params(matrix=mat, k=k, m_subs=m))
    assert (gc.cpu().numpy().view(np.uint32) == want_c).all()
    assert (gd.cpu().numpy() == want_d).all()
    ctx.close()


@pytest.mark.parametrize("scale,k,m", [(3, 6, 25), (4, 6, 50), (4, 3, 128), (3, 1, 23), (2, 6, 128)])
def test_far_cuts(scale, k, m):
    rng = np.random.default_rng(scale * 100 + m)
    roots = np.unique(rng.choice(24 ** k, size=min(600, 24 ** k), replace=False).astype(np.uint32))
    _check(roots, k, m, (MAT.astype(np.int32) * scale).astype(np.int8))


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 400])
@pytest.mark.parametrize("m", [1, 33, 34, 35, 68, 69, 89])
def test_cta_widths(n, m):
    rng = np.random.default_rng(1000 * n + m)
    _check(np.sort(rng.choice(24 ** 6, size=n, replace=False)).astype(np.uint32), 6, m, MAT)
