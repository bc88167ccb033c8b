"""FP32 Gram products of more than 48 columns (csrc/blas.cu, gram_kernel): tiles
of 28 to 64 columns, several a side, rows that fill no 32-row stage, columns that
are no multiple of 16 bytes apart."""

import numpy as np
import pytest

from paper_1506_08147_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(18, 20, 15), (18, 15, 15)])
@pytest.mark.parametrize("m", [49, 52, 56, 57, 64, 65, 72, 104, 128, 129, 144])
def test_tiles(m, n):
    ng = int(np.prod(n))
    c = B.Context([dict(n=n, L=(8.0, 8.0, 8.0), e_lo=(0, 0, 0), e_hi=n, m=m, J=m)], precision=B.DGDFT_PREC_MIXED)
    c.dgdft_alb_set_potential(0, np.zeros(ng))
    blk = np.random.default_rng(m).standard_normal((6, m, ng)).astype(np.float32).astype(np.float64)
    a, b, xtw = c.dgdft_alb_lobpcg_gram(0, blk, has_p=True, stage=0)
    c.close()
    s, hs = blk[:3].reshape(3 * m, ng), blk[3:].reshape(3 * m, ng)
    upper = np.kron(np.triu(np.ones((3, 3))), np.ones((m, m)))
    # FP32 sums of 32 products, added up with their rounding errors
    tol = 33 * 2.0 ** -24
    for got, left in ((a, hs), (b, s)):
        bound = tol * (np.abs(left) @ np.abs(s).T)
        assert np.all(np.abs(got - (left @ s.T) * upper) <= bound)
    assert np.all(np.abs(xtw - blk[0] @ blk[1].T) <= tol * (np.abs(blk[0]) @ np.abs(blk[1]).T))
