"""FP64 Gram products of narrow blocks (csrc/fp64_tensor.cu) at
many widths, on grids whose rows do not fill the chunks."""

import numpy as np
import pytest

from paper_1506_08147_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(8, 9, 5), (16, 16, 16), (18, 20, 15)])
@pytest.mark.parametrize("m", [1, 4, 5, 9, 13, 16, 17, 21, 25, 32, 33, 36, 37, 48])
def test_narrow_blocks(m, n):
    ng = int(np.prod(n))
    c = B.Context([dict(n=n, L=(8.0, 8.0, 8.0), e_lo=(0, 0, 0), e_hi=n, m=m, J=m)], precision=B.DGDFT_PREC_FP64)
    c.dgdft_alb_set_potential(0, np.zeros(ng))
    blk = np.random.default_rng(100 * m + ng).standard_normal((6, m, ng))
    a, b, xtw = c.dgdft_alb_lobpcg_gram(0, blk, has_p=True)
    c.close()
    s, hs = blk[:3].reshape(3 * m, ng), blk[3:].reshape(3 * m, ng)
    upper = np.kron(np.triu(np.ones((3, 3))), np.ones((m, m)))
    # sums of ng products, in any order: ng eps |row| |column|
    tol = ng * 2.3e-16
    for got, left in ((a, hs), (b, s)):
        bound = tol * np.linalg.norm(left, axis=1)[:, None] * np.linalg.norm(s, axis=1)[None, :]
        assert np.all(np.abs(got - (left @ s.T) * upper) <= bound)
    assert np.max(np.abs(xtw - blk[0] @ blk[1].T)) <= tol * ng * 2
