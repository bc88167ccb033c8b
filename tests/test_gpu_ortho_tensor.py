"""The orthonormalisation's products (csrc/fp64_tensor.cu): widths on both sides
of the operand tiles and of the 64-column tiles, row counts that fill no chunk
or stage, columns of very different norms."""

import numpy as np
import pytest

from paper_1506_08147_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lo,hi", [((12, 9, 8), (2, 1, 1), (11, 8, 8)), ((20, 18, 20), (0, 0, 0), (20, 18, 19))])
@pytest.mark.parametrize("J", [1, 2, 16, 17, 33, 48, 49, 64, 65, 129])
def test_orthonormalise(J, n, lo, hi):
    ng = int(np.prod(n))
    L = (6.0, 5.0, 4.0)
    gen = np.random.default_rng(J)
    x = gen.standard_normal((J, ng)) * 2.0 ** gen.integers(-6, 6, (J, 1))
    c = B.Context([dict(n=n, L=L, e_lo=lo, e_hi=hi, m=J, J=J)], precision=B.DGDFT_PREC_FP64)
    c.dgdft_alb_set_potential(0, np.zeros(ng))
    phi = np.asarray(c.dgdft_alb_restrict_orthonormalise(0, x, J))
    c.close()
    r = x.reshape(J, n[2], n[1], n[0])[:, lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]].reshape(J, -1)
    phi = phi.reshape(J, -1) * np.sqrt(np.prod(np.asarray(L) / np.asarray(n)))
    # orthonormal to a few J eps; the same span: the restricted columns lie in it
    # to the rounding of a basis of condition cond (below 1e4 here), squared in the Gram
    assert np.max(np.abs(phi @ phi.T - np.eye(J))) <= 20 * max(J, 10) * 2.3e-16
    out = r - (r @ phi.T) @ phi
    assert np.all(np.linalg.norm(out, axis=1) <= 1e-11 * np.linalg.norm(r, axis=1))
