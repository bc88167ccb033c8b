"""The FP64 stage's Gram products and block updates (csrc/fp64_tensor.cu): widths
on both sides of the operand tiles (16, 32, 48, 64 columns), more than one tile,
grids whose rows do not fill a 128-row tile or a 64-row stage, inputs of very
different norms, one block on both sides of a product, without P; infinities."""

import numpy as np
import pytest

from paper_1506_08147_gb300 import binding as B

pytestmark = pytest.mark.gpu

EPS = 2.3e-16


def _context(n, m):
    c = B.Context([dict(n=n, L=(8.0, 8.0, 8.0), e_lo=(0, 0, 0), e_hi=n, m=m, J=m)], precision=B.DGDFT_PREC_FP64)
    c.dgdft_alb_set_potential(0, np.zeros(int(np.prod(n))))
    return c


@pytest.mark.parametrize("has_p", [True, False])
@pytest.mark.parametrize("n", [(12, 9, 5), (18, 20, 15)])
@pytest.mark.parametrize("m", [1, 15, 16, 17, 32, 33, 48, 49, 64, 65, 96, 97, 130])
def test_update(m, n, has_p):
    ng = int(np.prod(n))
    gen = np.random.default_rng(m)
    # columns of very different norms, the coefficients of the small ones large
    scale = 2.0 ** gen.integers(-60, 60, (3, m))
    blk = gen.standard_normal((6, m, ng)) * np.concatenate([scale, scale])[:, :, None]
    y = gen.standard_normal((3 * m, m)) / scale.reshape(-1)[:, None]
    c = _context(n, m)
    out = c.dgdft_alb_lobpcg_update(0, blk, y, has_p=has_p, stage=1)
    c.close()
    s, hs = blk[:3].reshape(3 * m, ng), blk[3:].reshape(3 * m, ng)
    k = (3 if has_p else 2) * m
    for got, left, lo in ((out[0], s, 0), (out[1], s, m), (out[2], hs, m)):
        ref = y[lo:k].T @ left[lo:k]
        # k terms, each to 2^-53 of the row's largest contribution (on either side)
        big = np.max(np.abs(left[lo:k]) * np.max(np.abs(y[lo:k]), axis=1)[:, None], axis=0)
        assert np.all(np.abs(got - ref) <= 4 * (k - lo) * EPS * big[None, :])


@pytest.mark.parametrize("m", [49, 64, 65, 130])
def test_wide_gram(m):
    n = (18, 20, 15)
    ng = int(np.prod(n))
    gen = np.random.default_rng(m)
    scale = 2.0 ** gen.integers(-200, 200, (6, m, 1))
    blk = gen.standard_normal((6, m, ng)) * scale
    c = _context(n, m)
    a, b, xtw = c.dgdft_alb_lobpcg_gram(0, blk, has_p=True, stage=1)
    c.close()
    s, hs = blk[:3].reshape(3 * m, ng), blk[3:].reshape(3 * m, ng)
    upper = np.kron(np.triu(np.ones((3, 3))), np.ones((m, m)))
    for got, left in ((a, hs), (b, s)):
        bound = ng * EPS * np.linalg.norm(left, axis=1)[:, None] * np.linalg.norm(s, axis=1)[None, :]
        assert np.all(np.abs(got - (left @ s.T) * upper) <= bound)
    assert np.all(np.abs(xtw - blk[0] @ blk[1].T) <=
                  ng * EPS * np.linalg.norm(blk[0], axis=1)[:, None] * np.linalg.norm(blk[1], axis=1)[None, :])


@pytest.mark.parametrize("p,q,ng", [(1, 1, 1), (3, 70, 63), (16, 16, 65), (64, 64, 4097), (130, 20, 1000)])
def test_gram_entry(p, q, ng):
    gen = np.random.default_rng(p)
    u, v = gen.standard_normal((p, ng)), gen.standard_normal((q, ng))
    v[0, 0] = np.inf
    c = _context((8, 8, 8), 4)
    got = np.asarray(c.dgdft_alb_gram(u, v))
    c.close()
    got = got if got.shape == (p, q) else got.T
    assert not np.any(np.isfinite(got[:, 0]))
    assert np.all(np.abs(got[:, 1:] - u @ v[1:].T) <=
                  ng * EPS * np.linalg.norm(u, axis=1)[:, None] * np.linalg.norm(v[1:], axis=1)[None, :] + 1e-300)
