"""Rayleigh-Ritz spread over many SMs (csrc/rr_wide.cu): the sizes at which its
kernels change shape -- the smallest pencils, one warp against four for the
vectors (64), one CTA against a cluster (160), register counts of the column
kernels (64, 96, 160, 256, 352, 448), the largest a cluster holds (608) and
the first beyond it -- against LAPACK."""

import numpy as np
import pytest
import scipy.linalg as sla

from paper_1506_08147_gb300 import binding as B

pytestmark = pytest.mark.gpu

ARITH = {"fp64": (B.DGDFT_PREC_FP64, 1, 2.3e-16), "dfloat": (B.DGDFT_PREC_MIXED, 0, 1.5e-14)}


def _context(prec):
    e = dict(n=(8, 8, 8), L=(6.0, 6.0, 6.0), e_lo=(0, 0, 0), e_hi=(8, 8, 8), m=4, J=4)
    return B.Context([e], precision=prec)


@pytest.mark.parametrize("arith", sorted(ARITH))
@pytest.mark.parametrize("n,m", [(1, 1), (2, 1), (3, 3), (31, 8), (33, 33), (64, 21), (65, 22), (96, 32), (97, 9), (129, 43),
                                 (160, 64), (161, 53), (256, 85), (257, 3), (353, 117), (449, 149), (608, 40), (609, 17)])
def test_sizes(n, m, arith):
    prec, stage, eps = ARITH[arith]
    if arith == "dfloat" and (n > 160 or m > 64):
        eps = ARITH["fp64"][2]  # FP64 beyond the double-float kernel's sizes
    gen = np.random.default_rng(1000 * n + m)
    a = gen.standard_normal((n, n))
    a = a + a.T
    q = gen.standard_normal((n, n))
    b = q @ q.T / n + np.eye(n)  # condition <= ~5
    c = _context(prec)
    theta, y = c.dgdft_alb_rayleigh_ritz(a, b, m, stage=stage)
    c.close()
    ref = sla.eigh(a, b, eigvals_only=True)
    norm = np.max(np.abs(ref))
    # backward errors of Cholesky, the solves and the reflectors: a few n eps
    # |A| |B^-1| each; 50 covers their constants and cond(B)
    tol = 50 * max(n, 16) * eps
    assert np.max(np.abs(theta - ref[:m])) <= tol * norm
    assert np.max(np.abs(a @ y - b @ y * theta)) <= tol * np.max(np.abs(a)) * np.sqrt(n)
    # vectors found one by one: eps / (orthogonalisation window) on top
    window = 1e-5 if eps < 1e-15 else 3e-5
    assert np.max(np.abs(y.T @ b @ y - np.eye(m))) <= tol + 10 * eps / window


@pytest.mark.parametrize("arith", sorted(ARITH))
@pytest.mark.parametrize("gap", [0.0, 1e-9, 2e-7, 1e-6, 1e-5, 1e-4])
def test_pairs_at_every_gap(gap, arith):
    """Pairs of eigenvalues gap |A| apart: clusters, and both sides of the
    threshold (5e-7) and of the orthogonalisation windows."""
    prec, stage, eps = ARITH[arith]
    n, m = 120, 40
    gen = np.random.default_rng(int(gap * 1e12) % 1000 + 7)
    low = np.sort(gen.uniform(-1.0, 1.0, m // 2))
    low = np.linspace(-1.0, 1.0, m // 2) + 0.02 * low
    ev = np.sort(np.r_[low, low + gap * 10.0, gen.uniform(2.0, 10.0, n - m)])
    q, _ = np.linalg.qr(gen.standard_normal((n, n)))
    a = (q * ev) @ q.T
    a = 0.5 * (a + a.T)
    c = _context(prec)
    theta, y = c.dgdft_alb_rayleigh_ritz(a, np.eye(n), m, stage=stage)
    c.close()
    tol = 50 * n * eps
    assert np.max(np.abs(np.sort(theta) - ev[:m])) <= tol * 10.0
    assert np.max(np.abs(a @ y - y * theta)) <= 10.0 * max(tol, 1e-11)
    assert np.max(np.abs(y.T @ y - np.eye(m))) <= tol + 10 * eps / (1e-5 if eps < 1e-15 else 3e-5)
