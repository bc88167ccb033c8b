"""The density's dense eigensolver (csrc/eigh.cu) where its kernels change:
clusters of CTAs up to 608 columns, the whole GPU above, rows in shared memory
and (from about 1,900 columns) in global memory; one and two columns."""

import numpy as np
import pytest

from paper_1506_08147_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _weights(n, length):
    leg = np.polynomial.legendre
    c = np.zeros(n)
    c[-1] = 1.0
    r = np.sort(leg.legroots(leg.legder(c)).real)
    x = np.concatenate([[-1.0], r, [1.0]])
    return length / (n * (n - 1) * leg.legval(x, c) ** 2)


@pytest.mark.parametrize("ne,J", [((1, 1, 1), 1), ((1, 1, 1), 2), ((3, 3, 1), 7), ((3, 3, 3), 6), ((3, 3, 3), 22), ((3, 3, 3), 23),
                                  ((3, 3, 3), 71)])
def test_sizes(ne, J):
    gen = np.random.default_rng(J)
    span = tuple(3 if n > 1 else 1 for n in ne)
    nq = tuple(6 * s for s in span)
    cell = tuple(4.0 * n for n in ne)
    nl = (12, 12, 12)
    d = B.DG(ne, cell, span, nq, nl, J, 20.0, 1)
    n_elem = int(np.prod(ne))
    n = n_elem * J
    for k in range(n_elem):
        d.dgdft_dg_set_potential(k, gen.standard_normal(int(np.prod(nl))))
    cols = [gen.standard_normal((J, int(np.prod(nq)))) for _ in range(n_elem)]
    d.dgdft_dg_assemble(cols)
    H = np.zeros((n, n))
    for k in range(n_elem):
        for q, blk in d.dgdft_dg_get_row(k).items():
            H[k * J:(k + 1) * J, q * J:(q + 1) * J] = blk
    H = 0.5 * (H + H.T)
    n_occ = (n + 1) // 2
    eig, rho = d.dgdft_dg_density(cols, n_occ)
    d.close()
    ref = np.linalg.eigvalsh(H)
    # a backward stable reduction: a few n eps |H|
    assert np.max(np.abs(eig - ref[:n_occ])) <= 10 * max(n, 10) * 2.3e-16 * np.max(np.abs(ref))
    # rho integrates to the number of states: the eigenvectors are unit vectors
    # in an orthonormal basis (the mass matrices here have conditions below 1e4)
    w = [_weights(m, c / e) for m, c, e in zip(nl, cell, ne)]
    tot = np.einsum("kcba,c,b,a->", rho.reshape(n_elem, *nl[::-1]), w[2], w[1], w[0])
    assert abs(tot - n_occ) <= 1e-9 * n_occ
