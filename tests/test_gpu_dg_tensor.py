"""The tensor-core contractions of the DG assembly (csrc/dg_tensor.cu) where
their tiles change: 16 to 128 inputs and outputs of an axis pass on both sides
of the chunk sizes, more than 128 inputs, 1 to 128 columns on both sides of the
widths of the Gram products, point counts below and beside a stage of 64; columns
of very different magnitudes; infinities and NaN."""

from types import SimpleNamespace

import numpy as np
import pytest

from oracle import dg as odg
from paper_1506_08147_gb300 import binding as B

pytestmark = pytest.mark.gpu

CELL = (4.0, 5.0, 6.0)

SHAPES = [
    ((2, 3, 2), (2, 2, 2), 1),
    ((16, 17, 6), (16, 17, 8), 1),
    ((33, 12, 32), (32, 9, 33), 15),
    ((48, 6, 49), (49, 10, 48), 16),
    ((64, 65, 4), (65, 64, 6), 17),
    ((128, 4, 6), (128, 5, 97), 33),
    ((129, 6, 5), (16, 12, 11), 48),
    ((6, 130, 5), (7, 65, 80), 49),
    ((20, 20, 20), (14, 13, 15), 64),
    ((20, 20, 20), (14, 13, 15), 65),
    ((20, 18, 20), (22, 13, 15), 81),
    ((20, 18, 20), (22, 13, 15), 128),
]


def _domain(nq, nl, J):
    one = np.ones(3)
    return SimpleNamespace(n_elem=1, nl=nl, nq=nq, J=J, le=one * CELL, lq=one * CELL, e_off=0.0 * one,
                           corner=lambda k: 0.0 * one, coords=lambda k: (0, 0, 0), index=lambda *i: 0)


@pytest.mark.parametrize("dfloat", [False, True])
@pytest.mark.parametrize("nq,nl,J", SHAPES)
def test_shapes(nq, nl, J, dfloat):
    gen = np.random.default_rng(J)
    dom = _domain(nq, nl, J)
    z = gen.standard_normal((J, int(np.prod(nq)))) * 2.0 ** gen.integers(-120, 120, (J, 1))
    v = gen.standard_normal(int(np.prod(nl)))
    d = B.DG((1, 1, 1), CELL, (1, 1, 1), nq, nl, J, 20.0, 1, dfloat=dfloat)
    d.dgdft_dg_set_potential(0, v)
    phi = d.dgdft_dg_lgl_basis(0, z)
    d.dgdft_dg_assemble([z])
    row = d.dgdft_dg_get_row(0)
    d.close()
    exp = odg.alb_on_lgl(dom, 0, z)
    none = (np.zeros(0, np.int32), np.zeros(1, np.int64), np.zeros(0, np.int32), np.zeros(0))
    ora = odg.Assembly(dom, {0: exp}, {0: v}, {0: none}, np.zeros(1), 20.0).row(0)
    # random columns: mass matrices with conditions below 1e4 (of unit columns),
    # tables that agree to 1e-14, sums of up to 200 terms per axis
    assert np.max(np.abs(phi - exp)) <= 1e-10 * np.max(np.abs(exp))
    assert np.max(np.abs(row[0] - ora[0])) <= 1e-9 * np.max(np.abs(ora[0]))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite_is_reported(bad):
    z = np.random.default_rng(1).standard_normal((3, 512))
    z[1, 100] = bad
    d = B.DG((1, 1, 1), CELL, (1, 1, 1), (8, 8, 8), (8, 8, 8), 3, 20.0, 1)
    with pytest.raises(Exception, match="positive definite"):
        d.dgdft_dg_assemble([z])
    d.close()
