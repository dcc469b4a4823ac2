"""Default sweep of the two-level variants (moving atmospheres, partial
redistribution): the shifted-plane kernel against the band sweep that
mg3d_set_fs_config selects, over ragged grids, one
row or column, odd and even frequency counts, and optical paths beyond the range
of the integer weights.

Tolerance: FP64, both sides round each of at most 9 plane steps to a few units of
2^-52, and the band sweep's 1 - (1 - e^-x)/x leaves up to 2^-52/x to rounding
(x >= 1e-4 where it matters to the intensity): 1e-11.  FP32, nine steps of about
ten roundings of 2^-24 each on both sides: 2e-5.
"""

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

pytestmark = pytest.mark.gpu

VARIANTS = {"moving": dict(velocity=1.0), "prd": dict(velocity=0.0)}


def compare(variant, shape, nf, prec, scale=1.0):
    atom = synth.TwoLevelAtom(n_freq=nf, gamma_prd=0.5 if variant == "prd" else 0.0)
    atm, atom = synth.stratified_two_level(*shape, eps=1e-3, sigma=0.3, seed=3, atom=atom,
                                           **VARIANTS[variant])
    atom.kappa *= scale
    rows = -(-shape[1] // 8)
    out = []
    for band in (False, True):
        h = m.mg3d_create(atm, atom, n_grids=1, fs_prec=prec)
        try:
            if band:
                m.mg3d_set_fs_config(h, 1, min(nf, 3), -(-shape[1] // rows), 64, 0, 0)
            m.mg3d_formal_solve(h, 1)   # PRD: the second one sees the first one's field
            out.append(m.mg3d_formal_solve(h, 1))
        finally:
            m.mg3d_destroy(h)
    tol = 1e-11 if prec == m.MG3D_PREC_F64 else 2e-5
    for i, (a, b) in enumerate(zip(*out)):
        assert np.isfinite(a).all()
        size = np.abs(b)
        if i == 1 and variant == "prd":   # sum of w (1 - w0 rho): a difference of values of
            size = np.maximum(size, 1.0)  # order 1, whose relative error has no bound
        assert np.max(np.abs(a - b) / size) < tol


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("prec", [m.MG3D_PREC_F64, m.MG3D_PREC_F32])
@pytest.mark.parametrize("shape,nf", [((1, 1, 3), 3), ((2, 3, 5), 4), ((5, 7, 9), 9),
                                      ((33, 1, 9), 8), ((1, 33, 9), 5), ((3, 34, 9), 17),
                                      ((21, 19, 7), 18), ((130, 5, 5), 33), ((72, 70, 3), 7)])
def test_shapes(variant, prec, shape, nf):
    compare(variant, shape, nf, prec)


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("scale", [1e-230, 1e-40, 1e30, 1e230])
def test_optical_paths_out_of_range(variant, scale):
    compare(variant, (9, 10, 9), 9, m.MG3D_PREC_F64, scale)
