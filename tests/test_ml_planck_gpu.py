"""Planck function of the bound-free continua, seen through the mean intensity of a background
so thick that J is the background's source function: FP64 and FP32 handles over exponents
x = h nu/(k T) from 6e-4 (hot) to 26 (cool), against expm1 in numpy.

Tolerance FP64: B to two units of 2^-53, its product with the opacity, the reciprocal and the
sums of 24 rays with four weights each, all of one sign: 40 units.  FP32: the operands and four
operations, rounded to 2^-24 each, and sums of 24 rays: 32 units.
"""

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [m.MG3D_PREC_F64, m.MG3D_PREC_F32])
@pytest.mark.parametrize("T", [3.5e6, 1e6, 1e5, 2e4, 5e3])
def test_thick_background_shows_the_planck_function(prec, T):
    atom = synth.hydrogen_like_atom(line_freq=3, cont_freq=9)
    atm = synth.chromosphere(6, 5, 7, atom, t_min=T, t_max=T, sigma_t=0.0, chi_c0=1e28)
    h = m.mg3d_create_ml(atm, atom, n_grids=1, fs_prec=prec)
    try:
        m.mg3d_init_zero_radiation(h, 1)
        jx, _ = m.mg3d_formal_solve_ml(h, 1)
    finally:
        m.mg3d_destroy(h)
    f = sum(ln.n_freq for ln in atom.lines)
    tol = 40 * 2.0 ** -53 if prec == m.MG3D_PREC_F64 else 32 * 2.0 ** -24
    for ct in atom.continua:
        for y in np.linspace(1.0, ct.y_max, ct.n_freq):
            B = (ct.rho * y) ** 3 / np.expm1(atom.theta_ref * ct.rho * y / T)
            inner = jx[f, 1:-1]   # the top plane's entering rays are dark
            assert np.max(np.abs(inner - B)) < tol * B, (ct.lower, y)
            f += 1
