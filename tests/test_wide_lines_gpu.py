"""FP64 formal solution of lines whose wings leave the range of the integer
weights: a Doppler profile falls below 2^-250 from 13.2 Doppler widths on, so the
outer slots of a group take the FP64 weights beside inner ones that take the
integer weights and share one exponent.  Against the 64-bit torch reference.

Tolerance: as for the integer weights' other tests (a few units in the last place
of each of nine steps on both sides).
"""

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth
from test_integer_weights_gpu import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x_max", [14.0, 20.0])
@pytest.mark.parametrize("n_freq", [8, 9, 10, 12, 16, 17, 18])
@pytest.mark.parametrize("scale", [1.0, 1e3])
def test_wings_beyond_the_integer_weights(x_max, n_freq, scale):
    atm, atom = synth.stratified_two_level(8, 8, 9, eps=1e-3, sigma=0.3, seed=5, tau_top=1e-2,
                                           tau_bottom=1e2,
                                           atom=synth.TwoLevelAtom(n_freq=n_freq, x_max=x_max))
    atom.kappa *= scale
    h = m.mg3d_create(atm, atom, n_grids=1)
    try:
        jeff, u = m.mg3d_formal_solve(h, 1)
        n = m.mg3d_get_populations(h, 1)
    finally:
        m.mg3d_destroy(h)
    jo, uo = reference(atm, atom, n)
    assert np.max(np.abs(jeff - jo) / np.abs(jo)) < 1e-12
    assert np.max(np.abs(u - uo) / np.abs(uo)) < 1e-12
