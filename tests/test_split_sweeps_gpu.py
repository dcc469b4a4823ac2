"""MALI sweeps give the same populations, bit for bit, however they are split
over calls: within a call the rate kernel leaves the opacity and source function
of its new populations to the next formal solution, between calls the opacity
kernel forms them, and both have to round alike.
"""

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [m.MG3D_PREC_F64, m.MG3D_PREC_F32])
@pytest.mark.parametrize("variant", ["static", "moving", "prd"])
def test_sweeps_of_one_call_equal_single_calls(variant, prec):
    wide = variant != "static"
    atom = synth.TwoLevelAtom(n_freq=9, x_max=5.0 if wide else 3.0,
                              gamma_prd=0.5 if variant == "prd" else 0.0)
    atm, atom = synth.stratified_two_level(48, 48, 65, eps=1e-4, sigma=0.3, seed=4, atom=atom,
                                           velocity=1.0 if variant == "moving" else 0.0)
    out = []
    for calls in ([6], [1] * 6, [2, 4], [5, 1]):
        h = m.mg3d_create(atm, atom, n_grids=1, fs_prec=prec)
        try:
            m.mg3d_init_zero_radiation(h, 1)
            for c in calls:
                m.mg3d_mali_sweep(h, 1, c)
            out.append(m.mg3d_get_populations(h, 1))
        finally:
            m.mg3d_destroy(h)
    for n in out[1:]:
        assert np.array_equal(n, out[0])
