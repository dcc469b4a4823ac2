"""Multi-level rates with the FP32 formal solution over the whole range of rate
coefficients.  The populations depend on the ratios of the rates alone, so all of
them (Einstein and photoionisation coefficients, collisions) times one power of
two leave the populations as they are, also where a coefficient times an
exponential or a mean intensity leaves the range of single precision.

Tolerance: the rates differ by their rounding in FP64 or pairs of floats (2^-40
at most), which can flip roundings of 2^-24 in the FP32 opacities of the next
formal solution; 20 planes of a few such roundings each: 1e-5.
"""

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

pytestmark = pytest.mark.gpu

VARIANTS = {"static": {}, "damped": dict(a_damp=0.05), "prd": dict(gamma_prd=0.5),
            "scattering": dict(scattering=2.0), "moving": dict(velocity=1.0)}


def populations(scale, theta_ref, a_damp=0.0, gamma_prd=0.0, **kw):
    atom = synth.hydrogen_like_atom(line_freq=7, cont_freq=5, theta_ref=theta_ref,
                                    a_damp=a_damp, gamma_prd=gamma_prd)
    atm = synth.chromosphere(9, 8, 11, atom, t_min=8000.0, t_max=10000.0, sigma_t=0.05, **kw)
    atm.c *= scale
    for ln in atom.lines:
        ln.a_ul *= scale
    for cn in atom.continua:
        cn.beta *= scale
    h = m.mg3d_create_ml(atm, atom, n_grids=1, fs_prec=m.MG3D_PREC_F32)
    try:
        m.mg3d_init_zero_radiation(h, 1)
        m.mg3d_mali_sweep(h, 1, 2)
        return m.mg3d_get_populations(h, 1)
    finally:
        m.mg3d_destroy(h)


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("theta_ref", [40000.0, 250000.0])
def test_rates_scale_out(variant, theta_ref):
    one = populations(1.0, theta_ref, **VARIANTS[variant])
    assert np.isfinite(one).all()
    for e in (-140, -100, -70, 70, 100, 140):
        n = populations(2.0 ** e, theta_ref, **VARIANTS[variant])
        assert np.max(np.abs(n - one) / np.abs(one)) < 1e-5, e
