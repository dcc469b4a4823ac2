"""The FP64 shifted-plane sweep forms its step weights in 64-bit integer
arithmetic for optical paths from 2^-700 to 2^700 and in FP64 beyond; the
series takes over from the closed form below 2^-10.  Formal solutions of boxes
whose opacity is scaled so that their optical paths fall on each side of those
lines, and across them, against the 64-bit torch reference of perf/cases.py.
(The CPU oracle takes 1 - (1 - e^-x)/x as it stands, which at x = 1e-3 leaves
2e-10 of w0 to rounding; the reference takes expm1 and a series below 0.05.)

Tolerance: with weights accurate to a few units in the last place on both sides
(the integer closed form is off by at most 2^-35 of w0 = x/2 at x = 2^-10, i.e.
2^-46 of the source term and step), 1e-12 allows for nine planes.
"""

import importlib.util
import os

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

pytestmark = pytest.mark.gpu


def reference(atm, atom, n):
    path = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "perf",
                        "cases.py")
    spec = importlib.util.spec_from_file_location("perf_cases", path)
    cases = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(cases)
    import torch
    weights = cases._weights

    def weights_u(x):   # u itself for thick steps, not 1 - w0
        ex, w0, wup, u = weights(x)
        return ex, w0, wup, torch.where(x < 0.05, u, -torch.expm1(-x) / x.clamp_min(0.05))

    cases._weights = weights_u
    p = cases._TwoLevel(atm, atom, 1)
    nd = torch.tensor(n, device="cuda").reshape(2, atm.nz, -1)
    return [a.cpu().numpy().reshape(atm.shape) for a in p.formal(p.grid[0], nd)]


@pytest.mark.parametrize("scale", [1e-240, 1e-205, 1e-30, 1e-6, 1e-3, 0.1, 1.0, 30.0, 1e4, 1e30,
                                   1e200, 1e230])
@pytest.mark.parametrize("nx,ny,shape", [(16, 16, None), (5, 7, (9, 2, 32, 0, 2)),
                                         (33, 3, (6, 1, 64, 0, 2)), (8, 8, (9, 1, 512, 0, 3))])
def test_optical_paths_of_every_size(scale, nx, ny, shape):
    atm, atom = synth.stratified_two_level(nx, ny, 9, eps=1e-3, sigma=0.3, seed=5,
                                           tau_top=1e-2, tau_bottom=1e2,
                                           atom=synth.TwoLevelAtom(n_freq=9))
    atom.kappa *= scale
    h = m.mg3d_create(atm, atom, n_grids=1)
    try:
        if shape is not None:
            m.mg3d_set_fs_config(h, 1, *shape)
        jeff, u = m.mg3d_formal_solve(h, 1)
        n = m.mg3d_get_populations(h, 1)
    finally:
        m.mg3d_destroy(h)
    jo, uo = reference(atm, atom, n)
    assert np.max(np.abs(jeff - jo) / np.abs(jo)) < 1e-12
    assert np.max(np.abs(u - uo) / np.abs(uo)) < 1e-12


@pytest.mark.parametrize("thick", [1e12, 1e18, 1e24, 1e200])
def test_thin_layers_above_a_thick_one(thick):
    """Steps of paths beyond 2^64, whose u is below a unit of the fractions,
    hand their source function (w0 = 1) to thin layers."""
    atm, atom = synth.stratified_two_level(8, 8, 9, eps=1e-3, sigma=0.3, seed=5,
                                           tau_top=1e-2, tau_bottom=1e2,
                                           atom=synth.TwoLevelAtom(n_freq=9))
    atm.n_tot[3:6] *= thick
    h = m.mg3d_create(atm, atom, n_grids=1)
    try:
        jeff, u = m.mg3d_formal_solve(h, 1)
        n = m.mg3d_get_populations(h, 1)
    finally:
        m.mg3d_destroy(h)
    jo, uo = reference(atm, atom, n)
    assert np.max(np.abs(jeff - jo) / np.abs(jo)) < 1e-12
    assert np.max(np.abs(u - uo) / np.abs(uo)) < 1e-12
