"""Per-frequency angle sums of mg3d_formal_solve_ml, added over the ray-group slots on the
device and copied in pieces of 2^20 values: the same, bit for bit, for one chunk of
several pieces and for chunks of one frequency (one ragged piece each), for every number
of slots, either output alone, and with partial redistribution, whose U takes a local
term by frequency and node.  Between numbers of slots the rays are added in another
order: 24 values of one sign, 48 roundings of 2^-53 (2^-24) on both sides.
"""

import ctypes

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

pytestmark = pytest.mark.gpu


def solve(h):
    m.mg3d_init_zero_radiation(h, 1)
    return m.mg3d_formal_solve_ml(h, 1)


@pytest.mark.parametrize("prec", [m.MG3D_PREC_F64, m.MG3D_PREC_F32])
@pytest.mark.parametrize("gamma_prd", [0.0, 0.5])
def test_pieces_chunks_and_slots(prec, gamma_prd):
    atom = synth.hydrogen_like_atom(line_freq=9, cont_freq=2, gamma_prd=gamma_prd)
    atm = synth.chromosphere(64, 60, 7, atom)
    h = m.mg3d_create_ml(atm, atom, n_grids=1, fs_prec=prec)
    try:
        nf = m.mg3d_n_levels(h)[1]
        assert nf * atm.n_tot.size > 1 << 20
        tol = 48 * (2.0 ** -53 if prec == m.MG3D_PREC_F64 else 2.0 ** -24)
        first = None
        for rays in (1, 4, 12):
            m.mg3d_set_ml_shape(h, 1, 8, rays, 128)
            m.mg3d_set_ml_chunk(h, 0)
            whole = solve(h)
            m.mg3d_set_ml_chunk(h, 1)
            parts = solve(h)
            assert all(np.array_equal(a, b) for a, b in zip(whole, parts))
            if gamma_prd == 0.0:
                first = first or whole
                for a, b in zip(whole, first):
                    assert np.max(np.abs(a - b) / np.abs(b)) < tol
        ux = np.empty((nf,) + atm.shape)
        m.mg3d_init_zero_radiation(h, 1)
        assert m.load().mg3d_formal_solve_ml(
            h, 1, None, ux.ctypes.data_as(ctypes.POINTER(ctypes.c_double))) == 0
        assert np.array_equal(ux, parts[1])
    finally:
        m.mg3d_destroy(h)
