"""Launch shapes of the variants' shifted-plane sweep (lean 3, stage 0): what
mg3d_get_fs_config returns, set again, leaves the running kernel and the results
as they are, bit for bit; every shape of it gives the same results up to the order
of its sums; a program can leave it for the band sweep and come back.

Tolerance between shapes: sums of 9 frequencies and 24 rays of one sign in another
order (40 roundings of 2^-53, or 2^-24 in FP32), and eight steps of about ten
operations that another instance of the kernel may contract differently: 128.  PRD
sees the mean intensity of an earlier solution of the same shape through a
redistribution sum: three times that; its U is a difference of values of order 1 and
is compared on that scale.
"""

import numpy as np
import pytest

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [(v, p) for v in ("moving", "prd") for p in (m.MG3D_PREC_F64, m.MG3D_PREC_F32)]


def create(variant, prec, shape=(21, 19, 9), n_freq=9, **kw):
    atom = synth.TwoLevelAtom(n_freq=n_freq, x_max=5.0,
                              gamma_prd=0.5 if variant == "prd" else 0.0)
    atm, atom = synth.stratified_two_level(*shape, eps=1e-3, sigma=0.3, seed=3, atom=atom,
                                           velocity=1.0 if variant == "moving" else 0.0)
    return m.mg3d_create(atm, atom, n_grids=1, fs_prec=prec, **kw)


def solve(h):
    m.mg3d_init_zero_radiation(h, 1)
    return m.mg3d_formal_solve(h, 1)


@pytest.mark.parametrize("variant,prec", CASES)
@pytest.mark.parametrize("shape,n_freq", [((1, 1, 5), 3), ((21, 19, 9), 9), ((48, 48, 9), 17),
                                          ((64, 60, 5), 18)])
@pytest.mark.parametrize("tuned", [False, True])
def test_get_then_set_changes_nothing(variant, prec, shape, n_freq, tuned):
    h = create(variant, prec, shape, n_freq)
    try:
        if tuned:
            m.mg3d_autotune(h)
        cfg = m.mg3d_get_fs_config(h, 1)
        if not tuned:
            assert cfg[3:] == (3, 0)
        before = solve(h)
        info = m.mg3d_get_fs_occupancy(h, 1, *cfg)
        m.mg3d_set_fs_config(h, 1, *cfg)
        assert m.mg3d_get_fs_config(h, 1) == cfg
        after = solve(h)
    finally:
        m.mg3d_destroy(h)
    assert all(np.array_equal(a, b) for a, b in zip(before, after))
    assert info[0] >= 1


@pytest.mark.parametrize("variant,prec", CASES)
def test_every_shape_gives_the_same_results(variant, prec):
    h = create(variant, prec)
    try:
        first = m.mg3d_get_fs_config(h, 1)
        ref = solve(h)
        tol = 128 * (2.0 ** -53 if prec == m.MG3D_PREC_F64 else 2.0 ** -24)
        tol *= 3 if variant == "prd" else 1
        for freq in ([9, 4, 2, 100] if variant == "prd" else [9, 5, 3, 1, 100]):
            for bands, threads in ((1, 512), (2, 64), (5, 96), (10, 32), (16, 32)):
                if (bands - 1) * -(-19 // bands) >= 19:
                    with pytest.raises(m.MG3DError, match="empty band"):
                        m.mg3d_set_fs_config(h, 1, freq, bands, threads, 3, 0)
                    continue
                m.mg3d_set_fs_config(h, 1, freq, bands, threads, 3, 0)
                assert m.mg3d_get_fs_config(h, 1) == (min(freq, 9), bands, threads, 3, 0)
                for i, (a, b) in enumerate(zip(solve(h), ref)):
                    size = np.maximum(np.abs(b), 1.0 if i and variant == "prd" else 0.0)
                    assert np.max(np.abs(a - b) / size) < tol
        m.mg3d_set_fs_config(h, 1, 3, 2, 64, 0, 0)   # the band sweep
        assert m.mg3d_get_fs_config(h, 1) == (3, 2, 64, 0, 0)
        m.mg3d_set_fs_config(h, 1, *first)
        assert all(np.array_equal(a, b) for a, b in zip(solve(h), ref))
    finally:
        m.mg3d_destroy(h)


def test_refusals():
    for variant in ("moving", "prd"):
        h = create(variant, m.MG3D_PREC_F64)
        try:
            for bad in [(9, 2, 48, 3, 0), (9, 2, 1024, 3, 0), (9, 17, 64, 3, 0), (0, 2, 64, 3, 0),
                        (9, 2, 64, 3, 1), (9, 2, 64, 4, 0)] + ([(3, 2, 64, 3, 0)]
                                                               if variant == "prd" else []):
                with pytest.raises(m.MG3DError):
                    m.mg3d_set_fs_config(h, 1, *bad)
        finally:
            m.mg3d_destroy(h)
    atm, atom = synth.stratified_two_level(16, 16, 9, eps=1e-3, sigma=0.3, seed=2)
    for kw in ({}, dict(sc_interp=1)):
        h = m.mg3d_create(atm, atom, n_grids=1, **kw)
        try:
            with pytest.raises(m.MG3DError, match="lean must be"):
                m.mg3d_set_fs_config(h, 1, 9, 2, 64, 3, 0)
        finally:
            m.mg3d_destroy(h)
