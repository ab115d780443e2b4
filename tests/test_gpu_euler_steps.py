"""Explicit Euler on the face-value kernel, which writes the other of two f buffers each step, against
the two-pass kernels: odd and even step counts, replayed and plain steps, statistics, a saved state
taken between buffers.  FP64 to 1e-12 of the largest f (rounding over 42 steps), FP32 to the bound
that the FP32 Euler parity test uses (1e-5)."""
import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(fvlbm.FVLBM_FP64, 1e-12), (fvlbm.FVLBM_FP32_DEV, 1e-5)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("make", [
    lambda: mg.cavity_delaunay(h_boundary=1 / 30, n_target=1500, re=200.0, cfl=0.1),
    lambda: mg.naca0012_cmesh(n_target=2000, re_c=500.0, alpha_deg=3.0, cfl=0.05),
], ids=["laminar", "sst"])
def test_euler_face_value_matches_twopass(make, prec, tol):
    case = make()
    a = fvlbm.Solver(case, precision=prec, device=0, scheme=fvlbm.SCHEME_EULER)
    b = fvlbm.Solver(case, precision=prec, device=0, scheme=fvlbm.SCHEME_EULER, kernel_path=1)
    assert a.footprint()[1] < b.footprint()[1]
    blob = None
    for n, stats in ((1, False), (17, False), (3, True), (16, False), (5, True)):
        sa, sb = a.step(n, stats=stats), b.step(n, stats=stats)
        if stats:
            assert abs(sa["mass"] - sb["mass"]) <= 10 * tol * sb["mass"]
        if blob is None:
            blob, ref = a.save_state(), a.get_f()
    fa, fb = a.get_f(), b.get_f()
    assert np.abs(fa - fb).max() <= tol * np.abs(fb).max()
    a.step(2)
    a.load_state(blob)
    np.testing.assert_array_equal(a.get_f(), ref)
    for n, stats in ((17, False), (3, True), (16, False), (5, True)):
        a.step(n, stats=stats)
    np.testing.assert_array_equal(a.get_f(), fa)
    a.close()
    b.close()
