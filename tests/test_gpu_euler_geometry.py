"""FP32 explicit Euler forms its geometry in FP64 in every kernel that runs it: on slim rotated cells,
where face normals and areas formed in float from the nodes cancel, the one-kernel step is as close to
FP64 as the two-pass kernels are.

Both read the same rounded offsets and normals and differ in the order of a few roundings, so their
errors are of one size: the root mean square over some 10,000 values may differ by half (formed in
float, it is two to five times the two-pass kernels')."""
import dataclasses

import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu
FP64, FP32 = fvlbm.FVLBM_FP64, fvlbm.FVLBM_FP32_DEV
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def _slim(tri, n=24, aspect=1000.0, angle=0.5):
    c = (mg.cavity_delaunay(h_boundary=1 / n, n_target=2 * n * n, re=400.0, cfl=0.5) if tri
         else mg.cavity_quad(n, re=400.0, jitter=0.2, seed=5))
    ca, sa = np.cos(angle), np.sin(angle)
    m = dataclasses.replace(c.mesh, xy=(c.mesh.xy * [1.0, 1.0 / aspect]) @ np.array([[ca, sa], [-sa, ca]]))
    rng = np.random.default_rng(7)
    rho, u, v = (a * rng.uniform(-1, 1, m.n_cells) for a in (1e-2, 0.1, 0.1))
    return dataclasses.replace(c, mesh=m, nu=1e-2, cfl=0.3, rho=1.0 + rho, u=u, v=v)


def _run(case, prec, path, steps, state):
    s = fvlbm.Solver(case, precision=prec, device=0, scheme=fvlbm.SCHEME_EULER, kernel_path=path)
    s.set_cells(np.arange(s.cells[0]), *state)
    launches = s.footprint()[1]
    s.step(steps)
    f, fields = s.get_f(), s.fields()
    s.close()
    return f, fields, launches


def _start(case, steps):
    """A state after some steps whose numbers are exact in both precisions."""
    s = fvlbm.Solver(case, precision=FP64, device=0, scheme=fvlbm.SCHEME_EULER, kernel_path=1)
    s.step(steps)
    f, k, omega, nut = s.get_cells(np.arange(s.cells[0]))
    s.close()
    short = [np.float64(np.float32(x)) for x in (f - W, k, omega, nut)]
    return [W + short[0]] + short[1:]


def _rms(f, ref):
    return np.sqrt(np.mean((f - ref) ** 2))


@pytest.mark.parametrize("steps", [1, 8])
@pytest.mark.parametrize("tri", [False, True], ids=["quads", "triangles"])
@pytest.mark.parametrize("n", [24, 170], ids=["small-items", "large-items"])
def test_slim_cells(tri, steps, n):
    case = _slim(tri, n)
    state = _start(case, 0)
    ref, _, _ = _run(case, FP64, 1, steps, state)
    two, _, l2 = _run(case, FP32, 1, steps, state)
    one, _, l1 = _run(case, FP32, 0, steps, state)
    assert l1 < l2
    assert _rms(one, ref) <= 1.5 * _rms(two, ref)


def test_sst_solve_and_far_field():
    """k, omega and nu_t of a step come from the same kernels on the same values, and f with the far
    field around it is as close."""
    case = mg.naca0012_cmesh(n_target=6000, re_c=2000.0, alpha_deg=3.0, cfl=0.05)
    state = _start(case, 10)
    ref, _, _ = _run(case, FP64, 1, 1, state)
    two, f2, l2 = _run(case, FP32, 1, 1, state)
    one, f1, l1 = _run(case, FP32, 0, 1, state)
    assert l1 < l2
    for key in ("k", "omega", "nut"):
        np.testing.assert_array_equal(f1[key], f2[key])
    assert _rms(one, ref) <= 1.5 * _rms(two, ref)
