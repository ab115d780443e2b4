"""The FP64 SST kernels of the face-value path against the generic ones of the two-pass path.

Both evaluate the same equations in double, in other orders; a few steps from a rough turbulence
field agree to rounding (the stages between them, which also differ in order, included): k, omega
and nu_t to 1e-10 of their largest values, far below any dropped term or branch."""
import dataclasses

import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu


def _rough(case, seed, zero_k=False):
    """Fields that take every branch: increments inside and outside the limiter's bounds, blending
    functions from 0 to 1, cells without turbulence (k = nu_t = 0)."""
    rng = np.random.default_rng(seed)
    n = case.mesh.n_cells
    k = case.k * 10.0 ** rng.uniform(-3, 1, n)
    if zero_k:
        k[rng.random(n) < 0.3] = 0.0
    w = case.omega * 10.0 ** rng.uniform(-1, 2, n)
    u = case.uref * (1.0 + 0.1 * rng.uniform(-1, 1, n))
    return dataclasses.replace(case, k=k, omega=w, u=u, v=0.1 * case.uref * rng.uniform(-1, 1, n))


def _no_walls():
    m = mg.naca0012_cmesh(n_target=1500, alpha_deg=2.0)
    b = m.mesh
    bt = np.full_like(b.bedge_type, mg.BC_FARFIELD)
    bv = np.tile(b.bedge_val[b.bedge_type == mg.BC_FARFIELD][:1], (b.n_bedges, 1))
    return dataclasses.replace(m, mesh=dataclasses.replace(b, bedge_type=bt, bedge_val=bv))


@pytest.mark.parametrize("make", [
    lambda: _rough(mg.naca0012_cmesh(n_target=6000, alpha_deg=5.0), 1),
    lambda: _rough(mg.bfs_hybrid(n_target=5000), 2, zero_k=True),
    lambda: dataclasses.replace(_rough(mg.naca0012_cmesh(n_target=3000, alpha_deg=1.0), 3), local_dt=True, cfl=0.2),
    lambda: _rough(_no_walls(), 4),
    lambda: dataclasses.replace(_rough(mg.bfs_hybrid(n_target=2000), 5), variant=10),
], ids=["airfoil", "step-zero-k", "airfoil-local", "no-walls", "variants"])
def test_fp64_sst_paths_agree(make):
    case = make()
    a = fvlbm.Solver(case, precision=fvlbm.FVLBM_FP64, device=0)
    b = fvlbm.Solver(case, precision=fvlbm.FVLBM_FP64, device=0, kernel_path=1)
    assert fvlbm.fvlbm_fv_items(a.h)[0] > 0
    for n in (1, 2):
        a.step(n)
        b.step(n)
        fa, fb = a.fields(), b.fields()
        for key in ("k", "omega", "nut", "u"):
            assert np.isfinite(fb[key]).all()
            assert np.abs(fa[key] - fb[key]).max() <= 1e-10 * np.abs(fb[key]).max(), (key, n)
    a.close()
    b.close()
