"""The kernels that small and large handles take, each seen to run, on meshes with split items and items
that need the overflow table of halo ids.

In FP64 a cell's value is the same chain of operations with four threads per cell and in 64-cell items:
bit for bit.  The two-pass kernels order the operations differently: 1e-10 of the largest f after 19
steps, the bound of the oracle tests."""
import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu
FP64 = fvlbm.FVLBM_FP64


def _periodic():
    m = mg.periodic_box(16, kind="tri", jitter=0.2, seed=9)
    rng = np.random.default_rng(3)
    return mg.Case(m, nu=2e-3, cfl=0.5, rho=1.0 + 1e-3 * rng.uniform(-1, 1, m.n_cells),
                   u=0.05 * rng.uniform(-1, 1, m.n_cells))


SMALL = {"quads": lambda: mg.cavity_quad(33, re=400.0),
         "triangles": lambda: mg.cavity_delaunay(h_boundary=1 / 40, n_target=3000, re=200.0, cfl=0.5),
         "hybrid-sst": lambda: mg.bfs_hybrid(n_target=4000),
         "airfoil-sst": lambda: mg.naca0012_cmesh(n_target=10000, alpha_deg=3.0),
         "periodic": _periodic}


@pytest.mark.parametrize("name", SMALL)
def test_fp64_four_threads_per_cell_and_small_items(name):
    case = SMALL[name]()
    lanes, items = (fvlbm.Solver(case, precision=FP64, device=0) for _ in range(2))
    two = fvlbm.Solver(case, precision=FP64, device=0, kernel_path=1)
    fvlbm.fvlbm_set_wait_limit(items.h, 1 << 25)    # the fused kernels, which have the wait
    nitem, n_split, n_ovf = fvlbm.fvlbm_fv_items(items.h)
    assert nitem >= case.mesh.n_cells / 64
    if name == "airfoil-sst":
        assert n_split >= 1 and n_ovf >= 1
    for s in (lanes, items, two):
        s.step(17)
        s.step(2)
    fl, ref = lanes.get_f(), two.get_f()
    np.testing.assert_array_equal(fl, items.get_f())
    for key in ("k", "omega", "nut"):
        np.testing.assert_array_equal(lanes.fields()[key], items.fields()[key])
    assert np.abs(fl - ref).max() <= 1e-10 * np.abs(ref).max()
    assert {"lane_flux1", "lane_flux2", "lane_flux3"} <= set(lanes.profile_kernels(1))
    assert {"fused_stage1", "fused_stage2", "fused_stage3"} <= set(items.profile_kernels(1))
    for s in (lanes, items, two):
        s.close()


@pytest.mark.parametrize("re_c,overflow", [(1e4, 0), (6e6, 1)], ids=["split", "split-and-overflow"])
def test_fp64_large_items(re_c, overflow):
    """256-cell items, some split, on the finer wall cells one with an overflowing halo, against the
    two-pass kernels: 1e-10 of the largest f, the bound of the oracle test of split items (whose FP64
    half runs 64-cell items, its FP32 half these)."""
    case = mg.naca0012_cmesh(n_target=100000, re_c=re_c, alpha_deg=4.0)
    s, ref = (fvlbm.Solver(case, precision=FP64, device=0, kernel_path=path) for path in (0, 1))
    nitem, n_split, n_ovf = fvlbm.fvlbm_fv_items(s.h)
    assert nitem < case.mesh.n_cells / 128 and n_split >= 1 and n_ovf >= overflow, (nitem, n_split, n_ovf)
    s.step(3)
    ref.step(3)
    f = ref.get_f()
    assert np.abs(s.get_f() - f).max() <= 1e-10 * np.abs(f).max()
    assert "fused_stage1" in s.profile_kernels(1)
    s.close()
    ref.close()
