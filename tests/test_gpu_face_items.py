"""Face-value stages at the two item sizes and across state blobs.

The item size (64 or 256 cells) follows from the size of the handle.  A cell's arithmetic does
not depend on it: every face value is the same chain of fused multiply-adds whether its cell is
an item cell or on the ring, so one mesh steps bit for bit alike in a small and a large handle.
"""
import struct

import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu
FP64, FP32 = fvlbm.FVLBM_FP64, fvlbm.FVLBM_FP32_DEV


@pytest.mark.parametrize("prec", [FP64, FP32], ids=["fp64", "fp32"])
def test_item_sizes_agree_bit_for_bit(prec):
    """Meshes below the size that takes 64-cell items (quads, triangles, a hybrid SST mesh with
    walls, inlet and outlet, a periodic box) alone, and together with a large mesh in a batch that
    takes 256-cell items."""
    small = [mg.cavity_quad(33, re=400.0), mg.cavity_delaunay(h_boundary=1 / 40, n_target=3000, re=200.0, cfl=0.5),
             mg.bfs_hybrid(n_target=4000), mg.naca0012_cmesh(n_target=7000, alpha_deg=3.0)]
    m = mg.periodic_box(16, kind="tri", jitter=0.2, seed=9)
    rng = np.random.default_rng(3)
    small.append(mg.Case(m, nu=2e-3, cfl=0.5, rho=1.0 + 1e-3 * rng.uniform(-1, 1, m.n_cells),
                         u=0.05 * rng.uniform(-1, 1, m.n_cells)))
    b = fvlbm.Solver(small + [mg.cavity_quad(280, re=400.0)], precision=prec, device=0)
    b.step(19)
    items_b = fvlbm.fvlbm_fv_items(b.h)[0]
    n_small = 0
    for i, c in enumerate(small):
        s = fvlbm.Solver(c, precision=prec, device=0)
        s.step(19)
        np.testing.assert_array_equal(s.get_f(), b.get_f(i))
        for key in ("k", "omega", "nut"):
            np.testing.assert_array_equal(s.fields()[key], b.fields(i)[key])
        n_small += fvlbm.fvlbm_fv_items(s.h)[0]
        s.close()
    assert items_b < 80000 // 256 + n_small  # the batch ran larger items
    b.close()


def test_blob_with_relaxed_state_still_loads():
    """A version 1 blob holds one array more (the relaxed f^(1), 9 values per padded cell, after
    f^n); it is accepted and that array is passed over."""
    case = mg.cavity_quad(20, re=400.0)
    s = fvlbm.Solver(case, precision=FP64, device=0)
    s.step(5)
    f = s.get_f()
    blob = s.save_state()
    head = struct.Struct("<8siiiiiiqQQ")
    magic, version, prec, np_cells, ninst, turb, pad, steps, order, payload = head.unpack_from(blob)
    assert version == 2 and payload == len(blob) - head.size
    extra = 9 * np_cells * 8
    at = head.size + extra
    old = head.pack(magic, 1, prec, np_cells, ninst, turb, pad, steps, order, payload + extra)
    old += blob[head.size:at] + b"\xff" * extra + blob[at:]
    s.step(3)
    s.load_state(old)
    np.testing.assert_array_equal(s.get_f(), f)
    s.step(2)
    g = s.get_f()
    s.load_state(blob)
    s.step(2)
    np.testing.assert_array_equal(s.get_f(), g)
    with pytest.raises(fvlbm.FvlbmError):
        s.load_state(head.pack(magic, 1, prec, np_cells, ninst, turb, pad, steps, order, payload) + blob[head.size:])
    s.close()
