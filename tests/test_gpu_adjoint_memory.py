"""Device memory of the shape gradient: beside what the gradient without it holds, the adjoints of the
geometry arrays (32 values per padded cell, three per boundary face) and nothing else."""
import threading

import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu


def _held(s, shape):
    """Bytes that the call holds on the device (its scratch is one allocation, held to its end)."""
    import torch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info(0)[0]
    low, stop = [before], threading.Event()

    def watch():
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info(0)[0])

    t = threading.Thread(target=watch)
    t.start()
    s.adjoint(60, 1.0, 0.5, shape=shape)
    stop.set()
    t.join()
    return before - low[0]


def test_shape_gradient_holds_its_adjoints_only():
    case = mg.cavity_quad(300, re=400.0)
    s = fvlbm.Solver(case, precision=fvlbm.FVLBM_FP64, device=0)
    s.step(2)
    s.set_adjoint_budget(1)             # one step's stage values at a time
    for shape in (False, True):         # the kernels are loaded
        s.adjoint(2, 1.0, 0.5, shape=shape)
    plain, shaped = _held(s, False), _held(s, True)
    np_cells = 90112                    # 90,000 cells, whole blocks of 256
    assert plain > 0
    # (allocations are multiples of 2 MiB)
    assert shaped - plain <= 32 * 8 * np_cells + 3 * 8 * 1200 + (4 << 20)
    s.close()
