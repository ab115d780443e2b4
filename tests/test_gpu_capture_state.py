"""What a stream capture leaves behind: calls that are refused change nothing.  Every comparison is bit
for bit with a handle that was never captured."""
import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu
FP64, FP32 = fvlbm.FVLBM_FP64, fvlbm.FVLBM_FP32_DEV
IMEX, EULER = fvlbm.SCHEME_IMEX, fvlbm.SCHEME_EULER


def _laminar():
    return mg.cavity_delaunay(h_boundary=1 / 30, n_target=1500, re=200.0, cfl=0.1)


def _sst():
    return mg.naca0012_cmesh(n_target=2000, re_c=500.0, alpha_deg=3.0, cfl=0.05)


def _same(a, b):
    np.testing.assert_array_equal(a.get_f(), b.get_f())
    fa, fb = a.fields(), b.fields()
    for key in fa:
        np.testing.assert_array_equal(fa[key], fb[key])


@pytest.mark.parametrize("make", [_laminar, _sst], ids=["laminar", "sst"])
@pytest.mark.parametrize("scheme", [IMEX, EULER], ids=["imex", "euler"])
@pytest.mark.parametrize("prec", [FP64, FP32], ids=["fp64", "fp32"])
def test_refused_calls_leave_the_state(make, scheme, prec):
    """Statistics, runs of 16 steps (whether or not their graph exists), the profiler and the tuner are
    refused on a capturing stream, whose capture goes on; the next step starts from the state before it."""
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = fvlbm.Solver(make(), precision=prec, device=0, stream=st.cuda_stream, scheme=scheme)
        ref = fvlbm.Solver(make(), precision=prec, device=0, scheme=scheme)
        calls = [lambda: s.step(1, stats=True), lambda: s.step(2, stats=True), lambda: s.step(16),
                 lambda: s.profile_kernels(1)] + [lambda: s.autotune(1)] * (scheme == IMEX)
        done = 3
        s.step(3)
        for run in (0, 16):     # the second time the graph of 16 steps exists
            s.step(run)
            done += run
            torch.cuda.synchronize()
            for call in calls:
                with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=st):
                    with pytest.raises(fvlbm.FvlbmError) as e:
                        call()
                    assert e.value.code == fvlbm.FVLBM_ERR_CUDA
        a, b = s.step(2, stats=True), ref.step(done + 2, stats=True)
        assert a == b
        _same(s, ref)
        s.close()
        ref.close()
