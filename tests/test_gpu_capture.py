"""Steps on a stream that the caller captures: refused on laminar handles (an Euler step swaps two
buffers on the host, which a replay would not), while an even number of steps of an SST handle
replays like as many plain steps, bit for bit."""
import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", [fvlbm.SCHEME_IMEX, fvlbm.SCHEME_EULER], ids=["imex", "euler"])
@pytest.mark.parametrize("prec", [fvlbm.FVLBM_FP64, fvlbm.FVLBM_FP32_DEV], ids=["fp64", "fp32"])
def test_laminar_steps_are_refused_under_capture(prec, scheme):
    import torch
    case = mg.cavity_delaunay(h_boundary=1 / 30, n_target=1500, re=200.0, cfl=0.1)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = fvlbm.Solver(case, precision=prec, device=0, stream=st.cuda_stream, scheme=scheme)
        ref = fvlbm.Solver(case, precision=prec, device=0, scheme=scheme)
        s.step(3)
        torch.cuda.synchronize()
        for n in (1, 2):
            with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=st):
                with pytest.raises(fvlbm.FvlbmError):
                    s.step(n)
        s.step(2)
        ref.step(5)
        np.testing.assert_array_equal(s.get_f(), ref.get_f())
        s.close()
        ref.close()


def test_an_even_number_of_sst_steps_replays():
    import torch
    case = mg.naca0012_cmesh(n_target=2000, alpha_deg=2.0)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = fvlbm.Solver(case, precision=fvlbm.FVLBM_FP32_DEV, device=0, stream=st.cuda_stream)
        ref = fvlbm.Solver(case, precision=fvlbm.FVLBM_FP32_DEV, device=0)
        s.step(2)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            s.step(2)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        ref.step(8)
        np.testing.assert_array_equal(s.get_f(), ref.get_f())
        s.close()
        ref.close()
