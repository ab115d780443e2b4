"""What a stream capture leaves behind: calls that are refused change nothing, a captured number of SST
steps replays in any number, and a captured exchange follows f^n between the two buffers of an
explicit Euler handle.  Every comparison is bit for bit with a handle that was never captured: a
replay launches the same kernels on the same values."""
import numpy as np
import pytest

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

pytestmark = pytest.mark.gpu
FP64, FP32, TAN = fvlbm.FVLBM_FP64, fvlbm.FVLBM_FP32_DEV, fvlbm.FVLBM_FP64_TANGENT
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


@pytest.mark.parametrize("n", [1, 2, 3])
@pytest.mark.parametrize("scheme,path", [(IMEX, 0), (IMEX, 1), (EULER, 0), (EULER, 1)],
                         ids=["imex", "imex-twopass", "euler", "euler-twopass"])
@pytest.mark.parametrize("prec", [FP64, FP32], ids=["fp64", "fp32"])
def test_captured_sst_steps_replay_in_any_number(prec, scheme, path, n):
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = fvlbm.Solver(_sst(), precision=prec, device=0, stream=st.cuda_stream, scheme=scheme, kernel_path=path)
        ref = fvlbm.Solver(_sst(), precision=prec, device=0, scheme=scheme, kernel_path=path)
        s.step(1)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            s.step(n)
        ref.step(1)
        _same(s, ref)           # capturing runs nothing
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        ref.step(3 * n)
        _same(s, ref)
        s.step(1)
        ref.step(1)
        _same(s, ref)
        s.close()
        ref.close()


def test_a_captured_step_and_exchange_of_an_sst_handle():
    """One capture of two rounds of a step and a pack: every call of it stands for itself."""
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = fvlbm.Solver(_sst(), precision=FP32, device=0, stream=st.cuda_stream)
        ref = fvlbm.Solver(_sst(), precision=FP32, device=0, stream=st.cuda_stream)
        n = s.cells[0]
        ls, lr = s.set_exchange_list(np.arange(n)), ref.set_exchange_list(np.arange(n))
        rows, want = (torch.zeros((2, n, 12), dtype=torch.float64, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            for q in range(2):
                s.step(1)
                s.pack_cells_dev(ls, rows[q].data_ptr())
        for _ in range(2):
            g.replay()
            for q in range(2):
                ref.step(1)
                ref.pack_cells_dev(lr, want[q].data_ptr())
            torch.cuda.synchronize()
            assert torch.equal(rows, want)
        s.close()
        ref.close()


@pytest.mark.parametrize("prec,path", [(FP64, 0), (FP32, 0), (FP32, 1), (TAN, 0)],
                         ids=["fp64", "fp32", "fp32-twopass", "tangent"])
def test_captured_exchange_follows_euler_steps(prec, path):
    """Pack and unpack captured once on a laminar Euler handle, replayed after odd and even numbers of
    steps, across a saved state and across a run from the 16-step graph."""
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s, ref = (fvlbm.Solver(_laminar(), precision=prec, device=0, stream=st.cuda_stream, scheme=EULER,
                               kernel_path=path) for _ in range(2))
        n = s.cells[0]
        some = np.arange(0, n, 3)
        pack, unpack = s.set_exchange_list(np.arange(n)), s.set_exchange_list(some)
        rpack, runpack = ref.set_exchange_list(np.arange(n)), ref.set_exchange_list(some)
        out, want = (torch.zeros((n, 12), dtype=torch.float64, device="cuda") for _ in range(2))
        back = torch.zeros((len(some), 12), dtype=torch.float64, device="cuda")
        idx = torch.as_tensor(some, device="cuda")
        torch.cuda.synchronize()
        gp, gu = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(gp, stream=st):
            s.pack_cells_dev(pack, out.data_ptr())
        with torch.cuda.graph(gu, stream=st):
            s.unpack_cells_dev(unpack, back.data_ptr())
        blob = None
        for steps in (1, 1, 2, 19, 1, 0, 3):
            s.step(steps)
            ref.step(steps)
            if steps == 0:      # a state saved from the other buffer
                s.load_state(blob)
                ref.load_state(blob)
            gp.replay()
            ref.pack_cells_dev(rpack, want.data_ptr())
            torch.cuda.synchronize()
            assert torch.equal(out, want), steps
            if blob is None:
                blob = s.save_state()
            back.copy_(1.001 * out[idx])
            gu.replay()
            ref.unpack_cells_dev(runpack, back.data_ptr())
            torch.cuda.synchronize()
            _same(s, ref)
        s.close()
        ref.close()
