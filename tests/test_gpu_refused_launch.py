"""A launch that the driver refuses is reported by the call that made it, and by no later one."""
import ctypes as C

import pytest

import hivis_inputs as hi
from tests.harness import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["prefill", "draft"])
@pytest.mark.parametrize("name", ["c1_tiny_f32_b1", "tiny_f32_b4_ragged", "mini_mha_b1"])
def test_calls_after_a_refused_one(name, what):
    """A stream whose capture was broken off takes no launches: nothing runs, and the calls that follow on a stream in order work."""
    import torch
    from paper_2509_23928_b200 import HivisError
    cuda = C.CDLL("libcuda.so.1")
    case = Case(hi.workload(name))
    try:
        dr = case.drafter
        case.gpu_prefill()
        want, _ = case.gpu_draft()
        case.gpu_restore()
        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        handle, graph = C.c_void_p(s.cuda_stream), C.c_void_p()
        out = torch.empty((case.wl.batch, case.wl.k), dtype=torch.int32, device="cuda")
        assert cuda.cuStreamBeginCapture_v2(handle, 2) == 0          # (relaxed: other streams go on as they were)
        assert cuda.cuStreamSynchronize(handle) != 0                 # not allowed in a capture, and breaks it off
        with torch.cuda.stream(s), pytest.raises(HivisError):
            if what == "prefill":
                dr.prefill(case.d_ids, case.d_hidden, [int(x) for x in case.cu], start_pos=[0] * case.wl.batch, resid0=case.d_resid[0])
            else:
                dr.draft(case.wl.batch, case.wl.k, case.d_resid, out_ids=out)
        assert cuda.cuStreamEndCapture(handle, C.byref(graph)) != 0 and not graph.value
        case.gpu_restore()
        got, _ = case.gpu_draft()
        assert (got == want).all()
        dr.status()
    finally:
        case.close()
