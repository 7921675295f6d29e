"""A launch that the runtime refuses is reported by the call that made it, and by no later one."""
import ctypes as C

import pytest
import torch

from tests import util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("refused", ["us_cast_fp8", "us_linear_fwd", "us_layer_norm_fwd"])
def test_an_error_of_one_launch_is_not_reported_by_the_next(refused):
    """A stream whose capture was invalidated (it was queried meanwhile) takes no launches; the next calls, on the default
    stream, read their status from the runtime's last error and must not find that refusal there."""
    from paper_2303_11257_b200 import lib as L
    x, q, y = U.empty(8, 64, "bf16"), U.empty(8, 64, "e4m3"), U.empty(8, 64, "bf16")
    w, ws, v = U.empty(64, 64, "e4m3"), L.new_workspace(), torch.ones(64, device="cuda")
    t, loss = torch.zeros(8, dtype=torch.int32, device="cuda"), torch.empty(8, device="cuda")
    calls = {"us_cast_fp8": lambda st=None: L.us_cast_fp8(x, 1.0, q, st), "us_linear_fwd": lambda st=None: L.us_linear_fwd(q, w, 1.0, y, ws, None, st),
             "us_layer_norm_fwd": lambda st=None: L.us_layer_norm_fwd(x, v, v, 1e-5, y, st)}
    later = [lambda: L.us_softmax_xent_fwd(x, t, loss), lambda: L.us_weighted_add([x, x], [0.5, 0.5], 1.0, y)]
    for fn in (*calls.values(), *later):                       # kernels loaded
        fn()
    torch.cuda.synchronize()
    rt, st, graph = C.CDLL("libcudart.so.12"), C.c_void_p(), C.c_void_p()
    assert rt.cudaStreamCreateWithFlags(C.byref(st), 1) == 0   # non-blocking
    try:
        assert rt.cudaStreamBeginCapture(st, 2) == 0           # relaxed: other streams go on as usual
        assert rt.cudaStreamQuery(st) != 0
        rt.cudaGetLastError()
        with pytest.raises(L.UnitScaleError) as e:
            calls[refused](st.value)
        assert e.value.status == L.US_ERR_CUDA
        for fn in later:
            fn()
    finally:
        rt.cudaStreamEndCapture(st, C.byref(graph))
        rt.cudaGetLastError()
        assert rt.cudaStreamDestroy(st) == 0
    torch.cuda.synchronize()
    assert L.us_workspace_status(ws) == 0
