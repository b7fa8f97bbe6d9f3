"""The gradient's fixed scratch: a call that reports an error which earlier work left in
the runtime waits for its kernels all the same, since its scratch goes to the next call.  The error
is a host-side one: a wait on a stream that is being captured, which the runtime refuses."""
import ctypes as C

import numpy as np
import pytest

import oracle
from paper_1309_1114_gb300 import scenes, scheduler
from paper_1309_1114_gb300 import splotch as S

pytestmark = pytest.mark.gpu


def runtime():
    for name in ("libcudart.so.13", "libcudart.so.12", "libcudart.so"):
        try:
            return C.CDLL(name)
        except OSError:
            pass
    pytest.skip("no shared CUDA runtime to begin a capture with")


def leave_an_error(torch, lib):
    """One refused call of the library on a capturing stream; its error is not taken."""
    rt, side = runtime(), torch.cuda.Stream()
    pal = np.ascontiguousarray(scenes.ramp_palette(), np.float32)
    h, graph, stream = C.c_void_p(), C.c_void_p(), C.c_void_p(side.cuda_stream)
    assert lib.spl_create(C.byref(h), 0, stream) == S.SPL_OK
    try:
        assert lib.spl_set_colormap(h, pal.ctypes.data, len(pal), 0.0, 1.0) == S.SPL_OK
        assert rt.cudaStreamBeginCapture(stream, 2) == 0            # relaxed
        rc = lib.spl_set_colormap(h, pal.ctypes.data, len(pal), 0.0, 1.0)
        rt.cudaStreamEndCapture(stream, C.byref(graph))
        if graph.value:
            rt.cudaGraphDestroy(graph)
        rt.cudaGetLastError()
        assert rc == S.SPL_ECUDA
    finally:
        assert lib.spl_destroy(h) == S.SPL_OK


def test_waits_when_an_earlier_error_is_reported():
    import torch
    lib = S.load_library()
    batch, rng = 500, np.random.default_rng(1)
    theta = scheduler.init_theta(3, bias=1.0)
    x = rng.uniform(0.0, 6.0, (batch, 32)).astype(np.float32)
    t = rng.uniform(8.0, 14.0, batch).astype(np.float32)
    th, xs, ts = (torch.from_numpy(a).cuda() for a in (theta, x, t))
    grad, loss = torch.zeros(S.SPL_MLP_NPARAM, device="cuda"), torch.zeros(1, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def call():
        with torch.cuda.stream(stream):
            torch.cuda._sleep(200_000_000)                          # about a tenth of a second
        rc = lib.spl_mlp_loss_grad(th.data_ptr(), xs.data_ptr(), ts.data_ptr(), batch, grad.data_ptr(),
                                   loss.data_ptr(), C.c_void_p(stream.cuda_stream))
        return rc, stream.query()

    l64, g64 = oracle.mlp_loss_grad(theta, x, t)
    # (a first call loads the kernels, which waits by itself)
    for error in (False, True, False):
        grad.zero_(), loss.zero_()
        torch.cuda.synchronize()
        if error:
            leave_an_error(torch, lib)
        assert call() == (S.SPL_ECUDA if error else S.SPL_OK, True)
        assert abs(float(loss) - l64) <= 1e-5 * abs(l64)
        assert np.max(np.abs(grad.cpu().numpy() - g64)) <= 1e-5 * np.max(np.abs(g64))
