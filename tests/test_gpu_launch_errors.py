"""A launch that fails is reported by its own call and by no later one.  The failure is made on the host: the stream's capture has been
invalidated, so the launch is refused and nothing reaches the device."""
import contextlib
import ctypes

import pytest
import torch

from paper_2504_13989_b200 import Plan, binding
from paper_2504_13989_b200 import build as gbs_build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
RELAXED = 2                                          # CU_STREAM_CAPTURE_MODE_RELAXED


@contextlib.contextmanager
def invalidated_capture():
    """The handle of a stream whose capture a wait for it has invalidated."""
    cu = ctypes.CDLL("libcuda.so.1")
    stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuStreamCreate(ctypes.byref(stream), 1) == 0
    assert cu.cuStreamBeginCapture_v2(stream, RELAXED) == 0
    assert cu.cuStreamSynchronize(stream) != 0
    yield stream.value
    cu.cuStreamEndCapture(stream, ctypes.byref(graph))
    assert not graph.value and cu.cuStreamDestroy_v2(stream) == 0


@pytest.mark.parametrize("d,group,inverse", [(4096, 128, False), (128, 128, False), (128, 128, True), (4096, 128, True), (128, 32, True), (4096, 8, True)])
def test_a_refused_dequantize_leaves_no_error_behind(d, group, inverse):
    gbs_build.build()
    with Plan(d, d, 1, 4, group) as plan:
        codes, scales, _ = plan.rotate_quantize(torch.randn((3000, d), device=DEV).to(torch.bfloat16))
        out = torch.empty((3000, d), dtype=torch.float32, device=DEV)
        torch.cuda.synchronize()
        with invalidated_capture() as stream:
            rc = binding.lib().gbs_dequantize(plan.handle, codes.data_ptr(), scales.data_ptr(), 3000, out.data_ptr(), binding.GBS_DTYPE_F32,
                                              binding.GBS_INVERSE_ROTATE if inverse else 0, stream)
        assert rc == binding.GBS_ERR_CUDA
        assert binding.gbs_selftest_wait_expiry(100)[0] == 7         # its launch is checked by the thread's last error
