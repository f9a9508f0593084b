"""KV rows restored (gbs_dequantize with inverse rotation, d' = 128): ragged last blocks and every output width, whose stores leave shared
memory in pieces of 128 bytes, both ways to ask for one scale per row, outputs on a 16-byte boundary, and the calls that the path leaves to
the general kernel; against the float64 transform of the dequantized codes, and nothing written behind the last row."""
import warnings

import numpy as np
import pytest
import scipy.linalg
import torch

from paper_2504_13989_b200 import Plan, binding
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def check(got, y, d, dtype):
    h = torch.from_numpy(scipy.linalg.hadamard(128).astype(np.float64)).to(DEV)
    want = (y @ h / np.sqrt(128.0))[:, :d]
    # y = q Delta + lo comes with two roundings of numbers up to 2 max|y|, and 128 of them add up here; the kernel multiplies the exact sum
    # (up to 2 * 128 max|y| / Delta) by Delta / sqrt(128), three roundings, and adds 128 lo / sqrt(128), three more
    bound = 2.0 ** -24 * (2 * 2 + 6 * 2) * 128 / np.sqrt(128.0) * y.abs().amax(dim=1, keepdim=True)
    bound = bound + (2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -23) * want.abs()
    assert bool(((got.double() - want).abs() <= bound).all())


@pytest.mark.parametrize("d", [32, 64, 96, 128])
@pytest.mark.parametrize("rows", [1, 31, 32, 33, 5000])
@pytest.mark.parametrize("bits,asym,dtype", [(4, True, torch.bfloat16), (3, False, torch.bfloat16), (3, True, torch.float32), (4, False, torch.float32)])
def test_rows_and_widths(d, rows, bits, asym, dtype):
    gbs_build.build()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(rows + d)
    x = torch.randn((rows, d), generator=gen, device=DEV).pow(3).to(torch.bfloat16)
    with Plan(d, 128, 1, bits, 128, 1.0, asymmetric=asym) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        y = plan.dequantize(codes, scales, inverse=False, dtype=torch.float32).double()
        out = torch.full((rows + 1, d), 7.0, dtype=dtype, device=DEV)
        plan.dequantize(codes, scales, inverse=True, out=out[:rows])
        torch.cuda.synchronize()
        assert plan.device_status() == 0 and bool((out[rows] == 7.0).all())
    check(out[:rows], y, d, dtype)


@pytest.mark.parametrize("group", [0, 128])
@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("scales_at", [0, 4, 8])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_alignment_of_output_and_scales(dtype, scales_at, asym, group, tmp_path):
    """Rows that start 16 bytes behind a 32-byte boundary; (Delta, lo) pairs that are not on 8 bytes take the general kernel."""
    gbs_build.build()
    rows, d = 1000, 128
    gen = torch.Generator(device=DEV)
    gen.manual_seed(scales_at)
    x = torch.randn((rows, d), generator=gen, device=DEV).to(torch.bfloat16)
    with Plan(d, 128, 1, 4, group, 1.0, asymmetric=asym) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        y = plan.dequantize(codes, scales, inverse=False, dtype=torch.float32).double()
        room = torch.zeros(scales.numel() + 2, device=DEV)
        moved = room[scales_at // 4:][:scales.numel()].view_as(scales).copy_(scales)
        size = torch.empty((), dtype=dtype).element_size()
        buf = torch.full((16 // size + rows * d + 64,), 7.0, dtype=dtype, device=DEV)
        out = buf[16 // size:][:rows * d].view(rows, d)
        assert out.data_ptr() % 32 == 16 and moved.data_ptr() % 16 == scales_at
        names = kernels_of(lambda: plan.dequantize(codes, moved, inverse=True, out=out), tmp_path / "kv.dot")
        assert ("k_row_inv" in names) == (not (asym and scales_at == 4))
        torch.cuda.synchronize()
        assert plan.device_status() == 0 and bool((buf[:16 // size] == 7.0).all()) and bool((buf[16 // size + rows * d:] == 7.0).all())
    check(out, y, d, dtype)


def test_more_rows_than_the_stores_count_take_the_general_kernel(tmp_path):
    """Captured and not run: no device holds these rows."""
    gbs_build.build()
    with Plan(128, 128, 1, 4, 128, 1.0, asymmetric=True) as plan:
        codes, scales, _ = plan.rotate_quantize(torch.randn((8, 128), device=DEV).to(torch.bfloat16))
        out = torch.empty((8, 128), dtype=torch.bfloat16, device=DEV)
        plan.dequantize(codes, scales, inverse=True, out=out)
        torch.cuda.synchronize()
        for rows, kernel in ((2 ** 31 - 1, "k_row_inv"), (2 ** 31, "k_dequantize_inverse")):
            graph = torch.cuda.CUDAGraph(keep_graph=True)
            with torch.cuda.graph(graph):
                rc = binding.lib().gbs_dequantize(plan.handle, codes.data_ptr(), scales.data_ptr(), rows, out.data_ptr(), binding.GBS_DTYPE_BF16,
                                                  binding.GBS_INVERSE_ROTATE, torch.cuda.current_stream().cuda_stream)
            assert rc == binding.GBS_OK
            graph.enable_debug_mode()
            with warnings.catch_warnings():
                warnings.simplefilter("ignore")
                graph.debug_dump(str(tmp_path / "rows.dot"))
            assert kernel in (tmp_path / "rows.dot").read_text()
