"""KV rows restored (gbs_dequantize with inverse rotation, d' = 128): ragged last blocks and every output width, whose stores leave shared
memory in pieces of 128 bytes; against the float64 transform of the dequantized codes, and nothing written behind the last row."""
import numpy as np
import pytest
import scipy.linalg
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [32, 64, 96, 128])
@pytest.mark.parametrize("rows", [1, 31, 32, 33, 5000])
@pytest.mark.parametrize("bits,asym,dtype", [(4, True, torch.bfloat16), (3, False, torch.bfloat16), (3, True, torch.float32), (4, False, torch.float32)])
def test_rows_and_widths(d, rows, bits, asym, dtype):
    gbs_build.build()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(rows + d)
    x = torch.randn((rows, d), generator=gen, device=DEV).pow(3).to(torch.bfloat16)
    h = torch.from_numpy(scipy.linalg.hadamard(128).astype(np.float64)).to(DEV)
    with Plan(d, 128, 1, bits, 128, 1.0, asymmetric=asym) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        y = plan.dequantize(codes, scales, inverse=False, dtype=torch.float32).double()
        out = torch.full((rows + 1, d), 7.0, dtype=dtype, device=DEV)
        plan.dequantize(codes, scales, inverse=True, out=out[:rows])
        torch.cuda.synchronize()
        assert plan.device_status() == 0 and bool((out[rows] == 7.0).all())
    want = (y @ h / np.sqrt(128.0))[:, :d]
    # y = q Delta + lo comes with two roundings of numbers up to 2 max|y|, and 128 of them add up here; the kernel multiplies the exact sum
    # (up to 2 * 128 max|y| / Delta) by Delta / sqrt(128), three roundings, and adds 128 lo / sqrt(128), three more
    bound = 2.0 ** -24 * (2 * 2 + 6 * 2) * 128 / np.sqrt(128.0) * y.abs().amax(dim=1, keepdim=True)
    bound = bound + (2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -23) * want.abs()
    assert bool(((out[:rows].double() - want).abs() <= bound).all())
