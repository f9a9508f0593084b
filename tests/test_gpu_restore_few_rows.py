"""gbs_dequantize with inverse rotation around the numbers of rows at which a tile takes one token more: a row's result does not depend
on how many are restored with it, and nothing is written behind the last."""
import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,m,group", [(3584, 28, 128), (4096, 1, 0), (4096, 1, 32), (5120, 20, 128), (8192, 1, 0)])
@pytest.mark.parametrize("bits,dtype", [(3, torch.float32), (4, torch.bfloat16)])
def test_rows_do_not_depend_on_their_number(d, m, group, bits, dtype):
    gbs_build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    total = 5 * sms + 3
    gen = torch.Generator(device=DEV)
    gen.manual_seed(d)
    x = torch.randn((total, d), generator=gen, device=DEV).pow(3).to(torch.bfloat16)
    with Plan(d, d, m, bits, group, 0.9) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        want = plan.dequantize(codes, scales, inverse=True, dtype=dtype)
        for n in [1, 2, 3, 5] + [k * sms + e for k in (1, 2, 3, 4) for e in (-1, 0, 1)]:
            out = torch.full((n + 1, d), 7.0, dtype=dtype, device=DEV)
            plan.dequantize(codes[:n], scales[:n], inverse=True, out=out[:n])
            assert torch.equal(out[:n], want[:n]) and bool((out[n] == 7.0).all())
        assert plan.device_status() == 0
