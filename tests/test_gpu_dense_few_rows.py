"""The full Paley order at one row that is not zero, and at the numbers of rows that on 148 SMs take each width of a cluster: the CTAs
launched, and every row against the dense definition in float64."""
import re

import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build
from parity_util import compare_rotate_quantize, kernels_of
from test_gpu_dense_splits import _reference

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("d,m,rows,ctas", [(1536, 1544, 1, 13), (1536, 1544, 772, 13), (1536, 1544, 1400, 9), (1536, 1544, 2600, 6),
                                           (1536, 1544, 4096, 4), (120, 128, 1, None), (256, 264, 1, None), (4000, 4080, 1, None)])
def test_rows_and_ctas(d, m, rows, ctas, bits, tmp_path):
    gbs_build.build()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(100 * rows + bits)
    x = torch.randn((rows, d), generator=gen, device=DEV).to(torch.bfloat16)
    x[rows // 2, d // 3] = 30.0
    ref = _reference(x, m, bits, 0.9)
    assert (ref["delta"] > 0).all()
    with Plan(d, m, m, bits, 0, 0.9) as plan:
        codes, scales, y = plan.rotate_quantize(x, want_y=True)
        graph = kernels_of(lambda: plan.rotate_quantize(x, out=(codes, scales, None)), tmp_path / "rq.dot")
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        compare_rotate_quantize(x, ref, codes, scales, y, bits, 0, m, 0.9)
    grid = int(re.search(r"k_tc_dense_rq.*?<\\?<\\?<(\d+),", graph).group(1))
    if ctas is not None and torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert grid == ctas * -(-rows // 128)                        # one wave: a cluster per 128 rows
