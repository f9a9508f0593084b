"""gbs_quantized_matmul of 33 to 64 tokens around the width at which its warps keep two steps of four-bit rows in flight: which form runs, and its
product against the exact one (tolerance: fp32, two roundings of 2^-24)."""
import re

import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of
from test_gpu_matmul_tiles import _codes

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n_tok", [33, 64])
@pytest.mark.parametrize("d,m,bits,steps", [(128, 1, 4, 1), (1024, 1, 4, 1), (2048, 1, 4, 1), (2560, 20, 4, 2), (3584, 28, 4, 2), (4096, 1, 4, 2),
                                            (4096, 1, 3, 1)])
def test_steps_in_flight(d, m, bits, steps, n_tok, tmp_path):
    gbs_build.build()
    n_out = 1061
    cx, qx = _codes(n_tok, d, bits, d + n_tok)
    cw, qw = _codes(n_out, d, bits, d + 1)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(4)
    sx = torch.rand((n_tok, 1), generator=gen, device=DEV) + 0.1
    sw = torch.rand((n_out, 1), generator=gen, device=DEV) + 0.1
    with Plan(d, d, m, bits) as plan:
        out = torch.full((n_tok + 1, n_out), float("nan"), dtype=torch.float32, device=DEV)
        graph = kernels_of(lambda: plan.quantized_matmul(cx, sx, plan, cw, sw, out=out[:n_tok]), tmp_path / "mm.dot")
        plan.quantized_matmul(cx, sx, plan, cw, sw, out=out[:n_tok])
        torch.cuda.synchronize()
        assert bool(torch.isnan(out[n_tok]).all())
        want = (qx @ qw.T) * sx.double() * sw.double().T
        assert bool(((out[:n_tok].double() - want).abs() <= 2.5e-7 * want.abs()).all())
    assert re.search(r"k_qgemvILi\dELi\dEfLi2ELi8ELi(\d)E", graph).group(1) == str(steps)
