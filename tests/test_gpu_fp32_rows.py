"""fp32 rows on the tensor cores (three bf16 planes per row): every width class, expansion, group sizes, ragged tiles, strided
rows, more rows than the grid's tiles, against the oracle; and an input of which every bit reaches the output.

The inputs are heavy-tailed rows.  A nearly constant row (1 + 1e-3 N(0, 1)) with group scales is no input for the fixed scale
tolerance of 1e-6: the contraction's partial sums reach U = 128, each of its 3 U / 16 = 24 fp32 accumulations may be off by
2^-23 of that, and a group's own values are only 0.06, so the bound there is 24 * 128 * 2^-23 / 0.06 = 6e-3 (3.5e-5 was seen)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build
from parity_util import compare_rotate_quantize

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,d_pad,m,bits,group,rows", [
    (4096, 4096, 1, 4, 0, 1), (4096, 4096, 1, 3, 128, 1203), (3584, 3584, 28, 3, 32, 5), (3968, 4096, 1, 4, 1024, 7),
    (1408, 1408, 44, 4, 0, 66), (512, 512, 1, 3, 64, 130), (352, 768, 12, 4, 32, 9),               # one warp per 32 rows
    (5120, 5120, 20, 4, 0, 3), (5056, 5120, 20, 3, 128, 303), (8192, 8192, 1, 3, 0, 301), (8192, 8192, 1, 4, 2048, 2),
    (8192, 8192, 1, 4, 64, 5), (4480, 4608, 72, 4, 0, 4),                                            # two warps share them
])
def test_fp32_rows_against_the_oracle(d, d_pad, m, bits, group, rows):
    gbs_build.build()
    rng = np.random.Generator(np.random.PCG64(d + rows))
    x = (0.5 * rng.standard_t(3.0, size=(rows, d))).astype(np.float32)
    x[:, rng.choice(d, 5, replace=False)] *= 50.0
    x[0] = 0.0
    x[0, d // 3] = 16777215.0                                                # 24 significant bits, alone in its row
    if rows > 2:
        x[2] = 0.0
    xt = torch.from_numpy(x)
    ref = oracle.rotate_quantize_rows(x, d, d_pad, m, bits, group, 0.9)
    with Plan(d, d_pad, m, bits, group, 0.9) as plan:
        wide = torch.full((rows, d + 8), float("nan"), device=DEV)
        wide[:, :d] = xt.to(DEV)
        for xd in (xt.to(DEV), wide[:, :d]):
            codes, scales, y = plan.rotate_quantize(xd, want_y=True)
            torch.cuda.synchronize()
            assert plan.device_status() == 0
            # every rotated value is +-x / sqrt(d'): one rounding, of the product with 1 / sqrt(d') (itself rounded)
            want = 16777215.0 / np.sqrt(d_pad)
            assert bool(((y[0].double().abs() - want).abs() <= 2.0 ** -22 * want).all())
            compare_rotate_quantize(xt, ref, codes, scales, y, bits, group, d_pad, 0.9)
        again, _, _ = plan.rotate_quantize(xd)
        assert torch.equal(again, codes)
