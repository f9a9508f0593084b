"""bf16 rows of 4096 < d' <= 8192 in one sweep: four lane quadrants and three (rows that move on from tile to tile), tiles of two
tokens with a last one of one, fewer tiles than blocks and many per block, expansion, strided rows, group sizes from two lanes
to a warp, against the oracle; the same bytes every time."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan, synth
from paper_2504_13989_b200 import build as gbs_build
from parity_util import compare_rotate_quantize

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,d_pad,m,bits,group,rows", [
    (8192, 8192, 1, 3, 0, 1), (8192, 8192, 1, 4, 0, 2403), (8128, 8192, 1, 3, 128, 297), (8192, 8192, 1, 4, 2048, 5), (8192, 8192, 1, 3, 512, 31),
    (5120, 5120, 20, 4, 0, 2), (5120, 5120, 20, 3, 0, 3007), (5056, 5120, 20, 4, 128, 1201), (5120, 5120, 20, 3, 256, 700),
    (4608, 4608, 72, 4, 0, 77), (6144, 6144, 12, 3, 512, 901), (7168, 7168, 28, 4, 256, 1500), (6912, 6912, 108, 3, 0, 9),
])
def test_rows_against_the_oracle(d, d_pad, m, bits, group, rows):
    gbs_build.build()
    rng = np.random.Generator(np.random.PCG64(d + rows))
    x = 0.5 * rng.standard_t(3.0, size=(rows, d))
    x[:, rng.choice(d, 5, replace=False)] *= 50.0
    if rows > 2:
        x[1] = 0.0
    xt = torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)
    at = np.unique(np.concatenate([np.arange(min(rows, 12)), np.arange(max(0, rows - 12), rows), rng.integers(0, rows, 40)]))
    ref = oracle.rotate_quantize_rows(synth.to_oracle_array(xt[at]), d, d_pad, m, bits, group, 0.9)
    with Plan(d, d_pad, m, bits, group, 0.9) as plan:
        wide = torch.full((rows, d + 64), float("nan"), dtype=torch.bfloat16, device=DEV)
        wide[:, :d] = xt.to(DEV)
        for xd in (xt.to(DEV), wide[:, :d]):
            codes, scales, y = plan.rotate_quantize(xd, want_y=True)
            torch.cuda.synchronize()
            assert plan.device_status() == 0
            compare_rotate_quantize(xt[at], ref, codes[at], scales[at], y[at], bits, group, d_pad, 0.9)
        for _ in range(3):
            again, s2, _ = plan.rotate_quantize(xd)
            assert torch.equal(again, codes) and torch.equal(s2, scales)
