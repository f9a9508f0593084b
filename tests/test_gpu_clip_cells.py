"""gbs_clip_error by histogram for every width of its table's cells, over more tiles than blocks, so that a block's running totals are read
more than once; against the oracle, within the tolerance the suite uses for these sums.  `cell_bits` repeats the host's search for the widest
cells (2^13 to 2^10 units of t: 512 to 4096 of them) that no two different thresholds share, so that a set of ratios shows which table it builds."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan, synth
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of

DEV = "cuda:0"
TOL = 1e-5
SCALE = 4194304.0 - 8.0                              # t = 1


def cell_bits(alphas, levels):
    thresholds = [math.ceil((j + 0.5) / levels * a * SCALE) for a in alphas for j in range(levels)]
    for bits in range(13, 9, -1):
        cells = {}
        for t in thresholds:
            cells.setdefault(t >> bits, []).append(t)
        if all(max(c) - min(c) <= 1 for c in cells.values()):
            return bits
    return 0                                         # served by the per-candidate kernel


def ratios(bits, levels):
    """Lowest thresholds 0.4 to 0.8 of a cell of 2^bits apart, on both sides of a border that wider cells do not have; bits = 0: in one cell
    of any width."""
    if bits == 0:
        return [float(np.float32(a)) for a in (0.6, 0.60001, 0.9)]
    for odd in range(1, 1 << (22 - bits), 2):
        for part in (0.2, 0.3, 0.4):
            alphas = [float(np.float32((odd + s * part) * 2.0 ** bits / SCALE * levels / 0.5)) for s in (-1, 1)] + [float(np.float32(0.9))]
            if 0.55 < alphas[0] and alphas[1] < 0.8 and cell_bits(alphas, levels) == bits:
                return alphas
    raise AssertionError("no such ratios")


WIDTHS = [13, 12, 11, 10, 0]


@pytest.mark.parametrize("levels", [3, 7])
@pytest.mark.parametrize("width", WIDTHS)
def test_every_width_of_cells_has_ratios(width, levels):
    assert cell_bits(ratios(width, levels), levels) == width


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("width", WIDTHS)
@pytest.mark.parametrize("d,m,rows", [(1024, 1, 1300), (3584, 28, 607)])
def test_cells(d, m, rows, width, bits, tmp_path):
    gbs_build.build()
    rng = np.random.Generator(np.random.PCG64(rows))
    x = 0.5 * rng.standard_t(3.0, size=(rows, d))
    x[5] = 0.0
    xt = torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)
    alphas = ratios(width, 2 ** (bits - 1) - 1)
    ref = oracle.clip_error_rows(synth.to_oracle_array(xt), d, d, m, bits, 0, alphas)
    with Plan(d, d, m, bits, 0, 0.9) as plan:
        xd = xt.to(DEV)
        names = kernels_of(lambda: plan.clip_error(xd, alphas), tmp_path / "clip.dot")
        assert ("k_tc_uv_clip" in names) == (width != 0) and ("k_tc_uv_rq" in names) == (width == 0)
        got = plan.clip_error(xd, alphas)
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        assert np.all(np.abs(got.cpu().numpy() - ref) <= TOL * ref)
