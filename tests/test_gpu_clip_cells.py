"""gbs_clip_error by histogram for every width of its table's cells (512 to 4096, by how close two thresholds come), over more tiles than
blocks, so that a block's running totals are read more than once; against the oracle, within the tolerance the suite uses for these sums."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan, synth
from paper_2504_13989_b200 import build as gbs_build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = 1e-5


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("apart", [0.02, 0.006, 0.004, 0.002])          # lowest thresholds apart / (2 D): one case per width at 3 bits
@pytest.mark.parametrize("d,m,rows", [(1024, 1, 1300), (3584, 28, 607)])
def test_cells(d, m, rows, apart, bits):
    gbs_build.build()
    rng = np.random.Generator(np.random.PCG64(rows))
    x = 0.5 * rng.standard_t(3.0, size=(rows, d))
    x[5] = 0.0
    xt = torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)
    alphas = [float(np.float32(a)) for a in (0.6, 0.6 + apart, 0.85, 1.0)]
    ref = oracle.clip_error_rows(synth.to_oracle_array(xt), d, d, m, bits, 0, alphas)
    with Plan(d, d, m, bits, 0, 0.9) as plan:
        got = plan.clip_error(xt.to(DEV), alphas)
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        assert np.all(np.abs(got.cpu().numpy() - ref) <= TOL * ref)
