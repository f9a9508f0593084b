"""gbs_clip_error by histogram (bf16 rows, one scale per token) at the edges of its dispatch: numbers of thresholds for each
copy count, thresholds that coincide, thresholds too close (the per-candidate kernel), ragged tiles and widths; against the
oracle, within the tolerance the suite uses for these sums."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan, synth
from paper_2504_13989_b200 import build as gbs_build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = 1e-5


@pytest.mark.parametrize("d,d_pad,m,bits,rows", [
    (4096, 4096, 1, 3, 1), (4096, 4096, 1, 4, 1203), (3584, 3584, 28, 3, 30), (3968, 4096, 1, 4, 3), (1408, 1408, 44, 3, 602), (512, 512, 1, 4, 5)])
@pytest.mark.parametrize("alphas", [
    [1.0], [0.7], list(np.linspace(0.5, 1.0, 8)), list((np.arange(32) + 33) / 64.0),       # 16/64-spaced ones share thresholds
    list((np.arange(63, -1, -1) + 1) / 64.0),                                              # all of them, descending
    [0.5, 0.5, 0.9], [0.6, 0.6 + 1e-5, 0.8],                                               # equal; too close for a cell
])
def test_sums_against_the_oracle(d, d_pad, m, bits, rows, alphas):
    gbs_build.build()
    rng = np.random.Generator(np.random.PCG64(d + rows))
    x = 0.5 * rng.standard_t(3.0, size=(rows, d))
    x[:, rng.choice(d, 4, replace=False)] *= 50.0
    if rows > 2:
        x[1] = 0.0
        x[2] = 0.0
        x[2, 7] = 3.0                                   # every |y| equal: at alpha = 1 this row adds no error at all
    xt = torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)
    a32 = [float(np.float32(a)) for a in alphas]
    ref = oracle.clip_error_rows(synth.to_oracle_array(xt), d, d_pad, m, bits, 0, a32)
    with Plan(d, d_pad, m, bits, 0, 0.9) as plan:
        got = plan.clip_error(xt.to(DEV), a32)
        err = torch.full((len(a32),), 2.0, dtype=torch.float64, device=DEV)
        plan.clip_error(xt.to(DEV), a32, err_sum=err)
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        assert np.all(np.abs(got.cpu().numpy() - ref) <= TOL * ref)
        assert np.all(np.abs(err.cpu().numpy() - 2.0 - ref) <= TOL * ref + 1e-15)
