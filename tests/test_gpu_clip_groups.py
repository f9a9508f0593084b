"""gbs_clip_error by histogram with group scales, at the edges of its dispatch: groups from one lane's 128 coordinates to eight lanes',
widths whose lanes are not all in use, thresholds for four tokens at a time, for two and too many; against the oracle.

Tolerances: the suite's; where one candidate nearly fits, a value's t = |y| / M is rounded to 2^-22 M with M <= the largest of all, so that
each residual is off by at most 2^-23 M and an error E over n values by 2^-22 M sqrt(n E) + n 2^-46 M^2; 1e-6 of E for the fp32 rotation."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan, synth
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = 1e-5


def _even(K):
    return [float(np.float32(0.5 + 0.5 * (i + 1) / K)) for i in range(K)]


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("K", [9, 32])                              # 4 bits, K = 32: two tokens at a time
@pytest.mark.parametrize("d,d_pad,m,group,rows", [
    (4096, 4096, 1, 128, 1), (4096, 4096, 1, 1024, 1203), (3584, 3584, 28, 128, 607), (512, 512, 1, 128, 5), (512, 512, 1, 512, 1200),
    (3968, 4096, 1, 256, 30), (1408, 1408, 44, 32, 9)])
def test_sums_against_the_oracle(d, d_pad, m, group, rows, K, bits, tmp_path):
    gbs_build.build()
    rng = np.random.Generator(np.random.PCG64(d + rows))
    x = 0.5 * rng.standard_t(3.0, size=(rows, d))
    x[:, rng.choice(d, 4, replace=False)] *= 50.0
    if rows > 2:
        x[1] = 0.0
        x[2] = 0.0
        x[2, 7] = 3.0
    xt = torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)
    alphas = _even(K)
    ref = oracle.clip_error_rows(synth.to_oracle_array(xt), d, d_pad, m, bits, group, alphas)
    with Plan(d, d_pad, m, bits, group, 0.9) as plan:
        xd = xt.to(DEV)
        names = kernels_of(lambda: plan.clip_error(xd, alphas), tmp_path / "clip.dot")
        assert ("k_tc_uv_clip" in names) == (group >= 128) and ("k_tc_uv_rq" in names) == (group < 128)
        got = plan.clip_error(xd, alphas).cpu().numpy()
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        assert np.all(np.abs(got - ref) <= TOL * ref)


@pytest.mark.parametrize("bits,K,rows,served", [(4, 64, 40, False), (3, 64, 40, True), (4, 8, 1776, False), (4, 8, 1780, True)])
def test_rule(bits, K, rows, served, tmp_path):
    gbs_build.build()
    x = synth.make_host("llama4096", 40).repeat(-(-rows // 40), 1)[:rows]
    alphas = _even(K)
    ref = oracle.clip_error_rows(synth.to_oracle_array(x[:40]), 4096, 4096, 1, bits, 128, alphas) if rows == 40 else None
    with Plan(4096, 4096, 1, bits, 128, 0.9) as plan:
        xd = x.to(DEV)
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        names = kernels_of(lambda: plan.clip_error(xd, alphas), tmp_path / "clip.dot")
        if K > 8 or sms == 148:
            assert ("k_tc_uv_clip" in names) == served and ("k_tc_uv_rq" in names) != served
        if ref is not None:
            assert np.all(np.abs(plan.clip_error(xd, alphas).cpu().numpy() - ref) <= TOL * ref)


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("noise", [0.0, 1e-3])
def test_groups_of_unlike_size(bits, noise):
    """|y| is one value per group but for what bf16 makes of the rows, and differs by orders of magnitude between groups."""
    gbs_build.build()
    d, group, rows = 4096, 128, 9
    rng = np.random.Generator(np.random.PCG64(bits))
    y = np.repeat(2.0 ** -rng.integers(0, 12, (rows, d // group)), group, axis=1)
    y *= np.where(rng.random((rows, d)) < 0.5, -1.0, 1.0)
    y += noise * y * rng.standard_normal((rows, d))
    H = oracle.hadamard_full(1, 12).astype(np.float64) / 64.0
    xt = torch.from_numpy((y @ H).astype(np.float32)).to(torch.bfloat16)
    alphas = [0.5, 0.5625, 0.625, 0.6875, 0.75, 0.8125, 0.875, 31.0 / 32, 1.0]
    ref = oracle.clip_error_rows(synth.to_oracle_array(xt), d, d, 1, bits, group, alphas)
    rot = np.abs(xt.double().numpy() @ H.T).reshape(rows, -1, group)
    m2 = float((rot.max(axis=2) ** 2).max())
    n = rows * d
    with Plan(d, d, 1, bits, group, 0.9) as plan:
        got = plan.clip_error(xt.to(DEV), alphas).cpu().numpy()
        bound = 1e-6 * ref + 2.0 ** -22 * np.sqrt(m2 * n * ref) + n * 2.0 ** -46 * m2
        assert np.all(got >= 0.0) and np.all(np.abs(got - ref) <= bound), (got, ref, bound)
        # a power of two leaves every code as it is, also where M is too small for its reciprocal
        small = plan.clip_error((xt.float() * 2.0 ** -105).to(torch.bfloat16).to(DEV), alphas).cpu().numpy()
        assert np.allclose(small * 2.0 ** 210, got, rtol=1e-9, atol=0.0)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_value_that_is_not_finite_shows_in_every_sum(bad):
    gbs_build.build()
    x = synth.make_host("llama4096", 9)
    x[4, 100] = bad
    for bits in (3, 4):
        with Plan(4096, 4096, 1, bits, 128, 0.9) as plan:
            assert not bool(torch.isfinite(plan.clip_error(x.to(DEV), _even(32))).any())
