"""gbs_clip_error by histogram on batches whose errors differ by many orders of magnitude between candidates: rows of one channel
(every rotated value has the same magnitude: alpha = 1 fits exactly) with noise from none to a few per cent, candidates in
either order, and rows too small or not finite.

Tolerance: a value's t = |y| / M is rounded to 2^-22 M, so each residual is off by at most 2^-23 M and an error E over n values by
2^-22 M sqrt(n E) + n 2^-46 M^2; 1e-6 of E more for the fp32 rotation and M."""
import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan, synth
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(got, ref, x, d_pad):
    # per-token maxima |y| <= sum |x| / sqrt(d'), reached by the rows used here up to their noise
    m2 = float((np.abs(x).sum(axis=1) ** 2).max()) / d_pad
    n = x.shape[0] * d_pad
    bound = 1e-6 * ref + 2.0 ** -22 * np.sqrt(m2 * n * ref) + n * 2.0 ** -46 * m2
    assert np.all(got >= 0.0) and np.all(np.abs(got - ref) <= bound), (got, ref, bound)


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("rows", [1, 64])
@pytest.mark.parametrize("noise", [0.0, 1e-4, 1e-3, 1e-2])
def test_one_channel_rows(bits, rows, noise):
    gbs_build.build()
    d = 4096
    rng = np.random.Generator(np.random.PCG64(rows + bits))
    x = noise * rng.standard_normal((rows, d)) * 3.0 / 64
    x[np.arange(rows), rng.integers(0, d, rows)] = rng.uniform(3.0, 6.0, rows)
    xt = torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)
    alphas = [0.5, 0.5625, 0.625, 0.6875, 0.75, 0.8125, 0.875, 31.0 / 32, 1.0]      # nine: the histogram at any number of rows
    with Plan(d, d, 1, bits, 0, 0.9) as plan:
        for a in (alphas, alphas[::-1], [1.0] * 9, [1.0]):
            ref = oracle.clip_error_rows(synth.to_oracle_array(xt), d, d, 1, bits, 0, a)
            _check(plan.clip_error(xt.to(DEV), a).cpu().numpy(), ref, xt.double().numpy(), d)
        torch.cuda.synchronize()
        assert plan.device_status() == 0


def test_rows_of_tiny_values():
    gbs_build.build()
    d = 512
    x = np.random.Generator(np.random.PCG64(5)).standard_normal((9, d)).astype(np.float32)
    xt = torch.from_numpy(x).to(torch.bfloat16)
    with Plan(d, d, 1, 4, 0, 0.9) as plan:
        a = [0.5 + i / 16 for i in range(9)]
        want = plan.clip_error(xt.to(DEV), a).cpu().numpy()
        # a power of two leaves every code as it is: the sums change by its square, exactly
        small = plan.clip_error((xt.float() * 2.0 ** -110).to(torch.bfloat16).to(DEV), a).cpu().numpy()
        assert np.allclose(small * 2.0 ** 220, want, rtol=1e-12, atol=0.0)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_a_value_that_is_not_finite_shows_in_every_sum(bad):
    gbs_build.build()
    x = synth.make_host("llama4096", 9)
    x[4, 100] = bad
    with Plan(4096, 4096, 1, 4, 0, 0.9) as plan:
        for a in ([0.5, 0.75, 1.0], [0.5 + i / 16 for i in range(9)]):
            assert not bool(torch.isfinite(plan.clip_error(x.to(DEV), a)).any())


@pytest.mark.parametrize("bits,K", [(3, 5), (3, 10), (3, 20), (3, 31), (3, 50), (4, 9), (4, 18), (4, 27), (4, 32), (4, 64)])
def test_evenly_spaced_candidates_take_the_histogram(bits, K, tmp_path):
    """Many thresholds (j + 1/2) alpha_k / D coincide but for a rounding of alpha to float; the call must not fall back for it."""
    gbs_build.build()
    x = synth.make_host("llama4096", 640)
    alphas = [float(np.float32(0.5 + 0.5 * (i + 1) / K)) for i in range(K)]
    ref = oracle.clip_error_rows(synth.to_oracle_array(x), 4096, 4096, 1, bits, 0, alphas)
    with Plan(4096, 4096, 1, bits, 0, 0.9) as plan:
        xd = x.to(DEV)
        names = kernels_of(lambda: plan.clip_error(xd, alphas), tmp_path / "clip.dot")
        assert "k_tc_uv_clip" in names and "k_tc_uv_rq" not in names
        got = plan.clip_error(xd, alphas).cpu().numpy()
        assert np.all(np.abs(got - ref) <= 1e-5 * ref)
        # a tile per block and one pass of the per-candidate kernel: that one
        names = kernels_of(lambda: plan.clip_error(xd[:500], alphas[:8]), tmp_path / "few.dot")
        assert "k_tc_uv_rq" in names and "k_tc_uv_clip" not in names
        # thresholds that are close but not the same still go to the per-candidate kernel
        names = kernels_of(lambda: plan.clip_error(xd, [0.6, 0.60001]), tmp_path / "other.dot")
        assert "k_tc_uv_rq" in names and "k_tc_uv_clip" not in names
