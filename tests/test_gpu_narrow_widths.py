"""Narrow widths without a Paley factor: on either side of the lines between the shared-memory kernel and the tensor-core kernels
(inverse rotation with group scales, fp32 rows), which kernel runs and that a row's result stays the same up to fp32 rounding."""
import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _x(n, d):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(d + n)
    return torch.randn((n, d), generator=gen, device=DEV).pow(3)


@pytest.mark.parametrize("d,group,dtype,per_sm", [
    (512, 128, torch.bfloat16, None), (512, 32, torch.float32, None), (1024, 128, torch.bfloat16, 6), (1024, 1024, torch.float32, 24),
    (2048, 32, torch.bfloat16, 2), (2048, 128, torch.float32, 5), (4096, 128, torch.float32, 0), (512, 0, torch.bfloat16, 0)])
def test_inverse(d, group, dtype, per_sm, tmp_path):
    gbs_build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with Plan(d, d, 1, 4, group, 0.9) as plan:
        n = (per_sm or 3) * sms + 1
        codes, scales, _ = plan.rotate_quantize(_x(n, d).to(torch.bfloat16))
        got = {}
        for rows in (n - 1, n):
            names = kernels_of(lambda: plan.dequantize(codes[:rows], scales[:rows], inverse=True, dtype=dtype), tmp_path / ("%d.dot" % rows))
            tensor = per_sm is not None and rows > per_sm * sms
            assert ("k_tc_uv_inv" in names) == tensor and ("k_dequantize_inverse" in names) == (not tensor)
            got[rows] = plan.dequantize(codes[:rows], scales[:rows], inverse=True, dtype=dtype)[:n - 1]
        # fp32: sums of d' terms in two orders, each rounding 2^-24 of partial sums at most sqrt(d') results in size
        diff = (got[n - 1].double() - got[n].double()).norm() / got[n].double().norm()
        assert float(diff) <= (1e-6 if dtype == torch.float32 else 4e-4)


@pytest.mark.parametrize("d,group,per_sm", [(512, 0, None), (512, 32, None), (1024, 0, 28), (1024, 128, 64), (2048, 0, 1.5), (2048, 128, 1.5),
                                            (4096, 0, 0)])
def test_fp32_rows(d, group, per_sm, tmp_path):
    gbs_build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with Plan(d, d, 1, 4, group, 0.9) as plan:
        n = int((per_sm or 3) * sms) + 1
        x = _x(n, d)
        got = {}
        for rows in (n - 1, n):
            names = kernels_of(lambda: plan.rotate_quantize(x[:rows]), tmp_path / ("%d.dot" % rows))
            tensor = per_sm is not None and rows > per_sm * sms
            assert ("k_tc_uvf" in names) == tensor and ("k_rotate_quantize" in names) == (not tensor)
            got[rows] = [t[:n - 1] for t in plan.rotate_quantize(x[:rows], want_y=True)]
        a, b = got[n - 1], got[n]
        assert float((a[2].double() - b[2].double()).norm() / b[2].double().norm()) <= 1e-6
        assert float(((a[1] - b[1]).abs() / b[1]).max()) <= 2e-6
        assert float((a[0] != b[0]).float().mean()) <= 1e-4
