"""Values at the ends of the number range through the kernels that replaced general ones: tiny rows and groups, scales near the
largest float, infinities.  Powers of two change no significand, so the results scale exactly; an infinity gives the scale and the
codes that the general kernel gives."""
import numpy as np
import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _rows(n, d, seed):
    x = 0.5 * np.random.Generator(np.random.PCG64(seed)).standard_t(3.0, size=(n, d))
    return torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16).to(DEV)


@pytest.mark.parametrize("d,m,group", [(8192, 1, 0), (8192, 1, 128), (5120, 20, 0), (5120, 20, 128)])
@pytest.mark.parametrize("bits", [3, 4])
def test_tiny_rows_and_groups_are_quantized_like_others(d, m, group, bits):
    gbs_build.build()
    x = _rows(9, d, d + bits)
    with Plan(d, d, m, bits, group, 0.9) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        small, s2, _ = plan.rotate_quantize((x.float() * 2.0 ** -110).to(torch.bfloat16))
        assert torch.equal(small, codes) and torch.equal(s2, scales * 2.0 ** -110)


@pytest.mark.parametrize("d,m,group,asym", [(4096, 1, 0, False), (3584, 28, 0, False), (8192, 1, 0, False), (4096, 1, 128, False),
                                            (128, 1, 0, False), (128, 1, 128, True)])
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_large_scales_are_restored(d, m, group, asym, bits, dtype):
    gbs_build.build()
    x = _rows(70, d, d + bits)
    with Plan(d, d, m, bits, group, 0.9, asymmetric=asym) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        up = 2.0 ** 112
        want = plan.dequantize(codes, scales, inverse=True, dtype=dtype)
        got = plan.dequantize(codes, scales * up, inverse=True, dtype=dtype)
        assert bool(torch.isfinite(got).all()) and torch.equal(got, want * up)


@pytest.mark.parametrize("d,m,group,at", [(4096, 1, 0, 0), (4096, 1, 128, 4095), (3584, 28, 0, 1000), (8192, 1, 0, 77), (5120, 20, 128, 5000)])
@pytest.mark.parametrize("value", [float("inf"), float("-inf")])
def test_an_infinity_in_an_fp32_row(d, m, group, at, value, monkeypatch):
    gbs_build.build()
    x = _rows(6, d, d).float() * 1.001
    want_rest = x.clone()
    x[3, at] = value
    with Plan(d, d, m, 4, group, 0.9) as plan:
        codes, scales, y = plan.rotate_quantize(x, want_y=True)
        rest = plan.rotate_quantize(want_rest)
    monkeypatch.setenv("GBS_FORCE_GENERIC", "1")
    with Plan(d, d, m, 4, group, 0.9) as plan:
        c2, s2, y2 = plan.rotate_quantize(x, want_y=True)
    assert bool(torch.isinf(scales[3]).all()) and torch.equal(scales[3], s2[3]) and torch.equal(codes[3], c2[3]) and torch.equal(y[3], y2[3])
    others = [0, 1, 2, 4, 5]
    assert torch.equal(codes[others], rest[0][others]) and torch.equal(scales[others], rest[1][others])


@pytest.mark.parametrize("d,m", [(1536, 1544), (480, 480), (8, 128)])
@pytest.mark.parametrize("at", [0, 1, 7, 15, 16, 300])
def test_an_infinity_in_a_row_of_a_full_order(d, m, at):
    gbs_build.build()
    x = _rows(133, d, d)
    with Plan(d, m, m, 4, 0, 0.9) as plan:
        want = plan.rotate_quantize(x)
        bad = x.clone()
        bad[130, at % d] = float("inf")
        codes, scales, _ = plan.rotate_quantize(bad)
    assert bool(torch.isinf(scales[130]).all())
    # every value times a factor of zero: NaN, which clips to the lowest code, -D
    assert bool((codes[130] == 0x99).all())
    others = [i for i in range(133) if i != 130]
    assert torch.equal(codes[others], want[0][others]) and torch.equal(scales[others], want[1][others])
