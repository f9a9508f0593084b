"""The full Paley order over the numbers of rows at which its contraction is split among 13, 10, 6 and 4 CTAs (on 148 SMs), with one tile and
with two or three per cluster, ragged ends, and rows of codes that start at any byte: every row against the dense definition in float64."""
import functools

import numpy as np
import pytest
import torch

import oracle
from paper_2504_13989_b200 import Plan, binding
from paper_2504_13989_b200 import build as gbs_build
from parity_util import compare_rotate_quantize

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@functools.lru_cache(maxsize=None)
def _hadamard(m):
    # the oracle's construction takes minutes at the largest orders: there the library's, whose defining property is checked
    if m < 2000:
        return oracle.hadamard_m(m)
    h = binding.gbs_hadamard_m(m).numpy()
    assert np.array_equal(h.astype(np.float32) @ h.T.astype(np.float32), m * np.eye(m, dtype=np.float32))
    return h


def _reference(x, m, bits, alpha):
    h = torch.from_numpy(_hadamard(m)).to(DEV).double()
    y = (x.double() @ h[:, : x.shape[1]].T) / np.sqrt(m)
    top = 2 ** (bits - 1) - 1
    delta = alpha * y.abs().amax(dim=1, keepdim=True) / top
    q = torch.where(delta > 0, y / torch.where(delta > 0, delta, 1.0), 0.0).round().clamp(-top, top)      # half to even
    return {"y": y.cpu().numpy(), "delta": delta.cpu().numpy(), "q": q.to(torch.int32).cpu().numpy()}


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("d,m,rows", [
    (1536, 1544, 1), (1536, 1544, 129), (1536, 1544, 1090), (1536, 1544, 1900), (1536, 1544, 4000), (1536, 1544, 5531), (1536, 1544, 12301),
    (120, 128, 40), (256, 264, 1000), (4000, 4080, 300)])
def test_every_row(d, m, rows, bits):
    gbs_build.build()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(rows + bits)
    x = (torch.randn((rows, d), generator=gen, device=DEV) * (1.0 + 20.0 * (torch.rand((rows, 1), generator=gen, device=DEV) < 0.02))).to(torch.bfloat16)
    x[rows // 2] = 0.0
    ref = _reference(x, m, bits, 0.9)
    with Plan(d, m, m, bits, 0, 0.9) as plan:
        nb = m * bits // 8
        codes = torch.full((rows + 1, nb), 0xEE, dtype=torch.uint8, device=DEV)
        scales = torch.full((rows + 1, 1), -1.0, dtype=torch.float32, device=DEV)
        for y in (torch.empty((rows, m), dtype=torch.float32, device=DEV), None):
            binding.gbs_rotate_quantize(plan.handle, x, codes[:rows], scales[:rows], y)
            torch.cuda.synchronize()
            assert plan.device_status() == 0
            assert bool((codes[rows] == 0xEE).all()) and float(scales[rows, 0]) == -1.0, "wrote past the last row"
            compare_rotate_quantize(x, ref, codes[:rows], scales[:rows], y, bits, 0, m, 0.9)
            codes[:rows] = 0x55
