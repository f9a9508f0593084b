"""The full Paley orders at the edges of their split over a cluster: one CTA to eight, the order that fills eight, the largest
tables, the largest order, batches of one row to several tiles per cluster.  The rotation is the float64 product with the order's
matrix (which test_gpu_dense.py compares with the oracle's at 1544 and below); the oracle's own dense rotation takes minutes
at these sizes."""
import numpy as np
import pytest
import torch

from paper_2504_13989_b200 import Plan, binding
from paper_2504_13989_b200 import build as gbs_build
from parity_util import compare_rotate_quantize

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,m,bits,rows", [(128, 128, 3, 1), (480, 480, 4, 257), (504, 504, 3, 40), (1000, 1032, 4, 128), (1536, 1544, 3, 6000),
                                           (2000, 2000, 4, 129), (3000, 3080, 3, 5), (4080, 4080, 4, 9), (4064, 4080, 3, 130)])
def test_orders_against_the_dense_definition(d, m, bits, rows):
    gbs_build.build()
    rng = np.random.Generator(np.random.PCG64(d + m + rows))
    x = torch.from_numpy((0.5 * rng.standard_t(3.0, size=(rows, d))).astype(np.float32)).to(torch.bfloat16)
    H = binding.gbs_hadamard_m(m).numpy().astype(np.float64)
    top = 2 ** (bits - 1) - 1
    y_ref = x.double().numpy() @ H[:, :d].T / np.sqrt(m)
    delta = 0.9 * np.abs(y_ref).max(axis=1, keepdims=True) / top
    ref = {"y": y_ref, "delta": delta, "q": np.clip(np.rint(y_ref / delta), -top, top).astype(np.int64)}
    with Plan(d, m, m, bits, 0, 0.9) as plan:
        xd = x.to(DEV)
        codes, scales, y = plan.rotate_quantize(xd, want_y=True)
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        compare_rotate_quantize(x, ref, codes, scales, y, bits, 0, m, 0.9)
        # nothing beyond the last row's bytes: rows of m * bits / 8 bytes start at any byte
        flat = torch.full((codes.numel() + 64,), 0xA5, dtype=torch.uint8, device=DEV)
        again = flat[:codes.numel()].view(rows, -1)
        plan.rotate_quantize(xd, out=(again, scales, None))
        torch.cuda.synchronize()
        assert torch.equal(again, codes) and bool((flat[codes.numel():] == 0xA5).all())
