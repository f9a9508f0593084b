"""gbs_quantized_matmul at the edges of its kernels: the few-token kernel and the tile kernel on either side of the rule between
them, narrow and wide tiles, ragged channels and tokens, every pair of bit widths.  Codes are drawn directly; the expected value is the
float64 product of the unpacked codes (exact: |sum| <= 49 d' < 2^53) times the two scales."""
import numpy as np
import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _codes(n, d, bits, seed):
    """Random codes in [-D, D], packed (little-endian bit stream), and the same as float64."""
    top = 2 ** (bits - 1) - 1
    q = np.random.default_rng(seed).integers(-top, top + 1, size=(n, d))
    u = (q & (2 ** bits - 1)).reshape(n, d // 8, 8).astype(np.int64)
    word = (u << (bits * np.arange(8))).sum(axis=2)
    packed = np.stack([(word >> (8 * i)) & 255 for i in range(bits)], axis=2).reshape(n, -1).astype(np.uint8)
    return torch.from_numpy(packed).to(DEV), torch.from_numpy(q.astype(np.float64)).to(DEV)


@pytest.mark.parametrize("d,n_tok,n_out", [
    (128, 1, 16), (128, 8, 17), (256, 9, 31), (1024, 17, 33), (1024, 33, 100), (1024, 64, 257),       # the few-token kernel
    (128, 1, 18000), (256, 16, 9001), (128, 16, 18300), (256, 17, 11003), (256, 33, 4400), (128, 64, 6001),   # few tokens, many channels
    (128, 65, 1), (384, 65, 127), (1024, 96, 128), (640, 129, 129), (1024, 191, 1000),                # tiles, few
    (512, 3000, 4090), (256, 4097, 5000), (128, 20000, 300), (384, 97, 40000),                        # several waves of tiles
])
@pytest.mark.parametrize("bx,bw,dtype", [(4, 4, torch.bfloat16), (3, 3, torch.float32), (3, 4, torch.float32), (4, 3, torch.bfloat16)])
def test_against_the_exact_integer_product(d, n_tok, n_out, bx, bw, dtype):
    gbs_build.build()
    cx, qx = _codes(n_tok, d, bx, d + n_tok)
    cw, qw = _codes(n_out, d, bw, d + n_out + 1)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(3)
    sx = torch.rand((n_tok, 1), generator=gen, device=DEV) + 0.1
    sw = torch.rand((n_out, 1), generator=gen, device=DEV) + 0.1
    m = {384: 12, 640: 20}.get(d, 1)                          # odd numbers of 128-code steps
    with Plan(d, d, m, bx) as px, Plan(d, d, m, bw) as pw:
        out = torch.full((n_tok + 1, n_out), float("nan"), dtype=dtype, device=DEV)
        px.quantized_matmul(cx, sx, pw, cw, sw, out=out[:n_tok])
        torch.cuda.synchronize()
        assert px.device_status() == 0 and bool(torch.isnan(out[n_tok]).all())
        want = (qx @ qw.T) * sx.double() * sw.double().T
        got = out[:n_tok].double()
        # fp32: two roundings of 2^-24 (the scales' product, its product with the exact sum); bf16: one more of 2^-9
        tol = 2.5e-7 if dtype == torch.float32 else 2.0 ** -8
        assert bool(((got - want).abs() <= tol * want.abs()).all())
