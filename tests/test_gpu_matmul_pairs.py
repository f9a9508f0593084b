"""gbs_quantized_matmul on pairs of SMs: widths of its tiles from 64 to 256 tokens, ragged channels and tokens (an SM of a pair without rows among
them), several waves, odd numbers of 128-code steps, every pair of bit widths; against the float64 product of the unpacked codes (exact:
|sum| <= 49 d' < 2^53) times the two scales."""
import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build
from test_gpu_matmul_tiles import DEV, _codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n_tok,n_out", [
    (4096, 4096, 1000), (4096, 1000, 4100), (4096, 300, 14336), (4096, 129, 18944), (4096, 65, 18817), (3584, 257, 9473), (3584, 2100, 2049),
    (8192, 200, 5000), (1024, 5000, 5121), (5120, 700, 129)])
@pytest.mark.parametrize("bx,bw,dtype", [(4, 4, torch.bfloat16), (3, 3, torch.float32), (3, 4, torch.float32), (4, 3, torch.bfloat16)])
def test_against_the_exact_integer_product(d, n_tok, n_out, bx, bw, dtype):
    gbs_build.build()
    cx, qx = _codes(n_tok, d, bx, d + n_tok)
    cw, qw = _codes(n_out, d, bw, d + n_out + 1)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(3)
    sx = torch.rand((n_tok, 1), generator=gen, device=DEV) + 0.1
    sw = torch.rand((n_out, 1), generator=gen, device=DEV) + 0.1
    m = {3584: 28, 5120: 20}.get(d, 1)
    with Plan(d, d, m, bx) as px, Plan(d, d, m, bw) as pw:
        out = torch.full((n_tok + 1, n_out), float("nan"), dtype=dtype, device=DEV)
        px.quantized_matmul(cx, sx, pw, cw, sw, out=out[:n_tok])
        torch.cuda.synchronize()
        assert px.device_status() == 0 and bool(torch.isnan(out[n_tok]).all())
        want = (qx @ qw.T) * sx.double() * sw.double().T
        # fp32: two roundings of 2^-24 (the scales' product, its product with the exact sum); bf16: one more of 2^-9
        tol = 2.5e-7 if dtype == torch.float32 else 2.0 ** -8
        assert bool(((out[:n_tok].double() - want).abs() <= tol * want.abs()).all())
