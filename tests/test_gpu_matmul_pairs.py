"""gbs_quantized_matmul on pairs of SMs: widths of its tiles from 64 to 256 tokens, ragged channels and tokens (an SM of a pair without rows among
them), several waves, odd numbers of 128-code steps, every pair of bit widths; against the float64 product of the unpacked codes (exact:
|sum| <= 49 d' < 2^53) times the two scales."""
import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of
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


@pytest.mark.parametrize("d,m,bits,shapes", [
    (128, 1, 3, [(15655, 2074), (1650, 19687)]), (384, 12, 3, [(486, 19635), (15343, 651)]), (896, 28, 4, [(808, 9614), (460, 14256)])])
def test_launches_in_a_row(d, m, bits, shapes, tmp_path):
    """Nothing between the launches, whose blocks follow one another on the SMs: what one of them still signals must not reach the next."""
    gbs_build.build()
    with Plan(d, d, m, bits) as px, Plan(d, d, m, bits) as pw:
        calls, wants = [], []
        for i, (n_tok, n_out) in enumerate(shapes):
            cx, qx = _codes(n_tok, d, bits, 10 + i)
            cw, qw = _codes(n_out, d, bits, 20 + i)
            sx, sw = torch.ones((n_tok, 1), device=DEV), torch.ones((n_out, 1), device=DEV)
            calls.append((cx, sx, pw, cw, sw))
            wants.append((qx @ qw.T).float())                  # whole numbers below 2^24
            names = kernels_of(lambda: px.quantized_matmul(*calls[i], dtype=torch.float32), tmp_path / ("%d.dot" % i))
            assert "k_tc_qgemm2" in names
        outs = [px.quantized_matmul(*calls[i % 2], dtype=torch.float32) for i in range(20)]
        torch.cuda.synchronize()
        assert px.device_status() == 0
        for i, out in enumerate(outs):
            assert torch.equal(out, wants[i % 2])
