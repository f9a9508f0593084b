"""gbs_quantized_matmul on pairs of SMs, for every width of its tiles: ragged channels and tokens, a last tile whose tokens all lie in the pair's
first SM, fewer tokens than half a tile, odd numbers of 128-code steps, several tiles per pair, every pair of bit widths; against the float64
product of the unpacked codes (exact: |sum| <= 49 d' < 2^53) times the two scales.  The rule that chooses the kernel says for each shape
which width it takes, and the captured call which kernel ran."""
import pytest
import torch

from paper_2504_13989_b200 import Plan
from paper_2504_13989_b200 import build as gbs_build
from parity_util import kernels_of
from test_matmul_rule import PAIRS, rule

DEV = "cuda:0"

# width of the tiles: (d', m, tokens, channels) with four bits on both sides, then with three bits on a side
SHAPES = {
    False: {64: [(4096, 1, 17, 41182), (3584, 28, 33, 40810)],
            96: [(20480, 20, 90, 19000)],
            128: [(3456, 108, 99, 21567), (3456, 108, 298, 10244), (3456, 108, 552, 6313)],
            160: [(1920, 60, 141, 19300), (4096, 1, 129, 10079), (1920, 60, 397, 9605)],
            192: [(1408, 44, 168, 20329), (896, 28, 808, 9614), (3584, 28, 845, 3121)],
            224: [(2176, 68, 193, 9680), (640, 20, 773, 15715), (3584, 28, 8075, 265)],
            256: [(640, 20, 233, 38016), (896, 28, 1121, 6783), (4096, 1, 4096, 1000), (1920, 60, 2084, 1829)]},
    True: {64: [(3456, 108, 1, 34318), (3456, 108, 33, 18973), (3456, 108, 32, 20225)],
           96: [(20480, 20, 90, 9500)],
           128: [(1920, 60, 97, 21375), (1920, 60, 300, 10264), (4096, 1, 2880, 529)],
           160: [(1408, 44, 138, 19749), (1408, 44, 387, 10846)],
           192: [(896, 28, 167, 20308), (896, 28, 3533, 1547), (256, 1, 565, 37812)],
           224: [(640, 20, 194, 19462), (384, 12, 1005, 9842), (256, 1, 1359, 12769)],
           256: [(384, 12, 237, 39040), (128, 1, 15655, 2074), (128, 1, 1650, 19687)]},
}
CASES = [(three, width) + shape for three in SHAPES for width in SHAPES[three] for shape in SHAPES[three][width]]
BITS = {False: [(4, 4, torch.bfloat16), (4, 4, torch.float32)], True: [(3, 3, torch.float32), (3, 4, torch.float32), (4, 3, torch.bfloat16)]}
# on either side of the rule
NEAR = [(4096, 1, 4096, 1000), (4096, 1, 1000, 4100), (4096, 1, 300, 14336), (4096, 1, 129, 18944), (4096, 1, 65, 18817), (3584, 28, 257, 9473),
        (3584, 28, 2100, 2049), (8192, 1, 200, 5000), (1024, 1, 5000, 5121), (5120, 20, 700, 129)]


@pytest.mark.parametrize("three,width,d,m,n_tok,n_out", CASES)
def test_shapes_reach_the_pairs_with_that_width(three, width, d, m, n_tok, n_out):
    assert rule(n_tok, n_out, d, three) == (PAIRS, width)


def test_shapes_cover_what_they_are_for():
    for three in SHAPES:
        assert sorted(SHAPES[three]) == list(range(64, 257, 32))
        shapes = [(width, d // 128, n_tok, n_out) for t, width, d, m, n_tok, n_out in CASES if t == three]
        assert any(n_tok < width // 2 for width, steps, n_tok, n_out in shapes)
        assert any(0 < n_tok % width <= width // 2 and n_tok > width for width, steps, n_tok, n_out in shapes)
        assert any(steps % 2 == 1 and -(-n_tok // width) * -(-n_out // 256) > 74 for width, steps, n_tok, n_out in shapes)
        assert any(0 < n_out % 256 <= 128 for width, steps, n_tok, n_out in shapes)


def _codes(n, d, bits, seed):
    """Random codes in [-D, D], packed (little-endian bit stream), and the same as float64."""
    top = 2 ** (bits - 1) - 1
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    q = torch.randint(-top, top + 1, (n, d), generator=gen, device=DEV, dtype=torch.int32)
    u = (q & (2 ** bits - 1)).view(n, d // 8, 8) << (bits * torch.arange(8, dtype=torch.int32, device=DEV))
    word = u.sum(dim=2, dtype=torch.int64)
    packed = torch.stack([((word >> (8 * i)) & 255).to(torch.uint8) for i in range(bits)], dim=2).reshape(n, -1)
    return packed, q.double()


def compare(d, m, n_tok, n_out, bx, bw, dtype, tmp_path):
    """Runs the product against its exact value; the kernels' names."""
    gbs_build.build()
    cx, qx = _codes(n_tok, d, bx, d + n_tok)
    cw, qw = _codes(n_out, d, bw, d + n_out + 1)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(3)
    sx = torch.rand((n_tok, 1), generator=gen, device=DEV) + 0.1
    sw = torch.rand((n_out, 1), generator=gen, device=DEV) + 0.1
    with Plan(d, d, m, bx) as px, Plan(d, d, m, bw) as pw:
        out = torch.full((n_tok + 1, n_out), float("nan"), dtype=dtype, device=DEV)
        names = kernels_of(lambda: px.quantized_matmul(cx, sx, pw, cw, sw, out=out[:n_tok]), tmp_path / "pairs.dot")
        torch.cuda.synchronize()
        assert px.device_status() == 0 and bool(torch.isnan(out[n_tok]).all())
        want = (qx @ qw.T) * sx.double() * sw.double().T
        # fp32: two roundings of 2^-24 (the scales' product, its product with the exact sum); bf16: one more of 2^-9
        tol = 2.5e-7 if dtype == torch.float32 else 2.0 ** -8
        assert bool(((out[:n_tok].double() - want).abs() <= tol * want.abs()).all())
    return names


@pytest.mark.gpu
@pytest.mark.parametrize("d,m,n_tok,n_out,bx,bw,dtype", [case[2:] + bits for case in CASES for bits in BITS[case[0]]])
def test_every_width_against_the_exact_integer_product(d, m, n_tok, n_out, bx, bw, dtype, tmp_path):
    assert "k_tc_qgemm2" in compare(d, m, n_tok, n_out, bx, bw, dtype, tmp_path)


@pytest.mark.gpu
@pytest.mark.parametrize("d,m,n_tok,n_out", NEAR)
@pytest.mark.parametrize("bx,bw,dtype", BITS[False] + BITS[True])
def test_against_the_exact_integer_product(d, m, n_tok, n_out, bx, bw, dtype, tmp_path):
    on_pairs = rule(n_tok, n_out, d, bx == 3 or bw == 3)[0] == PAIRS
    assert ("k_tc_qgemm2" in compare(d, m, n_tok, n_out, bx, bw, dtype, tmp_path)) == on_pairs


@pytest.mark.gpu
@pytest.mark.parametrize("d,m,bits,shapes", [
    (128, 1, 3, [(15655, 2074), (1650, 19687)]), (384, 12, 3, [(486, 19635), (15343, 651)]), (896, 28, 4, [(808, 9614), (460, 14256)])])
def test_launches_in_a_row(d, m, bits, shapes):
    """Nothing between the launches, whose blocks follow one another on the SMs: what one of them still signals must not reach the next."""
    gbs_build.build()
    with Plan(d, d, m, bits) as px, Plan(d, d, m, bits) as pw:
        calls, wants = [], []
        for i, (n_tok, n_out) in enumerate(shapes):
            assert rule(n_tok, n_out, d, bits == 3)[0] == PAIRS
            cx, qx = _codes(n_tok, d, bits, 10 + i)
            cw, qw = _codes(n_out, d, bits, 20 + i)
            sx, sw = torch.ones((n_tok, 1), device=DEV), torch.ones((n_out, 1), device=DEV)
            calls.append((cx, sx, pw, cw, sw))
            wants.append((qx @ qw.T).float())                  # whole numbers below 2^24
        outs = [px.quantized_matmul(*calls[i % 2], dtype=torch.float32) for i in range(20)]
        torch.cuda.synchronize()
        assert px.device_status() == 0
        for i, out in enumerate(outs):
            assert torch.equal(out, wants[i % 2])
