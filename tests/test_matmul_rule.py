"""The rule by which gbs_quantized_matmul chooses its kernel (host arithmetic), for a whole B200 and for parts of one."""
import ctypes

import pytest

from paper_2504_13989_b200 import binding, build as gbs_build

FEW_TOKENS, TILES, PAIRS = 0, 1, 2


def rule(n_tok, n_out, d_pad, three=False, sms=148, pairs=None):
    """(kernel, tokens per tile)"""
    gbs_build.build()
    fn = binding.lib().gbs_matmul_rule
    fn.argtypes = [ctypes.c_int64, ctypes.c_int64] + [ctypes.c_int] * 4 + [ctypes.POINTER(ctypes.c_int)]
    tokens = ctypes.c_int(0)
    kernel = fn(n_tok, n_out, d_pad // 128, int(three), sms, sms // 2 if pairs is None else pairs, ctypes.byref(tokens))
    return kernel, tokens.value


@pytest.mark.parametrize("three", [False, True])
@pytest.mark.parametrize("sms,pairs", [(1, 0), (1, None), (2, 1), (17, None), (148, 0), (148, 60), (148, None)])
@pytest.mark.parametrize("n_tok,n_out,d_pad", [(1, 1, 128), (64, 4096, 4096), (300, 14336, 4096), (4096, 4096, 4096), (1, 2000000, 128)])
def test_a_part_of_the_chip_is_served(n_tok, n_out, d_pad, three, sms, pairs):
    """Without pairs the kernel on single SMs takes the call; widths are those that the kernels have."""
    kernel, tokens = rule(n_tok, n_out, d_pad, three, sms, pairs)
    if kernel == FEW_TOKENS:
        assert n_tok <= 64
    else:
        assert tokens % 32 == 0 and (64 if kernel == PAIRS else 32) <= tokens <= 256
    if (sms // 2 if pairs is None else pairs) == 0:
        assert kernel != PAIRS


def test_large_outputs_take_pairs():
    assert rule(4096, 4096, 4096) == (PAIRS, 256)
    assert rule(4096, 4096, 4096, pairs=0) == (TILES, 256)


@pytest.mark.parametrize("sms", [148, 100])
def test_few_tokens_beyond_sixteen_are_counted_in_waves_of_32_channels_per_sm(sms):
    wave = 32 * sms
    for n_tok, three, waves in ((17, False, 2), (32, False, 2), (33, False, 1), (64, False, 1), (33, True, 1), (64, True, 1)):
        assert rule(n_tok, waves * wave, 4096, three, sms)[0] == FEW_TOKENS
        assert rule(n_tok, waves * wave + 1, 4096, three, sms)[0] != FEW_TOKENS
        assert rule(n_tok, 128 * sms + 1, 4096, three, sms)[0] != FEW_TOKENS          # the tiles' second wave
    assert rule(65, 16, 4096, False, sms)[0] != FEW_TOKENS
