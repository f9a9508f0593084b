"""The split of a full Paley order's contraction (host arithmetic): which one each number of rows takes, and what becomes of a device that
cannot say how many clusters of a size run at once."""
import ctypes

import pytest

from paper_2504_13989_b200 import binding, build as gbs_build

MAX_CTAS = 16
SMEM = 232448
QUERY = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_int)


class Device:
    """Clusters of `ctas` that run at once, by the bits of the kernel; -1 in `fails`: the question cannot be answered."""

    def __init__(self, at_once=lambda bits, ctas: 140 // ctas):
        self.at_once, self.fails, self.asked = at_once, set(), []
        self.known = (ctypes.c_int * (2 * (MAX_CTAS + 1)))()

    def split(self, n_rows, m=1544, d=1536, bits=4):
        """(CTAs that share a token's coordinates, output blocks of each)"""
        gbs_build.build()
        fn = binding.lib().gbs_dense_rule
        fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, QUERY, ctypes.c_void_p,
                       ctypes.POINTER(ctypes.c_int)]

        def query(_, bits, ctas):
            self.asked.append((bits, ctas))
            return -1 if ctas in self.fails else self.at_once(bits, ctas)
        blocks = ctypes.c_int(0)
        ctas = fn(m, d, n_rows, bits, SMEM, ctypes.addressof(self.known), QUERY(query), None, ctypes.byref(blocks))
        return ctas, blocks.value


def test_a_question_that_failed_is_asked_again():
    want = Device().split(1)
    device = Device()
    device.fails = set(range(MAX_CTAS + 1))
    assert device.split(1)[0] == 0 and device.split(1)[0] == 0
    device.fails = set()
    assert device.split(1) == want


def test_a_size_that_failed_once_serves_the_next_call():
    want = Device().split(1)
    device = Device()
    device.fails = {want[0]}
    assert device.split(1)[0] not in (0, want[0])
    device.fails = set()
    assert device.split(1) == want


def test_answers_are_kept_also_that_none_fits():
    device = Device(lambda bits, ctas: 0 if ctas > 8 else 140 // ctas)
    assert 0 < device.split(1)[0] <= 8
    n = len(device.asked)
    assert len(set(device.asked)) == n
    device.split(1)
    device.split(4096)
    assert len(device.asked) == n


def test_each_kernel_has_its_own_answer():
    device = Device(lambda bits, ctas: 140 // ctas if bits == 4 else (1 if ctas == 4 else 0))
    four = device.split(1, bits=4)
    assert four[0] != 4 and device.split(1, bits=3)[0] == 4 and device.split(1, bits=4) == four


@pytest.mark.parametrize("m,d", [(128, 120), (264, 256), (1544, 1536), (4080, 4000)])
@pytest.mark.parametrize("n_rows", [1, 129, 2000, 100000, 2 ** 31 - 129])
def test_a_split_covers_the_order(m, d, n_rows):
    for sms in (148, 16, 15):
        ctas, blocks = Device(lambda bits, n: sms // n).split(n_rows, m, d)
        assert 1 <= ctas <= MAX_CTAS and blocks % 4 == 0 and blocks <= 64 and (ctas - 1) * blocks < m // 8 <= ctas * blocks
