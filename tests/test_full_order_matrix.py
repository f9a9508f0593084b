"""The matrices of Algorithm 2, written out from its definition, up to orders at which the oracle's own construction takes minutes."""
import numpy as np
import pytest

import oracle
from paper_2504_13989_b200 import binding, build as gbs_build


@pytest.mark.parametrize("m", [20, 128, 504, 1032, 2000, 2064, 3080, 4080])
def test_the_matrix_of_an_order_is_algorithm_2s(m):
    """H[0][0] = 1, the rest of row 0 and column 0 -1, H[i][j] = -chi(j - i) for i != j with the squares modulo m - 1, -1 on the diagonal."""
    gbs_build.build()
    p = m - 1
    chi = np.full(p, -1, dtype=np.int8)
    chi[np.arange(1, p, dtype=np.int64) ** 2 % p] = 1
    chi[0] = 1                                                        # the diagonal
    i = np.arange(p)
    want = np.full((m, m), -1, dtype=np.int8)
    want[0, 0] = 1
    want[1:, 1:] = -chi[(i[None, :] - i[:, None]) % p]
    assert np.array_equal(binding.gbs_hadamard_m(m).numpy(), want)
    if m <= 504:
        assert np.array_equal(oracle.hadamard_m(m), want)
