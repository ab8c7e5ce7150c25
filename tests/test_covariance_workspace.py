"""The size of the covariance's workspace (computed on the host): in proportion to the
matrix, or small, and none past the mocks that its 64-bit sums hold -- what the direct
path could multiply must not fail for a scratch of many times its size."""
import ctypes
import random

import pytest

from paper_1708_05303_gb300 import build, bsp


@pytest.fixture(scope="module")
def size():
    build.build()
    lib = bsp.load()

    def f(m, d):
        n = ctypes.c_size_t()
        assert lib.bsp_covariance_workspace_size(m, d, ctypes.byref(n)) == 0
        return n.value

    return f


def test_known_sizes(size):
    for m, d in [(10 ** 8, 1), (10 ** 6, 3), (2 ** 22 + 1, 64), (2 ** 31 - 1, 1), (3 * 10 ** 7, 32), (50, 50), (2, 1)]:
        assert size(m, d) == 0, (m, d)
    for m, d in [(512, 4962), (100, 1), (400_000, 3), (10 ** 5, 100), (2 ** 22, 32), (2, 4500)]:
        assert size(m, d) > 0, (m, d)


def test_in_proportion(size):
    rng = random.Random(1)
    for _ in range(2000):
        m, d = int(2 ** rng.uniform(1, 31)) - 1 or 2, int(2 ** rng.uniform(0, 17))
        n = size(max(m, 2), d)
        # 16 bytes a value of at most four times the columns, whole chunks of 32 mocks, an exponent and a bit a column
        assert n <= max(2 ** 30, 64 * (m + 32) * d + 5 * (d + 128) + 512), (m, d, n)
