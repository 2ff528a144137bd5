"""The workspace of the offline solve, by host arithmetic alone: no GPU is needed."""
import random

import pytest

import paper_2410_21271_b200 as eora
from paper_2410_21271_b200 import build as eora_build


@pytest.fixture(scope="module", autouse=True)
def lib():
    eora_build.build()


def width(cols):
    """The columns of an iterate in whole tiles of 64, 96, 128 or 160."""
    return min(-(-cols // w) * w for w in (64, 96, 128, 160))


def matrices(d, k, n, r, over=0):
    """Bytes of dW, X~ (where it is needed in whole tiles), P, the larger of C and dW - B'A, three iterates and the small problems."""
    a256, up = lambda v: -(-v // 256) * 256, lambda v: -(-v // 128) * 128
    m = min(r + (over or 32), d)
    dp, kp, np_ = up(d), up(k), up(n)
    side = np_ if m <= n < d else dp
    ldm, rows = width(m), max(dp, np_)
    return sum(map(a256, (4 * dp * kp, 4 * kp * np_ if k % 128 or n % 128 else 0, 4 * dp * np_, 4 * max(side * side, d * k), 4 * rows * ldm, 4 * rows * ldm,
                          4 * max(rows, kp) * ldm, 8 * m * m, 32 * 8 * m * m, (m + 15) // 16 * 2048, 8 * m * m, 8 * (2 * m + 128), 4 * ldm * ldm)))


def reported(d, k, n, r, over=0):
    return eora.eora_solve_workspace_bytes(eora.eora_solve_config(d, k, n, r, over, 0))


def most(d, k, n, r, over=0):
    """What may be reported: the matrices, and a quarter of that or 48 MB so that products go in few parts."""
    m = matrices(d, k, n, r, over)
    return m + max(m // 4 + 512, 48 << 20)


@pytest.mark.parametrize("d,k,n,r", [(4096, 4096, 2048, 128), (14336, 4096, 2048, 128), (128, 128, 100000, 32), (354, 24, 43, 7)])
def test_the_operands_of_the_tensor_cores_take_no_memory_of_their_own(d, k, n, r):
    assert 0 < reported(d, k, n, r) <= matrices(d, k, n, r)


@pytest.mark.parametrize("d,k,n,r", [(4096, 4096, 8192, 128), (4096, 4096, 16384, 128), (14336, 4096, 16384, 128), (1024, 4096, 2048, 128), (4096, 14336, 2048, 128)])
def test_nor_much_beyond_the_matrices_of_many_columns(d, k, n, r):
    assert 0 < reported(d, k, n, r) <= most(d, k, n, r)


def test_workspace_of_any_shape():
    """Beyond that only a layer with far fewer inputs than the smaller side has rows needs more than its matrices, for C's three parts."""
    rng = random.Random(3)
    log_int = lambda lo, hi: round(lo * (hi / lo) ** rng.random())
    seen = 0
    for _ in range(20000):
        d, k, n, r, over = log_int(1, 20000), log_int(1, 20000), log_int(1, 30000), log_int(1, 480), rng.choice([0, 0, 1, 20])
        m = min(r + (over or 32), d)
        got = reported(d, k, n, r, over)
        if r > m or m > 512:
            assert got == 0
            continue
        side = n if m <= n < d else d
        assert got > 0
        if 3 * width(m) <= side <= k:
            assert got <= most(d, k, n, r, over), (d, k, n, r, over)
            seen += 1
        assert got <= most(d, k, n, r, over) + matrices(d, k, n, r, over) // 2, (d, k, n, r, over)
    assert seen > 1000
