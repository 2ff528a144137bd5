"""The tiles of the tensor-core path for more than 32 tokens, by host arithmetic alone: no GPU is needed."""
import random

import pytest

from paper_2410_21271_b200 import build as eora_build
from helpers import prefill_plan as plan


@pytest.fixture(scope="module", autouse=True)
def lib():
    eora_build.build()


@pytest.mark.parametrize("w,ab,K,N,r,M", [
    ("q4", "q8", 4096, 4096, 256, 500),     # 128 rows x 256 tokens, four stages, weights through shared memory, an odd number of units per CTA
    ("q3", "q4", 14336, 4096, 256, 490),
    ("q4", "q4", 4224, 11328, 256, 143),    # weights in tensor memory: three stages, the last row tile has one half
    ("q3", "f16", 8832, 10048, 128, 809),
])
def test_dequantising_warps_do_not_pass_over_a_whole_ring(w, ab, K, N, r, M):
    """A warp that waits for a ring's stage by parity has to have waited within the last `stages` k-blocks."""
    main, _ = plan(w, ab, K, N, r, M)
    assert main.stages <= 4
    assert main.longest_step <= main.stages


def test_no_shape_lets_a_warp_pass_over_a_whole_ring():
    rng = random.Random(1)
    short = 0
    for _ in range(4000):
        w, ab = rng.choice(["q4", "q3", "sp24", "sq4"]), rng.choice(["f16", "q4", "q3", "q8"])
        K, N, r = 128 * rng.randint(1, 112), 32 * rng.randint(1, 448), rng.choice([0, 64, 128, 256, 384, 512, 1024])
        M = rng.choice([rng.randint(33, 160), rng.randint(160, 1100), rng.randint(1100, 4096)])
        for t in plan(w, ab, K, N, r, M, rng.choice([64, 128])):
            assert t.longest_step <= 3 and t.longest_step <= max(t.stages, 1), (w, ab, K, N, r, M, t.rows, t.tokens, t.stages, t.longest_step)
            short += 0 < t.stages <= 4
    assert short > 200


def test_planning_takes_no_longer_with_many_tilings_to_choose_from():
    """A forward plans its tiles in every call.  200 tokens with adapters of rank 512 have the most tilings (hundreds of pairs of a main product's and
    one for t), 2048 tokens the fewest."""
    import time

    def best(*shape):
        times = []
        for _ in range(30):
            t = time.perf_counter()
            for _ in range(50):
                plan(*shape)
            times.append(time.perf_counter() - t)
        return min(times)

    few, many = best("q4", "f16", 4096, 1024, 128, 2048), best("q4", "f16", 4096, 1024, 512, 200)
    assert many < 1.5 * few
