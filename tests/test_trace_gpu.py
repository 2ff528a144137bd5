"""The time stamps behind eora_linear_set_trace stay inside a buffer of exactly the size the header asks for."""
import pytest

pytestmark = pytest.mark.gpu

import eora_inputs as gen
import paper_2410_21271_b200 as eora
from helpers import make_case, run_layer

GUARD = -0x5A5A5A5A5A5A5A5A


def traced(L, x, values):
    """Forward with a trace buffer of `values` values and guard words behind it: the buffer, after checking the guards."""
    import torch
    buf = torch.full((values + 4096,), GUARD, dtype=torch.int64, device="cuda:0")
    assert eora.eora_linear_set_trace(L.handle, buf) == eora.EORA_OK
    run_layer(L, x, "f16")
    assert eora.eora_linear_set_trace(L.handle, None) == eora.EORA_OK
    assert bool((buf[values:] == GUARD).all()), "written past the documented size"
    return buf[:values]


@pytest.mark.parametrize("K,N,r,M", [(512, 256, 0, 33), (1024, 4096, 128, 64), (4096, 544, 24, 100), (512, 4096, 512, 300), (1024, 2048, 136, 1100)])
def test_prefill_stamps_stay_inside_the_buffer(K, N, r, M):
    wf, af, bf = make_case(101, K, N, r)
    L = eora.Layer(wf, af, bf, max_m=M)
    buf = traced(L, gen.make_x(102, M, K), 4 * ((K + r) // 64 + 4))
    assert bool((buf[:4] != GUARD).all())                        # the first k-block's four stamps
    L.close()


@pytest.mark.parametrize("M", [1, 8])
def test_decode_stamps_stay_inside_the_buffer(M):
    K, N, r = 1024, 2048, 128
    wf, af, bf = make_case(103, K, N, r, w="q3")
    L = eora.Layer(wf, af, bf, max_m=M)
    buf = traced(L, gen.make_x(104, M, K), 64 * eora.eora_linear_decode_grid(L.handle, M))
    assert int((buf != GUARD).sum()) > 0
    L.close()


def test_nine_to_32_tokens_record_nothing():
    K, N, r, M = 512, 256, 64, 16
    wf, af, bf = make_case(105, K, N, r)
    L = eora.Layer(wf, af, bf, max_m=M)
    assert bool((traced(L, gen.make_x(106, M, K), 0) == GUARD).all())
    L.close()


def test_one_token_ctas_of_a_keep_their_place():
    """The CTAs that hold A are done long before the others and keep their places until a launch behind has entered or the others are about
    to store, so that a late launch finds one place per SM.  Alone on the chip: CTA 0 (which holds A) leaves after the last CTA's
    products with the backbone."""
    import torch
    K, N, r = 14336, 4096, 128
    wf, af, bf = make_case(107, K, N, r, w="q3")
    L = eora.Layer(wf, af, bf, max_m=1)
    x = gen.make_x(108, 1, K)
    grid = eora.eora_linear_decode_grid(L.handle, 1)
    for _ in range(3):
        t = traced(L, x, 64 * grid).view(grid, 16, 4)
        torch.cuda.synchronize()
        assert int(t[0, 0, 3]) >= int(t[grid - 1, 0, 2])
    L.close()
