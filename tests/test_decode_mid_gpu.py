"""GPU parity of the kernel for nine to 32 tokens where its cuts can go wrong: the smallest and largest of each range of tokens,
one pair of reduction tiles (no cluster), unequal halves of the reduction axis, more units than a cluster takes (several waves),
more pairs of X than slots, t in several chunks, fused layers in one CTA.  Tolerance as for every forward (tests/helpers.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import eora_oracle as orc
import eora_inputs as gen
import paper_2410_21271_b200 as eora
from helpers import make_case, run_layer, check_parity, x_to_torch
from test_multi_adapter_gpu import adapters_for, reference


@pytest.mark.parametrize("w,ab,K,N,r,M,xd,group", [
    ("q4", "f16", 128, 32, 8, 9, "f16", 128),
    ("q3", "q8", 384, 96, 72, 16, "bf16", 64),
    ("sp24", "f16", 640, 160, 0, 17, "f16", 128),
    ("sq4", "q4", 1152, 64, 128, 32, "f16", 64),
    ("q4", "q3", 256, 42016, 64, 25, "f16", 128),       # 1313 pairs of row tiles: more than sixteen per cluster
    ("q3", "f16", 14336, 64, 64, 32, "f16", 128),       # 56 pairs per half
    ("q4", "f16", 512, 96, 4096, 24, "f16", 128),       # 32 pairs of t, 256 row tiles of A
])
def test_mid_cuts(w, ab, K, N, r, M, xd, group):
    wf, af, bf = make_case(61, K, N, r, w=w, ab=ab, group=group)
    x = gen.make_x(62, M, K, xd)
    L = eora.Layer(wf, af, bf, max_m=M, x_dtype=xd)
    assert L.launches(M) == (2 if xd == "bf16" else 1)
    y_ref = orc.forward(x, xd, wf, af, bf)
    for rep in range(2):
        check_parity(run_layer(L, x, xd), y_ref, f"{w}/{ab} K{K} N{N} r{r} M{M} call {rep}")
    L.close()


def test_mid_fused_layers_share_a_cta():
    import torch
    K, r, M = 512, 128, 21
    layers = [make_case(65 + i, K, N, r, w="q4") for i, N in enumerate((128, 4096, 256, 4224))]
    x = gen.make_x(66, M, K)
    F = eora.FusedLayers(layers, max_m=M)
    ys = F.forward(x_to_torch(x, "f16"))
    torch.cuda.synchronize()
    for i, (wf, af, bf) in enumerate(layers):
        check_parity(ys[i].float().cpu().numpy().astype(np.float64), orc.forward(x, "f16", wf, af, bf), f"layer {i}")
    F.close()


def test_mid_several_adapters():
    import torch
    K, N, r, n = 640, 160, 64, 3
    ids = [(7 * i) % 5 - 1 for i in range(30)]                # -1 and 3: no adapter
    wf, _, _ = make_case(67, K, N, 0, w="q3")
    adapters = adapters_for(K, N, r, "q4", n, 68)
    x = gen.make_x(69, len(ids), K)
    L = eora.MultiAdapterLayer(wf, adapters, max_m=len(ids))
    y = L.forward(x_to_torch(x, "f16"), ids)
    torch.cuda.synchronize()
    check_parity(y.float().cpu().numpy().astype(np.float64), reference(x, "f16", wf, adapters, ids), "multi")
    L.close()


@pytest.mark.parametrize("w,ab,K,N,r,n,group", [
    ("q4", "f16", 2048, 512, 64, 3, 128),
    ("q3", "q4", 2048, 512, 64, 3, 64),
    ("q4", "q8", 2048, 512, 40, 2, 128),
    ("sp24", "f16", 2048, 512, 128, 3, 128),
    ("sq4", "q3", 2048, 512, 64, 3, 128),
    ("q4", "f16", 128, 32, 64, 2, 128),                  # one pair: no cluster
    ("q3", "q4", 640, 96, 512, 8, 128),                  # 32 pairs of t, several chunks
])
def test_several_adapters_are_as_exact_at_every_number_of_tokens(w, ab, K, N, r, n, group):
    """A request's result must not depend on how many others share its batch: products of exact operands (fp16 X, integer q - z, t as
    an fp16 high and low part) summed in fp32, whatever kernel serves the number of tokens.  The bound, against float64 with an fp32 Y:
    the sums' rounding (a few 2^-24 of the partial sums, which are at most a few times Y) and the low part's (2^-22 of the compensation)
    stay below 2^-18; t or the weights rounded once to fp16 would show as 2^-13 to 2^-15."""
    import torch
    ids = [i % (n + 1) - 1 for i in range(32)]
    wf, _, _ = make_case(91, K, N, 0, w=w, group=group)
    adapters = adapters_for(K, N, r, ab, n, 92)
    x = gen.make_x(93, len(ids), K)
    ref = reference(x, "f16", wf, adapters, ids)
    L = eora.MultiAdapterLayer(wf, adapters, max_m=len(ids), y_dtype="f32")
    for m in (8, 9, 16, 17, 32):
        y = L.forward(x_to_torch(x[:m], "f16"), ids[:m])
        torch.cuda.synchronize()
        assert L.device_status() == 0
        rel = orc.parity_errors(y.cpu().numpy().astype(np.float64), ref[:m])[0]
        assert rel <= 2.0 ** -18, (m, rel)
    L.close()


@pytest.mark.parametrize("xd", ["f16", "bf16"])
def test_launches_of_several_adapters(xd):
    """eora_linear_launches and eora_linear_decode_grid follow the rule that a multi-adapter forward is dispatched by."""
    K, N, r = 512, 96, 64
    wf, _, _ = make_case(94, K, N, 0)
    L = eora.MultiAdapterLayer(wf, adapters_for(K, N, r, "f16", 2, 95), max_m=40, x_dtype=xd)
    for m in (1, 8, 9, 16, 17, 24, 32, 33, 40):
        one = xd == "f16" and 9 <= m <= 32
        assert eora.eora_linear_launches(L.handle, m) == (1 if one else (m + 7) // 8), m
        grid = eora.eora_linear_decode_grid(L.handle, m)
        # three pairs of row tiles: a cluster of two each, beside the CTAs that hold A; the kernel for eight tokens has one per row tile
        assert grid > 0 and (grid != eora.eora_linear_decode_grid(L.handle, 8)) == one, (m, grid)
    L.close()
