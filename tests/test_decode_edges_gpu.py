"""GPU parity of the decode kernel where its cuts can go wrong: one pair of reduction tiles (no cluster), an odd number of pairs
(unequal halves), fewer row tiles than CTAs, more than a cluster's shared memory holds, a reduction axis in several chunks, t
in several chunks, row tiles of different fused layers in one CTA.  Tolerance as for every forward (tests/helpers.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import eora_oracle as orc
import eora_inputs as gen
import paper_2410_21271_b200 as eora
from helpers import make_case, run_layer, check_parity, x_to_torch


@pytest.mark.parametrize("w,ab,K,N,r,M,xd,group", [
    ("q4", "f16", 128, 32, 8, 1, "f16", 128),          # one pair: a cluster of one, the shortest run (one blob)
    ("q3", "f16", 128, 96, 0, 8, "bf16", 64),
    ("q3", "f16", 384, 64, 128, 1, "f16", 128),        # three pairs: halves of two and one
    ("q4", "q8", 640, 160, 72, 7, "f16", 64),
    ("q4", "f16", 256, 61024, 16, 1, "f16", 128),      # 3814 row tiles: more than 48 per cluster, several waves of CTAs
    ("q3", "f16", 256, 61024, 16, 8, "f16", 128),
    ("q4", "f16", 14336, 64, 64, 8, "f16", 128),       # 56 pairs per half: two chunks of activations
    ("sp24", "q4", 14336, 32, 128, 5, "bf16", 128),
    ("q3", "f16", 512, 96, 2048, 8, "f16", 128),       # 16 pairs of t, four at a time
    ("sq4", "q3", 512, 96, 1024, 2, "f16", 128),
])
def test_decode_cuts(w, ab, K, N, r, M, xd, group):
    wf, af, bf = make_case(41, K, N, r, w=w, ab=ab, group=group)
    x = gen.make_x(42, M, K, xd)
    L = eora.Layer(wf, af, bf, max_m=M, x_dtype=xd)
    assert L.path(M) == eora.EORA_PATH_DECODE
    y_ref = orc.forward(x, xd, wf, af, bf)
    for rep in range(2):
        check_parity(run_layer(L, x, xd), y_ref, f"{w}/{ab} K{K} N{N} r{r} M{M} call {rep}")
    L.close()


@pytest.mark.parametrize("M", [1, 6])
def test_decode_bf16_beyond_fp16(M):
    """bf16 activations outside fp16's range (and blocks of very small ones) through a layer without an adapter."""
    K, N = 512, 96
    wf, _, _ = make_case(43, K, N, 0, w="q4")
    rng = np.random.default_rng(44)
    mag = np.repeat(np.exp2(rng.integers(-40, 30, (M, K // 128))), 128, axis=1)
    x = gen.f32_to_bf16_bits((rng.standard_normal((M, K)) * mag).astype(np.float32))
    L = eora.Layer(wf, None, None, max_m=M, x_dtype="bf16", y_dtype="f32")
    check_parity(run_layer(L, x, "bf16"), orc.forward(x, "bf16", wf, None, None), f"M{M}")
    L.close()


@pytest.mark.parametrize("M", [1, 2, 5, 8])
def test_decode_bf16_over_its_whole_range(M):
    """Blocks of bf16 activations whose largest magnitude lies anywhere between 2^-112 and 2^122 (a sum of 256 products with weights
    below one still fits a float): each is a block of a power of two times fp16 numbers, so none may be lost or overflow."""
    K, N = 256, 96
    wf, _, _ = make_case(47, K, N, 0, w="q3")
    rng = np.random.default_rng(48)
    L = eora.Layer(wf, None, None, max_m=M, x_dtype="bf16", y_dtype="f32")
    for e in (-110, -104, -96, -95, 0, 112, 113, 118):
        x = rng.uniform(1.0, 2.0, (M, K)) * rng.choice([-1.0, 1.0], (M, K))
        xb = gen.f32_to_bf16_bits(np.ldexp(x, e).astype(np.float32))
        ref = orc.forward(xb, "bf16", wf, None, None)
        scale = 2.0 ** -e                                        # (compared near one: squares of 1e-33 would underflow)
        check_parity(run_layer(L, xb, "bf16") * scale, ref * scale, f"M{M} 2^{e}")
    L.close()


def test_decode_fused_layers_share_a_cta():
    """Four layers of one to five row tiles each: a cluster's row tiles belong to several layers, with different pairs of t."""
    import torch
    K, r, M = 512, 128, 4
    layers = [make_case(45 + i, K, N, r, w="q3") for i, N in enumerate((32, 4096, 64, 4160))]
    x = gen.make_x(46, M, K)
    F = eora.FusedLayers(layers, max_m=M)
    ys = F.forward(x_to_torch(x, "f16"))
    torch.cuda.synchronize()
    for i, (wf, af, bf) in enumerate(layers):
        check_parity(ys[i].float().cpu().numpy().astype(np.float64), orc.forward(x, "f16", wf, af, bf), f"layer {i}")
    F.close()


@pytest.mark.parametrize("M", [1, 8])
def test_decode_of_very_many_outputs(M):
    """400 000 outputs: more row tiles than a thousand CTAs take, in waves."""
    K, N = 128, 400000
    wf, _, _ = make_case(49, K, N, 0, w="q3")
    x = gen.make_x(50, M, K)
    L = eora.Layer(wf, None, None, max_m=M)
    assert L.path(M) == eora.EORA_PATH_DECODE
    check_parity(run_layer(L, x, "f16"), orc.forward(x, "f16", wf, None, None), f"M{M}")
    L.close()


def test_decode_of_many_long_2to4_rows():
    """2:4, eight tokens, a reduction axis in several parts, 48 row tiles per cluster and four pairs of t: with those, activations, sums and rings of
    large blobs do not fit at once, and the launch is cut finer.  Every quad keeps its first two places, so that a few columns are quickly checked."""
    import torch
    K, N, r, M = 14848, 57344, 512, 8
    g = torch.Generator(device="cuda:0").manual_seed(51)
    vals = (torch.randn((N, K // 2), device="cuda:0", generator=g) * 0.02).half()
    meta = torch.full((N, K // 32), 0x44444444, dtype=torch.int32, device="cuda:0")
    cfg, wts = eora.eora_linear_config(), eora.eora_linear_weights()
    cfg.d_in, cfg.d_out, cfg.rank, cfg.w_format, cfg.w_bits, cfg.w_group = K, N, r, eora.EORA_W_SPARSE24, 4, 128
    cfg.ab_format, cfg.ab_group, cfg.x_dtype, cfg.y_dtype, cfg.max_m = eora.EORA_AB_F16, 128, eora.EORA_X_F16, eora.EORA_Y_F32, M
    a = (torch.randn((K, r), device="cuda:0", generator=g) * 0.02).half()
    b = (torch.randn((r, N), device="cuda:0", generator=g) * 0.02).half()
    wts.w_codes, wts.w_zeros, wts.a, wts.b = vals.data_ptr(), meta.data_ptr(), a.data_ptr(), b.data_ptr()
    h = eora.eora_linear_create(cfg, wts)
    x = torch.randn((M, K), device="cuda:0", generator=g).half()
    y = torch.empty((M, N), device="cuda:0")
    assert eora.eora_linear_path(h, M) == eora.EORA_PATH_DECODE
    eora.eora_linear_forward(h, x, M, y)
    torch.cuda.synchronize()
    assert eora.eora_linear_last_device_status(h) == 0
    eora.eora_linear_destroy(h)
    cols = torch.arange(0, N, 331, device="cuda:0")
    kept = x.double().reshape(M, K // 4, 4)[:, :, :2].reshape(M, K // 2)
    ref = kept @ vals[cols].double().T + (x.double() @ a.double()) @ b[:, cols].double()
    check_parity(y[:, cols].double().cpu().numpy(), ref.cpu().numpy())
