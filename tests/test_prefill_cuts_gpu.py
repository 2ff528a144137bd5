"""GPU parity of the tensor-core path for more than 32 tokens where its cuts can go wrong: clusters that share a reduction axis
(uneven shares, an extension longer than one share, the fewest k-blocks that are split), token tiles with a remainder, rows that
end inside a tile, fused layers of 128-row tiles, launches chained back to back.  Tolerance as for every forward (tests/helpers.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import eora_oracle as orc
import eora_inputs as gen
import paper_2410_21271_b200 as eora
from helpers import make_case, run_layer, check_parity, x_to_torch, prefill_plan


@pytest.mark.parametrize("w,ab,K,N,r,M,xd,yd,group", [
    ("q4", "f16", 128, 32, 0, 33, "f16", "f16", 128),       # two k-blocks, one ragged row tile: no split
    ("q4", "f16", 512, 128, 64, 33, "f16", "f32", 64),      # eight k-blocks, a float result
    ("q4", "f16", 2048, 384, 128, 64, "f16", "f16", 128),
    ("q3", "q8", 4096, 544, 512, 48, "bf16", "bf16", 128),  # shares of eight CTAs, 544 = 4 * 128 + 32 rows
    ("q3", "f16", 512, 512, 2048, 70, "f16", "f16", 128),   # an extension four times as long as the backbone's reduction axis
    ("sp24", "q4", 1152, 1024, 64, 100, "f16", "f32", 128), # 18 k-blocks: pairs do not divide evenly
    ("sq4", "f16", 2048, 2080, 0, 257, "f16", "f16", 128),  # two token tiles, the second ragged
    ("q4", "q3", 14336, 512, 256, 333, "bf16", "f16", 128),
    ("q4", "f16", 1024, 4096, 24, 700, "f16", "f16", 128),
])
def test_prefill_cuts(w, ab, K, N, r, M, xd, yd, group):
    wf, af, bf = make_case(71, K, N, r, w=w, ab=ab, group=group)
    x = gen.make_x(72, M, K, xd)
    L = eora.Layer(wf, af, bf, max_m=M, x_dtype=xd, y_dtype=yd)
    ref = orc.forward(x, xd, wf, af, bf)
    for rep in range(2):
        check_parity(run_layer(L, x, xd), ref, f"{w}/{ab} K{K} N{N} r{r} M{M} call {rep}")
    L.close()


@pytest.mark.parametrize("M", [40, 130])
def test_prefill_fused_calls_in_a_row(M):
    """Calls that follow each other without a wait, each reading what the one in front wrote: X of the second is Y of the first."""
    import torch
    K, r = 1024, 64
    layers = [make_case(75 + i, K, N, r, w="q4") for i, N in enumerate((1024, 128, 384))]
    F = eora.FusedLayers(layers, max_m=M)
    one = eora.Layer(*layers[0], max_m=M)
    x = gen.make_x(76, M, K)
    xt = x_to_torch(x, "f16")
    for rep in range(3):
        y = one.forward(xt)
        ys = F.forward(y)
    torch.cuda.synchronize()
    check_parity(y.float().cpu().numpy().astype(np.float64), orc.forward(x, "f16", *layers[0]), "first")
    x2 = y.cpu().numpy()
    for i, case in enumerate(layers):
        check_parity(ys[i].float().cpu().numpy().astype(np.float64), orc.forward(x2, "f16", *case), f"layer {i}")
    F.close()
    one.close()


@pytest.mark.parametrize("w,ab,K,N,r,M,group", [
    ("q4", "f16", 256, 38144, 64, 160, 128),   # 256 rows x 160 tokens: the accumulators leave tensor memory for three stages of weights
    ("q4", "f16", 256, 38144, 64, 161, 128),   # one token more: 128 rows x 176 tokens
    ("q4", "f16", 256, 38144, 64, 352, 128),
    ("sp24", "q8", 384, 38144, 128, 64, 128),  # units of one tile (2:4) and of two (8-bit)
    ("q3", "q3", 640, 18944, 256, 224, 128),   # 128 rows x 224 tokens
    ("sq4", "q4", 256, 288, 64, 40, 128),      # row tiles past the matrix
    ("q4", "f16", 128, 2048, 64, 34, 128),     # fewer units than a warp's ring has slots
    ("q4", "f16", 640, 544, 64, 50, 64),       # a scale entry per tile
    ("q3", "q8", 4096, 2176, 512, 100, 64),    # clusters; the halves of the reduction axis; rings that go round
])
def test_prefill_weights_in_tensor_memory(w, ab, K, N, r, M, group):
    """Where the dequantised weights go to tensor memory and where they do not: tiles of weight rows and tokens around the limit, rows past the
    matrix, rings that are not filled and rings that go round, both sizes of a unit of work, one or two scale entries."""
    wf, af, bf = make_case(77, K, N, r, w=w, ab=ab, group=group)
    x = gen.make_x(78, M, K, "f16")
    L = eora.Layer(wf, af, bf, max_m=M)
    check_parity(run_layer(L, x, "f16"), orc.forward(x, "f16", wf, af, bf), f"{w}/{ab} K{K} N{N} r{r} M{M}")
    L.close()


@pytest.mark.parametrize("w,ab,K,N,r,M,stages,tm", [
    ("q4", "q4", 640, 3936, 256, 1100, 3, 0),     # 256 rows x 256 tokens, five units of W and two of B
    ("q4", "f16", 640, 3936, 64, 1100, 3, 0),     # units of B of one k-block
    ("q4", "f16", 512, 3936, 64, 1100, 3, 0),     # an even number of units
    ("q4", "q4", 640, 19040, 256, 143, 3, 1),     # weights in tensor memory
    ("q3", "f16", 384, 19040, 128, 143, 3, 1),
    ("q4", "q8", 256, 19040, 256, 143, 3, 1),
    ("sp24", "q4", 640, 19040, 256, 143, 3, 1),   # units of W of one k-block
    ("q4", "q3", 640, 19040, 256, 100, 4, 1),
    ("sq4", "q8", 640, 544, 256, 1100, 4, 1),     # 128 rows x 256 tokens
])
def test_prefill_short_rings(w, ab, K, N, r, M, stages, tm):
    """The shortest rings, with tiles of one half (two warps to a row tile): odd and even numbers of units in front of the extension's."""
    main = prefill_plan(w, ab, K, N, r, M)[0]
    assert (main.stages, main.in_tensor_memory) == (stages, tm) and 0 < (N - 1) % main.rows + 1 <= 128
    wf, af, bf = make_case(79, K, N, r, w=w, ab=ab)
    x = gen.make_x(80, M, K, "f16")
    L = eora.Layer(wf, af, bf, max_m=M)
    ref = orc.forward(x, "f16", wf, af, bf)
    for rep in range(3):
        check_parity(run_layer(L, x, "f16"), ref, f"{w}/{ab} K{K} N{N} r{r} M{M} call {rep}")
    L.close()


@pytest.mark.parametrize("w,ab,K,N,r,M,main_cut,t_cut", [
    # the plan's tiles and clusters: (rows, CTAs that share a tile's reduction axis) of the main product and of t = X.A
    ("sq4", "q4", 2560, 192, 1024, 33, (128, 3), (128, 8)),
    ("sp24", "f16", 4096, 8768, 1024, 167, (256, 3), (128, 3)),     # through shared memory
    ("q3", "q4", 1408, 9280, 512, 34, (256, 3), (128, 4)),
    ("sp24", "q4", 5248, 1856, 512, 37, (128, 5), (128, 8)),
    ("q4", "q8", 3968, 4960, 512, 43, (256, 5), (128, 4)),
    ("sq4", "q3", 4992, 192, 512, 35, (128, 6), (128, 8)),
    ("q3", "q8", 4096, 4128, 64, 33, (256, 6), (128, 8)),
    ("q3", "q3", 4096, 128, 384, 34, (128, 7), (128, 8)),
    ("sp24", "q8", 4736, 2848, 512, 46, (256, 7), (128, 8)),
    ("sq4", "q8", 2688, 5600, 64, 34, (128, 3), (128, 3)),
    ("q4", "q4", 2688, 5408, 2048, 292, (128, 1), (256, 3)),
    ("q3", "f16", 5760, 1568, 2048, 36, (128, 3), (128, 5)),
    ("sq4", "f16", 4480, 5664, 2048, 43, (128, 2), (256, 5)),
    ("q3", "q4", 5376, 2336, 64, 36, (128, 6), (128, 6)),
    ("sp24", "q4", 5376, 5312, 256, 34, (128, 3), (256, 6)),
    ("sq4", "f16", 3968, 256, 384, 492, (128, 8), (128, 7)),
    # the fewest k-blocks of a share: four
    ("q3", "q3", 512, 128, 1024, 173, (128, 2), (128, 1)),
    ("q3", "f16", 1024, 128, 0, 35, (128, 4), (0, 0)),
    ("sq4", "q4", 1920, 384, 2048, 223, (128, 7), (128, 4)),        # and an extension longer than a share
    ("sq4", "q8", 2048, 192, 0, 33, (128, 8), (0, 0)),
    # an extension longer than a share
    ("q3", "q8", 896, 160, 1024, 33, (128, 2), (128, 2)),
    ("q3", "f16", 1024, 128, 384, 173, (128, 4), (128, 4)),
    ("q3", "q3", 2048, 160, 384, 182, (128, 8), (128, 8)),
])
def test_prefill_clusters_of_every_size(w, ab, K, N, r, M, main_cut, t_cut):
    """Even and uneven deals of k-blocks and of epilogue units, which the plan is asked for first."""
    main, t = prefill_plan(w, ab, K, N, r, M)
    assert ((main.rows, main.cluster), (t.rows, t.cluster)) == (main_cut, t_cut)
    wf, af, bf = make_case(81, K, N, r, w=w, ab=ab)
    x = gen.make_x(82, M, K, "f16")
    L = eora.Layer(wf, af, bf, max_m=M)
    ref = orc.forward(x, "f16", wf, af, bf)
    for rep in range(2):
        check_parity(run_layer(L, x, "f16"), ref, f"{w}/{ab} K{K} N{N} r{r} M{M} call {rep}")
    L.close()
