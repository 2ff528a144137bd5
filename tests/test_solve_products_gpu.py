"""GPU parity of the offline solve where its tensor-core products can go wrong: both tile widths, fewer reduction elements than a chunk of the
accumulators and a chunk with a remainder, padded sizes (X~ needed as whole tiles), iterates whose column tiles begin inside a block
of 128, one to four blocks of the Cholesky factor, and values at the ends of the range that three bf16 parts cover.  The error has rank r plus noise a hundred times smaller, so the compensation B'A and the singular values are unique and comparable with the float64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import eora_solve_oracle as sol
import eora_inputs as gen
from test_solve_gpu import run_solve

# fp32 accuracy of the products: 4096 terms carry at most 1e-6 relative (2-norm) into dW X~ and its square; over the gap of 100 between the
# singular values on both sides of the cut that is far below the rounding of W - W^ itself (|W| / |dW| * 2^-24 < 1e-5).
PRODUCT_RTOL = 1e-4
SIGMA_RTOL = 1e-6


@pytest.mark.parametrize("d,k,n,r", [
    (4736, 256, 1024, 24),      # 37 x 8 tiles: the wide tile; n side, an iterate of 56 columns on the CUDA cores
    (128, 128, 128, 8),         # one tile, four stages
    (300, 1100, 500, 40),       # padded everywhere; chunks of eight stages with a remainder
    (1024, 320, 384, 100),      # iterate of 132 columns: two tiles of 96, on the CUDA cores
    (700, 640, 900, 250),       # 282 columns: three tiles of 96, two blocks of the factor
    (640, 600, 700, 400),       # 432 columns: three blocks of the factor
    (1000, 1000, 1100, 480),    # 512 columns: four
    (512, 520, 600, 268),       # 300 columns on the tensor cores: two tiles of 160, the second beginning inside a block
])
def test_compensation_and_spectrum(d, k, n, r):
    w, w_hat, x = gen.make_solve_case(41, d, k, n, kind="gap", rank_signal=r)
    ref = sol.solve(w, w_hat, x, r)
    b, a, s, _ = run_solve(w, w_hat, x, r)
    want = ref["B"] @ ref["A"]
    assert np.linalg.norm(b @ a - want) <= PRODUCT_RTOL * np.linalg.norm(want)
    assert np.linalg.norm(s - ref["sigma"]) <= SIGMA_RTOL * np.linalg.norm(ref["sigma"])


@pytest.mark.parametrize("scale", [2.0 ** -40, 2.0 ** 40])
def test_scaled_activations_scale_sigma_alone(scale):
    """Powers of two change no rounding anywhere: sigma scales with X~, B'A stays the same bit for bit."""
    import torch
    import paper_2410_21271_b200 as eora
    d, k, n, r = 256, 384, 512, 32
    w, w_hat, x = (torch.from_numpy(v).cuda() for v in gen.make_solve_case(42, d, k, n))
    b0, a0, s0 = eora.solve(w, w_hat, x, r)
    b1, a1, s1 = eora.solve(w, w_hat, x * scale, r)
    torch.cuda.synchronize()
    assert torch.equal(s0 * scale, s1)
    assert torch.equal(b0 * scale, b1) and torch.equal(a0, a1 * scale)


def test_not_a_number_in_not_a_number_out():
    """One infinite activation makes every column of P that it meets infinite or NaN: nothing finite may be made up from it."""
    import torch
    import paper_2410_21271_b200 as eora
    w, w_hat, x = (torch.from_numpy(v).cuda() for v in gen.make_solve_case(43, 128, 128, 256))
    x[3, 5] = float("inf")
    b, a, s = eora.solve(w, w_hat, x, 16)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(b @ a).all())


@pytest.mark.parametrize("d,k,n,r", [(256, 256, 512, 16), (1024, 512, 1024, 64), (640, 384, 600, 350)])      # the last: eigenproblem in one CTA
@pytest.mark.parametrize("where,value", [("w", "nan"), ("w_hat", "inf"), ("x", "nan"), ("x", "-inf")])
def test_what_is_not_finite_shows_in_every_result(d, k, n, r, where, value):
    """sigma and A are not zero ("no error to compensate") where B' is not a number: every element of all three is not finite."""
    import torch
    import paper_2410_21271_b200 as eora
    t = dict(zip(("w", "w_hat", "x"), (torch.from_numpy(v).cuda() for v in gen.make_solve_case(44, d, k, n))))
    t[where][5, 7] = float(value)
    b, a, s = eora.solve(t["w"], t["w_hat"], t["x"], r)
    torch.cuda.synchronize()
    for name, v in (("B'", b), ("A", a), ("sigma", s)):
        assert not bool(torch.isfinite(v).any()), name


@pytest.mark.parametrize("d,k,n,r", [
    (1024, 1024, 4000, 60),     # without room beyond the matrices: dW's place used in between, every product but C's own in parts
    (1500, 1024, 1000, 60),     # the same on the n side
    (1500, 300, 1000, 60),      # few inputs: C split over itself in slabs; in the smallest workspace products with C itself
    (1100, 200, 1300, 60),      # the same on the d side
    (1700, 300, 1300, 30),      # an iterate's parts among the matrices', not among the small problems
    (60, 40, 3000, 20),         # small matrices, many columns
])
def test_workspaces_down_to_the_matrices_alone(d, k, n, r):
    """The reported workspace, less than that, and one that holds dW, P, C and the iterates and nothing else: results as ever, and nothing behind it is touched."""
    import torch
    import paper_2410_21271_b200 as eora
    from test_solve_plan_cpu import matrices
    w, w_hat, x = gen.make_solve_case(45, d, k, n, kind="gap", rank_signal=r)
    ref = sol.solve(w, w_hat, x, r)
    want = ref["B"] @ ref["A"]
    cfg = eora.eora_solve_config(d, k, n, r, 0, 0)
    tw, th, tx = (torch.from_numpy(v).cuda() for v in (w, w_hat, x))
    most = eora.eora_solve_workspace_bytes(cfg)
    for size in sorted({most, max(most - 1, matrices(d, k, n, r)), matrices(d, k, n, r)}):
        ws = torch.full((size + 65536,), 0xA5, dtype=torch.uint8, device="cuda:0")
        b, a, s = torch.empty((d, r), device="cuda:0"), torch.empty((r, k), device="cuda:0"), torch.empty(r, device="cuda:0")
        loss = torch.zeros(1, dtype=torch.float64, device="cuda:0")
        eora.eora_solve(cfg, tw, th, tx, b, a, s, ws[:size])
        eora.eora_solve_loss(cfg, tw, th, tx, b, a, loss, ws[:size])
        torch.cuda.synchronize()
        assert bool((ws[size:] == 0xA5).all())
        got = b.cpu().numpy().astype(np.float64) @ a.cpu().numpy()
        assert np.linalg.norm(got - want) <= PRODUCT_RTOL * np.linalg.norm(want)
        assert np.linalg.norm(s.cpu().numpy() - ref["sigma"]) <= SIGMA_RTOL * np.linalg.norm(ref["sigma"])


def test_more_tiles_than_clusters_of_two():
    """An iterate of 512 columns with 2432 rows: 76 tiles of its product with C, a CTA each."""
    d, k, n, r = 2432, 600, 2500, 32
    w, w_hat, x = gen.make_solve_case(46, d, k, n, kind="gap", rank_signal=r)
    ref = sol.solve(w, w_hat, x, r)
    want = ref["B"] @ ref["A"]
    b, a, s, _ = run_solve(w, w_hat, x, r, oversample=480)
    assert np.linalg.norm(b @ a - want) <= PRODUCT_RTOL * np.linalg.norm(want)
    assert np.linalg.norm(s - ref["sigma"]) <= SIGMA_RTOL * np.linalg.norm(ref["sigma"])


def test_tensor_core_products_side_by_side_on_three_streams():
    """Three solves whose clusters share the GPU: every one gives what it gives alone, bit for bit."""
    import torch
    import paper_2410_21271_b200 as eora
    cases = [(1024, 900, 1100, 64), (1500, 1024, 1024, 100), (900, 1024, 1000, 128)]
    ins = [(tuple(torch.from_numpy(v).cuda() for v in gen.make_solve_case(47 + i, d, k, n)), r) for i, (d, k, n, r) in enumerate(cases)]
    alone = [eora.solve(*t, r) for t, r in ins]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in cases]
    for rep in range(3):
        outs = []
        for st, (t, r) in zip(streams, ins):
            with torch.cuda.stream(st):
                outs.append(eora.solve(*t, r, stream=st))
    torch.cuda.synchronize()
    for one, other in zip(alone, outs):
        assert all(torch.equal(u, v) for u, v in zip(one, other))
