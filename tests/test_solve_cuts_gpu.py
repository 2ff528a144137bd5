"""GPU parity of the offline solve where its cuts can go wrong: the side of the iteration (n < d and n >= d), iterates of one to
several column tiles (64, 96, 128, 160 wide) and both eigensolvers (up to 320 columns and above), dimensions that are no whole tiles,
few and odd numbers of iterations, spectra that fall fast or end.  Compared with the float64 oracle through what is unique: the remaining
loss and the singular values, within the bounds of the solve's other tests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import eora_solve_oracle as sol
import eora_inputs as gen
from test_solve_gpu import run_solve, LOSS_RTOL, SIGMA_RTOL


@pytest.mark.parametrize("d,k,n,r", [
    (129, 127, 65, 3),          # n side, one tile and a bit
    (257, 100, 300, 60),        # d side, 92 columns
    (300, 129, 260, 90),        # n side, 122 columns
    (400, 300, 390, 150),       # 182 columns: two blocks of two columns per lane group
    (420, 500, 700, 280),       # 312 columns, the last of the cluster's eigensolver
    (420, 500, 410, 300),       # 332 columns: the one behind it
    (50, 70, 40, 30),           # n < m: the d side although n is smaller, an iterate of 50 columns and rank 40
])
def test_solve_cuts(d, k, n, r):
    w, w_hat, x = gen.make_solve_case(31, d, k, n)
    ref = sol.solve(w, w_hat, x, r)
    b, a, s, _ = run_solve(w, w_hat, x, r)
    opt, got = sol.layer_loss(ref["dW"], ref["B"], ref["A"], x), sol.layer_loss(ref["dW"], b, a, x)
    assert got <= opt * (1 + LOSS_RTOL), (got, opt)
    assert np.allclose(s, ref["sigma"], rtol=SIGMA_RTOL), (s[:4], ref["sigma"][:4])


@pytest.mark.parametrize("iters", [2, 4, 5, 6, 7])
def test_solve_few_iterations(iters):
    """Single products, pairs and a single one left over: with a spectrum of rank 8 and little noise every count has converged."""
    d, k, n, r = 160, 128, 256, 8
    w, w_hat, x = gen.make_solve_case(32, d, k, n, kind="gap", rank_signal=r)
    ref = sol.solve(w, w_hat, x, r)
    b, a, s, _ = run_solve(w, w_hat, x, r, iters=iters)
    opt, got = sol.layer_loss(ref["dW"], ref["B"], ref["A"], x), sol.layer_loss(ref["dW"], b, a, x)
    assert got <= opt * (1 + LOSS_RTOL), (got, opt)
    assert np.allclose(s, ref["sigma"], rtol=SIGMA_RTOL)


@pytest.mark.parametrize("decades,scale", [(2, 1.0), (3, 1e-6), (3, 1e4)])
def test_solve_falling_spectrum(decades, scale):
    """Singular values that fall by `decades` over the iterate's columns, at three scales: the iteration squares them twice."""
    d, k, n, r = 256, 256, 256, 64
    rng = np.random.default_rng(33)
    w, w_hat, _ = gen.make_solve_case(33, d, k, n)
    q1, q2 = (np.linalg.qr(rng.standard_normal((n, n)))[0] for _ in range(2))
    sv = 10.0 ** (-decades * np.arange(n) / 96)
    x = np.ascontiguousarray(((q1 * sv) @ q2 * scale).astype(np.float32))
    ref = sol.solve(w, w_hat, x, r)
    b, a, s, _ = run_solve(w, w_hat, x, r)
    opt, got = sol.layer_loss(ref["dW"], ref["B"], ref["A"], x), sol.layer_loss(ref["dW"], b, a, x)
    assert got <= opt * (1 + LOSS_RTOL), (got, opt)
    assert np.allclose(s, ref["sigma"], rtol=SIGMA_RTOL)


@pytest.mark.parametrize("d,k,n,r", [(130, 1500, 200, 20), (1500, 130, 200, 20), (256, 512, 1000, 64)])
def test_solve_needs_no_more_than_the_reported_workspace(d, k, n, r):
    """Solve and loss check in a workspace of exactly the reported size, with guard bytes behind it."""
    import torch
    import paper_2410_21271_b200 as eora
    w, w_hat, x = gen.make_solve_case(34, d, k, n)
    cfg = eora.eora_solve_config(d, k, n, r, 0, 0)
    size = eora.eora_solve_workspace_bytes(cfg)
    ws = torch.full((size + 65536,), 0xA5, dtype=torch.uint8, device="cuda:0")
    tw, th, tx = (torch.from_numpy(v).to("cuda:0") for v in (w, w_hat, x))
    b, a, s = torch.empty((d, r), device="cuda:0"), torch.empty((r, k), device="cuda:0"), torch.empty(r, device="cuda:0")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda:0")
    eora.eora_solve(cfg, tw, th, tx, b, a, s, ws[:size])
    eora.eora_solve_loss(cfg, tw, th, tx, b, a, loss, ws[:size])
    torch.cuda.synchronize()
    assert bool((ws[size:] == 0xA5).all())
    ref = sol.solve(w, w_hat, x, r)
    opt = sol.layer_loss(ref["dW"], ref["B"], ref["A"], x)
    assert abs(float(loss.item()) ** 0.5 - opt) <= opt * LOSS_RTOL
    assert eora.eora_solve(cfg, tw, th, tx, b, a, s, ws[:size - 1], check=False) == eora.EORA_ERR_BAD_SHAPE
