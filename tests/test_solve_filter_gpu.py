"""GPU parity of the offline solve's default iteration (fourteen products with a Chebyshev filter) with the plain one of 24 products, over the shapes that
a spectrum of the projected error can have, with few and many extra vectors: it has to come at least as close to the optimum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import paper_2410_21271_b200 as eora


def spectrum(kind, q, r):
    """q falling singular values; `r`: the rank that will be asked for."""
    i = np.arange(q, dtype=np.float64)
    return {"power law": (1 + i) ** -0.5, "flat": 1 - 0.5 * i / q, "nearly flat": 1 - 0.05 * i / q, "ends at the rank": np.where(i < r, 1 - 0.5 * i / q, 0.0),
            "ends before the rank": np.where(i < r // 2, 1 - 0.5 * i / q, 0.0), "falling": 10.0 ** (-4 * i / q), "plateau": np.where(i < r // 2, 2.0, 1 - 0.1 * i / q),
            "gap": np.where(i < r, 1 - 0.3 * i / q, 0.02 * (1 - 0.5 * i / q)), "spiked": np.where(i < 3, 300.0 / (1 + i), 1 - 0.5 * i / q)}[kind]


def case(kind, d, q, r, seed):
    """dW = U diag(s) V^T with the rows of X~ orthonormal: dW X~ has the singular values s, and the optimum is what is left of them."""
    rng = np.random.default_rng(seed)
    s = spectrum(kind, q, r)
    u, v, x = (np.linalg.qr(rng.standard_normal((n, q)))[0] for n in (d, q, q))
    return ((u * s) @ v.T).astype(np.float32), x.T.astype(np.float32).copy(), s


def excess(dw, x, r, s, **kw):
    """Remaining loss squared over the optimum's, less one (where nothing is left: over the whole error)."""
    import torch
    w, xt = torch.from_numpy(dw).cuda(), torch.from_numpy(x).cuda()
    b, a, _ = eora.solve(w, torch.zeros_like(w), xt, r, **kw)
    left = (w.double() - b.double() @ a.double()) @ xt.double()
    best = float((torch.linalg.svdvals(w.double() @ xt.double())[r:] ** 2).sum())
    whole = float(np.sum(s ** 2))
    return (float((left ** 2).sum()) - best) / (best if best > 1e-9 * whole else whole)


# Rounding alone: at the optimum the loss does not change to first order in the factors' span, so a product's error of at most 2^-21 of the whole counts
# squared, 2.3e-13 of the whole, and the whole is up to 4000 times the optimum ("gap", "spiked").
ROUNDING = 1e-9


@pytest.mark.parametrize("over", [1, 4, 32])
@pytest.mark.parametrize("kind", ["power law", "flat", "nearly flat", "ends at the rank", "ends before the rank", "falling", "plateau", "gap", "spiked"])
def test_default_iteration_converges_as_far_as_24_plain_products(kind, over):
    d, q, r = 320, 256, 32
    dw, x, s = case(kind, d, q, r, 51)
    filtered, plain = excess(dw, x, r, s, oversample=over), excess(dw, x, r, s, oversample=over, iters=24)
    print(f"{kind}, {over} extra: filtered {filtered:.3e}, plain {plain:.3e}, 14 plain {excess(dw, x, r, s, oversample=over, iters=14):.3e}")
    assert filtered <= plain + ROUNDING


@pytest.mark.parametrize("kind", ["power law", "flat", "plateau"])
def test_default_iteration_with_products_on_the_tensor_cores(kind):
    d, q, r = 1100, 1024, 64
    dw, x, s = case(kind, d, q, r, 52)
    filtered, plain = excess(dw, x, r, s), excess(dw, x, r, s, iters=24)
    print(f"{kind}: filtered {filtered:.3e}, plain {plain:.3e}, 14 plain {excess(dw, x, r, s, iters=14):.3e}")
    assert filtered <= plain + ROUNDING
