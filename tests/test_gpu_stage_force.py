"""The stage's force product f = W^T (W x) on whole numbers: every product and
sum is exact in any order, so the result is compared bit for bit (a rounding
bound for rows of thousands of values would let a lost part of a row pass)."""
import pytest
import torch

import lgf_inputs as li

pytestmark = pytest.mark.gpu


# row lengths 3 nm of every class of the one-pass product (up to 512, 1024, 2048, 4096
# vectors of 16 bytes), their ends, rows that are no whole vectors, a factor off
# the 16-byte alignment (shift), the longest one-pass rows and rows beyond them
@pytest.mark.parametrize("prec,nm,shift", [("f32", 1, 0), ("f32", 60, 0), ("f32", 60, 1), ("f32", 682, 0), ("f32", 683, 0),
                                           ("f32", 1365, 0), ("f32", 1366, 0), ("f32", 2730, 0), ("f32", 2732, 0),
                                           ("f32", 2733, 0), ("f32", 4096, 3), ("f32", 5120, 0), ("f32", 5461, 0),
                                           ("f32", 5462, 0), ("f64", 1, 0), ("f64", 341, 0), ("f64", 342, 1),
                                           ("f64", 682, 0), ("f64", 1366, 0), ("f64", 2730, 0), ("f64", 2731, 0)])
def test_force_product_exact(prec, nm, shift, ctx64, ctx32):
    """W is +-1 everywhere and x is +-1 (one 2 where the row length is even), so that every
    (W x)_r is odd: each element of W and each row changes the result."""
    ctx = ctx64 if prec == "f64" else ctx32
    dt, n, b, D = ctx.dtype, 3 * nm, 8, li.box_blocks(2, 2, 2)
    gen = torch.Generator("cuda").manual_seed(nm)
    sign = lambda *s: torch.randint(0, 2, s, device="cuda", generator=gen, dtype=torch.int8).to(dt) * 2 - 1
    X = 2.0 + 12.0 * torch.rand(nm, 3, dtype=torch.float64, device="cuda", generator=gen)
    W = sign(n * n + shift)[shift:].view(n, n)
    x = sign(n)
    if n % 2 == 0:
        x[n // 2] = 2
    r = torch.zeros(3 * D.shape[0] * b ** 3, dtype=dt, device="cuda")
    u, f = torch.empty_like(r), torch.full((n,), float("nan"), dtype=dt, device="cuda")
    # r = 0 makes U = 0 exactly, so the right-hand side U - u_Gamma is x
    ctx.nested_projection_stage(b, D, r, u, X_prev=X, X=X, ub=-x, W1=W, alpha=0.1, f=f)
    ref, size = torch.zeros(n, dtype=torch.float64, device="cuda"), 0.0
    for a in range(0, n, 2048):
        y = W[a:a + 2048].double() @ x.double()
        assert bool((y.remainder(2) == 1).all())
        ref += W[a:a + 2048].double().T @ y
        size += float(y.abs().sum())
    assert size < 2 ** 24     # every partial sum, in any order, is a whole number below this
    assert torch.equal(f.double(), ref)
