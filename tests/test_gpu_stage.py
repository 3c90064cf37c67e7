"""The nested-projection stage (Sec. 3.1, Eq. nested_proj: ip -> f -> pc -> vc)
on the GPU against the oracle's composition of the same steps, element by
element: u on every face of D, d_hat on every cell of D, f_hat at every
marker.  FP64 at 1e-12 and FP32 at 1e-5 relative L-infinity.

With W1 = C^-1 (the oracle's force Schur complement of Eq. force_schur) the
GPU's u also meets the no-slip row I^i u = u_Gamma at the markers."""
import numpy as np
import pytest
import torch

import lgf_inputs as li
from conftest import rel_linf

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-12, "f32": 1e-5}


def _case(nm, move, seed):
    rng = np.random.default_rng(seed)
    b = 8
    D = li.box_blocks(4, 3, 3)
    c = np.array([16.0, 12.0, 12.0])
    ang = np.linspace(0, 2 * np.pi, nm, endpoint=False)
    X = c + np.stack([3.5 * np.cos(ang), 3.0 * np.sin(ang), 1.2 * np.cos(3 * ang)], axis=1)
    Xp = X + move * np.array([1.0, -0.5, 0.25])
    r = rng.uniform(-1, 1, size=(3, D.shape[0], b ** 3))
    ub = rng.normal(size=(3, nm))
    return b, D, X, Xp, r, ub


def _run(ctx, b, D, X, Xp, r, ub, W1, W2, alpha, dx):
    dt = ctx.dtype
    dev = "cuda"
    nD = D.shape[0]
    rt = torch.tensor(r.reshape(-1), dtype=dt, device=dev)
    u = torch.full((3 * nD * b ** 3,), float("nan"), dtype=dt, device=dev)
    d = torch.full((nD * b ** 3,), float("nan"), dtype=dt, device=dev)
    kw = {}
    f = None
    if X.shape[0]:
        f = torch.full((3 * X.shape[0],), float("nan"), dtype=dt, device=dev)
        kw = dict(X_prev=torch.tensor(Xp, dtype=torch.float64, device=dev),
                  X=torch.tensor(X, dtype=torch.float64, device=dev),
                  ub=torch.tensor(ub.reshape(-1), dtype=dt, device=dev),
                  W1=torch.tensor(W1, dtype=dt, device=dev),
                  W2=None if W2 is None else torch.tensor(W2, dtype=dt, device=dev), f=f)
    ctx.nested_projection_stage(b, D, rt, u, alpha=alpha, dx=dx, d=d, **kw)
    torch.cuda.synchronize()
    return (u.cpu().numpy().reshape(3, nD, -1), d.cpu().numpy().reshape(nD, -1),
            None if f is None else f.cpu().numpy().reshape(3, -1))


def test_stage_fp64_no_slip_with_exact_schur_inverse(ctx64, oracle):
    b, D, X, Xp, r, ub = _case(8, 0.0, 11)
    alpha, dx = 0.15, 0.5
    C = oracle.force_schur(b, D, Xp, X, alpha, dx, R=64)
    W1, W2 = np.linalg.inv(C), np.eye(C.shape[0])
    u, d, f = _run(ctx64, b, D, X, Xp, r, ub, W1, W2, alpha, dx)
    ur, dr, fr = oracle.nested_projection_stage(b, D, r, Xp, X, ub, W1, W2, alpha=alpha, dx=dx, R=64)
    assert rel_linf(u, ur) < TOL["f64"]
    assert rel_linf(d, dr) < TOL["f64"]
    assert rel_linf(f, fr) < TOL["f64"]
    U = oracle.ib_interp(b, D, X, u[None].astype(np.float64))[0]
    assert np.abs(U - ub).max() < 1e-9 * np.abs(ub).max()


@pytest.mark.parametrize("prec,move,nm", [("f64", 0.3, 6), ("f32", 0.0, 8), ("f32", 0.3, 6), ("f64", 0.0, 0)])
def test_stage_matches_oracle(prec, move, nm, ctx64, ctx32, oracle):
    ctx = ctx64 if prec == "f64" else ctx32
    b, D, X, Xp, r, ub = _case(nm, move, 12 + nm)
    alpha, dx = 0.25, 1.0
    W1 = np.random.default_rng(3).normal(size=(3 * nm, 3 * nm)) * 0.2
    W2 = None if move == 0.0 else np.random.default_rng(4).normal(size=(3 * nm, 3 * nm)) * 0.2
    u, d, f = _run(ctx, b, D, X, Xp, r, ub, W1, W2, alpha, dx)
    ur, dr, fr = oracle.nested_projection_stage(b, D, r, Xp, X, ub, W1, W2, alpha=alpha, dx=dx, R=64)
    assert not np.isnan(u).any() and not np.isnan(d).any()
    assert rel_linf(u, ur) < TOL[prec]
    assert rel_linf(d, dr) < TOL[prec]
    if nm:
        assert rel_linf(f, fr) < TOL[prec]


def test_stage_empty_flow_set(ctx64):
    f = torch.full((6,), float("nan"), dtype=torch.float64, device="cuda")
    X = torch.zeros((2, 3), dtype=torch.float64, device="cuda")
    ub = torch.zeros(6, dtype=torch.float64, device="cuda")
    W = torch.zeros((6, 6), dtype=torch.float64, device="cuda")
    ctx64.nested_projection_stage(8, np.zeros((0, 3), np.int32), None, None, X_prev=X, X=X, ub=ub, W1=W, f=f)
    torch.cuda.synchronize()
    assert torch.equal(f, torch.zeros_like(f))


@pytest.mark.parametrize("prec,nm,shift", [("f32", 1, 0), ("f32", 60, 0), ("f32", 60, 1), ("f32", 682, 0), ("f32", 683, 0),
                                           ("f32", 1366, 0), ("f32", 2732, 0), ("f32", 5462, 0), ("f64", 1, 0),
                                           ("f64", 341, 0), ("f64", 342, 1), ("f64", 1366, 0), ("f64", 2731, 0)])
def test_stage_force_product_sizes(prec, nm, shift, ctx64, ctx32):
    """f = W^T W (U - u_Gamma) with r = 0, so that U = 0 exactly: rows of every
    length class of the one-pass product, rows that are no whole vectors, a
    factor off the 16-byte alignment (shift) and rows beyond the one-pass limit.
    Any summation order of n products meets 2 (n + 1) u |W|^T |W| |x| (u the
    unit roundoff), with one more such factor for the second product."""
    ctx = ctx64 if prec == "f64" else ctx32
    dt, n = ctx.dtype, 3 * nm
    b, D = 8, li.box_blocks(2, 2, 2)
    gen = torch.Generator("cuda").manual_seed(nm)
    X = 2.0 + 12.0 * torch.rand(nm, 3, dtype=torch.float64, device="cuda", generator=gen)
    W = torch.randn(n * n + shift, dtype=dt, device="cuda", generator=gen)[shift:].view(n, n)
    ub = torch.randn(n, dtype=dt, device="cuda", generator=gen)
    r = torch.zeros(3 * D.shape[0] * b ** 3, dtype=dt, device="cuda")
    u, f = torch.empty_like(r), torch.full((n,), float("nan"), dtype=dt, device="cuda")
    ctx.nested_projection_stage(b, D, r, u, X_prev=X, X=X, ub=ub, W1=W, alpha=0.1, f=f)
    ref, bound = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    for a in range(0, n, 2048):   # the rows in FP64, a part at a time
        w = W[a:a + 2048].double()
        ref -= w.T @ (w @ ub.double())
        bound += w.abs().T @ (w.abs() @ ub.double().abs())
    tol = 4 * (n + 2) * torch.finfo(dt).eps / 2
    assert bool(((f.double() - ref).abs() <= tol * bound).all())


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("b", [4, 8, 16])
def test_stage_right_hand_side_off_the_vector_alignment(prec, b, ctx64, ctx32):
    """r one value off the 16-byte alignment: the same bits as aligned."""
    ctx = ctx64 if prec == "f64" else ctx32
    D = li.random_sparse(9, b=b, nsrc=5, ntgt=1, extent=(3, 2, 2)).src
    r = torch.randn(3 * D.shape[0] * b ** 3 + 1, dtype=ctx.dtype, device="cuda")
    u = [torch.empty(3 * D.shape[0] * b ** 3, dtype=ctx.dtype, device="cuda") for _ in range(2)]
    ctx.nested_projection_stage(b, D, r[1:], u[0], alpha=0.1)
    ctx.nested_projection_stage(b, D, r[1:].clone(), u[1], alpha=0.1)
    assert torch.equal(u[0], u[1])
