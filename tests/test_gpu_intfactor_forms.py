"""The integrating factor's passes have more than one form; which one a launch
takes depends on the block edge, the radius class, the precision and the
number of blocks and fields.  Fields are independent and every form adds in the same
order, so a call of many fields equals the calls of one field each bit for
bit, also where the two lie on different sides of a rule."""
import numpy as np
import pytest
import torch

import lgf_inputs as li
import paper_1604_01814_gb300 as lgf
from conftest import build_lib, rel_linf

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-12, "f32": 1e-5}
# one alpha per radius class (4, 8, 12, 16) at the contexts' truncation tolerance
ALPHAS = {"f32": {4: 0.02, 8: 0.3, 12: 1.0, 16: 2.0}, "f64": {4: 1e-4, 8: 0.05, 12: 0.25, 16: 0.75}}


def _class(ctx, alpha):
    R, _ = ctx.intfactor_weights(alpha)
    return next(c for c in (4, 8, 12, 16) if R <= c)


# FP32, blocks of 32: the z pass changes at 192 blocks and fields (windows 4 and 8);
# FP64, blocks of 16: the x+y pass at 32 blocks or pairs and fields (windows 12 and 16)
@pytest.mark.parametrize("prec,b,extent,nf,cls", [("f32", 32, (5, 5, 4), 2, 4), ("f32", 32, (5, 5, 4), 2, 8),
                                                  ("f64", 16, (2, 2, 2), 9, 12), ("f64", 16, (2, 2, 2), 9, 16),
                                                  ("f64", 16, (3, 1, 1), 16, 12), ("f64", 16, (3, 1, 1), 16, 16)])
def test_forms_agree(ctx32, ctx64, prec, b, extent, nf, cls):
    ctx = ctx64 if prec == "f64" else ctx32
    alpha, c = ALPHAS[prec][cls], li.box_blocks(*extent)
    assert _class(ctx, alpha) == cls
    f = torch.randn(nf, c.shape[0] * b ** 3, dtype=ctx.dtype, device="cuda")
    u, one = torch.full_like(f, float("nan")), torch.full_like(f, float("nan"))
    ctx.intfactor_apply(alpha, b, c, c, f, u, ncomp=nf)
    for k in range(nf):
        ctx.intfactor_apply(alpha, b, c, c, f[k], one[k])
    assert torch.equal(u, one)


@pytest.mark.parametrize("cls", [4, 8, 12, 16])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_forms_agree_in_one_launch_of_several_sets(prec, cls):
    """The ragged launches choose over all their jobs: 12 sets of blocks of 16
    together against each alone."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build_lib()
    ctx = lgf.Context(prec, flags=lgf._binding.LGF_FLAG_BATCH_RAGGED)
    b, alpha, probs = 16, ALPHAS[prec][cls], []
    for k in range(12):
        c = li.box_blocks(1 + k % 3, 1 + k % 4, 1 + k % 2)
        f = torch.randn(c.shape[0] * b ** 3, dtype=ctx.dtype, device="cuda")
        probs.append(dict(b=b, src=c, tgt=c, f=f, u=torch.full_like(f, float("nan")), op=lgf.LGF_OP_INTFACTOR,
                          alpha=alpha))
    ctx.batch_apply(probs)
    for p in probs:
        one = torch.full_like(p["f"], float("nan"))
        ctx.intfactor_apply(alpha, b, p["src"], p["tgt"], p["f"], one)
        assert torch.equal(p["u"], one)
    torch.cuda.synchronize()
    ctx.close()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("b,extent", [(8, (4, 4, 3)), (16, (1, 4, 1)), (16, (1, 1, 3)), (32, (1, 3, 1)), (32, (1, 1, 3))])
def test_every_window_class_reached(ctx32, ctx64, oracle, prec, b, extent):
    """Every radius class on a box and on columns of blocks in y and in z, sources on
    every other block, every point against the oracle (no result is zero)."""
    ctx = ctx64 if prec == "f64" else ctx32
    t = li.box_blocks(*extent)
    s = np.ascontiguousarray(t[::2])
    f = np.random.default_rng(b).uniform(-1, 1, (s.shape[0], b ** 3))
    fd = torch.tensor(f.reshape(-1), dtype=ctx.dtype, device="cuda")
    seen = set()
    for alpha in ALPHAS[prec].values():
        seen.add(_class(ctx, alpha))
        u = torch.full((t.shape[0] * b ** 3,), float("nan"), dtype=ctx.dtype, device="cuda")
        ctx.intfactor_apply(alpha, b, s, t, fd, u)
        ref = oracle.intfactor_blocks(alpha, b, s, f, t).reshape(t.shape[0], -1)
        assert np.abs(ref[::2]).max(axis=1).min() > 0
        assert rel_linf(u.cpu().numpy(), ref) < TOL[prec], alpha
    assert seen == {4, 8, 12, 16}
