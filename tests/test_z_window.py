"""The shifted window along z: which problems take it (the library's own
geometry, on the CPU) and its z pass at every transform length that it can
reach, with and without the symmetry in ky (GPU, against the oracle)."""
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

import lgf_inputs as li
from conftest import ROOT, rel_linf

TOL = {"f64": 1e-12, "f32": 1e-5}
# every length but 4096: the union spans at most 2048 points, so an even length is never above 4096
LENGTHS = (32, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512, 640, 768, 1024, 1280, 1536, 2048, 2560, 3072)


def problem(M, yshift, mirror=False):
    """A body and its flow with M - 1 distinct offsets along z, shifted along x (32
    points for 31 offsets) and, with yshift, along y."""
    b, lt = 8, min(M // 8 - 1, 256)          # blocks of the flow along z (2048 points at most)
    ls = M // 8 - lt                         # and of the body
    zs = sorted({0, ls - 1})
    at = 0 if mirror else lt - ls
    src = [[0, 0, at + z] for z in zs]
    zt = sorted({0, lt // 3, lt - 1})
    tgt = sorted({(x, y, z) for z in zt for x in (0, 2) for y in ((0, 2) if yshift else (0,))})
    rng = np.random.default_rng(M + 2 * yshift + mirror)
    f = rng.uniform(-1, 1, (1, 2, len(src), b ** 3))
    return li.Problem("z", b, np.array(src, np.int32), np.array(tgt, np.int32), f)


def library_geometry(tmp_path, problems, choice=""):
    """(M_x, M_y, M_z, shifted x, y, z) of the plans that the library makes by default, or
    for a choice as a tuning file states it."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    csrc = os.path.join(ROOT, "paper_1604_01814_gb300", "csrc")
    objs = glob.glob(os.path.join(ROOT, "_build", "*.cu.o"))
    srcs = glob.glob(os.path.join(csrc, "*.cu*"))
    if not os.path.exists(nvcc) or len(objs) < len(glob.glob(os.path.join(csrc, "*.cu"))):
        pytest.skip("the library's objects are not built")
    if min(map(os.path.getmtime, objs)) < max(map(os.path.getmtime, srcs)):
        pytest.skip("the library's objects are older than its sources")
    main = tmp_path / "geometry.cu"
    main.write_text(r"""
#include <algorithm>
#include <cstdio>
#include "lgf_internal.cuh"
#include "lgf_tune.h"
int main(int argc, char **argv)
{
    lgf::TuneChoiceText text;
    if (argc > 1 && !lgf::tune_parse_plan_value(argv[1], &text)) return 3;
    int b, ns, nt;
    while (scanf("%d %d %d", &b, &ns, &nt) == 3) {
        lgf::PoissonPlan p;
        p.b = b;
        for (int d = 0; d < 3; ++d) { p.slo[d] = p.tlo[d] = 1 << 30; p.shi[d] = p.thi[d] = -(1 << 30); }
        for (int i = 0; i < ns + nt; ++i)
            for (int d = 0; d < 3; ++d) {
                int v;
                if (scanf("%d", &v) != 1) return 1;
                int *lo = i < ns ? p.slo : p.tlo, *hi = i < ns ? p.shi : p.thi;
                lo[d] = std::min(lo[d], v);
                hi[d] = std::max(hi[d], v);
            }
        lgf::PoissonGeom g{};
        int64_t A, B;
        if (!lgf::poisson_geometry(p, argc > 1 ? lgf::tune_choice(text) : lgf::poisson_default_choice(p, true), &g, &A, &B))
            return 2;
        printf("%d %d %d %d %d %d\n", g.M[0], g.M[1], g.M[2], g.xasym, g.yasym, g.zasym);
    }
}
""")
    exe = tmp_path / "geometry"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "include"), "-I", csrc, "-o", str(exe), str(main), *objs], check=True)
    text = "".join(f"{p.b} {len(p.src)} {len(p.tgt)}\n" + "\n".join(" ".join(map(str, c)) for c in np.concatenate([p.src, p.tgt])) +
                   "\n" for p in problems)
    run = lambda *args: [tuple(map(int, line.split())) for line in
                         subprocess.run([str(exe), *args], input=text, check=True, capture_output=True, text=True).stdout.splitlines()]
    return run(choice) if choice else run()


def test_choices_of_older_files_keep_z_even(tmp_path):
    """A choice written before z had a shifted window was timed with z even and names
    that geometry still; one written now ends with w1."""
    probs = [problem(64, 1), problem(320, 0)]
    new = library_geometry(tmp_path, probs, "x1 y0 bx0 by0 bz0 z0 f0 w1")
    assert [g[2] for g in new] == [64, 320] and all(g[5] for g in new)
    for old in ("x1 y0 bx0 by0 bz0 z0", "x1 y0 bx0 by0 bz0 z0 f0"):
        got = library_geometry(tmp_path, probs, old)
        assert [g[2] for g in got] == [128, 640] and not any(g[5] for g in got)
    assert library_geometry(tmp_path, probs[1:], "x1 y0 bx0 by0 bz1 z0")[0][2] == 768


def test_default_geometry(tmp_path):
    """The problems below take the shifted z window at their length; random sets
    have the geometry that the benchmark states."""
    import bench
    probs = [problem(M, y, m) for M in LENGTHS for y in (0, 1) for m in (False, True)]
    rng = np.random.default_rng(1)
    rnd = []
    for i in range(200):
        se, te = rng.integers(1, 9, 3), rng.integers(1, 25, 3)
        at = rng.integers(-4, 12, 3)
        s, t = li.box_blocks(1, 1, 1), np.array([[0, 0, 0], te - 1], np.int32)
        s = np.array([at, at + se - 1], np.int32)
        rnd.append(li.Problem("r", (4, 8, 16, 32)[i % 4], s, t, np.zeros((1, 1, 2, 1))))
    got = library_geometry(tmp_path, probs + rnd)
    for (M, y), g in zip([(M, y) for M in LENGTHS for y in (0, 1) for _ in range(2)], got):
        assert g == (32, 32, M, 1, y, 1), (M, y, g)
    assert sum(g[5] for g in got[len(probs):]) > 50
    for p, g in zip(rnd, got[len(probs):]):
        assert list(g[:3]) == bench.geometry(p)[0]
        assert g[5] <= (g[3] or g[4])


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("yshift", [0, 1])
@pytest.mark.parametrize("M", LENGTHS)
def test_every_length(M, yshift, prec, ctx64, ctx32, oracle):
    """Sampled targets of a body at either end of its flow."""
    ctx = ctx64 if prec == "f64" else ctx32
    for mirror in (False, True):
        p = problem(M, yshift, mirror)
        f = torch.tensor(p.f.reshape(-1), dtype=ctx.dtype, device="cuda")
        u = torch.full((2 * p.tgt.shape[0] * 512,), float("nan"), dtype=ctx.dtype, device="cuda")
        ctx.poisson_apply(p.b, p.src, p.tgt, f, u, ncomp=2, dx=0.5)
        got = u.cpu().numpy().astype(np.float64).reshape(2, -1)
        assert np.isfinite(got).all()
        idx = np.random.default_rng(M).choice(got.shape[1], size=300, replace=False)
        ref = oracle.poisson_direct_multi(p.b, p.src, p.f[0], oracle.block_points(p.b, p.tgt)[idx], dx=0.5, R=64)
        assert rel_linf(got[:, idx], ref) < TOL[prec]
