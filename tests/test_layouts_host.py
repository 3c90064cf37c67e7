"""How the FP64 and long-line kernels split their work, from the constants they
are compiled with (host programs over the kernel headers, no GPU needed).

FP64 issues two lanes a clock and SM, so what it pays for is warps issued, full
or not, and SMs without work; shared memory is paid in 128-byte wavefronts."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1604_01814_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def run(tmp_path, header, body):
    """Lines of integers that `body` prints."""
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(f'#include <cstdio>\n#include "{header}"\nusing namespace lgf;\n{body}\n')
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [[int(v) for v in line.split()] for line in out.splitlines()]


def test_fp64_xy_items_fill_warps_and_planes_spread(tmp_path):
    """The x+y pass of small FP64 sets: every z-plane (two with blocks of 8) is a
    CTA of its own, and the x and y items of a single block and of a pair are whole
    warps; the wide form only where it is chosen, on larger sets."""
    rows = run(tmp_path, "lgf_intfactor_win.cuh", r"""
template <int LB, int R> void one() {
    using C = win::XYCfg<double, LB, R, false>;
    printf("%d %d %d %d %d %d %d %d %d %d\n", C::b, R, C::NS, C::EY1 * C::GX * C::NS, C::EY * C::GX * C::NS,
           C::b * C::NS * C::GY, C::THREADS, (int)win::xy_wide<double, LB, R>(31), (int)win::xy_wide<double, LB, R>(32),
           (int)win::xy_wide<float, LB, R>(1));
}
template <int LB> void all() { one<LB, 4>(); one<LB, 8>(); one<LB, 12>(); one<LB, 16>(); }
int main() { all<3>(); all<4>(); all<5>(); }""")
    assert len(rows) == 12
    for b, R, ns, x1, x2, y1, threads, small, large, f32 in rows:
        assert ns == (2 if b == 8 else 1)
        assert x1 % 32 == x2 % 32 == y1 % 32 == 0 and threads % 32 == 0
        assert f32 == 1
        assert small == (b == 32 and R == 16)
        assert large == (small or (b == 16 and R >= 12))


def test_z_pass_choice(tmp_path):
    """Which z pass: blocks of 16 stream in FP32, and in FP64 from window 8 on;
    blocks of 32 stream in FP32 only, at windows 4 and 8, on large sets."""
    rows = run(tmp_path, "lgf_intfactor_win.cuh", r"""
template <int LB, int R> void one() {
    printf("%d %d %d %d %d %d\n", 1 << LB, R, (int)win::z_march<float, LB, R>(1), (int)win::z_march<float, LB, R>(192),
           (int)win::z_march<double, LB, R>(1), (int)win::z_march<double, LB, R>(100000));
}
template <int LB> void all() { one<LB, 4>(); one<LB, 8>(); one<LB, 12>(); one<LB, 16>(); }
int main() { all<3>(); all<4>(); all<5>(); }""")
    for b, R, few, many, few64, many64 in rows:
        assert few == (b == 16) and many == (b == 16 or (b == 32 and R <= 8))
        assert few64 == many64 == (b == 16 and R >= 8)


SIZES = (32, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512, 640, 768, 1024, 1280, 1536, 2048, 2560, 3072, 4096)


def _warps(active):
    """Warps with an active lane, of a list of lane flags."""
    return sum(any(active[i:i + 32]) for i in range(0, len(active), 32))


def _idle(threads, lane, groups, tpc):
    """Warps issued over warps' worth of groups: thread i of `threads` is lane(i)
    of its line's tpc, and takes groups lane, lane + tpc, ..."""
    issued = sum(_warps([lane(i) + r < groups for i in range(threads)]) for r in range(0, groups, tpc))
    lines = threads // tpc
    return issued * 32 / (lines * groups)


def test_fp64_x_passes_leave_no_lanes_idle(tmp_path):
    rows = run(tmp_path, "lgf_poisson_kernels.cuh", r"""
template <int M> void one() {
    using P = pk::Plan<M>; using L = pk::RowLay<double, M>;
    printf("%d %d %d %d %d\n", M, L::THREADS, L::TPC, P::G0, P::GL);
}
template <int... M> void all() { (one<M>(), ...); }
int main() { all<""" + ", ".join(map(str, SIZES)) + ">(); }")
    assert len(rows) == len(SIZES)
    for M, threads, tpc, g0, gl in rows:
        lpc = threads // tpc
        first = _idle(threads, lambda i: i % tpc, g0, tpc)      # lanes along the groups of a line
        last = _idle(threads, lambda i: i // lpc, gl, tpc)      # lanes along the lines
        assert first <= 1.2 and last <= 1.0, (M, first, last)
        if M != 80:
            assert first == 1.0, (M, first)


def test_fp64_column_passes_leave_few_lanes_idle(tmp_path):
    """Columns side by side in a warp; the idle part weighted by the stages' radix
    (five flops per point and binary digit)."""
    import math
    rows = run(tmp_path, "lgf_poisson_kernels.cuh", r"""
template <int M> void one() {
    using P = pk::Plan<M>; using C = pk::ColCfg<double, M>;
    printf("%d %d %d %d %d %d %d\n", M, C::W, P::TPC, P::G0, P::GL, P::R0, P::RL);
}
template <int... M> void all() { (one<M>(), ...); }
int main() { all<""" + ", ".join(map(str, SIZES)) + ">(); }")
    for M, w, tpc, g0, gl, r0, rl in rows:
        cost = [math.log2(r0), math.log2(rl)]
        idle = [_idle(w * tpc, lambda i: i // w, g, tpc) for g in (g0, gl)]
        assert sum(c * i for c, i in zip(cost, idle)) / sum(cost) < 1.1, (M, idle)


def test_middle_stage_wavefronts(tmp_path):
    """Shared-memory wavefronts of the column passes' middle stage (FP32, element m
    of column w at m W + w, 16 lanes of 8 bytes): at most a third above the least."""
    rows = run(tmp_path, "lgf_poisson_kernels.cuh", r"""
template <int M> void one() {
    using P = pk::Plan<M>; using C = pk::ColCfg<float, M>;
    if constexpr (P::NST == 3)
        printf("%d %d %d %d %d %d\n", M, C::W, P::TPC, pk::MidSplit<M>::TJ, pk::MidSplit<M>::TS, P::N1);
}
template <int... M> void all() { (one<M>(), ...); }
int main() { all<""" + ", ".join(map(str, SIZES)) + ">(); }")
    assert [r[0] for r in rows] == [m for m in SIZES if m >= 384]
    for M, w, tpc, tj, ts, n1 in rows:
        assert tj * ts == tpc
        waves = least = 0
        for half in range(0, w * tpc, 16):
            words = set()
            for i in range(half, min(half + 16, w * tpc)):
                t = i // w
                words.add(((t // tj) * n1 + t % tj) * w + i % w)
            banks = [v % 16 for v in words]
            waves += max(banks.count(k) for k in set(banks))
            least += 1
        assert waves <= 4 / 3 * least, (M, waves, least)


def test_twiddle_tables_take_one_allocation_and_no_upload(tmp_path):
    """Entry i of a length's table in the order of its stages (the first use of a
    length forms it on the device): w_M^{j q} at (q - 1) G0 + j, then w_{N1}^{j q}."""
    rows = run(tmp_path, "lgf_poisson_kernels.cuh", r"""
template <int M> void one() {
    using P = pk::Plan<M>;
    printf("%d %d %d", M, P::R0, P::R1);
    for (int i = 0; i < M; ++i) printf(" %d", pk::twiddle_exponent(i, M, P::R0, P::R1));
    printf("\n");
}
template <int... M> void all() { (one<M>(), ...); }
int main() { all<""" + ", ".join(map(str, SIZES)) + ">(); }")
    for M, r0, r1, *e in rows:
        g0, rl = M // r0, M // r0 // r1
        want = [j * q for q in range(1, r0) for j in range(g0)] + [j * q * r0 for q in range(1, r1) for j in range(rl)]
        assert e == want + [0] * (M - len(want)), M
    text = open(os.path.join(CSRC, "lgf_poisson.cu")).read()
    body = text[text.index("const void *twiddles("):]
    body = body[:body.index("\n}\n")]
    assert body.count("cudaMalloc(") == 1 and "cudaMemcpy" not in body
