// Pass kernels of the Poisson apply, specialised on the transform length.
//
// Every length M = 2^k, 3 * 2^k or 5 * 2^k (32..4096) has a fixed plan of two
// or three DIF stages (radix <= 20), see Plan below.  A line (a column of W adjacent kx
// values, or one packed pair of x rows) is handled by TPC threads:
//   - the first forward stage loads its operands straight from global memory
//     into registers (all loads of a thread in flight together), does the
//     butterflies and writes the stage result to shared memory;
//   - the middle stage (three-stage plans only) works in shared memory;
//   - the last forward stage reads shared memory into registers; its outputs
//     are final spectrum values, stored straight to global memory (y pass) or
//     multiplied by the kernel spectrum and sent straight into the first
//     inverse stage (z pass).
// The inverse sweep mirrors this (adjoint stages, conjugate twiddles).  One
// shared-memory transpose per stage boundary, one __syncthreads per boundary.
#pragma once
#include <type_traits>

#include "lgf_internal.cuh"

namespace lgf {
namespace pk {

constexpr int cgcd(int a, int b) { return b == 0 ? a : cgcd(b, a % b); }

// Stage plan of a length M (2^k, 3 * 2^k or 5 * 2^k, 32..4096): a first stage
// of radix R0, for M >= 384 a middle stage of radix R1 (R0, R1 powers of two),
// and a last stage of even radix RL.  Every stage before the last splits off
// a power of two, so its twiddle index stays j q M/N with M/N a power of two.
// TPC threads share a line.  In the three-stage plans it is the greatest common
// divisor of the stages' group counts, so that every thread owns a whole number of
// groups in every stage; the two-stage plans have one group per thread in the
// longer stage, and the threads past the shorter stage's groups (whole warps,
// as lanes run along columns) sit it out.  (Length 32 keeps the divisor, 4: its threads own
// whole groups of both stages.)
// Lengths 96, 192 and 320 had three stages (4 x 2 x 12, 4 x 4 x 12, 4 x 4 x 20), 80 and
// 160 a radix of 20: with two stages half the shared-memory passes and barriers go,
// and more of the butterflies are packed.  z pass at length 320 (refresh of 556 blocks)
// 315 -> 297 us, the refresh 660 -> 631 us, the 64-plate batch 3.96 -> 3.89 ms.
template <int ML>
struct Plan {
    static constexpr int M = ML;
    static constexpr int R0 = M == 32 || M == 64 || M == 80 || M == 96 || M == 384 || M == 512 || M == 640 || M == 768 ||
                                      M == 1280
                                  ? 8
                                  : 16;
    static constexpr int R1 = M == 384 || M == 640 ? 4
                            : M == 512 || M == 768 || M == 1024 || M == 1280 || M == 1536 || M == 2560 ? 8
                            : M == 2048 || M == 3072 || M == 4096 ? 16 : 1;
    static constexpr int RL = M / (R0 * R1);
    static constexpr int NST = R1 > 1 ? 3 : 2;
    static constexpr int N1 = M / R0;                             // sub-problem size entering stage 1
    static constexpr int G0 = M / R0, G1 = M / R1, GL = M / RL;   // groups per stage
    static constexpr int TPC = NST == 3 ? cgcd(cgcd(G0, G1), GL)
                             : cgcd(G0, GL) <= 4 && M != 32 ? (G0 > GL ? G0 : GL)
                                                                         : cgcd(G0, GL);
    static constexpr int NG0 = (G0 + TPC - 1) / TPC, NGL = (GL + TPC - 1) / TPC;   // rounds of groups
    static constexpr bool MASK0 = G0 % TPC != 0, MASKL = GL % TPC != 0;            // the last round is partial
    static constexpr int TW1 = (R0 - 1) * G0;                     // first twiddle of the middle stage
    static_assert(R0 * R1 * RL == M && RL <= 20 && RL >= 4 && RL % 2 == 0, "plan must cover the length");
    static_assert(NST == 2 || (G0 % TPC == 0 && G1 % TPC == 0 && GL % TPC == 0), "whole groups per thread");
};

// Position of frequency k after the forward sweep, and back: position
// q0 M/R0 + q1 RL + qL holds frequency q0 + R0 q1 + R0 R1 qL.
template <int ML>
__device__ __forceinline__ int pos_of(int k)
{
    using P = Plan<ML>;
    const int q0 = k % P::R0;
    k /= P::R0;
    const int q1 = k % P::R1;
    const int qL = k / P::R1;
    return q0 * (ML / P::R0) + q1 * P::RL + qL;
}

// The column passes are bound by instruction issue (76 % of the slots of the z
// pass at length 320), and more than a quarter of their instructions were index
// arithmetic: twiddles gathered at j q M/N from one natural-order table, a division
// per middle-stage group, 64-bit offsets formed per access.  Tables in the order
// of the stages, a middle stage that splits each line as sub-problems times groups
// and pointers that walk took the refresh of 556 blocks (x 640, y and z 320) from
// 826 to 730 us, the 64-plate batch from 4.85 to 4.42 ms and the 512x256x256 wake
// from 7.39 to 6.90 ms, every output bit the same; the x passes also lost the bank
// conflicts of the gathered twiddles.
// Exponent e of entry i of a length's twiddle table (the entry is
// exp(-2 pi i e / M)): the first stage's w_M^{j q} at (q - 1) G0 + j, then the
// middle stage's w_{N1}^{j q} = w_M^{j q R0} at TW1 + (q - 1) RL + j; 0 past them.
__host__ __device__ inline int twiddle_exponent(int i, int M, int R0, int R1)
{
    const int G0 = M / R0, RL = G0 / R1, TW1 = (R0 - 1) * G0;
    if (i < TW1) return (i % G0) * (i / G0 + 1);
    i -= TW1;
    return i < (R1 - 1) * RL ? (i % RL) * (i / RL + 1) * R0 : 0;   // (none with R1 = 1)
}

template <int ML>
__device__ __forceinline__ int freq_of(int pos)
{
    using P = Plan<ML>;
    const int q0 = pos / (ML / P::R0);
    const int r0 = pos % (ML / P::R0);
    return q0 + P::R0 * (r0 / P::RL) + P::R0 * P::R1 * (r0 % P::RL);
}

// Forward butterfly of one group of a stage that is not the last: DFT then
// the twiddles w_N^{j q}, which the table holds at tw[(q - 1) J + j] for the
// stage's J groups (see twiddle_exponent), so that one address per thread
// and constant offsets reach all of them.  HALF: the inputs a[R/2..R) are zero
// (not read).
template <int R, int J, bool HALF = false, typename T>
__device__ __forceinline__ void dif_group(Cx<T> *a, int j, const Cx<T> *tw)
{
    if constexpr (HALF)
        dft_half_in<R, -1, T>(a);
    else
        Dft<R, -1, T>::run(a);
#pragma unroll
    for (int q = 1; q < R; ++q) a[q] = cmul(a[q], tw[(q - 1) * J + j]);
}

// A group whose only nonzero input is a[0] (the data of the line end before
// M/R): the DFT gives a[0] at every output, so the stage is the twiddles.
template <int R, int J, typename T>
__device__ __forceinline__ void dif_group_single(Cx<T> *a, int j, const Cx<T> *tw)
{
#pragma unroll
    for (int q = 1; q < R; ++q) a[q] = cmul(a[0], tw[(q - 1) * J + j]);
}

// Its adjoint.  HALF: only the outputs a[0..R/2) are formed.
template <int R, int J, bool HALF = false, typename T>
__device__ __forceinline__ void dit_group(Cx<T> *a, int j, const Cx<T> *tw)
{
#pragma unroll
    for (int q = 1; q < R; ++q) a[q] = cmulc(a[q], tw[(q - 1) * J + j]);
    if constexpr (HALF)
        dft_half_out<R, 1, T>(a);
    else
        Dft<R, 1, T>::run(a);
}

// Middle stage (three-stage plans): shared memory to shared memory.  The
// threads of a line split as TJ groups times TS sub-problems, so that every
// group's address is the thread's own plus a constant.
template <int ML>
struct MidSplit {
    using P = Plan<ML>;
    // Consecutive threads take consecutive groups, which are neighbours in shared
    // memory; sub-problems are a multiple of all banks apart.  With the
    // sub-problems along the threads the 11 threads of a warp at length 4096 (three
    // columns) met on the same banks: z pass of 64x64x2048 points 450 us (373 before that
    // split, 325 now), y passes of 32x1024x512 264 and 217 (249 and 207; 251 and 202 now);
    // at 512 (1024x512x512, 12 fields) z 7.2 -> 6.3 ms.
    static constexpr int TJ = cgcd(P::TPC, P::RL), TS = P::TPC / TJ;
    static_assert(P::NST == 2 || (P::R0 % TS == 0 && P::RL % TJ == 0), "whole groups per thread");
};
template <int ML, int DIR, typename T, class Addr>
__device__ __forceinline__ void middle_stage(Cx<T> *s, const Addr &ad, int line, int t, const Cx<T> *tw)
{
    using P = Plan<ML>;
    if constexpr (P::NST == 3) {
        constexpr int N = P::N1, R = P::R1, NP = N / R;
        constexpr int TS = MidSplit<ML>::TS, TJ = MidSplit<ML>::TJ;
        const int j0 = t % TJ;
        const Cx<T> *tw1 = tw + P::TW1 + j0;
        const int o = (t / TJ) * N + j0;
#pragma unroll
        for (int sub = 0; sub < P::R0; sub += TS) {
#pragma unroll
            for (int j = 0; j < NP; j += TJ) {
                Cx<T> a[R];
                if (DIR < 0) {
#pragma unroll
                    for (int p = 0; p < R; ++p) a[p] = s[ad(line, o + sub * N + j + p * NP)];
                    dif_group<R, NP>(a, j, tw1);
#pragma unroll
                    for (int q = 0; q < R; ++q) s[ad(line, o + sub * N + q * NP + j)] = a[q];
                } else {
#pragma unroll
                    for (int q = 0; q < R; ++q) a[q] = s[ad(line, o + sub * N + q * NP + j)];
                    dit_group<R, NP>(a, j, tw1);
#pragma unroll
                    for (int p = 0; p < R; ++p) s[ad(line, o + sub * N + j + p * NP)] = a[p];
                }
            }
        }
    }
}

// Shared-memory layouts.
struct ColAddrW {   // element m of column w: m * W + w
    int W;
    __device__ __forceinline__ int operator()(int w, int m) const { return m * W + w; }
};
// The twiddles, which no pass writes, may be fetched while the previous pass still
// runs; everything else waits for it (chain_wait).  A, B, f and u, which the passes
// hand on, are therefore plain pointers in every body and kernel that may be
// chained: const with __restrict__, or __restrict__ alone, promises that nobody
// else writes them while the kernel runs, and a load under that promise may use the
// read-only path or move ahead of chain_wait, when the previous pass still writes.
// (The f of the x forward pass is not handed on by a pass, and that kernel is
// never chained.)
template <typename T>
__device__ __forceinline__ void load_twiddles(Cx<T> *tw, const Cx<T> *__restrict__ twg, int M)
{
    for (int i = threadIdx.x; i < M; i += blockDim.x) tw[i] = twg[i];
    chain_wait();
}

// ---------------------------------------------------------------------------
// Column passes.  Data in global memory: rows of K complex values (kx), row
// `r` of the current column set at base + r * rs.  Most CTAs own W adjacent
// kx of one plane; the K mod W leftover kx of every plane (the Nyquist column
// kx = M/2 when K = M/2 + 1) are packed W (plane, kx) pairs per CTA, so no
// CTA runs mostly empty columns.  Those CTAs come first in the grid: their
// scattered accesses are slower, and they then overlap the rest instead of
// trailing it.
// ---------------------------------------------------------------------------
// Row-block occupancy for the y-forward pass: row y of plane pl (both
// relative to the source region) holds data unless its (z, y) row block has
// no block along x (the x-forward pass then skipped it); bit y >> lb of
// mask[pl >> lb].
struct RowFlags {
    const unsigned long long *mask = nullptr;   // nullptr: every row holds data
    int lb = 0;
    __device__ __forceinline__ unsigned long long plane(int pl) const { return mask ? mask[pl >> lb] : ~0ull; }
    // only with a mask: every region then has at most 64 row blocks, so the
    // shift stays below 64
    __device__ __forceinline__ bool row(unsigned long long pm, int y) const { return (pm >> (y >> lb)) & 1ull; }
};

template <int W>
__host__ __device__ __forceinline__ int col_ctas(int K, int nplanes)
{
    const int nfull = K / W, rem = K - nfull * W;
    return nfull * nplanes + (rem * nplanes + W - 1) / W;
}

// Column (kx, plane) of lane w of CTA `cta`; false for padding lanes of the
// last packed CTA (kx, plane set to 0 so that addresses stay in range).
template <int W>
__device__ __forceinline__ bool column_of(int cta, int w, int K, int nplanes, int &kx, int &pl)
{
    const int nfull = K / W, rem = K - nfull * W;
    const int ntail = (rem * nplanes + W - 1) / W;
    if (cta >= ntail) {
        const int c = cta - ntail;
        pl = c / nfull;
        kx = (c - pl * nfull) * W + w;
        return true;
    }
    const int i = cta * W + w;
    pl = i / rem;
    kx = nfull * W + (i - pl * rem);
    if (pl < nplanes) return true;
    pl = 0;
    kx = 0;
    return false;
}

// Forward along the column: rows [lo, lo + n) hold data (row m at
// in + (m - lo) * rs), others are zero; the spectrum (natural order) goes to
// out + k * os.  Used by the y pass and by the spectrum build's z pass.
// HALF: the data rows lie in [0, M/2), which holds for every pass of an
// apply (the transform length is at least twice the box), so the first
// stage's upper inputs are zero at compile time and its first butterfly
// layer is skipped.  Row addresses advance by a fixed stride per radix digit
// (the last stage's digit is the top digit of the frequency).
// (The body of every pass kernel takes its CTA coordinates as arguments: the
// kernels below run it at their own blockIdx, the ragged kernels at the
// coordinates of a CTA inside one job of a job table.)
template <typename T, int ML, int W, bool HALF>
__device__ __forceinline__ void col_forward_body(int bx, int by, const Cx<T> *in, Cx<T> *out,
                                                 int K, int nplanes, int lo, int n, int64_t rs, int64_t os,
                                                 int64_t in_plane, int64_t out_plane, int64_t in_field,
                                                 int64_t out_field, const Cx<T> *__restrict__ twg, RowFlags rf)
{
    using P = Plan<ML>;
    constexpr int M = P::M;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *tw = reinterpret_cast<Cx<T> *>(smem_raw);
    Cx<T> *s = tw + M;
    load_twiddles(tw, twg, M);
    const int w = threadIdx.x % W, t = threadIdx.x / W;
    int kx, pl;
    const bool live = column_of<W>(bx, w, K, nplanes, kx, pl);
    const Cx<T> *ib = in + by * in_field + pl * in_plane + kx;
    Cx<T> *ob = out + by * out_field + pl * out_plane + kx;
    const ColAddrW ad{W};
    constexpr int R0 = P::R0;
    constexpr int NG0 = P::NG0;
    constexpr int NP = HALF ? R0 / 2 : R0;
    const int64_t istep = (int64_t)P::G0 * rs;
    Cx<T> a[NG0][R0];
    if (rf.mask == nullptr) {   // every row holds data (uniform branch)
#pragma unroll
        for (int i = 0; i < NG0; ++i) {
            const int r = t + i * P::TPC - lo;   // data row of digit p = 0
            const Cx<T> *src = ib + (int64_t)r * rs;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const bool ok = live && (unsigned)(r + p * P::G0) < (unsigned)n && (!P::MASK0 || t + i * P::TPC < P::G0);
                a[i][p] = ok ? *src : Cx<T>{T(0), T(0)};
                src += istep;
            }
        }
    } else {
        const unsigned long long pm = rf.plane(pl);
#pragma unroll
        for (int i = 0; i < NG0; ++i) {
            const int r = t + i * P::TPC - lo;
            const Cx<T> *src = ib + (int64_t)r * rs;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const int y = r + p * P::G0;
                const bool ok =
                    live && (unsigned)y < (unsigned)n && rf.row(pm, y) && (!P::MASK0 || t + i * P::TPC < P::G0);
                a[i][p] = ok ? *src : Cx<T>{T(0), T(0)};
                src += istep;
            }
        }
    }
    __syncthreads();   // twiddles
#pragma unroll
    for (int i = 0; i < NG0; ++i) {
        const int g = t + i * P::TPC;
        if (P::MASK0 && g >= P::G0) break;
        dif_group<P::R0, P::G0, HALF>(a[i], g, tw);
#pragma unroll
        for (int q = 0; q < R0; ++q) s[ad(w, q * P::G0 + g)] = a[i][q];
    }
    __syncthreads();
    if constexpr (P::NST == 3) {
        middle_stage<ML, -1>(s, ad, w, t, tw);
        __syncthreads();
    }
    constexpr int RL = P::RL;
    const int64_t ostep = (int64_t)(M / RL) * os;
#pragma unroll
    for (int g = t; g < P::GL; g += P::TPC) {
        Cx<T> c[RL];
#pragma unroll
        for (int q = 0; q < RL; ++q) c[q] = s[ad(w, (g * P::RL) + q)];
        Dft<RL, -1, T>::run(c);
        if (live) {
            Cx<T> *dst = ob + (int64_t)freq_of<ML>(g * P::RL) * os;
#pragma unroll
            for (int q = 0; q < RL; ++q) {
                *dst = c[q];
                dst += ostep;
            }
        }
    }
}

template <typename T, int ML, int W, bool HALF>
__global__ void __launch_bounds__(W * Plan<ML>::TPC) k_col_forward(const Cx<T> *in, Cx<T> *out,
                                                                     int K, int nplanes, int lo, int n, int64_t rs,
                                                                     int64_t os, int64_t in_plane, int64_t out_plane,
                                                                     int64_t in_field, int64_t out_field,
                                                                     const Cx<T> *__restrict__ twg, RowFlags rf)
{
    col_forward_body<T, ML, W, HALF>(blockIdx.x, blockIdx.y, in, out, K, nplanes, lo, n, rs, os, in_plane, out_plane,
                                     in_field, out_field, twg, rf);
}

// Inverse along the column: spectrum rows (natural order, row k at
// in + k * rs) in; rows [lo, lo + n) of the result written to
// out + (m - lo) * os.  HALF_OUT: the written rows lie in [0, M/2), so the
// last stage forms only the lower half of its outputs (otherwise, the
// shifted y window with targets past M/2, all of them).
template <typename T, int ML, int W, bool HALF_OUT>
__device__ __forceinline__ void col_inverse_body(int bx, int by, const Cx<T> *in, Cx<T> *out,
                                                 int K, int nplanes, int lo, int n, int64_t rs, int64_t os,
                                                 int64_t in_plane, int64_t out_plane, int64_t in_field,
                                                 int64_t out_field, const Cx<T> *__restrict__ twg)
{
    using P = Plan<ML>;
    constexpr int M = P::M;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *tw = reinterpret_cast<Cx<T> *>(smem_raw);
    Cx<T> *s = tw + M;
    load_twiddles(tw, twg, M);
    const int w = threadIdx.x % W, t = threadIdx.x / W;
    int kx, pl;
    const bool live = column_of<W>(bx, w, K, nplanes, kx, pl);
    const Cx<T> *ib = in + by * in_field + pl * in_plane + kx;
    Cx<T> *ob = out + by * out_field + pl * out_plane + kx;
    const ColAddrW ad{W};
    constexpr int RL = P::RL;
    constexpr int NGL = P::NGL;
    const int64_t istep = (int64_t)(M / RL) * rs;
    Cx<T> c[NGL][RL];
#pragma unroll
    for (int i = 0; i < NGL; ++i) {
        const int g = t + i * P::TPC;
        if (P::MASKL && g >= P::GL) break;
        const Cx<T> *src = ib + (int64_t)freq_of<ML>(g * P::RL) * rs;
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            c[i][q] = live ? *src : Cx<T>{T(0), T(0)};
            src += istep;
        }
    }
#pragma unroll
    for (int i = 0; i < NGL; ++i) {
        const int g = t + i * P::TPC;
        if (P::MASKL && g >= P::GL) break;
        Dft<RL, 1, T>::run(c[i]);
#pragma unroll
        for (int q = 0; q < RL; ++q) s[ad(w, (g * P::RL) + q)] = c[i][q];
    }
    __syncthreads();
    if constexpr (P::NST == 3) {
        middle_stage<ML, 1>(s, ad, w, t, tw);
        __syncthreads();
    }
    constexpr int R0 = P::R0;
    constexpr int NOUT = HALF_OUT ? R0 / 2 : R0;
    const int64_t ostep = (int64_t)P::G0 * os;
#pragma unroll
    for (int g = t; g < P::G0; g += P::TPC) {
        Cx<T> a[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) a[q] = s[ad(w, q * P::G0 + g)];
        dit_group<P::R0, P::G0, HALF_OUT>(a, g, tw);
        if (live) {
            const int r = g - lo;
            Cx<T> *dst = ob + (int64_t)r * os;
#pragma unroll
            for (int p = 0; p < NOUT; ++p) {
                if ((unsigned)(r + p * P::G0) < (unsigned)n) *dst = a[p];
                dst += ostep;
            }
        }
    }
}

template <typename T, int ML, int W, bool HALF_OUT>
__global__ void __launch_bounds__(W * Plan<ML>::TPC) k_col_inverse(const Cx<T> *in, Cx<T> *out,
                                                                     int K, int nplanes, int lo, int n, int64_t rs,
                                                                     int64_t os, int64_t in_plane, int64_t out_plane,
                                                                     int64_t in_field, int64_t out_field,
                                                                     const Cx<T> *__restrict__ twg)
{
    col_inverse_body<T, ML, W, HALF_OUT>(blockIdx.x, blockIdx.y, in, out, K, nplanes, lo, n, rs, os, in_plane,
                                         out_plane, in_field, out_field, twg);
}

// z pass: forward along z over the source planes, times the real even kernel
// spectrum, inverse along z, target planes written back in place.  The field
// is the fastest part of the CTA index, so the CTAs of every field of one
// column set run back to back and read that part of the spectrum from L2:
// for big boxes the spectrum is larger than L2.  Source and target planes
// lie in [0, M/2): the first stage skips its zero upper inputs and the last
// stage forms only its lower outputs.
// Resident CTAs per SM that the register allocation must allow (FP32): four of
// 256 threads up to length 256 (64 registers; the 64-plate batch 3.88 -> 3.82 ms against
// the compiler's own choice below 160), five of 160 at 320, three at 384 and 512, two
// at the long mixed lengths (no spills beyond a few bytes).
// ZV = 1 (the tuner's alternative, FP32 only) asks for one more resident CTA
// per SM than the default, i.e. a tighter register cap (where the default
// leaves the choice to the compiler, 3).
template <typename T, int ML, int ZV = 0>
struct ConvOcc {
    static constexpr int base = sizeof(T) == 4 ? (ML <= 256 ? 4 : ML == 320 ? 5 : ML == 384 || ML == 512 ? 3 : ML == 640 || ML == 1536 || ML == 2560 || ML == 3072 ? 2 : 1) : 1;
    static constexpr int value = ZV == 0 ? base : (base == 1 ? 3 : base + 1);
};

// SPEC: 0 the real spectrum of the even embedding ([kz][ky <= My/2][kx]);
// 1 the complex spectrum of the shifted x window (same layout); 2 the complex
// spectrum of the shifted y window ([kz][ky < My][kx], no mirror in ky); 3 that of the
// shifted z window ([kz < Mz], ky <= My/2 where y is even (ysym), else all), whose
// target planes reach past M/2, so that the last stage forms all its outputs.  A
// shifted z pays where the targets outreach the sources, a body and its flow: 192
// points instead of 256 along z of the sphere set, whose Poisson apply went from 152.0
// to 145.9 us in FP32 and from 3.53 to 3.05 ms in FP64.
template <typename T, int ML, int W, int SPEC>
__device__ __forceinline__ void col_convolve_body(int bx, int nf, Cx<T> *B, const void *__restrict__ specv,
                                                  int K, int ld, int lds, int My, int ysym, int s0, int ns, int t0,
                                                  int nt, int64_t field, const Cx<T> *__restrict__ twg)
{
    constexpr bool CPLX = SPEC > 0;
    using SpecT = typename std::conditional<CPLX, Cx<T>, T>::type;
    const SpecT *__restrict__ spec = reinterpret_cast<const SpecT *>(specv);
    using P = Plan<ML>;
    constexpr int M = P::M;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *tw = reinterpret_cast<Cx<T> *>(smem_raw);
    Cx<T> *s = tw + M;
    load_twiddles(tw, twg, M);
    const int w = threadIdx.x % W, t = threadIdx.x / W;
    int kx, ky;
    const int field_i = bx % nf;
    const bool live = column_of<W>(bx / nf, w, K, My, kx, ky);
    const int64_t plane = (int64_t)My * ld;
    Cx<T> *bb = B + field_i * field + (int64_t)ky * ld + kx;
    const ColAddrW ad{W};
    constexpr int R0 = P::R0;
    constexpr int NG0 = P::NG0;
    const int64_t step0 = (int64_t)P::G0 * plane;
    {
        Cx<T> a[NG0][R0];
#pragma unroll
        for (int i = 0; i < NG0; ++i) {
            const int r = t + i * P::TPC - s0;
            const Cx<T> *src = bb + (int64_t)r * plane;
#pragma unroll
            for (int p = 0; p < R0 / 2; ++p) {
                const bool ok = live && (unsigned)(r + p * P::G0) < (unsigned)ns && (!P::MASK0 || t + i * P::TPC < P::G0);
                a[i][p] = ok ? *src : Cx<T>{T(0), T(0)};
                src += step0;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NG0; ++i) {
            const int g = t + i * P::TPC;
            if (P::MASK0 && g >= P::G0) break;
            dif_group<P::R0, P::G0, true>(a[i], g, tw);
#pragma unroll
            for (int q = 0; q < R0; ++q) s[ad(w, q * P::G0 + g)] = a[i][q];
        }
    }
    __syncthreads();
    if constexpr (P::NST == 3) {
        middle_stage<ML, -1>(s, ad, w, t, tw);
        __syncthreads();
    }
    constexpr int RL = P::RL;
    constexpr int S = M / RL;   // frequency step of the last stage's digit
    const bool yfull = SPEC == 2 || (SPEC == 3 && !ysym);
    const int Khy = yfull ? My : My / 2 + 1;
    const int kyr = yfull ? ky : (ky <= My - ky ? ky : My - ky);
    const SpecT *sp = spec + (int64_t)kyr * lds + kx;
    const int64_t sp_plane = (int64_t)Khy * lds, sp_step = S * sp_plane;
#pragma unroll
    for (int g = t; g < P::GL; g += P::TPC) {
        // frequency of digit q: kb + q S; its mirror M - kb - q S once past M/2
        const int kb = freq_of<ML>(g * P::RL);
        const SpecT *spl = sp + (int64_t)kb * sp_plane;
        const SpecT *sph = sp + (int64_t)(M - kb - (RL / 2) * S) * sp_plane;
        Cx<T> c[RL];
        SpecT gk[RL];
        if constexpr (SPEC == 3) {   // no mirror in kz
#pragma unroll
            for (int q = 0; q < RL; ++q) {
                gk[q] = *spl;
                spl += sp_step;
            }
        } else {
#pragma unroll
            for (int q = 0; q < RL / 2; ++q) {
                gk[q] = *spl;
                gk[RL / 2 + q] = *sph;
                spl += sp_step;
                sph -= sp_step;
            }
        }
#pragma unroll
        for (int q = 0; q < RL; ++q) c[q] = s[ad(w, (g * P::RL) + q)];
        Dft<RL, -1, T>::run(c);
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            if constexpr (CPLX) {
                c[q] = cmul(c[q], gk[q]);
            } else {
                c[q].x *= gk[q];
                c[q].y *= gk[q];
            }
        }
        Dft<RL, 1, T>::run(c);
#pragma unroll
        for (int q = 0; q < RL; ++q) s[ad(w, (g * P::RL) + q)] = c[q];
    }
    __syncthreads();
    if constexpr (P::NST == 3) {
        middle_stage<ML, 1>(s, ad, w, t, tw);
        __syncthreads();
    }
    const int64_t step1 = (int64_t)P::G0 * plane;
#pragma unroll
    for (int g = t; g < P::G0; g += P::TPC) {
        Cx<T> a[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) a[q] = s[ad(w, q * P::G0 + g)];
        dit_group<P::R0, P::G0, SPEC != 3>(a, g, tw);
        if (live) {
            const int r = g - t0;
            Cx<T> *dst = bb + (int64_t)r * plane;
#pragma unroll
            for (int p = 0; p < (SPEC == 3 ? R0 : R0 / 2); ++p) {
                if ((unsigned)(r + p * P::G0) < (unsigned)nt) *dst = a[p];
                dst += step1;
            }
        }
    }
}

template <typename T, int ML, int W, int SPEC, int ZV>
__global__ void __launch_bounds__(W * Plan<ML>::TPC, ConvOcc<T, ML, ZV>::value) k_col_convolve(Cx<T> *B, const void *__restrict__ specv,
                                                                      int K, int ld, int lds, int My, int ysym, int s0,
                                                                      int ns, int t0, int nt, int64_t field,
                                                                      const Cx<T> *__restrict__ twg)
{
    col_convolve_body<T, ML, W, SPEC>(blockIdx.x, gridDim.x / col_ctas<W>(K, My), B, specv, K, ld, lds, My, ysym, s0, ns,
                                      t0, nt, field, twg);
}

// ---------------------------------------------------------------------------
// Row passes along x (real <-> half complex), two real rows per complex line.
// ---------------------------------------------------------------------------
// Layout and thread split of the x passes.  LPC lines (packed row pairs) share
// a CTA and a line's M values are strided over shared memory: value r of
// sub-problem q0 (position q0 N1 + r) of line l at base(q0) + r LD + l, LD odd.
// Three access patterns have to be free of bank conflicts (16 lanes of 8 bytes):
//   - the middle and last stages, lanes on consecutive lines, then on
//     consecutive sub-problems: 16 lines are contiguous; with 8 or 4 lines,
//     base() steps by LPC modulo 16 over the next 2 or 4 sub-problems;
//   - the first stage, lanes on consecutive groups (so that the global accesses
//     of the same thread are contiguous along x): stride LD, odd;
//   - the pass over the half spectrum, lanes on consecutive frequencies k =
//     q0 + R0 q1 + R0 R1 qL: base(q0) congruent to C1 (q0 mod 2^SH) +
//     C2 (q0 >> SH) modulo 16, chosen per plan so that 16 consecutive k fall on
//     16 different banks.
// Every address is a thread constant plus a compile-time offset.
// The passes are bound by shared-memory wavefronts and latency.  With every line
// contiguous (padded or swizzled per length) and its threads side by side, 62 %
// of the x inverse's wavefronts at length 640 were conflicts and it fetched
// every half spectrum twice (for k and M - k): refresh of 556 blocks (length 640)
// x inverse 101 -> 66 us, x forward 68 -> 53; 64-plate batch 797 -> 672 and 384 ->
// 346 us; 512x256x256 wake (length 1024) x inverse 762 -> 656 us, x forward 634 -> 648.
constexpr int congruent(int v, int c) { return v + (((c - v) % 16) + 16) % 16; }   // smallest >= v equal to c mod 16

template <typename T, int ML>
struct RowLay {
    using P = Plan<ML>;
    // threads per line: 8 to 48 values each; TPC is a multiple of R0 in the
    // three-stage plans.  Where TPC does not divide the first stage's groups, the
    // lanes past them are idle in the last round: free in FP32, but FP64 issues a
    // warp over 16 cycles whatever its lanes do, so it takes the counts that leave
    // none idle (x forward, 3 fields of 96 x 96 lines: length 192 145 -> 130 us, 160 162 -> 129; 512x512
    // lines of length 32, half a warp a CTA before, 279 -> 145)
    static constexpr bool F64 = sizeof(T) == 8;
    static constexpr int TPC = F64 && (ML == 80 || ML == 160) ? 10
                             : F64 && (ML == 96 || ML == 192) ? 12
                             : F64 && ML == 640 ? 16
                             : ML <= 32 ? 4
                             : ML <= 160 ? 8
                             : ML == 320 ? 20
                             : ML <= 384 ? 16
                             : ML <= 768 || ML == 1280 ? 32
                             : ML == 2048 || ML == 4096 ? 128
                                         : 64;
    // lines per CTA: 8 up to length 768 and at 1280 (32 for the shortest lines in
    // FP32, which would leave a CTA of one warp), 4 above, or 2 or 1 where 4 lines do not
    // fit, so that several CTAs of an SM overlap
    // their loads, stages and stores and a small box still fills the GPU: 16 lines at
    // length 256 took the 128^3 box's batch from 99.7 to 105.3 us, 8 lines
    // at length 1024 the wake's x forward from 648 to 804 us.  FP64: 4 at 64 and 128,
    // so that every SM has lines (below), 16 at 160 for whole warps
    static constexpr int SIZE = int(sizeof(Cx<T>));
    static constexpr bool fit(int l) { return (ML * (l + 1) + 64 + ML) * SIZE <= 112 * 1024; }
    static constexpr int LPC = F64 && (ML == 64 || ML == 128) ? 4
                             : F64 && ML == 160 ? 16
                             : F64 && ML < 128 ? 8
                             : TPC == 4 ? 32
                             : (ML <= 768 || ML == 1280) && fit(8) ? 8
                             : fit(4) ? 4 : ML * SIZE <= 48 * 1024 ? 2 : 1;
    static constexpr int LD = LPC > 1 ? LPC + 1 : 1;
    static constexpr bool FEW = LPC < 16;
    static constexpr int C1 = FEW ? LPC : P::R0 == 16 ? 1 : P::NST == 2 ? 2 : 1;
    static constexpr int SH = FEW ? (LPC == 8 ? 1 : LPC == 4 ? 2 : 3)
                            : P::R0 == 16 ? 4
                            : P::NST == 2 || P::RL == 8 ? 3 : 2;
    static constexpr int S1 = congruent(P::N1 * LD, C1);
    static constexpr int S2 = congruent(((1 << SH) - 1) * S1 + P::N1 * LD, FEW ? 1 : 8);
    static __host__ __device__ constexpr int base(int q0) { return (q0 & ((1 << SH) - 1)) * S1 + (q0 >> SH) * S2; }
    static constexpr int THREADS = LPC * TPC;
    static constexpr size_t SMEM = sizeof(Cx<T>) * (size_t)(ML + base(P::R0 - 1) + P::N1 * LD);
    // resident CTAs the register allocation must allow: FP32 up to 1024 threads
    // per SM (64 registers), FP64 leaves it to the compiler
    static constexpr int BYSMEM = int(227 * 1024 / (SMEM + 1024)), BYREG = 1024 / THREADS;
    static constexpr int OCC = sizeof(T) == 8 ? 1 : BYSMEM < BYREG ? (BYSMEM < 1 ? 1 : BYSMEM) : (BYREG < 1 ? 1 : BYREG);
    static_assert(SMEM <= 227 * 1024 && THREADS <= 1024, "a CTA's lines fit");
    static_assert(TPC % P::R0 == 0 || P::NST == 2, "the middle stage owns a sub-problem per thread");
    // slot of frequency k
    static __device__ __forceinline__ int freq_slot(int k)
    {
        const int q0 = k % P::R0, q1 = k / P::R0 % P::R1, qL = k / (P::R0 * P::R1);
        return base(q0) + (q1 * P::RL + qL) * LD;
    }
};

// The stages between the first one and the spectrum, lanes on consecutive
// lines: DIR < 0 middle then last stage, DIR > 0 last then middle, all in
// shared memory.  Barriers between and after the stages.
template <typename T, int ML, int DIR>
__device__ __forceinline__ void row_inner_stages(Cx<T> *__restrict__ s, const Cx<T> *__restrict__ tw)
{
    using P = Plan<ML>;
    using L = RowLay<T, ML>;
    constexpr int RL = P::RL, LD = L::LD;
    const int l = threadIdx.x % L::LPC, t = threadIdx.x / L::LPC;
    auto last = [&]() {
#pragma unroll
        for (int i = 0; i < (P::GL + L::TPC - 1) / L::TPC; ++i) {
            const int g = t + i * L::TPC;
            if (P::GL % L::TPC != 0 && g >= P::GL) break;
            Cx<T> *p = s + L::base(g % P::R0) + (g / P::R0) * RL * LD + l;
            Cx<T> c[RL];
#pragma unroll
            for (int q = 0; q < RL; ++q) c[q] = p[q * LD];
            Dft<RL, DIR, T>::run(c);
#pragma unroll
            for (int q = 0; q < RL; ++q) p[q * LD] = c[q];
        }
        __syncthreads();
    };
    auto middle = [&]() {
        if constexpr (P::NST == 3) {
            constexpr int R = P::R1, NP = RL, TJ = L::TPC / P::R0;
            static_assert(NP % TJ == 0, "whole groups per thread");
            const int j0 = t / P::R0;
            Cx<T> *p = s + L::base(t % P::R0) + j0 * LD + l;
            const Cx<T> *tw1 = tw + P::TW1 + j0;
#pragma unroll
            for (int j = 0; j < NP; j += TJ) {
                Cx<T> a[R];
#pragma unroll
                for (int q = 0; q < R; ++q) a[q] = p[(j + q * NP) * LD];
                if (DIR < 0)
                    dif_group<R, NP>(a, j, tw1);
                else
                    dit_group<R, NP>(a, j, tw1);
#pragma unroll
                for (int q = 0; q < R; ++q) p[(j + q * NP) * LD] = a[q];
            }
            __syncthreads();
        }
    };
    if (DIR < 0) {
        middle();
        last();
    } else {
        last();
        middle();
    }
}

// Forward: rows (y, y+1) of source plane z, x in [s0x, s0x + Lsx), from the
// block layout (HALF: the apply, where the row lies in [0, M/2) so the first
// stage's upper inputs are zero at compile time) or from a dense box with row
// length dense_ld (the spectrum build, full rows).
template <typename T, int ML, bool HALF>
__device__ __forceinline__ void row_forward_body(int bx, int by, const T *__restrict__ f, Cx<T> *__restrict__ A,
                                                 const PoissonGeom &g, const Cx<T> *__restrict__ twg, int npairs,
                                                 int lb, int dense_ld)
{
    using P = Plan<ML>;
    using L = RowLay<T, ML>;
    constexpr int M = P::M, TPC = L::TPC;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *tw = reinterpret_cast<Cx<T> *>(smem_raw);
    Cx<T> *s = tw + M;
    load_twiddles(tw, twg, M);
    const int t = threadIdx.x % TPC, l = threadIdx.x / TPC;
    const int pr = bx * L::LPC + l;
    const bool live = pr < npairs;
    const int hp = g.Ls[1] >> 1;
    const int zi = live ? pr / hp : 0, yi = live ? 2 * (pr - zi * hp) : 0;
    // a CTA whose lines all lie in row blocks without source blocks has
    // nothing to transform (the y pass does not read those rows)
    if (g.srcrow && !__syncthreads_or(live && ((g.srcrow[zi >> lb] >> (yi >> lb)) & 1ull))) return;
    const T *ff = f + by * g.fstride;
    constexpr int R0 = P::R0;
    constexpr int NG0 = (P::G0 + TPC - 1) / TPC;
    constexpr bool MASKED = P::G0 % TPC != 0;   // the last round of groups is partial
    Cx<T> a[NG0][R0];
    if constexpr (HALF) {
        // the block-map row and the in-block offset of rows (y, y+1) are
        // fixed per line; y is even and b >= 2, so both rows share a block
        const int bm = (1 << lb) - 1;
        const int *mrow = g.srcmap + ((zi >> lb) * g.nbs[1] + (yi >> lb)) * g.nbs[0];
        const int inner = (((zi & bm) << lb) + (yi & bm)) << lb;
#pragma unroll
        for (int i = 0; i < NG0; ++i) {
            const int xr = t + i * TPC - g.s0[0];
#pragma unroll
            for (int p = 0; p < R0 / 2; ++p) {
                const int x = xr + p * P::G0;
                Cx<T> v{T(0), T(0)};
                if (live && (unsigned)x < (unsigned)g.Ls[0] && (!MASKED || t + i * TPC < P::G0)) {
                    const int bi = mrow[x >> lb];
                    if (bi >= 0) {
                        const T *q = ff + ((int64_t)bi << (3 * lb)) + inner + (x & bm);
                        v.x = q[0];
                        v.y = q[1 << lb];
                    }
                }
                a[i][p] = v;
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < NG0; ++i) {
            const int gg = t + i * TPC;
            const T *row = ff + ((int64_t)(g.s0[2] + zi) * g.M[1] + (g.s0[1] + yi)) * dense_ld;
#pragma unroll
            for (int p = 0; p < R0; ++p) {
                const int x = gg + p * P::G0;
                Cx<T> v{T(0), T(0)};
                if (live && x >= g.s0[0] && x < g.s0[0] + g.Ls[0] && (!MASKED || gg < P::G0)) {
                    v.x = row[x];
                    v.y = row[dense_ld + x];
                }
                a[i][p] = v;
            }
        }
    }
    __syncthreads();
    // source rows that end before M/R0 (a small body in a long box): one
    // nonzero input per first-stage group (uniform over the launch)
    const bool single = HALF && g.s0[0] + g.Ls[0] <= P::G0;
#pragma unroll
    for (int i = 0; i < NG0; ++i) {
        const int gg = t + i * TPC;
        if (MASKED && gg >= P::G0) break;
        if (single)
            dif_group_single<P::R0, P::G0>(a[i], gg, tw);
        else
            dif_group<P::R0, P::G0, HALF>(a[i], gg, tw);
#pragma unroll
        for (int q = 0; q < R0; ++q) s[L::base(q) + gg * L::LD + l] = a[i][q];
    }
    __syncthreads();
    row_inner_stages<T, ML, -1>(s, tw);
    if (!live) return;
    // the two rows' half spectra from the packed line
    Cx<T> *row = A + by * g.Astride + ((int64_t)zi * g.ldA_y + yi) * g.ld, *row2 = row + g.ld;
    const Cx<T> *sl = s + l;
    auto unpack = [&](int k) {
        const Cx<T> zk = sl[L::freq_slot(k)];
        const Cx<T> zm = sl[L::freq_slot(k == 0 ? 0 : M - k)];
        row[k] = Cx<T>{T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y)};
        row2[k] = Cx<T>{T(0.5) * (zk.y + zm.y), T(-0.5) * (zk.x - zm.x)};
    };
#pragma unroll 4
    for (int i = 0; i < M / 2 / TPC; ++i) unpack(t + i * TPC);
    if (t == 0) unpack(M / 2);
}

template <typename T, int ML, bool HALF>
__global__ void __launch_bounds__(RowLay<T, ML>::THREADS, RowLay<T, ML>::OCC)
    k_row_forward(const T *__restrict__ f, Cx<T> *__restrict__ A, PoissonGeom g, const Cx<T> *__restrict__ twg,
                  int npairs, int lb, int dense_ld)
{
    row_forward_body<T, ML, HALF>(blockIdx.x, blockIdx.y, f, A, g, twg, npairs, lb, dense_ld);
}

// Inverse: rows (y, y+1) of target plane z from their half spectra; x in
// [t0x, t0x + Ltx) scaled by dx^2 and scattered to the target block layout.
// HALF_OUT: the target x lies in [0, M/2) (even embedding), so only the
// lower half of the last stage's outputs is formed; otherwise (the shifted x
// window, targets up to M) every output is.
template <typename T, int ML, bool HALF_OUT>
__device__ __forceinline__ void row_inverse_body(int bx, int by, const Cx<T> *A, T *u,
                                                 const PoissonGeom &g, const Cx<T> *__restrict__ twg, int npairs,
                                                 int lb)
{
    using P = Plan<ML>;
    using L = RowLay<T, ML>;
    constexpr int M = P::M, TPC = L::TPC;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *tw = reinterpret_cast<Cx<T> *>(smem_raw);
    Cx<T> *s = tw + M;
    load_twiddles(tw, twg, M);
    const int t = threadIdx.x % TPC, l = threadIdx.x / TPC;
    const int pr = bx * L::LPC + l;
    const bool live = pr < npairs;
    const int hp = g.Lt[1] >> 1;
    const int zi = live ? pr / hp : 0, yi = live ? 2 * (pr - zi * hp) : 0;
    // a CTA whose lines all lie in row blocks without target blocks has
    // nothing to write
    if (g.tgtrow && !__syncthreads_or(live && ((g.tgtrow[zi >> lb] >> (yi >> lb)) & 1ull))) return;
    // Hermitian extension of the two half spectra, packed as Z = G1 + i G2: the
    // values at k give Z at k and at M - k, stored at the positions the inverse
    // sweep expects; NB loads of each row in flight
    const Cx<T> *row = A + by * g.Astride + ((int64_t)zi * g.ldA_y + yi) * g.ld, *row2 = row + g.ld;
    Cx<T> *sl = s + l;
    constexpr int NI = M / 2 / TPC, NB = NI % 8 == 0 ? 8 : NI % 6 == 0 ? 6 : NI % 5 == 0 ? 5 : NI % 4 == 0 ? 4 : 1;
    if (live) {
        const Cx<T> e1 = t == 0 ? row[M / 2] : Cx<T>{T(0), T(0)};
        const Cx<T> e2 = t == 0 ? row2[M / 2] : Cx<T>{T(0), T(0)};
#pragma unroll 1
        for (int i0 = 0; i0 < NI; i0 += NB) {
            Cx<T> g1[NB], g2[NB];
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                g1[i] = row[t + (i0 + i) * TPC];
                g2[i] = row2[t + (i0 + i) * TPC];
            }
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const int k = t + (i0 + i) * TPC;
                if (k == 0) g1[i].y = g2[i].y = T(0);
                sl[L::freq_slot(k)] = Cx<T>{g1[i].x - g2[i].y, g1[i].y + g2[i].x};
                if (k != 0) sl[L::freq_slot(M - k)] = Cx<T>{g1[i].x + g2[i].y, g2[i].x - g1[i].y};
            }
        }
        if (t == 0) sl[L::freq_slot(M / 2)] = Cx<T>{e1.x, e2.x};
    } else {
        for (int k = t; k < M; k += TPC) sl[L::freq_slot(k)] = Cx<T>{T(0), T(0)};
    }
    __syncthreads();
    row_inner_stages<T, ML, 1>(s, tw);
    if (!live) return;
    const T sc = T(g.scale);
    const int bm = g.b - 1;
    const int *__restrict__ mrow = g.tgtmap + ((zi >> lb) * g.nbt[1] + (yi >> lb)) * g.nbt[0];
    const int inner = (((zi & bm) << lb) + (yi & bm)) << lb;
    T *uu = u + by * g.ustride;
    constexpr int R0 = P::R0;
    constexpr int NOUT = HALF_OUT ? R0 / 2 : R0;
#pragma unroll
    for (int i = 0; i < (P::G0 + TPC - 1) / TPC; ++i) {
        const int gg = t + i * TPC;
        if (P::G0 % TPC != 0 && gg >= P::G0) break;
        Cx<T> a[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) a[q] = sl[L::base(q) + gg * L::LD];
        dit_group<P::R0, P::G0, HALF_OUT>(a, gg, tw);
        const int xr = gg - g.t0[0];
#pragma unroll
        for (int p = 0; p < NOUT; ++p) {
            const int xi = xr + p * P::G0;
            if ((unsigned)xi >= (unsigned)g.Lt[0]) continue;
            const int bi0 = mrow[xi >> lb];
            if (bi0 < 0) continue;
            T *q = uu + ((int64_t)bi0 << (3 * lb)) + inner + (xi & bm);
            q[0] = sc * a[p].x;
            q[1 << lb] = sc * a[p].y;   // row y + 1 of the same block (y is even, b >= 2)
        }
    }
}

template <typename T, int ML, bool HALF_OUT>
__global__ void __launch_bounds__(RowLay<T, ML>::THREADS, RowLay<T, ML>::OCC)
    k_row_inverse(const Cx<T> *A, T *u, PoissonGeom g, const Cx<T> *__restrict__ twg,
                  int npairs, int lb)
{
    row_inverse_body<T, ML, HALF_OUT>(blockIdx.x, blockIdx.y, A, u, g, twg, npairs, lb);
}

// ---------------------------------------------------------------------------
// Ragged launches: one pass of many independent problems that share the
// transform length (and the kernel's compile-time variant) in one launch.
// The job table travels in the kernel's parameter space; job j owns the CTAs
// [cta0_j, cta0_{j+1}) of the one-dimensional grid, and every CTA finds its
// job by a binary search over cta0 (the same for all threads of a CTA), then
// runs the pass body at its coordinates inside that job.  No CTA waits on
// another, so problems of any size mix in one launch.
// ---------------------------------------------------------------------------
constexpr int kRagJobs = 64;   // jobs per launch (longer lists go in several launches)

template <class J>
struct RagTable {
    J j[kRagJobs];
    int n;
};

template <class J>
__device__ __forceinline__ const J &rag_job(const RagTable<J> &t)
{
    int lo = 0, hi = t.n - 1;
    const int c = blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (t.j[mid].cta0 <= c) lo = mid;
        else hi = mid - 1;
    }
    return t.j[lo];
}

// x passes: in = f (forward) or A (inverse), out = A or u; CTAs (gx, nf).
template <typename T>
struct RowJob {
    PoissonGeom g;
    const void *in;
    void *out;
    const Cx<T> *tw;
    int npairs, lb, nf;
    int cta0, gx;
};
// y passes: the argument list of k_col_forward / k_col_inverse; CTAs (gx, nf).
template <typename T>
struct ColJob {
    const Cx<T> *in;
    Cx<T> *out;
    const Cx<T> *tw;
    RowFlags rf;
    int64_t rs, os, in_plane, out_plane, in_field, out_field;
    int K, nplanes, lo, n, nf;
    int cta0, gx;
};
// z pass: the argument list of k_col_convolve; CTAs nf * col_ctas.
template <typename T>
struct ConvJob {
    Cx<T> *B;
    const void *spec;
    const Cx<T> *tw;
    int64_t field;
    int K, ld, lds, My, ysym, s0, ns, t0, nt, nf;
    int cta0, gx;
};

template <typename T, int ML, bool HALF>
__global__ void __launch_bounds__(RowLay<T, ML>::THREADS, RowLay<T, ML>::OCC) k_row_forward_rag(const __grid_constant__ RagTable<RowJob<T>> t)
{
    const RowJob<T> &J = rag_job(t);
    const int c = (int)blockIdx.x - J.cta0;
    row_forward_body<T, ML, HALF>(c % J.gx, c / J.gx, (const T *)J.in, (Cx<T> *)J.out, J.g, J.tw, J.npairs, J.lb,
                                       0);
}

template <typename T, int ML, bool HALF_OUT>
__global__ void __launch_bounds__(RowLay<T, ML>::THREADS, RowLay<T, ML>::OCC) k_row_inverse_rag(const __grid_constant__ RagTable<RowJob<T>> t)
{
    const RowJob<T> &J = rag_job(t);
    const int c = (int)blockIdx.x - J.cta0;
    row_inverse_body<T, ML, HALF_OUT>(c % J.gx, c / J.gx, (const Cx<T> *)J.in, (T *)J.out, J.g, J.tw, J.npairs,
                                           J.lb);
}

template <typename T, int ML, int W>
__global__ void __launch_bounds__(W * Plan<ML>::TPC) k_col_forward_rag(const __grid_constant__ RagTable<ColJob<T>> t)
{
    const ColJob<T> &J = rag_job(t);
    const int c = (int)blockIdx.x - J.cta0;
    col_forward_body<T, ML, W, true>(c % J.gx, c / J.gx, J.in, J.out, J.K, J.nplanes, J.lo, J.n, J.rs, J.os,
                                     J.in_plane, J.out_plane, J.in_field, J.out_field, J.tw, J.rf);
}

template <typename T, int ML, int W, bool HALF_OUT>
__global__ void __launch_bounds__(W * Plan<ML>::TPC) k_col_inverse_rag(const __grid_constant__ RagTable<ColJob<T>> t)
{
    const ColJob<T> &J = rag_job(t);
    const int c = (int)blockIdx.x - J.cta0;
    col_inverse_body<T, ML, W, HALF_OUT>(c % J.gx, c / J.gx, J.in, J.out, J.K, J.nplanes, J.lo, J.n, J.rs, J.os,
                                         J.in_plane, J.out_plane, J.in_field, J.out_field, J.tw);
}

template <typename T, int ML, int W, int SPEC, int ZV>
__global__ void __launch_bounds__(W * Plan<ML>::TPC, ConvOcc<T, ML, ZV>::value) k_col_convolve_rag(
    const __grid_constant__ RagTable<ConvJob<T>> t)
{
    const ConvJob<T> &J = rag_job(t);
    col_convolve_body<T, ML, W, SPEC>((int)blockIdx.x - J.cta0, J.nf, J.B, J.spec, J.K, J.ld, J.lds, J.My, J.ysym, J.s0,
                                      J.ns, J.t0, J.nt, J.field, J.tw);
}

// ---------------------------------------------------------------------------
// Host-side launch helpers.
// ---------------------------------------------------------------------------
template <typename T, int ML>
struct ColCfg {
    static constexpr int TPC = Plan<ML>::TPC;
    // FP64 runs at two lanes a clock and SM: what counts is that every SM has
    // columns, not how many CTAs share one.  With 32 columns a CTA the 32^3 box (length
    // 64) had 33 CTAs in the y passes and 66 in z: 72.6 us, now 51.2; the FP64 sphere
    // Poisson apply 3623 -> 3548 us
    // At length 160 the 10 groups of the first stage are 2.5 warps of 8 columns, half
    // a warp idle in the dearer stage: 16 columns (z pass of 96x96x80 points, 3 fields: 890 -> 814 us)
    static constexpr int W0 = sizeof(T) == 8 ? (ML == 160 ? 16 : 8) : TPC <= 8 ? 32 : TPC <= 20 ? 16 : 8;
    static constexpr int WMAX = int(98304 / (sizeof(Cx<T>) * ML)) < 1 ? 1 : int(98304 / (sizeof(Cx<T>) * ML));
    static constexpr int W = W0 < WMAX ? W0 : WMAX;
    static constexpr size_t SMEM = sizeof(Cx<T>) * (((size_t)ML) * (W + 1));
};

// The z pass's width: 8 columns at length 320, where five CTAs of 160 threads keep
// their 72 registers (three of 320 had 64 and spilled: 295 against 283 us for the
// refresh of 556 blocks).  Elsewhere the column passes' width: 8 columns at 192, 256
// and 384 took the sphere Poisson apply from 152.4 to 156.6 us and the
// 512x256x256 wake from 6.10 to 7.18 ms.
template <typename T, int ML>
struct ConvCfg : ColCfg<T, ML> {
    static constexpr int W = ML == 320 ? 8 : ColCfg<T, ML>::W;
    static constexpr size_t SMEM = sizeof(Cx<T>) * (((size_t)ML) * (W + 1));
};
}  // namespace pk

// Launch entry points (one set per precision, instantiated in
// lgf_poisson_f32.cu / lgf_poisson_f64.cu).
template <typename T>
lgf_status launch_row_forward(lgf_ctx *ctx, const PoissonGeom &g, const T *f, Cx<T> *A, const Cx<T> *tw, int nfields,
                              int lb, int dense_ld, cudaStream_t s);
template <typename T>
lgf_status launch_row_inverse(lgf_ctx *ctx, const PoissonGeom &g, const Cx<T> *A, T *u, const Cx<T> *tw, int nfields,
                              int lb, cudaStream_t s);
template <typename T>
lgf_status launch_col_forward(lgf_ctx *ctx, int M, int K, int nplanes, int nfields, const Cx<T> *in, Cx<T> *out,
                              int lo, int n, int64_t rs, int64_t os, int64_t in_plane, int64_t out_plane,
                              int64_t in_field, int64_t out_field, const Cx<T> *tw, pk::RowFlags rf, cudaStream_t s,
                              const char *name);
template <typename T>
lgf_status launch_col_inverse(lgf_ctx *ctx, int M, int K, int nplanes, int nfields, const Cx<T> *in, Cx<T> *out,
                              int lo, int n, int64_t rs, int64_t os, int64_t in_plane, int64_t out_plane,
                              int64_t in_field, int64_t out_field, const Cx<T> *tw, cudaStream_t s, const char *name);
template <typename T, int SPEC>
lgf_status launch_col_convolve(lgf_ctx *ctx, const PoissonGeom &g, Cx<T> *B, const T *spec, const Cx<T> *tw,
                               int nfields, cudaStream_t s);
// Ragged launches of one pass over jobs that share the transform length M
// (and the variant named by the other arguments); every job field but cta0
// and gx is set by the caller.
template <typename T>
lgf_status launch_row_forward_rag(lgf_ctx *ctx, int M, pk::RowJob<T> *jobs, int n, cudaStream_t s);
template <typename T>
lgf_status launch_row_inverse_rag(lgf_ctx *ctx, int M, bool half_out, pk::RowJob<T> *jobs, int n, cudaStream_t s);
template <typename T>
lgf_status launch_col_forward_rag(lgf_ctx *ctx, int M, pk::ColJob<T> *jobs, int n, cudaStream_t s);
template <typename T>
lgf_status launch_col_inverse_rag(lgf_ctx *ctx, int M, bool half_out, pk::ColJob<T> *jobs, int n, cudaStream_t s);
template <typename T, int SPEC>
lgf_status launch_col_convolve_rag(lgf_ctx *ctx, int M, int zvar, pk::ConvJob<T> *jobs, int n, cudaStream_t s);

}  // namespace lgf

namespace lgf {
namespace pk {

template <class K>
inline lgf_status set_smem(lgf_ctx *ctx, K kern, size_t smem)
{
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute");
    }
    return LGF_OK;
}

template <typename T, int ML>
lgf_status row_forward_m(lgf_ctx *ctx, const PoissonGeom &g, const T *f, Cx<T> *A, const Cx<T> *tw, int nfields,
                         int lb, int dense_ld, cudaStream_t s)
{
    using C = RowLay<T, ML>;
    auto kern = k_row_forward<T, ML, true>;
    if (dense_ld) {
        // full dense rows: only the FP64 spectrum build
        if constexpr (sizeof(T) == 8)
            kern = k_row_forward<T, ML, false>;
        else
            return fail(ctx, LGF_EINVAL, "row forward: FP32 dense rows");
    } else if (g.s0[0] < 0 || 2 * (g.s0[0] + g.Ls[0]) > g.M[0]) {
        return fail(ctx, LGF_EINVAL, "row forward: source beyond half the transform length");
    }
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    const int npairs = (g.Ls[1] / 2) * g.Ls[2];
    dim3 grid((npairs + C::LPC - 1) / C::LPC, nfields);
    const int ph = prof_begin(ctx, s, dense_ld ? "spectrum_x_forward" : "poisson_x_forward");
    kern<<<grid, C::THREADS, C::SMEM, s>>>(f, A, g, tw, npairs, lb, dense_ld);
    LGF_CHECK_LAUNCH(ctx, "poisson x-forward");
    prof_end(ctx, s, ph);
    return LGF_OK;
}

template <typename T, int ML>
lgf_status row_inverse_m(lgf_ctx *ctx, const PoissonGeom &g, const Cx<T> *A, T *u, const Cx<T> *tw, int nfields,
                         int lb, cudaStream_t s)
{
    using C = RowLay<T, ML>;
    auto kern = k_row_inverse<T, ML, true>;
    if (g.t0[0] < 0 || g.t0[0] + g.Lt[0] > g.M[0])
        return fail(ctx, LGF_EINVAL, "row inverse: target beyond the transform length");
    if (2 * (g.t0[0] + g.Lt[0]) > g.M[0]) kern = k_row_inverse<T, ML, false>;
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    const int npairs = (g.Lt[1] / 2) * g.Lt[2];
    dim3 grid((npairs + C::LPC - 1) / C::LPC, nfields);
    const int ph = prof_begin(ctx, s, "poisson_x_inverse");
    LGF_CUDA(ctx, chain_launch(ctx->chain, kern, grid, C::THREADS, C::SMEM, s, A, u, g, tw, npairs, lb));
    prof_end(ctx, s, ph);
    return LGF_OK;
}

template <typename T, int ML>
lgf_status col_forward_m(lgf_ctx *ctx, int K, int nplanes, int nfields, const Cx<T> *in, Cx<T> *out, int lo, int n,
                         int64_t rs, int64_t os, int64_t in_plane, int64_t out_plane, int64_t in_field,
                         int64_t out_field, const Cx<T> *tw, RowFlags rf, cudaStream_t s, const char *name)
{
    using C = ColCfg<T, ML>;
    auto kern = k_col_forward<T, ML, C::W, true>;
    if (lo + n > ML / 2) {
        // full-length input: only the FP64 spectrum build's z pass
        if constexpr (sizeof(T) == 8)
            kern = k_col_forward<T, ML, C::W, false>;
        else
            return fail(ctx, LGF_EINVAL, "column forward: FP32 input beyond half the transform length");
    }
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    dim3 grid(col_ctas<C::W>(K, nplanes), nfields);
    const int ph = prof_begin(ctx, s, name);
    LGF_CUDA(ctx, chain_launch(ctx->chain, kern, grid, C::W * C::TPC, C::SMEM, s, in, out, K, nplanes, lo, n, rs, os,
                               in_plane, out_plane, in_field, out_field, tw, rf));
    prof_end(ctx, s, ph);
    return LGF_OK;
}

template <typename T, int ML>
lgf_status col_inverse_m(lgf_ctx *ctx, int K, int nplanes, int nfields, const Cx<T> *in, Cx<T> *out, int lo, int n,
                         int64_t rs, int64_t os, int64_t in_plane, int64_t out_plane, int64_t in_field,
                         int64_t out_field, const Cx<T> *tw, cudaStream_t s, const char *name)
{
    using C = ColCfg<T, ML>;
    auto kern = k_col_inverse<T, ML, C::W, true>;
    if (lo < 0 || lo + n > ML) return fail(ctx, LGF_EINVAL, "column inverse: rows beyond the length");
    if (lo + n > ML / 2) kern = k_col_inverse<T, ML, C::W, false>;
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    dim3 grid(col_ctas<C::W>(K, nplanes), nfields);
    const int ph = prof_begin(ctx, s, name);
    LGF_CUDA(ctx, chain_launch(ctx->chain, kern, grid, C::W * C::TPC, C::SMEM, s, in, out, K, nplanes, lo, n, rs, os,
                               in_plane, out_plane, in_field, out_field, tw));
    prof_end(ctx, s, ph);
    return LGF_OK;
}

template <typename T, int ML, int SPEC>
lgf_status col_convolve_m(lgf_ctx *ctx, const PoissonGeom &g, Cx<T> *B, const T *spec, const Cx<T> *tw, int nfields,
                          cudaStream_t s)
{
    using C = ConvCfg<T, ML>;
    // the register variant is an FP32 choice (FP64 runs one CTA per SM)
    auto kern = (sizeof(T) == 4 && g.zvar) ? k_col_convolve<T, ML, C::W, SPEC, sizeof(T) == 4 ? 1 : 0>
                                           : k_col_convolve<T, ML, C::W, SPEC, 0>;
    if (g.s0[2] < 0 || g.t0[2] < 0 || 2 * (g.s0[2] + g.Ls[2]) > g.M[2] ||
        (SPEC == 3 ? 1 : 2) * (g.t0[2] + g.Lt[2]) > g.M[2])
        return fail(ctx, LGF_EINVAL, "z pass: planes beyond the transform's inputs or outputs");
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    dim3 grid(nfields * col_ctas<C::W>(g.Kx, g.M[1]));
    const int ph = prof_begin(ctx, s, "poisson_z_convolve");
    LGF_CUDA(ctx, chain_launch(ctx->chain, kern, grid, C::W * C::TPC, C::SMEM, s, B, spec, g.Kx, g.ld, g.ld, g.M[1],
                               !g.yasym, g.s0[2], g.Ls[2], g.t0[2], g.Lt[2], g.Bstride, tw));
    prof_end(ctx, s, ph);
    return LGF_OK;
}

// Send jobs in tables of kRagJobs, CTA ranges assigned in order; jobs with
// no CTAs are skipped.
template <class J, class Kern>
lgf_status rag_send(lgf_ctx *ctx, Kern kern, int threads, size_t smem, J *jobs, int n, cudaStream_t s,
                    const char *name)
{
    static_assert(sizeof(RagTable<J>) <= 32000, "job table beyond the kernel parameter space");
    for (int c0 = 0; c0 < n;) {
        RagTable<J> t;
        t.n = 0;
        int64_t ctas = 0;
        for (; c0 < n && t.n < kRagJobs; ++c0) {
            J &j = jobs[c0];
            const int64_t nc = (int64_t)j.gx * j.nf;
            if (nc <= 0) continue;
            j.cta0 = (int)ctas;
            t.j[t.n++] = j;
            ctas += nc;
        }
        if (t.n == 0) continue;
        if (ctas > 0x7fffffff) return fail(ctx, LGF_EUNSUPPORTED, "ragged launch: too many CTAs");
        const int ph = prof_begin(ctx, s, name);
        kern<<<(unsigned)ctas, threads, smem, s>>>(t);
        LGF_CHECK_LAUNCH(ctx, name);
        prof_end(ctx, s, ph);
    }
    return LGF_OK;
}

template <typename T, int ML>
lgf_status row_forward_rag_m(lgf_ctx *ctx, RowJob<T> *jobs, int n, cudaStream_t s)
{
    using C = RowLay<T, ML>;
    auto kern = k_row_forward_rag<T, ML, true>;
    for (int i = 0; i < n; ++i) {
        const PoissonGeom &g = jobs[i].g;
        if (g.M[0] != ML || g.s0[0] < 0 || 2 * (g.s0[0] + g.Ls[0]) > g.M[0])
            return fail(ctx, LGF_EINVAL, "ragged row forward: source beyond half the transform length");
        jobs[i].gx = (jobs[i].npairs + C::LPC - 1) / C::LPC;
    }
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    return rag_send(ctx, kern, C::THREADS, C::SMEM, jobs, n, s, "poisson_x_forward");
}

template <typename T, int ML>
lgf_status row_inverse_rag_m(lgf_ctx *ctx, bool half_out, RowJob<T> *jobs, int n, cudaStream_t s)
{
    using C = RowLay<T, ML>;
    auto kern = half_out ? k_row_inverse_rag<T, ML, true> : k_row_inverse_rag<T, ML, false>;
    for (int i = 0; i < n; ++i) {
        const PoissonGeom &g = jobs[i].g;
        if (g.M[0] != ML || g.t0[0] < 0 || g.t0[0] + g.Lt[0] > g.M[0] ||
            (half_out && 2 * (g.t0[0] + g.Lt[0]) > g.M[0]))
            return fail(ctx, LGF_EINVAL, "ragged row inverse: target beyond the transform length");
        jobs[i].gx = (jobs[i].npairs + C::LPC - 1) / C::LPC;
    }
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    return rag_send(ctx, kern, C::THREADS, C::SMEM, jobs, n, s, "poisson_x_inverse");
}

template <typename T, int ML>
lgf_status col_forward_rag_m(lgf_ctx *ctx, ColJob<T> *jobs, int n, cudaStream_t s)
{
    using C = ColCfg<T, ML>;
    auto kern = k_col_forward_rag<T, ML, C::W>;
    for (int i = 0; i < n; ++i) {
        if (jobs[i].lo < 0 || jobs[i].lo + jobs[i].n > ML / 2)
            return fail(ctx, LGF_EINVAL, "ragged column forward: input beyond half the transform length");
        jobs[i].gx = col_ctas<C::W>(jobs[i].K, jobs[i].nplanes);
    }
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    return rag_send(ctx, kern, C::W * C::TPC, C::SMEM, jobs, n, s, "poisson_y_forward");
}

template <typename T, int ML>
lgf_status col_inverse_rag_m(lgf_ctx *ctx, bool half_out, ColJob<T> *jobs, int n, cudaStream_t s)
{
    using C = ColCfg<T, ML>;
    auto kern = half_out ? k_col_inverse_rag<T, ML, C::W, true> : k_col_inverse_rag<T, ML, C::W, false>;
    for (int i = 0; i < n; ++i) {
        if (jobs[i].lo < 0 || jobs[i].lo + jobs[i].n > (half_out ? ML / 2 : ML))
            return fail(ctx, LGF_EINVAL, "ragged column inverse: rows beyond the length");
        jobs[i].gx = col_ctas<C::W>(jobs[i].K, jobs[i].nplanes);
    }
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    return rag_send(ctx, kern, C::W * C::TPC, C::SMEM, jobs, n, s, "poisson_y_inverse");
}

template <typename T, int ML, int SPEC>
lgf_status col_convolve_rag_m(lgf_ctx *ctx, int zvar, ConvJob<T> *jobs, int n, cudaStream_t s)
{
    using C = ConvCfg<T, ML>;
    auto kern = (sizeof(T) == 4 && zvar) ? k_col_convolve_rag<T, ML, C::W, SPEC, sizeof(T) == 4 ? 1 : 0>
                                         : k_col_convolve_rag<T, ML, C::W, SPEC, 0>;
    for (int i = 0; i < n; ++i) {
        const ConvJob<T> &j = jobs[i];
        if (j.s0 < 0 || j.t0 < 0 || 2 * (j.s0 + j.ns) > ML || (SPEC == 3 ? 1 : 2) * (j.t0 + j.nt) > ML)
            return fail(ctx, LGF_EINVAL, "ragged z pass: planes beyond the transform's inputs or outputs");
        jobs[i].gx = col_ctas<C::W>(j.K, j.My);
    }
    lgf_status st = set_smem(ctx, kern, C::SMEM);
    if (st != LGF_OK) return st;
    return rag_send(ctx, kern, C::W * C::TPC, C::SMEM, jobs, n, s, "poisson_z_convolve");
}

#define LGF_DISPATCH_ML(M_RT, CALL)                                             \
    switch (M_RT) {                                                             \
    case 32: { constexpr int LM = 32; return CALL; }                            \
    case 64: { constexpr int LM = 64; return CALL; }                            \
    case 80: { constexpr int LM = 80; return CALL; }                            \
    case 160: { constexpr int LM = 160; return CALL; }                          \
    case 320: { constexpr int LM = 320; return CALL; }                          \
    case 640: { constexpr int LM = 640; return CALL; }                          \
    case 1280: { constexpr int LM = 1280; return CALL; }                        \
    case 2560: { constexpr int LM = 2560; return CALL; }                        \
    case 96: { constexpr int LM = 96; return CALL; }                            \
    case 128: { constexpr int LM = 128; return CALL; }                          \
    case 192: { constexpr int LM = 192; return CALL; }                          \
    case 256: { constexpr int LM = 256; return CALL; }                          \
    case 384: { constexpr int LM = 384; return CALL; }                          \
    case 512: { constexpr int LM = 512; return CALL; }                          \
    case 768: { constexpr int LM = 768; return CALL; }                          \
    case 1024: { constexpr int LM = 1024; return CALL; }                        \
    case 1536: { constexpr int LM = 1536; return CALL; }                        \
    case 2048: { constexpr int LM = 2048; return CALL; }                        \
    case 3072: { constexpr int LM = 3072; return CALL; }                        \
    case 4096: { constexpr int LM = 4096; return CALL; }                        \
    default: return fail(ctx, LGF_EUNSUPPORTED, "transform length not 2^k, 3*2^k or 5*2^k in 32..4096"); \
    }

}  // namespace pk

template <typename T>
lgf_status launch_row_forward(lgf_ctx *ctx, const PoissonGeom &g, const T *f, Cx<T> *A, const Cx<T> *tw, int nfields,
                              int lb, int dense_ld, cudaStream_t s)
{
    LGF_DISPATCH_ML(g.M[0], (pk::row_forward_m<T, LM>(ctx, g, f, A, tw, nfields, lb, dense_ld, s)));
}

template <typename T>
lgf_status launch_row_inverse(lgf_ctx *ctx, const PoissonGeom &g, const Cx<T> *A, T *u, const Cx<T> *tw, int nfields,
                              int lb, cudaStream_t s)
{
    LGF_DISPATCH_ML(g.M[0], (pk::row_inverse_m<T, LM>(ctx, g, A, u, tw, nfields, lb, s)));
}

template <typename T>
lgf_status launch_col_forward(lgf_ctx *ctx, int M, int K, int nplanes, int nfields, const Cx<T> *in, Cx<T> *out,
                              int lo, int n, int64_t rs, int64_t os, int64_t in_plane, int64_t out_plane,
                              int64_t in_field, int64_t out_field, const Cx<T> *tw, pk::RowFlags rf, cudaStream_t s,
                              const char *name)
{
    LGF_DISPATCH_ML(M, (pk::col_forward_m<T, LM>(ctx, K, nplanes, nfields, in, out, lo, n, rs, os,
                                                               in_plane, out_plane, in_field, out_field, tw, rf,
                                                               s, name)));
}

template <typename T>
lgf_status launch_col_inverse(lgf_ctx *ctx, int M, int K, int nplanes, int nfields, const Cx<T> *in, Cx<T> *out,
                              int lo, int n, int64_t rs, int64_t os, int64_t in_plane, int64_t out_plane,
                              int64_t in_field, int64_t out_field, const Cx<T> *tw, cudaStream_t s, const char *name)
{
    LGF_DISPATCH_ML(M, (pk::col_inverse_m<T, LM>(ctx, K, nplanes, nfields, in, out, lo, n, rs, os,
                                                               in_plane, out_plane, in_field, out_field, tw,
                                                               s, name)));
}

template <typename T, int SPEC>
lgf_status launch_col_convolve(lgf_ctx *ctx, const PoissonGeom &g, Cx<T> *B, const T *spec, const Cx<T> *tw,
                               int nfields, cudaStream_t s)
{
    LGF_DISPATCH_ML(g.M[2], (pk::col_convolve_m<T, LM, SPEC>(ctx, g, B, spec, tw, nfields, s)));
}

template <typename T>
lgf_status launch_row_forward_rag(lgf_ctx *ctx, int M, pk::RowJob<T> *jobs, int n, cudaStream_t s)
{
    LGF_DISPATCH_ML(M, (pk::row_forward_rag_m<T, LM>(ctx, jobs, n, s)));
}

template <typename T>
lgf_status launch_row_inverse_rag(lgf_ctx *ctx, int M, bool half_out, pk::RowJob<T> *jobs, int n, cudaStream_t s)
{
    LGF_DISPATCH_ML(M, (pk::row_inverse_rag_m<T, LM>(ctx, half_out, jobs, n, s)));
}

template <typename T>
lgf_status launch_col_forward_rag(lgf_ctx *ctx, int M, pk::ColJob<T> *jobs, int n, cudaStream_t s)
{
    LGF_DISPATCH_ML(M, (pk::col_forward_rag_m<T, LM>(ctx, jobs, n, s)));
}

template <typename T>
lgf_status launch_col_inverse_rag(lgf_ctx *ctx, int M, bool half_out, pk::ColJob<T> *jobs, int n, cudaStream_t s)
{
    LGF_DISPATCH_ML(M, (pk::col_inverse_rag_m<T, LM>(ctx, half_out, jobs, n, s)));
}

template <typename T, int SPEC>
lgf_status launch_col_convolve_rag(lgf_ctx *ctx, int M, int zvar, pk::ConvJob<T> *jobs, int n, cudaStream_t s)
{
    LGF_DISPATCH_ML(M, (pk::col_convolve_rag_m<T, LM, SPEC>(ctx, zvar, jobs, n, s)));
}

}  // namespace lgf
