// Step (a), FP64: R_ij(E) = (1/2a) sum_k w_ik w_jk / (E_k - E)  (Section "Overview",
// Eq. rmatrix), the upper triangle of each energy's R in the packed layout
// (tri_idx, stride tri_ld(n)).
//
// This is the plain-FP64 baseline the mixed-precision path is measured
// against. Only the upper triangle is computed and stored, so every R is
// exactly symmetric. d_k = 1/(E_k - E) is formed once per (CTA, k) in shared
// memory and folded into the j-operand.
#include "rm_internal.cuh"

namespace rmgb {
namespace {

// Where packed_wins(n): the packed pairs p = (i <= j) of one energy dealt out 32 to a
// warp load, PT loads a warp, so that no FP64 FMA is spent on an entry that is
// not stored. GB300 issues 2 FP64 FMAs per clock and SM, and everything else
// (two shared loads per FMA, the staging) fits beside them; a 64 x 64 tile
// kernel spends 3072 FMAs per pole where 64 channels need 2080, and 21504
// where 132 need 8778. 4000 energies of 64 channels x 1920 poles: 39.9 ms
// tiled, 27.6 ms packed (floor 27.4); 200 of 132 x 3960: 30.4 and 13.1 ms
// (floor 11.9).
//
// A CTA takes NW PT warp loads of one energy, from row rlo on: per chunk of TK
// poles it stages the rows rlo .. n - 1 of W and of W d (DIV: W / (E_k - E),
// n < 32) in shared memory (row stride TK + 1 doubles: lanes on consecutive
// rows j read distinct banks), the next chunk's W and the chunk after that
// one's d already on their way. Every entry is one chain of FMAs over
// ascending poles.
constexpr int PK_MAX_WARPS = 16;

template <int PT, int TK, bool DIV>
__global__ void __launch_bounds__(PK_MAX_WARPS * 32)
    form_r_packed(PwDev pw, const double *__restrict__ E, double *__restrict__ R)
{
    extern __shared__ double sm[];
    const int n = pw.n, N = pw.N, np = tri_count(n);
    const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31;
    const double x = E[blockIdx.y];
    const int p_cta = blockIdx.x * nthr * PT;
    auto row_of = [&](int p) {   // row of packed pair p
        const float t = (float)(2 * n + 1);
        int i = (int)((t - sqrtf(fmaxf(t * t - 8.0f * (float)p, 0.0f))) * 0.5f);
        i = min(max(i, 0), n - 1);
        while (i > 0 && tri_idx(i, i, n) > p) --i;
        while (i + 1 < n && tri_idx(i + 1, i + 1, n) <= p) ++i;
        return i;
    };
    const int rlo = row_of(p_cta), nr = n - rlo;
    constexpr int LD = TK + 1;
    double *Ws = sm, *Wd = sm + nr * LD, *dk = Wd + nr * LD;   // dk: [2][TK]
    // offsets of the pairs' rows; past the end, those of the last pair
    int io[PT], jo[PT];
    double acc[PT];
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int p = min(p_cta + (warp * PT + q) * 32 + lane, np - 1);
        const int i = row_of(p);
        io[q] = (i - rlo) * LD;
        jo[q] = (i + (p - tri_idx(i, i, n)) - rlo) * LD;
        acc[q] = 0.0;
    }
    const int total = nr * TK;
    const double *Wg = pw.W + (size_t)rlo * N;
    auto den = [&](int k) { return k < N ? pw.Ek[k] - x : 1.0; };
    if (tid < 2 * TK) dk[tid] = DIV ? den(tid) : (tid < N ? 1.0 / den(tid) : 0.0);
    constexpr int PRE = 4;   // elements of the next chunk a thread holds
    double pre[PRE];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < PRE; ++u) {
            const int q = tid + u * nthr, r = q / TK, c = q - r * TK;
            pre[u] = q < total && k0 + c < N ? Wg[(size_t)r * N + k0 + c] : 0.0;
        }
    };
    fetch(0);
    __syncthreads();
    for (int k0 = 0, b = 0; k0 < N; k0 += TK, b ^= 1) {
        const double *dc = dk + b * TK;
        auto put = [&](int q, double w) {
            const int r = q / TK, c = q - r * TK;
            Ws[r * LD + c] = w;
            Wd[r * LD + c] = DIV ? w / dc[c] : w * dc[c];
        };
#pragma unroll
        for (int u = 0; u < PRE; ++u)
            if (tid + u * nthr < total) put(tid + u * nthr, pre[u]);
        for (int q = tid + PRE * nthr; q < total; q += nthr) {
            const int r = q / TK, c = q - r * TK;
            put(q, k0 + c < N ? Wg[(size_t)r * N + k0 + c] : 0.0);
        }
        __syncthreads();
        if (k0 + TK < N) fetch(k0 + TK);
        if (tid < TK) {
            const int k = k0 + 2 * TK + tid;
            dk[b * TK + tid] = DIV ? den(k) : (k < N ? 1.0 / den(k) : 0.0);
        }
#pragma unroll
        for (int c = 0; c < TK; ++c)
#pragma unroll
            for (int q = 0; q < PT; ++q) acc[q] = fma(Ws[io[q] + c], Wd[jo[q] + c], acc[q]);
        __syncthreads();
    }
    const double h = 0.5 / pw.a;
    double *Re = R + (size_t)blockIdx.y * tri_ld(n);
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int p = p_cta + (warp * PT + q) * 32 + lane;
        if (p < np) Re[p] = acc[q] * h;
    }
}

template <int PT, int TK, bool DIV>
cudaError_t launch_packed(const PwDev &pw, const double *E, int nE, double *R, int nw, int ctas, cudaStream_t s)
{
    const size_t smem = ((size_t)2 * pw.n * (TK + 1) + 2 * TK) * sizeof(double);
    const cudaError_t e = allow_smem(form_r_packed<PT, TK, DIV>, smem);
    if (e != cudaSuccess) return e;
    form_r_packed<PT, TK, DIV><<<dim3(ctas, nE), nw * 32, smem, s>>>(pw, E, R);
    return cudaGetLastError();
}

// Loads per warp, warps and CTAs per energy.
struct PkPlan {
    int pt, nw, ctas;
};

// From 32 channels on, the least of CTAs x (warp-load lanes + rows to be
// scaled), the FP64 work of a pole.
PkPlan pk_plan(int n)
{
    const int nq = (tri_count(n) + 31) / 32;
    if (n < 32) {
        const int pt = nq <= 4 ? 1 : (nq <= 8 ? 2 : 4);
        return {pt, (nq + pt - 1) / pt, 1};
    }
    PkPlan best = {};
    long long least = 0;
    for (int p = 4; p <= 8; ++p)
        for (int w = 4; w <= PK_MAX_WARPS; ++w) {
            const int c = (nq + p * w - 1) / (p * w);
            const long long cost = (long long)c * (32 * p * w + n);
            if (least == 0 || cost < least) {
                least = cost;
                best = {p, w, c};
            }
        }
    return best;
}

// Packed pairs or tiles: both run at the FP64 pipe (600 and 610 GFMA/s counted
// as here), so the fewer FP64 operations of a pole win. Packed pairs: every
// lane of every warp load and the rows a CTA scales, those from its first
// pair's on. Tiles: 64 x 64 (48 x 64 on the diagonal) and 64 columns to scale.
// ms for 1000 poles, packed and tiled: 200 x 1000 energies 35.0, 61.4; 320 x
// 400 37.6, 37.8; 384 x 300 40.3, 40.1; 448 x 200 36.7, 35.9; 500 x 160 37.1,
// 37.4; 512 x 160 39.2, 37.2; 530 x 160 41.9, 46.7; 660 x 100 41.6, 43.3; 700
// x 100 46.6, 43.3; 769 x 64 36.9, 38.5. Above PK_MAX_N one CTA of staged rows
// fills an SM and the pipe idles at its barriers (833 x 64: 48.2, 44.4).
constexpr int PK_MAX_N = 784;

bool packed_wins(int n, const PkPlan &pl)
{
    if (n < 32) return true;
    if (n > PK_MAX_N) return false;
    const int span = 32 * pl.pt * pl.nw, t = (n + 63) / 64;
    long long packed = 0;
    for (int c = 0, i = 0; c < pl.ctas; ++c) {
        while (i + 1 < n && tri_idx(i + 1, i + 1, n) <= c * span) ++i;
        packed += span + n - i;
    }
    const long long tiled = (long long)t * (t - 1) / 2 * (64 * 64 + 64) + (long long)t * (48 * 64 + 64);
    return 51 * packed <= 50 * tiled;
}

cudaError_t launch_packed_any(const PwDev &pw, const PkPlan &pl, const double *E, int nE, double *R, cudaStream_t s)
{
    const int n = pw.n, pt = pl.pt, nw = pl.nw, ctas = pl.ctas;
#define RM_PK(P, K, D) launch_packed<P, K, D>(pw, E, nE, R, nw, ctas, s)
    if (n < 32) return pt == 1 ? RM_PK(1, 16, true) : (pt == 2 ? RM_PK(2, 16, true) : RM_PK(4, 16, true));
    // poles per chunk: at most ~70 KB of shared memory (three CTAs per SM) up
    // to 512 channels, two CTAs above (with 4 poles a chunk instead, 530 x 160
    // took 47.5 ms, 41.9 so: a barrier comes too often)
#define RM_PK_TK(P) (n <= 256 ? RM_PK(P, 16, false) : RM_PK(P, 8, false))
    switch (pt) {
    case 4: return RM_PK_TK(4);
    case 5: return RM_PK_TK(5);
    case 6: return RM_PK_TK(6);
    case 7: return RM_PK_TK(7);
    default: return RM_PK_TK(8);
    }
#undef RM_PK_TK
#undef RM_PK
}

constexpr int TB = 64;   // output tile
constexpr int TK = 16;   // pole chunk
constexpr int TT = 4;    // outputs per thread per dimension

// The rest: CTA per (energy, 64x64 upper tile); 256 threads x 4x4 outputs.
// Off-diagonal tiles: thread (ty, tx) = (tid/16, tid%16) owns rows 4ty.., cols
// 4tx... Diagonal tiles: the 32x32 quadrant below the diagonal is not needed,
// so whole warps are assigned to the three upper quadrants (2 warps each) and
// warps 6-7 sit out; the FP64 pipe is not spent on discarded outputs.
__global__ void __launch_bounds__(256) form_r_tiled(PwDev pw, const double *__restrict__ E,
                                                    double *__restrict__ R)
{
    const int ti = blockIdx.y, tj = blockIdx.x;
    if (tj < ti) return;
    const int e = blockIdx.z;
    const int n = pw.n, N = pw.N;
    const int i0 = ti * TB, j0 = tj * TB;
    __shared__ double Wi[TK][TB + 1];
    __shared__ double Wj[TK][TB + 1];
    __shared__ double dk[TK];
    const int tid = threadIdx.x;
    int tx = tid & 15, ty = tid >> 4;
    bool active = true;
    if (ti == tj) {
        const int w = tid >> 5, l = tid & 31;
        const int quad = w >> 1;             // 0: (0,0), 1: (0,1), 2: (1,1), 3: idle
        const int sub = (w & 1) * 32 + l;    // 64 threads per 32x32 quadrant
        const int qy = (quad == 2) ? 1 : 0, qx = (quad == 0) ? 0 : 1;
        ty = qy * 8 + (sub >> 3);
        tx = qx * 8 + (sub & 7);
        active = quad < 3;
    }
    const double x = E[e];
    double acc[TT][TT];
#pragma unroll
    for (int a = 0; a < TT; ++a)
#pragma unroll
        for (int b = 0; b < TT; ++b) acc[a][b] = 0.0;

    for (int k0 = 0; k0 < N; k0 += TK) {
        if (tid < TK) {
            const int k = k0 + tid;
            dk[tid] = (k < N) ? 1.0 / (pw.Ek[k] - x) : 0.0;
        }
        __syncthreads();
        // 64 rows x 16 poles per operand: 4 elements per thread, k fastest
#pragma unroll
        for (int t = 0; t < (TB * TK) / 256; ++t) {
            const int q = tid + t * 256;
            const int r = q / TK, c = q - (q / TK) * TK;
            const int k = k0 + c;
            const int gi = i0 + r, gj = j0 + r;
            Wi[c][r] = (gi < n && k < N) ? pw.W[(size_t)gi * N + k] : 0.0;
            Wj[c][r] = (gj < n && k < N) ? pw.W[(size_t)gj * N + k] * dk[c] : 0.0;
        }
        __syncthreads();
        if (active) {
#pragma unroll
        for (int c = 0; c < TK; ++c) {
            double av[TT], bv[TT];
#pragma unroll
            for (int a = 0; a < TT; ++a) av[a] = Wi[c][ty * TT + a];
#pragma unroll
            for (int b = 0; b < TT; ++b) bv[b] = Wj[c][tx * TT + b];
#pragma unroll
            for (int a = 0; a < TT; ++a)
#pragma unroll
                for (int b = 0; b < TT; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
        }
        }
        __syncthreads();
    }
    if (!active) return;
    const double h = 0.5 / pw.a;
    double *Re = R + (size_t)e * tri_ld(n);
#pragma unroll
    for (int a = 0; a < TT; ++a) {
        const int i = i0 + ty * TT + a;
#pragma unroll
        for (int b = 0; b < TT; ++b) {
            const int j = j0 + tx * TT + b;
            if (i < n && j < n && i <= j) Re[tri_idx(i, j, n)] = acc[a][b] * h;
        }
    }
}

}  // namespace

cudaError_t launch_form_r_fp64(const PwDev &pw, const double *E, int nE, double *R,
                               cudaStream_t s)
{
    if (nE == 0) return cudaSuccess;
    const PkPlan pl = pk_plan(pw.n);
    if (packed_wins(pw.n, pl)) return launch_packed_any(pw, pl, E, nE, R, s);
    const int t = (pw.n + TB - 1) / TB;
    dim3 grid(t, t, nE);
    form_r_tiled<<<grid, 256, 0, s>>>(pw, E, R);
    return cudaGetLastError();
}

}  // namespace rmgb
