// FP32 dense kernels of the global-memory solver's mixed-precision path
// (rm_opts.solve_precision = RM_FP32, channel counts above the shared-memory
// solver's limit). One CTA works on one energy's matrices in global memory: 128
// or 256 threads for the narrower systems, so that several share an SM, 512 for
// the wider ones (launch_lu32_any and launch_zsweep_any, solve_large.cu):
//
//   lu32_factor_solve   [A | B] -> solves A X = B for the trailing rows of X
//                       (the matching system, Section "Overview", Eq. match):
//                       blocked right-looking LU with partial pivoting. The
//                       current panel of PB columns (all rows below its
//                       diagonal) is factored with its rows in registers
//                       (one barrier per column) and left in shared memory,
//                       column-major; its row interchanges are applied to the
//                       columns to its right as one permutation per panel;
//                       U12 = L11^{-1} A12 is solved one column per thread;
//                       the trailing matrix takes the rank-PB update
//                       A22 -= L21 U12 in strips of 128 columns with 4 x 8
//                       or (two panel rows a thread) 8 x 8 register tiles per
//                       thread, packed FMAs (the U12 strips copied
//                       asynchronously into two shared buffers in turn).
//                       Back-substitution of the
//                       requested rows runs in the same blocked form, upwards.
//   zsweep_invert       Z <- -Z^{-1} for a complex symmetric Z whose
//                       Hermitian part is positive definite (Z = 1 - iK, the
//                       T step of Section "Glossary of terms"): the sweep
//                       operator applied PB pivots at a time, no pivoting
//                       (every leading block of such a Z is nonsingular).
//                       Per block of pivots K: the PB x PB block is swept in
//                       shared memory (B -> -B^{-1}), the panel
//                       P = Z[:, K] B^{-1} is formed in shared memory, every
//                       other entry takes Z_ij -= P_i Z_Kj (rank-PB complex
//                       update in strips of 64 columns, 4 x 4 per thread,
//                       packed FMAs), and
//                       Z[:, K], Z[K, :] become P and P^T. Z stays symmetric,
//                       so only the upper triangle is kept current: tiles
//                       wholly below the diagonal are skipped and every read
//                       takes the entry (min(i, j), max(i, j)).
//
// At 1000 channels both stream their trailing matrix through HBM once per
// panel (152 CTAs hold 1.2 GB), but what their inner loops wait for is shared
// memory, from which every FMA's operands come (64 energies: L1 and shared
// memory 48% and 75% busy in LU and sweep, FMA pipe 46% and 48%, DRAM 10% and
// 7%); below about 300 they were bound by the latency of the panel's columns,
// which the registers and the second CTA per SM take away. ms for 304 or more
// systems filling the GPU, before and after: LU of 110 unknowns (1216 systems) 1.61 -> 0.46, 203 (912)
// 2.85 -> 1.11, 431 (456) 5.37 -> 3.44, 1000 (304, 600 right-hand sides) 22.1
// -> 19.1; sweep of 80 (1216) 0.63 -> 0.39, 150 (912) 1.38 -> 1.00, 300 (456)
// 2.79 -> 2.30, 600 (304) 11.5 -> 11.0. Every entry keeps its chain of FMAs,
// so the results are the same to the bit.
//
// Both kernels read and write their matrix through global memory (L2), with
// no waits other than __syncthreads. A zero or non-finite pivot marks the
// energy RM_ESINGULAR and the CTA returns.
#pragma once

#include <math.h>
#include <type_traits>

#include "rm_internal.cuh"

namespace rmgb {
namespace f32d {

constexpr int UW = 128;    // real strip width (columns)
constexpr int UWC = 64;    // complex strip width (columns)
constexpr int LU_SLOT = 36;   // floats of one warp's pivot candidate: its row (32), key, position

// Layout of the real augmented matrix of n unknowns and np right-hand sides:
// columns [0, n) A, [n, rhs0(n)) zero, [rhs0(n), rhs0(n) + np) B, zero up to ld.
__host__ __device__ inline int rhs0(int n) { return (n + 3) & ~3; }
__host__ __device__ inline int aug_ld(int n, int np) { return (rhs0(n) + np + 3) & ~3; }
// Column stride of the shared-memory panel (4 mod 32 floats: the row-wise
// panel load hits 4-way bank conflicts at most, float4 reads stay aligned).
__host__ __device__ inline int lu_npad(int n) { return ((rhs0(n) + 31) & ~31) + 4; }
// Complex matrix of order m: row stride, and the panel's column stride.
__host__ __device__ inline int z_ld(int m) { return (m + 3) & ~3; }
__host__ __device__ inline int z_npad(int m) { return ((m + 7) & ~7) + 8; }

template <int PB, int NTH, int RPT> __host__ __device__ inline size_t lu_smem(int n)
{
    const size_t f = (size_t)PB * lu_npad(n) + 2 * (size_t)PB * (UW + 4) + (RPT > 0 ? 2 * (NTH / 32) * LU_SLOT : 0);
    // perm [npad], move lists [2 PB], counters [8], reduction keys
    // [NWARP x 64 bit], reduction values [NWARP], and slack
    const size_t i = (size_t)lu_npad(n) + 2 * PB + 8 + 3 * (NTH / 32) + 16;
    return f * sizeof(float) + i * sizeof(int);
}

// LEAN: one strip, and operand pairs formed at each use instead of stored
// (the widest systems whose panel of PB columns still fits).
template <int PB, bool LEAN> __host__ __device__ inline size_t z_smem(int m)
{
    const size_t panel = (size_t)PB * z_npad(m) * sizeof(float2), block = (size_t)PB * (PB + 1) * sizeof(float2);
    if (LEAN) return panel + (size_t)PB * (UWC + 2) * sizeof(float2) + block;
    return panel + 2 * (size_t)PB * (UWC + 2) * sizeof(float4) + (size_t)PB * PB * sizeof(float4) + block;
}

// Packed FP32 FMA: each half is fma(a, b, c) of that half, rounded as the
// scalar instruction rounds it. The FMA pipe takes two clocks for it, so the
// rank updates run at the pipe's rate with half the issue slots.
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long pack2(float x, float y)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool in)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = in ? 16 : 0;   // 0: the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// Packed key of a pivot candidate: larger magnitude first, then lower row.
// Magnitudes are non-negative floats, whose bit patterns order as integers;
// a NaN counts as +infinity (it is then caught as a non-finite pivot).
__device__ __forceinline__ unsigned long long piv_key(float v, int r)
{
    float m = fabsf(v);
    if (m != m) m = __int_as_float(0x7f800000);
    return ((unsigned long long)__float_as_uint(m) << 32) | (unsigned)(0x7fffffff - r);
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long k)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, k, off);
        k = o > k ? o : k;
    }
    return k;
}

// ---- real blocked LU ---------------------------------------------------------

// Prefetch into L2 of the line at p.
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Rows [rlo, rhi) (stored from rstore; rlo a multiple of 4), columns
// [c_lo, w): C += Lp x U, Lp the column-major panel of PB columns (stride
// npad) holding the negated multipliers, U = rows [u0, u0 + PB) of M (final,
// zero from column w to ld). Strips of 128 columns, their U copied
// asynchronously into two shared buffers in turn (one barrier per strip);
// thread (ty, tx) = (tid / 16, tid % 16) takes rows TI ty .. TI ty + TI - 1 of
// each tile of TI NTH / 16 rows and columns 4 tx .. 4 tx + 3 and 64 + 4 tx ..
// 64 + 4 tx + 3 (a quarter-warp's float4 reads of U hit distinct banks). The C
// tile after the current one, the next strip's first at a strip's end, is on
// its way meanwhile. Shared memory delivers 128 bytes a clock to a warp's
// lanes, broadcast or not, and bounds the product: TI = 4 reads 48 bytes for
// 32 FMAs and holds the next tile in registers, TI = 8 reads 64 for 64 and has
// only L2 for the next tile. TI = 8 with two panel rows a thread: the solve of
// 152 systems of 513 open channels 8.96 -> 8.39 ms, of 640 13.2 -> 12.4, of
// 1000 43.3 -> 41.8, the elimination of 512 of 331 (256 threads) 2.13 -> 1.90;
// with one row a thread, where a tile is most of the matrix, it is 2-7 % slower.
template <int PB, int NTH, int TI>
__device__ void lu_update_rows(float *M, int ld, int u0, int rlo, int rhi, int rstore, int c_lo, int w, const float *Lp,
                               int npad, float *Us)
{
    constexpr int TR = TI * NTH / 16;   // rows per tile
    constexpr bool REGS = TI == 4;     // the next tile in registers
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int nstrip = (w - c_lo + UW - 1) / UW;
    auto stage = [&](int s, float *buf) {
        for (int q = tid; q < PB * (UW / 4); q += NTH) {
            const int k = q / (UW / 4), j4 = 4 * (q - (q / (UW / 4)) * (UW / 4));
            const int c = c_lo + s * UW + j4;
            cp_async16(buf + k * (UW + 4) + j4, M + (size_t)(u0 + k) * ld + min(c, ld - 4), c < ld);
        }
    };
    auto load = [&](int rb, int c0, unsigned long long (&v)[TI][4]) {
#pragma unroll
        for (int i = 0; i < TI; ++i) {
            const int r = rb + i;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = c0 + 64 * h + 4 * tx;
                ulonglong2 q = make_ulonglong2(0ull, 0ull);
                if (r < rhi && r >= rstore && c < ld) q = *reinterpret_cast<const ulonglong2 *>(M + (size_t)r * ld + c);
                v[i][2 * h] = q.x;
                v[i][2 * h + 1] = q.y;
            }
        }
    };
    stage(0, Us);
    unsigned long long acc[TI][4], nxt[REGS ? TI : 1][4];
    const int rb0 = rlo + TI * ty;
    if constexpr (REGS) load(rb0, c_lo, acc);
    for (int s = 0; s < nstrip; ++s) {
        const float *cur = Us + (s & 1) * PB * (UW + 4);
        const int c0 = c_lo + s * UW;
        cp_async_wait();
        __syncthreads();
        if (s + 1 < nstrip) stage(s + 1, Us + ((s + 1) & 1) * PB * (UW + 4));
        int rb = rb0;
        for (int r0 = rlo; r0 < rhi; r0 += TR, rb += TR) {
            const bool last = r0 + TR >= rhi;
            if constexpr (REGS) {
                if (!last) load(rb + TR, c0, nxt);
                else if (s + 1 < nstrip) load(rb0, c0 + UW, nxt);
            } else {
                load(rb, c0, acc);
                // half a row's 128 columns a lane: two lines of 128 bytes
                const int rn = (last ? rb0 : rb + TR) + (tx >> 1), cn = (last ? c0 + UW : c0) + 64 * (tx & 1);
                if (rn < rhi && cn < ld) prefetch_l2(M + (size_t)rn * ld + cn);
                if (rn < rhi && cn + 32 < ld) prefetch_l2(M + (size_t)rn * ld + cn + 32);
            }
            if (rb < rhi) {   // reads of Lp past rhi stay in shared memory and feed rows that are not stored
#pragma unroll (REGS ? 4 : 2)
                for (int k = 0; k < PB; ++k) {
                    float av[TI];
#pragma unroll
                    for (int i = 0; i < TI; i += 4) {
                        const float4 q = *reinterpret_cast<const float4 *>(Lp + k * npad + rb + i);
                        av[i] = q.x, av[i + 1] = q.y, av[i + 2] = q.z, av[i + 3] = q.w;
                    }
                    const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(cur + k * (UW + 4) + 4 * tx);
                    const ulonglong2 b1 = *reinterpret_cast<const ulonglong2 *>(cur + k * (UW + 4) + 64 + 4 * tx);
                    const unsigned long long b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
                    for (int i = 0; i < TI; ++i) {
                        const unsigned long long a = pack2(av[i], av[i]);
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[i][j] = fma2(a, b[j], acc[i][j]);
                    }
                }
#pragma unroll
                for (int i = 0; i < TI; ++i) {
                    const int r = rb + i;
                    if (r >= rhi || r < rstore) continue;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int c = c0 + 64 * h + 4 * tx;
                        if (c < ld)
                            *reinterpret_cast<ulonglong2 *>(M + (size_t)r * ld + c) =
                                make_ulonglong2(acc[i][2 * h], acc[i][2 * h + 1]);
                    }
                }
            }
            if constexpr (REGS) {
#pragma unroll
                for (int i = 0; i < TI; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = nxt[i][j];
            }
        }
    }
    __syncthreads();
}

// Factors the panel of columns [k0, k0 + kb), rows [k0, n), with partial
// pivoting (largest magnitude, then lowest row). On return Lp[j][r] holds the
// factored panel in its final row order, entries below the diagonal negated,
// and perm[r] the row that position r came from. A thread keeps RPT rows of
// the panel in registers, so a column costs one barrier: every warp puts its
// candidate (the row itself, key and position) into a slot before it, and all
// take the best slot after it; rows change position only in a register.
// Measured with the panel's rows in shared memory and two barriers: 2300 (203
// rows) to 2900 (1000 rows) clocks a column.
template <int PB, int NTH, int RPT>
__device__ bool lu_panel_regs(const float *M, int ld, int n, int k0, int kb, float *Lp, int npad, int *perm, float *slots)
{
    constexpr int NW = NTH / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float a[RPT][PB];
    int pos[RPT];
    bool live[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int r = k0 + tid + q * NTH;
        pos[q] = r;
        live[q] = r < n;
#pragma unroll
        for (int g = 0; g < PB; g += 4) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < n && k0 + g < ld) v = *reinterpret_cast<const float4 *>(M + (size_t)r * ld + k0 + g);
            a[q][g] = v.x;
            a[q][g + 1] = v.y;
            a[q][g + 2] = v.z;
            a[q][g + 3] = v.w;
        }
    }
#pragma unroll
    for (int j = 0; j < PB; ++j) {
        if (j >= kb) break;
        const int c = k0 + j;
        float *slot = slots + (j & 1) * NW * LU_SLOT;
        // key 0: no row left; a NaN counts as infinity (and is then not finite)
        unsigned mag = 0u;
        int mp = 0x7fffffff, mq = 0;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            unsigned u = __float_as_uint(fabsf(a[q][j]));
            u = u > 0x7f800000u ? 0x7f800000u : u;
            if (live[q] && (mp == 0x7fffffff || u > mag || (u == mag && pos[q] < mp))) {
                mag = u;
                mp = pos[q];
                mq = q;
            }
        }
        const unsigned wm = __reduce_max_sync(0xffffffffu, mag);
        const unsigned wp = __reduce_min_sync(0xffffffffu, mag == wm ? (unsigned)mp : 0x7fffffffu);
        if (mag == wm && (unsigned)mp == wp && wp != 0x7fffffffu) {
            float *dst = slot + warp * LU_SLOT;
#pragma unroll
            for (int q = 0; q < RPT; ++q)
                if (mq == q) {
#pragma unroll
                    for (int g = (j & ~3); g < PB; g += 4)
                        *reinterpret_cast<float4 *>(dst + g) = make_float4(a[q][g], a[q][g + 1], a[q][g + 2], a[q][g + 3]);
                }
            *reinterpret_cast<float2 *>(dst + PB) = make_float2(__uint_as_float(wm), __int_as_float((int)wp));
        } else if (lane == 0 && wp == 0x7fffffffu) {
            *reinterpret_cast<float2 *>(slot + warp * LU_SLOT + PB) = make_float2(0.f, __int_as_float(0x7fffffff));
        }
        __syncthreads();
        float2 cand = make_float2(0.f, __int_as_float(0x7fffffff));
        if (lane < NW) cand = *reinterpret_cast<const float2 *>(slot + lane * LU_SLOT + PB);
        const unsigned cm = __float_as_uint(cand.x), cp = (unsigned)__float_as_int(cand.y);
        const unsigned bm = __reduce_max_sync(0xffffffffu, cm);
        const unsigned p = __reduce_min_sync(0xffffffffu, cm == bm ? cp : 0x7fffffffu);
        const int win = __ffs(__ballot_sync(0xffffffffu, cm == bm && cp == p)) - 1;
        const float *pr = slot + win * LU_SLOT;
        const float pv = pr[j];
        if (!(fabsf(pv) > 0.f) || !isfinite(pv)) return false;   // the same decision in every thread
        const float ipv = 1.0f / pv;
        float l[RPT];   // 0 for rows already placed: they keep their entries
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            l[q] = 0.f;
            if (live[q]) {
                if (pos[q] == (int)p) {
                    live[q] = false;
                    pos[q] = c;
                } else {
                    if (pos[q] == c) pos[q] = (int)p;
                    l[q] = a[q][j] * ipv;
                    a[q][j] = -l[q];
                }
            }
        }
#pragma unroll
        for (int g = (j & ~3); g < PB; g += 4) {
            const float4 v4 = *reinterpret_cast<const float4 *>(pr + g);
            const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
            for (int q = 0; q < RPT; ++q)
                if (live[q]) {
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        if (g + h > j) a[q][g + h] = fmaf(-l[q], v[h], a[q][g + h]);
                }
        }
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int r = k0 + tid + q * NTH;
        if (r < n) {
            perm[pos[q]] = r;
#pragma unroll
            for (int j = 0; j < PB; ++j) Lp[j * npad + pos[q]] = a[q][j];
        }
    }
    return true;
}

// The same with the panel's rows in shared memory (any number of rows).
template <int PB, int NTH>
__device__ bool lu_panel_smem(const float *M, int ld, int n, int k0, int kb, float *Lp, int npad, int *perm,
                              unsigned long long *red, float *red_val)
{
    constexpr int NWARP = NTH / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < (n - k0) * kb; q += NTH) {
        const int r = k0 + q / kb, j = q - (q / kb) * kb;
        Lp[j * npad + r] = M[(size_t)r * ld + k0 + j];
    }
    for (int r = k0 + tid; r < n; r += NTH) perm[r] = r;
    __syncthreads();
    // pivot candidates of the panel's first column
    {
        unsigned long long key = 0ull;
        float kv = 0.f;
        for (int r = k0 + tid; r < n; r += NTH) {
            const float v = Lp[r];
            const unsigned long long kk = piv_key(v, r);
            if (kk > key) {
                key = kk;
                kv = v;
            }
        }
        const unsigned long long wk = warp_max_u64(key);
        const unsigned ball = __ballot_sync(0xffffffffu, key == wk && wk != 0ull);
        if (lane == 0) red[warp] = wk;
        if (ball && lane == __ffs(ball) - 1) red_val[warp] = kv;
    }
    __syncthreads();
    for (int j = 0; j < kb; ++j) {
        const int c = k0 + j;
        unsigned long long best = red[0];
        float pv = red_val[0];
#pragma unroll
        for (int q = 1; q < NWARP; ++q)
            if (red[q] > best) {
                best = red[q];
                pv = red_val[q];
            }
        const int p = 0x7fffffff - (int)(unsigned)(best & 0xffffffffu);
        const bool bad = best == 0ull || !(fabsf(pv) > 0.f) || !isfinite(pv);
        if (!bad && p != c) {
            if (tid < kb) {
                const float t = Lp[tid * npad + c];
                Lp[tid * npad + c] = Lp[tid * npad + p];
                Lp[tid * npad + p] = t;
            }
            if (tid == PB) {
                const int t = perm[c];
                perm[c] = perm[p];
                perm[p] = t;
            }
        }
        __syncthreads();
        if (bad) return false;
        // multipliers and the rank-1 update of the panel's remaining
        // columns; each thread's rows of column j + 1 are final here, so
        // their pivot candidates are taken on the way
        const float ipv = 1.0f / pv;
        unsigned long long key = 0ull;
        float kv = 0.f;
        for (int r = c + 1 + tid; r < n; r += NTH) {
            const float l = Lp[j * npad + r] * ipv;
            Lp[j * npad + r] = -l;
            for (int jj = j + 1; jj < kb; ++jj) Lp[jj * npad + r] = fmaf(-l, Lp[jj * npad + c], Lp[jj * npad + r]);
            if (j + 1 < kb) {
                const float v = Lp[(j + 1) * npad + r];
                const unsigned long long kk = piv_key(v, r);
                if (kk > key) {
                    key = kk;
                    kv = v;
                }
            }
        }
        if (j + 1 < kb) {
            const unsigned long long wk = warp_max_u64(key);
            const unsigned ball = __ballot_sync(0xffffffffu, key == wk && wk != 0ull);
            if (lane == 0) red[warp] = wk;
            if (ball && lane == __ffs(ball) - 1) red_val[warp] = kv;
        }
        __syncthreads();
    }
    return true;
}

// Solves A X = B in place for the n x w augmented matrix M (row stride ld,
// A in columns [0, n), right-hand sides in [rhs, w), zero padding between and
// after), leaving X in rows [row_lo, n) of the right-hand-side columns.
// RPT: rows of a panel per thread (n <= RPT NTH), 0: panel in shared memory.
// Returns false if a pivot is zero or not finite.
template <int PB, int NTH, int RPT>
__device__ bool lu32_factor_solve(float *M, int ld, int n, int w, int rhs, int row_lo, float *smem)
{
    constexpr int NWARP = NTH / 32;
    constexpr int TI = RPT == 2 ? 8 : 4;   // rows of a thread in the updates
    const int tid = threadIdx.x;
    const int npad = lu_npad(n);
    float *Lp = smem;
    float *Us = Lp + (size_t)PB * npad;
    float *slots = Us + 2 * PB * (UW + 4);
    int *perm = reinterpret_cast<int *>(slots + (RPT > 0 ? 2 * NWARP * LU_SLOT : 0));
    int *mv_dst = perm + npad;
    int *mv_src = mv_dst + PB;
    int *sh_int = mv_src + PB;                 // [0]: move count
    unsigned long long *red = reinterpret_cast<unsigned long long *>(sh_int + 8);   // [NWARP]
    float *red_val = reinterpret_cast<float *>(red + NWARP);                        // [NWARP]

    for (int k0 = 0; k0 < n; k0 += PB) {
        const int kb = min(PB, n - k0);
        if (tid == 0) sh_int[0] = 0;
        if constexpr (RPT > 0) {
            if (!lu_panel_regs<PB, NTH, RPT>(M, ld, n, k0, kb, Lp, npad, perm, slots)) return false;
            __syncthreads();
        } else {
            if (!lu_panel_smem<PB, NTH>(M, ld, n, k0, kb, Lp, npad, perm, red, red_val)) return false;
        }
        // U11 to global memory; rows moved below the panel by its interchanges
        for (int q = tid; q < kb * kb; q += NTH) {
            const int i = q / kb, j = q - (q / kb) * kb;
            if (i <= j) M[(size_t)(k0 + i) * ld + k0 + j] = Lp[j * npad + k0 + i];
        }
        for (int r = k0 + kb + tid; r < n; r += NTH)
            if (perm[r] != r) {
                const int s = atomicAdd(&sh_int[0], 1);
                mv_dst[s] = r;
                mv_src[s] = perm[r];
            }
        __syncthreads();
        const int nmv = sh_int[0];
        if (k0 + kb >= w) continue;
        // trailing columns: interchanges and U12 = L11^{-1} A12, one thread per
        // column; U12 goes to rows [k0, k0 + kb) of global memory
        for (int c = k0 + kb + tid; c < w; c += NTH) {
            float x[PB];
            // The new rows k0 .. k0 + kb come from perm[], which may name rows
            // below the panel; those rows are then move destinations, so they
            // are read first. A row below the panel only ever receives a row
            // of [k0, k0 + kb) (a position of the panel is never swapped
            // again once its pivot is chosen), and those rows are written
            // last, so the moves need no further ordering.
#pragma unroll
            for (int j = 0; j < PB; ++j) x[j] = j < kb ? M[(size_t)perm[k0 + j] * ld + c] : 0.f;
            for (int i0 = 0; i0 < nmv; i0 += 8) {
                float y[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i0 + i < nmv) y[i] = M[(size_t)mv_src[i0 + i] * ld + c];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i0 + i < nmv) M[(size_t)mv_dst[i0 + i] * ld + c] = y[i];
            }
            // x_j -= L_ji x_i, i ascending for every j; four j a shared read
#pragma unroll
            for (int i = 0; i < PB - 1; ++i) {
                if (i + 1 < kb) {
#pragma unroll
                    for (int g = ((i + 1) & ~3); g < PB; g += 4) {
                        const float4 l = *reinterpret_cast<const float4 *>(Lp + i * npad + k0 + g);
                        if (g > i) x[g] = fmaf(l.x, x[i], x[g]);
                        if (g + 1 > i) x[g + 1] = fmaf(l.y, x[i], x[g + 1]);
                        if (g + 2 > i) x[g + 2] = fmaf(l.z, x[i], x[g + 2]);
                        if (g + 3 > i) x[g + 3] = fmaf(l.w, x[i], x[g + 3]);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < PB; ++j)
                if (j < kb) M[(size_t)(k0 + j) * ld + c] = x[j];
        }
        __syncthreads();
        if (k0 + kb < n) lu_update_rows<PB, NTH, TI>(M, ld, k0, k0 + kb, n, k0 + kb, k0 + kb, w, Lp, npad, Us);
    }
    // back-substitution of rows [row_lo, n) for the right-hand sides
    const int rs = row_lo & ~3;
    int t1 = n;
    while (t1 > row_lo) {
        const int t0 = max(row_lo, t1 - PB);
        const int tb = t1 - t0;
        // -U of the block's columns: rows above it into the panel, the block
        // itself row by row into Us (four columns a read)
        for (int q = tid; q < (t1 - rs) * tb; q += NTH) {
            const int r = rs + q / tb, j = q - (q / tb) * tb;
            const float v = r >= row_lo ? -M[(size_t)r * ld + t0 + j] : 0.f;
            if (r < t0) Lp[j * npad + r] = v;
            else Us[(r - t0) * PB + j] = v;
        }
        __syncthreads();
        for (int c = rhs + tid; c < w; c += NTH) {
            float x[PB];
#pragma unroll
            for (int j = 0; j < PB; ++j) x[j] = j < tb ? M[(size_t)(t0 + j) * ld + c] : 0.f;
#pragma unroll
            for (int i = PB - 1; i >= 0; --i) {
                if (i < tb) {
                    float sum = x[i];
#pragma unroll
                    for (int g = (i & ~3); g < PB; g += 4) {
                        const float4 u = *reinterpret_cast<const float4 *>(Us + i * PB + g);
                        const float v[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (g + j > i && g + j < tb) sum = fmaf(v[j], x[g + j], sum);
                    }
                    x[i] = sum / -Us[i * PB + i];
                }
            }
#pragma unroll
            for (int j = 0; j < PB; ++j)
                if (j < tb) M[(size_t)(t0 + j) * ld + c] = x[j];
        }
        __syncthreads();
        if (t0 > row_lo) lu_update_rows<PB, NTH, TI>(M, ld, t0, rs, t0, row_lo, rhs, w, Lp, npad, Us);
        t1 = t0;
    }
    return true;
}

// ---- complex symmetric sweep -------------------------------------------------

__device__ __forceinline__ float2 cfma_neg(float2 a, float2 b, float2 c)
{
    // c - a b
    c.x = fmaf(-a.x, b.x, fmaf(a.y, b.y, c.x));
    c.y = fmaf(-a.x, b.y, fmaf(-a.y, b.x, c.y));
    return c;
}

__device__ __forceinline__ float2 crcp_safe(float2 d)
{
    const float s = fmaxf(fabsf(d.x), fabsf(d.y));
    const float xr = d.x / s, xi = d.y / s;
    const float t = 1.0f / (s * fmaf(xr, xr, xi * xi));
    return make_float2(xr * t, -xi * t);
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// Entry (i, j) of a symmetric Z of which only the upper triangle is current.
__device__ __forceinline__ float2 zu(const float2 *Z, int ldz, int i, int j)
{
    return i <= j ? Z[(size_t)i * ldz + j] : Z[(size_t)j * ldz + i];
}

// The operands of c -= a b with packed FMAs: b1 = (b.y, -b.x), b2 = -b; then
// c = fma2((a.x, a.x), b2, fma2((a.y, a.y), b1, c)) rounds as cfma_neg does.
__device__ __forceinline__ float4 zpair(float2 b) { return make_float4(b.y, -b.x, -b.x, -b.y); }

// How a multiplicand is kept in shared memory: as its pair, or (LEAN) itself.
template <bool LEAN> struct ZOp {
    using type = float4;
    static __device__ __forceinline__ float4 make(float2 b) { return zpair(b); }
};
template <> struct ZOp<true> {
    using type = float2;
    static __device__ __forceinline__ float2 make(float2 b) { return b; }
};
__device__ __forceinline__ ulonglong2 zget(const float4 *p) { return *reinterpret_cast<const ulonglong2 *>(p); }
__device__ __forceinline__ ulonglong2 zget(const float2 *p)
{
    const float4 q = zpair(*p);
    return make_ulonglong2(pack2(q.x, q.y), pack2(q.z, q.w));
}

// Z (m x m complex symmetric, row stride ldz, zero padding to ldz) <- -Z^{-1}
// in its upper triangle (the lower triangle is left stale).
template <int PB, int NTH, bool LEAN>
__device__ bool zsweep_invert(float2 *Z, int ldz, int m, float2 *smem)
{
    using Op = typename ZOp<LEAN>::type;
    constexpr int TR = NTH / 4;                   // rows per tile
    constexpr int SPT = PB * UWC / NTH;           // strip elements per thread
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int npz = z_npad(m);
    float2 *Lp = smem;
    Op *Us = reinterpret_cast<Op *>(Lp + (size_t)PB * npz);   // two strips (LEAN: one)
    Op *Bp = Us + (LEAN ? 1 : 2) * PB * (UWC + 2);
    float2 *Bs = reinterpret_cast<float2 *>(Bp + (LEAN ? 0 : PB * PB));
    for (int k0 = 0; k0 < m; k0 += PB) {
        const int kb = min(PB, m - k0);
        if (tid < PB * PB) {
            const int i = tid / PB, j = tid - (tid / PB) * PB;
            Bs[i * (PB + 1) + j] = (i < kb && j < kb) ? zu(Z, ldz, k0 + i, k0 + j) : make_float2(0.f, 0.f);
        }
        __syncthreads();
        // sweep of the diagonal block: B -> -B^{-1}
        for (int p = 0; p < kb; ++p) {
            const float2 d = Bs[p * (PB + 1) + p];
            const bool bad = !(fabsf(d.x) + fabsf(d.y) > 0.f) || !isfinite(d.x) || !isfinite(d.y);
            if (bad) return false;   // the same decision in every thread
            float2 v = make_float2(0.f, 0.f);
            const int i = tid / PB, j = tid - (tid / PB) * PB;
            const bool own = tid < PB * PB && i < kb && j < kb;
            if (own) {
                const float2 dinv = crcp_safe(d);
                if (i == p && j == p) {
                    v = make_float2(-dinv.x, -dinv.y);
                } else if (i == p) {
                    v = cmul(Bs[p * (PB + 1) + j], dinv);
                } else if (j == p) {
                    v = cmul(Bs[i * (PB + 1) + p], dinv);
                } else {
                    v = cfma_neg(cmul(Bs[i * (PB + 1) + p], dinv), Bs[p * (PB + 1) + j], Bs[i * (PB + 1) + j]);
                }
            }
            __syncthreads();
            if (own) Bs[i * (PB + 1) + j] = v;
            __syncthreads();
        }
        if constexpr (!LEAN) {
            if (tid < PB * PB) Bp[tid] = zpair(Bs[(tid / PB) * (PB + 1) + (tid - (tid / PB) * PB)]);
            __syncthreads();
        }
        // panel P_i = Z[i, K] B^{-1} = -Z[i, K] Bs for rows i outside K; a
        // thread takes half a row's columns
        for (int t = tid; t < 2 * m; t += NTH) {
            const int i = t < m ? t : t - m, kh = t < m ? 0 : PB / 2;
            unsigned long long P[PB / 2];
#pragma unroll
            for (int k = 0; k < PB / 2; ++k) P[k] = 0ull;
            if (i < k0 || i >= k0 + kb) {
                float2 zq[PB];
#pragma unroll
                for (int q = 0; q < PB; ++q) zq[q] = q < kb ? zu(Z, ldz, i, k0 + q) : make_float2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < PB; ++q) {
                    if (q < kb) {
                        const unsigned long long ax = pack2(zq[q].x, zq[q].x), ay = pack2(zq[q].y, zq[q].y);
#pragma unroll
                        for (int k = 0; k < PB / 2; ++k) {
                            ulonglong2 b;
                            if constexpr (LEAN) b = zget(Bs + q * (PB + 1) + kh + k);
                            else b = zget(Bp + q * PB + kh + k);
                            P[k] = fma2(ax, b.y, fma2(ay, b.x, P[k]));
                        }
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < PB / 2; ++k)
                Lp[(kh + k) * npz + i] = (kh + k < kb) ? unpack2(P[k]) : make_float2(0.f, 0.f);
        }
        // Z_ij -= P_i Z_Kj for i, j outside K, i <= j, 64 columns at a time (the
        // first strip is the one with fewer, where there are the fewest rows:
        // 512 systems of 150 / 200 / 260 open channels .670, 1.28, 2.43 ms with it
        // last, .638, 1.14, 2.20 so); the
        // next strip's Z_Kj and the next tile's Z_ij are on their way meanwhile.
        // A warp leaves out its 8 rows of a tile where they lie below the
        // strip's last column, and the strip's first half where they lie below
        // that: the solve of 152 systems of 290 open channels 2.33 -> 2.28 ms, of 513
        // 8.44 -> 7.95, of 640 12.5 -> 11.8, of 1000 41.9 -> 40.5.
        const int nstrip = (m + UWC - 1) / UWC;
        const int w0 = ((m + 1) & ~1) - (nstrip - 1) * UWC;   // columns of strip 0
        auto strip0 = [&](int s) { return s ? w0 + (s - 1) * UWC : 0; };
        float2 st[SPT];
        auto fetch = [&](int s) {   // strips left of K lie in columns of Z: k fastest there
            const int c0 = strip0(s);
            const bool left = c0 < k0;
#pragma unroll
            for (int u = 0; u < SPT; ++u) {
                const int q = tid + u * NTH;
                const int k = left ? q % PB : q / UWC, c = c0 + (left ? q / PB : q % UWC);
                const bool in = k < kb && c < m && (c < k0 || c >= k0 + kb);
                st[u] = in ? zu(Z, ldz, k0 + k, c) : make_float2(0.f, 0.f);
            }
        };
        auto put = [&](int s) {
            const bool left = strip0(s) < k0;
            Op *buf = Us + (LEAN ? 0 : (s & 1)) * PB * (UWC + 2);
#pragma unroll
            for (int u = 0; u < SPT; ++u) {
                const int q = tid + u * NTH;
                const int k = left ? q % PB : q / UWC, jj = left ? q / PB : q % UWC;
                // column 32 h + 2 x + e of the strip at 16 (2 h + e) + x: a
                // thread's four columns are four conflict-free reads
                buf[k * (UWC + 2) + 16 * (2 * (jj >> 5) + (jj & 1)) + ((jj & 31) >> 1)] = ZOp<LEAN>::make(st[u]);
            }
        };
        auto zload = [&](int rb, int c0, unsigned long long (&v)[4][4]) {
            const int c_end = c0 ? c0 + UWC : w0, r_end = min(m, c_end);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = rb + i;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c = c0 + 32 * h + 2 * tx;
                    ulonglong2 q = make_ulonglong2(0ull, 0ull);
                    if (r < r_end && c < c_end) q = *reinterpret_cast<const ulonglong2 *>(Z + (size_t)r * ldz + c);
                    v[i][2 * h] = q.x;
                    v[i][2 * h + 1] = q.y;
                }
            }
        };
        unsigned long long acc[4][4], nxt[4][4];
        // columns 32 H0 .. 63 of the strip cur at c0, rows rb .. rb + 3
        auto update = [&](auto h0, const Op *cur, int c0, int c_end, int rb) {
            constexpr int H0 = decltype(h0)::value;
#pragma unroll 4
            for (int k = 0; k < PB; ++k) {
                const float4 a0 = *reinterpret_cast<const float4 *>(Lp + k * npz + rb);
                const float4 a1 = *reinterpret_cast<const float4 *>(Lp + k * npz + rb + 2);
                const Op *b = cur + k * (UWC + 2) + tx;
                ulonglong2 bj[4];
#pragma unroll
                for (int j = 2 * H0; j < 4; ++j) bj[j] = zget(b + 16 * j);
                const float ax[4] = {a0.x, a0.z, a1.x, a1.z}, ay[4] = {a0.y, a0.w, a1.y, a1.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const unsigned long long y = pack2(ay[i], ay[i]), x = pack2(ax[i], ax[i]);
#pragma unroll
                    for (int j = 2 * H0; j < 4; ++j) acc[i][j] = fma2(y, bj[j].x, acc[i][j]);
#pragma unroll
                    for (int j = 2 * H0; j < 4; ++j) acc[i][j] = fma2(x, bj[j].y, acc[i][j]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = rb + i;
                if (r >= m) continue;
#pragma unroll
                for (int h = H0; h < 2; ++h) {
                    const int c = c0 + 32 * h + 2 * tx;
                    if (c < c_end)
                        *reinterpret_cast<ulonglong2 *>(Z + (size_t)r * ldz + c) =
                            make_ulonglong2(acc[i][2 * h], acc[i][2 * h + 1]);
                }
            }
        };
        fetch(0);
        if (!LEAN) put(0);
        const int rb0 = ty * 4;
        zload(rb0, 0, acc);
        for (int s = 0; s < nstrip; ++s) {
            const int c0 = strip0(s), c_end = c0 ? c0 + UWC : w0;
            const Op *cur = Us + (LEAN ? 0 : (s & 1)) * PB * (UWC + 2);
            if (LEAN) {
                __syncthreads();
                put(s);
            }
            __syncthreads();   // strip s (and, the first time, the panel) is complete
            if (s + 1 < nstrip) fetch(s + 1);
            const int r_end = min(m, c_end);   // row tiles starting past this are below the diagonal
            int rb = rb0;
            for (int r0 = 0; r0 < r_end; r0 += TR, rb += TR) {
                const bool last = r0 + TR >= r_end;
                if (!last) zload(rb + TR, c0, nxt);
                else if (s + 1 < nstrip) zload(rb0, c_end, nxt);
                const int rw = rb & ~7;   // the warp's first row
                if (rw >= c0 + 32 && rb < r_end) update(std::integral_constant<int, 1>(), cur, c0, c_end, rb);
                else if (rb < r_end) update(std::integral_constant<int, 0>(), cur, c0, c_end, rb);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = nxt[i][j];
            }
            if (!LEAN && s + 1 < nstrip) put(s + 1);
        }
        __syncthreads();
        // upper-triangle positions of Z[i, K] = P_i and Z[K, i] = P_i^T, and
        // Z[K, K] = -B^{-1}
        for (int q = tid; q < k0 * PB; q += NTH) {
            const int i = q / PB, k = q - (q / PB) * PB;
            if (k < kb) Z[(size_t)i * ldz + k0 + k] = Lp[k * npz + i];
        }
        for (int q = tid; q < kb * (m - k0 - kb); q += NTH) {
            const int k = q / (m - k0 - kb), i = k0 + kb + (q - (q / (m - k0 - kb)) * (m - k0 - kb));
            Z[(size_t)(k0 + k) * ldz + i] = Lp[k * npz + i];
        }
        if (tid < PB * PB) {
            const int i = tid / PB, j = tid - (tid / PB) * PB;
            if (i < kb && j < kb) Z[(size_t)(k0 + i) * ldz + k0 + j] = Bs[i * (PB + 1) + j];
        }
        __syncthreads();
    }
    return true;
}

}  // namespace f32d
}  // namespace rmgb
