// The block exchanges of the Gauss-Jordan sweep (see tcgemm.cu for the
// arithmetic) for float64 / complex128 fronts, as exact integer products on
// the BF16 tensor cores.
//
// GB300's FP64 pipe runs 1.25 TFLOP/s, and the rank-kb sweep of a 256 x 256
// P2 Helmholtz matrix (277 GFLOP of float64 updates) spends half of its time
// at that rate.  Here every operand is written as a sum of integers the tensor
// core takes exactly (the error-free transformation of Ozaki, Ogita, Oishi &
// Rump, Numer. Algorithms 2012, with a shared exponent per row): with e the
// exponent of the largest entry of the row (a row of the slab, a column of
// -M(P, :)) once the pivots are levelled,
//
//      v = 2^(e - 6) sum_{s < 8} d_s 2^(-8 s),   |d_0| <= 64, |d_s| <= 128,
//
// 62 bits below the row's largest entry.  The products d_p d_q with p + q = s
// < 8 are accumulated per s in their own tensor-memory accumulator: 36 MMAs
// per K step.  A sum of at most T64_KB2 x 2 = 128 such terms per pair is an
// integer below 2^24 for every s, so FP32 accumulation is exact in any order;
// what is left out (p + q >= 8) is below 2^-59 of the product of the two rows'
// largest entries per term: under the rounding of a float64 dot product of that
// length where no pivot's products are far below the others'.
//
// Levelling sees to that.  Unknowns on different scales (A -> D A E, D and E
// diagonal) multiply column q of M'(:, P) by 1 / D_q and row q of M(P, :) by D_q:
// the products keep their size, but a row's largest entry is that of the pivot
// with the smallest D_q, and the others lose bits.  pivot_levels reads the
// pivots' scales off the inverse of their own block, M'(P, P), whose rows all
// combine every pivot: with r_p the exponent of the largest entry of its row p,
// column q goes up by s_q = min_p (r_p - exponent of (p, q)) powers of two and
// row q of M down by as many (exact: exponents only).  Errors of one exchange
// relative to D_i E_j, scales over 2^24 / 2^48 / 2^80: 1e-11 / 6e-5 / 1 without
// levelling, 1e-16 / 7e-16 / 5e-16 with it, 4e-16 in float64.
//
// The epilogue joins the eight integers into two of 51 bits in integer
// arithmetic, those into one float64 value rounded once (two FMAs, ints_scaled)
// and adds it to the front: three FP64 instructions per element (summing the
// eight in float64 would make the FP64 pipe the bound again).
//
// Rows with an infinity or a NaN give NaN.
//
// One 128 x 64 output tile per CTA: eight accumulators of 64 columns fill the
// 512 tensor-memory columns.  A stage is 32 K values of all eight digits of
// both operands (96 KB, 64-byte swizzle rows), two stages in flight, one
// thread issues the MMAs (72 per stage, ~2300 clocks of tensor pipe against
// ~2000 clocks of L2 traffic).  Outer blocks are 64 pivots wide: the rank-kb
// steps inside the slab stay on the FP64 pipe, 8 m w flops per pivot, and from
// interior blocks of TC64_INNER_MIN on only those inside the 16-column panel:
// the block's other columns are exchanged here too, panel by panel.
//
// Factorization of the 256 x 256 P2 Helmholtz matrix in complex128: 560 ms with
// the rank-kb sweep over whole fronts (284 ms of updates), 305 ms with 64-pivot
// blocks exchanged here, 232 ms with the panels' exchanges as well and the
// panels over clusters (panel_cluster_kernel).  The epilogue does not overlap a
// tile's MMAs (the accumulators fill the tensor memory) and was over half of its
// ~31,000 clocks: front entries loaded eight columns at a time after the MMAs and
// four FP64 instructions per element.  With the entries loaded while the MMAs run
// and three instructions, all launches of this kernel in that factorization take
// 25.7 ms instead of 41.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cstdlib>
#include <vector>

#include "driver.h"
#include "factor.cuh"
#include "tcgen05.cuh"

namespace ndhss {
namespace {

constexpr int D64 = 8;                         // digits per operand
constexpr int T64_M = 128, T64_N = 64;         // output tile (real rows, columns)
constexpr int T64_BK = 32;                     // K values per stage: one 64-byte swizzle row
constexpr int T64_STAGES = 2;
constexpr int T64_THREADS = 320;               // warps 0-7 epilogue, 8 loads, 9 issues MMAs
constexpr uint32_t T64_A_BYTES = T64_M * T64_BK * 2, T64_B_BYTES = T64_N * T64_BK * 2;
constexpr uint32_t T64_STAGE_BYTES = D64 * (T64_A_BYTES + T64_B_BYTES);
constexpr uint32_t T64_TMEM_COLS = D64 * T64_N;
constexpr size_t T64_SMEM = (size_t)T64_STAGES * T64_STAGE_BYTES + 1024;
constexpr int NONFINITE = 1 << 20;             // row exponent of a row with an infinity or a NaN
static_assert(T64_TMEM_COLS == 512, "the eight accumulators fill the tensor memory");

// One front's part of an exchange: pivots [k0, k0 + w), nb columns from column
// j0 on (the pivots skipped), first packed row and first row exponent of its
// operands (A: m rows, then B: nb columns).
struct Front64 {
    int64_t foff, row0;
    int32_t m, w, nb, e0;
};
// The exchange of one front (as TcJob of tcgemm.cu): digit s of A starts at
// packed row a_row + s a_pstride, of B at b_row + s b_pstride.
struct Job64 {
    int32_t a_row, a_pstride, b_row, b_pstride;
    int32_t M, N, K, w;
    int64_t out;
    int32_t ldo, ea, eb, pad;
};
// front column of the exchange's column r
__device__ __forceinline__ int64_t col_of(int64_t r, int j0, int k0, int w) {
    const int64_t j = j0 + r;
    return j < k0 ? j : j + w;
}
// K values of a packed operand row for pivot blocks up to KW wide (one stage at least)
template <typename T, int KW>
constexpr int packed_k() { return (Tr<T>::cplx ? 2 : 1) * KW < T64_BK ? T64_BK : (Tr<T>::cplx ? 2 : 1) * KW; }

// ---------------------------------------------------------------- pack
// v 2^lev as an integer X: v 2^lev = X 2^(E - 1084), |X| < 2^62, E the largest
// levelled exponent of the row (level_exp)
__device__ __forceinline__ int64_t to_fixed(double v, int lev, int E) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int f = (int)((b >> 52) & 0x7ff);
    const uint64_t mant = (b & 0xfffffffffffffull) | (f ? 1ull << 52 : 0ull);
    const int sh = min(9, 9 - (E - max(f, 1) - lev));       // 9 at most but for zeros
    const uint64_t x = sh >= 0 ? mant << sh : sh > -55 ? (mant + (1ull << (-sh - 1))) >> -sh : 0ull;
    return (b >> 63) ? -(int64_t)x : (int64_t)x;
}
// exponent field of v 2^lev, subnormals counting as field 1; INT_MIN for zero,
// NONFINITE for an infinity or a NaN
__device__ __forceinline__ int level_exp(double v, int lev) {
    const int f = (int)((__double2hiint(v) >> 20) & 0x7ff);
    return v == 0.0 ? INT_MIN : f == 0x7ff ? NONFINITE : max(f, 1) + lev;
}
__device__ __forceinline__ int level_exp(c128 v, int lev) { return max(level_exp(v.x, lev), level_exp(v.y, lev)); }

// The powers of two s_q that level the pivots of an exchange (top of the file)
// into lev, by a CTA of 256 threads.  Every packing CTA forms them itself (64 KB
// to read from L2 at most, beside its own 32 KB tile and 100 KB of digits): a
// launch of its own for them took 7 us, 19 -> 26 per exchange.
template <int KW> struct LevelSmem {
    int ex[KW][KW + 1];
    int rmax[KW];
};
template <typename T, int KW>
__device__ __forceinline__ void pivot_levels(const T* __restrict__ front, const Front64& P, int k0, LevelSmem<KW>& S, int* lev) {
    const int w = P.w, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T* D = front + P.foff + (int64_t)k0 * P.m + k0;
    for (int q = threadIdx.x; q < w * w; q += 256) S.ex[q % w][q / w] = level_exp(D[(int64_t)(q / w) * P.m + q % w], 0);
    __syncthreads();
    for (int p = warp; p < w; p += 8) {
        int r = INT_MIN;
        for (int q = lane; q < w; q += 32) r = max(r, S.ex[p][q]);
        r = __reduce_max_sync(0xffffffffu, r);
        if (lane == 0) S.rmax[p] = r;
    }
    __syncthreads();
    for (int q = warp; q < w; q += 8) {
        int s = INT_MAX;
        for (int p = lane; p < w; p += 32)
            if (S.ex[p][q] != INT_MIN) s = min(s, S.rmax[p] - S.ex[p][q]);
        s = __reduce_min_sync(0xffffffffu, s);
        if (lane == 0) lev[q] = s == INT_MAX ? 0 : min(s, 4096);
    }
}

// the low digit of x (-128 .. 127) split off
__device__ __forceinline__ float next_digit(int64_t& x, bool last) {
    const int d = last ? (int)x : (int)(signed char)(x & 0xff);
    x = (x - d) >> 8;
    return (float)d;
}

// One CTA per 32 logical rows of one operand of one front (blockIdx.y): the A
// rows (pivot columns, i < m: M'(i, k0 + q)) come first, then the B rows
// (columns of the exchange: -M(k0 + q, column)).  LPR lanes take a row, over
// the pivots; pivots from w on are zeros.
template <typename T, int KW>
__global__ void __launch_bounds__(256)
tc64_pack_kernel(const Front64* __restrict__ fronts, const T* __restrict__ front, int k0, int j0,
                 __nv_bfloat16* __restrict__ packed, int32_t* __restrict__ rexp) {
    constexpr bool CPLX = Tr<T>::cplx;
    constexpr int CX = CPLX ? 2 : 1;
    constexpr int Kp = packed_k<T, KW>(), KL = Kp / CX;      // packed values and entries of a row
    constexpr int LPR = KL < 32 ? KL : 32, UL = KL / LPR, RW = 32 / LPR;
    // the levels' scratch, then the tile
    constexpr size_t TS = sizeof(T) * 32 * (KL + 1);
    __shared__ __align__(16) unsigned char sm[TS > sizeof(LevelSmem<KW>) ? TS : sizeof(LevelSmem<KW>)];
    __shared__ int s_lev[KW];
    T (*ts)[KL + 1] = reinterpret_cast<T(*)[KL + 1]>(sm);
    const Front64 P = fronts[blockIdx.y];
    const int m = P.m, w = P.w, nb = P.nb;
    const int rt_a = (m + 31) / 32, rt_b = (nb + 31) / 32;
    if ((int)blockIdx.x >= rt_a + rt_b) return;
    const bool is_a = (int)blockIdx.x < rt_a;
    const int r0 = ((int)blockIdx.x - (is_a ? 0 : rt_a)) * 32, rows = is_a ? m : nb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane / LPR, ll = lane % LPR;
    const T* F = front + P.foff;
    pivot_levels<T, KW>(front, P, k0, *reinterpret_cast<LevelSmem<KW>*>(sm), s_lev);
    __syncthreads();
    if (is_a) {
        for (int l = warp; l < KL; l += 8) {
            const int r = r0 + lane;
            ts[lane][l] = (r < rows && l < w) ? F[(int64_t)(k0 + l) * m + r] : zero<T>();
        }
    } else {
        for (int rr = RW * warp + sub; rr < 32; rr += 8 * RW) {
            const int r = r0 + rr;
            const int64_t j = col_of(r, j0, k0, w);
            for (int l = ll; l < KL; l += LPR)
                ts[rr][l] = (r < rows && l < w) ? -F[j * m + k0 + l] : zero<T>();
        }
    }
    __syncthreads();
    const int64_t a_rows = (int64_t)CX * m;
    const unsigned mask = RW == 1 ? 0xffffffffu : 0xffffu << (16 * sub);
    static_assert(RW == 1 || LPR == 16, "whole or half warps");
    int lv[UL];
#pragma unroll
    for (int u = 0; u < UL; ++u) {
        const int l = ll + LPR * u;
        const int s = l < w ? s_lev[l] : 0;
        lv[u] = is_a ? s : -s;
    }
    for (int rr = RW * warp + sub; rr < 32; rr += 8 * RW) {
        const int r = r0 + rr;
        T v[UL];
        int E = INT_MIN;
#pragma unroll
        for (int u = 0; u < UL; ++u) {
            v[u] = ts[rr][ll + LPR * u];
            E = max(E, level_exp(v[u], lv[u]));
        }
        E = __reduce_max_sync(mask, E);
        if (r >= rows) continue;
        if (E == INT_MIN) E = 1023;                    // a row of zeros
        const bool bad = E == NONFINITE;
        if (ll == 0) rexp[P.e0 + (is_a ? 0 : m) + r] = bad ? NONFINITE : E;
#pragma unroll
        for (int u = 0; u < UL; ++u) {
            const int l = ll + LPR * u;
            if constexpr (CPLX) {
                int64_t xr = bad ? 0 : to_fixed(v[u].x, lv[u], E), xi = bad ? 0 : to_fixed(v[u].y, lv[u], E);
                __nv_bfloat162* o0 = reinterpret_cast<__nv_bfloat162*>(
                    packed + (is_a ? P.row0 + 2 * (int64_t)r : P.row0 + D64 * a_rows + r) * Kp + 2 * l);
                const int64_t ps = (is_a ? a_rows : nb) * (int64_t)(Kp / 2);
#pragma unroll
                for (int s = D64 - 1; s >= 0; --s) {
                    const float dr = next_digit(xr, s == 0), di = next_digit(xi, s == 0);
                    if (is_a) {
                        o0[s * ps] = __floats2bfloat162_rn(dr, -di);
                        o0[s * ps + Kp / 2] = __floats2bfloat162_rn(di, dr);
                    } else {
                        o0[s * ps] = __floats2bfloat162_rn(dr, di);
                    }
                }
            } else {
                int64_t x = bad ? 0 : to_fixed(v[u], lv[u], E);
                __nv_bfloat16* o0 = packed + (is_a ? P.row0 + r : P.row0 + D64 * a_rows + r) * Kp + l;
                const int64_t ps = (is_a ? a_rows : nb) * (int64_t)Kp;
#pragma unroll
                for (int s = D64 - 1; s >= 0; --s) o0[s * ps] = __float2bfloat16_rn(next_digit(x, s == 0));
            }
        }
    }
}

// ---------------------------------------------------------------- GEMM
// Descriptor of a K-major operand tile with 64-byte swizzle: 8-row groups 512
// bytes apart (stride byte offset), the leading byte offset unused, layout
// type 4.
constexpr uint32_t SW64_HI = (512u >> 4) | 1u << 14 | 4u << 29;
__device__ __forceinline__ uint32_t sw64_lo(uint32_t saddr) { return (saddr >> 4) | 1u << 16; }

// (hi + lo 2^-32) 2^(f - 1023) for integers |hi|, |lo| < 2^51, rounded once, in
// two FP64 instructions: x + 1.5 2^52 is written down as bits for both, the
// first FMA takes both constants off again (hi - 1.5 2^20 is an integer below
// 2^52: exact)
__device__ __forceinline__ double ints_scaled(long long hi, long long lo, int f) {
    const double s = __longlong_as_double((long long)f << 52), s32 = __longlong_as_double((long long)(f - 32) << 52);
    // -(1.5 2^52 + 1.5 2^20) 2^(f - 1023)
    const double c = __longlong_as_double(
        (long long)((1ull << 63) | ((unsigned long long)(f + 52) << 52) | (0x8000000000000ull + 0x180000ull)));
    const double h = fma(__longlong_as_double(hi + 0x4338000000000000ll), s, c);
    return fma(__longlong_as_double(lo + 0x4338000000000000ll), s32, h);
}

template <typename T>
__global__ void __launch_bounds__(T64_THREADS, 1)
tc64_gemm_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
                 const Job64* __restrict__ jobs, const int2* __restrict__ tiles, const int32_t* __restrict__ rexp,
                 int k0, int j0, T* __restrict__ front, DevStatus* status) {
    constexpr bool CPLX = Tr<T>::cplx;
    extern __shared__ unsigned char dsm[];
    __shared__ __align__(8) uint64_t full_bar[T64_STAGES];
    __shared__ __align__(8) uint64_t empty_bar[T64_STAGES];
    __shared__ __align__(8) uint64_t acc_bar;
    __shared__ uint32_t tmem_holder;
    __shared__ int s_abort;
    __shared__ int s_eb[T64_N];

    const int2 tl = tiles[blockIdx.x];
    const Job64 J = jobs[tl.x];
    const int tiles_m = (J.M + T64_M - 1) / T64_M;
    const int m0 = (tl.y % tiles_m) * T64_M, n0 = (tl.y / tiles_m) * T64_N;
    const int nk = (J.K + T64_BK - 1) / T64_BK;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t base = (tc::smem_u32(dsm) + 1023u) & ~1023u;
    auto tileA = [&](int s, int p) { return base + (uint32_t)s * T64_STAGE_BYTES + (uint32_t)p * T64_A_BYTES; };
    auto tileB = [&](int s, int p) {
        return base + (uint32_t)s * T64_STAGE_BYTES + D64 * T64_A_BYTES + (uint32_t)p * T64_B_BYTES;
    };

    if (tid == 0) {
        for (int s = 0; s < T64_STAGES; ++s) {
            tc::mbar_init(&full_bar[s], 1);
            tc::mbar_init(&empty_bar[s], 1);
        }
        tc::mbar_init(&acc_bar, 1);
        s_abort = 0;
    }
    if (tid < T64_N) s_eb[tid] = n0 + tid < J.N ? rexp[J.eb + n0 + tid] : 1;
    if (warp == 0) tc::tmem_alloc(&tmem_holder, T64_TMEM_COLS);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_holder;

    int issued = 0;                                   // producer: stages loaded
    if (tid == 256) {
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % T64_STAGES;
            if (kb >= T64_STAGES && !tc::bar_wait(&empty_bar[s], ((kb / T64_STAGES) & 1) ^ 1)) {
                atomicExch(&s_abort, 1);
                break;
            }
            if (*(volatile int*)&s_abort) break;
            tc::bar_expect_tx(&full_bar[s], T64_STAGE_BYTES);
            for (int p = 0; p < D64; ++p) {
                tc::tma_load_2d(tileA(s, p), &amap, kb * T64_BK, J.a_row + p * J.a_pstride + m0, &full_bar[s]);
                tc::tma_load_2d(tileB(s, p), &bmap, kb * T64_BK, J.b_row + p * J.b_pstride + n0, &full_bar[s]);
            }
            issued = kb + 1;
        }
    } else if (tid == 288) {
        const uint32_t idesc = tc::idesc_bf16(T64_M, T64_N);
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % T64_STAGES;
            if (!tc::bar_wait(&full_bar[s], (kb / T64_STAGES) & 1)) {
                atomicExch(&s_abort, 1);
                break;
            }
            tc::fence_after();
            const uint32_t la = sw64_lo(tileA(s, 0)), lb = sw64_lo(tileB(s, 0));
#pragma unroll
            for (int kk = 0; kk < T64_BK / 16; ++kk) {
#pragma unroll
                for (int g = 0; g < D64; ++g)
#pragma unroll
                    for (int p = 0; p <= g; ++p)
                        tc::mma_f16(tmem + (uint32_t)g * T64_N, la + (uint32_t)p * (T64_A_BYTES >> 4) + 2u * kk,
                                    lb + (uint32_t)(g - p) * (T64_B_BYTES >> 4) + 2u * kk, SW64_HI, idesc,
                                    (kk || p || kb) ? 1u : 0u);
            }
            tc::commit(&empty_bar[s]);
        }
        tc::commit(&acc_bar);                         // fires once every MMA issued above has retired
        tc::bar_wait(&acc_bar, 0);
    } else if (warp < 8) {
        // epilogue: warp w takes the tile's rows 32 (w % 4) .. + 31 and columns
        // 32 (w / 4) .. + 31, eight columns of all eight accumulators at a time
        const int rr = (warp & 3) * 32 + lane, cb = (warp >> 2) * 32;
        const int64_t grow = m0 + rr;
        const bool rowok = grow < J.M;
        const int64_t crow = CPLX ? grow >> 1 : grow;
        const bool piv = crow >= k0 && crow < k0 + J.w;
        const int ea = rowok ? rexp[J.ea + crow] : 1;
        T* out = front + J.out + crow;
        // the front's entries of this thread (complex: even lanes hold Re, odd
        // lanes Im of complex row grow / 2; even lanes write the even columns, odd
        // lanes the odd ones), read while the MMAs run (real: half of them, the
        // others as these are used; all 32 spill)
        constexpr int NV = CPLX ? 4 : 8;              // per eight columns
        constexpr int NO = 16;                        // held at a time
        T old[NO];
        auto entry = [&](int q) -> T* {
            const int64_t col = n0 + cb + (CPLX ? 2 * q + (lane & 1) : q);
            return rowok && col < J.N ? out + col_of(col, j0, k0, J.w) * J.ldo : nullptr;
        };
#pragma unroll
        for (int q = 0; q < NO; ++q) {
            const T* ptr = entry(q);
            old[q] = (ptr && !piv) ? *ptr : zero<T>();
        }
        const bool ok = tc::bar_wait(&acc_bar, 0);
        tc::fence_after();
        if (!ok || *(volatile int*)&s_abort) {
            if (lane == 0 && atomicCAS(&status->code, 0, (int)NDHSS_ERR_TIMEOUT) == 0) status->node = -1;
        } else {
            const uint32_t t0 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cb;
#pragma unroll
            for (int c0 = 0; c0 < 32; c0 += 8) {
                if (n0 + cb + c0 >= J.N) break;
                uint32_t v[D64][8];
#pragma unroll
                for (int g = 0; g < D64; ++g) tc::tmem_ld8_async(t0 + (uint32_t)(g * T64_N + c0), v[g]);
                tc::tmem_wait_ld();
#pragma unroll
                for (int g = 0; g < D64; ++g) tc::tmem_landed(v[g]);
                double val[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    int d[D64];
#pragma unroll
                    for (int g = 0; g < D64; ++g) d[g] = __float2int_rn(__uint_as_float(v[g][u]));
                    // |d_0| <= 2^19, |d_1| <= 2^21, |d_2| <= 2^22.6, |d_3| <= 2^23: the pairs fit 32 bits
                    const long long hi = (long long)(d[0] * 256 + d[1]) * 65536 + (d[2] * 256 + d[3]);
                    const long long lo = ((long long)d[4] * 256 + d[5]) * 65536 + ((long long)d[6] * 256 + d[7]);
                    // V = hi 2^(ea + eb - 36) + lo 2^(ea + eb - 68) with unbiased row
                    // exponents (field - 1022).  ints_scaled wants its powers of two
                    // inside the normal range; what a product below 2^-954 or above
                    // 2^1003 lacks (a matrix of entries near 2^-960 or 2^960) is put
                    // on afterwards, rounded once (a shift beyond 2^+-1022 gives zero
                    // or infinity either way)
                    const int e = ea + s_eb[cb + c0 + u];
                    const int f = min(max(e - 1057, 33), 1990);
                    val[u] = ints_scaled(hi, lo, f);
                    const int shift = e - 1057 - f;
                    if (shift != 0)
                        val[u] *= __longlong_as_double(e >= NONFINITE ? 0x7ff8000000000000ll
                                                                      : (long long)(1023 + min(max(shift, -1022), 1023)) << 52);
                }
#pragma unroll
                for (int h = 0; h < NV; ++h) {
                    T nv;
                    if constexpr (CPLX) {
                        const int odd = lane & 1;
                        const double send = odd ? val[2 * h] : val[2 * h + 1];
                        const double recv = __shfl_xor_sync(0xffffffffu, send, 1);
                        nv.x = odd ? recv : val[2 * h];
                        nv.y = odd ? val[2 * h + 1] : recv;
                    } else {
                        nv = val[h];
                    }
                    const int q = c0 / 8 * NV + h;
                    if (T* ptr = entry(q)) *ptr = old[q % NO] + nv;
                    if (q + NO < 4 * NV) {
                        const T* ptr = entry(q + NO);
                        old[q % NO] = (ptr && !piv) ? *ptr : zero<T>();
                    }
                }
            }
        }
    }
    // leave only once every copy issued by this CTA has landed
    if (tid == 256) {
        for (int kb = max(0, issued - T64_STAGES); kb < issued; ++kb)
            if (!tc::bar_wait(&full_bar[kb % T64_STAGES], (kb / T64_STAGES) & 1)) break;
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, T64_TMEM_COLS);
}

// ---------------------------------------------------------------- without packed operands
// The exchange in float64 on the CUDA cores, straight from the front: a CTA
// takes the columns [16 blockIdx.x, + 16) of front blockIdx.y, holds -M(P, :) of
// them in shared memory (no other CTA reads or writes these columns) and walks
// over the rows, a row per thread.  Taken when there is no memory for packed
// operands; bound by the FP64 pipe (2 DFMA per clock and SM).
constexpr int T64_PC = 16;
template <typename T>
__global__ void __launch_bounds__(256)
tc64_plain_kernel(const Front64* __restrict__ fronts, T* __restrict__ front, int k0, int j0) {
    __shared__ T bs[TC64_KB2][T64_PC];
    const Front64 P = fronts[blockIdx.y];
    const int m = P.m, w = P.w, c0 = (int)blockIdx.x * T64_PC;
    if (c0 >= P.nb) return;
    T* F = front + P.foff;
    for (int q = threadIdx.x; q < w * T64_PC; q += 256) {
        const int l = q % w, c = q / w;
        bs[l][c] = c0 + c < P.nb ? -F[col_of(c0 + c, j0, k0, w) * m + k0 + l] : zero<T>();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += 256) {
        T acc[T64_PC];
#pragma unroll
        for (int c = 0; c < T64_PC; ++c) acc[c] = zero<T>();
        for (int l = 0; l < w; ++l) {
            const T a = F[(int64_t)(k0 + l) * m + i];
#pragma unroll
            for (int c = 0; c < T64_PC; ++c) acc[c] = fmac(a, bs[l][c], acc[c]);
        }
        const bool piv = i >= k0 && i < k0 + w;
#pragma unroll
        for (int c = 0; c < T64_PC; ++c) {
            if (c0 + c >= P.nb) break;
            T* ptr = F + col_of(c0 + c, j0, k0, w) * m + i;
            *ptr = piv ? acc[c] : *ptr + acc[c];
        }
    }
}

// Packed operands of one batch of fronts, and no more: they come on top of the
// factor itself (6 KB per row of a complex128 front and 64 pivots, more than the
// front's own 16 m bytes up to m = 384), and a batch of this size already has
// thousands of tiles.  NDHSS_TC64_SCRATCH sets another limit in bytes (0: no
// packed operands at all).
int64_t scratch_limit() {
    const char* e = std::getenv("NDHSS_TC64_SCRATCH");
    return e ? std::max<int64_t>(0, std::atoll(e)) : (int64_t)1 << 30;
}

template <typename T, int KW>
ndhss_status tc64_block_run(FactorData& F, const std::vector<int>& nodes, int k0, int width, int j0, int j1,
                            DevStatus* d_status, cudaStream_t st) {
    constexpr int CX = Tr<T>::cplx ? 2 : 1;
    constexpr int64_t Kp = packed_k<T, KW>();
    NDHSS_CUDA_TRY(cudaFuncSetAttribute(tc64_gemm_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T64_SMEM));
    // fronts in batches whose packed operands stay below the limit and the tensor
    // map's 2^31 rows; a batch that finds no memory is halved, and a front that
    // finds none by itself goes without
    int64_t max_rows = std::min<int64_t>(((int64_t)1 << 31) - 4096, scratch_limit() / (Kp * 2));
    size_t at = 0;
    while (at < nodes.size()) {
        std::vector<Front64> fr;
        std::vector<Job64> jobs;
        std::vector<int2> tiles;
        int64_t rows = 0, nexp = 0, need_max = 0;
        int rt_max = 0, nb_max = 0;
        const size_t first = at;
        bool packed = true;
        for (; at < nodes.size(); ++at) {
            const int s = nodes[at];
            const int mi = F.m_i(s), m = mi + F.m_b(s);
            if (mi <= k0) continue;
            const int w = std::min(width, mi - k0), nb = std::min(j1 == INT_MAX ? m : mi, j1) - j0 - w;
            if (nb <= 0) continue;                         // the pivots are all of the columns
            const int64_t a_rows = (int64_t)CX * m, need = D64 * (a_rows + nb);
            if (!fr.empty() && (fr.size() >= 65535 || packed != (need <= max_rows) || (packed && rows + need > max_rows))) break;
            packed = need <= max_rows;
            fr.push_back({F.foff[s], rows, m, w, nb, (int32_t)nexp});
            nb_max = std::max(nb_max, nb);
            if (!packed) continue;
            const Job64 j{(int32_t)rows, (int32_t)a_rows, (int32_t)(rows + D64 * a_rows), nb, (int32_t)a_rows, nb, CX * w,
                          w, F.foff[s], m, (int32_t)nexp, (int32_t)(nexp + m), 0};
            rows += need;
            need_max = std::max(need_max, need);
            nexp += m + nb;
            const int id = (int)jobs.size();
            jobs.push_back(j);
            const int nt = ((j.M + T64_M - 1) / T64_M) * ((j.N + T64_N - 1) / T64_N);
            for (int q = 0; q < nt; ++q) tiles.push_back(make_int2(id, q));
            rt_max = std::max(rt_max, (m + 31) / 32 + (nb + 31) / 32);
        }
        if (fr.empty()) break;
        // one pool allocation: packed digits, row exponents, then the tables
        auto r256 = [](size_t b) { return (b + 255) / 256 * 256; };
        const size_t packed_bytes = r256((size_t)rows * Kp * 2), exp_bytes = packed ? r256((size_t)nexp * 4) : 0;
        const size_t fr_bytes = r256(fr.size() * sizeof(Front64)), job_bytes = r256(jobs.size() * sizeof(Job64));
        const size_t t_bytes = r256(tiles.size() * sizeof(int2));
        std::vector<unsigned char> tab(fr_bytes + job_bytes + t_bytes);
        std::copy_n(reinterpret_cast<const unsigned char*>(fr.data()), fr.size() * sizeof(Front64), tab.data());
        std::copy_n(reinterpret_cast<const unsigned char*>(jobs.data()), jobs.size() * sizeof(Job64), tab.data() + fr_bytes);
        std::copy_n(reinterpret_cast<const unsigned char*>(tiles.data()), tiles.size() * sizeof(int2),
                    tab.data() + fr_bytes + job_bytes);
        unsigned char* buf = nullptr;
        if (pool_malloc_async((void**)&buf, packed_bytes + exp_bytes + tab.size(), st) != cudaSuccess) {
            cudaGetLastError();
            if (!packed) return set_error(NDHSS_ERR_OOM, "ndhss_factor: %zu bytes of front tables", tab.size());
            max_rows = fr.size() > 1 ? std::max(rows / 2, need_max) : rows - 1;
            at = first;
            continue;
        }
        int32_t* d_exp = reinterpret_cast<int32_t*>(buf + packed_bytes);
        unsigned char* d_tab = buf + packed_bytes + exp_bytes;
        const Front64* d_fr = reinterpret_cast<const Front64*>(d_tab);
        T* front = static_cast<T*>(F.d_front);
        ndhss_status rc = NDHSS_OK;
        if (cudaMemcpyAsync(d_tab, tab.data(), tab.size(), cudaMemcpyHostToDevice, st) != cudaSuccess)
            rc = set_error(NDHSS_ERR_CUDA, "ndhss_factor: upload of the tensor-core tables failed");
        auto launched = [&](const char* name) {
            const cudaError_t e = cudaGetLastError();
            note_launches(1);
            ++F.launches;
            if (e != cudaSuccess) rc = set_error(NDHSS_ERR_CUDA, "launch of %s failed: %s", name, cudaGetErrorString(e));
        };
        if (!packed) {
            if (rc == NDHSS_OK) {
                tc64_plain_kernel<T><<<dim3((unsigned)((nb_max + T64_PC - 1) / T64_PC), (unsigned)fr.size()), 256, 0, st>>>(
                    d_fr, front, k0, j0);
                launched("tc64_plain_kernel");
            }
            cudaFreeAsync(buf, st);
            if (rc != NDHSS_OK) return rc;
            for (const auto& f : fr) F.update_flops += (Tr<T>::cplx ? 8.0 : 2.0) * (double)f.m * (double)f.nb * f.w;
            continue;
        }
        CUtensorMap amap, bmap;
        const cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)Kp * 2};
        const cuuint32_t abox[2] = {(cuuint32_t)T64_BK, (cuuint32_t)T64_M}, bbox[2] = {(cuuint32_t)T64_BK, (cuuint32_t)T64_N};
        const cuuint32_t estr[2] = {1, 1};
        if (rc == NDHSS_OK)
            rc = drv_encode_tiled(&amap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, buf, dims, strides, abox, estr,
                                  CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (rc == NDHSS_OK)
            rc = drv_encode_tiled(&bmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, buf, dims, strides, bbox, estr,
                                  CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (rc == NDHSS_OK) {
            tc64_pack_kernel<T, KW><<<dim3((unsigned)rt_max, (unsigned)fr.size()), 256, 0, st>>>(
                d_fr, front, k0, j0, reinterpret_cast<__nv_bfloat16*>(buf), d_exp);
            launched("tc64_pack_kernel");
        }
        if (rc == NDHSS_OK) {
            tc64_gemm_kernel<T><<<(unsigned)tiles.size(), T64_THREADS, T64_SMEM, st>>>(
                amap, bmap, reinterpret_cast<const Job64*>(d_tab + fr_bytes),
                reinterpret_cast<const int2*>(d_tab + fr_bytes + job_bytes), d_exp, k0, j0, front, d_status);
            launched("tc64_gemm_kernel");
        }
        cudaFreeAsync(buf, st);
        if (rc != NDHSS_OK) return rc;
        for (const auto& f : fr) F.tc_flops += (Tr<T>::cplx ? 8.0 : 2.0) * (double)f.m * (double)f.nb * f.w;
    }
    return NDHSS_OK;
}

}  // namespace

// Complex fronts: blocks from 24 interior unknowns on, panels from 64 on.  A
// rank-16 update of a 64 x 64 tile holds an SM's FP64 pipe for 64 us there, more
// than the launches of an exchange cost (some 20 us).  Real fronts: 16 us, so the
// exchanges pay only where a level has more tiles than SMs.  A level whose rank-16
// updates fill less than two waves stays on the CUDA cores unless its pivots go in
// several blocks (96 unknowns), and the panels are exchanged in blocks whose
// slabs, one 64-column tile per 64 rows, fill one and a half.
TcPath tc64_front_path(const FactorData& F, const std::vector<int>& nodes, int64_t mi_max, bool forced) {
    if (F.vtype == NDHSS_C128 || forced) return {true, mi_max >= TC64_INNER_MIN};
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t slab = 0, all = 0;                      // 64 x 64 tiles of a slab's and of a whole level's update
    for (int s : nodes) {
        const int64_t t = F.m_i(s) > 0 ? (F.m_i(s) + F.m_b(s) + 63) / 64 : 0;
        slab += t;
        all += t * t;
    }
    const bool blocks = mi_max >= 96 || all >= 2 * sms;
    return {blocks, blocks && mi_max >= TC64_INNER_MIN && 2 * slab >= 3 * sms};
}

ndhss_status tc64_block_exchange(FactorData& F, const std::vector<int>& nodes, int k0, int width, int j0, int j1,
                                 DevStatus* d_status, cudaStream_t st) {
    // the packed width by the call's widest pivot block
    int wmax = 0;
    for (int s : nodes) wmax = std::max(wmax, std::min(width, F.m_i(s) - k0));
    auto run = [&](auto v) {
        using T = decltype(v);
        return wmax <= TC64_KB1 ? tc64_block_run<T, TC64_KB1>(F, nodes, k0, width, j0, j1, d_status, st)
               : wmax <= 32     ? tc64_block_run<T, 32>(F, nodes, k0, width, j0, j1, d_status, st)
                                : tc64_block_run<T, TC64_KB2>(F, nodes, k0, width, j0, j1, d_status, st);
    };
    return F.vtype == NDHSS_C128 ? run(c128{}) : run(double{});
}

}  // namespace ndhss
