// bv_fix_tile.cuh -- 16 x 16 tiles of the fixed-point Cholesky factorisation, shared by the
// block kernel (bv_fix_ll.cu) and the exact likelihood (bv_exact.cu): the diagonal tile's
// factor, the rows below it, their digits, and the update C -= L_I L_J^T on the tensor cores.
//
// Tiles are stored in the order in which a warp's accumulator fragment holds them (lane 4 g +
// t: rows g, g + 8, columns 2 t, 2 t + 1 of either half), 16 bytes a lane: every access of the
// update is a conflict-free 128-bit one.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "bv_device.cuh"
#include "bv_fix.cuh"
#include "bv_internal.h"

namespace {

using bvfix::Bal;
using bvfix::Dist;
using bvfix::Fac;

constexpr int kTileB = 2048;   // bytes of a 16 x 16 tile of 64-bit entries
constexpr int kDig = 6;        // digits of a factor entry
constexpr int kLd = 24;            // entries of a diagonal factor's column (16, then zeros)
constexpr int kDigB = kDig * 512;  // bytes of a tile's digits
constexpr int kFail = 1, kOver = 2;  // a thread's findings about the block
// The data row's headroom: |y| / sqrt(D) < 2^-(kYRoom + row_limit(N)) at first, so that a solved entry
// may be 2^kYRoom / 2 of the largest |y| / sqrt(D).  When one is larger, the row is scaled down by
// 2^kYStep, kYMax times at most (beyond any ratio that the pivots leave).
constexpr int kYRoom = 5, kYStep = 8, kYMax = 16;
// A pivot of at most this (2^-54 of the diagonal, below one FP64 rounding of it) counts as not
// positive: what a singular matrix leaves is noise of this size, of either sign.
constexpr int64_t kPivMin = 64;
constexpr int kFixSmemCap = 227 * 1024 - 8192;  // dynamic shared memory beside the tables

// Tile rows of N points and the data row; bytes of the tiles, and of a block's shared memory
// beside them: digits of one panel's rows | diagonal factor | its reciprocal square roots |
// coordinates, y, pivots, z row.
__host__ __device__ inline int fix_tiles(int nmax) { return (nmax + 16) >> 4; }
__host__ __device__ inline size_t fix_tile_bytes(int nmax) {
    const size_t T = fix_tiles(nmax);
    return T * (T + 1) / 2 * kTileB;
}
__host__ __device__ inline size_t fix_work_bytes(int nmax, int d) {
    const size_t T = fix_tiles(nmax);
    return (T - 1) * kDigB + (16 * kLd + 16) * sizeof(int4) + 16 * 16 + (((size_t)(d + 3) * nmax * 8 + 15) & ~(size_t)15);
}

__device__ __forceinline__ int ftile(int I, int J) { return ((I * (I + 1)) >> 1) + J; }

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint2& a0, const uint2& a1, const uint2& b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0.x), "r"(a1.x), "r"(a0.y), "r"(a1.y), "r"(b.x), "r"(b.y));
}

__device__ __forceinline__ int64_t shfl64(int64_t v, int src) { return (int64_t)__shfl_sync(0xffffffffu, (long long)v, src); }

// x = v rs in factor units from v in matrix units and rs = r 2^(e-62), rounded: v 2^e 2^60 r 2^-62,
// with |v| 2^e <= 1 / (r 2^-62).
__device__ __forceinline__ int64_t fix_scale(int64_t v, Bal r, int e) {
    const Bal b = bvfix::bal((int64_t)((uint64_t)v << (e + 1)));
    const int64_t mid = bvfix::smad(b.h, r.l, bvfix::smad(b.l, r.h, 0x80000000ll));
    return bvfix::smad(b.h, r.h, mid >> 32);
}

// The panel's reciprocal square roots, by column.
struct __align__(16) FixRs {
    Bal r;
    int e;
    int pad;
};

// A solved data entry x = v 2^e r, r in [1, 2), is below 2^-lim when v 2^e is below half of that.
__device__ __forceinline__ bool out_of_range(int64_t v, int e, int lim) { return ((v < 0 ? -v : v) >> (59 - lim - e)) != 0; }

// The diagonal factor in shared memory: column c's entries L[j][c] at c kLd + j.  The loops
// below read past j = 15, where the row loop needs zeros.

// The warp that factors the diagonal tile tells the warps that solve the rows below of every
// finished pair of columns through an mbarrier in shared memory (eight of them, one arrival a
// phase, one phase a panel; the hardware's named barriers are too few for eight CTAs an SM).
__device__ __forceinline__ void pair_ready(uint64_t* mb, int lane) {
    if (lane == 0)
        asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"((uint32_t)__cvta_generic_to_shared(mb)) : "memory");
}
// False when the wait ran out (it is bounded: about 2^20 polls).
__device__ __forceinline__ bool pair_wait(uint64_t* mb, uint32_t parity) {
    const uint32_t ad = (uint32_t)__cvta_generic_to_shared(mb);
    for (int it = 0; it < (1 << 20); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(ad), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// Factor the diagonal tile of a panel (columns k0 .. k0 + nc - 1), one warp: lane r + 16 h
// holds row r, columns of parity h, and the row's diagonal entry.  What bounds it is the chain
// from one pivot to the next, which needs the diagonal entry alone (d -= x^2, no exchange; a
// whole-number product, which has no conversions in the chain and no rounding of the cross term);
// the updates of the other columns by column c are done in the shadow of column c + 1's
// reciprocal square root.  Two columns a turn and the registers moved down by one, so that the
// code stays small: unrolled over the 16 columns, this and the row loop below ran at the rate
// of instruction fetches (10,000 clocks a tile and a row pass).  The pivots and the data row's
// entries (row N, if it lies in the tile) are stored.  PART (the one-warp CTAs, in which nobody waits):
// a last panel's columns beyond nc are left out; elsewhere the loop's known length is worth more (1.3%
// at N = 47).
template <bool PART>
__device__ __forceinline__ void fix_diag(const longlong2* tile, int nc, int k0, int N, int lim, int lane, int4* Ld, FixRs* rsv,
                                         int64_t* piv, int64_t* zrow, uint64_t* mb, int& flags) {
    const int r = lane & 15, par = lane >> 4;
    int64_t a[8];  // columns 2 (k + q) + par in turn k
    float fc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const longlong2 v = tile[((q >> 2) * 2 + (r >> 3)) * 32 + 4 * (r & 7) + (q & 3)];
        a[q] = par ? v.y : v.x;
        fc[q] = 0.0f;
    }
    int64_t dg;
    {
        const longlong2 v = tile[(r >> 3) * 96 + 4 * (r & 7) + ((r & 7) >> 1)];
        dg = (r & 1) ? v.y : v.x;
    }
    const int ry = N - k0;
    Fac f;
    f.h = 0;
    f.hf = f.lf = 0.0f;
    const int4* lp = Ld;  // the column last factored
    const int kend = PART ? (nc + 1) >> 1 : 8;
#pragma unroll 1
    for (int k = 0; k < kend; ++k) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int c = 2 * k + s;
            const bool on = c < nc;
            const int64_t p0 = shfl64(dg, c);
            const bool bad = on && p0 <= kPivMin;
            const int64_t p = p0 > kPivMin ? p0 : 1;
            const bvfix::Rsq rs = bvfix::rsqrt_fix(p);
            const Bal rb = bvfix::bal(on ? rs.r : 0);
            if (s || k) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {  // (columns already factored, and past the tile: not used again)
                    const int4 l = lp[2 * q + par];
                    bvfix::msub(a[q], fc[q], -f.h, -f.hf, -f.lf, l.x, __int_as_float(l.y), __int_as_float(l.z));
                }
            }
            const int64_t v = shfl64(bvfix::smad(bvfix::f2i(fc[0]), 4, a[0]), r + 16 * s);
            const int64_t x = fix_scale(v, rb, rs.e);
            f = bvfix::fac(x);
            dg = bvfix::sub_square(dg, x, f.h);
            if (par == 0) {
                Ld[c * kLd + r] = make_int4(f.h, __float_as_int(f.hf), __float_as_int(f.lf), 0);
                if (r == ry && on) {
                    zrow[k0 + c] = x;
                    if (out_of_range(v, rs.e, lim)) flags |= kOver;
                }
            }
            if (lane == 0) {
                FixRs o;
                o.r = rb;
                o.e = on ? rs.e : 0;
                o.pad = 0;
                rsv[c] = o;
                if (bad) flags |= kFail;
                if (on) piv[k0 + c] = p;
            }
            __syncwarp();
            lp = Ld + c * kLd + 2 * (k + s);
        }
        if (!PART) pair_ready(mb + k, lane);  // (after the columns' __syncwarp)
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            a[q] = a[q + 1];
            fc[q] = fc[q + 1];
        }
    }
}

// Four columns c0 .. c0 + 3 of one row of the panel, right-looking: a[0 .. W-1] are the
// columns from c0 on; a solved entry goes to the back as the others move down by one.  With
// wait, the columns come in pairs from the warp at work on the diagonal tile.
template <int W>
__device__ __forceinline__ void fix_row4(int64_t* a, float* fc, int c0, const int4* Ld, const FixRs* rsv, bool yrow,
                                         int lim, int64_t* z, int nc, bool wait, uint64_t* mb, uint32_t parity, int& flags) {
#pragma unroll 1
    for (int c = c0; c < c0 + 4; ++c) {
        if (wait && !(c & 1) && !pair_wait(mb + (c >> 1), parity)) flags |= kFail;
        const int64_t v = bvfix::smad(bvfix::f2i(fc[0]), 4, a[0]);
        const FixRs rs = rsv[c];
        const int64_t x = fix_scale(v, rs.r, rs.e);
        const Fac f = bvfix::fac(x);
        const int4* lp = Ld + c * kLd + c;
#pragma unroll
        for (int j = 1; j < W; ++j) {
            const int4 l = lp[j];
            a[j - 1] = a[j];
            fc[j - 1] = fc[j];
            bvfix::msub(a[j - 1], fc[j - 1], -f.h, -f.hf, -f.lf, l.x, __int_as_float(l.y), __int_as_float(l.z));
        }
        a[W - 1] = x;
        fc[W - 1] = 0.0f;
        if (yrow && c < nc) {
            z[c] = x;
            if (out_of_range(v, rs.e, lim)) flags |= kOver;
        }
    }
}

// One row of the panel below the diagonal tile: x L^T = a, then its digits.
__device__ __forceinline__ void fix_row(const longlong2* tile, const int4* Ld, const FixRs* rsv, int r, bool yrow, int lim,
                                        int64_t* z, int nc, bool wait, uint64_t* mb, uint32_t parity, uint32_t* dig, int& flags) {
    const int g = r & 7, rr = r >> 3;
    int64_t a[16];
    float fc[16];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const longlong2 v = tile[((q >> 2) * 2 + rr) * 32 + 4 * g + (q & 3)];
        a[2 * q] = v.x;
        a[2 * q + 1] = v.y;
        fc[2 * q] = fc[2 * q + 1] = 0.0f;
    }
    fix_row4<16>(a, fc, 0, Ld, rsv, yrow, lim, z, nc, wait, mb, parity, flags);   // a: columns 4 .. 15, x of 0 .. 3
    fix_row4<12>(a, fc, 4, Ld, rsv, yrow, lim, z, nc, wait, mb, parity, flags);   // columns 8 .. 15, x of 4 .. 7, 0 .. 3
    fix_row4<8>(a, fc, 8, Ld, rsv, yrow, lim, z, nc, wait, mb, parity, flags);
    fix_row4<4>(a, fc, 12, Ld, rsv, yrow, lim, z, nc, wait, mb, parity, flags);   // x of 12 .. 15, 8 .. 11, 4 .. 7, 0 .. 3
    // digits: x + 512 sum 2^10k has the digits plus 512 in six ten-bit fields; 1024 + field
    // is the FP16 number 0x6400 + field.  Word i of a row: columns 2 i, 2 i + 1 (the order of
    // the columns inside a product's sum is free).
    const uint64_t kBias = 512ull * (1ull | 1ull << 10 | 1ull << 20 | 1ull << 30 | 1ull << 40 | 1ull << 50);
    const __half2 off = __half2half2(__ushort_as_half(0xE600));  // -1536
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
        uint64_t u[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {  // columns 8 q + j
            const int o = 8 + ((j + 4) & 7);
            u[j] = (uint64_t)a[o] + kBias;
            a[o] = a[o - 8];
        }
#pragma unroll
        for (int s = 0; s < kDig; ++s) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t mask = s == 0 ? 2047u : 1023u;  // the top digit may be 512
                const uint32_t fa = (uint32_t)(u[2 * j] >> (50 - 10 * s)) & mask;
                const uint32_t fb = (uint32_t)(u[2 * j + 1] >> (50 - 10 * s)) & mask;
                const uint32_t pk2 = 0x64006400u + fa + (fb << 16);
                const __half2 h = __hadd2(*reinterpret_cast<const __half2*>(&pk2), off);
                w[j] = *reinterpret_cast<const uint32_t*>(&h);
            }
            reinterpret_cast<uint4*>(dig + s * 128 + rr * 64 + g * 8)[q] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// The sum of the digit products of one entry (orders 0 .. 5: units 2^-18 .. 2^-68; f6: what is
// added in units of order 5) in matrix units.  FAST: the FP32 whole numbers f become integers
// kB + f by adding 1.5 2^23 (a quarter of a clock each, a conversion takes two); right while all
// are below 2^22 in size, else *wide shows bits above.  Orders 0 and 1 are that small: of two rows
// of norm 1 (first digits of norm 514 with their rounding, second ones up to 512 each) at most
// 514^2 and 2 x 512 x 4 x 514 < 2^21.1; of a row and the data row, whose entries are below 1/2 (first
// digits up to 256), at most 4 x 256 x 514 and 16 x 256 x 512 + 512 x 4 x 514 < 2^21.6.  So only the
// others are looked at.  The weights are multiply-adds on the FMA pipe, the offsets kB one constant: the ALU is
// what bounds the update.
template <bool FAST>
__device__ __forceinline__ int64_t digit_sum(const float (&f)[kDig], uint32_t f6, uint32_t& wide) {
    constexpr uint32_t kB = 0x4B400000u;
    constexpr uint64_t kOff = 0ull - (((uint64_t)kB << 22) + ((uint64_t)kB << 12) + ((uint64_t)kB << 2) + (kB >> 8));
    uint32_t u[kDig];
#pragma unroll
    for (int k = 0; k < kDig; ++k) {
        // (order 5 with half of the 2^8 that it is cut by: rounded)
        u[k] = FAST ? __float_as_uint(f[k] + (k == 5 ? 12583040.0f : 12582912.0f))
                    : kB + (uint32_t)__float2int_rn(f[k]) + (k == 5 ? 128u : 0u);
        if (FAST && k > 1) wide |= u[k] ^ 0x4B000000u;
    }
    // orders 0 and 1 have weights 2^42 and 2^32: the high word alone
    const uint32_t top = (u[0] << 10) + u[1] - ((kB << 10) + kB);
    const uint64_t mid = bvfix::umad(u[2], 1u << 22, bvfix::umad(u[3], 1u << 12, bvfix::umad(u[4], 4u, bvfix::umad((u[5] + f6) >> 8, 1u, kOff))));
    return (int64_t)(mid + ((uint64_t)top << 32));
}

template <bool FAST>
__device__ __forceinline__ bool digit_sums(int64_t (&o)[4], const float (&acc)[kDig][4], const float (&a6)[4], bool diag) {
    uint32_t wide = 0, f6[4] = {0, 0, 0, 0};
    if (diag) {
#pragma unroll
        for (int e = 0; e < 4; ++e) f6[e] = (uint32_t)(__float2int_rn(a6[e]) >> 10);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        float f[kDig];
#pragma unroll
        for (int k = 0; k < kDig; ++k) f[k] = acc[k][e];
        o[e] = digit_sum<FAST>(f, f6[e], wide);
    }
    return !FAST || !__any_sync(0xffffffffu, wide >= 0x800000u);
}

// L_I's digits as a warp's A fragments.
__device__ __forceinline__ void load_digits(uint2 (&A)[kDig][2], const uint32_t* dI, int lane) {
#pragma unroll
    for (int s = 0; s < kDig; ++s)
#pragma unroll
        for (int h = 0; h < 2; ++h) A[s][h] = reinterpret_cast<const uint2*>(dI + s * 128 + h * 64)[lane];
}

// The products L_I L_J^T of one column half h of a tile (this lane's four entries), in matrix
// units.  On a diagonal tile (diag) the squares of the digits of order 3, which have one sign,
// are taken too: left out, they would raise every pivot by 2^-61.6 per column.
__device__ __forceinline__ void digit_dot(int64_t (&o)[4], const uint2 (&A)[kDig][2], const uint32_t* dJ, int h, bool diag,
                                          int lane) {
    float acc[kDig][4], a6[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < kDig; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[k][e] = 0.0f;
#pragma unroll
    for (int s = 0; s < kDig; ++s) {
        const uint2 B = reinterpret_cast<const uint2*>(dJ + s * 128 + h * 64)[lane];
#pragma unroll
        for (int k = s; k < kDig; ++k) mma_f16(acc[k], A[k - s][0], A[k - s][1], B);
        if (s == 3 && diag) mma_f16(a6, A[3][0], A[3][1], B);
    }
    if (!digit_sums<true>(o, acc, a6, diag)) digit_sums<false>(o, acc, a6, diag);
}

// C -= L_I L_J^T for one tile, one warp; dI, dJ: the tiles' digits.
__device__ __forceinline__ void fix_update(longlong2* C, const uint32_t* dI, const uint32_t* dJ, bool diag, int lane) {
    uint2 A[kDig][2];
    load_digits(A, dI, lane);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        longlong2 v0 = C[h * 64 + lane], v1 = C[h * 64 + 32 + lane];
        int64_t o[4];
        digit_dot(o, A, dJ, h, diag, lane);
        v0.x -= o[0];
        v0.y -= o[1];
        v1.x -= o[2];
        v1.y -= o[3];
        C[h * 64 + lane] = v0;
        C[h * 64 + 32 + lane] = v1;
    }
}

// The general smoothness through K_nu, in matrix units (not inlined: it is as long as all the rest).
__device__ __noinline__ int64_t gen_direct(const DevTheta* th, double x, uint64_t ratio) {
    const uint64_t rho = (uint64_t)bvfix::unit_fix(fmin(matern_gen_corr(*th, x), 1.0)) << 3;
    return (int64_t)((bvfix::mulhi64(rho, ratio) + 2) >> 2);
}

// What a tile (I, J) holds beside pairs of points, the data row and the identity, in the quarters s of
// the mask: rows 8 (s & 1) .., columns 8 (s >> 1) ...
__device__ __forceinline__ void fill_rest(longlong2* tp, int I, int J, int mask, int N, int lane, const int64_t* yfix) {
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
        if (!(mask >> s & 1)) continue;
        const int r = 16 * I + (lane >> 2) + 8 * (s & 1), c = 16 * J + 8 * (s >> 1) + 2 * (lane & 3);
        int64_t v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) v[e] = r == N && c + e < N ? yfix[c + e] : c + e == r ? 1ll << bvfix::kUnitC : 0;
        tp[s * 32 + lane] = make_longlong2(v[0], v[1]);
    }
}

// One covariance tile (I, J), one warp, entries in matrix units: rows and columns of the points
// at px (pre-scaled coordinates, dimension k at k np), row N the data row yfix.  GEN: the
// general smoothness beside the closed forms, through its table gt.  PAD: rows m .. m16 - 1 are no points but rows of the identity.
// PART: as in fix_diag.
template <bool GEN, bool PAD, bool PART>
__device__ __forceinline__ void fix_fill(longlong2* tp, int I, int J, int m, int m16, int N, int lane, const double* px, int d,
                                         const int64_t* yfix, const DevTheta* th, int nu_code, uint64_t ratio, const int64_t* gt,
                                         const uint64_t* tA, const uint64_t* tB, int& flags) {
    const int g = lane >> 2, t = lane & 3;
    // Column halves: entries (g + 8 i, c0 + e), four chains.  PART: a tile row of the data row alone takes
    // no pass, one of at most eight rows a single pass over them (both halves), and a half without
    // points none.
    const bool top = PART && 16 * I + 8 > N;
    const int hend = !PART ? 2 : 16 * I >= N ? 0 : top || 16 * J + 8 >= N ? 1 : 2;
#pragma unroll 1
    for (int h = 0; h < hend; ++h) {
        const int c0 = 16 * J + 8 * h + 2 * t, r0 = 16 * I + g, c1 = top ? c0 + 8 : c0, r1 = top ? r0 : r0 + 8;
        const int ra = min(r0, N - 1), rb = min(r1, N - 1);
        const int ca = min(c0, N - 1), cb = min(c0 + 1, N - 1), cc = min(c1, N - 1), cd = min(c1 + 1, N - 1);
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
        for (int k = 0; k < d; ++k) {
            const double* pk1 = px + k * N;
            const double xa = pk1[ra], xb = pk1[rb], ya = pk1[ca], yb = pk1[cb], yc = pk1[cc], yd = pk1[cd];
            acc[0] = fma(xa - ya, xa - ya, acc[0]);
            acc[1] = fma(xa - yb, xa - yb, acc[1]);
            acc[2] = fma(xb - yc, xb - yc, acc[2]);
            acc[3] = fma(xb - yd, xb - yd, acc[3]);
        }
        int64_t v[4];
        if (GEN && nu_code == NU_GENERAL) {
#pragma unroll 1
            for (int e = 0; e < 4; ++e) {
                const double ac = e == 0 ? acc[0] : e == 1 ? acc[1] : e == 2 ? acc[2] : acc[3];
                const Dist x = bvfix::dist_fix(bvfix::dbits(ac));
                int64_t w = bvfix::matern_gen_fix<GTAB_DEG, -GTAB_E0>(x, gt, tA, tB);
                if (x.q < 1 + GTAB_E0 && x.q > -511)  // nearer than the table, and not 0: K_nu itself
                    w = gen_direct(th, bvfix::scale2((double)x.X, x.q - 63), ratio);
                if (e == 0) v[0] = w;
                else if (e == 1) v[1] = w;
                else if (e == 2) v[2] = w;
                else v[3] = w;
            }
        } else {
            Dist x[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = bvfix::dist_fix(bvfix::dbits(acc[e]));
            bvfix::matern_fix<4>(nu_code == NU_HALF ? 0 : nu_code == NU_3HALF ? 1 : 2, x, tA, tB, v);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = e < 2 ? r0 : r1, c = (e < 2 ? c0 : c1) + (e & 1);
            const int ex = (int)(bvfix::dbits(acc[e]) >> 52);
            if ((ex & 0x7ff) == 0x7ff) flags |= kFail;  // a squared distance beyond FP64's range
            if (ex == 0) v[e] = (int64_t)(tA[0] >> 2);
            if (PAD && ((r >= m && r < m16) || (c >= m && c < m16))) v[e] = 0;
            if (c >= r || r >= N) v[e] = c == r ? 1ll << bvfix::kUnitC : 0;
            if (r == N && c < N) v[e] = yfix[c];
        }
        tp[(2 * h) * 32 + lane] = make_longlong2(v[0], v[1]);
        tp[(top ? 2 : 2 * h + 1) * 32 + lane] = make_longlong2(v[2], v[3]);
    }
    if (PART && hend < 2) fill_rest(tp, I, J, hend == 0 ? 15 : top ? 10 : 12, N, lane, yfix);
}

__device__ __forceinline__ int64_t y_step(int64_t v) { return (v + (1ll << (kYStep - 1))) >> kYStep; }

// The data row (row N) from tile column p on, and the solved entries of the columns before, times
// 2^-kYStep.
template <int NT>
__device__ __forceinline__ void fix_rescale(longlong2* tiles, int p, int TC, int N, int64_t* zrow) {
    const int tid = threadIdx.x, I = N >> 4, r = N & 15;
    const int cnt = (min(I + 1, TC) - p) << 3;
#pragma unroll 1
    for (int i = tid; i < cnt; i += NT) {
        const int q = i & 7;
        longlong2* e = tiles + ftile(I, p + (i >> 3)) * 128 + ((q >> 2) * 2 + (r >> 3)) * 32 + 4 * (r & 7) + (q & 3);
        const longlong2 v = *e;
        *e = make_longlong2(y_step(v.x), y_step(v.y));
    }
#pragma unroll 1
    for (int k = tid; k < 16 * p; k += NT) zrow[k] = y_step(zrow[k]);
}

// Eliminate the first NP panels of 16 columns of the T x T tiles (rows 0 .. N, row N the data
// row; TC tile columns of points) by one CTA.  Warp 0 factors a panel's diagonal tile; the
// other warps follow it, two columns behind, on the rows below, one row a thread (rows beyond
// one a thread, in the largest blocks, after that; a CTA of one warp does them after the tile); then all update the trailing tiles.  A data
// entry out of range scales the data row down and the panel, whose tiles are as they were, is
// solved again.  Returns the scalings, or -1 at a bad pivot (or more than kYMax scalings).
template <int NT>
__device__ __forceinline__ int fix_panels(longlong2* tiles, int T, int TC, int NP, int N, uint32_t* dig, int4* Ld, FixRs* rsv,
                                          int64_t* piv, int64_t* zrow, uint64_t* mb, uint32_t& parity) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lim = bvfix::row_limit(N);
    int scaled = 0;
#pragma unroll 1
    for (int p = 0; p < NP; ++p) {
        const int k0 = p << 4, nc = min(16, N - k0), rows = (T - p - 1) << 4;
        int flags = 0;
        if (NT == 32) {
            fix_diag<true>(tiles + ftile(p, p) * 128, nc, k0, N, lim, lane, Ld, rsv, piv, zrow, mb, flags);
#pragma unroll 1
            for (int rw = lane; rw < rows; rw += 32) {
                const int I = p + 1 + (rw >> 4);
                fix_row(tiles + ftile(I, p) * 128, Ld, rsv, rw & 15, (I << 4) + (rw & 15) == N, lim, zrow + k0, nc, false, mb,
                        parity, dig + (rw >> 4) * (kDigB / 4), flags);
            }
        } else if (warp == 0) {
            fix_diag<false>(tiles + ftile(p, p) * 128, nc, k0, N, lim, lane, Ld, rsv, piv, zrow, mb, flags);
        } else {
#pragma unroll 1
            for (int rw = tid - 32; rw < rows; rw += NT - 32) {
                const int I = p + 1 + (rw >> 4);
                fix_row(tiles + ftile(I, p) * 128, Ld, rsv, rw & 15, (I << 4) + (rw & 15) == N, lim, zrow + k0, nc, rw < NT - 32,
                        mb, parity, dig + (rw >> 4) * (kDigB / 4), flags);
            }
        }
        parity ^= 1;
        if (__syncthreads_or(flags)) {
            if (__syncthreads_or(flags & kFail) || ++scaled > kYMax) return -1;
            fix_rescale<NT>(tiles, p--, TC, N, zrow);
            __syncthreads();
            continue;
        }
        const int S = T - p - 1, cnt = (S * (S + 1)) >> 1;
#pragma unroll 1
        for (int q = warp; q < cnt; q += NT / 32) {
            int ii, jj;
            tri_rc(q, ii, jj);
            const int I = p + 1 + ii, J = p + 1 + jj;
            if (J >= TC) continue;
            fix_update(tiles + ftile(I, J) * 128, dig + ii * (kDigB / 4), dig + jj * (kDigB / 4), ii == jj, lane);
        }
        __syncthreads();
    }
    return scaled;
}

}  // namespace
