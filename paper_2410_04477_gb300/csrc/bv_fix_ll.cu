// bv_fix_ll.cu -- the FP64-accurate block-Vecchia log-likelihood kernel (Eq. 4, Algorithm 1)
// in 64-bit fixed point, with the trailing updates on the tensor cores.
//
// The computation is the one of bv_loglik.cu: one Cholesky factorisation of the block's
// augmented (N+1) x (N+1) matrix.  FP64 arithmetic bounded it: the SM executes 2 FP64 lanes
// per clock, and a block needs N^3/6 of them for the updates and about 10 N^2 for the
// covariance.  Dividing by D = sigma^2 + tau^2 makes the diagonal 1, so that every entry,
// Schur complement and factor entry lies in [-1, 1] and 64-bit integers hold them with an
// absolute error below FP64's (which rounds at 2^-54 of values near 1):
//   covariance   bv_fix.cuh: squared distances in FP64, the rest on the integer pipe;
//   panel        16 columns: the diagonal tile by one warp, the rows below one per thread;
//   update       C_IJ -= L_I L_J^T on the tensor cores, exactly: every factor entry is cut
//                into six signed 10-bit digits, held as FP16; products of digits sum to whole
//                numbers below 2^24 over 16 columns and up to four digit pairs, which FP32
//                accumulation adds without rounding.  The 21 digit pairs of combined order
//                <= 5 are taken (the pairs of order 4 and 5, five and six to a sum, could
//                round in the last bit only on sums that real digits do not reach, by one
//                unit of 2^-58); what is left out is below 2^-57 of 1.
// The data row is scaled by a power of two that leaves solved entries room for 16 times the
// largest |y| / sqrt(D); where one is larger (the parameters are far from the data's), the row is
// scaled further and the panel solved again.
//
// Against a 113-bit factorisation of the same scaled coordinates, the quadratic form and the log-
// determinant err by 2.2e-14 and 2.8e-16 (RMS, relative; n = 4,000, m = 60, nu = 3/2, tau^2 = 1e-4), FP64
// arithmetic by 1.4e-13 and 2.2e-15; classic Vecchia at m = 30 by 1.9e-14 and 1.4e-16 against 1.3e-13 and
// 1.1e-14.  Time of an evaluation, FP64 arithmetic and this kernel:
//   n = 200,000, m = 60 (N about 70)        5.09 ms   2.38 ms
//   n = 36,931, m = 113                     3.58      1.16
//   n = 100,000, 3D, m = 200                42.6      9.38
//   n = 50,000, blocks of 1, m = 30         2.35      1.25
//   n = 100,000, m = 60, nu = 1.2           4.93      2.25
//   n = 2,000, m = 30                       0.126     0.096
// What bounds it: for few blocks the pivots' chain (a tile's 16 pivots take some 12,000 clocks,
// in which the other warps follow two columns behind); else instruction issue and fetch, shared
// by the covariance, the panel rows and the sums of digit products, with the tensor cores busy
// for a twentieth of the time at N about 70 and an eightieth at N = 31.  More warps an SM, and starting a panel's chain
// beside the update before it, were measured and lose; halving the code gained 3 to 4%.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "bv_device.cuh"
#include "bv_fix.cuh"
#include "bv_fix_tile.cuh"
#include "bv_internal.h"
#include "bv_ll_block.cuh"

namespace {


// GLOB: the tiles live in a global-memory slot of the CTA (they stay in L2), where they would not
// leave room for as many CTAs in shared memory.
// WARPS: resident warps an SM that the registers leave room for: 20 (96 registers) up to N = 111,
// where more blocks an SM hide the pivots' chains (n = 200,000, m = 60: 2.40 ms, with 16 2.50),
// 16 (128 registers) beyond, where spills cost more (3D, m = 200: 10.2 ms, with 16 9.34); 24
// lose in both (2.58, 10.8).
template <int NT, bool GEN, bool GLOB, int WARPS>
__global__ void __launch_bounds__(NT, WARPS * 32 / NT) k_ll_fix(LLArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint64_t tA[256], tBs[NT == 32 ? 1 : 256];  // (one-warp CTAs: as many as fit count more)
    __shared__ int s_w;
    __shared__ unsigned s_ymax;  // largest high word of |y| / sqrt(D)
    __shared__ __align__(8) uint64_t s_mb[8];
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (NT > 32) {
#pragma unroll 1
        for (int j = tid; j < 256; j += NT) tBs[j] = a.fixtab[256 + j];
    }
    const uint64_t* tB = NT > 32 ? tBs : a.fixtab + 256;
    const int nwork = work_count(a);
    if (tid < 8)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(s_mb + tid)) : "memory");
    uint32_t parity = 0;  // of the panel's phase of the mbarriers
    if (tid == 0) s_w = take_work(a.ctr, blockIdx.x);
    __syncthreads();
    int dsprev = -1;
#pragma unroll 1
    for (int w = s_w; w < nwork; w = s_w) {
        const int nx = tid == 0 ? take_work(a.ctr, w + gridDim.x) : 0;
        const int blk = a.work[w];
        const int64_t b0 = a.bptr[blk], n0 = a.nptr[blk];
        const int b = (int)(a.bptr[blk + 1] - b0), m = (int)(a.nptr[blk + 1] - n0);
        const int N = m + b, T = fix_tiles(N), TC = (N + 15) >> 4;
        const int ds = a.bds[blk];
        const DevTheta th = a.theta[ds];
        const int d = a.d;
        unsigned char* wk = GLOB ? smraw : smraw + (size_t)((T * (T + 1)) >> 1) * kTileB;
        longlong2* tiles = GLOB ? reinterpret_cast<longlong2*>(a.ws + (int64_t)blockIdx.x * a.ws_stride)
                                : reinterpret_cast<longlong2*>(smraw);
        uint32_t* dig = reinterpret_cast<uint32_t*>(wk);
        int4* Ld = reinterpret_cast<int4*>(wk + (size_t)(T - 1) * kDigB);
        FixRs* rsv = reinterpret_cast<FixRs*>(Ld + 16 * kLd + 16);
        double* px = reinterpret_cast<double*>(rsv + 16);
        double* yv = px + d * N;
        int64_t* piv = reinterpret_cast<int64_t*>(yv + N);
        int64_t* zrow = piv + N;

        const double D = th.diag, isd = th.diag_rsqrt;
        const uint64_t ratio = th.diag_ratio;
        if (ds != dsprev) {  // A[j] = 2^(-j/256) sigma^2 / D
#pragma unroll 1
            for (int j = tid; j < 256; j += NT) tA[j] = bvfix::mulhi64(a.fixtab[j], ratio) << 1;
            dsprev = ds;
        }
        if (tid == 0) s_ymax = 0;
#pragma unroll 1
        for (int j = tid; j < 16 * kLd + 16; j += NT)
            if (j % kLd >= 16) Ld[j] = make_int4(0, 0, 0, 0);
        __syncthreads();
        unsigned ym = 0;
#pragma unroll 1
        for (int t = tid; t < N; t += NT) {
            const int g = t < m ? a.nidx[n0 + t] : a.pidx[b0 + (t - m)];
#pragma unroll 1
            for (int k = 0; k < d; ++k) px[k * N + t] = a.locs[(int64_t)k * a.n_tot + g] * inv_range_k(th, k);
            const double y = a.y[g] * isd;
            yv[t] = y;  // (in place of its fixed-point value until the scale is known)
            ym = max(ym, (unsigned)__double2hiint(y) & 0x7fffffffu);
        }
        ym = __reduce_max_sync(0xffffffffu, ym);
        if (lane == 0) atomicMax(&s_ymax, ym);
        __syncthreads();
        const int ye = (int)(s_ymax >> 20);
        const bool valid = D > 0.0 && D < INFINITY && ye != 0x7ff;
        int E = (ye > 0 ? ye - 1022 : -1021) + kYRoom + bvfix::row_limit(N);

        int64_t* yfix = reinterpret_cast<int64_t*>(yv);
        int flags = valid ? 0 : kFail;
#pragma unroll 1
        for (int t = tid; t < N; t += NT) yfix[t] = __double2ll_rn(bvfix::scale2(yv[t], bvfix::kUnitC - E));
        __syncthreads();
        const int ntile = (T * (T + 1)) >> 1;
#pragma unroll 1
        for (int q = warp; q < ntile; q += NW) {
            int I, J;
            tri_rc(q, I, J);
            if (J >= TC) continue;
            fix_fill<GEN, false, NT == 32>(tiles + q * 128, I, J, N, N, N, lane, px, d, yfix, a.theta + ds, th.nu_code, ratio,
                                         a.gtabi + (int64_t)ds * GTAB_SIZE, tA, tB, flags);
        }
        bool fail = __syncthreads_or(flags);
        if (!fail) {
            const int scaled = fix_panels<NT>(tiles, T, TC, TC, N, dig, Ld, rsv, piv, zrow, s_mb, parity);
            fail = scaled < 0;
            E += kYStep * scaled;
        }

        if (warp == 0) {
            const double zs = bvfix::scale2(1.0, E - bvfix::kUnitL), ps = D * 0x1p-60;
            const double2 s2 = warp_terms(m, N, lane, [&](int k) { return fail ? 0.0 : (double)zrow[k] * zs; },
                                          [&](int k) { return fail ? 0.0 : log((double)piv[k] * ps); });
            if (lane == 0) {
                double ell = -0.5 * (s2.x + (double)b * kLog2Pi);
                if (fail || !(ell == ell)) {
                    ell = -INFINITY;
                    record_fail(a.fail, blk);
                }
                a.ell_blk[blk] = ell;
                a.u_blk[blk] = s2.y;
                s_w = nx;
            }
        }
        __syncthreads();
    }
}

// The instantiation of a kind, CTA size and smoothness.
using FixKernel = void (*)(LLArgs);
template <bool GEN>
FixKernel fix_kernel_g(int kind, int threads) {
    if (threads == 256) return kind == 7 ? k_ll_fix<256, GEN, false, 16> : k_ll_fix<256, GEN, true, 16>;
    if (kind == 7) return threads == 64 ? k_ll_fix<64, GEN, false, 20> : nullptr;
    if (threads == 32) return k_ll_fix<32, GEN, true, 20>;
    if (threads != 128) return nullptr;
    return kind == 8 ? k_ll_fix<128, GEN, true, 20> : k_ll_fix<128, GEN, true, 16>;
}
cudaError_t fix_kernel(int kind, int threads, bool gen, FixKernel* k) {
    *k = gen ? fix_kernel_g<true>(kind, threads) : fix_kernel_g<false>(kind, threads);
    return *k ? cudaFuncSetAttribute(*k, cudaFuncAttributeMaxDynamicSharedMemorySize, kFixSmemCap) : cudaErrorInvalidValue;
}

}  // namespace

// CTA size: one warp for the diagonal tiles, the others for the rows below, with which four warps cover
// blocks up to N = 111 in one pass and large ones take eight.  A bin of few blocks (two an SM) takes eight
// as well: there a block's latency counts, not the SM's rate.  Up to three tile rows with tiles in the
// workspace (8): one warp for everything, 16 to 20 of them an SM.
int bv_fix_threads(int kind, int nmax, int nwork, int num_sms) {
    if (kind == 7) return nwork <= 2 * num_sms ? 256 : 64;
    if (fix_tiles(nmax) <= 3) return 32;
    return nwork > 2 * num_sms && nmax <= 239 ? 128 : 256;
}

size_t bv_fix_smem_bytes(int kind, int nmax, int d) {
    return fix_work_bytes(nmax, d) + (kind == 7 ? fix_tile_bytes(nmax) : 0);
}

// The kernel form of a bin of largest size nmax: -1 when even the panel's digits do not fit; tiles in a
// workspace (8; 9 from N = 112 on, with more registers), or, up to three tile rows, in shared memory (7)
// when the evaluation has few blocks in all (total): then latency counts, and one kernel for all small
// bins, since fetching a kernel's code takes some 13 us.  Many small blocks go to one-warp CTAs, since a
// second warp mostly waits on the pivots and as many CTAs do not fit with their tiles: 50,000 blocks of N =
// 8, 11, 18, 24, 31, 36, 47 take 0.37, 0.43, 1.00, 1.13, 1.25, 2.10, 2.40 ms (two warps and tiles in
// shared memory: 0.74, 0.74, 1.50, 1.51, 1.53, 2.67, 2.69; FP64, a warp a block: 0.46, 0.59, 0.97, 1.45,
// 2.18, 2.84, 4.78).  With fewer blocks an SM the second warp helps: up to 8 for N <= 24 (1,000 blocks of N
// = 21: 105 us a call either way), some 20 beyond (3,000 blocks of N = 31: 160 us with one, 141 with two;
// 2,000 of N = 47: 208 and 171).
int bv_fix_kind(int nmax, int total, int num_sms, int d) {
    const int T = fix_tiles(nmax);
    if (T <= 3) return total <= (T == 1 ? 2 : nmax <= 24 ? 8 : 21) * num_sms ? 7 : 8;
    if (bv_fix_smem_bytes(8, nmax, d) > (size_t)kFixSmemCap) return -1;
    return nmax <= 111 ? 8 : 9;
}
int bv_fix_max_n(int d) {
    int n = 64;
    while (bv_fix_kind(n + 1, 0, 0, d) > 0) ++n;
    return n;
}
size_t bv_fix_slot_bytes(int nmax) { return fix_tile_bytes(nmax); }

int bv_fix_occupancy(int kind, int threads, size_t smem) {
    int n[2] = {0, 0};
    for (int gen = 0; gen < 2; ++gen) {
        FixKernel k;
        if (fix_kernel(kind, threads, gen, &k) != cudaSuccess) return 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n[gen], k, threads, smem);
    }
    return n[0] > n[1] ? n[0] : n[1];
}

cudaError_t bv_fix_launch(int kind, int threads, int grid, size_t smem, const LLArgs& a, cudaStream_t s) {
    FixKernel k;
    const cudaError_t e = fix_kernel(kind, threads, a.gen, &k);
    if (e != cudaSuccess) return e;
    k<<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

// The exponential's tables (bv_fix.cuh): 2^(-j/256) in units 2^-62, then 2^(-j/65536) in units
// 2^-63, the first of them one unit below 1.
void bv_fix_tables(uint64_t* t) {
    for (int j = 0; j < 256; ++j) {
        t[j] = (uint64_t)(exp2l(-(long double)j / 256.0L) * 0x1p62L + 0.5L);
        t[256 + j] = j ? (uint64_t)(exp2l(-(long double)j / 65536.0L) * 0x1p63L + 0.5L) : (1ull << 63) - 1;
    }
}

// The Box-Muller pairs' tables (bv_fix.cuh).
size_t bv_sim_table_bytes() { return sizeof(bvfix::SimTab); }
void bv_sim_table(void* out) {
    bvfix::SimTab& t = *static_cast<bvfix::SimTab*>(out);
    const long double half_pi = 1.570796326794896619231321691639751442L;
    for (int j = 0; j < 256; ++j) {
        const long double x = ((long double)j + 0.5L) / 256.0L;
        t.c[j] = (uint16_t)(j == 0 ? 32768 : j == 255 ? 16384 : (int)(32768.0L / (1.0L + x) + 0.5L));
        t.ln[j] = (int64_t)floorl(-logl((long double)t.c[j] / 32768.0L * (j >= bvfix::kLnHalf ? 2.0L : 1.0L)) * 0x1p60L + 0.5L);
        t.cs[j] = (int64_t)(cosl(half_pi * x) * 0x1p62L + 0.5L);
        t.sn[j] = (int64_t)(sinl(half_pi * x) * 0x1p62L + 0.5L);
    }
}
