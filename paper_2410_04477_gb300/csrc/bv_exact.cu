// bv_exact.cu -- the exact Gaussian log-likelihood (Eq. 1) by a dense tiled Cholesky
// factorisation on the GPU, and the KL divergence of the block-Vecchia approximation
// (Eq. 7 of Sec. 3.1: KL = ell_0(theta; 0) - ell_a(theta; 0)).
//
// The (n+1) x (n+1) augmented matrix [[Sigma, .], [y^T, .]], divided by the diagonal D =
// sigma^2 + tau^2, in the fixed-point form of bv_fix_tile.cuh: packed lower 16 x 16 tiles of
// 64-bit entries, products of factor entries on the tensor cores through their digits.  At n =
// 8,000 21.8 ms; FP64 arithmetic, 2 lanes a clock and SM, took 188.7 ms (n^3 / 3 operations at
// 72% of its peak).  Right-looking by panels of 64 columns (four tiles), three launches a panel:
//   k_ex_diag    the 64 x 64 diagonal block, one CTA
//   k_ex_rows    the rows below it, 32 of them a warp: four solves against the 16 x 16
//                diagonal tiles with the updates between them, and the rows' digits
//   k_ex_update  A_IJ -= sum over the panel's four tiles of L_I L_J^T, a CTA per 64 x 64 block,
//                the sums of a block kept in registers so that it is read and written once;
//                the next panel's block column first, so that its diagonal block and rows run
//                on a stream of higher priority beside the update of the rest
// The factor's row n is z = L^-1 y, so y^T Sigma^-1 y = |z|^2 and log|Sigma| is the sum of the
// pivots' logarithms.  The data row is scaled by a power of two; should a solved entry leave
// the fixed-point range, or the squares sum to more than 16, the factorisation is done again with a larger one.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "bv_device.cuh"
#include "bv_fix_tile.cuh"
#include "bv_internal.h"

namespace {

constexpr int kExStep = 8, kExPasses = 13;                // the data row's scalings (a pass each)
constexpr int kP = 4;                                     // tiles of a panel
constexpr int kLdN = 16 * kLd + 16;                       // entries of a tile's factor in memory

__device__ __forceinline__ int64_t etile(int64_t I, int64_t J) { return ((I * (I + 1)) / 2 + J) * 128; }

struct ExArgs {
    const double* locs;  // SoA d x n
    const double* y;     // null: y = 0
    int64_t n;
    int d;
    int T, TC;           // tile rows of the n + 1 rows, tile columns of the n columns
    DevTheta th;
    longlong2* A;        // packed lower tiles
    uint32_t* dig;       // digits of the panel's rows: tile row I, panel tile s at (I kP + s)
    int4* Ld;            // the panel's four diagonal factors, their reciprocal roots and the
    FixRs* rsv;          // digits of the tiles between them (i, s), i > s, at i (i - 1) / 2 + s
    uint32_t* ddig;
    int64_t* piv;        // pivots and data row, by column
    int64_t* zrow;
    const uint64_t* fixtab;
    int E;               // data row in units of 2^(E - 60) sqrt(D)
    int* flags;
};

// One warp per tile.
template <bool GEN>
__global__ void __launch_bounds__(256) k_ex_fill(ExArgs a, int64_t ntiles) {
    __shared__ uint64_t tA[256], tB[256];
    tA[threadIdx.x] = bvfix::mulhi64(a.fixtab[threadIdx.x], a.th.diag_ratio) << 1;
    tB[threadIdx.x] = a.fixtab[256 + threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t f = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (f >= ntiles) return;
    int64_t I = (int64_t)((sqrt(8.0 * (double)f + 1.0) - 1.0) * 0.5);
    while ((I + 1) * (I + 2) / 2 <= f) ++I;
    while (I * (I + 1) / 2 > f) --I;
    const int64_t J = f - I * (I + 1) / 2, n = a.n;
    longlong2* tp = a.A + f * 128;
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
        const int64_t r = 16 * I + g + 8 * (s & 1), c0 = 16 * J + 8 * (s >> 1) + 2 * t;
        int64_t v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int64_t c = c0 + e, rr = min(r, n - 1), cc = min(c, n - 1);
            double acc = 0.0;
            for (int k = 0; k < a.d; ++k) {
                const double dt = (a.locs[k * n + rr] - a.locs[k * n + cc]) * inv_range_k(a.th, k);
                acc = fma(dt, dt, acc);
            }
            const int ex = (int)(bvfix::dbits(acc) >> 52);
            // a squared distance beyond FP64's range: e^-x and K_nu give 0 there, the other forms have no value
            if ((ex & 0x7ff) == 0x7ff && a.th.nu_code != NU_HALF && !GEN) atomicOr(a.flags, kFail);
            if (GEN) v[e] = c < r && r < n ? gen_direct(&a.th, sqrt(acc), a.th.diag_ratio) : 0;
            else if (ex == 0) v[e] = (int64_t)(tA[0] >> 2);
            else {
                const Dist x[1] = {bvfix::dist_fix(bvfix::dbits(acc))};
                int64_t o[1];
                bvfix::matern_fix<1>(a.th.nu_code == NU_HALF ? 0 : a.th.nu_code == NU_3HALF ? 1 : 2, x, tA, tB, o);
                v[e] = o[0];
            }
            if (c >= r || r >= n) v[e] = c == r ? 1ll << bvfix::kUnitC : 0;
            if (r == n && c < n && a.y) v[e] = __double2ll_rn(ldexp(a.y[c] * a.th.diag_rsqrt, bvfix::kUnitC - a.E));
        }
        tp[((s >> 1) * 2 + (s & 1)) * 32 + lane] = make_longlong2(v[0], v[1]);
    }
}

// Largest high word of |y| / sqrt(D).
__global__ void __launch_bounds__(256) k_ex_ymax(const double* y, int64_t n, double isd, unsigned* out) {
    unsigned m = 0;
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += 256ll * gridDim.x)
        m = max(m, (unsigned)__double2hiint(y[i] * isd) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// The diagonal block of panel P: at most 4 x 4 tiles, factored as a block of its own
// (bv_fix_ll.cu); the bound is the chain of its 64 pivots.
__global__ void __launch_bounds__(128) k_ex_diag(ExArgs a, int P) {
    __shared__ longlong2 tiles[10 * 128];
    __shared__ __align__(16) uint32_t dig[3 * kDigB / 4];
    __shared__ int4 Ld[kLdN];
    __shared__ FixRs rsv[16];
    __shared__ __align__(8) uint64_t mb[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int I0 = kP * P, tr = min(kP, a.T - I0), tc = min(kP, a.TC - I0);
    if (tid < 8)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(mb + tid)) : "memory");
    for (int q = 0; q < ((tr * (tr + 1)) >> 1); ++q) {
        int i, j;
        tri_rc(q, i, j);
        tiles[q * 128 + tid] = a.A[etile(I0 + i, I0 + j) + tid];
    }
    for (int j = tid; j < kLdN; j += 128) Ld[j] = make_int4(0, 0, 0, 0);
    __syncthreads();
    int flags = 0;
    for (int p = 0; p < tc; ++p) {
        const int64_t k0 = 16ll * (I0 + p);
        const int nc = (int)min((int64_t)16, a.n - k0), rows = (tr - p - 1) << 4, ry = (int)min(a.n - k0, (int64_t)1 << 20);
        if (warp == 0) {
            fix_diag<false>(tiles + ftile(p, p) * 128, nc, 0, ry, 1, lane, Ld, rsv, a.piv + k0, a.zrow + k0, mb, flags);
        } else if (tid - 32 < rows) {
            const int rw = tid - 32, i = p + 1 + (rw >> 4);
            fix_row(tiles + ftile(i, p) * 128, Ld, rsv, rw & 15, 16 * (i - p) + (rw & 15) == ry, 1, a.zrow + k0, nc, true,
                    mb, p & 1, dig + (rw >> 4) * (kDigB / 4), flags);
        }
        __syncthreads();
        for (int j = tid; j < kLdN; j += 128) a.Ld[p * kLdN + j] = Ld[j];
        if (tid < 16) a.rsv[p * 16 + tid] = rsv[tid];
        for (int i = p + 1; i < tr; ++i)
            for (int j = tid; j < kDigB / 16; j += 128)
                reinterpret_cast<uint4*>(a.ddig + (i * (i - 1) / 2 + p) * (kDigB / 4))[j] =
                    reinterpret_cast<const uint4*>(dig + (i - p - 1) * (kDigB / 4))[j];
        const int S = tr - p - 1;
        for (int q = warp; q < ((S * (S + 1)) >> 1); q += 4) {
            int ii, jj;
            tri_rc(q, ii, jj);
            if (I0 + p + 1 + jj >= a.TC) continue;
            fix_update(tiles + ftile(p + 1 + ii, p + 1 + jj) * 128, dig + ii * (kDigB / 4), dig + jj * (kDigB / 4), ii == jj,
                       lane);
        }
        __syncthreads();
    }
    if (flags) atomicOr(a.flags, flags);
}

// The rows below panel P's diagonal block: 32 rows (two tile rows) a warp.
constexpr size_t kRowsSmem = kP * kLdN * sizeof(int4) + kP * 16 * sizeof(FixRs) + 6 * kDigB + 4 * 2 * kDigB;
__global__ void __launch_bounds__(128) k_ex_rows(ExArgs a, int P) {
    extern __shared__ __align__(16) unsigned char smx[];
    int4* Ld = reinterpret_cast<int4*>(smx);
    FixRs* rsv = reinterpret_cast<FixRs*>(Ld + kP * kLdN);
    uint32_t* dd = reinterpret_cast<uint32_t*>(rsv + kP * 16);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* dw = dd + 6 * (kDigB / 4) + warp * 2 * (kDigB / 4);
    const int I0 = kP * P, tc = min(kP, a.TC - I0);
    for (int j = tid; j < tc * kLdN; j += 128) Ld[j] = a.Ld[j];
    if (tid < tc * 16) rsv[tid] = a.rsv[tid];
    for (int j = tid; j < 6 * kDigB / 16; j += 128) reinterpret_cast<uint4*>(dd)[j] = reinterpret_cast<const uint4*>(a.ddig)[j];
    __syncthreads();
    const int Iw = I0 + kP + 2 * (blockIdx.x * 4 + warp);  // the warp's first tile row
    if (Iw >= a.T) return;
    const int nI = min(2, a.T - Iw), I = Iw + min(lane >> 4, nI - 1);
    int flags = 0;
    for (int s = 0; s < tc; ++s) {
        const int64_t k0 = 16ll * (I0 + s);
        const int nc = (int)min((int64_t)16, a.n - k0);
        if ((lane >> 4) < nI)
            fix_row(a.A + etile(I, I0 + s), Ld + s * kLdN, rsv + s * 16, lane & 15, 16ll * I + (lane & 15) == a.n, 1, a.zrow + k0,
                    nc, false, nullptr, 0, dw + (lane >> 4) * (kDigB / 4), flags);
        __syncwarp();
        for (int i = 0; i < nI; ++i) {
            uint4* out = reinterpret_cast<uint4*>(a.dig + ((int64_t)(Iw + i) * kP + s) * (kDigB / 4));
            const uint4* src = reinterpret_cast<const uint4*>(dw + i * (kDigB / 4));
            for (int j = lane; j < kDigB / 16; j += 32) out[j] = src[j];
            for (int j = s + 1; j < tc; ++j)
                fix_update(a.A + etile(Iw + i, I0 + j), dw + i * (kDigB / 4), dd + (j * (j - 1) / 2 + s) * (kDigB / 4), false,
                           lane);
        }
        __syncwarp();
    }
    if (flags) atomicOr(a.flags, flags);
}

// Trailing 64 x 64 blocks (bi, bj), bj <= bi: those of block column j0 (first) or all beyond it.
// Warp w has tile row w / 2 and two tile columns of the block.
__global__ void __launch_bounds__(256, 2) k_ex_update(ExArgs a, int P, int j0, bool first) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t f = blockIdx.x;
    int bi, bj;
    if (first) {
        bi = j0 + (int)f;
        bj = j0;
    } else {
        int64_t x = (int64_t)((sqrt(8.0 * (double)f + 1.0) - 1.0) * 0.5);
        while ((x + 1) * (x + 2) / 2 <= f) ++x;
        while (x * (x + 1) / 2 > f) --x;
        bi = j0 + 1 + (int)x;
        bj = j0 + 1 + (int)(f - x * (x + 1) / 2);
    }
    const int I = kP * bi + (warp >> 1), J0 = kP * bj + 2 * (warp & 1), tc = min(kP, a.TC - kP * P);
    if (I >= a.T || J0 > I || J0 >= a.TC) return;
    const bool two = J0 + 1 <= I && J0 + 1 < a.TC;
    int64_t sum[2][2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) sum[j][h][e] = 0;
#pragma unroll 1
    for (int s = 0; s < tc; ++s) {
        uint2 A[kDig][2];
        load_digits(A, a.dig + ((int64_t)I * kP + s) * (kDigB / 4), lane);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (j && !two) break;
            const uint32_t* dJ = a.dig + ((int64_t)(J0 + j) * kP + s) * (kDigB / 4);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int64_t o[4];
                digit_dot(o, A, dJ, h, I == J0 + j, lane);
#pragma unroll
                for (int e = 0; e < 4; ++e) sum[j][h][e] += o[e];
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        if (j && !two) break;
        longlong2* C = a.A + etile(I, J0 + j);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
                longlong2 v = C[(2 * h + rr) * 32 + lane];
                v.x -= sum[j][h][2 * rr];
                v.y -= sum[j][h][2 * rr + 1];
                C[(2 * h + rr) * 32 + lane] = v;
            }
    }
}

// log-det and quadratic form from the factor: one CTA, fixed-order sums.
__global__ void __launch_bounds__(256) k_exact_terms(const int64_t* piv, const int64_t* zrow, int64_t n, double ps, double zs,
                                                     double* out) {
    __shared__ double s1[256], s2[256];
    double ld = 0.0, q = 0.0;
    for (int64_t g = threadIdx.x; g < n; g += 256) {
        ld += log((double)piv[g] * ps);
        const double z = (double)zrow[g] * zs;
        q = fma(z, z, q);
    }
    s1[threadIdx.x] = ld;
    s2[threadIdx.x] = q;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int t = 0; t < 256; ++t) {
            a += s1[t];
            b += s2[t];
        }
        out[0] = a;
        out[1] = b;
    }
}

// The call's device memory, taken from the stream's pool, and its second stream, given back on
// every path: the second stream's work is waited for before the memory goes.
struct ExBuf {
    cudaStream_t s, hi = nullptr;
    cudaEvent_t ready = nullptr, rest = nullptr;  // on s: a panel's rows are wanted; the rest is updated
    cudaEvent_t rows = nullptr;                   // on hi: a panel's rows and digits are there
    void* p = nullptr;
    explicit ExBuf(cudaStream_t st) : s(st) {}
    ~ExBuf() {
        if (hi) cudaStreamSynchronize(hi);
        if (p) cudaFreeAsync(p, s);
        for (cudaEvent_t e : {ready, rest, rows})
            if (e) cudaEventDestroy(e);
        if (hi) cudaStreamDestroy(hi);
    }
};

}  // namespace

extern "C" int bv_exact_loglik(bv_ctx* c, const bv_theta* theta, int32_t use_y, double* out_loglik,
                               double* out_quad, double* out_logdet) {
    if (!c || !theta) return BV_EINVAL;
    if (c->ndata != 1) return c->ndata == 0 ? BV_ESTATE : BV_EINVAL;
    if (use_y && !c->have_y) return BV_ESTATE;
    const int64_t n = c->n_tot;
    if (n <= 0 || n > 65536) return BV_EINVAL;
    DevTheta th;
    BV_TRY(bv_theta_to_dev(theta, c->d, &th));
    BV_CUDA(cudaSetDevice(c->device));
    const cudaStream_t st = c->stream;
    ExArgs a;
    a.locs = c->d_locs;
    a.y = use_y ? c->d_y : nullptr;
    a.n = n;
    a.d = c->d;
    a.T = (int)((n + 16) / 16);
    a.TC = (int)((n + 15) / 16);
    a.th = th;
    a.fixtab = c->d_fixtab;
    const int64_t ntiles = (int64_t)a.T * (a.T + 1) / 2;
    // one allocation: tiles | row digits | factors, roots and digits of the diagonal block |
    // pivots | data row | terms, flags, largest |y|
    const size_t szA = (size_t)ntiles * kTileB, szD1 = (size_t)a.T * kP * kDigB, szD = 2 * szD1, szL = kP * kLdN * sizeof(int4);
    const size_t szR = kP * 16 * sizeof(FixRs), szE = 6 * kDigB, szN = (size_t)a.TC * 16 * sizeof(int64_t);
    ExBuf buf(st);
    BV_CUDA(cudaMallocAsync(&buf.p, szA + szD + szL + szR + szE + 2 * szN + 32, st));
    unsigned char* q = static_cast<unsigned char*>(buf.p);
    a.A = reinterpret_cast<longlong2*>(q);
    a.dig = reinterpret_cast<uint32_t*>(q += szA);
    a.Ld = reinterpret_cast<int4*>(q += szD);
    a.rsv = reinterpret_cast<FixRs*>(q += szL);
    a.ddig = reinterpret_cast<uint32_t*>(q += szR);
    a.piv = reinterpret_cast<int64_t*>(q += szE);
    a.zrow = reinterpret_cast<int64_t*>(q += szN);
    struct {
        double term[2];
        int flags;
        unsigned ymax;
    } h = {};
    double* terms = reinterpret_cast<double*>(q += szN);
    a.flags = reinterpret_cast<int*>(terms + 2);
    BV_CUDA(cudaMemsetAsync(a.Ld, 0, szL + szR + szE + 2 * szN + 32, st));
    BV_CUDA(cudaFuncSetAttribute(k_ex_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowsSmem));
    uint32_t* const dig0 = a.dig;
    {
        int lo = 0, hi = 0;
        BV_CUDA(cudaDeviceGetStreamPriorityRange(&lo, &hi));
        BV_CUDA(cudaStreamCreateWithPriority(&buf.hi, cudaStreamNonBlocking, hi));
        for (cudaEvent_t* e : {&buf.ready, &buf.rest, &buf.rows}) BV_CUDA(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    }
    int E = 0;
    if (use_y) {
        k_ex_ymax<<<(unsigned)std::min<int64_t>((n + 255) / 256, c->num_sms), 256, 0, st>>>(c->d_y, n, th.diag_rsqrt,
                                                                                         reinterpret_cast<unsigned*>(a.flags + 1));
        BV_CUDA(cudaGetLastError());
        BV_CUDA(cudaMemcpyAsync(&h.ymax, a.flags + 1, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
        BV_CUDA(cudaStreamSynchronize(st));
        const int ye = (int)(h.ymax >> 20);
        E = (ye > 0 ? ye - 1022 : -1021) + kYRoom + 1;
    }
    const bool valid = th.diag > 0.0 && th.diag < INFINITY && (int)(h.ymax >> 20) != 0x7ff;
    const int np = (a.TC + kP - 1) / kP, nb = (a.T + kP - 1) / kP;
    for (int pass = 0; valid; ++pass) {
        a.E = E;
        BV_CUDA(cudaMemsetAsync(a.flags, 0, sizeof(int), st));
        const unsigned fg = (unsigned)((ntiles + 7) / 8);
        if (th.nu_code == NU_GENERAL) k_ex_fill<true><<<fg, 256, 0, st>>>(a, ntiles);
        else k_ex_fill<false><<<fg, 256, 0, st>>>(a, ntiles);
        BV_CUDA(cudaGetLastError());
        BV_CUDA(cudaEventRecord(buf.ready, st));
        BV_CUDA(cudaStreamWaitEvent(buf.hi, buf.ready, 0));
        for (int P = 0; P < np; ++P) {
            // hi: the panel (its block column is up to date), then the next block column, which
            // the rest of panel P - 1's update has to have passed; st: the rest of this panel's
            // update.  The digits of two panels are in use at a time.
            a.dig = dig0 + (P & 1) * (szD1 / 4);
            k_ex_diag<<<1, 128, 0, buf.hi>>>(a, P);
            const int64_t strips = a.T - (int64_t)kP * (P + 1), m = nb - P - 1;
            if (strips <= 0) break;
            k_ex_rows<<<(unsigned)((strips + 7) / 8), 128, kRowsSmem, buf.hi>>>(a, P);
            BV_CUDA(cudaEventRecord(buf.rows, buf.hi));
            BV_CUDA(cudaStreamWaitEvent(st, buf.rows, 0));
            if (P > 0) BV_CUDA(cudaStreamWaitEvent(buf.hi, buf.rest, 0));
            k_ex_update<<<(unsigned)m, 256, 0, buf.hi>>>(a, P, P + 1, true);
            if (m > 1) k_ex_update<<<(unsigned)(m * (m - 1) / 2), 256, 0, st>>>(a, P, P + 1, false);
            BV_CUDA(cudaEventRecord(buf.rest, st));
        }
        BV_CUDA(cudaGetLastError());
        BV_CUDA(cudaEventRecord(buf.rows, buf.hi));
        BV_CUDA(cudaStreamWaitEvent(st, buf.rows, 0));
        k_exact_terms<<<1, 256, 0, st>>>(a.piv, a.zrow, n, th.diag * 0x1p-60, ldexp(1.0, E - bvfix::kUnitL), terms);
        BV_CUDA(cudaGetLastError());
        BV_CUDA(cudaMemcpyAsync(&h, terms, sizeof(double) * 2 + sizeof(int), cudaMemcpyDeviceToHost, st));
        BV_CUDA(cudaStreamSynchronize(st));
        // the data row's Schur complements are below 2^-5 + |z| in units of 2^E sqrt(D); while the
        // squares sum to at most 16 none has left the range of +-8 (an entry that had would have
        // come after entries whose squares sum to more)
        if (!(h.term[1] <= ldexp(16.0, 2 * E))) h.flags |= kOver;
        if (!(h.flags & kOver) || (h.flags & kFail) || pass + 1 == kExPasses) break;
        E += kExStep;
    }
    if (!valid || h.flags) {
        if (out_loglik) *out_loglik = -INFINITY;
        return BV_ENOTPD;
    }
    const double logdet = h.term[0], quad = h.term[1];
    if (out_logdet) *out_logdet = logdet;
    if (out_quad) *out_quad = quad;
    if (out_loglik) *out_loglik = -0.5 * (quad + logdet + (double)n * 1.8378770664093454835606594728112);
    return BV_OK;
}

extern "C" int bv_exact_flops(int64_t n, double* flops) {
    if (n <= 0 || !flops) return BV_EINVAL;
    const double N = (double)(n + 1);
    *flops = N * N * N / 3.0 + N * N;  // Cholesky of the augmented matrix, leading terms
    return BV_OK;
}

extern "C" int bv_kl_divergence(bv_ctx* c, const bv_theta* theta, int32_t precision, double* out_kl,
                                double* out_logdet_exact, double* out_logdet_approx) {
    if (!c || !theta || !out_kl) return BV_EINVAL;
    if (!c->have_nn) return BV_ESTATE;
    // log-determinants do not depend on y: any observations (zeros if none) serve
    if (!c->have_y) {
        std::vector<double> zero(c->n_tot, 0.0);
        BV_TRY(bv_set_observations(c, zero.data(), 0));
    }
    double d0 = 0.0, da = 0.0, la = 0.0;
    BV_TRY(bv_exact_loglik(c, theta, 0, nullptr, nullptr, &d0));
    BV_TRY(bv_loglik_terms(c, theta, precision, &la, nullptr, &da));
    if (out_logdet_exact) *out_logdet_exact = d0;
    if (out_logdet_approx) *out_logdet_approx = da;
    // Eq. 7 with tr(Sigma_a^-1 Sigma_0) = n for Vecchia-type approximations:
    // KL = ell_0(theta; 0) - ell_a(theta; 0) = (log|Sigma_a| - log|Sigma_0|) / 2
    *out_kl = 0.5 * (da - d0);
    return BV_OK;
}
