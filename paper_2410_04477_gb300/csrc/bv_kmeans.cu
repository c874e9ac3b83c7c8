// bv_kmeans.cu -- K-means blocks on the GPU (Sec. 2.1; Algorithm 1 "Clustering").
//
// The paper names K-means without fixing its details; this library fixes them so the
// blocks are a deterministic function of (locations, k, seed, iterations), identical
// bit for bit to the plain definition:
//   * squared distance D2(x, c) = sum_k (x_k - c_k)^2, left to right, every -, * and +
//     rounded separately (no fused multiply-add);
//   * k-means++ seeding (Arthur and Vassilvitskii 2007): first centre = point
//     floor(r_0 n / 2^64); centre t is drawn with probability proportional to D2 to the
//     nearest chosen centre, on integer weights w_j = floor(D2_j 2^s) with s fixed from n
//     and the bounding box (sum w < 2^62): target = floor(r_t W / 2^64), the pick is the
//     first point whose inclusive prefix sum of w exceeds the target (W = 0: point
//     floor(r_t n / 2^64));
//   * Lloyd iterations: nearest centre with the lowest index on ties; centre = mean of its
//     members computed as ((double)S / count) 2^-q from the exact int64 sum S of
//     llrint(x 2^q); an empty cluster keeps its centre; a final assignment after the last
//     update gives the labels.
// r_t = SplitMix64 draw t of stream BV_STREAM_KPP(seed).
//
// GPU formulation.  The assignment scans all centres with FP32 arithmetic to find, per
// point, the smallest FP32 squared distance d32min; every centre whose FP32 distance is
// within a proven rounding margin of d32min is then re-scored with the exact FP64 rule.
// The margin bounds |d32 - D2| (coordinate rounding to FP32, the subtraction, the
// squares and the sum), so the exact minimiser is always among the re-scored centres.
// Centroid sums are exact integers (order-free atomics), so the update is bit-exact.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "bv_fix.cuh"
#include "bv_internal.h"

namespace {

// Exact squared distance, no contraction.
__device__ __forceinline__ double d2_exact(const double* x, const double* c, int d) {
    double acc = 0.0;
    for (int k = 0; k < d; ++k) {
        const double t = __dsub_rn(x[k], c[k]);
        acc = __dadd_rn(acc, __dmul_rn(t, t));
    }
    return acc;
}

// Upper bound on |d32 - D2| for a squared distance whose FP32 value is about v, with
// coordinates bounded by amax in magnitude (derivation in the design notes: coordinate
// rounding eta = 1.01 u (|x|+|c|+|t|) <= 4.04 u amax per axis, error of the squares
// eta (2|t| + eta), FP32 sum rounding (d+1) u v; all doubled for safety).
__device__ __forceinline__ float fp32_margin(float v, float amax, int d) {
    const float u = 5.9604645e-8f;  // 2^-24
    const float eta = 4.04f * u * amax;
    const float D = sqrtf(fmaxf(v, 0.0f)) + 2.0f * eta;
    const float e = sqrtf((float)d) * eta * (2.0f * D + eta) + (float)(d + 2) * u * (v + 1e-30f);
    return 4.0f * e + 1e-30f;
}

constexpr int kTile = 256;  // centres per shared-memory tile

// Lloyd assignment.  x: SoA FP64 points [d][n_tot] (this dataset's slice at `off`), cent:
// row-major FP64 centres [k][d].  L lanes a point, each with every L-th centre.  One FP32 pass
// keeps the smallest two distances and the smallest one's centre: unless the second lies within
// the rounding margin of the first, that centre is the exact minimiser.  The few points where it
// does are scored exactly over the centres inside the margin.  76 us at n = 20,000, k = 2,000;
// scoring every point's candidates in a second pass over all centres, with one lane a point and
// half of the SMs without a block, took 218 us.
template <int L>
__global__ void __launch_bounds__(256) k_assign(const double* __restrict__ locs, int64_t n_tot,
                                                int64_t off, int64_t n, int d,
                                                const double* __restrict__ cent, int64_t k,
                                                float amax, int32_t* __restrict__ label) {
    __shared__ float4 cf[kTile];
    const int part = threadIdx.x % L;
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / L;
    const bool live = i < n;
    double x[3] = {0.0, 0.0, 0.0};
    if (live)
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (q < d) x[q] = locs[(int64_t)q * n_tot + off + i];
    const float xf[3] = {(float)x[0], (float)x[1], (float)x[2]};
    float best32 = INFINITY, second = INFINITY;
    int32_t bi = 0;
    for (int64_t c0 = 0; c0 < k; c0 += kTile) {
        const int nt = (int)min((int64_t)kTile, k - c0);
        __syncthreads();
        for (int t = threadIdx.x; t < nt; t += blockDim.x) {
            const double* cc = cent + (c0 + t) * d;
            cf[t] = make_float4((float)cc[0], d > 1 ? (float)cc[1] : 0.f, d > 2 ? (float)cc[2] : 0.f, 0.f);
        }
        __syncthreads();
#pragma unroll 4
        for (int t = part; t < nt; t += L) {
            const float4 c = cf[t];
            const float a0 = xf[0] - c.x, a1 = xf[1] - c.y, a2 = xf[2] - c.z;
            const float v = fmaf(a2, a2, fmaf(a1, a1, a0 * a0));
            second = fminf(second, fmaxf(v, best32));
            if (v < best32) {
                best32 = v;
                bi = (int32_t)(c0 + t);
            }
        }
    }
#pragma unroll
    for (int o = 1; o < L; o <<= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best32, o), os = __shfl_xor_sync(0xffffffffu, second, o);
        const int32_t oi = __shfl_xor_sync(0xffffffffu, bi, o);
        second = fminf(fminf(second, os), fmaxf(best32, ob));
        if (ob < best32) {
            best32 = ob;
            bi = oi;
        }
    }
    const float thr = best32 + 2.0f * fp32_margin(best32 * 1.001f, amax, d);
    const bool close = live && !(second > thr);
    if (__any_sync(0xffffffffu, close)) {
        // exact FP64 score of every centre inside the margin; the lowest index among equals
        double best = INFINITY;
        int32_t be = 0;
        if (close) {
            for (int64_t t = part; t < k; t += L) {
                const double* cc = cent + t * d;
                const float a0 = xf[0] - (float)cc[0], a1 = xf[1] - (d > 1 ? (float)cc[1] : 0.f),
                            a2 = xf[2] - (d > 2 ? (float)cc[2] : 0.f);
                if (fmaf(a2, a2, fmaf(a1, a1, a0 * a0)) <= thr) {
                    const double e = d2_exact(x, cc, d);
                    if (e < best) {
                        best = e;
                        be = (int32_t)t;
                    }
                }
            }
        }
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            const double ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int32_t oi = __shfl_xor_sync(0xffffffffu, be, o);
            if (ob < best || (ob == best && oi < be)) {
                best = ob;
                be = oi;
            }
        }
        if (close) bi = best < INFINITY ? be : 0;
    }
    if (live && part == 0) label[i] = bi;
}

// Four lanes a point until every SM has four warps a scheduler with one (the same labels).
cudaError_t launch_assign(const double* locs, int64_t n_tot, int64_t off, int64_t n, int d, const double* cent, int64_t k,
                          float amax, int32_t* label, cudaStream_t s) {
    if (n < 75000) k_assign<4><<<(unsigned)((4 * n + 255) / 256), 256, 0, s>>>(locs, n_tot, off, n, d, cent, k, amax, label);
    else k_assign<1><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(locs, n_tot, off, n, d, cent, k, amax, label);
    return cudaGetLastError();
}

// Exact integer centroid sums.
__global__ void k_accum(const double* __restrict__ locs, int64_t n_tot, int64_t off, int64_t n,
                        int d, const int32_t* __restrict__ label, int q,
                        unsigned long long* __restrict__ S, unsigned long long* __restrict__ cnt) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t c = label[i];
    atomicAdd(cnt + c, 1ull);
    for (int k = 0; k < d; ++k) {
        const long long v = llrint(ldexp(locs[(int64_t)k * n_tot + off + i], q));
        atomicAdd(S + c * d + k, (unsigned long long)v);
    }
}

__global__ void k_finalize(const unsigned long long* __restrict__ S,
                           const unsigned long long* __restrict__ cnt, int64_t k, int d, int q,
                           double* __restrict__ cent, int64_t* __restrict__ counts) {
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= k) return;
    const unsigned long long nc = cnt[c];
    if (counts) counts[c] = (int64_t)nc;
    if (nc == 0) return;
    for (int j = 0; j < d; ++j) {
        const long long s = (long long)S[c * d + j];
        cent[c * d + j] = ldexp(__ll2double_rn(s) / __ull2double_rn(nc), -q);
    }
}

// ---- k-means++ ---------------------------------------------------------------------
constexpr int kChunk = 1024;  // points per seeding chunk (one CTA)

// D2 <- min(D2, D2(x, c_new)) (or init), and exact per-chunk weight sums.
__global__ void __launch_bounds__(kChunk) k_kpp_update(const double* __restrict__ locs,
                                                       int64_t n_tot, int64_t off, int64_t n,
                                                       int d, const double* __restrict__ cnew,
                                                       int init, int s, double* __restrict__ D2,
                                                       unsigned long long* __restrict__ chunk_sum) {
    __shared__ unsigned long long red[kChunk / 32];
    const int64_t i = blockIdx.x * (int64_t)kChunk + threadIdx.x;
    unsigned long long w = 0;
    if (i < n) {
        double x[3];
        for (int q = 0; q < d; ++q) x[q] = locs[(int64_t)q * n_tot + off + i];
        const double v = d2_exact(x, cnew, d);
        double cur = init ? v : D2[i];
        if (!init && v < cur) cur = v;
        D2[i] = cur;
        w = (unsigned long long)ldexp(cur, s);
    }
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int j = 0; j < kChunk / 32; ++j) t += red[j];
        chunk_sum[blockIdx.x] = t;
    }
}

// Inclusive scan of one value per thread over a kChunk-thread block (exact integers).
__device__ __forceinline__ unsigned long long block_incl_scan(unsigned long long v,
                                                              unsigned long long* sh) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        unsigned long long x = lane < kChunk / 32 ? sh[lane] : 0ull;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        if (lane < kChunk / 32) sh[lane] = x;
    }
    __syncthreads();
    const unsigned long long r = v + (w > 0 ? sh[w - 1] : 0ull);
    __syncthreads();
    return r;
}

// Pick centre t: the first point whose inclusive prefix weight exceeds the target.  One
// CTA: scan of the chunk sums (in pieces of kChunk) to find the chunk, then a scan of
// that chunk's weights.
__global__ void __launch_bounds__(kChunk) k_kpp_pick(const double* __restrict__ locs,
                                                     int64_t n_tot, int64_t off, int64_t n, int d,
                                                     const double* __restrict__ D2, int s,
                                                     const unsigned long long* __restrict__ chunk_sum,
                                                     int64_t nchunks, uint64_t stream, int64_t t,
                                                     double* __restrict__ cent_t) {
    __shared__ unsigned long long sh[kChunk / 32];
    __shared__ unsigned long long s_base, s_total;
    __shared__ long long s_chunk, s_pick;
    const int tid = threadIdx.x;
    // exact total weight
    unsigned long long part = 0;
    for (int64_t c = tid; c < nchunks; c += kChunk) part += chunk_sum[c];
    const unsigned long long tot = block_incl_scan(part, sh);
    if (tid == kChunk - 1) s_total = tot;
    if (tid == 0) {
        s_pick = -1;
        s_chunk = -1;
    }
    __syncthreads();
    const unsigned long long W = s_total;
    const uint64_t r = bv_sm64(stream, (uint64_t)t);
    if (W == 0) {
        if (tid == 0) s_pick = (long long)__umul64hi(r, (uint64_t)n);
        __syncthreads();
    } else {
        const unsigned long long target = __umul64hi(r, W);
        unsigned long long base = 0;
        for (int64_t c0 = 0; c0 < nchunks; c0 += kChunk) {
            const int64_t c = c0 + tid;
            const unsigned long long v = c < nchunks ? chunk_sum[c] : 0ull;
            const unsigned long long inc = block_incl_scan(v, sh) + base;
            const unsigned long long exc = inc - v;
            if (c < nchunks && inc > target && exc <= target) {
                s_chunk = c;
                s_base = exc;
            }
            __syncthreads();
            if (s_chunk >= 0) break;
            // base for the next piece: inclusive value of the last thread
            if (tid == kChunk - 1) s_base = inc;
            __syncthreads();
            base = s_base;
            __syncthreads();
        }
        // s_chunk is always found (target < W); the clamps only keep indices in range
        const long long ch = s_chunk >= 0 ? s_chunk : nchunks - 1;
        const unsigned long long rem = s_chunk >= 0 ? target - s_base : 0ull;
        const int64_t i = ch * kChunk + tid;
        const unsigned long long w = i < n ? (unsigned long long)ldexp(D2[i], s) : 0ull;
        const unsigned long long inc = block_incl_scan(w, sh);
        if (i < n && inc > rem && inc - w <= rem) s_pick = (long long)i;
        __syncthreads();
    }
    __syncthreads();
    const long long pick = (s_pick >= 0 && s_pick < n) ? s_pick : n - 1;
    if (tid < d) cent_t[tid] = locs[(int64_t)tid * n_tot + off + pick];
}

// All picks of k-means++ in one launch, for sets that fit one cluster's registers: 8 CTAs of
// 1,024 threads, P consecutive points a thread, so that the order of (CTA, warp, lane, point)
// is the points' order.  The two launches a pick above cost their latency whatever the work: at
// n = 20,000 and k = 2,000 the set-up (K-means, neighbours) took 37.0 ms with them, and takes
// 13.2 ms with this kernel (8.4 ms) and the assignment above.  Here a pick is two cluster
// barriers: the CTAs exchange their weight sums; the one that holds the target scans its warps'
// sums and then that warp's lanes, and writes the new centre into every CTA's shared memory.
// Weights are whole numbers, so the sums (kept up to date by differences) do not depend on the
// order of additions.  A point's exact distance is only computed when its FP32 distance to the
// new centre is not above thr, its current distance and the rounding margin.
constexpr int kKppCtas = 8, kKppMaxP = 5;

// Barrier of all the cluster's threads, releasing and acquiring their writes to its shared memory.
// The .aligned form needs a converged warp, which a branch taken by some of its lanes does not
// leave by itself.
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int P>
__global__ void __cluster_dims__(kKppCtas, 1, 1) __launch_bounds__(kChunk, 1)
    k_kpp_all(const double* __restrict__ locs, int64_t n_tot, int64_t off, int64_t n, int d, int s, float amax, uint64_t stream,
              int64_t k, double* __restrict__ cent) {
    extern __shared__ double s_x[];                    // the CTA's points: coordinate q of point i at q kChunk P + i
    __shared__ double s_c[3];                          // the newest centre
    __shared__ unsigned long long s_sum[kKppCtas];     // weight sums of the CTAs
    __shared__ unsigned long long s_warp[kChunk / 32], s_tot, s_rem;
    __shared__ int s_w;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x;  // one cluster
    const int64_t i0 = ((int64_t)rank * kChunk + tid) * P;
    float xf[P][3], thr[P];
    double D2[P];
    unsigned long long w[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const bool live = i0 + p < n;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double v = live && q < d ? locs[(int64_t)q * n_tot + off + i0 + p] : 0.0;
            if (q < d) s_x[(q * kChunk + tid) * P + p] = v;
            xf[p][q] = (float)v;
        }
        thr[p] = live ? INFINITY : -1.0f;
        D2[p] = INFINITY;
        w[p] = 0;
    }
    if (lane == 0) s_warp[warp] = 0;
    if (tid == 0) s_tot = 0;
    if (tid < 3) s_c[tid] = tid < d ? cent[tid] : 0.0;
    cluster_sync();  // (another CTA's shared memory may be written once that CTA is known to run)
    for (int64_t t = 1; t < k; ++t) {
        const float c0 = (float)s_c[0], c1 = (float)s_c[1], c2 = (float)s_c[2];
        const uint64_t r = bv_sm64(stream, (uint64_t)t);
        unsigned long long dw = 0;  // change of the thread's weight (modulo 2^64)
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float a0 = xf[p][0] - c0, a1 = xf[p][1] - c1, a2 = xf[p][2] - c2;
            if (!(fmaf(a2, a2, fmaf(a1, a1, a0 * a0)) > thr[p])) {  // (also when FP32 overflows)
                double v = 0.0;  // d2_exact
                for (int q = 0; q < d; ++q) {
                    const double df = __dsub_rn(s_x[(q * kChunk + tid) * P + p], s_c[q]);
                    v = __dadd_rn(v, __dmul_rn(df, df));
                }
                if (v < D2[p]) {
                    D2[p] = v;
                    const unsigned long long wn = (unsigned long long)bvfix::scale2(v, s);  // as ldexp: exact, or below 1
                    dw += wn - w[p];
                    w[p] = wn;
                    const float vf = __double2float_ru(v);
                    thr[p] = vf + 2.0f * fp32_margin(vf * 1.001f, amax, d);
                }
            }
        }
        if (__any_sync(0xffffffffu, dw != 0)) {
            for (int o = 16; o > 0; o >>= 1) dw += __shfl_xor_sync(0xffffffffu, dw, o);
            if (lane == 0) {
                s_warp[warp] += dw;
                atomicAdd(&s_tot, dw);
            }
        }
        __syncthreads();
        if (tid < kKppCtas) {  // this CTA's sum into CTA tid's table
            uint32_t ra;
            const uint32_t la = (uint32_t)__cvta_generic_to_shared(s_sum + rank);
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(tid));
            asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(ra), "l"(s_tot) : "memory");
        }
        cluster_sync();
        unsigned long long W = 0;
#pragma unroll
        for (int q = 0; q < kKppCtas; ++q) W += s_sum[q];
        int owner = kKppCtas - 1;
        unsigned long long target = 0, base = 0;
        int64_t pick = -1;
        if (W == 0) {
            pick = (int64_t)__umul64hi(r, (uint64_t)n);
            owner = (int)(pick / ((int64_t)kChunk * P));
        } else {
            target = __umul64hi(r, W);
            for (int q = 0; q < kKppCtas; ++q) {  // the first CTA whose inclusive sum exceeds the target
                if (target < base + s_sum[q]) {
                    owner = q;
                    break;
                }
                base += s_sum[q];
            }
        }
        if (owner == rank) {
            if (W != 0) {
                if (warp == 0) {
                    const unsigned long long v = s_warp[lane];
                    unsigned long long inc = v;
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned long long u = __shfl_up_sync(0xffffffffu, inc, o);
                        if (lane >= o) inc += u;
                    }
                    const unsigned long long rem = target - base;
                    if (rem < inc && rem >= inc - v) {
                        s_w = lane;
                        s_rem = rem - (inc - v);
                    }
                }
                __syncthreads();
                if (warp == s_w) {
                    unsigned long long v = 0;
#pragma unroll
                    for (int p = 0; p < P; ++p) v += w[p];
                    unsigned long long inc = v;
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned long long u = __shfl_up_sync(0xffffffffu, inc, o);
                        if (lane >= o) inc += u;
                    }
                    unsigned long long rem = s_rem;
                    if (rem < inc && rem >= inc - v) {
                        rem -= inc - v;
#pragma unroll
                        for (int p = 0; p < P; ++p) {
                            if (pick < 0) {
                                if (rem < w[p]) pick = i0 + p;
                                else rem -= w[p];
                            }
                        }
                    }
                }
            }
            if (pick >= 0 && (W != 0 || tid == 0)) {  // one thread
                for (int q = 0; q < d; ++q) {
                    const double v = s_x[q * kChunk * P + (int)(pick - (int64_t)rank * kChunk * P)];  // a point of this CTA
                    cent[t * d + q] = v;
                    const uint32_t la = (uint32_t)__cvta_generic_to_shared(s_c + q);
                    for (int z = 0; z < kKppCtas; ++z) {
                        uint32_t ra;
                        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(z));
                        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
                    }
                }
            }
        }
        cluster_sync();
    }
}

}  // namespace

// Whether a cluster of the one-launch seeding can be placed on this device (a part of one may have no eight
// SMs of a cluster's size, or not the shared memory).  BV_FAULT_CLUSTER says no, for tests.
template <class K>
static bool kpp_cluster_fits(K kern, size_t smem) {
    const char* f = getenv("BV_FAULT_CLUSTER");
    if (f && *f && strcmp(f, "0") != 0) return false;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kKppCtas);
    cfg.blockDim = dim3(kChunk);
    cfg.dynamicSmemBytes = smem;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

static int ceil_log2_u64(uint64_t v) {
    int e = 0;
    while (e < 64 && ((uint64_t)1 << e) < v) ++e;
    return e;
}

int bv_kmeans_scales(const double* h, int64_t n, int d, int* s_out, int* q_out) {
    double lo[3], hi[3];
    for (int k = 0; k < d; ++k) lo[k] = hi[k] = h[k];
    for (int64_t i = 0; i < n; ++i)
        for (int k = 0; k < d; ++k) {
            const double v = h[i * d + k];
            lo[k] = std::min(lo[k], v);
            hi[k] = std::max(hi[k], v);
        }
    double d2max = 0.0, amax = 0.0;
    for (int k = 0; k < d; ++k) {
        const double e = hi[k] - lo[k];
        d2max += e * e;
        amax = std::max(amax, std::max(fabs(lo[k]), fabs(hi[k])));
    }
    int ed = 0, ea = 0;
    frexp(d2max, &ed);
    frexp(amax, &ea);
    const int ln = ceil_log2_u64((uint64_t)n);
    *s_out = 61 - ln - (ed + 1);
    *q_out = 61 - ln - (ea + 1);
    return BV_OK;
}

int bv_centroids_device(const double* d_locs, int64_t n_tot, int64_t off, int64_t n, int d,
                        const int32_t* d_label, int64_t k, int q, double* d_cent,
                        int64_t* d_counts, cudaStream_t s) {
    unsigned long long *S = nullptr, *cnt = nullptr;
    BV_CUDA(cudaMallocAsync(&S, sizeof(unsigned long long) * k * d, s));
    BV_CUDA(cudaMallocAsync(&cnt, sizeof(unsigned long long) * k, s));
    BV_CUDA(cudaMemsetAsync(S, 0, sizeof(unsigned long long) * k * d, s));
    BV_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * k, s));
    k_accum<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d_locs, n_tot, off, n, d, d_label, q, S, cnt);
    BV_CUDA(cudaGetLastError());
    k_finalize<<<(unsigned)((k + 255) / 256), 256, 0, s>>>(S, cnt, k, d, q, d_cent, d_counts);
    BV_CUDA(cudaGetLastError());
    BV_CUDA(cudaFreeAsync(S, s));
    BV_CUDA(cudaFreeAsync(cnt, s));
    return BV_OK;
}

// Full K-means of one dataset (points [off, off+n) of the SoA array): seeding, `iters`
// Lloyd iterations and the final assignment.  d_label[n] and d_cent[k x d] are outputs.
int bv_kmeans_device(const double* d_locs, int64_t n_tot, int64_t off, int64_t n, int d,
                     int64_t k, uint64_t seed, int iters, int32_t* d_label, double* d_cent,
                     cudaStream_t s) {
    // scales and the coordinate bound from a host copy of this slice
    std::vector<double> h((size_t)n * d);
    {
        std::vector<double> col((size_t)n);
        for (int q = 0; q < d; ++q) {
            BV_CUDA(cudaMemcpyAsync(col.data(), d_locs + (int64_t)q * n_tot + off, sizeof(double) * n,
                                    cudaMemcpyDeviceToHost, s));
            BV_CUDA(cudaStreamSynchronize(s));
            for (int64_t i = 0; i < n; ++i) h[(size_t)i * d + q] = col[(size_t)i];
        }
    }
    int sc = 0, q = 0;
    bv_kmeans_scales(h.data(), n, d, &sc, &q);
    double amax = 0.0;
    for (double v : h) amax = std::max(amax, fabs(v));

    const uint64_t stream = BV_STREAM_KPP(seed);
    const int64_t nchunks = (n + kChunk - 1) / kChunk;
    // first centre
    {
        const uint64_t r0 = bv_sm64(stream, 0);
        const int64_t first = (int64_t)(((unsigned __int128)r0 * (unsigned __int128)(uint64_t)n) >> 64);
        for (int q2 = 0; q2 < d; ++q2)
            BV_CUDA(cudaMemcpyAsync(d_cent + q2, d_locs + (int64_t)q2 * n_tot + off + first, sizeof(double),
                                    cudaMemcpyDeviceToDevice, s));
    }
    const int64_t per = (n + kKppCtas * kChunk - 1) / (kKppCtas * kChunk);  // points a thread of the one-launch form
    // (the shared-memory limit is the kernel's, not the call's: the same for all dimensions, so that calls
    // of several threads do not take it from one another)
    auto kern = per == 1 ? k_kpp_all<1> : per == 2 ? k_kpp_all<2> : per == 3 ? k_kpp_all<3> : per == 4 ? k_kpp_all<4> : k_kpp_all<5>;
    if (per <= kKppMaxP && kpp_cluster_fits(kern, sizeof(double) * kChunk * per * 3)) {
        const size_t sm = sizeof(double) * kChunk * per * d;
        kern<<<kKppCtas, kChunk, sm, s>>>(d_locs, n_tot, off, n, d, sc, (float)amax, stream, k, d_cent);
        BV_CUDA(cudaGetLastError());
    } else {
        double* D2 = nullptr;
        unsigned long long* csum = nullptr;
        BV_CUDA(cudaMallocAsync(&D2, sizeof(double) * n, s));
        BV_CUDA(cudaMallocAsync(&csum, sizeof(unsigned long long) * nchunks, s));
        for (int64_t t = 1; t < k; ++t) {
            k_kpp_update<<<(unsigned)nchunks, kChunk, 0, s>>>(d_locs, n_tot, off, n, d, d_cent + (t - 1) * d,
                                                              t == 1, sc, D2, csum);
            BV_CUDA(cudaGetLastError());
            k_kpp_pick<<<1, kChunk, 0, s>>>(d_locs, n_tot, off, n, d, D2, sc, csum, nchunks, stream, t,
                                            d_cent + t * d);
            BV_CUDA(cudaGetLastError());
        }
        BV_CUDA(cudaFreeAsync(D2, s));
        BV_CUDA(cudaFreeAsync(csum, s));
    }
    // Lloyd
    for (int it = 0; it < iters; ++it) {
        BV_CUDA(launch_assign(d_locs, n_tot, off, n, d, d_cent, k, (float)amax, d_label, s));
        BV_TRY(bv_centroids_device(d_locs, n_tot, off, n, d, d_label, k, q, d_cent, nullptr, s));
    }
    BV_CUDA(launch_assign(d_locs, n_tot, off, n, d, d_cent, k, (float)amax, d_label, s));
    return BV_OK;
}
