// bv_fix.cuh -- 64-bit fixed-point arithmetic of the FP64-accurate block kernel
// (bv_fix_ll.cu): products, reciprocal square root, exponential and the closed-form Matern
// correlation, on the integer pipe.
//
// Why: this part's SM executes 2 FP64 lanes per clock but 64 or more 32 x 32 -> 64-bit
// integer multiply-adds.  A correlation matrix normalised to a unit diagonal has entries,
// Schur complements and factor entries all in [-1, 1], so 64-bit fixed point holds them
// with an absolute error of 2^-60 or less, where FP64 arithmetic leaves 2^-54 on values
// near 1.
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define BV_FIX __device__ __forceinline__
#else  // host build of the arithmetic's own test
#include <string.h>
#define BV_FIX static inline
#endif

namespace bvfix {

#ifdef __CUDACC__
BV_FIX int clz64(uint64_t v) { return __clzll((long long)v); }
BV_FIX float rsq32(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
BV_FIX int f2i(float x) { return __float2int_rn(x); }
BV_FIX uint64_t dbits(double x) { return (uint64_t)__double_as_longlong(x); }
BV_FIX double bitsd(uint64_t x) { return __longlong_as_double((long long)x); }
#else
BV_FIX int clz64(uint64_t v) { return v ? __builtin_clzll(v) : 64; }
BV_FIX float rsq32(float x) { return (float)(1.0 / sqrt((double)x)) * (1.0f + 1.2e-7f); }  // a last-bit error, as the unit has
BV_FIX int f2i(float x) { return (int)rintf(x); }
BV_FIX uint64_t dbits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
BV_FIX double bitsd(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
#endif

// v 2^e, |e| <= 2040 (exact unless the result is subnormal); ldexp without its special cases.
BV_FIX double scale2(double v, int e) {
    const int a = e / 2;
    return v * bitsd((uint64_t)(1023 + a) << 52) * bitsd((uint64_t)(1023 + e - a) << 52);
}

BV_FIX uint32_t hi32(uint64_t a) { return (uint32_t)(a >> 32); }
BV_FIX uint32_t lo32(uint64_t a) { return (uint32_t)a; }

// a b + c, 32 x 32 + 64 bits: one instruction, 64 lanes a clock (written out, since the
// compiler does not always see that both factors are 32 bits wide).
#ifdef __CUDACC__
BV_FIX int64_t smad(int32_t a, int32_t b, int64_t c) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
    return c;
}
BV_FIX uint64_t umad(uint32_t a, uint32_t b, uint64_t c) {
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
    return c;
}
#else
BV_FIX int64_t smad(int32_t a, int32_t b, int64_t c) { return (int64_t)((uint64_t)((int64_t)a * b) + (uint64_t)c); }
BV_FIX uint64_t umad(uint32_t a, uint32_t b, uint64_t c) { return (uint64_t)a * b + c; }
#endif

// High 64 bits of a b within 2 units, without bias (the low x low product is left out and the
// middle one cut off, 0.75 units on average, which are added); a, b < 2^63, so that the two
// middle products sum without a carry: three multiply-adds.
BV_FIX uint64_t mulhi63(uint64_t a, uint64_t b) {
    const uint64_t mid = umad(hi32(a), lo32(b), umad(lo32(a), hi32(b), 0xC0000000ull));
    return umad(hi32(a), hi32(b), hi32(mid));
}
// The same for any a, b.
BV_FIX uint64_t mulhi64(uint64_t a, uint64_t b) {
    const uint64_t p = umad(hi32(a), lo32(b), 0xA0000000ull), q = umad(lo32(a), hi32(b), 0xA0000000ull);
    return umad(hi32(a), hi32(b), hi32(p)) + hi32(q);
}

// A signed 64-bit value as h 2^32 + l with both halves signed (l in [-2^31, 2^31)), so that
// all partial products are signed 32 x 32 -> 64.
struct Bal {
    int32_t h, l;
};
BV_FIX Bal bal(int64_t v) {
    Bal b;
    b.l = (int32_t)(uint32_t)v;
    b.h = (int32_t)(((uint64_t)v + 0x80000000ull) >> 32);
    return b;
}
// a / b in units 2^-63, rounded, for finite 0 < a <= b (host).  A rounding of sigma^2 / D to FP64's
// 53 bits would be up to 64 units of 2^-60, of one sign in every covariance entry of a dataset.
inline uint64_t ratio63(double a, double b) {
    int ea = 0, eb = 0;
    unsigned __int128 rem = (uint64_t)ldexp(frexp(a, &ea), 53);
    const uint64_t den = (uint64_t)ldexp(frexp(b, &eb), 53);
    uint64_t q = rem >= den ? 1 : 0;
    rem -= q ? den : 0;
    const int bits = 63 + ea - eb;  // (<= 63: a <= b)
    if (bits < -1) return 0;
    if (bits < 0) return q;         // a / b in [2^-65, 2^-63), rounded at 2^-64
    for (int i = 0; i < bits; ++i) {
        rem <<= 1;
        q <<= 1;
        if (rem >= den) {
            rem -= den;
            ++q;
        }
    }
    return q + (2 * rem >= den ? 1 : 0);
}

// Scales: matrix entries and Schur complements in units of 2^-60 (kUnitC), factor entries in
// units of 2^-59 (kUnitL).
constexpr int kUnitC = 60, kUnitL = 59;

// A factor entry x = h 2^29 + l for products: h h exactly on the integer pipe, the two cross
// products in FP32, whose accumulators are half as wide: they are below 2^-31 |x| |y|, so that
// FP32's 2^-24 leaves 2^-55 |x| |y|; l l is below 2^-62.
struct Fac {
    int32_t h;
    float hf, lf;  // h and l 2^-31
};
BV_FIX Fac fac(int64_t x) {
    Fac f;
    f.h = (int32_t)((x + (1ll << 28)) >> 29);
    f.hf = (float)f.h;
    f.lf = (float)((int32_t)((uint32_t)x << 3) >> 3) * 4.656612873077392578125e-10f;
    return f;
}
// a 2^-60 + c 2^-58 -= x y.
BV_FIX void msub(int64_t& a, float& c, int32_t nxh, float nxhf, float nxlf, int32_t yh, float yhf, float ylf) {
    a = smad(nxh, yh, a);
    c = fmaf(nxhf, ylf, c);
    c = fmaf(nxlf, yhf, c);
}

// a - x^2 in matrix units for a factor entry x = h 2^29 + l, rounded: h h, 2 h l and l l (to 14 bits
// of l) in whole numbers.  In FP32, as in msub, the cross term of an x near 1 errs by up to 2^-55,
// and l l, left out, raises every pivot by 2^-63.6 a column.
BV_FIX int64_t sub_square(int64_t a, int64_t x, int32_t h) {
    const int32_t l = (int32_t)((uint32_t)x << 3) >> 3, lq = l >> 15;
    return smad(-h, h, a) - (smad(h, l, smad(lq, lq, 1ll << 27)) >> 28);
}

// Largest size of a solved data entry, as a power of two: below 2^-row_limit(N).  A row of the
// factor has a norm of at most 1, so the data row's Schur complements stay below 2^-5 + sqrt(N)
// 2^-row_limit(N) < 4.1, in the range of +-8 of a 64-bit entry in matrix units (and entries below
// 1/2 keep the digits' sums in range).
BV_FIX int row_limit(int n) {
    int g = 1;
    while (n > 16 << (2 * g)) ++g;
    return g;
}

// 1 / sqrt(P), P = p 2^-60, for p in [1, 2^60]: r 2^(e - 62) with r in [2^62, 2^63) and e >= 0,
// within 2^-59 relative and exact for P = 1.  The hardware seed's mantissa Y (24 bits, error
// 2^-22) takes a Newton step with the second-order term in fixed point, which cubes its error.
struct Rsq {
    int64_t r;
    int e;
};
BV_FIX uint32_t fbits(float x) {
#ifdef __CUDACC__
    return __float_as_uint(x);
#else
    uint32_t u;
    memcpy(&u, &x, 4);
    return u;
#endif
}
BV_FIX Rsq rsqrt_fix(int64_t p) {
    Rsq o;
    const float pf = fmaf((float)(int32_t)hi32((uint64_t)p), 4294967296.0f, (float)lo32((uint64_t)p));
    const uint32_t u = fbits(rsq32(pf));
    const uint32_t Y = (u & 0x7fffffu) | 0x800000u;       // units 2^-23
    o.e = (int)(u >> 23) - 127 + 30;
    const uint64_t M = (uint64_t)p << (2 * o.e + 3);      // P 4^e in (1/4, 1], units 2^-63
    const int64_t e60 = (1ll << 60) - (int64_t)mulhi63(M, umad(Y, Y, 0) << 15);  // 1 - P 4^e y^2
    const int32_t es = (int32_t)(e60 >> 20);              // units 2^-40
    const int64_t c = e60 + (smad(es, es + es + es, 0) >> 22);  // e + 3 e^2 / 4
    const int64_t pr = smad((int32_t)Y, (int32_t)(c >> 16), smad((int32_t)Y, (int32_t)(c & 0xffff), 0) >> 16);
    o.r = ((int64_t)Y << 39) + (pr >> 6);                 // y (1 + c / 2)
    return o;
}

// sqrt(M) 2^31 for M in [2^62, 2^64), within 2^-62 relative: 24 bits from the hardware
// reciprocal square root and two residual corrections.
BV_FIX uint64_t sqrt_fix(uint64_t M) {
    const float mf = (float)hi32(M);                    // M 2^-32 in [2^30, 2^32]
    const float y = rsq32(mf);
    const uint32_t s0 = (uint32_t)f2i(mf * y * 256.0f);  // sqrt(M) 2^-8
    const int64_t r = (int64_t)(M - (umad(s0, s0, 0) << 16));
    const float h = y * 7.62939453125e-6f;               // 1 / (2 sqrt(M)): y 2^-16 / 2
    const int32_t c1 = f2i((float)(int32_t)(r >> 13) * (h * 67108864.0f));        // r h in units 2^-13
    const int64_t r2 = (int64_t)((uint64_t)r << 16) - (int64_t)((uint64_t)smad((int32_t)s0, c1, 0) << 12) - (smad(c1, c1, 0) >> 10);
    const int32_t c2 = f2i((float)(int32_t)(r2 >> 9) * (h * 33554432.0f));        // units 2^-32
    return ((uint64_t)s0 << 39) + (uint64_t)((int64_t)c1 << 18) + (uint64_t)(int64_t)(c2 >> 1);
}

// The scaled distance x = sqrt(acc) of a normal acc > 0 as x = X 2^(q - 63), X in
// [2^62, 2^63), from acc's 53-bit significand.
struct Dist {
    uint64_t X;
    int q;
};
BV_FIX Dist dist_fix(uint64_t accbits) {
    Dist o;
    const int k = (int)(accbits >> 52) - 1023;
    o.q = (k >> 1) + 1;
    o.X = sqrt_fix(((accbits & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << (10 + (k & 1)));
    return o;
}

// Tables of the exponential: A[j] = 2^(-j/256) w in units 2^-62 (w <= 1, a weight of the
// caller's) and B[j] = 2^(-j/65536) in units 2^-63 (B[0] one unit below 1).
BV_FIX uint64_t shr(uint64_t v, int n) { return v >> (n < 63 ? n : 63); }

// w e^-x = w 2^-z from z in units 2^-57: W 2^-i with W in units 2^-61.  z = i + j1/256 +
// j2/65536 + g: tables for the middle parts, e^-r - 1 for r = g ln 2 < 2^-16 as -r + (r^2/2 -
// r^3/6) with the bracket in FP32 (below 2^-33, its rounding below 2^-57 of the result).
struct Exp {
    uint64_t W;
    int i;
};
template <typename TA, typename TB>
BV_FIX Exp exp2_fix(uint64_t zf, const TA* A, const TB* B) {
    const uint64_t r = mulhi63((zf & 0x1FFFFFFFFFFull) << 22, 0x58B90BFBE8E7BCD6ull);  // units 2^-78; ln 2 in 2^-63
    const float rf = (float)(int32_t)hi32(r);                      // units 2^-46
    const int32_t q2 = f2i(rf * rf * 1.862645149230957e-9f * (1.0f - rf * 4.736951571734001e-15f));  // r^2/2 - r^3/6, 2^-64
    const uint64_t E = r - ((uint64_t)(uint32_t)q2 << 14);
    const uint64_t P = mulhi63(A[(zf >> 49) & 255], B[(zf >> 41) & 255]);
    Exp o;
    o.W = P - ((mulhi63(P, E) + 8192) >> 14);
    o.i = (int)(zf >> 57);
    return o;
}

// w rho(x) in matrix units for the closed forms: nu = 0 (1/2), 1 (3/2) or 2 (5/2), for K scaled
// distances at once (independent chains that the compiler interleaves; one copy of the code for
// all nu, which branch on it only for the polynomial).  x >= 64 gives 0 (rho below 2^-80).
template <int K, typename TA, typename TB>
BV_FIX void matern_fix(int nu, const Dist (&x)[K], const TA* A, const TB* B, int64_t (&out)[K]) {
    Exp e[K];
    uint64_t v[K];
    int q[K];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < K; ++k) {
        const uint64_t Z = mulhi63(x[k].X, 0x5C551D94AE0BF85Eull);  // log2 e in units 2^-62
        q[k] = x[k].q > 6 ? 6 : x[k].q < -55 ? -55 : x[k].q;
        const int sh = 6 - q[k];
        e[k] = exp2_fix(((Z << 2) + ((1ull << sh) >> 1)) >> sh, A, B);
        v[k] = shr(e[k].W, e[k].i);
    }
    if (nu > 0) {
        uint64_t H[K];
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int k = 0; k < K; ++k) {
            H[k] = mulhi63(x[k].X, e[k].W);                         // units 2^(q - 60)
            v[k] += shr(H[k] << 1, e[k].i - q[k]);
        }
        if (nu > 1) {
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int k = 0; k < K; ++k) {
                const uint64_t H2 = mulhi63(x[k].X, mulhi63(H[k], 0x5555555555555555ull));  // units 2^(2 q - 59)
                v[k] += shr(H2 << 6, e[k].i - 2 * q[k] + 4);
            }
        }
    }
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < K; ++k) out[k] = x[k].q > 6 ? 0 : (int64_t)((v[k] + 1) >> 1);
}

// The general smoothness: rho = e^-(x - L(x)), L a polynomial of degree DEG - 1 in t = 2 m - 3
// on each octave x = m 2^o, m in [1, 2), its coefficients (power basis, units 2^-57, |L| < 64)
// at tab + (o + OCT0) DEG, evaluated by Horner's rule.  For 2^-OCT0 <= x; x >= 128 gives 0.
template <int DEG, int OCT0, typename TA, typename TB>
BV_FIX int64_t matern_gen_fix(Dist x, const int64_t* tab, const TA* A, const TB* B) {
    const int q = x.q > 7 ? 7 : x.q < 1 - OCT0 ? 1 - OCT0 : x.q;
    const int64_t* c = tab + (q - 1 + OCT0) * DEG;
    const Bal t = bal((int64_t)(2 * x.X) - (3ll << 62));           // units 2^-62
    int64_t b = c[DEG - 1];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = DEG - 2; k >= 0; --k) {
        const Bal y = bal(b);
        const int64_t mid = smad(y.h, t.l, smad(y.l, t.h, 1ll << 29));
        b = c[k] + (int64_t)((uint64_t)smad(y.h, t.h, 0) << 2) + (mid >> 30);
    }
    const uint64_t xf = q > 6 ? x.X << 1 : x.X >> (6 - q);         // x in units 2^-57
    const int64_t y = (int64_t)(xf - (uint64_t)b);                 // x - L; from 64 on its sign bit is set
    const bool far = x.q > 7 || (q >= 6 && y < 0) || (q == 7 && b <= 0);
    const uint64_t yc = y < 0 ? 0 : (uint64_t)y;
    const Exp e = exp2_fix(mulhi64(yc, 0xB8AA3B295C17F0BCull) << 1, A, B);  // log2 e in units 2^-63
    return far ? 0 : (int64_t)((shr(e.W, e.i) + 1) >> 1);
}

// A double in [0, 1] in matrix units, truncated.
BV_FIX int64_t unit_fix(double v) {
    const uint64_t b = dbits(v);
    const int k = (int)(b >> 52) - 1023;  // v = 1.f 2^k, k <= 0
    if (k < -61) return 0;
    return (int64_t)(((b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 8 >> (-k));
}

// High 64 bits of the signed product a b, up to a unit off (the low x low product is left out);
// |a|, |b| < 2^63 - 2^31.
BV_FIX int64_t mulh(int64_t a, int64_t b) {
    const Bal x = bal(a), y = bal(b);
    return smad(x.h, y.h, smad(x.h, y.l, smad(x.l, y.h, 0)) >> 32);
}

// Tables of the Box-Muller pairs: c[j] 2^-15 ~ 1 / (1 + (j + 1/2) / 256) (1 for j = 0, 1/2 for
// j = 255), with -ln of it -- of its double where j >= kLnHalf -- in units 2^-60, and cosine and
// sine of (pi / 2) (j + 1/2) / 256 in units 2^-62.
constexpr int kLnHalf = 106;  // 1 + 106/256: about sqrt(2)
struct SimTab {
    uint16_t c[256];
    int64_t ln[256];
    int64_t cs[256], sn[256];
};

// One pair: two uniforms u1 = 1 - k1 2^-53, u2 = k2 2^-53 give rho = sqrt(-2 ln u1) and the
// angle 2 pi u2.  V = rho^2 in units 2^-56, rho = X 2^(q - 63) (X = 0 for u1 = 1), cs and sn in
// units 2^-62; all within a few 2^-57.
struct Pair {
    uint64_t V, X;
    int q;
    int64_t cs, sn;
};
BV_FIX Pair pair_fix(uint64_t k1, uint64_t k2, const SimTab& T) {
    Pair o;
    {   // -ln u1 = -e ln 2 - ln c^-1 - ln(1 + r), u1 = m 2^e, r = m c - 1, |r| < 2^-7.9
        const uint64_t U = (1ull << 53) - k1;
        const int lz = clz64(U);
        const uint64_t M = U << lz;                      // m 2^63
        const int j = (int)(M >> 55) & 255;
        const uint32_t c = T.c[j];
        const int64_t hi = (int64_t)umad(hi32(M), c, 0) - (1ll << 46);  // (m c - 1) 2^46, top part
        const int64_t R = (int64_t)((uint64_t)hi << 24) + (int64_t)(umad(lo32(M), c, 0) >> 8);  // r, units 2^-70
        const float r = (float)(int32_t)(R >> 32) * 3.637978807091713e-12f;     // units 2^-38
        const float g = fmaf(r, fmaf(r, fmaf(r, -1.0f / 7.0f, 1.0f / 6.0f), -0.2f), 0.25f);
        const int64_t t1 = 0x1555555555555555ll - ((int64_t)f2i(r * g * 1099511627776.0f) << 22);  // 1/3 - r g, units 2^-62
        const int64_t t2 = (1ll << 61) - (mulh(R, t1) >> 6);                                       // 1/2 - r t1
        const int64_t l = (R >> 10) - (mulh(mulh(R, R), t2) >> 14);             // ln(1 + r), units 2^-60
        const int e = 10 - lz + (j >= kLnHalf);
        // -e ln 2 in units 2^-58 (up to 2^63.2, unsigned), ln 2 to 4 more bits
        const uint64_t S = (uint64_t)(-e) * 0x2C5C85FDF473DE6ull + (uint64_t)((-e * 11 + 8) >> 4) - (uint64_t)((T.ln[j] + l + 2) >> 2);
        o.V = (S + 1) >> 1;                              // 2 (-ln u1) in units 2^-56
    }
    {
        const int sh = clz64(o.V | 1) & ~1;
        o.q = 4 - (sh >> 1);
        o.X = o.V ? sqrt_fix(o.V << sh) : 0;
    }
    {   // angle (pi / 2) (quarter + f): f's top 8 bits by table, the rest d = (pi / 2) 2^-8 f'
        const uint64_t A = k2 << 11;
        const int quarter = (int)(A >> 62), j = (int)(A >> 54) & 255;
        const int64_t D = mulh((int64_t)((A << 10) ^ (1ull << 63)) >> 1, 0x3243F6A8885A308Dll);  // units 2^-68; pi / 2 in 2^-61
        const int64_t D2 = mulh(D, D);                   // units 2^-72, < 2^-16.6
        const float d2 = (float)(int32_t)(D2 >> 26) * 1.4210854715202004e-14f;   // units 2^-46
        const int64_t c1 = -(D2 >> 7) + (int64_t)f2i(d2 * d2 * fmaf(d2, -1.0f / 720.0f, 1.0f / 24.0f) * 7.378697629483821e19f);  // cos d - 1, 2^-66
        // d^2 / 6 - d^4 / 120, units 2^-70
        const int64_t t = (mulh(D2, 0x2AAAAAAAAAAAAAABll) >> 2) - (int64_t)f2i(d2 * d2 * (1.0f / 120.0f) * 1.180591620717411e21f);
        const int64_t s1 = D - (mulh(D, t) >> 6);        // sin d, units 2^-68
        const int64_t C = T.cs[j], S = T.sn[j];
        const int64_t x = C + (mulh(C, c1) >> 2) - (mulh(S, s1) >> 4);
        const int64_t y = S + (mulh(S, c1) >> 2) + (mulh(C, s1) >> 4);
        const int64_t a = quarter & 1 ? y : x, b = quarter & 1 ? x : y;
        o.cs = quarter == 1 || quarter == 2 ? -a : a;
        o.sn = quarter >= 2 ? -b : b;
    }
    return o;
}

}  // namespace bvfix
