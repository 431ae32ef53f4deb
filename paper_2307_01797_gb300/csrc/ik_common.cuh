// ik_common.cuh -- device-side building blocks of libitokmc (sm_103a).
//
// Counter-based random numbers (Philox4x32-10, Salmon et al. SC'11), the
// uniform and normal maps, FP64 log/exp/sincos(2 pi u) written from their
// series so that every device agrees with any other IEEE-754 implementation
// of the same operation sequence, the Poisson sampler of the tau-leap, and
// grid helpers.  All translation units are compiled with -fmad=false: each
// FP64 expression below is evaluated as written, one rounding per operation.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ik {

// ---------------------------------------------------------------- parameters
// Kernel-argument copy of the configuration (one realization's grid; all
// realizations share it).
struct Params {
    int n, n3;              // cells per axis, cells per realization
    int R;                  // realizations
    int S;                  // particle species blocks: 1 (electrons), or 3 with mobile ions
    int B;                  // particle blocks S R: block b holds species b / R of realization b % R
    int log2n;
    int ppc, n_new, n_crit, n_ssa, frac_bits;
    int dep_win;            // largest shared deposit window (cells) a push block uses, <= DEP_WIN_MAX
    double lo[3], hi[3], h[3], rh[3];   // rh = 1/h
    // 1/h to 96 bits (cells are cubes): h = mh 2^h_exp with 53-bit mh, and
    // floor(2^148 / mh) in three words, lowest first
    uint32_t rh96[3];
    int h_exp;
    double dt, mu, D, alpha_A, alpha_B, eta, photon_ratio, kappa_lo, kappa_hi, eps;
    double sdt;             // sqrt(2 D dt)
    double k_ep, k_np;      // recombination frequencies per pair, beta / dV (1/s)
    double E0;
    uint64_t seed0;
    uint32_t step;
    // graph-replayed steps read the step counter from device memory (the
    // last node of a step advances it); otherwise null and step is used
    const uint32_t* step_dev;
    // FP32 form constants (cell units)
    float f_drift;          // -mu dt / h   (multiplies E in V/m)
    float f_diff;           // sqrt(2 D dt) / h
    // per species (electrons, positive ions, negative ions): drift
    // coefficient sgn(Z) mu (V = cmu E), sqrt(2 D dt), the FP32 form's
    // cmu dt / h and sqrt(2 D dt) / h, and the push and product stream tags
    double cmu_sp[3], sdt_sp[3];
    float f_drift_sp[3], f_diff_sp[3];
    uint32_t push_tag_sp[3], prod_tag_sp[3];
};

constexpr int DEP_WIN_MAX = 2048;   // cells of the push's shared deposit window (16 KB)

enum : uint32_t {
    TAG_INIT = 1u, TAG_PUSH = 2u, TAG_KMC = 3u, TAG_PRODUCT = 4u, TAG_PHOTON = 5u,
    TAG_PUSH_POS = 6u, TAG_PUSH_NEG = 7u, TAG_PRODUCT_POS = 8u, TAG_PRODUCT_NEG = 9u
};

// Device error word bits (OR-ed by kernels, read by the host after a stage).
enum : uint32_t {
    DERR_CAPACITY = 1u, DERR_OVERFLOW = 2u, DERR_KMC = 4u, DERR_TIMEOUT = 8u, DERR_INTERNAL = 16u
};

// ---------------------------------------------------------------- Philox
struct u32x4 { uint32_t x, y, z, w; };

__device__ __forceinline__ u32x4 philox10(u32x4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = u32x4{ hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0 };
    }
    return c;
}

// A draw stream (key = seed, counter = (index, step, tag<<24|sub, block));
// words are consumed in order, a block is generated every four words.
// (2k+1) 2^-53 for a 52-bit k, assembled from its bits with integer
// instructions (the value is exact: 2k+1 < 2^53).
__device__ __forceinline__ double u53(uint64_t k)
{
    const uint64_t m = 2ull * k + 1ull;
    const int p = 63 - __clzll((long long)m);            // leading bit, 0..52
    const uint64_t bits = ((uint64_t)(p - 53 + 1023) << 52) | ((m << (52 - p)) & 0x000fffffffffffffull);
    return __longlong_as_double((long long)bits);
}

// m 2^-53 for m < 2^53, exact.
__device__ __forceinline__ double u53_mul(uint64_t m)
{
    if (m == 0) return 0.0;
    const int p = 63 - __clzll((long long)m);
    return __longlong_as_double((long long)(((uint64_t)(p - 53 + 1023) << 52) | ((m << (52 - p)) & 0x000fffffffffffffull)));
}

struct Stream {
    uint32_t k0, k1, c0, c1, c2, blk;
    u32x4 buf;
    int pos;
    __device__ __forceinline__ Stream(uint64_t seed, uint32_t index, uint32_t step, uint32_t tag,
                                      uint32_t sub)
        : k0((uint32_t)seed), k1((uint32_t)(seed >> 32)), c0(index), c1(step),
          c2((tag << 24) | sub), blk(0), buf{0, 0, 0, 0}, pos(4) {}
    __device__ __forceinline__ uint32_t u32()
    {
        if (pos == 4) {
            buf = philox10(u32x4{ c0, c1, c2, blk }, k0, k1);
            ++blk;
            pos = 0;
        }
        const uint32_t v = pos == 0 ? buf.x : pos == 1 ? buf.y : pos == 2 ? buf.z : buf.w;
        ++pos;
        return v;
    }
    // uniform on (0,1): k = 52 random bits, (2k+1) 2^-53 (exact)
    __device__ __forceinline__ double uniform() { return u53(bits52()); }
    __device__ __forceinline__ uint64_t bits52()
    {
        const uint32_t a = u32();
        const uint32_t b = u32();
        return ((uint64_t)a << 20) | (uint64_t)(b >> 12);
    }
};

// The stream consumed two words at a time (the word order of Stream): pair
// k is words 2k, 2k+1; uniform() is the FP64 uniform of the next pair,
// uniform32() the FP32 uniform of its high word.
struct PairStream {
    uint32_t k0, k1, c0, c1, c2, blk;
    u32x4 buf;
    bool hi_half;                 // next pair is (buf.z, buf.w)
    __device__ __forceinline__ PairStream(uint64_t seed, uint32_t index, uint32_t step, uint32_t tag, uint32_t sub)
        : k0((uint32_t)seed), k1((uint32_t)(seed >> 32)), c0(index), c1(step), c2((tag << 24) | sub), blk(0),
          buf{ 0, 0, 0, 0 }, hi_half(false)
    {
        buf = philox10(u32x4{ c0, c1, c2, blk }, k0, k1);
        ++blk;
    }
    __device__ __forceinline__ void pair(uint32_t& a, uint32_t& b)
    {
        if (hi_half) {
            a = buf.z; b = buf.w;
            buf = philox10(u32x4{ c0, c1, c2, blk }, k0, k1);
            ++blk;
        } else {
            a = buf.x; b = buf.y;
        }
        hi_half = !hi_half;
    }
    __device__ __forceinline__ double uniform()
    {
        uint32_t a, b;
        pair(a, b);
        return u53((((uint64_t)a) << 20) | (uint64_t)(b >> 12));
    }
    __device__ __forceinline__ float uniform32();
};

// FP32 uniform on (0,1) from the high word of an FP64 uniform: its top 23
// bits k give (2k+1) 2^-24 (exact in FP32), the FP64 uniform to within an
// FP32 ulp.
__device__ __forceinline__ float uniform_f32(uint32_t v)
{
    return (float)(2u * (v >> 9) + 1u) * 0x1p-24f;
}

__device__ __forceinline__ float PairStream::uniform32()
{
    uint32_t a, b;
    pair(a, b);
    return uniform_f32(a);
}

// ---------------------------------------------------------------- FP64 math
// log: x = 2^e m, m in [1/sqrt2, sqrt2); s = (m-1)/(m+1);
// ln m = 2s + 2s z P(z), z = s^2, P(z) = sum_{j=0..9} z^j / (2j+3).
// ln x = e*LN2_HI + (e*LN2_LO + ln m); LN2_HI = ln2 with 21 low bits cleared.
__device__ __forceinline__ double dlog(double x)
{
    if (!(x > 0.0)) return (x == 0.0) ? -__longlong_as_double(0x7ff0000000000000ll) : __longlong_as_double(0x7ff8000000000000ll);
    if (x == __longlong_as_double(0x7ff0000000000000ll)) return x;
    int e = 0;
    uint64_t b = (uint64_t)__double_as_longlong(x);
    int bexp = (int)((b >> 52) & 0x7ff);
    if (bexp == 0) {
        x = x * 0x1p54;
        e = -54;
        b = (uint64_t)__double_as_longlong(x);
        bexp = (int)((b >> 52) & 0x7ff);
    }
    e += bexp - 1023;
    double m = __longlong_as_double((long long)((b & 0x000fffffffffffffull) | 0x3ff0000000000000ull));
    if (m > 1.41421356237309504880) { m = m * 0.5; e += 1; }
    const double f = m - 1.0;
    const double s = f / (2.0 + f);
    const double z = s * s;
    double p = 1.0 / 21.0;
    p = __fma_rn(p, z, 1.0 / 19.0);
    p = __fma_rn(p, z, 1.0 / 17.0);
    p = __fma_rn(p, z, 1.0 / 15.0);
    p = __fma_rn(p, z, 1.0 / 13.0);
    p = __fma_rn(p, z, 1.0 / 11.0);
    p = __fma_rn(p, z, 1.0 / 9.0);
    p = __fma_rn(p, z, 1.0 / 7.0);
    p = __fma_rn(p, z, 1.0 / 5.0);
    p = __fma_rn(p, z, 1.0 / 3.0);
    const double t = 2.0 * s;
    const double lnm = __fma_rn(t, z * p, t);
    const double de = (double)e;
    return de * 6.93147180369123816490e-01 + (de * 1.90821492927058770002e-10 + lnm);
}

// exp: n = rint(x / ln2), r = (x - n LN2_HI) - n LN2_LO, Taylor to r^13.
__device__ __forceinline__ double dexp(double x)
{
    if (x != x) return x;
    if (x > 709.78) return __longlong_as_double(0x7ff0000000000000ll);
    if (x < -745.2) return 0.0;
    const double nd = rint(x * 1.44269504088896340736);
    const double r = (x - nd * 6.93147180369123816490e-01) - nd * 1.90821492927058770002e-10;
    double p = 1.0 / 6227020800.0;
    p = __fma_rn(p, r, 1.0 / 479001600.0);
    p = __fma_rn(p, r, 1.0 / 39916800.0);
    p = __fma_rn(p, r, 1.0 / 3628800.0);
    p = __fma_rn(p, r, 1.0 / 362880.0);
    p = __fma_rn(p, r, 1.0 / 40320.0);
    p = __fma_rn(p, r, 1.0 / 5040.0);
    p = __fma_rn(p, r, 1.0 / 720.0);
    p = __fma_rn(p, r, 1.0 / 120.0);
    p = __fma_rn(p, r, 1.0 / 24.0);
    p = __fma_rn(p, r, 1.0 / 6.0);
    p = __fma_rn(p, r, 0.5);
    p = __fma_rn(p, r, 1.0);
    p = __fma_rn(p, r, 1.0);
    const int n = (int)nd;
    if (n > 1023) return (p * 2.0) * __longlong_as_double((long long)(n - 1 + 1023) << 52);
    if (n < -1020) {
        const double sc = p * __longlong_as_double((long long)(n + 600 + 1023) << 52);
        return sc * 0x1p-600;
    }
    return p * __longlong_as_double((long long)(n + 1023) << 52);
}

// sin and cos of 2 pi u: q = rint(4u), f = 4u - q, a = f pi/2, Taylor series
// of sin a through a^17 and cos a through a^18, quadrant by q mod 4.
__device__ __forceinline__ void dsincos2pi(double u, double* so, double* co)
{
    const double t = 4.0 * u;
    const double q = rint(t);
    const double f = t - q;
    const double a = f * 1.57079632679489661923;
    const double z = a * a;
    double sp = -1.0 / 355687428096000.0;
    sp = __fma_rn(sp, z, 1.0 / 1307674368000.0);
    sp = __fma_rn(sp, z, -1.0 / 6227020800.0);
    sp = __fma_rn(sp, z, 1.0 / 39916800.0);
    sp = __fma_rn(sp, z, -1.0 / 362880.0);
    sp = __fma_rn(sp, z, 1.0 / 5040.0);
    sp = __fma_rn(sp, z, -1.0 / 120.0);
    sp = __fma_rn(sp, z, 1.0 / 6.0);
    const double sa = __fma_rn(-a, z * sp, a);
    double cp = 1.0 / 6402373705728000.0;
    cp = __fma_rn(cp, z, -1.0 / 20922789888000.0);
    cp = __fma_rn(cp, z, 1.0 / 87178291200.0);
    cp = __fma_rn(cp, z, -1.0 / 479001600.0);
    cp = __fma_rn(cp, z, 1.0 / 3628800.0);
    cp = __fma_rn(cp, z, -1.0 / 40320.0);
    cp = __fma_rn(cp, z, 1.0 / 720.0);
    cp = __fma_rn(cp, z, -1.0 / 24.0);
    cp = __fma_rn(cp, z, 0.5);
    const double ca = __fma_rn(-z, cp, 1.0);
    switch (((int)q) & 3) {
    case 0: *so = sa; *co = ca; break;
    case 1: *so = ca; *co = -sa; break;
    case 2: *so = -sa; *co = -ca; break;
    default: *so = -ca; *co = sa; break;
    }
}

// ---------------------------------------------------------------- Poisson
// log k!: exact product below 10, Stirling series through k^-7 above.
__device__ __forceinline__ double dlogfact(int64_t k)
{
    if (k < 10) {
        double f = 1.0;
        for (int64_t i = 2; i <= k; ++i) f = f * (double)i;
        return dlog(f);
    }
    const double x = (double)k;
    const double r = 1.0 / x;
    const double r2 = r * r;
    double ser = 1.0 / 1680.0;
    ser = 1.0 / 1260.0 - r2 * ser;
    ser = 1.0 / 360.0 - r2 * ser;
    ser = 1.0 / 12.0 - r2 * ser;
    ser = r * ser;
    return (((x + 0.5) * dlog(x) - x) + 0.91893853320467274178) + ser;
}

// ---- pairs of floats: a value hi + lo to about 2^-44
// The Poisson draws are whole numbers: FP64 arithmetic only decides floors and
// comparisons.  These pairs decide the same ones outside a margin that covers
// their error many times over, with FP32 instructions (GB300 issues 64 of them
// in the time of one FP64 instruction); inside the margin FP64 decides (5e-5 of
// the trials, 2e-3 of the logarithmic tests).  k_kmc over a channel with
// recombination on 128^3 is bound by that pipe: 857 us with FP64 draws, 224 us
// with these (6.26 million FP64 warp instructions to 2.74 million).
struct FF { float h, l; };
__device__ __forceinline__ FF ff_norm(float h, float l)            // |h| >= |l|
{
    const float s = h + l;
    return FF{ s, l - (s - h) };
}
__device__ __forceinline__ FF ff_add(FF a, FF b)
{
    const float s = a.h + b.h, t = s - a.h, e = (a.h - (s - t)) + (b.h - t);
    return ff_norm(s, e + (a.l + b.l));
}
__device__ __forceinline__ FF ff_mul(FF a, FF b)
{
    const float p = a.h * b.h, e = __fmaf_rn(a.h, b.h, -p);
    return ff_norm(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e)));
}
__device__ __forceinline__ FF ff_div(FF a, FF b)
{
    const float q = __fdividef(a.h, b.h);
    const float r = __fmaf_rn(-q, b.h, a.h) + __fmaf_rn(-q, b.l, a.l);      // a - q b
    return ff_norm(q, __fdividef(r, b.h));
}
// The constant c to 48 bits.
#define IK_FF(c) (FF{ (float)(c), (float)((c) - (double)(float)(c)) })
// m 2^-53 for m < 2^53.
__device__ __forceinline__ FF ff_frac53(uint64_t m)
{
    const float h = (float)(uint32_t)(m >> 29), l = (float)(uint32_t)(m & 0x1fffffffu);   // 24 and 29 bits
    return ff_norm(h * 0x1p-24f, l * 0x1p-53f);
}
// The same for small m: its own leading bits.
__device__ __forceinline__ FF ff_small53(uint64_t m)
{
    const int z = __clzll((long long)m) - 11;                      // m > 0
    const FF f = ff_frac53(m << z);
    const float sc = __int_as_float((127 - z) << 23);
    return FF{ f.h * sc, f.l * sc };
}
// A positive double in float's range.
__device__ __forceinline__ FF ff_from(double v)
{
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int e = (int)(b >> 52) - 1023;
    const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);
    const FF f = ff_frac53(m);                                     // v 2^-(e + 1)
    const float sc = __int_as_float((e + 128) << 23);
    return FF{ f.h * sc, f.l * sc };
}

// One PTRS acceptance test by logarithms, in FP64 (the specification).
static __device__ __noinline__ bool ptrs_log_test(double mu, double kd, double us, double V)
{
    const double b = 0.931 + 2.53 * sqrt(mu);
    const double a = -0.059 + 0.02483 * b;
    const double invalpha = 1.1239 + 1.1328 / (b - 3.4);
    // the acceptance test as one logarithm (Hoermann's form)
    const double lhs = dlog((V * invalpha) / ((a / (us * us)) + b));
    const double rhs = ((-mu) + kd * dlog(mu)) - dlogfact((int64_t)kd);
    return lhs <= rhs;
}
// The trial's count and its test against vr, in FP64.
static __device__ __noinline__ double ptrs_trial(double mu, double U, double us, double V, bool& below_vr)
{
    const double b = 0.931 + 2.53 * sqrt(mu);
    const double a = -0.059 + 0.02483 * b;
    below_vr = V <= 0.9277 - 3.6224 / (b - 2.0);
    return floor(((((2.0 * a) / us) + b) * U + mu) + 0.43);
}
// Inversion by sequential search, in FP64.
static __device__ __noinline__ int64_t poisson_search(double mu, double u)
{
    double p = dexp(-mu);
    double F = p;
    int64_t k = 0;
    while (u > F && k < 200) {
        k += 1;
        p = (p * mu) / (double)k;
        F = F + p;
    }
    return k;
}

// P(mu): 0 without a draw for mu <= 0; inversion by sequential search (one
// uniform) for mu < 10; PTRS transformed rejection (Hoermann 1993, two
// uniforms per trial) above.  Returns -1 if PTRS exhausts its trial limit.
__device__ __forceinline__ int64_t dpoisson_inl(Stream& s, double mu)
{
    if (!(mu > 0.0)) return 0;
    const bool small = mu < 10.0;
    // the pairs serve means up to 2^24; a search whose first term would leave
    // float's range does not occur (exp(-10) = 4.5e-5), a mean near 0 does
    const bool pairs = mu < 0x1p24 && mu > 0x1p-60;
    const FF m = ff_from(pairs ? mu : 1.0);
    if (small) {
        const uint32_t a = s.u32(), c = s.u32();
        const uint64_t ku = ((uint64_t)a << 20) | (uint64_t)(c >> 12);
        if (pairs) {
            // errors below 1e-5: expf and p to 1e-6 relative over the few steps
            const float u = ff_frac53(2 * ku + 1).h, mf = m.h;
            float p = expf(-mf), F = p;
            int k = 0;
            bool clear = fabsf(u - F) > 1e-5f;
            while (clear && u > F && k < 100) {
                k += 1;
                p = __fdividef(p * mf, (float)k);
                F += p;
                clear = fabsf(u - F) > 1e-5f;
            }
            if (clear && k < 100) return k;
        }
        return poisson_search(mu, u53(ku));
    }
    // b, a and vr of the transformed rejection
    const float r0 = sqrtf(m.h), rl = __fdividef(__fmaf_rn(-r0, r0, m.h) + m.l, r0 + r0);
    const FF b = ff_add(IK_FF(0.931), ff_mul(IK_FF(2.53), ff_norm(r0, rl)));
    const FF a = ff_add(IK_FF(-0.059), ff_mul(IK_FF(0.02483), b));
    const float vr = 0.9277f - __fdividef(3.6224f, b.h - 2.0f);
    const float invalpha = 1.1239f + __fdividef(1.1328f, b.h - 3.4f);
    for (int it = 0; it < 1000000; ++it) {
        const uint32_t w0 = s.u32(), w1 = s.u32(), w2 = s.u32(), w3 = s.u32();
        const uint64_t ku = 2ull * (((uint64_t)w0 << 20) | (uint64_t)(w1 >> 12)) + 1ull;
        const uint64_t kv = 2ull * (((uint64_t)w2 << 20) | (uint64_t)(w3 >> 12)) + 1ull;
        // U = ku 2^-53 - 1/2, us = 1/2 - |U| and V = kv 2^-53 are exact: so are
        // the comparisons among them
        const bool neg = ku < (1ull << 52);
        const uint64_t au = neg ? (1ull << 52) - ku : ku - (1ull << 52), kus = (1ull << 52) - au;
        const FF us = ff_small53(kus), Uabs = ff_frac53(au);
        const FF U = neg ? FF{ -Uabs.h, -Uabs.l } : Uabs;
        double kd = 0.0;
        int64_t kk = 0;
        bool below_vr = false, known = false;
        if (pairs) {
            const FF q = ff_div(FF{ 2.0f * a.h, 2.0f * a.l }, us);
            const FF v = ff_add(ff_add(ff_mul(ff_add(q, b), U), m), IK_FF(0.43));
            const float fh = floorf(v.h), fr = (v.h - fh) + v.l, fl = floorf(fr), at = fr - fl;
            const float slack = 1e-5f + (m.h + fabsf(v.h)) * 0x1p-38f, dv = ff_frac53(kv).h - vr;
            known = at > slack && at < 1.0f - slack && fabsf(dv) > 1e-5f && fabsf(v.h) < 0x1p30f;
            kk = (int64_t)(int)fh + (int)fl;
            below_vr = dv < 0.0f;
        }
        if (!known) {
            kd = ptrs_trial(mu, neg ? -u53_mul(au) : u53_mul(au), u53_mul(kus), u53_mul(kv), below_vr);
            kk = (int64_t)kd;
        }
        if (kus >= 630503947831870ull && below_vr) return kk;             // us >= 0.07
        const bool negk = known ? kk < 0 : kd < 0.0;
        if (negk || (kus < 117093590311633ull && kv > kus)) continue;     // us < 0.013
        if (known && kk >= 4 && us.h > 1e-9f) {
            // k ln mu - mu - ln k! = -(k h(x) + ln(2 pi k) / 2 + 1 / 12 k - 1 / 360 k^3 + ...)
            // with x = (mu - k) / k, h(x) = x - ln(1 + x): errors below 1e-4
            const float kf = (float)kk, d = (m.h - kf) + (m.l - (float)(kk - (int64_t)kf));
            const float x = __fdividef(d, kf);
            const float h = fabsf(x) < 0.05f
                                ? x * x * (0.5f + x * (-1.0f / 3.0f + x * (0.25f + x * (-0.2f + x * (1.0f / 6.0f + x * (-1.0f / 7.0f))))))
                                : x - log1pf(x);
            const float rk = __fdividef(1.0f, kf);
            const float rhs = -(kf * h) - 0.5f * logf(6.2831853f * kf) - rk * (1.0f / 12.0f - rk * rk * (1.0f / 360.0f));
            const float lhs = logf(__fdividef(ff_frac53(kv).h * invalpha, __fdividef(a.h, us.h * us.h) + b.h));
            const float gap = rhs - lhs;
            // kf h carries the relative errors of d and of the logarithm
            if (fabsf(gap) > 1e-3f + kf * h * 1e-4f) {
                if (gap > 0.0f) return kk;
                continue;
            }
        }
        if (ptrs_log_test(mu, known ? (double)kk : kd, u53_mul(kus), u53_mul(kv))) return kk;
    }
    return -1;
}
static __device__ __noinline__ int64_t dpoisson(Stream& s, double mu) { return dpoisson_inl(s, mu); }

// An exponential time -ln(u) / A, u the uniform of the bits k; infinity where
// it lies above the limit for certain (the caller does nothing else with such
// a time), which FP32 decides for most draws.  logf and the rounding of u
// to 24 bits are off by less than 2e-7 (1 + l).
static __device__ __noinline__ double exp_time_exact(uint64_t k, double A) { return (-dlog(u53(k))) / A; }
__device__ __forceinline__ double exp_time(Stream& s, double A, double limit)
{
    const uint64_t k = s.bits52();
    const float l = -logf(ff_frac53(2 * k + 1).h);
    if (l - 1e-5f * (1.0f + l) > (float)(A * limit) * 1.00001f) return __longlong_as_double(0x7ff0000000000000ll);
    return exp_time_exact(k, A);
}

// ---------------------------------------------------------------- grid
__device__ __forceinline__ int clampi(int i, int n) { return i < 0 ? 0 : (i > n - 1 ? n - 1 : i); }

// CIC stencil along one axis for an absolute coordinate (FP64 form):
// u = (x - lo)/h - 1/2, i0 = floor(u), f = u - i0, indices folded to [0,n-1].
// (x-lo)/h in grid units: q0 = d r, q = q0 + (d - q0 h) r with r = 1/h (one
// fused correction; the same operations as the specification's).
__device__ __forceinline__ double grid_quot(double x, double lo, double h, double rh)
{
    // x - 0 is x itself (also for -0): a domain corner at 0 (uniform across
    // the launch) needs no subtraction on the FP64 pipe
    double d = x;
    if (__double_as_longlong(lo) != 0) d = x - lo;
    const double q0 = d * rh;
    return __fma_rn(__fma_rn(-q0, h, d), rh, q0);
}

// a / b given r = 1/b, with the same fused correction.
__device__ __forceinline__ double quot_r(double a, double b, double r)
{
    const double q0 = a * r;
    return __fma_rn(__fma_rn(-q0, b, a), r, q0);
}

// Cell of a coordinate known to lie in [lo, hi): floor((x-lo)/h), clamped.
__device__ __forceinline__ int cell_axis(double x, double lo, double h, double rh, int n)
{
    const int i = (int)floor(grid_quot(x, lo, h, rh));
    return i > n - 1 ? n - 1 : (i < 0 ? 0 : i);
}

// Cell quotients qd in [1/2, 2^31) split from their bits.  For such qd the
// stencil coordinate u = qd - 1/2 is exact (1/2 is a multiple of ulp(qd)),
// and so are floor(u), the fraction f = u - floor(u) = F 2^-sh and
// floor(f 2^s) = F >> (sh - s): the FP64 subtract / floor / convert
// sequence yields the same values, and these integer steps keep the FP64
// pipe (a small fraction of the FP32 rate on GB300) for the arithmetic
// that rounds.  qc = floor(qd) is the cell index.
struct QSplit {
    int qc, i0, sh;
    unsigned long long F, fb;        // fb 2^-sh = qd - qc
};
__device__ __forceinline__ bool qsplit(double qd, QSplit& r)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(qd);
    const int e = (int)(b >> 52);                  // biased exponent (>= 2048 when negative)
    if (e < 1022 || e > 1053) return false;        // qd < 1/2, qd >= 2^31, negative, NaN
    const unsigned long long m = (b & 0xfffffffffffffull) | (1ull << 52);
    const int sh = 1075 - e;                       // fraction bits of qd, 22..53
    const unsigned long long fb = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    r.qc = (int)(m >> sh);
    r.sh = sh;
    r.fb = fb;
    if (fb >= half) { r.i0 = r.qc; r.F = fb - half; }
    else { r.i0 = r.qc - 1; r.F = fb + half; }
    return true;
}
// The quotient q = (x - lo) / h of axis a (grid_quot) rounded to 53 bits and
// split, by integer multiplication with the 96-bit reciprocal: the product's
// upper 96 bits are within a few units of 2^-96 of the quotient, and grid_quot's
// result is the quotient rounded to nearest up to an error of 2^-52 units of
// the last place before its rounding; so both round the same way unless the
// bits below the 53rd lie within 2^-29 of a half.  Those, and quotients
// outside qsplit's range, return false (the caller takes grid_quot).  GB300 has
// 2 FP64 lanes per SM and clock: the three FP64 instructions of a quotient
// hold the pipe for the time in which an SM issues 192 others.  (Products
// rounded by integer instructions, about 50 each, gained nothing.)
__device__ __forceinline__ bool quot_split(const Params& P, double x, int a, QSplit& r)
{
    double d = x;
    if (__double_as_longlong(P.lo[a]) != 0) d = x - P.lo[a];
    const uint32_t dh = (uint32_t)__double2hiint(d), dl = (uint32_t)__double2loint(d);
    const int e = (int)(dh >> 20);                  // biased exponent (>= 2048 when negative)
    const uint32_t m1 = (dh << 11) | (dl >> 21) | 0x80000000u, m0 = dl << 11;
    const uint64_t u = (uint64_t)m1 * P.rh96[1], v = (uint64_t)m0 * P.rh96[2];
    const uint64_t w = (uint64_t)(uint32_t)u + (uint32_t)v + __umulhi(m1, P.rh96[0]) + __umulhi(m0, P.rh96[1]);
    uint64_t top = (uint64_t)m1 * P.rh96[2] + (u >> 32) + (v >> 32) + (w >> 32);
    uint32_t g = (uint32_t)w;
    int E = e - 1075 - P.h_exp;                     // q = top 2^(E - 63)
    if (!(top >> 63)) {
        top = (top << 1) | (g >> 31);
        g <<= 1;
        --E;
    }
    const uint32_t low = ((uint32_t)top << 21) | (g >> 11);
    const int sh = 52 - E;                          // fraction bits
    if (e == 0 || e >= 2047 || sh < 22 || sh > 53 || low - 0x7ffffffcu <= 8u) return false;
    const uint64_t m = (top >> 11) + (low >> 31);
    const uint64_t fb = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    r.qc = (int)(m >> sh);
    r.sh = sh;
    r.fb = fb;
    if (fb >= half) { r.i0 = r.qc; r.F = fb - half; }
    else { r.i0 = r.qc - 1; r.F = fb + half; }
    return true;
}
// x >= lo and x < hi by order-preserving integer keys (-0 taken as +0; a NaN
// fails one of the two tests, as in the FP64 comparisons).
__device__ __forceinline__ unsigned long long dkey(double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    b = b == 0x8000000000000000ull ? 0ull : b;
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__device__ __forceinline__ uint64_t seed_of(const Params& P, int r) { return P.seed0 + (uint64_t)r; }
// The step counter of the Philox streams.
__device__ __forceinline__ uint32_t step_of(const Params& P) { return P.step_dev ? *P.step_dev : P.step; }

// Particle block b: species b / R, realization b % R (at most three species:
// two comparisons instead of a division).
__host__ __device__ __forceinline__ int species_of(const Params& P, int b) { return (b >= P.R) + (b >= 2 * P.R); }
__host__ __device__ __forceinline__ int phys_of(const Params& P, int b) { return b - species_of(P, b) * P.R; }

// ---------------------------------------------------------------- warp helpers
__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// Inclusive segmented sum over runs of equal keys that are contiguous in
// lane order; returns true in the last lane of each run (which then holds
// the run total in v / c).
__device__ __forceinline__ bool warp_run_sum(uint32_t key, bool valid, unsigned long long& v,
                                             unsigned& c)
{
    const unsigned lane = lane_id();
    const unsigned full = 0xffffffffu;
    const uint32_t kprev = __shfl_up_sync(full, key, 1);
    const bool vprev = __shfl_up_sync(full, valid ? 1 : 0, 1);
    const bool head = (lane == 0) || !vprev || kprev != key || !valid;
    const unsigned heads = __ballot_sync(full, head);
    // segment start lane for this lane: highest head at or below lane
    const unsigned below = heads & (0xffffffffu >> (31 - lane));
    const int seg_start = 31 - __clz(below);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long ov = __shfl_up_sync(full, v, d);
        const unsigned oc = __shfl_up_sync(full, c, d);
        if ((int)lane - d >= seg_start) { v += ov; c += oc; }
    }
    const uint32_t knext = __shfl_down_sync(full, key, 1);
    const bool vnext = __shfl_down_sync(full, valid ? 1 : 0, 1);
    const bool tail = (lane == 31) || !vnext || knext != key;
    return valid && tail;
}

}  // namespace ik
