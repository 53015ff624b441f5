// eri_fixaux.cuh -- the auxiliary integrals [r]^(0) of one primitive quartet
// (Eqs. boys, 0m and r-rr) in 64-bit fixed point.
//
// The FP64 path spends 24 (L = 0) to 800 (L = 8) FP64 instructions on a
// primitive quartet, at 17 clocks per warp and SM each (68 on the quarter of the
// SM a warp lives in); the integer pipe does a 64-bit product in three
// multiply-adds of 1.1 clocks and about ten other instructions.
//
// Quantities and units (powers of two unless said otherwise):
//  * u = 1/zeta of either side, as mantissa and exponent; w = u_p + u_q = 1/rho;
//    V = 1/sqrt(w) (a float seed and one third-order step), rho = V^2.  The
//    prefactor is V once zeta^(-3/2) of each side is in its E products.
//  * X = P - Q from fixed coordinates, exact; T = rho X^2.
//  * Boys: F_n by five-term Taylor expansion about the nearest grid point
//    T_j = j/256, with every order n = 0..L straight from the row's F_n..F_n+5.
//    Row j holds F_m alpha_j^m (alpha_j real, chosen so that F_m alpha_j^m <= F_0 for
//    every m of the row), so a large T costs no relative precision.
//    T >= 320: F_n = (2n-1)!! / (2T)^n sqrt(pi/T)/2 (erf(sqrt T) = 1).
//  * recursion: R^(n)_t of order N is held times u^-(N + 2n), u^2 = 2 rho / alpha_j
//    (kappa / |X| for T >= 320): then R^(n)_0 = (-1)^n F_n alpha^n, and
//    [t+1]^(n) = (X u) [t]^(n+1) + t [t-1]^(n+1) without further factors.
//    Order N carries a shift of N bits more (it exceeds R_0 by up to (N-1)!!), so
//    a step is (X u / 2) [t]^(n+1) + (t/4) [t-1]^(n+1).  The last step multiplies order N by V (u / s)^N, s = 2^sigma the
//    Hermite unit of the transforms.
//
// Every value keeps 2^-60 of the largest it may have, where FP64 keeps 2^-53 of itself.
// Checked on the host against long double (tests/test_fixed_aux_cpu.py).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "eri_internal.h"

namespace eri {

constexpr int kFixBoysInvStep = 256, kFixBoysLog2 = 8;
constexpr int kFixBoysRows = (int)(kBoysTmax * kFixBoysInvStep) + 1;
constexpr int kFixBoysK = 5;         // Taylor terms beyond the first
constexpr int kFixAuxLmax = 10;      // largest order of the fixed-point auxiliary integrals
// Bits kept free above F_0 for the recursion of order L, whose values pass it
constexpr int fix_headroom(int L) { return L > 8 ? 1 : 0; }
// 8-byte words of a table row of order L: F_m alpha^m 2^(h - headroom), m = 0..L+5, in
// units of 2^-61; sqrt(2/alpha) in units of 2^-60; 1/alpha in units
// of 2^-31 (low word) and h - headroom (high word)
constexpr int fix_boys_words(int L) { return (L + kFixBoysK + 4) & ~1; }
// constants of T >= 320 for order L, 8-byte words: sqrt(pi)/2 (2n-1)!! kappa^(-2n),
// n = 0..kFixAuxLmax, in units of 2^-61, then kappa in units of 2^-60
constexpr int kFixFarWords = kFixAuxLmax + 2;

// One primitive pair: centre in units of 2^-f, 1/zeta = um 2^(ue - 62), um in [2^61, 2^62)
struct alignas(8) FixPrim {
    long long x[3];
    long long um;
    int ue;
    float zeta;
};

#ifdef __CUDACC__
#define FIX_HD __host__ __device__ __forceinline__
#else
#define FIX_HD inline
#endif

FIX_HD int fix_clz(unsigned long long v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
FIX_HD float fix_rsqrt_seed(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / std::sqrt(x);
#endif
}
FIX_HD float fix_pow2(int e)  // -126 <= e <= 127
{
#ifdef __CUDA_ARCH__
    return __int_as_float((127 + e) << 23);
#else
    return std::ldexp(1.0f, e);
#endif
}
FIX_HD unsigned fix_float_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned b;
    std::memcpy(&b, &x, 4);
    return b;
#endif
}

FIX_HD float fix_inverse(float x)  // correctly rounded
{
#ifdef __CUDA_ARCH__
    return __frcp_rn(x);
#else
    return 1.0f / x;
#endif
}

// sigma with mu 2^sigma >= 1.1 sqrt(2 rho), at most a factor 2 above; c = 2.42 / mu^2
FIX_HD int fix_sigma(float rho, float c)
{
    const int e = (int)(fix_float_bits(c * rho) >> 23) - 127;  // 2^e <= y < 2^(e+1)
    return (e + 2) >> 1;
}
// Reduced exponent of two sums of exponents.  Every operation is rounded to
// nearest, so it never falls as zb grows: the tile's scales rely on that, and
// zb (zk / (zb + zk)) does fall, by its last place, in one of twelve steps.
FIX_HD float fix_reduced(float zb, float zk) { return fix_inverse(fix_inverse(zb) + fix_inverse(zk)); }

// two consecutive 8-byte words, 16-byte aligned
FIX_HD void fix_load2(const long long* p, long long& a, long long& b)
{
#ifdef __CUDA_ARCH__
    const longlong2 v = __ldg(reinterpret_cast<const longlong2*>(p));
    a = v.x;
    b = v.y;
#else
    a = p[0];
    b = p[1];
#endif
}

// v = hi 2^32 + lo with lo signed
FIX_HD int fix_lo(long long v) { return (int)v; }
FIX_HD int fix_hi(long long v) { return (int)(v >> 32) + (int)((unsigned)(int)v >> 31); }
FIX_HD long long fix_wide(int a, int b) { return (long long)a * b; }

// a b 2^-62 for |a|, |b| <= 2^62 (one unit off at most)
FIX_HD long long fix_mul62(long long a, long long b)
{
    const int a1 = fix_hi(a), a0 = fix_lo(a), b1 = fix_hi(b), b0 = fix_lo(b);
    return (fix_wide(a1, b1) << 2) + ((fix_wide(a1, b0) + (1LL << 29)) >> 30) + (fix_wide(a0, b1) >> 30);
}

// 2^61 / sqrt(W 2^-62) for W in [2^60, 2^62], to a unit or two: result in [2^61, 2^62]
FIX_HD long long fix_rsqrt(long long W)
{
    const unsigned w1 = (unsigned)((unsigned long long)W >> 32), w0 = (unsigned)W;
    float y = fix_rsqrt_seed((float)w1 * 0x1p-30f);
    y = y < 1.99999988f ? y : 1.99999988f;
    const unsigned yb = fix_float_bits(y);
    const unsigned Y = yb >= 0x3f800000u ? ((yb & 0x7fffffu) | 0x800000u) : 0x800000u;  // y 2^23
    const unsigned long long Y2 = (unsigned long long)Y * Y;                            // y^2 2^46
    const unsigned y1 = (unsigned)(Y2 >> 32), y0 = (unsigned)Y2;
    // E = 2^62 (1 - W 2^-62 y^2)
    unsigned long long m = (unsigned long long)w0 * y0;
    m = (unsigned long long)w0 * y1 + (m >> 32);
    m = (unsigned long long)w1 * y0 + m;
    const long long E = (1LL << 62) - (long long)((((unsigned long long)w1 * y1) << 18) + (m >> 14));
    // (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ...
    const int Eh = (int)(E >> 20);
    const long long c = (E >> 1) + ((3 * fix_wide(Eh, Eh)) >> 25);
    return ((long long)Y << 38) + (((long long)Y * (c >> 4)) >> 20);
}

// The scales of one primitive quartet's integrals.
struct FixBase {
    long long V;    // prefactor: V 2^(ve - 61)
    int ve;
    int ue;         // u = U 2^(ue - 62)
    long long U;
    long long x[3]; // X u / 2 in units of 2^-58
};

// F[n] = (-alpha)^n F_n, n = 0..L (units 2^-61), and the scales.
// L <= LMAX; with L a constant every loop unrolls.
template <int LMAX>
FIX_HD void fix_base(int L, const FixPrim& p, const FixPrim& q, int f, const long long* __restrict__ tab,
                     const long long* __restrict__ far, long long (&F)[LMAX + 1], FixBase& b)
{
    // P - Q, scaled up to 62 bits; |X|^2 = S 2^(64 - 2 nx - 2 f)
    long long d[3];
    unsigned long long top = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        d[i] = p.x[i] - q.x[i];
        top |= (unsigned long long)(d[i] ^ (d[i] >> 63));
    }
    const int nx = fix_clz(top | 1) - 2;
    long long S = 0, c = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        d[i] = (long long)((unsigned long long)d[i] << nx);
        const int x1 = fix_hi(d[i]), x0 = fix_lo(d[i]);
        S += fix_wide(x1, x1);
        c += fix_wide(x1, x0);
    }
    S += c >> 31;
    // 1/rho = W 2^(e - 62), W in [2^60, 2^62), e even; 1/sqrt of it V 2^(-61 - e/2)
    int e = p.ue > q.ue ? p.ue : q.ue;
    const int dp = e - p.ue, dq = e - q.ue;
    long long W = (p.um >> (dp < 63 ? dp : 63)) + (q.um >> (dq < 63 ? dq : 63));
    const int s1 = (int)(W >> 62);
    W >>= s1;
    e += s1;
    const int s2 = e & 1;
    W >>= s2;
    e = (e + s2) >> 1;
    const long long V = fix_rsqrt(W);
    const int v1 = fix_hi(V), v0 = fix_lo(V);
    const long long VV = (fix_wide(v1, v1) << 2) + (fix_wide(v1, v0) >> 29);  // rho = VV 2^(-60 - 2e)
    const int q1 = fix_hi(VV), q0 = fix_lo(VV), r1 = fix_hi(S), r0 = fix_lo(S);
    const long long TT = (fix_wide(r1, q1) << 3) + ((fix_wide(r1, q0) + fix_wide(r0, q1)) >> 29);
    const int sT = 2 * (nx + f + e) - 118;  // T 2^53 = TT 2^-sT
    const long long Tend = (long long)kBoysTmax << 53;
    if (sT >= 0 ? (TT >> (sT < 63 ? sT : 63)) < Tend : (sT > -62 && TT < (Tend >> -sT))) {
        const long long Tf = sT >= 0 ? (sT < 63 ? TT >> sT : 0) : TT << -sT;
        const int j = (int)((Tf + (1LL << (52 - kFixBoysLog2))) >> (53 - kFixBoysLog2));
        const long long md = ((long long)j << (53 - kFixBoysLog2)) - Tf;  // (T_j - T) 2^53, |md| <= 2^45
        const long long* row = tab + (size_t)j * fix_boys_words(L);
        const long long w = row[L + kFixBoysK + 2];
        const int ia = (int)w;
        b.V = V;
        b.ve = -e - (int)(w >> 32);
        // p_k = (md/alpha)^k / k! in units of 2^-60: |p1| <= 2^51, |p3| < 2^31
        const long long p1 = (fix_wide((int)(md >> 16), ia) >> 8) + (fix_wide((int)(md & 0xffff), ia) >> 24);
        const int a1 = fix_hi(p1), a0 = fix_lo(p1);
        const int t1 = (int)(p1 >> 21), tl = (int)p1 & 0x1fffff;  // units of 2^-39 and 2^-60
        const long long p2 = (fix_wide(t1, t1) + (fix_wide(t1, tl) >> 20)) >> 19;
        const int b1 = fix_hi(p2), b0 = fix_lo(p2);
        // t1 p2 2^-39 / 3, by 2/3 in units of 2^-31
        const int p3 = (int)((fix_wide((int)(fix_wide(t1, (int)(p2 >> 11)) >> 29), 1431655765) + (1LL << 30)) >> 31);
        const int p4 = (int)((fix_wide(t1, p3) + (1LL << 40)) >> 41);
        const int p5 = (int)((fix_wide((int)(fix_wide(t1, p4) >> 39), 13107) + (1 << 15)) >> 16);
        long long g[LMAX + kFixBoysK + 2];
#pragma unroll
        for (int m = 0; m <= LMAX + kFixBoysK; m += 2)
            if (m <= L + kFixBoysK) fix_load2(row + m, g[m], g[m + 1]);
#pragma unroll
        for (int n = 0; n <= LMAX; ++n) {
            if (n <= L) {
                const int g1 = fix_hi(g[n + 1]), g2 = fix_hi(g[n + 2]);
                const long long H = fix_wide(g1, a1) + fix_wide(g2, b1);
                const long long M = fix_wide(g1, a0) + fix_wide(fix_lo(g[n + 1]), a1) + fix_wide(g2, b0) +
                                    fix_wide(fix_lo(g[n + 2]), b1) + fix_wide(fix_hi(g[n + 3]), p3) +
                                    fix_wide(fix_hi(g[n + 4]), p4) + fix_wide(fix_hi(g[n + 5]), p5);
                const long long v = g[n] + (H << 4) + (M >> 28);
                F[n] = n & 1 ? -v : v;
            }
        }
        if (L > 0) {
            b.U = fix_mul62(V, row[L + kFixBoysK + 1]);
            b.ue = 3 - e;
        }
    } else {
        // 1/|X| = Y 2^(-61 + z + nx + f - 63)
        const int z = (fix_clz((unsigned long long)S) - 2) >> 1;
        b.V = fix_rsqrt(S << (2 * z));
        const int ye = z + nx + f - 63;
        b.ve = ye + fix_headroom(L);
#pragma unroll
        for (int n = 0; n <= LMAX; ++n)
            if (n <= L) F[n] = n & 1 ? -far[n] : far[n];
        if (L > 0) {
            b.U = fix_mul62(b.V, far[kFixAuxLmax + 1]);
            b.ue = ye + 3;
        }
    }
    if (L > 0) {
        // X u / 2 = (d U 2^-62) 2^(ue - 1 - nx - f), to units of 2^-58
        const int s = nx + f - b.ue - 57;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const long long pr = fix_mul62(d[i], b.U);
            b.x[i] = s >= 0 ? pr >> (s < 63 ? s : 63) : (long long)((unsigned long long)pr << (-s & 63));
        }
    }
}

// One recursion step: the limbs x1 2^29 + x0, x0s = 8 x0, of X u / 2 in units of
// 2^-58 times R, plus (c/4) R2.
FIX_HD long long fix_step(int x1, int x0s, long long R)
{
    const int r1 = fix_hi(R), r0 = fix_lo(R);
    const long long m = fix_wide(x1, r0) + (fix_wide(x0s, r1) + (1LL << 28));
    return (fix_wide(x1, r1) << 3) + (m >> 29);
}
FIX_HD long long fix_step(int x1, int x0s, long long R, int c, long long R2)
{
    return fix_step(x1, x0s, R) + ((R2 * c) >> 2);
}

// The factors V (u/s)^N 2^N that turn order N of the recursion into
// its integral over s^N, s = mu 2^sigma (rmu = 2^62 / mu), in units of 2^(g - 62): phi[N] in units of
// 2^-61, then a right shift sh[N] (fix_finish; below zero for orders well under
// their bound).
template <int LMAX>
FIX_HD void fix_factors(int L, const FixBase& b, int sigma, long long rmu, int g, long long (&phi)[LMAX + 1], int (&sh)[LMAX + 1])
{
    long long m = b.V;  // V 2^(ve - 61) = m 2^-62 2^(ve + 1)
    int ex = b.ve + 1;
    const long long U0 = L > 0 ? fix_mul62(b.U, rmu) : 0;
    const int nu = L > 0 ? fix_clz((unsigned long long)U0) - 2 : 0;
    const long long U = U0 << nu;
    const int du = b.ue - nu - sigma;
#pragma unroll
    for (int N = 0; N <= LMAX; ++N) {
        if (N <= L) {
            if (N > 0) {
                m = fix_mul62(m, U);
                const int up = m < (1LL << 61);  // back to [2^61, 2^62]
                m <<= up;
                ex += du - up;
            }
            phi[N] = m >> 1;
            sh[N] = g - ex - N;
        }
    }
}

// R of the recursion times its factor
FIX_HD long long fix_finish(long long R, long long phi, int sh)
{
    const int a1 = fix_hi(R), a0 = fix_lo(R), b1 = fix_hi(phi), b0 = fix_lo(phi);
    const long long v = (fix_wide(a1, b1) << 4) + ((fix_wide(a1, b0) + fix_wide(a0, b1)) >> 28);
    return sh < 0 ? (long long)((unsigned long long)v << (-sh & 63)) : v >> (sh > 63 ? 63 : sh);
}

// |P - Q|^2 in floats, from the whole coordinates (units of 2^-f): cut to their
// high words, centres at the far end of the range would be off by 2^-7 bohr
FIX_HD float fix_distance2(const FixPrim& p, const FixPrim& q, int f)
{
    const float unit = fix_pow2(-f);
    float r2 = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float d = (float)(p.x[i] - q.x[i]) * unit;
        r2 += d * d;
    }
    return r2;
}

// Exponent g with |order N of the integrals| s^-N < 2^g for N <= L, from the
// exponents and |X|^2: at any distance sqrt(rho) (2 rho)^(N/2) (N-1)!!/(N+1) (the
// value at X = 0), and sqrt(pi)/2 N! / |X|^(N+1) up to a factor below 3.
// At X = 0 that is no estimate but the value itself, so top is raised by
// kFixBoundMargin: rho (a product, a sum and an approximate division of floats) is
// within 2^-21, the root's seed and imu within 2^-22 of theirs, to powers of up to
// 5.5 and 10, with a rounding for each product: less than 2^-17 together.  Next to a
// power of two a bound that fell short would take the limbs (2^62 - 2^30) past their end.
constexpr float kFixBoundMargin = 1.0f + 0x1p-15f;
FIX_HD int fix_bound(int L, float rho, float r2, int sigma, float imu)
{
    const float is = fix_pow2(-sigma) * imu, ir = r2 > 1e-30f ? fix_rsqrt_seed(r2) : 1e15f;
    float near = rho * fix_rsqrt_seed(rho), far = 0.8863f * ir, top = 0.f;
    const float rn = 2.0f * rho * is * is, rf = ir * is;
    float even = near;  // order N at X = 0 (N even), without 1/(N + 1)
    for (int N = 0; N <= L; ++N) {
        if (N > 0) far *= (float)N * rf;
        if (N > 0 && !(N & 1)) even *= (float)(N - 1) * rn;
        // an odd order stays below the larger of its neighbours
        const float nr = (N & 1) ? fmaxf(even / (float)N, even * (float)N * rn / (float)(N + 2)) : even / (float)(N + 1);
        top = fmaxf(top, fminf(nr, 3.0f * far));
    }
    top *= kFixBoundMargin;
    return top > 1e-37f ? (int)(fix_float_bits(top) >> 23) - 126 : -126;
}

// ---- host: tables ----------------------------------------------------------
// Coarse rows F_0..F_kBoysMtab, exp(-T) every 1/32 (build_boys_master) to the
// row j of order L.  Orders above L + 5 come from the nearest coarse row by
// Taylor, the others by the downward recursion.
inline void fix_boys_row(const long double* master, int L, int j, int64_t* out)
{
    const int W = kBoysMtab + 2, M = L + kFixBoysK, per = kFixBoysInvStep / kBoysInvStep;
    const int c = (j + per / 2) / per;
    const long double T = (long double)j / kFixBoysInvStep, d = (long double)(j - c * per) / kFixBoysInvStep;
    const long double* row = master + (size_t)c * W;
    long double F[kFixAuxLmax + kFixBoysK + 1], t = 1.0L, s = 0.0L, ed = 0.0L;
    for (int k = 0; k <= 8; ++k) {
        s += row[M + k] * t;
        ed += t;
        t *= -d / (k + 1);
    }
    const long double eT = row[kBoysMtab + 1] * ed;
    F[M] = s;
    for (int m = M - 1; m >= 0; --m) F[m] = (2.0L * T * F[m + 1] + eT) / (2 * m + 1);
    double la = 1e300;  // log alpha: F_m alpha^m <= F_0
    for (int m = 1; m <= M; ++m) la = std::fmin(la, std::log((double)(F[0] / F[m])) / m);
    const int ia = (int)(2147483648.0 / std::exp(la)) + 2;
    const long double alpha = 2147483648.0L / ia;
    int h = 0;
    while (F[0] * (1LL << (h + 1)) <= 1.0L) ++h;
    h -= fix_headroom(L);
    long double am = ldexpl(1.0L, 61 + h);
    for (int m = 0; m <= M; ++m) {
        out[m] = (int64_t)llroundl(F[m] * am);
        am *= alpha;
    }
    out[M + 1] = (int64_t)llroundl(sqrtl(2.0L / alpha) * 0x1p60L);
    out[M + 2] = (int64_t)(((uint64_t)(uint32_t)h << 32) | (uint32_t)ia);
}

inline void fix_far_constants(int L, int64_t* out)
{
    // kappa^2 >= ((2n-1)!!)^(1/n) for the orders of a row, as alpha_j at large T
    long double df = 1.0L, k2 = 1.0L;
    for (int n = 1; n <= L + kFixBoysK; ++n) {
        df *= 2 * n - 1;
        k2 = fmaxl(k2, powl(df, 1.0L / n));
    }
    long double t = 0.886226925452758013649083741670572591L;  // sqrt(pi)/2
    for (int n = 0; n <= kFixAuxLmax; ++n) {
        out[n] = n <= L ? (int64_t)llroundl(ldexpl(t, 61 - fix_headroom(L))) : 0;
        t *= (2 * n + 1) / k2;
    }
    out[kFixAuxLmax + 1] = (int64_t)llroundl(sqrtl(k2) * 0x1p60L);
}

// A primitive pair's scalars: exponent zeta, centre P (host and device).
FIX_HD void fix_split_exponent(double v, long long* m, int* e)
{
    // v > 0 normal: v = m 2^(e - 62), m in [2^61, 2^62)
    long long bits;
    std::memcpy(&bits, &v, 8);
    *m = ((bits & 0xfffffffffffffLL) | 0x10000000000000LL) << 9;
    *e = (int)((bits >> 52) & 0x7ff) - 1022;
}
FIX_HD long long fix_coordinate(double x, int f)
{
    // x 2^f, |x 2^f| < 2^61
    long long m;
    int e;
    if (x == 0.0) return 0;
    fix_split_exponent(x < 0 ? -x : x, &m, &e);
    const int s = 62 - e - f;  // m 2^(e - 62 + f)
    const long long v = s <= 0 ? m << -s : (s > 62 ? 0 : ((m >> (s - 1)) + 1) >> 1);
    return x < 0 ? -v : v;
}

}  // namespace eri
