// eri_fixed.cuh -- the forward tile with fixed-point transforms.
//
// What bounds the FP64 tile is the FP64 pipe: 1.9 lanes per clock and SM,
// against 30 for the 32 x 32 + 64 bit integer multiply-add (IMAD.WIDE), both
// measured on GB300.  The ket and bra transforms are sums of products whose
// magnitudes are known beforehand, so they run here on 64-bit fixed-point
// numbers, three multiply-adds per product; so do the auxiliary integrals (eri_fixaux.cuh).
// The E products and the epilogue stay FP64.
// What bounds it: no pipe.  (pp|ps) and (dp|pp), K = 3: issue slots 37 and 40 % busy,
// the IMAD pipe 39 and 43 %, with the four warps a scheduler that 128 registers
// leave; of 10 cycles an instruction 3 to 3.6 are barriers between the stages, 2 the
// latency of dependent integer operations.  1e5 quartets of (pp|ps): FP64 tile 3.5 ms,
// this one 2.26; 6.5e4 of (dp|pp): 10.7 and 8.1.
//
// Scales (all powers of two, so scaling rounds nothing):
//  * Hermite orders carry a length: for bra primitive i a unit s = mu 2^sigma
//    with s >= 1.1 sqrt(2 rho), rho the largest reduced exponent i meets or, at a
//    distance r of the two pairs, kFixFarT / r^2 if that is less, and mu
//    in [1, 2) fixed for the batch (exact for its largest rho; the E products
//    come with mu^|q|); R of order N is taken times s^(-N), E of order |q|
//    times 2^(sigma |q|).  sigma_i (bra alone, rho -> zeta_i) bounds it from above.
//    At a distance order N falls as N! / r^N, so that in units of sqrt(2 rho) high
//    orders, which are the whole integral of one-centre pairs such as p_x p_y, would
//    keep few of the bits that all orders share; in units of about 3 / r they stay level.
//  * R of one (quartet, bra primitive) is relative to 2^g, a bound of its
//    entries over the ket primitives (fix_bound); |R| <= 2^62 units.
//  * each column (component pair) of E is relative to the 1-norm of its
//    terms over all ket primitives (2^h), so no sum of products overflows:
//    |sum E R| <= 2^60 2^62.  Likewise the bra's E, over all its primitives.
//  * X (the ket-transformed integrals) is aligned to the quartet's largest g and
//    h before the bra transform, whose sums over bra primitives then add without
//    further scaling.
//  * the bra's limbs are formed once a pair, with sigma_i; X of order n is then
//    shifted by n (sigma_i - sigma) to meet them.  A column without low orders
//    (p_x p_y of one centre has order 2 alone) would lose those bits: a
//    quartet in which a column may lose more than kFixWeakBits forms its limbs
//    from the E products at its own sigmas, relative to a bound F of the 1-norm
//    there, and leaves X as it is.
// A number is held as two signed limbs, hi 2^31 + lo (R), hi 2^32 + lo (X) or
// hi 2^29 + lo (E); a product keeps hi hi, hi lo and lo hi, and the dropped lo lo is below
// 2^-64 of the bound.
//
// Precision: FP64 transforms round every product and sum at 2^-53 of its own
// size; here every operand is rounded at 2^-60 or 2^-61 of the largest the
// sum may hold.  The difference between the two is how far the bound lies above
// the sum, which grows with the spread of exponents inside a pair,
// (largest / smallest zeta)^((l1 + l2) / 2), and with the order.  So does the FP64
// tile's error with the distance inside a pair, which its recursion forms
// magnify.  fixed_eligible (eri_fwd.cu) admits what measured no larger a relative
// 2-norm error over a batch than the FP64 tile in the form that would have run:
// order 6 and 5 bits of spread anywhere, order 8 and 6 bits where some pair's
// centres lie kFixWide apart.  These are errors of blocks: an entry far below the
// others of its column, over short distances, keeps fewer digits than FP64.
#pragma once

#include <climits>
#include <type_traits>
#include <utility>

#include "eri_fixaux.cuh"
#include "eri_tile.cuh"

namespace eri {

// log2 of the largest spread factor of a pair, and the largest order, for the
// fixed-point tile: anywhere, and where a pair's centres lie kFixWide bohr apart.
// Relative 2-norm error against the long double oracle, fixed point over FP64 in the
// form that either would run, pairs of two centres (and half of one centre):
//  cube of, bohr              1.5          4            8     12
//  2.4 bits, (dp|dp), K = 2   0.8 (0.9)    0.7 (1.0)    0.9   1.0 (1.0)
//  4.8 bits, (dp|dp), K = 3   1.1 (1.6)    0.7 (1.1)    0.5   1.0 (1.0)
//  5.9 bits, (pp|pp), K = 2   2.7 (2.2)    0.9 (1.0)    1.0   1.3 (1.0)
//            (dp|dp), K = 2   4.5 (6.0)    1.4 (2.1)    1.1   1.1 (1.2)
//  order 7,  (dd|dp), K = 3   3.4 (4.1)    1.2 (1.6)    0.4   0.4 (1.0)
//            (fd|pp), K = 2   2.6 (2.0)    1.2 (1.2)    0.6   0.8 (1.0)
//  order 8,  (dd|dd), K = 3   3.7 (3.4)    1.5 (2.0)    1.1   0.4 (0.6)
//            (ff|pp), K = 2   3.7 (2.9)    1.3 (1.2)    0.4   0.4 (0.7)
//  order 9,  (fd|dd), K = 2                9.4          4.8   2.2 (2.1)
//  order 10, (fd|fd), K = 2                13           8.7   7.6 (6.8)
// (order 5 and less, 4.8 bits and less, both tiles in the plain form: 0.4 to 1.02)
constexpr float kFixSpreadBits = 5.0f, kFixSpreadBitsWide = 6.0f;
constexpr int kFixLmaxNear = 6, kFixLmax = 8;
constexpr float kFixWide = 8.0f;
static_assert(kFixLmax <= kFixAuxLmax, "order of the fixed-point auxiliary integrals");
// products per low-limb accumulator between folds: each below 2^28 2^31.  Even:
// the ket transform reads its operands in aligned pairs from each multiple on.
constexpr int kFixFold = 14;
static_assert(kFixFold % 2 == 0, "pairs of ket primitives stay 16-byte aligned");

// T = rho r^2 from which the Hermite unit follows the distance: s r >= 1.1 sqrt(8) = 3.1,
// at most twice that, keeps N! / (s r)^N between 2^-7 and 2^3 for N <= 8
constexpr float kFixFarT = 4.0f;
// bits a bra column may lose to the shift of X before its quartet forms the limbs
// itself (shifted throughout, components of (dp|ps) with one-centre bra pairs came out
// 1.9e-11 of themselves off with bra exponents 2e3 times the ket's, 5.4e-9 with 1e5
// times; FP64 4e-16)
constexpr int kFixWeakBits = 4;

template <int N>
using IntC = std::integral_constant<int, N>;

// order t + u + v of Hermite index e (tetrahedral numbering)
__host__ __device__ __forceinline__ int herm_order(int e)
{
    int n = 0;
    while ((n + 1) * (n + 2) * (n + 3) / 6 <= e) ++n;
    return n;
}

// x 2^sh rounded to the nearest integer; |x 2^sh| < 2^62, zero and denormals give 0
__device__ __forceinline__ long long fix_from(double x, int sh)
{
    const int hi = __double2hiint(x);
    const int e = (hi >> 20) & 0x7ff;
    unsigned long long m = ((((unsigned long long)((hi & 0xfffff) | 0x100000)) << 32) |
                            (unsigned)__double2loint(x)) << 10;  // |x| = m 2^(e - 1085)
    const int r = 1085 - e - sh;  // >= 1
    m = ((m >> (max(1, min(r, 64)) - 1)) + 1) >> 1;
    if (r > 63 || e == 0) m = 0;
    return hi < 0 ? -(long long)m : (long long)m;
}

template <int BITS>
__device__ __forceinline__ int2 fix_limbs(long long v)
{
    if (BITS == 32) return make_int2(fix_lo(v), fix_hi(v));
    const int h = (int)((v + (1LL << (BITS - 1))) >> BITS);
    return make_int2((int)v - (int)((unsigned)h << (BITS & 31)), h);
}
constexpr int kLimbR = 31, kLimbE = 29, kLimbX = 32;

// Sums of products of E limbs (29 bits) with R limbs (31 bits) in the ket
// transform, X limbs (32 bits) in the bra transform: a low limb of BITS bits
// gives the weights 2^(29 + BITS), 2^29 and 2^BITS.
struct FixAcc {
    long long h, a, b;
    __device__ __forceinline__ FixAcc() : h(0), a(0), b(0) {}
};
__device__ __forceinline__ void fix_mac(FixAcc& s, int e0, int e1, int r0, int r1)
{
    s.h += (long long)e1 * r1;
    s.a += (long long)e1 * r0;
    s.b += (long long)e0 * r1;
}
// fold the accumulator whose terms are not bounded by the 1-norm
__device__ __forceinline__ void fix_fold(FixAcc& s)
{
    s.h += s.b >> 29;
    s.b &= (1LL << 29) - 1;
}
// ket transform: 2^122 of product units is the bound; in units of 2^59 (63 bits)
__device__ __forceinline__ long long fix_ket_sum(const FixAcc& s)
{
    return (s.h << 1) + ((s.a + (1LL << 29)) >> 30) + ((s.b + (1LL << 27)) >> 28);
}
// bra transform: the bound is 2^123; in units of 2^61 (62 bits)
__device__ __forceinline__ long long fix_bra_sum(const FixAcc& s)
{
    return s.h + ((s.a + (1LL << 31)) >> 32) + ((s.b + (1LL << 28)) >> 29);
}

// ---- pair tables -----------------------------------------------------------
// One thread per (pair, component pair) over its terms and primitives: the
// column's 1-norms per Hermite order go to norm[8], relative to 2^ex.  Ket role:
// of the products themselves, which each quartet scales by its own sigma.  Bra
// role: of the products times 2^(sigma_i |p|); their limbs, relative to the whole
// 1-norm (2^ex again); and the bits by which its order 0 lies below that, the
// largest of a pair to weak.
struct FixPairArgs {
    const double* E;      // ket role [npairs][T][KS], bra role [npairs][KS][T]
    int2* limbs;          // [npairs][KS][T] (bra role)
    int* weak;            // [npairs], zeros (bra role)
    const FixPrim* ps;    // [npairs][KS]
    const int32_t* kp;    // [npairs]
    const int* start;     // [ncol + 1] terms of a column
    const int16_t* herm;  // [T] Hermite index of a term
    int64_t npairs;
    int KS, T, ncol, ket;
    float c;              // 2.42 / mu^2 (fix_sigma)
    int* ex;              // [npairs][ncol]
    float* norm;          // [npairs][ncol][8]
    float* box;           // [npairs][6] smallest, largest coordinates of the primitive pairs' centres
    int f;                // their units 2^-f
};

__device__ __forceinline__ int fix_norm_exp(const float* n, int base, int sigma)
{
    float s = 0.f;
    for (int o = 0; o < 7; ++o) s = __fadd_ru(s, n[o] * __int_as_float(min(254, max(1, 127 + sigma * o)) << 23));
    return s > 0.f ? base + (__float_as_int(s) >> 23) - 126 : base;
}

static __global__ void __launch_bounds__(128) fix_pairs_kernel(FixPairArgs a)
{
    const int64_t total = a.npairs * a.ncol;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = g / a.ncol;
        const int c = (int)(g - j * a.ncol), K = a.kp[j];
        const double* E = a.E + (size_t)j * a.T * a.KS;
        const FixPrim* ps = a.ps + (size_t)j * a.KS;
        if (c == 0)
            for (int x = 0; x < 3; ++x) {
                long long lo = ps[0].x[x], hi = lo;
                for (int k = 1; k < K; ++k) {
                    lo = min(lo, ps[k].x[x]);
                    hi = max(hi, ps[k].x[x]);
                }
                a.box[6 * j + x] = (float)lo * fix_pow2(-a.f);
                a.box[6 * j + 3 + x] = (float)hi * fix_pow2(-a.f);
            }
        const int t0 = a.start[c], t1 = a.start[c + 1], ts = a.ket ? a.KS : 1, ks = a.ket ? 1 : a.T;
        int top = 0;
        for (int t = t0; t < t1; ++t)
            for (int k = 0; k < K; ++k) top = max(top, __double2hiint(E[t * ts + k * ks]) & 0x7fffffff);
        // magnitudes relative to 2^base, rounded up to floats (below 2^-120: nothing)
        const int base = (top >> 20) - 1023;
        float n[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        float sum = 0.f;
        for (int t = t0; t < t1; ++t) {
            const int o = herm_order(a.herm[t]);
            for (int k = 0; k < K; ++k) {
                const int hi = __double2hiint(E[t * ts + k * ks]) & 0x7fffffff;
                const int e = (hi >> 20) - 1023 - base;
                float v = e > -120 ? __int_as_float((((e + 127) << 23) | ((hi & 0xfffff) << 3)) + 8) : 0.f;
                if (!a.ket) {
                    v *= __int_as_float((127 + fix_sigma(ps[k].zeta, a.c) * o) << 23);
                    sum = __fadd_ru(sum, v);
                }
#pragma unroll
                for (int i = 0; i < 7; ++i)
                    if (i == o) n[i] = __fadd_ru(n[i], v);
            }
        }
        // (bra: in units of the 1-norm, a power of two)
        const int up = a.ket ? 0 : (__float_as_int(sum) >> 23) - 126;
        for (int i = 0; i < 8; ++i) a.norm[8 * g + i] = a.ket ? n[i] : ldexpf(n[i], -up);
        a.ex[g] = top ? base + up : -1000;
        if (!a.ket) {
            const int f = top ? base + up : -1000;
            if (top) atomicMax(&a.weak[j], n[0] > 0.f ? (__float_as_int(sum) >> 23) - (__float_as_int(n[0]) >> 23) : 1000);
            for (int t = t0; t < t1; ++t) {
                const int o = herm_order(a.herm[t]);
                for (int k = 0; k < K; ++k) {
                    const int sg = fix_sigma(ps[k].zeta, a.c) * o;
                    a.limbs[((size_t)j * a.KS + k) * a.T + t] = fix_limbs<kLimbE>(fix_from(E[t + k * ks], 60 + sg - f));
                }
            }
        }
    }
}

// ---- tile ------------------------------------------------------------------

// Stage B: rows u0..u1-1 of the E products of C columns (E[c], KS apart)
// against P bra Hermite functions.  One read of R feeds C columns, one read of
// E (the same for most lanes) feeds P functions: shared memory would
// otherwise bound the stage (its 128 B per clock and SM against 3.2 clocks of
// multiply-adds per product and warp).
// KT > 0: the tile's ket primitives, a constant (the usual contraction degrees).
template <int P, int C, int KT>
__device__ __forceinline__ void fix_ket_rows(FixAcc (&s)[P][2], const int2* const (&E)[C], const int2* Rc,
                                             const uint16_t* const (&row)[P], const int16_t* s_q, int u0, int u1,
                                             int KKt, int KS, int per_fold, int& left)
{
    auto pair = [&](const int2* const (&Eu)[C], const int2* const (&R)[P], int k) {
        int4 e[C];
#pragma unroll
        for (int c = 0; c < C; ++c) e[c] = *reinterpret_cast<const int4*>(Eu[c] + k);
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const int4 r = *reinterpret_cast<const int4*>(R[j] + k);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                fix_mac(s[j][c], e[c].x, e[c].y, r.x, r.y);
                fix_mac(s[j][c], e[c].z, e[c].w, r.z, r.w);
            }
        }
    };
    auto one = [&](const int2* const (&Eu)[C], const int2* const (&R)[P], int k) {
        int2 e[C];
#pragma unroll
        for (int c = 0; c < C; ++c) e[c] = Eu[c][k];
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const int2 r = R[j][k];
#pragma unroll
            for (int c = 0; c < C; ++c) fix_mac(s[j][c], e[c].x, e[c].y, r.x, r.y);
        }
    };
    auto fold = [&]() {
        if (--left == 0) {
            left = per_fold;
#pragma unroll
            for (int j = 0; j < P; ++j)
#pragma unroll
                for (int c = 0; c < C; ++c) fix_fold(s[j][c]);
        }
    };
    for (int u = u0; u < u1; ++u) {
        const int q = s_q[u];
        const int2 *R[P], *Eu[C];
#pragma unroll
        for (int j = 0; j < P; ++j) R[j] = Rc + row[j][q];
#pragma unroll
        for (int c = 0; c < C; ++c) Eu[c] = E[c] + u * KS;
        if constexpr (KT > 0) {
#pragma unroll
            for (int k = 0; k + 1 < KT; k += 2) pair(Eu, R, k);
            if (KT & 1) one(Eu, R, KT - 1);
            fold();
        } else {
            for (int k0 = 0; k0 < KKt; k0 += kFixFold) {
                const int ke = min(KKt, k0 + kFixFold);
                int k = k0;
                for (; k + 1 < ke; k += 2) pair(Eu, R, k);
                if (k < ke) one(Eu, R, k);
                fold();
            }
        }
    }
}

// One step of the auxiliary recursion (Eq. r-rr): byte offsets of its sources
// in R, axis and coefficient.
struct alignas(16) FixStep {
    int o1, o2, axis, c;
};

// The item's auxiliary integrals from its base, through R (one column, rows NIs
// entries apart): levels as in r_recursion, then every order times its factor,
// as limbs.  G consecutive lanes of a warp (a power of two, the same for every
// item of the warp) share the item, lane j of them: G entries of a level at a
// time, all sources read before any is written (a lane alone takes four).
// on: false for lanes without an item, which only keep the warp's barriers.
__device__ __forceinline__ void fix_recursion(int L, const long long* F, const int (&x1)[3], const int (&x0s)[3],
                                              const long long* phi, const int* sh, const FixStep* st,
                                              const int16_t* ord, long long* R, int NIs, int G, int j, bool on)
{
    const char* Rb = reinterpret_cast<const char*>(R);
    auto step = [&](const FixStep& s) {
        const int a = s.axis == 0 ? x1[0] : (s.axis == 1 ? x1[1] : x1[2]);
        const int b = s.axis == 0 ? x0s[0] : (s.axis == 1 ? x0s[1] : x0s[2]);
        long long v = fix_step(a, b, *reinterpret_cast<const long long*>(Rb + s.o1));
        if (s.c) v += (*reinterpret_cast<const long long*>(Rb + s.o2) * s.c) >> 2;
        return v;
    };
    if (G > 1) {
        if (on && j == 0) R[0] = F[L];
        __syncwarp();
        for (int n = L - 1; n >= 0; --n) {
            const int N = L - n;
            int e = (N + 1) * (N + 2) * (N + 3) / 6 - 1 - j;
            long long* Re = R + e * NIs;
            for (int left = e + j; left >= 1; left -= G, e -= G, Re -= G * NIs) {
                long long v = 0;
                const bool act = on && e >= 1;
                if (act) v = step(st[e]);
                __syncwarp();
                if (act) *Re = v;
                __syncwarp();
            }
            if (on && j == 0) R[0] = F[n];
            __syncwarp();
        }
        const int nhl = (L + 1) * (L + 2) * (L + 3) / 6;
        if (on)
            for (int e = j; e < nhl; e += G) {
                const int N = ord[e];
                *reinterpret_cast<int2*>(&R[e * NIs]) = fix_limbs<kLimbR>(fix_finish(R[e * NIs], phi[N], sh[N]));
            }
        return;
    }
    if (!on) return;
    R[0] = F[L];
    for (int n = L - 1; n >= 0; --n) {
        const int N = L - n;
        int e = (N + 1) * (N + 2) * (N + 3) / 6 - 1;
        long long* Re = R + e * NIs;
        for (; e >= 4; e -= 4, Re -= 4 * NIs) {
            FixStep s[4];
            long long v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] = st[e - i];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = step(s[i]);
#pragma unroll
            for (int i = 0; i < 4; ++i) Re[-i * NIs] = v[i];
        }
        for (; e >= 1; --e, Re -= NIs) *Re = step(st[e]);
        R[0] = F[n];
    }
    int e = 0;
    long long* Re = R;
    for (int N = 0; N <= L; ++N) {
        const long long f = phi[N];
        const int s = sh[N];
        for (const int top = (N + 1) * (N + 2) * (N + 3) / 6; e < top; ++e, Re += NIs)
            *reinterpret_cast<int2*>(Re) = fix_limbs<kLimbR>(fix_finish(*Re, f, s));
    }
}

// f(IntC<0>()), ..., f(IntC<N - 1>()): loops whose index is a constant expression
template <typename F, int... I>
__device__ __forceinline__ void static_for(std::integer_sequence<int, I...>, F f)
{
    (f(IntC<I>()), ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F f)
{
    static_for(std::make_integer_sequence<int, N>(), f);
}

// A step of the recursion (the axis rule of build_rstep_table)
struct StepC {
    int order, axis, c, s1, s2;
};
__host__ __device__ constexpr StepC step_c(int e)
{
    int h[3] = {0, 0, 0};
    herm_tuv_c(e, h[0], h[1], h[2]);
    StepC s{h[0] + h[1] + h[2], h[0] == 1 ? 0 : (h[1] == 1 ? 1 : (h[2] == 1 ? 2 : -1)), 0, 0, 0};
    if (s.axis < 0) {
        int best = 1 << 20;
        for (int i = 0; i < 3; ++i)
            if (h[i] > 0 && h[i] < best) {
                best = h[i];
                s.axis = i;
            }
    }
    if (s.axis < 0) return s;  // e = 0
    s.c = h[s.axis] - 1;
    h[s.axis] -= 1;
    s.s1 = herm_idx_c(h[0], h[1], h[2]);
    if (s.c > 0) {
        h[s.axis] -= 1;
        s.s2 = herm_idx_c(h[0], h[1], h[2]);
    }
    return s;
}

// The same with L known, in registers.
template <int L>
__device__ __forceinline__ void fix_recursion_c(const long long (&F)[L + 1], const int (&x1)[3], const int (&x0s)[3],
                                                const long long (&phi)[L + 1], const int (&sh)[L + 1], long long* R,
                                                int NIs)
{
    long long r[host_nh(L)];
    r[0] = F[L];
    static_for<L>([&](auto level) {
        constexpr int N = decltype(level)::value + 1;
        static_for<host_nh(N) - 1>([&](auto i) {
            constexpr int e = host_nh(N) - 1 - decltype(i)::value;
            constexpr StepC s = step_c(e);
            if constexpr (s.c > 0)
                r[e] = fix_step(x1[s.axis], x0s[s.axis], r[s.s1], s.c, r[s.s2]);
            else
                r[e] = fix_step(x1[s.axis], x0s[s.axis], r[s.s1]);
        });
        r[0] = F[L - N];
    });
    static_for<host_nh(L)>([&](auto i) {
        constexpr int e = decltype(i)::value, N = step_c(e).order;
        *reinterpret_cast<int2*>(&R[e * NIs]) = fix_limbs<kLimbR>(fix_finish(r[e], phi[N], sh[N]));
    });
}

// Stage A of one primitive quartet into its column of R, relative to 2^g (L > 0).
template <int LMAX, int FIXED>
__device__ __forceinline__ void fix_aux_item(int Lr, const FixPrim& p, const FixPrim& q, int f,
                                             const long long* __restrict__ tab, const long long* __restrict__ far,
                                             int sigma, long long rmu, int g, const FixStep* st, const int16_t* ord,
                                             long long* R, int NIs, int G, int j, bool on)
{
    const int L = FIXED ? LMAX : Lr;
    long long F[LMAX + 1], phi[LMAX + 1];
    int sh[LMAX + 1];
    FixBase b;
    fix_base<LMAX>(L, p, q, f, tab, far, F, b);
    fix_factors<LMAX>(L, b, sigma, rmu, g, phi, sh);
    int x1[3], x0s[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        x1[i] = (int)((b.x[i] + (1LL << 28)) >> 29);
        x0s[i] = (int)((unsigned)(int)(b.x[i] - ((long long)x1[i] << 29)) << 3);
    }
    if constexpr (FIXED)
        fix_recursion_c<LMAX>(F, x1, x0s, phi, sh, R, NIs);
    else
        fix_recursion(L, F, x1, x0s, phi, sh, st, ord, R, NIs, G, j, on);
}

// Shared-memory tables of a class and tile shape (stage_fixed_tables).
struct FixTables {
    const int *bstart, *kstart;
    const uint16_t* bp;   // [Tab] offset into X of a bra term's row
    const int16_t* kq;    // [Tcd]
    const uint16_t* pq;   // [nhb][nhk] offset into R of p+q
    const int16_t* tc;    // [Tcd] 8 column + order of a ket term
    const int16_t* bc;    // [Tab] and of a bra term
    const int16_t* ord;   // [nhl] order of a Hermite function
    const int16_t *kpair, *bpair; // [nkpair][2], [nbpair][2]
    const FixStep* st;    // [nhl]
    __device__ __forceinline__ FixTables(const ClassTables& ct, double* tab)
    {
        st = reinterpret_cast<const FixStep*>(tab);
        bstart = reinterpret_cast<const int*>(st + ct.nhl);
        kstart = bstart + ct.nab + 1;
        bp = reinterpret_cast<const uint16_t*>(kstart + ct.ncd + 1);
        kq = reinterpret_cast<const int16_t*>(bp + ct.Tab);
        pq = reinterpret_cast<const uint16_t*>(kq + ct.Tcd);
        tc = reinterpret_cast<const int16_t*>(pq + ct.nhb * ct.nhk);
        bc = tc + ct.Tcd;
        ord = bc + ct.Tab;
        kpair = ord + ct.nhl;
        bpair = kpair + 2 * ct.nkpair;
    }
};
inline size_t fix_table_bytes(const ClassTables& ct)
{
    return sizeof(FixStep) * (size_t)ct.nhl + 4 * (ct.nab + ct.ncd + 2) +
           2 * (2 * ct.Tab + 2 * ct.Tcd + ct.nhb * ct.nhk + ct.nhl + 2 * ct.nkpair + 2 * ct.nbpair);
}

// The tile's scratch: ints, per (quartet, bra primitive) sigma and the bound g;
// per bra primitive whether any quartet's ket E change there; per quartet G, the
// largest exponent of the bounds, and the largest rho for its distance (a float);
// per (quartet, ket column) the exponent H (largest sigma) and its distance to the
// current sigma's.  Then 16-bit words (two tiles of some shapes only just share an
// SM), per (quartet, bra primitive) sigma_i - sigma, and flags: bit 0 the ket's E
// change there, bit 1 the quartet forms its bra limbs itself; per (quartet, bra
// column) the exponent F.
__host__ __device__ __forceinline__ int fix_scratch_ints(int TQ, int KB, int nab, int ncd)
{
    return 2 * TQ * KB + KB + 2 * TQ + 2 * TQ * ncd + (2 * TQ * KB + TQ * nab + 1) / 2;
}

constexpr int kFixRegL = 4;  // auxiliary integrals in registers up to this order

template <int NT>
__device__ void tile_fixed(const FwdArgs& a, int64_t q0, int nqt, double* sm, double* s_red)
{
    const ClassTables& ct = a.ct;
    const int tid = threadIdx.x, lane = tid & 31;
    const int TQ = a.TQ, KB = a.KB, KK = a.KK;
    const int nhb = ct.nhb, nhk = ct.nhk, ncd = ct.ncd, nab = ct.nab;
    const int KS = (KK + 1) & ~1;                 // ket primitives per row, 16-byte pairs
    const int QS = r_row_stride(a.IC * KS, 1);    // R columns of a quartet
    const int NIs = r_row_stride(TQ * QS, 1);     // R row stride
    const int XS = nhb * ncd * TQ;                // X of one bra primitive
    const FixTables tb(ct, sm + a.o_tab);
    int* s_q = reinterpret_cast<int*>(sm + a.o_q);
    int64_t* s_qq = reinterpret_cast<int64_t*>(sm + a.o_dj);
    int* s_sig = reinterpret_cast<int*>(sm + a.o_fx);
    int* s_g = s_sig + TQ * KB;
    int* s_any = s_g + TQ * KB;
    int* s_G = s_any + KB;
    float* s_lim = reinterpret_cast<float*>(s_G + TQ);
    int* s_dh = s_G + 2 * TQ;
    int* s_H = s_dh + TQ * ncd;
    int16_t* s_ds = reinterpret_cast<int16_t*>(s_H + TQ * ncd);
    int16_t* s_ch = s_ds + TQ * KB;
    int16_t* s_F = s_ch + TQ * KB;
    const int lgTQ = 31 - __clz(TQ);  // TQ is a power of two
    const FastDiv d_ncd(ncd), d_kb(KB);
    __shared__ int s_kmax[2], s_next;
    int2* sEb = reinterpret_cast<int2*>(sm + a.o_Eb);
    int2* sEk = reinterpret_cast<int2*>(sm + a.o_Ek);
    FixPrim* sPb = reinterpret_cast<FixPrim*>(sm + a.o_Pb);
    FixPrim* sPk = reinterpret_cast<FixPrim*>(sm + a.o_Pk);
    long long* sR = reinterpret_cast<long long*>(sm + a.o_R);
    int2* sX = reinterpret_cast<int2*>(sm + a.o_X);
    long long* sA = reinterpret_cast<long long*>(sm + a.o_acc);
    if (tid == 0) s_kmax[0] = s_kmax[1] = 0;
    __syncthreads();
    {
        int mkb = 0, mkk = 0;
        for (int q = tid; q < TQ; q += NT) {
            int b = 0, k = 0, kb = 0, kk = 0, weak = 0;
            const int64_t qq = q < nqt && a.order ? a.order[q0 + q] : q0 + q;
            if (q < nqt) {
                quartet_pairs(a, qq, &b, &k);
                kb = a.bra_kp[b];
                kk = a.ket_kp[k];
                weak = a.bra_weak[b] > kFixWeakBits;
            }
            // the distance of the pairs' boxes
            float r2 = 0.f;
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                const float *B = a.bra_box + 6 * (int64_t)b + x, *K = a.ket_box + 6 * (int64_t)k + x;
                const float d = fmaxf(0.f, fmaxf(B[0] - K[3], K[0] - B[3]));
                r2 = fmaf(d, d, r2);
            }
            s_lim[q] = __fdividef(kFixFarT, r2);
            s_ch[q * KB] = weak;
            s_q[4 * q] = b;
            s_q[4 * q + 1] = k;
            s_q[4 * q + 2] = kb;
            s_q[4 * q + 3] = kk;
            if (a.order) s_qq[q] = qq;
            mkb = max(mkb, kb);
            mkk = max(mkk, kk);
        }
        mkb = __reduce_max_sync(0xffffffffu, mkb);
        mkk = __reduce_max_sync(0xffffffffu, mkk);
        if (lane == 0 && mkb > 0) {
            atomicMax(&s_kmax[0], mkb);
            atomicMax(&s_kmax[1], mkk);
        }
    }
    __syncthreads();
    const int KBt = s_kmax[0], KKt = s_kmax[1];
    const FastDiv d_kkt(KKt);
    {
        // (slots past a pair's own count keep what the pair kernel put there)
        constexpr int W = sizeof(FixPrim) / 8;
        long long *pb = reinterpret_cast<long long*>(sPb), *pk = reinterpret_cast<long long*>(sPk);
        const FastDiv d_b(KB * W), d_k(KK * W);
        for (int idx = tid; idx < TQ * KB * W; idx += NT) {
            const int q = d_b.div(idx), r = idx - q * KB * W;
            pb[idx] = reinterpret_cast<const long long*>(a.bra_ps)[(size_t)s_q[4 * q] * KB * W + r];
        }
        for (int idx = tid; idx < TQ * KK * W; idx += NT) {
            const int q = d_k.div(idx), r = idx - q * KK * W;
            pk[idx] = reinterpret_cast<const long long*>(a.ket_ps)[(size_t)s_q[4 * q + 1] * KK * W + r];
        }
    }
    const int nC = TQ * nab * ncd;
    for (int idx = tid; idx < nC; idx += NT) sA[idx] = 0;
    __syncthreads();
    // sigma of (quartet, bra primitive i): the pairs' slots are sorted by
    // exponent, descending, so ket slot 0 gives the largest reduced exponent, and
    // sigma never grows with i
    auto sigma_of = [&](int q, int i) {
        const float zb = sPb[q * KB + i].zeta, zk = sPk[q * KK].zeta;
        return min(fix_sigma(zb, a.fx_c), fix_sigma(fminf(fix_reduced(zb, zk), s_lim[q]), a.fx_c));
    };
    auto norm_exp = [&](int q, int cd, int sigma) {
        const int64_t g = (int64_t)s_q[4 * q + 1] * ncd + cd;
        return fix_norm_exp(a.ket_norm + 8 * g, a.ket_ex[g], sigma);
    };
    for (int idx = tid; idx < TQ * KB; idx += NT) {
        const int q = d_kb.div(idx), i = idx - q * KB;
        const bool on = i < s_q[4 * q + 2];
        const int sg = on ? sigma_of(q, i) : INT_MIN;
        s_sig[idx] = sg;
        s_ds[idx] = on ? fix_sigma(sPb[idx].zeta, a.fx_c) - sg : 0;
        s_g[idx] = -1000;
    }
    __syncthreads();
    for (int idx = tid; idx < TQ * ncd; idx += NT) {
        const int q = d_ncd.div(idx);
        s_H[idx] = q < nqt ? norm_exp(q, idx - q * ncd, s_sig[q * KB]) : 0;
    }
    // whether quartet q forms its bra limbs itself; lo: the smallest sigma_i - sigma
    auto own_limbs = [&](int q, int* lo) {
        int hi = 0;
        *lo = 1000;
        if (!s_ch[q * KB]) return false;  // (so far: whether the pair has a weak column)
        for (int i = 0; i < s_q[4 * q + 2]; ++i) {
            hi = max(hi, s_ds[q * KB + i]);
            *lo = min(*lo, s_ds[q * KB + i]);
        }
        return hi * (ct.la + ct.lb) > kFixWeakBits;
    };
    for (int idx = tid; idx < TQ * nab; idx += NT) {
        const int q = idx & (TQ - 1), ab = idx >> lgTQ;
        int lo;
        if (!own_limbs(q, &lo)) continue;
        const int64_t g = (int64_t)s_q[4 * q] * nab + ab;
        s_F[idx] = fix_norm_exp(a.bra_norm + 8 * g, a.bra_ex[g], -lo);
    }
    // bounds of the auxiliary integrals
    {
        const FastDiv d_bk(KBt * KKt);
        for (int idx = tid; idx < TQ * KBt * KKt; idx += NT) {
            const int q = d_bk.div(idx), r = idx - q * KBt * KKt, i = d_kkt.div(r), k = r - i * KKt;
            if (i >= s_q[4 * q + 2] || k >= s_q[4 * q + 3]) continue;
            const FixPrim &p = sPb[q * KB + i], &c = sPk[q * KK + k];
            const float r2 = fix_distance2(p, c, a.fx_f), rho = __fdividef(p.zeta * c.zeta, p.zeta + c.zeta);
            atomicMax(&s_g[q * KB + i], fix_bound(ct.L, rho, r2, s_sig[q * KB + i], a.fx_imu));
        }
    }
    __syncthreads();
    for (int i = tid; i < KB; i += NT) s_any[i] = 0;
    __syncthreads();
    for (int q = tid; q < TQ; q += NT) {
        int G = -1000, cur = INT_MIN, lo;
        const bool own = own_limbs(q, &lo);
        for (int i = 0; i < s_q[4 * q + 2]; ++i) {
            G = max(G, s_g[q * KB + i]);
            if (own) s_ds[q * KB + i] = 0;
        }
        for (int i = 0; i < KB; ++i) {
            const int sg = s_sig[q * KB + i];
            int ch = 0;
            if (sg != INT_MIN) {
                ch = sg != cur;
                cur = sg;
                if (ch) s_any[i] = 1;
            }
            s_ch[q * KB + i] = ch + 2 * own;
        }
        s_G[q] = G;
    }

    const int nhbu = nhb - ct.pb0, npg = nhbu > 1 ? (nhbu + 1) >> 1 : 1;
    const int per_fold = KKt >= kFixFold ? 1 : kFixFold / KKt;
    const int nCP = (TQ * ncd + 31) & ~31;
    const FastDiv d_npg(npg), d_ncp(nCP);
    // the CTAs of an SM start their few stage-A items at different warps
    const int a_rot = 32 * (int)((blockIdx.x / a.nsm) & 3);
    int n = 0;  // bra primitives of the chunk
    for (int i0 = 0; i0 < KBt; i0 += n) {
        __syncthreads();
        // a chunk ends where a quartet's sigma changes
        for (n = 1; n < a.IC && i0 + n < KBt && !s_any[i0 + n]; ++n) {
        }
        const int NIt = TQ * n * KKt;
        const FastDiv d_n(n), d_nk(n * KKt);
        // ---- A: auxiliary integrals
        // (columns of primitives a quartet lacks keep whatever they hold: the E
        // products they meet are zero)
        const bool regs = ct.L <= kFixRegL;
        // lanes per item: as many as put every thread to work, up to four (each
        // lane repeats the item's base), or more where a warp would hold few items
        const int fill = max(1, NT / NIt);
        const int G = regs ? 1 : min(fill > 32 ? 32 : 4, 1 << (31 - __clz(fill)));
        const int first = ((tid + a_rot) & (NT - 1)) / G;
        for (int it0 = first; it0 - (lane / G) < NIt; it0 += NT / G) {
            const bool in = it0 < NIt;
            const int item = in ? it0 : 0;
            const int q = d_nk.div(item), r = item - q * n * KKt, ii = d_kkt.div(r), k = r - ii * KKt;
            const int i = i0 + ii;
            const bool on = in && i < s_q[4 * q + 2] && k < s_q[4 * q + 3];
            if (G == 1 && !on) continue;
            long long* R = sR + q * QS + ii * KS + k;
            const int sg = s_sig[q * KB + i], g = s_g[q * KB + i];
            auto run = [&](auto lmax, auto fixed) {
                fix_aux_item<decltype(lmax)::value, decltype(fixed)::value>(
                    ct.L, sPb[q * KB + i], sPk[q * KK + k], a.fx_f, a.fx_tab, a.fx_far, sg, a.fx_rmu, g, tb.st, tb.ord, R,
                    NIs, G, lane & (G - 1), on);
            };
            switch (regs ? ct.L : -1) {
                case 1: run(IntC<1>(), IntC<1>()); break;
                case 2: run(IntC<2>(), IntC<1>()); break;
                case 3: run(IntC<3>(), IntC<1>()); break;
                case 4: run(IntC<4>(), IntC<1>()); break;
                default: run(IntC<kFixLmax>(), IntC<0>());
            }
        }
        {
            // the chunk's bra E products
            const int nb = n * ct.Tab;
            const FastDiv d_nb(nb), d_tab(ct.Tab);
            for (int idx = tid; idx < TQ * nb; idx += NT) {
                const int q = d_nb.div(idx), r = idx - q * nb, ii = d_tab.div(r);
                const size_t src = ((size_t)s_q[4 * q] * KB + i0) * ct.Tab + r;
                int2 e = make_int2(0, 0);
                if (i0 + ii < s_q[4 * q + 2]) {
                    if (s_ch[q * KB] & 2) {
                        const int bc = tb.bc[r - ii * ct.Tab];
                        const int sh = 60 + s_sig[q * KB + i0 + ii] * (bc & 7) - s_F[(bc >> 3) * TQ + q];
                        e = fix_limbs<kLimbE>(fix_from(a.bra_E[src], sh));
                    } else {
                        e = a.bra_limbs[src];
                    }
                }
                sEb[q * a.sEbS + r] = e;
            }
        }
        if (s_any[i0]) {
            // ket E products of the quartets whose sigma changed, relative
            // to their columns' 1-norms at the new sigma
            for (int idx = tid; idx < TQ * ncd; idx += NT) {
                const int q = d_ncd.div(idx);
                if (s_ch[q * KB + i0] & 1) s_dh[idx] = s_H[idx] - norm_exp(q, idx - q * ncd, s_sig[q * KB + i0]);
            }
            __syncthreads();
            const int nk = KK * ct.Tcd;
            const FastDiv d_qk(nk), d_kk(KK);
            for (int idx = tid; idx < TQ * nk; idx += NT) {
                const int q = d_qk.div(idx), r = idx - q * nk, t = d_kk.div(r), k = r - t * KK;
                if (!(s_ch[q * KB + i0] & 1)) continue;
                const int tc = tb.tc[t], c = q * ncd + (tc >> 3);
                const int sh = 60 + s_sig[q * KB + i0] * (tc & 7) - s_H[c] + s_dh[c];
                sEk[q * a.sEkS + t * KS + k] =
                    k < s_q[4 * q + 3]
                        ? fix_limbs<kLimbE>(fix_from(a.ket_E[(size_t)s_q[4 * q + 1] * nk + r], sh))
                        : make_int2(0, 0);
            }
        }
        if (tid == 0) s_next = NT;
        __syncthreads();
        // ---- B: ket transform and contraction, two bra Hermite functions and
        // a pair of columns per item (pairs are sorted longest first; a warp
        // takes the next 32 items when it is done with its last, which evens
        // out their lengths)
        const int nB = TQ * n * npg * ct.nkpair;
        auto ket_stage = [&](auto kt) {
            constexpr int KT = decltype(kt)::value;
            for (int item = tid;;) {
                if (item - lane >= nB) break;
                if (item < nB) {
                    const int q = item & (TQ - 1), r = item >> lgTQ, s = d_n.div(r), ii = r - s * n;
                    const int pr = d_npg.div(s), pg = s - pr * npg, x = q * KB + i0 + ii;
                    const int c1 = tb.kpair[2 * pr], c2 = tb.kpair[2 * pr + 1];
                    const int t1 = tb.kstart[c1], n1 = tb.kstart[c1 + 1] - t1;
                    const int t2 = c2 < 0 ? t1 : tb.kstart[c2], n2 = c2 < 0 ? 0 : tb.kstart[c2 + 1] - t2;
                    const int2* Rc = reinterpret_cast<const int2*>(sR) + q * QS + ii * KS;
                    const int p0 = ct.pb0 + pg, p1 = ct.pb0 + pg + npg;
                    // (for a quartet without primitive i the bra's E are zero, and X immaterial;
                    // ds is 0 where the quartet forms its own bra limbs)
                    const int dG = s_G[q] - s_g[x], ds = s_ds[x];
                    int2* X = sX + ii * XS + q;
                    auto put = [&](int p, int cd, const FixAcc& v) {
                        const int sh = max(0, min(s_dh[q * ncd + cd] + dG + ds * (int)tb.ord[p], 62));
                        X[(p * ncd + cd) * TQ] = fix_limbs<kLimbX>((fix_ket_sum(v) + ((1LL << sh) >> 1)) >> sh);
                    };
                    int left = per_fold;
                    const int2 *E1 = sEk + q * a.sEkS + t1 * KS, *E2 = sEk + q * a.sEkS + t2 * KS;
                    const int16_t* kq = tb.kq + t1;
                    const int2 *const Ea[2] = {E1, E2}, *const Eb[1] = {E1};
                    if (nhbu > 1) {
                        const uint16_t* const row[2] = {tb.pq + p0 * nhk, tb.pq + (p1 < nhb ? p1 : p0) * nhk};
                        FixAcc s2[2][2];
                        fix_ket_rows<2, 2, KT>(s2, Ea, Rc, row, kq, 0, n2, KKt, KS, per_fold, left);
                        fix_ket_rows<2, 1, KT>(s2, Eb, Rc, row, kq, n2, n1, KKt, KS, per_fold, left);
                        put(p0, c1, s2[0][0]);
                        if (c2 >= 0) put(p0, c2, s2[0][1]);
                        if (p1 < nhb) {
                            put(p1, c1, s2[1][0]);
                            if (c2 >= 0) put(p1, c2, s2[1][1]);
                        }
                    } else {
                        const uint16_t* const row[1] = {tb.pq + p0 * nhk};
                        FixAcc s2[1][2];
                        fix_ket_rows<1, 2, KT>(s2, Ea, Rc, row, kq, 0, n2, KKt, KS, per_fold, left);
                        fix_ket_rows<1, 1, KT>(s2, Eb, Rc, row, kq, n2, n1, KKt, KS, per_fold, left);
                        put(p0, c1, s2[0][0]);
                        if (c2 >= 0) put(p0, c2, s2[0][1]);
                    }
                }
                int next = 0;
                if (lane == 0) next = atomicAdd(&s_next, 32);
                item = __shfl_sync(0xffffffffu, next, 0) + lane;
            }
        };
        switch (KKt) {
            case 1: ket_stage(IntC<1>()); break;
            case 3: ket_stage(IntC<3>()); break;
            case 9: ket_stage(IntC<9>()); break;
            default: ket_stage(IntC<0>());
        }
        __syncthreads();
        // ---- C: bra transform and contraction over the chunk's bra primitives
        // (an item: a pair of rows of one (quartet, cd) over one read of X; a pair's
        // items fill whole warps, so that a warp walks one pair's terms)
        for (int item = tid; item < ct.nbpair * nCP; item += NT) {
            const int pr = d_ncp.div(item), r = item - pr * nCP;
            if (r >= TQ * ncd) continue;
            const int q = r & (TQ - 1), a1 = tb.bpair[2 * pr], a2 = tb.bpair[2 * pr + 1];
            const int t1 = tb.bstart[a1], n1 = tb.bstart[a1 + 1] - t1;
            const int t2 = a2 < 0 ? t1 : tb.bstart[a2], n2 = a2 < 0 ? 0 : tb.bstart[a2 + 1] - t2;
            const int2 *E1 = sEb + q * a.sEbS + t1, *E2 = sEb + q * a.sEbS + t2;
            const int2* X = sX + r;
            const uint16_t* bp = tb.bp + t1;
            FixAcc f1, f2;
            int left = kFixFold;
            for (int ii = 0; ii < n; ++ii, E1 += ct.Tab, E2 += ct.Tab, X += XS) {
                int u = 0;
                for (; u < n2; ++u) {
                    const int2 x = X[bp[u]], e1 = E1[u], e2 = E2[u];
                    fix_mac(f1, e1.x, e1.y, x.x, x.y);
                    fix_mac(f2, e2.x, e2.y, x.x, x.y);
                    if (--left == 0) {
                        left = kFixFold;
                        fix_fold(f1);
                        fix_fold(f2);
                    }
                }
                for (; u < n1; ++u) {
                    const int2 x = X[bp[u]], e1 = E1[u];
                    fix_mac(f1, e1.x, e1.y, x.x, x.y);
                    if (--left == 0) {
                        left = kFixFold;
                        fix_fold(f1);
                        fix_fold(f2);
                    }
                }
            }
            sA[a1 * TQ * ncd + r] += fix_bra_sum(f1);
            if (a2 >= 0) sA[a2 * TQ * ncd + r] += fix_bra_sum(f2);
        }
    }
    __syncthreads();
    // units of 2^(G + H + f - 62)
    tile_epilogue<NT, 0>(
        a,
        [&](int, int item) {
            const int q = item & (TQ - 1), r = item >> lgTQ, ab = d_ncd.div(r), cd = r - ab * ncd;
            if (q >= nqt) return 0.0;
            const int F = s_ch[q * KB] & 2 ? s_F[ab * TQ + q] : a.bra_ex[(size_t)s_q[4 * q] * nab + ab];
            const int e = s_G[q] + s_H[q * ncd + cd] + F - 62;
            // two factors: e may pass the exponent range of one
            const int eh = max(-1000, min(1000, e)), el = max(-1000, min(1000, e - eh));
            double v = (double)sA[item] * __hiloint2double((1023 + eh) << 20, 0);
            if (el) v *= __hiloint2double((1023 + el) << 20, 0);
            return v;
        },
        q0, nqt, sm, s_q, s_qq, s_red);
}

// Class tables into shared memory: the FP64 tile's, with the Hermite indices
// turned into offsets of this tile shape, the terms' columns and orders,
// the Hermite orders.
template <int NT>
__device__ __forceinline__ void stage_fixed_tables(const FwdArgs& a, double* sm)
{
    const ClassTables& ct = a.ct;
    const int tid = threadIdx.x;
    const int KS = (a.KK + 1) & ~1, NIs = r_row_stride(a.TQ * r_row_stride(a.IC * KS, 1), 1);
    const FixTables tb(ct, sm + a.o_tab);
    for (int i = tid; i <= ct.nab; i += NT) const_cast<int*>(tb.bstart)[i] = ct.bra_start[i];
    for (int i = tid; i <= ct.ncd; i += NT) const_cast<int*>(tb.kstart)[i] = ct.ket_start[i];
    // offsets are into at most the 227 KB of a CTA, in 8-byte entries
    for (int i = tid; i < ct.Tab; i += NT) const_cast<uint16_t*>(tb.bp)[i] = (uint16_t)(ct.bra_p[i] * ct.ncd * a.TQ);
    for (int i = tid; i < ct.Tcd; i += NT) const_cast<int16_t*>(tb.kq)[i] = ct.ket_q[i];
    for (int i = tid; i < ct.nhb * ct.nhk; i += NT) const_cast<uint16_t*>(tb.pq)[i] = (uint16_t)(ct.pq[i] * NIs);
    for (int cd = tid; cd < ct.ncd; cd += NT)
        for (int t = ct.ket_start[cd]; t < ct.ket_start[cd + 1]; ++t)
            const_cast<int16_t*>(tb.tc)[t] = (int16_t)(cd * 8 + herm_order(ct.ket_q[t]));
    for (int ab = tid; ab < ct.nab; ab += NT)
        for (int t = ct.bra_start[ab]; t < ct.bra_start[ab + 1]; ++t)
            const_cast<int16_t*>(tb.bc)[t] = (int16_t)(ab * 8 + herm_order(ct.bra_p[t]));
    for (int e = tid; e < ct.nhl; e += NT) {
        const_cast<int16_t*>(tb.ord)[e] = (int16_t)herm_order(e);
        const RStep r = a.rsteps[e];
        const_cast<FixStep*>(tb.st)[e] = FixStep{8 * r.src1 * NIs, r.coef ? 8 * r.src2 * NIs : 0, r.axis, r.coef};
    }
    for (int i = tid; i < 2 * ct.nkpair; i += NT) const_cast<int16_t*>(tb.kpair)[i] = ct.kpairs[i];
    for (int i = tid; i < 2 * ct.nbpair; i += NT) const_cast<int16_t*>(tb.bpair)[i] = ct.bpairs[i];
}

template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) fwd_fixed_kernel(FwdArgs a)
{
    extern __shared__ __align__(16) double sm[];
    __shared__ double s_red;
    if (threadIdx.x == 0) s_red = 0.0;
    stage_fixed_tables<NT>(a, sm);
    for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        const int64_t q0 = tile * a.TQ;
        tile_fixed<NT>(a, q0, (int)min((int64_t)a.TQ, a.nq - q0), sm, &s_red);
    }
}

}  // namespace eri
