// eri_fwd.cu -- forward ERI batches: eri_boys and eri_batch.
//
// Per class and batch (Section 3.1: bra pair list x ket pair list):
//  1. prepass_kernel   validates indices, angular momenta and contraction
//                      degrees and finds the largest K on each centre;
//  2. pair_kernel      per primitive pair: zeta_p, P, 2pi^(5/2)/zeta_p or
//                      1/zeta_q, and the products E^x E^y E^z of the
//                      Hermite expansion coefficients (Eqs. E2rr1/E2rr2/
//                      E2-000) for every nonzero (Cartesian pair, Hermite)
//                      term, with c_a c_b folded in and, on the ket, the
//                      sign (-1)^{l_q} of Eq. pq-from-r;
//  3. fwd_kernel       per tile of quartets, staged through shared memory:
//       A. [r]^(0) for every primitive quartet of the tile (Boys function,
//          Eq. 0m, Eq. r-rr);
//       B. ket transform and ket contraction (Eq. ket-from-hermite):
//          X[p][cd] = sum_k sum_q E^cd_{k,q} [p+q]^(0)_{ik};
//       C. bra transform and bra contraction (Eq. bra-from-hermite):
//          (ab|cd) += sum_p E^ab_{i,p} X[p][cd], accumulated over bra
//          primitives i in registers (or in `out` for very large shellsets),
//     then coalesced stores of the quartet-fastest output.
// Every FP64 operation of the path runs in these kernels.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "eri_device.cuh"
#include "eri_fixed.cuh"
#include "eri_internal.h"
#include "eri_tile.cuh"

namespace eri {

// ---------------------------------------------------------------------------
// 1. prepass
// ---------------------------------------------------------------------------
struct PrepassArgs {
    const int32_t* shell_l;
    const int32_t* shell_K;
    int32_t nshell;
    const int32_t* bra;
    int64_t nbra;
    const int32_t* ket;
    int64_t nket;
    const int64_t* quartets;
    int64_t nq;
    int l[4];
    int unit_b;  // 1: every bra pair's second shell is -1, the unit function (3-centre)
    int* info;   // [0..3] max K per centre, [4] error, [5..6] recursion risk (float bits)
    // recursion risk (risk = 1): per pair (2|A-B|)^l2 max_ij exp(-mu_ij |A-B|^2),
    // the factor by which the horizontal recursion can magnify the pair's
    // rounding relative to its integrals; the largest over bra (ket) pairs
    int risk;
    const double* centres;
    const int32_t* shell_atom;
    const int32_t* shell_off;
    const double* exps;
    int* kmin;   // optional [2]: INT_MAX less the smallest primitive-pair count K1 K2 over bra (ket) pairs
    // optional [7]: the largest zeta_max / zeta_min of a bra (ket) pair (float
    // bits), 1 if a primitive lies outside the fixed-point tile's range, the
    // largest |coordinate|, the largest zeta of a bra (ket) pair and the largest
    // distance of a pair's centres (float bits)
    int* spread;
    const double* coefs;
};

// The fixed-point tile's range of primitives: exponents and coefficients far
// from the ends of the FP64 range, and finite (the FP64 tile takes the rest).
__device__ __forceinline__ bool fix_range(double z, double c)
{
    return z >= 1e-8 && z <= 1e8 && fabs(c) <= 1e30;
}

// zeta_max / zeta_min over the primitive pairs of shells s1, s2 (s2 < 0: the
// unit function); *bad set where a primitive or centre is out of range, *far
// raised to the largest |coordinate|, *wide to the distance of the centres, *zmax
// the largest zeta
__device__ float pair_spread(const PrepassArgs& a, int s1, int s2, bool* bad, float* far, float* wide, float* zmax)
{
    float lo = 0.f, hi = 0.f, r2 = 0.f;
    for (int x = 0; x < 3 && s2 >= 0; ++x) {
        const float d = (float)(a.centres[3 * a.shell_atom[s1] + x] - a.centres[3 * a.shell_atom[s2] + x]);
        r2 = fmaf(d, d, r2);
    }
    *wide = fmaxf(*wide, sqrtf(r2));
    for (int c = 0; c < 2; ++c) {
        const int s = c ? s2 : s1;
        if (s < 0) continue;
        float zl = 3e38f, zh = 0.f;
        for (int i = a.shell_off[s]; i < a.shell_off[s] + a.shell_K[s]; ++i) {
            *bad |= !fix_range(a.exps[i], a.coefs[i]);
            zl = fminf(zl, (float)a.exps[i]);
            zh = fmaxf(zh, (float)a.exps[i]);
        }
        for (int x = 0; x < 3; ++x) {
            const double r = fabs(a.centres[3 * a.shell_atom[s] + x]);
            *bad |= !(r <= 1e6);
            *far = fmaxf(*far, __double2float_ru(r));
        }
        lo += zl;
        hi += zh;
    }
    *zmax = hi;
    return hi / lo;
}

// Copies the prepass results to mapped host memory.
__global__ void info_to_host_kernel(const int* __restrict__ src, int n, int* dst)
{
    if ((int)threadIdx.x < n) dst[threadIdx.x] = src[threadIdx.x];
}

// (2|A-B|)^l2 max over primitive pairs of exp(-z1 z2 / (z1 + z2) |A-B|^2), the
// maximum being that of the smallest exponents.  In floats from the FP64
// distance (to about 1e-5: the guard compares it with a round power of ten);
// FP64 pow and exp and a division per primitive pair took 26 of the 30 us that
// this kernel was of a batch of 1000 (pp|pp) (143 us); in floats it took 13.
__device__ float pair_recursion_risk(const PrepassArgs& a, int s1, int s2, int l2)
{
    if (l2 == 0) return 1.0f;
    const double* A = a.centres + 3 * a.shell_atom[s1];
    const double* B = a.centres + 3 * a.shell_atom[s2];
    const double d2 = (A[0] - B[0]) * (A[0] - B[0]) + (A[1] - B[1]) * (A[1] - B[1]) + (A[2] - B[2]) * (A[2] - B[2]);
    const float r2 = d2 > 1e30 ? 1e30f : (float)d2;  // finite: no inf - inf below
    float z1 = 3.0e38f, z2 = 3.0e38f;
    for (int i = 0; i < a.shell_K[s1]; ++i) z1 = fminf(z1, (float)a.exps[a.shell_off[s1] + i]);
    for (int j = 0; j < a.shell_K[s2]; ++j) z2 = fminf(z2, (float)a.exps[a.shell_off[s2] + j]);
    const float lo = fminf(z1, z2), mu = lo / (1.0f + lo / fmaxf(z1, z2));
    return fminf(expf((float)l2 * logf(2.0f * sqrtf(r2)) - mu * r2), 3.0e38f);
}

__device__ __forceinline__ void set_err(int* p, int code) { atomicCAS(p, 0, code); }

// The largest of a warp's v into *p (0 or more; floats by their bits): the pairs
// of a batch all meet in a few words, whose atomics took most of this kernel.
__device__ __forceinline__ void warp_max_into(int* p, int v)
{
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && v > 0) atomicMax(p, v);
}

__global__ void prepass_kernel(PrepassArgs a)
{
    const int64_t n = max(max(a.nbra, a.nket), a.nq);
    // this thread's largest values, reduced per warp at the end
    int kmax[4] = {0, 0, 0, 0}, kmin[2] = {0, 0}, risk[2] = {0, 0}, ratio[2] = {0, 0}, zeta[2] = {0, 0}, coord = 0, apart = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const int32_t* pr = side == 0 ? a.bra : a.ket;
            const int64_t np = side == 0 ? a.nbra : a.nket;
            if (i >= np) continue;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int32_t s = pr[2 * i + c];
                if (a.unit_b && side == 0 && c == 1) {
                    if (s != -1) set_err(&a.info[4], DEV_EINDEX);
                    kmax[1] = 1;
                    continue;
                }
                if (s < 0 || s >= a.nshell) {
                    set_err(&a.info[4], DEV_EINDEX);
                    continue;
                }
                const int l = a.shell_l[s], K = a.shell_K[s];
                if (l != a.l[2 * side + c]) set_err(&a.info[4], DEV_ECLASS);
                if (K < 1 || K > kKmax) {
                    set_err(&a.info[4], DEV_EK);
                    continue;
                }
                kmax[2 * side + c] = max(kmax[2 * side + c], K);
            }
            if (a.kmin) {
                const int s1 = pr[2 * i], s2 = pr[2 * i + 1];
                const bool unit = a.unit_b && side == 0;
                if (s1 >= 0 && s1 < a.nshell && (unit || (s2 >= 0 && s2 < a.nshell)))
                    kmin[side] = max(kmin[side], INT_MAX - max(0, a.shell_K[s1] * (unit ? 1 : a.shell_K[s2])));
            }
            if (a.spread) {
                const int s1 = pr[2 * i], s2 = pr[2 * i + 1];
                const bool unit = a.unit_b && side == 0;
                if (s1 >= 0 && s1 < a.nshell && (unit || (s2 >= 0 && s2 < a.nshell))) {
                    const int K1 = a.shell_K[s1], K2 = unit ? 1 : a.shell_K[s2];
                    if (K1 >= 1 && K1 <= kKmax && K2 >= 1 && K2 <= kKmax) {
                        bool bad = false;
                        float far = 0.f, wide = 0.f, zmax;
                        const float r = pair_spread(a, s1, unit ? -1 : s2, &bad, &far, &wide, &zmax);
                        apart = max(apart, __float_as_int(wide));
                        zeta[side] = max(zeta[side], __float_as_int(zmax));
                        ratio[side] = max(ratio[side], __float_as_int(r));  // r >= 1: int order = float order
                        if (bad) a.spread[2] = 1;
                        coord = max(coord, __float_as_int(far));
                    }
                }
            }
            if (a.risk) {
                const int s1 = pr[2 * i], s2 = pr[2 * i + 1];
                if (s1 >= 0 && s1 < a.nshell && s2 >= 0 && s2 < a.nshell) {
                    const int K1 = a.shell_K[s1], K2 = a.shell_K[s2];
                    if (K1 >= 1 && K1 <= kKmax && K2 >= 1 && K2 <= kKmax) {
                        const float r = pair_recursion_risk(a, s1, s2, a.l[2 * side + 1]);
                        risk[side] = max(risk[side], __float_as_int(r));  // r >= 0: int order = float order
                    }
                }
            }
        }
        if (a.quartets && i < a.nq) {
            const int64_t b = a.quartets[2 * i], k = a.quartets[2 * i + 1];
            if (b < 0 || b >= a.nbra || k < 0 || k >= a.nket) set_err(&a.info[4], DEV_EINDEX);
        }
    }
    // every thread of the block reaches this point
    for (int c = 0; c < 4; ++c) warp_max_into(&a.info[c], kmax[c]);
    for (int side = 0; side < 2; ++side) {
        if (a.kmin) warp_max_into(&a.kmin[side], kmin[side]);
        if (a.risk) warp_max_into(&a.info[5 + side], risk[side]);
        if (!a.spread) continue;
        warp_max_into(&a.spread[side], ratio[side]);
        warp_max_into(&a.spread[4 + side], zeta[side]);
    }
    if (!a.spread) return;
    warp_max_into(&a.spread[3], coord);
    warp_max_into(&a.spread[6], apart);
}

// ---------------------------------------------------------------------------
// 2. primitive-pair tables
// ---------------------------------------------------------------------------
struct PairArgs {
    const double* centres;
    const int32_t* shell_atom;
    const int32_t* shell_K;
    const int32_t* shell_off;
    const double* exps;
    const double* coefs;
    const int32_t* pairs;
    int64_t npairs;
    int l1, l2;
    int KS;                 // primitive-pair slots per pair
    int T;                  // terms
    const uint8_t* fac;     // [T][3] per-axis E-table indices
    int ket;                // 1: ket side (sign (-1)^{l_q}, scale 1/zeta_q)
    double* ps;             // [npairs][KS][PS_N]
    double* E;              // [npairs][T][KS] (slot fastest)
    int32_t* kprim;         // [npairs] number of valid slots K1*K2
    // adjoint only (ax == nullptr otherwise): per-axis tables with both
    // indices raised by up to 2, ax[(g*3 + axis)*eax + (i*(l2+3) + j)*(l1+l2+5) + t]
    double* ax;
    int eax;
    double* zz;             // [npairs][KS][2]: the two exponents
    int split;              // 1: E products stored as float pairs (hi, lo) in the double slots
    int hrr;                // 1: terms of E_{e,0}, |e| = l1..l1+l2 (horizontal-recursion form)
    const double* scale;    // [T] per-term factors (solid-harmonic side), or null
    // fixed-point tile (never with ax): a pair's slots in descending order of
    // zeta, ps holds FixPrim with coordinates in units of 2^-fx_f, and the E
    // products carry a further zeta^(-1/2),
    int fixed, fx_f;
    int32_t* weak;          // [npairs], zeroed here (bra)
    double mu;              // and mu^(Hermite order) (eri_fixed.cuh)
};

constexpr int kPairThreads = 128;
constexpr double kPairWarpSlots = 640.0;  // times sqrt(terms): at most this many slots take a warp each
constexpr int kEax = (kLmax + 3) * (kLmax + 3) * (2 * kLmax + 5);  // per-axis E table bound (adjoint shifts)
constexpr int kEfw = (kLmax + 1) * (kLmax + 1) * (2 * kLmax + 1);  // without the shifts (also the HRR form's)

// c1 c2 k zeta^(-3/2) (times 2 pi^(5/2) on the bra), rounded once at the end: the
// fixed-point tile takes its E products as they come, so the roundings of this
// factor, two more than the FP64 tile's, would be most of its error.
__device__ __forceinline__ double fix_e00(double c1, double c2, double k, double p, double invp, int ket)
{
    // products as unevaluated sums hi + lo
    const double a = c1 * c2, al = fma(c1, c2, -a);
    const double b = a * k, bl = fma(a, k, -b) + al * k;
    const double s = sqrt(invp), sl = fma(-s, s, invp) * (0.5 / s);
    double w = invp * s;
    // (1/zeta)^(3/2) = invp^(3/2) (1 + 3/2 (1 - invp zeta))
    double wl = fma(invp, s, -w) + invp * sl + 1.5 * w * fma(-invp, p, 1.0);
    if (!ket) {
        const double v = w * kTwoPi52;
        wl = fma(w, kTwoPi52, -v) + (wl * kTwoPi52 + w * kTwoPi52Lo);
        w = v;
    }
    const double r = b * w;
    return r + (fma(b, w, -r) + (b * wl + bl * w));
}

// RAISED: the adjoint's tables (a.ax != NULL): the per-axis E tables with
// both indices raised by 2, one thread per (slot, axis).  The adjoint reads
// no E products of that side, so none are formed.  Otherwise one thread per
// slot forms the three tables and the E products of the class's terms; WARP: a
// warp does, lanes 0..2 a table each (in shared memory), then every lane its
// share of the products.  A batch of few slots with long term lists leaves one
// thread per slot latency bound on 16 of the 152 SMs: 2048 uncontracted (ff|
// pairs 917 us, of a batch of 7.2 ms.
template <bool RAISED, bool WARP>
__global__ void __launch_bounds__(kPairThreads) pair_kernel_t(PairArgs a)
{
    static_assert(!(RAISED && WARP), "the raised tables take a thread per axis");
    constexpr int NX = RAISED || WARP ? 1 : 3;  // axes per thread
    constexpr int PER = RAISED ? 3 : (WARP ? 32 : 1);  // threads per slot
    __shared__ double s_E[WARP ? kPairThreads / 32 : 1][3][WARP ? kEfw : 1];
    const int lane = WARP ? threadIdx.x & 31 : 0;
    const int64_t total = a.npairs * a.KS * PER;
    for (int64_t gg = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; gg < total;
         gg += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = gg / PER;                     // the slot
        const int x0 = RAISED ? (int)(gg - g * 3) : 0;  // its first axis
        if (WARP) __syncwarp();                         // the last slot's tables are read
        const int64_t j = g / a.KS;
        const int s = (int)(g - j * a.KS);
        // s2 = -1: the unit function (exponent 0, coefficient 1) of a 3-centre
        // bra; its centre is immaterial and taken as the first shell's
        const int s1 = a.pairs[2 * j], s2 = a.pairs[2 * j + 1];
        const int K1 = a.shell_K[s1], K2 = s2 < 0 ? 1 : a.shell_K[s2];
        if (s == 0 && x0 == 0 && lane == 0) {
            a.kprim[j] = K1 * K2;
            if (!RAISED && a.weak) a.weak[j] = 0;
        }
        if (s >= K1 * K2) {  // padding slot: finite zeros, never contributes
            if (RAISED) {
                for (int q = 0; q < a.eax; ++q) a.ax[((size_t)g * 3 + x0) * a.eax + q] = 0.0;
                if (x0 != 0) continue;
                a.zz[2 * g] = a.zz[2 * g + 1] = 1.0;
            } else {
                for (int t = lane; t < a.T; t += WARP ? 32 : 1)
                    a.E[a.fixed && !a.ket ? (size_t)g * a.T + t : ((size_t)j * a.T + t) * a.KS + s] = 0.0;
            }
            if (lane != 0) continue;
            if (!RAISED && a.fixed) {
                reinterpret_cast<FixPrim*>(a.ps)[g] = FixPrim{{0, 0, 0}, 1LL << 61, 1, 1.0f};
                continue;
            }
            double* o = a.ps + (size_t)g * PS_N;
            o[PS_P] = 1.0;
            o[PS_PX] = o[PS_PY] = o[PS_PZ] = 0.0;
            continue;
        }
        const int i1 = s / K2, i2 = s - i1 * K2;
        const int p1 = a.shell_off[s1] + i1, p2 = s2 < 0 ? -1 : a.shell_off[s2] + i2;
        const double z1 = a.exps[p1], z2 = s2 < 0 ? 0.0 : a.exps[p2];
        const double c2 = s2 < 0 ? 1.0 : a.coefs[p2];
        const double* A = a.centres + 3 * a.shell_atom[s1];
        const double* B = s2 < 0 ? A : a.centres + 3 * a.shell_atom[s2];
        const double p = z1 + z2;
        const double invp = 1.0 / p;
        int so = s;  // output slot
        if (!RAISED && a.fixed) {
            so = 0;
            for (int x1 = 0; x1 < K1; ++x1)
                for (int x2 = 0; x2 < K2; ++x2) {
                    const double z = a.exps[a.shell_off[s1] + x1] + (s2 < 0 ? 0.0 : a.exps[a.shell_off[s2] + x2]);
                    so += z > p || (z == p && x1 * K2 + x2 < s);
                }
        }
        const double inv2p = 0.5 * invp;
        double P[3], AB2 = 0.0;
        for (int x = 0; x < 3; ++x) {
            P[x] = (z1 * A[x] + z2 * B[x]) * invp;
            const double d = A[x] - B[x];
            AB2 = fma(d, d, AB2);
        }
        auto PA = [&](int x) { return (x == 0 ? P[0] : (x == 1 ? P[1] : P[2])) - A[x]; };
        auto PB = [&](int x) { return (x == 0 ? P[0] : (x == 1 ? P[1] : P[2])) - B[x]; };
        // K_AB c_1 c_2 carried by the x-axis bootstrap E_00^0 (Eq. E2-000),
        // 1 on y and z: the products E^x E^y E^z are unchanged.  So is the
        // pair's factor of the Eq. 0m prefactor, 2 pi^(5/2) / zeta_p on the
        // bra and 1 / zeta_q on the ket: every E of the pair (per-axis tables
        // and products alike) carries it once, and [0]^(m) needs only the
        // quartet's 1/sqrt(zeta_p + zeta_q).
        const double kab = exp(-z1 * z2 * invp * AB2);
        // (fixed point: with zeta^(-1/2), 1/sqrt(zeta_p + zeta_q) = sqrt(rho / (zeta_p zeta_q)))
        const double e00x = !RAISED && a.fixed ? fix_e00(a.coefs[p1], c2, kab, p, invp, a.ket)
                                               : a.coefs[p1] * c2 * kab * (a.ket ? invp : kTwoPi52 * invp);
        const int ext = RAISED ? 2 : 0;
        // largest raised indices: the adjoint raises both by 2; the
        // horizontal-recursion form needs E_{i,0} for i <= l1 + l2
        const int m1 = a.hrr ? a.l1 + a.l2 : a.l1 + ext, m2 = a.hrr ? 0 : a.l2 + ext;
        const int L12 = a.l1 + a.l2, n2 = m2 + 1, nt = m1 + m2 + 1;
        double El[WARP ? 1 : NX][WARP ? 1 : (RAISED ? kEax : kEfw)];
        for (int xi = 0; xi < NX; ++xi) {
            const int x = WARP ? lane : x0 + xi;
            if (WARP && x >= 3) break;
            double* Ex = WARP ? s_E[threadIdx.x >> 5][x] : El[xi];
            for (int q = 0; q < (m1 + 1) * n2 * nt; ++q) Ex[q] = 0.0;
            Ex[0] = x == 0 ? e00x : 1.0;
            const double pa = PA(x), pb = PB(x);
            // raise the first index at j = 0 (Eq. E2rr1)
            for (int i = 0; i < m1; ++i)
                for (int t = 0; t <= i + 1; ++t) {
                    double v = 0.0;
                    if (t >= 1) v = inv2p * Ex[(i * n2) * nt + t - 1];
                    if (t <= i) v = fma(pa, Ex[(i * n2) * nt + t], v);
                    if (t + 1 <= i) v = fma((double)(float)(t + 1), Ex[(i * n2) * nt + t + 1], v);
                    Ex[((i + 1) * n2) * nt + t] = v;
                }
            // raise the second index for every first index (Eq. E2rr2)
            for (int i = 0; i <= m1; ++i)
                for (int jj = 0; jj < m2; ++jj)
                    for (int t = 0; t <= i + jj + 1; ++t) {
                        const int b0 = (i * n2 + jj) * nt;
                        double v = 0.0;
                        if (t >= 1) v = inv2p * Ex[b0 + t - 1];
                        if (t <= i + jj) v = fma(pb, Ex[b0 + t], v);
                        if (t + 1 <= i + jj) v = fma((double)(float)(t + 1), Ex[b0 + t + 1], v);
                        Ex[(i * n2 + jj + 1) * nt + t] = v;
                    }
        }
        if (RAISED) {
            double* o = a.ax + ((size_t)g * 3 + x0) * a.eax;
            for (int q = 0; q < (m1 + 1) * n2 * nt; ++q) o[q] = El[0][q];
            if (x0 != 0) continue;
            a.zz[2 * g] = z1;
            a.zz[2 * g + 1] = z2;
        } else {
            // term t at Eout[t * es]: slot fastest, or (fixed-point bra) term fastest
            const size_t es = a.fixed && !a.ket ? 1 : a.KS;
            double* Eout = a.E + (a.fixed && !a.ket ? ((size_t)j * a.KS + so) * a.T : (size_t)j * a.T * a.KS + so);
            const int ntc = L12 + 1, n2c = a.hrr ? 1 : a.l2 + 1;  // dims the class-table indices use
            const double* T0 = WARP ? s_E[threadIdx.x >> 5][0] : El[0];
            const double* T1 = WARP ? s_E[threadIdx.x >> 5][1] : El[NX > 1 ? 1 : 0];
            const double* T2 = WARP ? s_E[threadIdx.x >> 5][2] : El[NX > 2 ? 2 : 0];
            if (WARP) __syncwarp();
            for (int t = lane; t < a.T; t += WARP ? 32 : 1) {
                int idx[3], lq = 0;
                for (int x = 0; x < 3; ++x) {
                    const int f = a.fac[3 * t + x];
                    const int tt = f % ntc, bb = (f / ntc) % n2c, aa = f / (ntc * n2c);
                    idx[x] = (aa * n2 + bb) * nt + tt;
                    lq += tt;
                }
                double v = T0[idx[0]] * T1[idx[1]] * T2[idx[2]];
                if (a.scale) v *= a.scale[t];
                if (a.ket && (lq & 1)) v = -v;
                if (a.fixed)
                    for (int x = 0; x < lq; ++x) v *= a.mu;
                if (a.split)
                    reinterpret_cast<float2*>(Eout)[t * es] = split_f64(v);
                else
                    Eout[t * es] = v;
            }
        }
        if (lane != 0) continue;
        if (!RAISED && a.fixed) {
            FixPrim f;
            for (int x = 0; x < 3; ++x) f.x[x] = fix_coordinate(P[x], a.fx_f);
            // 1/zeta to 62 bits: the rounded reciprocal and its residual
            fix_split_exponent(invp, &f.um, &f.ue);
            f.um += (long long)(fma(-invp, p, 1.0) * (double)f.um);
            f.zeta = (float)p;
            reinterpret_cast<FixPrim*>(a.ps)[j * a.KS + so] = f;
            continue;
        }
        double* o = a.ps + (size_t)(j * a.KS + so) * PS_N;
        o[PS_P] = p;
        o[PS_PX] = P[0];
        o[PS_PY] = P[1];
        o[PS_PZ] = P[2];
    }
}

// grid: blocks of 128 threads for one thread per slot; the raised kernel
// takes three per slot
static void launch_pair(const PairArgs& p, int grid, cudaStream_t st)
{
    // A warp per slot where the slots are few for one thread each: one thread takes the
    // same time for any number of slots up to the chip's threads, warps queue from about
    // 3000 on.  Calls of one quartet, us, one thread | one warp per slot: (pp|, 33 terms,
    // 1000 slots 99 | 87, 3000 98 | 95, 4500 99 | 105, 8192 103 | 124; (dp|, 108, 6000
    // 136 | 126, 8192 132 | 140; (dd|, 336, 8192 240 | 182, 16384 242 | 276; (ff|, 1920,
    // 16384 984 | 646: they cross near 640 sqrt(terms).  Lists of fewer than 16 terms
    // leave most lanes idle.
    const int64_t slots = p.npairs * p.KS;
    if (p.ax)
        pair_kernel_t<true, false><<<(int)std::min<int64_t>(3LL * grid, 24LL * sm_count()), kPairThreads, 0, st>>>(p);
    else if (p.T >= 16 && (double)slots <= kPairWarpSlots * std::sqrt((double)p.T))
        pair_kernel_t<false, true><<<(int)std::max<int64_t>(1, std::min<int64_t>((32 * slots + kPairThreads - 1) / kPairThreads, 16LL * sm_count())),
                                     kPairThreads, 0, st>>>(p);
    else
        pair_kernel_t<false, false><<<grid, kPairThreads, 0, st>>>(p);
}

static const auto fwd_kernel = fwd_kernel_t<false, kNT>;
static const auto fwd_kernel_split = fwd_kernel_t<true, kNT>;

// A tile whose shared memory leaves room for one CTA per SM (each CTA also
// takes a 1 KB system reserve and a few bytes of static shared memory).
static bool one_cta_per_sm(size_t bytes) { return 2 * (bytes + 1024 + 64) > (size_t)smem_per_sm(); }

// The forward kernel for the transforms' arithmetic and a CTA width (kNT or kNTWide).
static void (*fwd_kern(int split, int nt))(FwdArgs)
{
    if (split == XF_FIXED)
        return nt == kNTWide ? fwd_fixed_kernel<kNTWide> : (nt == kNTSlim ? fwd_fixed_kernel<kNTSlim> : fwd_fixed_kernel<kNT>);
    if (nt == kNTWide) return split ? fwd_kernel_t<true, kNTWide> : fwd_kernel_t<false, kNTWide>;
    return split ? fwd_kernel_split : fwd_kernel;
}

// ---------------------------------------------------------------------------
// Boys entry kernel
// ---------------------------------------------------------------------------
__global__ void boys_kernel(int mmax, const double* T, int64_t n, const double* tab, double* F)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double f[ERI_BOYS_MMAX + 1];
        boys_eval(mmax, T[i], tab, f);
        for (int m = 0; m <= mmax; ++m) F[i * (mmax + 1) + m] = f[m];
    }
}

int sm_count()
{
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

int smem_per_sm()
{
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        if (n <= 0) n = 64 * 1024;
    }
    return n;
}

int max_smem_optin()
{
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (n <= 0) n = 48 * 1024;
    }
    return n;
}

// ---------------------------------------------------------------------------
// Tile planning: pick (TQ, IC, e_smem, acc_regs) so that shared memory fits
// and the auxiliary-integral stage has enough independent items.
// ---------------------------------------------------------------------------
static int odd_up(int n) { return n | 1; }

// Ping-pong buffers of the epilogue's horizontal recursions: level g of the
// combined sequence (ket levels 0..ld, then bra levels 1..lb) lives in
// buffer g % 2; *A and *B are the largest even and odd level (doubles).
static void hrr_buffers(const ClassTables& ct, int TQ, size_t* A, size_t* B)
{
    *A = *B = 0;
    for (int g = 0; g <= ct.ld + ct.lb; ++g) {
        const size_t n = g <= ct.ld ? (size_t)TQ * ct.nab * ct.kn[g] : (size_t)TQ * ct.ncd_f * ct.bn[g - ct.ld];
        size_t& m = (g & 1) ? *B : *A;
        m = std::max(m, n);
    }
}

bool tile_layout(const ClassTables& ct, int KB, int KK, int TQ, int IC, int e_smem, TilePlan* tp, int split, int nt)
{
    size_t off = 0;
    auto take = [&](size_t nd) {
        size_t o = off;
        off += (nd + 1) & ~size_t(1);  // keep 16-byte alignment
        return (int)o;
    };
    auto even = [](size_t nd) { return (nd + 1) & ~size_t(1); };
    tp->TQ = TQ;
    tp->IC = IC;
    tp->e_smem = e_smem;
    tp->sEbS = e_smem ? odd_up(KB * ct.Tab) : 0;
    tp->sEkS = e_smem ? odd_up(KK * ct.Tcd) : 0;
    // the fixed-point tile: E staged, register accumulators, ket primitives
    // in 16-byte pairs (rows of KS, quartets and rows an odd number of pairs apart)
    const bool fixed = split == XF_FIXED;
    const int nx = fixed ? IC : 1;  // X of a chunk's bra primitives, or of one
    const int ps_n = fixed ? (int)(sizeof(FixPrim) / 8) : PS_N;
    if (fixed && ct.L > kFixLmax) return false;
    if (fixed && !e_smem) return false;
    const int KS = (KK + 1) & ~1;
    if (fixed) {
        tp->sEkS = r_row_stride(KS * ct.Tcd, 1);
        tp->sEbS = odd_up(IC * ct.Tab);  // a chunk's bra primitives
    }
    // the paired layout of the auxiliary integrals where the split form's
    // blocked ket stage packs two ket primitives per FP32 instruction, for
    // tiles that accumulate in memory: with register accumulators live
    // through the ket stage the packed loop runs short of registers (measured
    // on (ff|dd), K = 5: 1.27 times slower than the unpacked loop; (ff|ff),
    // K = 5, accumulating in memory: 1.06 times faster)
    const bool acc_regs = TQ * ct.nab * ct.ncd <= kNT * kNACC;
    tp->r_pairs = split == XF_SPLIT && split_block_width(ct.nhb - ct.pb0) && KK >= 2 && !acc_regs ? 1 : 0;
    const int KKr = tp->r_pairs ? (KK + 1) & ~1 : KK;
    size_t r_need = (size_t)(fixed ? r_row_stride(TQ * r_row_stride(IC * KS, 1), 1)
                                   : r_row_stride(TQ * IC * KKr, tp->r_pairs)) * ct.nhl;
    size_t hA = 0, hB = 0;
    if (ct.hrr || ct.sph) {
        // the recursion (and solid-harmonic) buffers alias every staging
        // region before the tables (E, pair scalars, R, X are dead in the
        // epilogue); grow R if short
        if (ct.hrr) hrr_buffers(ct, TQ, &hA, &hB);
        if (ct.sph) {  // each solid-harmonic step reads one buffer and writes the other
            const size_t nf = (size_t)TQ * ct.nab_f * ct.ncd_f;
            hA = std::max(hA, nf);
            hB = std::max(hB, nf);
        }
        const size_t staged = even((size_t)TQ * tp->sEbS) + even((size_t)TQ * tp->sEkS) +
                              even((size_t)TQ * KB * ps_n) + even((size_t)TQ * KK * ps_n) + even(r_need) +
                              even((size_t)TQ * ct.nhb * ct.ncd * nx);
        const size_t need = even(hA) + even(hB);
        if (staged < need) r_need += need - staged;
    }
    {
        // the Coulomb digestion of plans stages the tile's values there too
        const size_t staged = even((size_t)TQ * tp->sEbS) + even((size_t)TQ * tp->sEkS) +
                              even((size_t)TQ * KB * ps_n) + even((size_t)TQ * KK * ps_n) + even(r_need) +
                              even((size_t)TQ * ct.nhb * ct.ncd * nx);
        const size_t need = even((size_t)TQ * ct.nab * ct.ncd);
        if ((fixed || TQ * ct.nab * ct.ncd <= kNT * kNACC) && staged < need) r_need += need - staged;
    }
    tp->o_Eb = take((size_t)TQ * tp->sEbS);
    tp->o_Ek = take((size_t)TQ * tp->sEkS);
    tp->o_Pb = take((size_t)TQ * KB * ps_n);
    tp->o_Pk = take((size_t)TQ * KK * ps_n);
    tp->o_R = take(r_need);
    tp->o_X = take((size_t)TQ * ct.nhb * ct.ncd * nx);
    tp->o_hB = (int)even(hA);
    const size_t tab_bytes =
        fixed ? fix_table_bytes(ct) : 4 * (ct.nab + ct.ncd + 2) + 2 * (ct.Tab + ct.Tcd + ct.nhb * ct.nhk);
    tp->o_tab = take((tab_bytes + 7) / 8);
    tp->o_q = take((size_t)TQ * 2);
    tp->o_geo = take(ct.hrr ? (size_t)TQ * 6 : 0);
    tp->o_dj = take((size_t)TQ + ct.nab_f);  // also the quartet indices of a sorted batch
    // one-quartet tiles only, and only where it fits: a tile without it
    // reads the bra E products from global memory
    tp->o_Ei = -1;
    if (!e_smem && TQ == 1 && (off + even(ct.Tab)) * 8 <= (size_t)max_smem_optin()) tp->o_Ei = take(ct.Tab);
    tp->o_Er = -1;  // added for the split form by add_e_ring
    tp->o_fx = fixed ? take((fix_scratch_ints(TQ, KB, ct.nab, ct.ncd) + 1) / 2) : -1;
    tp->o_acc = fixed ? take((size_t)TQ * ct.nab * ct.ncd) : -1;
    tp->bytes = off * 8;
    tp->nt = fixed ? nt : kNT;
    tp->acc_regs = (fixed || TQ * ct.nab * ct.ncd <= kNT * kNACC) ? 1 : 0;
    if (ct.hrr && !tp->acc_regs) return false;
    return tp->bytes + (fixed ? 64 : 0) <= (size_t)max_smem_optin();  // (and a few words of static shared memory)
}

// Split form: when the blocked ket stage reads its ket E rows from global
// memory, give every warp (tp->nt / 32 of them) a ring of kRingRows rows (KK
// float pairs each) at the end of the tile's shared memory, if it fits.
static void add_e_ring(const ClassTables& ct, int KK, TilePlan* tp)
{
    tp->o_Er = -1;
    if (tp->e_smem || !split_block_width(ct.nhb - ct.pb0)) return;
    const size_t off = (tp->bytes / 8 + 1) & ~size_t(1), nd = (size_t)(tp->nt / 32) * kRingRows * KK;
    if ((off + nd) * 8 > (size_t)max_smem_optin()) return;
    tp->o_Er = (int)off;
    tp->bytes = (off + nd) * 8;
}

// Tile shape of the fixed-point tile where none has been timed: the least
// modelled time.  A stage's round (one item per thread) costs its unit, in
// clocks of an SM whose 512 threads (registers allow no more) all run it, shared
// by the threads that do, but at least a third of it (one warp's latency); chunks
// and tiles add their barriers and set-up.  The units are rough figures of the
// stages timed on (pp|ps) and (dd|dd).
static bool plan_fixed_tile(const ClassTables& ct, int KB, int KK, int64_t nq, TilePlan* best, double* time_out = nullptr)
{
    bool found = false;
    double best_time = 0.0;
    const double unit_a_low[5] = {200, 350, 550, 800, 1300};
    const double unit_a = ct.L <= 4 ? unit_a_low[ct.L] : 12.0 * ct.nhl * ct.L;
    const double unit_b = 150 + 24.0 * KK * ct.Tcd / ct.ncd, unit_c = 150;
    for (int nt : {kNTSlim, kNT, kNTWide}) {
        for (int TQ = 1; TQ <= 128 && (TQ == 1 || TQ < 2 * nq); TQ *= 2)
            for (int IC : {KB, (KB + 1) / 2, (KB + 2) / 3, 1}) {
                TilePlan tp;
                if (!tile_layout(ct, KB, KK, TQ, IC, 1, &tp, XF_FIXED, nt)) continue;
                const int64_t tiles = (nq + TQ - 1) / TQ;
                int64_t per_sm = std::min<int64_t>(kNTWide / nt, (int64_t)smem_per_sm() / (int64_t)(tp.bytes + 1088));
                if (per_sm < 1) continue;
                per_sm = std::min<int64_t>(per_sm, (tiles + sm_count() - 1) / sm_count());
                const double share = std::max(1.0 / 3, (double)(per_sm * nt) / kNTWide);
                auto rounds = [&](double items) { return std::ceil(items / nt); };
                const int chunks = (KB + IC - 1) / IC;
                const double t_chunk =
                    800 + share * (rounds((double)TQ * IC * KK) * unit_a +
                                   rounds(0.25 * TQ * IC * (ct.nhb - ct.pb0) * ct.ncd) * unit_b +
                                   rounds(0.5 * TQ * ct.nab * ct.ncd) * (unit_c + 10.0 * IC * ct.Tab / ct.nab));
                const double time = std::ceil((double)tiles / (double)(per_sm * sm_count())) *
                                    (4000 + share * rounds((double)TQ * KB * KK) * 60 + chunks * t_chunk);
                if (!found || time < best_time) {
                    best_time = time;
                    *best = tp;
                    found = true;
                }
            }
    }
    if (found && time_out) *time_out = best_time;
    return found;
}

bool plan_tiles(const ClassTables& ct, int KB, int KK, int64_t nq, TilePlan* best, size_t max_bytes, int split)
{
    if (split == XF_FIXED) return plan_fixed_tile(ct, KB, KK, nq, best);
    bool found = false;
    double best_score = -1.0;
    for (int e_smem = 1; e_smem >= 0; --e_smem) {
        for (int TQ = 128; TQ >= 1; TQ /= 2) {
            if (TQ > 1 && TQ * ct.nab * ct.ncd > kNT * kNACC) continue;  // prefer register accumulation
            if (TQ > 1 && (int64_t)TQ > 2 * nq) continue;
            for (int IC = KB; IC >= 1; IC = (IC + 1) / 2 - (IC == 1)) {
                TilePlan tp;
                if (!tile_layout(ct, KB, KK, TQ, IC, e_smem, &tp, split) || (max_bytes && tp.bytes > max_bytes)) {
                    if (IC == 1) break;
                    continue;
                }
                // score: utilisation of the stage-A items, the ket-stage items
                // and the bra-stage items (fraction of kNT-wide rounds used)
                auto util = [](int64_t n) {
                    const int64_t rounds = (n + kNT - 1) / kNT;
                    return rounds ? (double)n / (double)(rounds * kNT) : 0.0;
                };
                const int64_t nA = (int64_t)TQ * IC * KK;
                const double wA = (double)ct.nhl * 2.0 + 40.0;
                const double wB = (double)ct.nhb * ct.Tcd * KK;
                const double wC = (double)ct.ncd * ct.Tab;
                const double score = (wA + wB + wC) /
                                     (wA / util(nA) + wB / util((int64_t)TQ * ct.nhb * ct.ncd) +
                                      wC / util((int64_t)TQ * ct.nab * ct.ncd)) +
                                     1e-3 * TQ * IC + (e_smem ? 0.05 : 0.0);
                if (score > best_score) {
                    best_score = score;
                    *best = tp;
                    found = true;
                }
                if (IC == 1) break;
            }
        }
        if (found) break;
    }
    return found;
}

// FP64 tile of a batch too small to be timed: plan_tiles fills one CTA's stages,
// which leaves a small batch's quartets on a few SMs (1000 (pp|pp), K = 1: 32 CTAs).
// Here the least modelled time of the whole batch, in clocks: every stage's
// warps on the busiest SM over its four FP64 pipes, 68 clocks an instruction, so
// a tile of few quartets costs nothing until four warps queue; and the latency of
// staging and barriers, once per wave of resident tiles.  *best (the shape of
// plan_tiles) stays unless another is modelled 10 % faster.  Measured per call, us:
// (pp|pp) K = 1, 50 / 1000 / 12000 quartets 140 / 145 / 211 -> 63 / 66 / 152; (ps|ps)
// K = 3, 50 / 1000 quartets 208 / 233 -> 77 / 89; (dd|dd) K = 3, 50 / 1000 quartets
// 1305 / 2377 -> 379 / 2140 (with the faster pair tables and checking pass).
// Returns the modelled time of *best.
static double plan_small_tile(const ClassTables& ct, int KB, int KK, int64_t nq, TilePlan* best)
{
    auto warps = [](double items) { return std::ceil(items / 32); };
    const int L = ct.L;
    const double base = 45.0 + 3.0 * L, steps = (L + 1.0) * (L + 2) * (L + 3) * (L + 4) / 24;
    auto model = [&](const TilePlan& tp) {
        const int64_t tiles = (nq + tp.TQ - 1) / tp.TQ, per_sm = (tiles + sm_count() - 1) / sm_count();
        const int64_t res = std::min<int64_t>(per_sm, one_cta_per_sm(tp.bytes) ? 1 : 2);
        const double nA = (double)tp.TQ * tp.IC * KK;  // below 64 items a warp takes each (stage A)
        auto pipe = [&](double w, double instr) { return std::ceil(res * w / 4) * instr * 68; };
        const double a = nA < 64 ? pipe(nA, base + steps / 16 + 2 * L) : pipe(warps(nA), base + steps);
        const double b = pipe(warps((double)tp.TQ * (ct.nhb - ct.pb0) * ct.ncd), (double)KK * ct.Tcd / ct.ncd);
        const double c = pipe(warps((double)tp.TQ * ct.nab * ct.ncd), (double)ct.Tab / ct.nab);
        const int chunks = (KB + tp.IC - 1) / tp.IC;
        return (double)((per_sm + res - 1) / res) * (5000 + chunks * (800 + a) + KB * (1000 + b + c));
    };
    const double planned = model(*best);
    double best_time = 0.9 * planned;
    bool other = false;
    for (int TQ = 1; TQ <= 128 && (TQ == 1 || TQ < 2 * nq); TQ *= 2) {
        if (TQ > 1 && TQ * ct.nab * ct.ncd > kNT * kNACC) break;
        for (int IC = KB, next; IC >= 1; IC = next) {  // KB, half of it, 1
            next = IC == 1 ? 0 : (IC == KB && KB > 2 ? (KB + 1) / 2 : 1);
            TilePlan tp;
            if (!tile_layout(ct, KB, KK, TQ, IC, best->e_smem, &tp, XF_FP64)) continue;
            const double t = model(tp);
            if (t < best_time) {
                best_time = t;
                *best = tp;
                other = true;
            }
        }
    }
    return other ? best_time : planned;
}

static int dev_err_to_code(int e)
{
    switch (e) {
        case DEV_OK: return ERI_OK;
        case DEV_ECLASS: return ERI_ECLASS;
        case DEV_EINDEX: return ERI_EINVAL;
        case DEV_EK: return ERI_EINVAL;
        case DEV_ETIMEOUT: return ERI_ETIMEOUT;
        default: return ERI_ECUDA;
    }
}

static size_t align_up(size_t n) { return (n + 255) & ~size_t(255); }

// Whether a batch of class cls may run the fixed-point tile: every primitive
// in its range, and neither order nor exponents' spread beyond what its
// precision allows (eri_fixed.cuh).  info: PrepassArgs::spread.
static bool fixed_eligible(eri_class_t cls, const int32_t* info)
{
    if (info[2]) return false;
    float apart;
    std::memcpy(&apart, &info[6], 4);
    const bool wide = apart >= kFixWide;
    if (cls.la + cls.lb + cls.lc + cls.ld > (wide ? kFixLmax : kFixLmaxNear)) return false;
    for (int side = 0; side < 2; ++side) {
        float r;
        std::memcpy(&r, &info[side], 4);
        const int l = side ? cls.lc + cls.ld : cls.la + cls.lb;
        if (!(0.5f * (float)l * std::log2(r) <= (wide ? kFixSpreadBitsWide : kFixSpreadBits))) return false;
    }
    return true;
}

// mu of the Hermite unit: 1.1 sqrt(2 rho) = mu 2^n, mu in [1, 2), for the
// largest reduced exponent rho of the batch (kept a little below, so that
// fix_sigma's float product does not round past the power of two).
static double fix_unit(double rho)
{
    const double s = 1.1 * std::sqrt(2.0 * rho);
    return s > 0.0 ? s / std::ldexp(1.0, std::ilogb(s)) * 1.00001 : 1.0;
}

// The fixed-point form of one side's pair tables.
static void launch_fix_pairs(const PairTables& t, const ClassTables& ct, int64_t npairs, int KS, int side, double mu,
                             int fx_f, cudaStream_t st)
{
    FixPairArgs f{};
    f.E = t.E;
    f.limbs = t.limbs;
    f.weak = t.weak;
    f.ps = reinterpret_cast<const FixPrim*>(t.ps);
    f.kp = t.kp;
    f.start = side ? ct.ket_start : ct.bra_start;
    f.herm = side ? ct.ket_q : ct.bra_p;
    f.npairs = npairs;
    f.KS = KS;
    f.T = side ? ct.Tcd : ct.Tab;
    f.ncol = side ? ct.ncd : ct.nab;
    f.ket = side;
    f.c = (float)(2.42 / (mu * mu));
    f.ex = t.ex;
    f.norm = t.norm;
    f.box = t.box;
    f.f = fx_f;
    const int64_t n = npairs * f.ncol;
    count_launch();
    fix_pairs_kernel<<<(int)std::max<int64_t>(1, std::min<int64_t>((n + 127) / 128, 16LL * sm_count())), 128, 0, st>>>(f);
}

// A batch too small to be timed takes the fixed-point tile from this many
// primitive quartets a quartet on: K = 2 (16), 16383 quartets, us, FP64 against
// fixed point: (ps|ss) 114 / 154, (pp|ps) 242 / 289, (dp|dp) 1570 / 2280.
constexpr int kFixSmallPrims = 81;
// And where its modelled time (plan_fixed_tile; rough clocks that a stage's
// threads share) and that of its pair tables' second pass (setup: terms of a
// column times primitives) stay below the FP64 tile's (plan_small_tile; clocks).
// Fitted to 23 classes of K = 3, 4 and 5 with 2000 to 16383 quartets: what it lets in
// measured 0.3 to 1.03 times the FP64 call, e.g. (pp|pp) K = 3, 8000 quartets 876 us / 530,
// (dp|pp) K = 3, 4000, 895 / 772; what it keeps out up to 1.6: (dd|ss) K = 3, 2000, 314 / 507,
// (ps|ss) K = 3, 2000, 106 / 145, (ff|ss) K = 4, 4000, 3840 / 5258.
static bool fix_small_faster(int L, double fix_time, double setup, double fp64_time)
{
    return (L >= 5 ? 14.0 : 11.0) * fix_time + 75e3 + 1800.0 * setup < fp64_time;
}

// Prepass + pair tables shared by the forward and adjoint entry points.
// On success fills the pair tables and the largest K on each centre.
// Largest product of bra and ket recursion risks for which the recursion
// forms are offered (see prepass_kernel): 1.1e-16 x 900 x O(10) ~ 1e-12.
constexpr double kRecursionRisk = 900.0;

// Forms eri_batch may use (eri_set_forms): bit o allows form o.
static std::atomic<int> g_form_mask{0xF};

// When the calling thread's batches take the fixed-point tile (eri_set_fixed).
static thread_local int g_fixed_mode = ERI_FIXED_RULE;
// Batches of at least this many quartets time their tile shapes and forms.
constexpr int64_t kTuneMinQuartets = 16384;

// Forms chosen by timing, per (device, class, K_bra, K_ket, precision).
static std::map<std::tuple<int, int, int, int, int, int, int, int, int>, int> g_forms;
static std::mutex g_forms_mu;

static std::tuple<int, int, int, int, int, int, int, int, int> form_key(eri_class_t cls, int KB, int KK, int split,
                                                                        int kind)
{
    int dev = 0;
    cudaGetDevice(&dev);
    return std::make_tuple(dev, cls.la, cls.lb, cls.lc, cls.ld, KB, KK, split, kind);
}

static int lookup_form(eri_class_t cls, int KB, int KK, int split, int kind)
{
    std::lock_guard<std::mutex> lk(g_forms_mu);
    auto it = g_forms.find(form_key(cls, KB, KK, split, kind));
    return it == g_forms.end() ? -1 : it->second;
}

// Whether the FP64 tile was timed faster than the fixed-point one, by the same key
// (arithmetic XF_FIXED); nothing where they were not compared.
static std::map<std::tuple<int, int, int, int, int, int, int, int, int>, bool> g_fp64_faster;

static int lookup_fp64_faster(eri_class_t cls, int KB, int KK, int kind)  // 1, 0, or -1: not compared
{
    std::lock_guard<std::mutex> lk(g_forms_mu);
    auto it = g_fp64_faster.find(form_key(cls, KB, KK, XF_FIXED, kind));
    return it == g_fp64_faster.end() ? -1 : (int)it->second;
}

static void remember_fp64_faster(eri_class_t cls, int KB, int KK, int kind, bool faster)
{
    std::lock_guard<std::mutex> lk(g_forms_mu);
    g_fp64_faster[form_key(cls, KB, KK, XF_FIXED, kind)] = faster;
}

void remember_form(eri_class_t cls, int KB, int KK, int split, int kind, int form)
{
    std::lock_guard<std::mutex> lk(g_forms_mu);
    g_forms[form_key(cls, KB, KK, split, kind)] = form;
}

int prepare_batch(eri_class_t cls, const eri_basis_t* basis, const int32_t* bra, int64_t nbra, const int32_t* ket,
                  int64_t nket, const int64_t* quartets, int64_t nq, int ldelta, cudaStream_t st,
                  const ClassTables** ct_out, PairTables* pb, PairTables* pk, int* KB, int* KK, int kmax[4],
                  int allow_swap, FormChoice* fc, int split, int kind, int* mixed)
{
    int err = ERI_OK;
    // kind 2: the caller's bra side (x, unit) is a solid harmonic
    // kind 3: solid-harmonic output on every centre (plain or recursion form)
    auto tables = [&](int la, int lb, int lc, int ld, int x_first, int hrr) {
        if (kind == 2) return get_class_tables_pure(la, lb, lc, ld, x_first ? 1 : 2, st, &err);
        if (kind == 3) return get_class_tables_sph(la, lb, lc, ld, hrr, st, &err);
        return hrr ? get_class_tables_hrr(la, lb, lc, ld, st, &err) : get_class_tables(la, lb, lc, ld, st, &err);
    };
    const ClassTables* ct = tables(cls.la, cls.lb, cls.lc, cls.ld, 1, 0);
    if (!ct) return err;
    *ct_out = ct;
    const int forced = fc ? fc->form : -1;
    if (fc) {
        fc->form = 0;
        fc->alt = -1;
        fc->cached = 0;
        fc->fixed = 0;
    }
    int* status = device_status();
    if (!status) return ERI_ECUDA;
    int32_t* hinfo = host_pinned_i32(16);
    if (!hinfo) return ERI_ENOMEM;
    // info lives in the status block (slots 8..16), separate from the error word:
    // [0..6] as PrepassArgs::info, [7..8] the smallest pair counts per side,
    // [9..15] PrepassArgs::spread
    int* dinfo = status + 8;
    // (one call: a small batch is bound by its launches, about 2 us each)
    if (cudaMemsetAsync(dinfo, 0, 16 * sizeof(int), st) != cudaSuccess) return ERI_ECUDA;
    // Where the fixed-point tile can be the faster one (GB300, ms, FP64 against fixed
    // point): contracted 4-centre classes above (ss|ss).  Not (ss|ss), 4e5 of mixed
    // degrees 5.12 / 5.37, whose tiles hold few primitive quartets; not uncontracted
    // batches, where set-up and barriers outweigh the products: (pp|ps) 3e5 0.43 / 0.49;
    // not 3-centre ones, (f|dp) 1e5 4.90 / 6.20; nor the smallest, which are not asked
    // for their spread either, nor is a basis without contracted shells (it adds 7 us
    // to the checking pass: (ps|ss) K = 1, 4000 quartets 62 / 69 us a call).
    const int64_t nqq = quartets ? nq : nbra * nket;
    const int L = cls.la + cls.lb + cls.lc + cls.ld;
    const bool by_rule = g_fixed_mode == ERI_FIXED_RULE;
    const bool try_fixed = fc && !fc->no_fixed && g_fixed_mode != ERI_FIXED_NEVER && !split && ldelta == 0 &&
                           (kind == 0 || kind == 3) && L > 0 && L <= kFixLmax &&
                           (!by_rule || (nqq >= 2000 && basis->nprim > basis->nshell));
    PrepassArgs pa{basis->shell_l, basis->shell_K, basis->nshell, bra, nbra, ket, nket, quartets,
                   quartets ? nq : (int64_t)0,
                   {cls.la, cls.lb, cls.lc, cls.ld}, (kind == 1 || kind == 2) ? 1 : 0, dinfo,
                   allow_swap > 1 ? 1 : 0, basis->centres, basis->shell_atom, basis->shell_off, basis->exps,
                   dinfo + 7, try_fixed ? dinfo + 9 : nullptr, basis->coefs};
    const int64_t n = std::max(std::max(nbra, nket), quartets ? nq : (int64_t)0);
    const int grid = (int)std::min<int64_t>((n + 255) / 256, 4 * sm_count());
    {
        ProfScope ps(PROF_PREPASS, st);
        prepass_kernel<<<std::max(grid, 1), 256, 0, st>>>(pa);
    }
    if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    // the info goes to the pinned host buffer through its mapped device
    // address, written by a kernel: a device-to-host copy would queue behind
    // any large read-back the caller has put on that copy engine
    int32_t* hmapped = nullptr;
    if (cudaHostGetDevicePointer((void**)&hmapped, hinfo, 0) == cudaSuccess && hmapped) {
        count_launch();
        info_to_host_kernel<<<1, 32, 0, st>>>(dinfo, 16, hmapped);
        if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    } else {
        cudaGetLastError();
        if (cudaMemcpyAsync(hinfo, dinfo, 16 * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return ERI_ECUDA;
    }
    if (cudaStreamSynchronize(st) != cudaSuccess) return ERI_ECUDA;
    if (hinfo[4] != 0) return dev_err_to_code(hinfo[4]);
    for (int c = 0; c < 4; ++c) kmax[c] = hinfo[c];
    *KB = kmax[0] * kmax[1];
    *KK = kmax[2] * kmax[3];
    if (mixed) *mixed = (INT_MAX - hinfo[7] < *KB || INT_MAX - hinfo[8] < *KK) ? 1 : 0;
    bool fix_ok = try_fixed && fixed_eligible(cls, hinfo + 9);
    if (fix_ok && by_rule)
        fix_ok = (int64_t)*KB * *KK >= (nqq < kTuneMinQuartets ? kFixSmallPrims : 4) && nqq * *KB * *KK >= 150000 &&
                 lookup_fp64_faster(cls, *KB, *KK, kind) != 1;
    if (allow_swap) {
        // Four forms: which side is transformed first (Section 3.2.2
        // transforms the ket first, assuming it has the lower l) and whether
        // the transforms run on (e0) functions followed by horizontal
        // recursions in the contracted basis.  The FP64-work model picks one
        // unless a form is forced or an earlier timing chose one.
        const ClassTables* opt[4] = {ct, tables(cls.lc, cls.ld, cls.la, cls.lb, 0, 0), nullptr, nullptr};
        if (!opt[1]) return err;
        // The recursion forms must keep their magnified rounding, about
        // 1.1e-16 x (bra risk) x (ket risk) x the integrals' scale, well
        // inside the 1e-11 absolute bar: they are offered only while the
        // product of the largest pair risks stays below kRecursionRisk.
        float rb, rk;
        std::memcpy(&rb, &hinfo[5], 4);
        std::memcpy(&rk, &hinfo[6], 4);
        const bool hrr_ok = (double)rb * (double)rk <= kRecursionRisk;
        if (allow_swap > 1 && (kind == 0 || kind == 3) && hrr_ok) {
            opt[2] = tables(cls.la, cls.lb, cls.lc, cls.ld, 1, 1);
            opt[3] = tables(cls.lc, cls.ld, cls.la, cls.lb, 0, 1);
            if (!opt[2] || !opt[3]) return err;
        }
        double cost[4];
        auto set_costs = [&]() {
            for (int o = 0; o < 4; ++o) {
                cost[o] = -1.0;  // infeasible
                const ClassTables* c = opt[o];
                if (!c) continue;
                const double kb = (o & 1) ? *KK : *KB, kk = (o & 1) ? *KB : *KK;
                if (c->hrr) {
                    // (f0|e0) must fit the register accumulators and the
                    // recursion buffers of the epilogue the shared memory
                    TilePlan tp;
                    if (c->nab * c->ncd > kNT * kNACC || !plan_tiles(*c, (int)kb, (int)kk, nqq, &tp)) continue;
                }
                // a recursion step is an FP64 operation, which costs several
                // products of the fixed-point transforms (where the smallest tile fits)
                TilePlan least;
                const bool fits = fix_ok && tile_layout(*c, (int)kb, (int)kk, 1, 1, 1, &least, XF_FIXED, kNTSlim);
                const double step = fits ? 6.0 : 1.0;
                cost[o] = kb * kk * ((c->nhb - c->pb0) * c->Tcd + 0.5 * c->nhl) + kb * c->ncd * c->Tab +
                          (c->hrr ? step * (c->nab * c->nks + c->ncd_f * c->nbs) : 0);
            }
            // the caller's form mask (eri_set_forms), unless it leaves no feasible form
            const int mask = g_form_mask.load();
            bool any = false;
            for (int o = 0; o < 4; ++o) any |= cost[o] >= 0 && (mask >> o & 1);
            if (any)
                for (int o = 0; o < 4; ++o)
                    if (!(mask >> o & 1)) cost[o] = -1.0;
        };
        auto cheapest = [&](int lo, int hi) {
            int b = -1;
            for (int o = lo; o < hi; ++o)
                if (cost[o] >= 0 && (b < 0 || cost[o] < cost[b])) b = o;
            return b;
        };
        int best = -1, cached = 0;
        auto choose = [&]() {  // false: the caller's form is not feasible
            set_costs();
            best = forced;
            if (forced >= 0) return forced <= 3 && cost[forced] >= 0;
            best = lookup_form(cls, *KB, *KK, fix_ok ? XF_FIXED : split, kind);
            cached = best >= 0 && cost[best] >= 0;
            if (!cached) best = cheapest(0, 4);
            return true;
        };
        if (!choose()) return ERI_EINVAL;
        if (fix_ok && by_rule && nqq < kTuneMinQuartets && forced < 0) {
            // a batch too small to be timed: the models of both tiles
            auto degree = [&](int o, bool ket) { return ((o & 1) != 0) == ket ? *KB : *KK; };
            const ClassTables& cf = *opt[best];
            const bool fix_plain = best < 2;
            double fix_time = 0.0, fp64_time = 1e300;
            TilePlan tp;
            if (plan_fixed_tile(cf, degree(best, 0), degree(best, 1), nqq, &tp, &fix_time)) {
                const double setup = (double)degree(best, 0) * cf.Tab / cf.nab + (double)degree(best, 1) * cf.Tcd / cf.ncd;
                fix_ok = false;
                if (!choose()) return ERI_EINVAL;
                const ClassTables& c64 = *opt[best];
                if (plan_tiles(c64, degree(best, 0), degree(best, 1), nqq, &tp))
                    fp64_time = plan_small_tile(c64, degree(best, 0), degree(best, 1), nqq, &tp);
                // (an FP64 recursion form, of the larger error, by 10 % against a plain one)
                if (fix_plain && best >= 2) fp64_time *= 1.1;
                fix_ok = fix_small_faster(L, fix_time, setup, fp64_time);
                if (fix_ok && !choose()) return ERI_EINVAL;
            }
        }
        if (fc) fc->cached = cached;
        if (fc) {
            fc->form = best;
            fc->alt = best >= 2 ? cheapest(0, 2) : cheapest(2, 4);
        }
        ct = opt[best];
        *ct_out = ct;
        if (best & 1) {
            cls = eri_class_t{cls.lc, cls.ld, cls.la, cls.lb};
            std::swap(bra, ket);
            std::swap(nbra, nket);
            std::swap(*KB, *KK);
            std::swap(kmax[0], kmax[2]);
            std::swap(kmax[1], kmax[3]);
        }
    }
    // the fixed-point tile where its precision and its shared memory allow
    TilePlan fix_tile;
    bool fixed = fix_ok && plan_tiles(*ct, *KB, *KK, nqq, &fix_tile, 0, XF_FIXED);
    if (fixed && !get_fix_boys_table(ct->L, st, &err)) {
        if (err != ERI_ENOMEM) return err;
        fixed = false;  // the FP64 tile needs less memory
        err = ERI_OK;
    }
    int fx_f = 0;
    double mu = 1.0;
    if (fixed) {  // |coordinate| 2^fx_f < 2^60
        float far;
        std::memcpy(&far, &hinfo[12], 4);
        fx_f = 60 - std::max(-10, far > 0.f ? std::ilogb(far) + 1 : -10);
        float zb, zk;
        std::memcpy(&zb, &hinfo[13], 4);
        std::memcpy(&zk, &hinfo[14], 4);
        mu = fix_unit((double)zb * zk / ((double)zb + zk));
    }
    // workspace: pair tables of both sides.
    // ldelta 1: the raised tables of the kernel bra only (the adjoint launch
    // for one side's channels); 2: of both sides, with the E products of
    // both (the adjoint launch for every channel)
    const int grad = ldelta > 0, grad_both = ldelta > 1;
    const int eaxb = (cls.la + 3) * (cls.lb + 3) * (cls.la + cls.lb + 5);
    const int eaxk = (cls.lc + 3) * (cls.ld + 3) * (cls.lc + cls.ld + 5);
    const size_t nb_E = align_up(sizeof(double) * nbra * *KB * ct->Tab);
    const size_t nk_E = align_up(sizeof(double) * nket * *KK * ct->Tcd);
    const size_t nb_k = align_up(sizeof(int32_t) * nbra), nk_k = align_up(sizeof(int32_t) * nket);
    const size_t nb_ax = grad ? align_up(sizeof(double) * nbra * *KB * 3 * eaxb) : 0;
    const size_t nk_ax = grad_both ? align_up(sizeof(double) * nket * *KK * 3 * eaxk) : 0;
    const size_t nb_z = grad ? align_up(sizeof(double) * nbra * *KB * 2) : 0;
    const size_t nk_z = grad_both ? align_up(sizeof(double) * nket * *KK * 2) : 0;
    const size_t n_grad = nb_ax + nk_ax + nb_z + nk_z;
    size_t nb_ps, nk_ps, nb_x, nk_x, nk_n, nb_n, nb_b, nk_b, nb_l, nb_w;
    auto total = [&]() {
        const size_t ps_n = fixed ? sizeof(FixPrim) / 8 : PS_N, on = fixed;
        nb_ps = align_up(sizeof(double) * nbra * *KB * ps_n);
        nk_ps = align_up(sizeof(double) * nket * *KK * ps_n);
        nb_x = on * align_up(sizeof(int32_t) * nbra * ct->nab);
        nk_x = on * align_up(sizeof(int32_t) * nket * ct->ncd);
        nk_n = on * align_up(sizeof(float) * 8 * nket * ct->ncd);
        nb_n = on * align_up(sizeof(float) * 8 * nbra * ct->nab);
        nb_b = on * align_up(sizeof(float) * 6 * nbra);
        nk_b = on * align_up(sizeof(float) * 6 * nket);
        nb_l = on * nb_E;
        nb_w = on * align_up(sizeof(int32_t) * nbra);
        return nb_ps + nb_E + nk_ps + nk_E + nb_k + nk_k + n_grad + nb_x + nk_x + nk_n + nb_n + nb_l + nb_w + nb_b + nk_b;
    };
    uint8_t* ws = (uint8_t*)workspace(total(), &err);
    if (!ws && fixed && err == ERI_ENOMEM) {
        fixed = false;  // no limbs, norms and boxes: what the FP64 tile needs
        err = ERI_OK;
        ws = (uint8_t*)workspace(total(), &err);
    }
    if (!ws) return err;
    if (fc) {
        fc->key = fix_ok ? XF_FIXED : split;
        fc->fixed = fixed;
        fc->fx_f = fx_f;
        fc->mu = mu;
    }
    {
        uint8_t* g0 = ws + nb_ps + nb_E + nk_ps + nk_E + nb_k + nk_k;
        pb->ax = grad ? (double*)g0 : nullptr;
        pk->ax = grad_both ? (double*)(g0 + nb_ax) : nullptr;
        pb->zz = grad ? (double*)(g0 + nb_ax + nk_ax) : nullptr;
        pk->zz = grad_both ? (double*)(g0 + nb_ax + nk_ax + nb_z) : nullptr;
        pb->eax = eaxb;
        pk->eax = eaxk;
        pb->ex = fixed ? (int32_t*)(g0 + n_grad) : nullptr;
        pk->ex = fixed ? (int32_t*)(g0 + n_grad + nb_x) : nullptr;
        pk->norm = fixed ? (float*)(g0 + n_grad + nb_x + nk_x) : nullptr;
        uint8_t* l0 = g0 + n_grad + nb_x + nk_x + nk_n;
        pb->norm = fixed ? (float*)l0 : nullptr;
        pb->limbs = fixed ? (int2*)(l0 + nb_n) : nullptr;
        pb->weak = fixed ? (int32_t*)(l0 + nb_n + nb_l) : nullptr;
        pk->limbs = nullptr;
        pk->weak = nullptr;
        pb->box = fixed ? (float*)(l0 + nb_n + nb_l + nb_w) : nullptr;
        pk->box = fixed ? (float*)(l0 + nb_n + nb_l + nb_w + nb_b) : nullptr;
    }
    pb->ps = (double*)ws;
    pb->E = (double*)(ws + nb_ps);
    pk->ps = (double*)(ws + nb_ps + nb_E);
    pk->E = (double*)(ws + nb_ps + nb_E + nk_ps);
    pb->kp = (int32_t*)(ws + nb_ps + nb_E + nk_ps + nk_E);
    pk->kp = (int32_t*)(ws + nb_ps + nb_E + nk_ps + nk_E + nb_k);
    for (int side = 0; side < 2; ++side) {
        PairArgs p{};
        p.centres = basis->centres;
        p.shell_atom = basis->shell_atom;
        p.shell_K = basis->shell_K;
        p.shell_off = basis->shell_off;
        p.exps = basis->exps;
        p.coefs = basis->coefs;
        p.pairs = side ? ket : bra;
        p.npairs = side ? nket : nbra;
        p.l1 = side ? cls.lc : cls.la;
        p.l2 = side ? cls.ld : cls.lb;
        p.KS = side ? *KK : *KB;
        p.T = side ? ct->Tcd : ct->Tab;
        p.fac = side ? ct->ket_fac : ct->bra_fac;
        p.ket = side;
        PairTables& t = side ? *pk : *pb;
        p.ps = t.ps;
        p.E = t.E;
        p.kprim = t.kp;
        p.ax = t.ax;
        p.eax = t.eax;
        p.zz = t.zz;
        p.split = split;
        p.fixed = fixed;
        p.fx_f = fx_f;
        p.mu = mu;
        p.weak = t.weak;
        p.hrr = ct->hrr;
        p.scale = side ? ct->ket_scale : ct->bra_scale;
        const int64_t tot = p.npairs * p.KS;
        const int g = (int)std::min<int64_t>((tot + 127) / 128, 8 * sm_count());
        ProfScope ps(PROF_PAIR, st);
        if (grad_both) {  // the E products as well as the raised tables (both write the same pair scalars)
            PairArgs pe = p;
            pe.ax = nullptr;
            pe.zz = nullptr;
            launch_pair(pe, std::max(g, 1), st);
        }
        launch_pair(p, std::max(g, 1), st);
        if (fixed) launch_fix_pairs(t, *ct, p.npairs, p.KS, side, mu, fx_f, st);
        if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    }
    return ERI_OK;
}

static int check_basis(const eri_basis_t* b)
{
    if (!b || !b->centres || !b->shell_atom || !b->shell_l || !b->shell_K || !b->shell_off || !b->exps || !b->coefs)
        return ERI_EINVAL;
    if (b->natom < 0 || b->nshell < 0 || b->nprim < 0) return ERI_EINVAL;
    return ERI_OK;
}

static int check_class(eri_class_t c)
{
    const int l[4] = {c.la, c.lb, c.lc, c.ld};
    for (int i = 0; i < 4; ++i)
        if (l[i] < 0 || l[i] > kLmax) return ERI_EINVAL;
    return ERI_OK;
}

int check_batch_args(eri_class_t cls, const eri_basis_t* basis, const int32_t* bra, int64_t nbra, const int32_t* ket,
                     int64_t nket, const int64_t* quartets, int64_t nq, int64_t len)
{
    if (check_class(cls) != ERI_OK || check_basis(basis) != ERI_OK) return ERI_EINVAL;
    if (nbra < 0 || nket < 0 || (quartets && nq < 0)) return ERI_EINVAL;
    if ((nbra > 0 && !bra) || (nket > 0 && !ket)) return ERI_EINVAL;
    if (nbra > INT32_MAX || nket > INT32_MAX) return ERI_EINVAL;
    const int64_t nqq = quartets ? nq : nbra * nket;
    const int64_t nab = host_nc(cls.la) * host_nc(cls.lb), ncd = host_nc(cls.lc) * host_nc(cls.ld);
    if (len < nqq * nab * ncd) return ERI_EINVAL;
    return ERI_OK;
}

// Autotuner of eri_batch: on the first large batch of a (class, form, K_bra,
// K_ket, precision) signature, time every feasible tile shape (TQ in 1..128 with
// register accumulation, IC in {K_bra, K_bra/2, 1}, E staged when it fits)
// on the batch's leading quartets (about four waves of tiles, at least
// kTuneQuartets) and remember the fastest with its time per quartet
// (eri_batch compares forms by it).  The trial launches write (part
// of) `out`; the real launch overwrites it.
constexpr int64_t kTuneQuartets = 8192;
static std::map<std::tuple<int, int, int, int, int, int, int, int, int, int>, std::pair<TilePlan, float>> g_tuned;
static std::mutex g_tuned_mu;

static bool tuned_tile(const FwdArgs& base, int split, cudaStream_t st, TilePlan* best, float* best_ms_out)
{
    int dev = 0;
    cudaGetDevice(&dev);
    const ClassTables& ct = base.ct;
    const auto key = std::make_tuple(dev, ct.la, ct.lb, ct.lc, ct.ld, ct.hrr, ct.pure, base.KB, base.KK, split);
    {
        std::lock_guard<std::mutex> lk(g_tuned_mu);
        auto it = g_tuned.find(key);
        if (it != g_tuned.end()) {
            *best = it->second.first;
            *best_ms_out = it->second.second;
            return true;
        }
    }
    std::vector<TilePlan> cands;
    for (int TQ = 1; TQ <= 128; TQ *= 2) {
        if (split == XF_FIXED) {
            for (int IC : {base.KB, (base.KB + 1) / 2, (base.KB + 2) / 3, 1})
                for (int nt : {kNTSlim, kNT, kNTWide}) {
                    TilePlan tp;
                    if (!tile_layout(ct, base.KB, base.KK, TQ, IC, 1, &tp, split, nt)) continue;
                    // at least half as many CTAs per SM as the registers hold
                    if ((kNTWide / nt) * (tp.bytes + 1088) > 2 * (size_t)smem_per_sm()) continue;
                    bool dup = false;
                    for (auto& c : cands) dup |= c.TQ == TQ && c.IC == IC && c.nt == nt;
                    // a chunk with too few or far too many items for the CTA is not worth timing
                    const int items = TQ * IC * base.KK;
                    if (!dup && (items * 8 >= nt || TQ == 1) && items <= 16 * nt) cands.push_back(tp);
                }
            continue;
        }
        if (TQ * ct.nab * ct.ncd > kNT * kNACC) break;
        for (int IC : {base.KB, (base.KB + 1) / 2, 1}) {
            for (int es = 1; es >= 0; --es) {
                TilePlan tp;
                if (tile_layout(ct, base.KB, base.KK, TQ, IC, es, &tp, split) && tp.acc_regs) {
                    bool dup = false;
                    for (auto& c : cands) dup |= (c.TQ == TQ && c.IC == IC && c.e_smem == es);
                    if (dup) break;
                    // a tile that leaves room for one CTA per SM is also tried
                    // with 512 threads (twice the warps in the same memory)
                    const bool wide = one_cta_per_sm(tp.bytes);
                    TilePlan tw = tp;
                    tw.nt = kNTWide;
                    if (split == XF_SPLIT) {
                        add_e_ring(ct, base.KK, &tp);
                        add_e_ring(ct, base.KK, &tw);
                    }
                    cands.push_back(tp);
                    if (wide && tw.bytes <= (size_t)max_smem_optin()) cands.push_back(tw);
                    break;
                }
            }
        }
    }
    if (cands.empty()) return false;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best_ms = 3e38f;  // per quartet
    bool ok = false;
    // per quartet, over about `waves` waves of tiles (steady state) and at least
    // kTuneQuartets quartets; 3e38: did not run
    auto time_tile = [&](const TilePlan& tp, int waves) {
        FwdArgs a = base;
        set_tile(a, tp);
        void (*kern)(FwdArgs) = fwd_kern(split, tp.nt);
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tp.bytes) != cudaSuccess) {
            cudaGetLastError();
            return 3e38f;
        }
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, tp.nt, tp.bytes);
        const int64_t slots = (int64_t)std::max(per_sm, 1) * sm_count();
        const int64_t nq = std::min(base.nq, std::max(kTuneQuartets, waves * slots * tp.TQ));
        a.ntiles = (nq + tp.TQ - 1) / tp.TQ;
        const int64_t grid = std::min<int64_t>(a.ntiles, slots);
        // one warm-up launch, then the fastest of three timed ones: candidates
        // often lie within a few per cent of each other
        float ms = 3e38f;
        bool timed = true;
        count_launch();
        kern<<<(int)grid, tp.nt, tp.bytes, st>>>(a);
        for (int rep = 0; rep < 3 && timed; ++rep) {
            float t = 0.f;
            cudaEventRecord(e0, st);
            count_launch();
            kern<<<(int)grid, tp.nt, tp.bytes, st>>>(a);
            cudaEventRecord(e1, st);
            timed = cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess;
            ms = std::min(ms, t);
        }
        if (!timed) {
            cudaGetLastError();
            return 3e38f;
        }
        return ms / (float)nq;
    };
    std::vector<float> first;
    for (const TilePlan& tp : cands) {
        const float ms = time_tile(tp, 4);
        first.push_back(ms);
        if (ms < best_ms) {
            best_ms = ms;
            *best = tp;
            ok = true;
        }
    }
    if (split == XF_FIXED && ok) {
        // fixed-point tiles of very different shapes tie in four waves and differ by
        // 3 % over a batch ((pp|ps) K = 3, 1e5 quartets, 2.27 ms in 256 threads of 8
        // quartets, 2.35 in 512 of 32): those within 4 % again, over 16 waves
        const float close = 1.04f * best_ms;
        best_ms = 3e38f;
        for (size_t i = 0; i < cands.size(); ++i) {
            if (first[i] > close) continue;
            const float ms = time_tile(cands[i], 16);
            if (ms < best_ms) {
                best_ms = ms;
                *best = cands[i];
            }
        }
        ok = best_ms < 3e38f;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (ok) {
        std::lock_guard<std::mutex> lk(g_tuned_mu);
        g_tuned[key] = std::make_pair(*best, best_ms);
        *best_ms_out = best_ms;
    }
    return ok;
}

// ---------------------------------------------------------------------------
// Processing order (build_order).  A batch may mix contraction degrees (a
// molecule's s shells of K = 6, 3 and 1); the tile loops run to the tile's
// largest primitive-pair counts, so the quartets are counting-sorted by the
// key kb (KK + 1) + kk, descending: histogram, offsets, scatter.  Equal keys
// keep no particular order (only the positions the tiles read and write from
// depend on it, not the values).
// ---------------------------------------------------------------------------
struct OrderArgs {
    const int64_t* quartets;  // NULL: product form
    int64_t nq, nbra;
    const int32_t* kpb;
    const int32_t* kpk;
    int KK, swap;
};

__device__ __forceinline__ int order_key(const OrderArgs& o, int64_t qq)
{
    int64_t ob, ok;
    if (o.quartets) {
        ob = o.quartets[2 * qq];
        ok = o.quartets[2 * qq + 1];
    } else {
        ob = qq % o.nbra;
        ok = qq / o.nbra;
    }
    const int64_t b = o.swap ? ok : ob, k = o.swap ? ob : ok;
    return o.kpb[b] * (o.KK + 1) + o.kpk[k];
}

__global__ void order_hist_kernel(OrderArgs o, unsigned long long* cnt)
{
    for (int64_t qq = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; qq < o.nq; qq += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[order_key(o, qq)], 1ULL);
}

// Exclusive sums of the counts from the last key down, by one block: a slice of
// kScanPer keys per thread and round, the slices' sums through warp shuffles.
// One thread walking the 1369 keys of K = 6 pairs took 0.26 ms, 5 % of a 4e5-quartet
// (ss|ss) batch, each step a memory round trip; this takes 3.3 us.
constexpr int kScanThreads = 256, kScanPer = 8;
__global__ void __launch_bounds__(kScanThreads) order_scan_kernel(int nbins, unsigned long long* cnt)
{
    __shared__ unsigned long long s_warp[kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    unsigned long long run = 0;
    for (int top = nbins; top > 0; top -= kScanThreads * kScanPer) {
        const int k0 = top - 1 - tid * kScanPer;  // this thread's keys k0, k0 - 1, ...
        unsigned long long c[kScanPer], own = 0;
#pragma unroll
        for (int j = 0; j < kScanPer; ++j) {
            c[j] = k0 - j >= 0 ? cnt[k0 - j] : 0;
            own += c[j];
        }
        unsigned long long sum = own;  // inclusive over the warp
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long v = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += v;
        }
        if (lane == 31) s_warp[tid >> 5] = sum;
        __syncthreads();
        unsigned long long before = run + sum - own, all = 0;
        for (int w = 0; w < kScanThreads / 32; ++w) {
            if (w < (tid >> 5)) before += s_warp[w];
            all += s_warp[w];
        }
        run += all;
#pragma unroll
        for (int j = 0; j < kScanPer; ++j)
            if (k0 - j >= 0) {
                cnt[k0 - j] = before;
                before += c[j];
            }
        __syncthreads();  // the next round writes s_warp again
    }
}

__global__ void order_scatter_kernel(OrderArgs o, unsigned long long* off, int64_t* order)
{
    for (int64_t qq = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; qq < o.nq; qq += (int64_t)gridDim.x * blockDim.x)
        order[atomicAdd(&off[order_key(o, qq)], 1ULL)] = qq;
}

int build_order(const int64_t* quartets, int64_t nq, int64_t nbra, const int32_t* kpb, const int32_t* kpk, int KB,
                int KK, int swap, int sort, cudaStream_t st, int64_t** order, unsigned long long** queue)
{
    int err = ERI_OK;
    const int nbins = (KB + 1) * (KK + 1);
    // [2] tile-queue counters, then (sort) [nbins] key counts and [nq] order
    const size_t n64 = 2 + (sort ? (size_t)nbins + (size_t)nq : 0);
    unsigned long long* buf = (unsigned long long*)order_workspace(sizeof(unsigned long long) * n64, &err);
    if (!buf) return err;
    *queue = buf;
    *order = nullptr;
    if (cudaMemsetAsync(buf, 0, sizeof(unsigned long long) * (sort ? 2 + (size_t)nbins : 2), st) != cudaSuccess)
        return ERI_ECUDA;
    if (!sort) return ERI_OK;
    unsigned long long* cnt = buf + 2;
    int64_t* ord = reinterpret_cast<int64_t*>(cnt + nbins);
    const OrderArgs o{quartets, nq, nbra, kpb, kpk, KK, swap};
    const int g = (int)std::min<int64_t>((nq + 255) / 256, (int64_t)sm_count() * 8);
    count_launch();
    order_hist_kernel<<<std::max(g, 1), 256, 0, st>>>(o, cnt);
    count_launch();
    order_scan_kernel<<<1, kScanThreads, 0, st>>>(nbins, cnt);
    count_launch();
    order_scatter_kernel<<<std::max(g, 1), 256, 0, st>>>(o, cnt, ord);
    if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    *order = ord;
    return ERI_OK;
}

}  // namespace eri

using namespace eri;

extern "C" int eri_boys(int mmax, const double* T, int64_t n, double* F, void* stream)
{
    if (mmax < 0 || mmax > ERI_BOYS_MMAX || n < 0) return ERI_EINVAL;
    if (n == 0) return ERI_OK;
    if (!T || !F) return ERI_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int err = ERI_OK;
    const double* tab = get_boys_table(mmax, st, &err);
    if (!tab) return err;
    const int grid = (int)std::min<int64_t>((n + 127) / 128, 16 * sm_count());
    count_launch();
    boys_kernel<<<grid, 128, 0, st>>>(mmax, T, n, tab, F);
    return cudaGetLastError() == cudaSuccess ? ERI_OK : ERI_ECUDA;
}

// Kernel arguments of one forward batch in form fc (the pair tables pb, pk
// of that form are built); the tile shape from the planner.
static int forward_args(const eri_basis_t* basis, const int32_t* bra_pairs, int64_t nbra,
                        const int32_t* ket_pairs, int64_t nket, const int64_t* quartets, int64_t nqq, double* out,
                        const ClassTables* ct, const PairTables& pb, const PairTables& pk, int KB, int KK, int swapped,
                        int split, const FormChoice& fc, cudaStream_t st, FwdArgs* a, TilePlan* tp)
{
    int err = ERI_OK;
    const double* boys = get_boys_table(ct->L, st, &err);
    if (!boys) return err;
    const RStep* rs = get_rsteps(st, &err);
    if (!rs) return err;
    if (!plan_tiles(*ct, KB, KK, nqq, tp, 0, split)) return ERI_EINVAL;
    if (split == XF_FP64 && nqq < kTuneMinQuartets) plan_small_tile(*ct, KB, KK, nqq, tp);
    *a = FwdArgs{};
    if (split == XF_FIXED) {
        const int64_t* fx = get_fix_boys_table(ct->L, st, &err);
        if (!fx) return err;
        a->fx_tab = reinterpret_cast<const long long*>(fx);
        a->fx_far = a->fx_tab + (size_t)kFixBoysRows * fix_boys_words(ct->L);
        a->fx_f = fc.fx_f;
        a->fx_c = (float)(2.42 / (fc.mu * fc.mu));
        a->fx_imu = (float)(1.0 / fc.mu);
        a->fx_rmu = (long long)(0x1p62L / (long double)fc.mu);
    }
    a->ct = *ct;
    a->boys = boys;
    a->rsteps = rs;
    a->bra_ps = pb.ps;
    a->bra_E = pb.E;
    a->bra_kp = pb.kp;
    a->ket_ps = pk.ps;
    a->ket_E = pk.E;
    a->ket_kp = pk.kp;
    a->bra_ex = pb.ex;
    a->bra_norm = pb.norm;
    a->bra_box = pb.box;
    a->ket_box = pk.box;
    a->bra_limbs = pb.limbs;
    a->bra_weak = pb.weak;
    a->ket_ex = pk.ex;
    a->ket_norm = pk.norm;
    a->quartets = quartets;
    a->nq = nqq;
    a->nbra = nbra;  // original roles: output layout and product-form decoding
    a->nket = nket;
    a->swap = swapped;
    const int nab_out = ct->sph ? ct->nab_s : ct->nab_f, ncd_out = ct->sph ? ct->ncd_s : ct->ncd_f;
    a->nab_o = swapped ? ncd_out : nab_out;
    a->ncd_o = swapped ? nab_out : ncd_out;
    a->out = out;
    a->bra_sh = swapped ? ket_pairs : bra_pairs;  // the kernel's lists
    a->ket_sh = swapped ? bra_pairs : ket_pairs;
    a->centres = basis->centres;
    a->shell_atom = basis->shell_atom;
    a->KB = KB;
    a->KK = KK;
    a->nsm = sm_count();
    set_tile(*a, *tp);
    a->ntiles = (nqq + tp->TQ - 1) / tp->TQ;
    return ERI_OK;
}

static thread_local int g_last_form = -1;
static thread_local TilePlan g_last_tile{};
static thread_local int g_last_arithmetic = XF_FP64;

// One forward batch of any kind (0: 4-centre; 1, 2: 3-centre with the unit
// function as the second bra shell, Cartesian or solid-harmonic x): form
// choice, pair tables, tile shape, launch.  Arguments already validated.
static int run_forward(eri_class_t cls, const eri_basis_t* basis, const int32_t* bra_pairs, int64_t nbra,
                       const int32_t* ket_pairs, int64_t nket, const int64_t* quartets, int64_t nq, double* out,
                       int split, int kind, cudaStream_t st)
{
    const int64_t nqq = quartets ? nq : nbra * nket;
    const ClassTables* ct = nullptr;
    PairTables pb{}, pk{};
    int KB = 0, KK = 0, kmax[4];
    FormChoice fc;
    // The recursion forms are FP64 only: the horizontal recursion multiplies
    // the (e0|f0) values by powers of A-B and C-D, which magnifies the split
    // transforms' rounding (about 1e-14 of those larger values) past the
    // 1e-10 bar when the centres are far apart.  3-centre batches have none.
    const int allow = (kind == 1 || kind == 2 || split) ? 1 : 2;
    // a batch that mixes contraction degrees runs its quartets sorted by
    // (kb, kk), each tile looping to its own largest counts; the order is
    // built once, in the first form's orientation (the grouping is the same
    // in the other)
    int mixed = 0;
    int64_t* order = nullptr;
    auto prepare = [&](FormChoice* f, FwdArgs* a, TilePlan* tp) -> int {
        int e = prepare_batch(cls, basis, bra_pairs, nbra, ket_pairs, nket, quartets, nq, 0, st, &ct, &pb, &pk, &KB,
                              &KK, kmax, allow, f, split, kind, &mixed);
        if (e != ERI_OK) return e;
        e = forward_args(basis, bra_pairs, nbra, ket_pairs, nket, quartets, nqq, out, ct, pb, pk, KB, KK,
                         f->form & 1, f->fixed ? XF_FIXED : split, *f, st, a, tp);
        if (e != ERI_OK) return e;
        if (mixed && !order && nqq > 1) {
            unsigned long long* queue = nullptr;
            e = build_order(quartets, nqq, nbra, pb.kp, pk.kp, KB, KK, f->form & 1, 1, st, &order, &queue);
            if (e != ERI_OK) return e;
        }
        a->order = order;
        return ERI_OK;
    };
    FwdArgs a;
    TilePlan tp;
    bool from_tuner = false;
    int err = prepare(&fc, &a, &tp);
    if (err != ERI_OK) return err;
    // large batches: tile shape from the autotuner (cached per kernel class,
    // form and signature); on the first such batch of a signature, the
    // cheapest plain and horizontal-recursion forms are both timed on the
    // batch's own leading quartets and the faster is remembered
    if (nqq >= kTuneMinQuartets) {
        struct Timed {
            FormChoice fc;
            TilePlan tile;
            float ms = 0.f;  // per quartet
            bool tuned = false;
        };
        // The form and tile of the arithmetic that fc came out with; leaves the
        // chosen form prepared (the pair tables share one workspace).
        auto select = [&](Timed* t) -> int {
            t->tuned = tuned_tile(a, t->fc.fixed ? XF_FIXED : split, st, &t->tile, &t->ms);
            if (t->fc.cached || t->fc.alt < 0) return ERI_OK;
            const int KB0 = (t->fc.form & 1) ? KK : KB, KK0 = (t->fc.form & 1) ? KB : KK;  // caller's orientation
            Timed other;
            other.fc.form = t->fc.alt;
            other.fc.no_fixed = t->fc.no_fixed;
            FwdArgs a1;
            TilePlan tp1;
            if (prepare(&other.fc, &a1, &tp1) == ERI_OK)
                other.tuned = tuned_tile(a1, other.fc.fixed ? XF_FIXED : split, st, &other.tile, &other.ms);
            // In fixed point a recursion form, whose epilogue rounds in FP64, has to
            // be 10 % faster: (dp|pp) K = 3, 65000 quartets 7.58 ms against 8.25, error
            // against 64 bits 1.8e-15 against 1.6e-15 (the FP64 tile's plain form 1.6e-15,
            // its recursion form 3.7e-15); (dp|dp) K = 2, 50000, 3.30 against 3.77 ms stays.
            auto weight = [](const FormChoice& f) { return f.fixed && f.form >= 2 ? 1.1f : 1.0f; };
            const bool take_alt = other.tuned && (!t->tuned || weight(other.fc) * other.ms < weight(t->fc) * t->ms);
            remember_form(cls, KB0, KK0, t->fc.key, kind, take_alt ? other.fc.form : t->fc.form);
            if (take_alt) {
                *t = other;
                a = a1;
                tp = tp1;
                return ERI_OK;
            }
            // rebuild the pair tables of the first form (the workspace was reused)
            FormChoice f0;
            f0.form = t->fc.form;
            f0.no_fixed = t->fc.no_fixed;
            return prepare(&f0, &a, &tp);
        };
        Timed best;
        best.fc = fc;
        err = select(&best);
        if (err != ERI_OK) return err;
        // Where fixed point is not surely the faster one, the FP64 tile is timed too,
        // once per signature: fewer than 81 primitive quartets each, or sides whose orders
        // lie four apart or of which one is (ss|.
        // 20000 quartets, ms, FP64 against fixed point: K = 2 (pp|ss) 0.199 / 0.225, (dd|ss)
        // 0.433 / 0.488, (pp|pp) 0.558 / 0.446; K = 3 (ff|ss) 3.81 / 5.39, (dd|ss) 1.26 / 1.06,
        // (ff|ps) 5.21 / 5.65, (fd|ps) 4.15 / 4.34, (ff|ds) 11.0 / 10.9 (16384);
        // elsewhere 0.46 to 0.99 times FP64 for K = 3 and 4, (ps|ps) to (dp|dp).
        const int KB0 = (best.fc.form & 1) ? KK : KB, KK0 = (best.fc.form & 1) ? KB : KK;
        if (best.fc.fixed && best.tuned && g_fixed_mode == ERI_FIXED_RULE && g_form_mask.load() == 0xF &&
            ((int64_t)KB * KK < kFixSmallPrims || cls.la + cls.lb == 0 || cls.lc + cls.ld == 0 ||
             std::abs(cls.la + cls.lb - cls.lc - cls.ld) >= 4) &&
            lookup_fp64_faster(cls, KB0, KK0, kind) < 0) {
            Timed fp64;
            fp64.fc.no_fixed = 1;
            err = prepare(&fp64.fc, &a, &tp);
            if (err == ERI_OK) err = select(&fp64);
            if (err != ERI_OK) return err;
            // (fixed point has to make up for the second pass over its pair tables,
            // about 40 us a call, and for what the timings scatter; an FP64 recursion
            // form, of the larger error, has to be 10 % faster than a plain one)
            const float w = fp64.fc.form >= 2 && best.fc.form < 2 ? 1.1f : 1.0f;
            const bool faster = fp64.tuned && w * fp64.ms * (float)nqq < 1.05f * best.ms * (float)nqq + 0.04f;
            remember_fp64_faster(cls, KB0, KK0, kind, faster);
            if (faster) {
                best = fp64;
            } else {
                FormChoice f0;
                f0.form = best.fc.form;
                err = prepare(&f0, &a, &tp);
                if (err != ERI_OK) return err;
            }
        }
        fc = best.fc;
        if (best.tuned) {
            tp = best.tile;
            set_tile(a, tp);
            a.ntiles = (nqq + tp.TQ - 1) / tp.TQ;
            from_tuner = true;
        }
    }
    if (!from_tuner) {
        // a tile the tuner did not choose (accumulation in memory, or a small
        // batch): 512 threads when the tile leaves room for one CTA per SM
        // only (measured on (ff|ff): FP64 1.07 and 1.14 times faster at K = 5
        // and 1, split 1.27 and 1.34), then, split, the ring of ket E rows;
        // the tuner's candidates come with both settled
        if (!fc.fixed && one_cta_per_sm(tp.bytes)) tp.nt = kNTWide;
        if (split) add_e_ring(a.ct, a.KK, &tp);
        set_tile(a, tp);
    }
    void (*kern)(FwdArgs) = fwd_kern(fc.fixed ? XF_FIXED : split, tp.nt);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tp.bytes) != cudaSuccess)
        return ERI_ECUDA;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, tp.nt, tp.bytes);
    if (per_sm < 1) per_sm = 1;
    const int64_t grid = std::min<int64_t>(a.ntiles, (int64_t)per_sm * sm_count());
    {
        ProfScope ps(PROF_FWD, st);
        kern<<<(int)grid, tp.nt, tp.bytes, st>>>(a);
    }
    if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    g_last_form = fc.form;
    g_last_tile = tp;
    g_last_arithmetic = fc.fixed ? XF_FIXED : split;
    return ERI_OK;
}

extern "C" int eri_batch(eri_class_t cls, const eri_basis_t* basis, const int32_t* bra_pairs, int64_t nbra,
                         const int32_t* ket_pairs, int64_t nket, const int64_t* quartets, int64_t nq, double* out,
                         int64_t out_len, int precision, void* stream)
{
    int err = check_batch_args(cls, basis, bra_pairs, nbra, ket_pairs, nket, quartets, nq, out_len);
    if (err != ERI_OK) return err;
    if (precision != ERI_PREC_FP64 && precision != ERI_PREC_SPLIT) return ERI_EINVAL;
    const int64_t nqq = quartets ? nq : nbra * nket;
    if (nqq == 0 || nbra == 0 || nket == 0) return ERI_OK;
    if (!out) return ERI_EINVAL;
    return run_forward(cls, basis, bra_pairs, nbra, ket_pairs, nket, quartets, nq, out,
                       precision == ERI_PREC_SPLIT, 0, (cudaStream_t)stream);
}

extern "C" int eri_solid_harmonics(int32_t l, double* out)
{
    if (l < 0 || l > ERI_LMAX || !out) return ERI_EINVAL;
    solid_harmonic_table(l, out);
    return ERI_OK;
}

extern "C" int eri_batch_sph(eri_class_t cls, const eri_basis_t* basis, const int32_t* bra_pairs, int64_t nbra,
                             const int32_t* ket_pairs, int64_t nket, const int64_t* quartets, int64_t nq,
                             double* out, int64_t out_len, int precision, void* stream)
{
    int err = check_batch_args(cls, basis, bra_pairs, nbra, ket_pairs, nket, quartets, nq, INT64_MAX);
    if (err != ERI_OK) return err;
    if (precision != ERI_PREC_FP64 && precision != ERI_PREC_SPLIT) return ERI_EINVAL;
    const int64_t nqq = quartets ? nq : nbra * nket;
    const int64_t ns = (int64_t)(2 * cls.la + 1) * (2 * cls.lb + 1) * (2 * cls.lc + 1) * (2 * cls.ld + 1);
    if (out_len < nqq * ns) return ERI_EINVAL;
    if (nqq == 0 || nbra == 0 || nket == 0) return ERI_OK;
    if (!out) return ERI_EINVAL;
    return run_forward(cls, basis, bra_pairs, nbra, ket_pairs, nket, quartets, nq, out,
                       precision == ERI_PREC_SPLIT, 3, (cudaStream_t)stream);
}

__global__ void unit_pairs_kernel(const int32_t* __restrict__ x, int64_t n, int32_t* __restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        out[2 * i] = x[i];
        out[2 * i + 1] = -1;
    }
}

extern "C" int eri_batch3(int32_t lx, int32_t lc, int32_t ld, const eri_basis_t* basis, const int32_t* x_shells,
                          int64_t nx, const int32_t* ket_pairs, int64_t nket, const int64_t* triples, int64_t nt,
                          int32_t pure, double* out, int64_t out_len, int precision, void* stream)
{
    const eri_class_t cls{lx, 0, lc, ld};
    if (pure != 0 && pure != 1) return ERI_EINVAL;
    // the pair-list checks of eri_batch (x shells stand in for the bra pairs)
    int err = check_batch_args(cls, basis, x_shells, nx, ket_pairs, nket, triples, nt, INT64_MAX);
    if (err != ERI_OK) return err;
    if (precision != ERI_PREC_FP64 && precision != ERI_PREC_SPLIT) return ERI_EINVAL;
    const int64_t ntt = triples ? nt : nx * nket;
    const int64_t ncx = pure ? 2 * lx + 1 : host_nc(lx);
    if (out_len < ntt * ncx * host_nc(lc) * host_nc(ld)) return ERI_EINVAL;
    if (ntt == 0 || nx == 0 || nket == 0) return ERI_OK;
    if (!out) return ERI_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int32_t* pairs = (int32_t*)aux_workspace(sizeof(int32_t) * 2 * (size_t)nx, &err);
    if (!pairs) return err;
    const int grid = (int)std::min<int64_t>((nx + 255) / 256, 4 * sm_count());
    unit_pairs_kernel<<<std::max(grid, 1), 256, 0, st>>>(x_shells, nx, pairs);
    if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    count_launch();
    return run_forward(cls, basis, pairs, nx, ket_pairs, nket, triples, nt, out, precision == ERI_PREC_SPLIT,
                       pure ? 2 : 1, st);
}

extern "C" int eri_set_forms(int32_t mask)
{
    if (mask < 0 || mask > 0xF) return ERI_EINVAL;
    return g_form_mask.exchange(mask ? mask : 0xF);
}

extern "C" int eri_last_tile(int32_t* tq, int32_t* ic, int32_t* threads, int32_t* smem_bytes)
{
    if (g_last_form < 0) return ERI_EINVAL;
    if (tq) *tq = g_last_tile.TQ;
    if (ic) *ic = g_last_tile.IC;
    if (threads) *threads = g_last_tile.nt;
    if (smem_bytes) *smem_bytes = (int32_t)g_last_tile.bytes;
    return ERI_OK;
}

static_assert(XF_FP64 == ERI_ARITH_FP64 && XF_SPLIT == ERI_ARITH_SPLIT && XF_FIXED == ERI_ARITH_FIXED, "one numbering");

extern "C" int eri_last_arithmetic(int32_t* arithmetic)
{
    if (!arithmetic || g_last_form < 0) return ERI_EINVAL;
    *arithmetic = g_last_arithmetic;
    return ERI_OK;
}

extern "C" int eri_set_fixed(int32_t mode)
{
    if (mode < ERI_FIXED_NEVER || mode > ERI_FIXED_ALWAYS) return ERI_EINVAL;
    const int prev = g_fixed_mode;
    g_fixed_mode = mode;
    return prev;
}

extern "C" int eri_last_form(int32_t* swapped, int32_t* hrr)
{
    if (!swapped || !hrr) return ERI_EINVAL;
    if (g_last_form < 0) return ERI_EINVAL;
    *swapped = g_last_form & 1;
    *hrr = (g_last_form >> 1) & 1;
    return ERI_OK;
}

namespace eri {

// ---------------------------------------------------------------------------
// The forward batch on tables and scratch the caller supplies (no allocation,
// no swap of the sides): used by the allocation-free entry point.  `dinfo`
// is 5 device ints, `scratch` holds the pair tables of both sides.
// ---------------------------------------------------------------------------
int fwd_batch_on(eri_class_t cls, const eri_basis_t* basis, const int32_t* bra, int64_t nbra, const int32_t* ket,
                 int64_t nket, const int64_t* quartets, int64_t nq, double* out, const ClassTables& ct,
                 const double* boys, const RStep* rs, int* dinfo, double* scratch, size_t scratch_doubles,
                 cudaStream_t st)
{
    if (cudaMemsetAsync(dinfo, 0, 5 * sizeof(int), st) != cudaSuccess) return ERI_ECUDA;
    PrepassArgs pa{basis->shell_l, basis->shell_K, basis->nshell, bra, nbra, ket, nket, quartets,
                   quartets ? nq : (int64_t)0, {cls.la, cls.lb, cls.lc, cls.ld}, 0, dinfo, 0,
                   nullptr, nullptr, nullptr, nullptr};
    const int64_t n = std::max(std::max(nbra, nket), quartets ? nq : (int64_t)0);
    const int grid = (int)std::min<int64_t>((n + 255) / 256, 4 * sm_count());
    count_launch();
    prepass_kernel<<<std::max(grid, 1), 256, 0, st>>>(pa);
    if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    int hinfo[5] = {0, 0, 0, 0, 0};
    if (cudaMemcpyAsync(hinfo, dinfo, sizeof(hinfo), cudaMemcpyDeviceToHost, st) != cudaSuccess) return ERI_ECUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return ERI_ECUDA;
    if (hinfo[4] != 0) return dev_err_to_code(hinfo[4]);
    const int KB = hinfo[0] * hinfo[1], KK = hinfo[2] * hinfo[3];
    // carve the scratch: [ps_b | E_b | ps_k | E_k | kp_b | kp_k], 32-double aligned pieces
    auto up = [](size_t d) { return (d + 31) & ~size_t(31); };
    const size_t n_psb = up((size_t)nbra * KB * PS_N), n_Eb = up((size_t)nbra * KB * ct.Tab);
    const size_t n_psk = up((size_t)nket * KK * PS_N), n_Ek = up((size_t)nket * KK * ct.Tcd);
    const size_t n_kpb = up(((size_t)nbra + 1) / 2), n_kpk = up(((size_t)nket + 1) / 2);
    if (n_psb + n_Eb + n_psk + n_Ek + n_kpb + n_kpk > scratch_doubles) return ERI_EINVAL;
    PairTables pb{}, pk{};
    pb.ps = scratch;
    pb.E = pb.ps + n_psb;
    pk.ps = pb.E + n_Eb;
    pk.E = pk.ps + n_psk;
    pb.kp = reinterpret_cast<int32_t*>(pk.E + n_Ek);
    pk.kp = reinterpret_cast<int32_t*>(pk.E + n_Ek + n_kpb);
    for (int side = 0; side < 2; ++side) {
        PairArgs p{};
        p.centres = basis->centres;
        p.shell_atom = basis->shell_atom;
        p.shell_K = basis->shell_K;
        p.shell_off = basis->shell_off;
        p.exps = basis->exps;
        p.coefs = basis->coefs;
        p.pairs = side ? ket : bra;
        p.npairs = side ? nket : nbra;
        p.l1 = side ? cls.lc : cls.la;
        p.l2 = side ? cls.ld : cls.lb;
        p.KS = side ? KK : KB;
        p.T = side ? ct.Tcd : ct.Tab;
        p.fac = side ? ct.ket_fac : ct.bra_fac;
        p.ket = side;
        const PairTables& t = side ? pk : pb;
        p.ps = t.ps;
        p.E = t.E;
        p.kprim = t.kp;
        const int64_t tot = p.npairs * p.KS;
        const int g = (int)std::min<int64_t>((tot + 127) / 128, 8 * sm_count());
        count_launch();
        launch_pair(p, std::max(g, 1), st);
        if (cudaGetLastError() != cudaSuccess) return ERI_ECUDA;
    }
    const int64_t nqq = quartets ? nq : nbra * nket;
    TilePlan tp;
    if (!plan_tiles(ct, KB, KK, nqq, &tp)) return ERI_EINVAL;
    FwdArgs a{};
    a.ct = ct;
    a.boys = boys;
    a.rsteps = rs;
    a.bra_ps = pb.ps;
    a.bra_E = pb.E;
    a.bra_kp = pb.kp;
    a.ket_ps = pk.ps;
    a.ket_E = pk.E;
    a.ket_kp = pk.kp;
    a.quartets = quartets;
    a.nq = nqq;
    a.nbra = nbra;
    a.nket = nket;
    a.swap = 0;
    a.nab_o = ct.nab_f;
    a.ncd_o = ct.ncd_f;
    a.out = out;
    a.KB = KB;
    a.KK = KK;
    set_tile(a, tp);
    a.ntiles = (nqq + tp.TQ - 1) / tp.TQ;
    if (cudaFuncSetAttribute(fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tp.bytes) != cudaSuccess)
        return ERI_ECUDA;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fwd_kernel, kNT, tp.bytes);
    if (per_sm < 1) per_sm = 1;
    const int64_t grid2 = std::min<int64_t>(a.ntiles, (int64_t)per_sm * sm_count());
    count_launch();
    fwd_kernel<<<(int)grid2, kNT, tp.bytes, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? ERI_OK : ERI_ECUDA;
}

}  // namespace eri

namespace eri {

// Pair tables of one list of shell pairs with a uniform K1*K2 = KS, written
// into caller-provided buffers (plans own theirs).
int build_pair_tables_on(const eri_basis_t* basis, const int32_t* d_pairs, int64_t npairs, int l1, int l2, int KS,
                         int T, const uint8_t* fac, int ket, int split, PairTables* out, cudaStream_t st)
{
    PairArgs p{};
    p.centres = basis->centres;
    p.shell_atom = basis->shell_atom;
    p.shell_K = basis->shell_K;
    p.shell_off = basis->shell_off;
    p.exps = basis->exps;
    p.coefs = basis->coefs;
    p.pairs = d_pairs;
    p.npairs = npairs;
    p.l1 = l1;
    p.l2 = l2;
    p.KS = KS;
    p.T = T;
    p.fac = fac;
    p.ket = ket;
    p.ps = out->ps;
    p.E = out->E;
    p.kprim = out->kp;
    p.split = split;
    const int64_t tot = npairs * KS;
    const int g = (int)std::min<int64_t>((tot + 127) / 128, 8 * sm_count());
    count_launch();
    launch_pair(p, std::max(g, 1), st);
    return cudaGetLastError() == cudaSuccess ? ERI_OK : ERI_ECUDA;
}

}  // namespace eri
