"""The fixed-point auxiliary integrals (csrc/eri_fixaux.cuh is host code too)
against a long double evaluation of Eqs. boys, 0m and r-rr, at every range of
the Boys argument, and their table rows at the row ends."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_12501_gb300", "csrc")

SOURCE = r"""
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>
#include "eri_fixaux.cuh"
using namespace eri;
typedef long double Q;
static void boys(int M, Q T, Q* F) {
    if (T < 60) {
        Q term = Q(1) / (2 * M + 1), s = term;
        for (int k = 1; k < 2000 && term > s * 1e-25L; ++k) { term *= 2 * T / (2 * M + 2 * k + 1); s += term; }
        const Q e = expl(-T);
        F[M] = e * s;
        for (int m = M - 1; m >= 0; --m) F[m] = (2 * T * F[m + 1] + e) / (2 * m + 1);
    } else {
        const Q e = expl(-T);
        F[0] = 0.5L * sqrtl(3.14159265358979323846264338327950288L / T) * erfl(sqrtl(T));
        for (int m = 0; m < M; ++m) F[m + 1] = ((2 * m + 1) * F[m] - e) / (2 * T);
    }
}
static int idx(int t, int u, int v) { const int N = t + u + v; return N * (N + 1) * (N + 2) / 6 + (u + v) * (u + v + 1) / 2 + v; }
int main() {
    const int W = kBoysMtab + 2;
    std::vector<Q> master((size_t)kBoysGrid * W);
    std::vector<bool> have(kBoysGrid, false);
    std::mt19937_64 g(7);
    auto uni = [&](double a, double b) { return a + (b - a) * ((g() >> 11) * 0x1p-53); };
    for (int L : {0, 1, 2, 3, 4, 6, 8, 10}) {
        const int words = fix_boys_words(L), nh = (L + 1) * (L + 2) * (L + 3) / 6;
        std::vector<int64_t> tab((size_t)kFixBoysRows * words, 0), far(kFixFarWords);
        std::vector<bool> row(kFixBoysRows, false);
        fix_far_constants(L, far.data());
        auto need = [&](int j) {  // the table's row j, and the coarse row it comes from
            if (j < 0 || j >= kFixBoysRows || row[j]) return;
            row[j] = true;
            const int per = kFixBoysInvStep / kBoysInvStep, c = (j + per / 2) / per;
            if (!have[c]) {
                Q F[kBoysMtab + 1];
                boys(kBoysMtab, (Q)c / kBoysInvStep, F);
                for (int m = 0; m <= kBoysMtab; ++m) master[(size_t)c * W + m] = F[m];
                master[(size_t)c * W + kBoysMtab + 1] = expl(-(Q)c / kBoysInvStep);
                have[c] = true;
            }
            fix_boys_row(master.data(), L, j, tab.data() + (size_t)j * words);
        };
        std::vector<int> hx(nh), hy(nh), hz(nh);
        for (int N = 0; N <= L; ++N)
            for (int t = N; t >= 0; --t)
                for (int u = N - t; u >= 0; --u) { const int e = idx(t, u, N - t - u); hx[e] = t; hy[e] = u; hz[e] = N - t - u; }
        double worst0 = 0, rms = 0, rmsd = 0, bound = 0;
        const int n = 1500;
        for (int it = 0; it < n; ++it) {
            const double zp = pow(10, uni(-1.3, 2)), zq = pow(10, uni(-1.3, 2)), rho = zp * zq / (zp + zq);
            const double r = it % 4 == 0 ? 0.0 : it % 4 == 1 ? sqrt(uni(0, 30) / rho) : it % 4 == 2 ? sqrt(uni(300, 340) / rho) : pow(10, uni(-3, 1.5));
            double P[3], C[3], d[3], len = 0;
            for (int i = 0; i < 3; ++i) { d[i] = uni(-1, 1); len += d[i] * d[i]; }
            const int f = 54;
            FixPrim a, b;
            for (int i = 0; i < 3; ++i) {
                P[i] = uni(-6, 6);
                C[i] = P[i] + r * d[i] / sqrt(len);
                a.x[i] = fix_coordinate(P[i], f);
                b.x[i] = fix_coordinate(C[i], f);
            }
            fix_split_exponent(1 / zp, &a.um, &a.ue);
            fix_split_exponent(1 / zq, &b.um, &b.ue);
            Q X[3], R2 = 0;
            const Q rq = 1 / ((Q)(1 / zp) + (Q)(1 / zq));
            for (int i = 0; i < 3; ++i) { X[i] = ((Q)a.x[i] - (Q)b.x[i]) / powl(2, f); R2 += X[i] * X[i]; }
            const Q T = rq * R2;
            if (T < 321) for (int j = -1; j <= 1; ++j) need((int)floorl(T * kFixBoysInvStep + 0.5L) + j);
            long long F[11], phi[11];
            int sh[11];
            FixBase B;
            fix_base<10>(L, a, b, f, (const long long*)tab.data(), (const long long*)far.data(), F, B);
            if (L == 0) B.U = 1LL << 61, B.ue = 0;
            const double mu = 1.37;
            const int sigma = ((int)floor(log2(2.42 / (mu * mu) * rho)) + 2) >> 1;
            const int gg = fix_bound(L, (float)rho, (float)R2, sigma, (float)(1 / mu));
            fix_factors<10>(L, B, sigma, (long long)(0x1p62L / (Q)mu), gg, phi, sh);
            std::vector<long long> R(nh);
            int x1[3], x0[3];
            for (int i = 0; i < 3 && L; ++i) { x1[i] = (int)((B.x[i] + (1LL << 28)) >> 29); x0[i] = (int)((B.x[i] - ((long long)x1[i] << 29)) * 8); }
            std::vector<Q> c(nh);
            std::vector<double> cd(nh);
            Q FQ[12], FD[12];
            boys(L, T, FQ);
            double Xd[3], Td = 0;
            for (int i = 0; i < 3; ++i) { Xd[i] = P[i] - C[i]; Td += Xd[i] * Xd[i]; }
            boys(L, (Q)(Td *= rho), FD);
            auto base = [&](int k) { return sqrtl(rq) * powl(-2 * rq, k) * FQ[k]; };
            auto based = [&](int k) { double v = sqrt(rho); for (int i = 0; i < k; ++i) v *= -2 * rho; return v * (double)FD[k]; };
            R[0] = F[L]; c[0] = base(L); cd[0] = based(L);
            for (int k = L - 1; k >= 0; --k) {
                const int N = L - k;
                for (int e = (N + 1) * (N + 2) * (N + 3) / 6 - 1; e >= 1; --e) {
                    int h[3] = {hx[e], hy[e], hz[e]}, ax = -1;
                    for (int i = 0; i < 3 && ax < 0; ++i) if (h[i] == 1) ax = i;
                    for (int i = 0, best = 99; i < 3 && (ax < 0 || best < 99); ++i) if (h[i] > 0 && h[i] < best) { best = h[i]; ax = i; }
                    const int m = h[ax] - 1;
                    h[ax] -= 1;
                    const int i1 = idx(h[0], h[1], h[2]);
                    int i2 = i1;
                    if (m) { h[ax] -= 1; i2 = idx(h[0], h[1], h[2]); }
                    R[e] = m ? fix_step(x1[ax], x0[ax], R[i1], m, R[i2]) : fix_step(x1[ax], x0[ax], R[i1]);
                    c[e] = X[ax] * c[i1] + (m ? m * c[i2] : 0);
                    cd[e] = Xd[ax] * cd[i1] + (m ? m * cd[i2] : 0);
                }
                R[0] = F[k]; c[0] = base(k); cd[0] = based(k);
            }
            for (int e = 0; e < nh; ++e) {
                const int N = hx[e] + hy[e] + hz[e];
                const Q s = powl(mu * powl(2, sigma), -N), ref = c[e] * s;
                const double er = (double)((Q)fix_finish(R[e], phi[N], sh[N]) * powl(2, gg - 62) - ref) / (double)c[0];
                const double ed = (double)((Q)cd[e] * s - ref) / (double)c[0];
                if (e == 0) worst0 = std::max(worst0, fabs(er));
                rms += er * er / nh; rmsd += ed * ed / nh;
                bound = std::max(bound, fabs((double)ref) * pow(2, -gg));
            }
        }
        printf("%d %.3e %.3e %.3e %.4f\n", L, worst0, sqrt(rms / n), sqrt(rmsd / n), bound);
    }
}
"""


@pytest.fixture(scope="module")
def figures(tmp_path_factory):
    d = tmp_path_factory.mktemp("aux")
    src = d / "aux.cpp"
    src.write_text(SOURCE)
    from paper_2506_12501_gb300.build import nvcc
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, "-I", inc, str(src), "-o", str(d / "aux")], check=True,
                   capture_output=True)
    out = subprocess.run([str(d / "aux")], check=True, capture_output=True, text=True, timeout=300).stdout
    return {int(w[0]): [float(x) for x in w[1:]] for w in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("L", [0, 1, 2, 3, 4, 6, 8, 10])
def test_fixed_auxiliary_integrals(figures, L):
    worst0, rms, rms_double, bound = figures[L]
    # order 0: units of 2^-61 of F_0's row, T to 2^-54 absolute and 2^-56 relative
    assert worst0 < 2.0 ** -53.5
    # every order: no further off than the same recursion in double precision
    assert rms < rms_double
    # the bound the integrals are scaled by holds (an excess would overflow the limbs)
    assert bound <= 1.0
