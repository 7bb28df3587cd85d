// Separable form of the energy denominators of Eq. (Pstatic):
//     2 / (E_c - E_v) = sum_{t < T} u_t(v) z_t(c)   to a stated relative accuracy, entry by entry.
//
// With x_v = -E_v and y_c = E_c the weights form a Cauchy matrix 2 / (x_v + y_c), positive because
// every E_c lies above every E_v.  Gaussian elimination of a Cauchy matrix has a closed form: after
// pivots (v_s, c_s), s < t, the remaining matrix is
//     R_t(v, c) = 2 a_t(v) b_t(c) / (x_v + y_c),
//     a_t(v) = prod_s (x_v - x_{v_s}) / (x_v + y_{c_s}),  b_t(c) = prod_s (y_c - y_{c_s}) / (x_{v_s} + y_c),
// so |a_t(v) b_t(c)| is the relative error left at (v, c): no cancellation, no O(nv nc) search.  The
// elimination stops once max|a| max|b| <= tol.  Each pivot is the largest entry of its row and column
// (a few alternating searches), the term is the cross through it,
//     u_t(v) = R_t(v, c_t),   z_t(c) = R_t(v_t, c) / R_t(v_t, c_t).
// Such pivots keep the terms small: their sizes add up to at most 1.3 of the weight at any (v, c) for a
// gap of 1/60 of the energy range, 2.8 for one of 1e-4 of it (pivots by |a| and |b| alone reach 50
// there), and to 0.8 to 1 of the weights in their root mean square.  The error falls geometrically with t
// (the numerical rank of a Cauchy matrix grows with the logarithm of the cross ratio of its two
// intervals): 8 to 13 terms reach 2^-26 for E_v in [-10, 0] eV and E_c in [0.5, 20] eV.  The factors are then
// rounded to FP32, which leaves about 1e-7 of a weight (measured at most 8.8e-8 with 32 x 480 and 64 x 1000 states), less
// than the 2^-23 that sqrt(2 / (E_c - E_v)) in FP32 carries into both factors of a pair density.
// The unoccupied states are taken from the highest energy down: z_0 falls with E_c, so the sums over c
// grow towards their end, and the truncating additions of the tensor cores lose less than on the way of
// a sum that is large from its start.
//
// Plain C++ (no CUDA), so that the CPU tests compile it too.
#pragma once
#include <cmath>
#include <cstddef>
#include <vector>

namespace gw {

constexpr double SEP_TOL = 0x1p-26;

struct SepFactors {
    int T = 0;                    // terms; 0: not reached within max_terms
    int ldu = 0;                  // values per term: nc and nv, each rounded up to `chunk`
    std::vector<float> tab;       // [T][ldu]: z_t(nc - 1 - i) 2^-e, zeros, then u_t(v) 2^-e', zeros (|.| <= 1)
    std::vector<float> scale;     // [T]: 2^(e + e')
};

// E: Hartree, nv occupied then nc unoccupied energies, in any order.
inline SepFactors sep_factors(const double *E, int nv, int nc, int chunk, int max_terms, double tol = SEP_TOL)
{
    SepFactors f;
    const double *Ev = E, *Ec = E + nv;
    std::vector<double> a(nv, 1.0), b(nc, 1.0), iv(nv), ic(nc);  // iv, ic: 1 / (E_c - E_v) along the pivot's cross
    auto biggest = [](const std::vector<double> &w, const std::vector<double> *by) {
        size_t best = 0;
        double m = -1.0;
        for (size_t i = 0; i < w.size(); ++i) {
            const double x = std::fabs(by ? w[i] * (*by)[i] : w[i]);
            if (x > m) {
                m = x;
                best = i;
            }
        }
        return best;
    };
    const int cpad = (nc + chunk - 1) / chunk * chunk, vpad = (nv + chunk - 1) / chunk * chunk;
    f.ldu = cpad + vpad;
    double lowest = Ec[0];
    for (int c = 1; c < nc; ++c)
        lowest = std::fmin(lowest, Ec[c]);
    for (int t = 0;; ++t) {
        if (std::fabs(a[biggest(a, nullptr)]) * std::fabs(b[biggest(b, nullptr)]) <= tol) {
            f.T = t;
            return f;
        }
        if (t == max_terms)
            return SepFactors();
        for (int v = 0; v < nv; ++v)
            iv[v] = 1.0 / (lowest - Ev[v]);
        size_t pv = biggest(a, &iv), pc = 0;
        for (int round = 0; round < 6; ++round) {
            for (int c = 0; c < nc; ++c)
                ic[c] = 1.0 / (Ec[c] - Ev[pv]);
            pc = biggest(b, &ic);
            for (int v = 0; v < nv; ++v)
                iv[v] = 1.0 / (Ec[pc] - Ev[v]);
            const size_t next = biggest(a, &iv);
            if (next == pv || round == 5)  // iv and ic belong to (pv, pc)
                break;
            pv = next;
        }
        // u = 2 a b_pc iv and z = b ic / (b_pc ic_pc), each with its largest power of two divided out
        const double us = 2.0 * b[pc], zs = 1.0 / (b[pc] * ic[pc]);
        int eu = 0, ez = 0;
        std::frexp(us * a[biggest(a, &iv)] * iv[biggest(a, &iv)], &eu);
        std::frexp(zs * b[biggest(b, &ic)] * ic[biggest(b, &ic)], &ez);
        if (!std::isfinite(us * a[pv] * iv[pv]) || eu + ez > 100 || eu + ez < -100)
            return SepFactors();  // gaps that FP32 scales cannot carry
        f.tab.resize((size_t)(t + 1) * f.ldu, 0.f);
        float *row = f.tab.data() + (size_t)t * f.ldu;
        const double u1 = std::ldexp(us, -eu), z1 = std::ldexp(zs, -ez);
        for (int v = 0; v < nv; ++v)
            row[cpad + v] = static_cast<float>(u1 * a[v] * iv[v]);
        for (int c = 0; c < nc; ++c)
            row[nc - 1 - c] = static_cast<float>(z1 * b[c] * ic[c]);
        f.scale.push_back(static_cast<float>(std::ldexp(1.0, eu + ez)));
        const double ev = Ev[pv], ec = Ec[pc];
        for (int v = 0; v < nv; ++v)
            a[v] *= (ev - Ev[v]) * iv[v];
        for (int c = 0; c < nc; ++c)
            b[c] *= (Ec[c] - ec) * ic[c];
    }
}

}  // namespace gw
