// lll_quadrature.cpp -- Gauss rule of the weight x^2 nu(x) on [-a, a] (host, FP64).
//
// The drift of Eq. (LIBOR-drift-PT) integrates an O(x^2) function against the
// Levy measure, so it is written against the bounded weight m(x) = x^2 nu(x):
// int g dF ~= sum_j W_j g(x_j) / x_j^2.  For NIG (Section 4 gives kappa;
// the density is Barndorff-Nielsen's)
//     m(x) = (dbar alpha / pi) |x| e^{beta x} K_1(alpha |x|).
// Steps: (1) discretise m with a composite Gauss-Legendre rule on panels
// graded geometrically towards the origin; (2) Stieltjes recurrence for the
// orthonormal polynomials of the discrete measure, with full
// re-orthogonalisation; (3) nodes = eigenvalues of the Jacobi matrix by
// Sturm-sequence bisection; (4) weights = Christoffel numbers
// 1 / sum_k p_k(x_j)^2.
#include <algorithm>
#include <cmath>
#include <vector>

namespace lll {
namespace {

// Gauss-Legendre nodes/weights on [-1, 1] by Newton iteration on P_G.
void gauss_legendre(int G, std::vector<double> &t, std::vector<double> &w)
{
    t.assign(G, 0.0);
    w.assign(G, 0.0);
    for (int i = 0; i < (G + 1) / 2; ++i) {
        double z = std::cos(M_PI * (i + 0.75) / (G + 0.5));
        double dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= G; ++k) {
                const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = G * (z * p1 - p0) / (z * z - 1.0);
            const double dz = p1 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        t[i] = -z;
        t[G - 1 - i] = z;
        w[i] = w[G - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

double x2nu(double x, double alpha, double beta, double dbar)
{
    const double ax = std::fabs(x);
    if (ax == 0.0) return dbar / M_PI;
    return dbar * alpha / M_PI * ax * std::exp(beta * x) * std::cyl_bessel_k(1.0, alpha * ax);
}

// Recurrence coefficients al[0..K), bt[1..K) of the polynomials orthonormal for
// the measure sum_i v_i delta_{y_i} (Stieltjes procedure with orthonormal
// vectors q_k(y_i) sqrt(v_i) and full re-orthogonalisation), extended on demand.
struct Jacobi {
    const std::vector<double> &y;
    double mu0 = 0.0;
    std::vector<double> al, bt; // bt[0] unused
    std::vector<std::vector<double>> qs;

    Jacobi(const std::vector<double> &y_, const std::vector<double> &v) : y(y_)
    {
        for (double w : v) mu0 += w;
        std::vector<double> q(v.size());
        for (size_t i = 0; i < v.size(); ++i) q[i] = std::sqrt(v[i] / mu0);
        qs.push_back(q);
        bt.push_back(0.0);
    }

    // Coefficients up to al[K-1]; 0 on success.
    int extend(int K)
    {
        if (!(mu0 > 0.0)) return -1;
        const size_t M = y.size();
        while ((int)al.size() < K) {
            const int k = (int)al.size();
            if (k > 0) { // the next vector
                const std::vector<double> &qk = qs[k - 1];
                std::vector<double> r(M);
                for (size_t i = 0; i < M; ++i)
                    r[i] = (y[i] - al[k - 1]) * qk[i] - (k > 1 ? bt[k - 1] * qs[k - 2][i] : 0.0);
                for (int pass = 0; pass < 2; ++pass)
                    for (const auto &qq : qs) {
                        double d = 0.0;
                        for (size_t i = 0; i < M; ++i) d += qq[i] * r[i];
                        for (size_t i = 0; i < M; ++i) r[i] -= d * qq[i];
                    }
                double nr = 0.0;
                for (size_t i = 0; i < M; ++i) nr += r[i] * r[i];
                nr = std::sqrt(nr);
                if (!(nr > 0.0)) return -2;
                for (size_t i = 0; i < M; ++i) r[i] /= nr;
                bt.push_back(nr);
                qs.push_back(r);
            }
            double a = 0.0;
            for (size_t i = 0; i < M; ++i) a += y[i] * qs[k][i] * qs[k][i];
            al.push_back(a);
        }
        return 0;
    }
};

// The Q-point Gauss rule of those coefficients (Q at most their number).
void gauss_of_jacobi(const std::vector<double> &al, const std::vector<double> &bt, double mu0, int Q, double *nodes,
                     double *weights)
{
    // Eigenvalues of the Jacobi matrix by bisection on Sturm counts.
    double lo = al[0], hi = al[0];
    for (int k = 0; k < Q; ++k) {
        const double rad = (k > 0 ? bt[k] : 0.0) + (k + 1 < Q ? bt[k + 1] : 0.0);
        lo = std::min(lo, al[k] - rad);
        hi = std::max(hi, al[k] + rad);
    }
    // All eigenvalues are bisected side by side: a Sturm sequence is a chain of
    // divisions, and Q independent chains overlap where one after the other waited for
    // each quotient (the search of shorter_rule that ends without a rule, 64 nodes:
    // 0.79 -> 0.36 ms).  The numbers are those of one bisection at a time.
    std::vector<double> a0(Q, lo), b0(Q, hi), mid(Q), d(Q);
    std::vector<int> below(Q);
    for (int it = 0; it < 200; ++it) {
        bool moving = false;
        for (int j = 0; j < Q; ++j) {
            mid[j] = 0.5 * (a0[j] + b0[j]);
            moving = moving || (mid[j] > a0[j] && mid[j] < b0[j]);
            d[j] = 1.0;
            below[j] = 0;
        }
        if (!moving) break;
        for (int k = 0; k < Q; ++k) {
            const double off = k > 0 ? bt[k] * bt[k] : 0.0, alk = al[k];
            for (int j = 0; j < Q; ++j) {
                double v = alk - mid[j] - off / d[j];
                v = v == 0.0 ? -1e-300 : v;
                below[j] += v < 0.0;
                d[j] = v;
            }
        }
        for (int j = 0; j < Q; ++j)
            if (mid[j] > a0[j] && mid[j] < b0[j]) (below[j] > j ? b0 : a0)[j] = mid[j];
    }
    for (int j = 0; j < Q; ++j) nodes[j] = 0.5 * (a0[j] + b0[j]);
    // Christoffel numbers from the orthonormal recurrence.
    for (int j = 0; j < Q; ++j) {
        const double xx = nodes[j];
        double pm = 0.0, pc = 1.0 / std::sqrt(mu0), s = pc * pc;
        for (int k = 0; k + 1 < Q; ++k) {
            const double pn = ((xx - al[k]) * pc - (k > 0 ? bt[k] * pm : 0.0)) / bt[k + 1];
            pm = pc;
            pc = pn;
            s += pc * pc;
        }
        weights[j] = 1.0 / s;
    }
}

}  // namespace

// Returns 0 on success.
int build_nig_rule(double alpha, double beta, double dbar, double a, int Q, double *nodes,
                   double *weights)
{
    const int G = 32;
    std::vector<double> gt, gw;
    gauss_legendre(G, gt, gw);
    std::vector<double> edges;
    edges.push_back(0.0);
    const int outer = 24;
    for (double e = 1e-14 * a; e < a / outer; e /= 0.35) edges.push_back(e);
    for (int i = 1; i <= outer; ++i) edges.push_back(a * i / outer);
    std::vector<double> y, v;
    for (int side = -1; side <= 1; side += 2)
        for (size_t p = 0; p + 1 < edges.size(); ++p) {
            const double lo = edges[p], hi = edges[p + 1];
            const double mid = 0.5 * (lo + hi), half = 0.5 * (hi - lo);
            for (int g = 0; g < G; ++g) {
                const double xx = side * (mid + half * gt[g]);
                y.push_back(xx);
                v.push_back(half * gw[g] * x2nu(xx, alpha, beta, dbar));
            }
        }
    Jacobi J(y, v);
    const int rc = J.extend(Q);
    if (rc != 0) return rc;
    gauss_of_jacobi(J.al, J.bt, J.mu0, Q, nodes, weights);
    return 0;
}

// ---- A shorter rule for the same measure -----------------------------------
// The path kernels integrate, for every path, step and rate,
//     A_i - C_i = sum_j W_j / x_j^2 (e^{lambda_i x_j} - 1) (P(x_j) - 1),
//     P(x) = prod_{l > i} (1 - w_l + w_l e^{lambda_l x}),  w_l in (0, 1).
// Expanded, P is a convex combination of exponentials e^{theta x}, theta a sum
// of some of the lambda_l, and
//     (e^{lambda x} - 1) (e^{theta x} - 1) / x^2 = int_0^lambda int_0^theta e^{(u+v) x} dv du,
// so every such integral is an integral over tau = u + v of the rule's moment
// generating function G(tau) = sum_j W_j e^{tau x_j}, tau between minus the sum
// of the negative and the sum of the positive lambda's.  A rule of q nodes
// whose generating function agrees with G to a relative eps over that interval
// therefore gives A_i - C_i to the relative error eps (against the absolute
// value of its terms, where the lambda's differ in sign), whatever the path's
// rates are.  The q-point Gauss rule of the discrete measure sum_j W_j
// delta_{x_j} is the natural one (Gautschi 2004, "Orthogonal Polynomials:
// Computation and Approximation", 2.2): exact to degree 2q - 1.
//
// eps = 2^-28, a sixteenth of FP32's unit roundoff, in which the integral is
// summed.  A second condition keeps the sum's rounding no larger than the
// given rule's: the terms c_j E_ij sum in absolute value to about
// |lambda| sum_j W_j / |x_j|, which a node next to 0 inflates.
constexpr double kRuleTol = 1.0 / 268435456.0;

static bool same_generating_function(const double *x, const double *W, int Q, const double *xr, const double *Wr,
                                     int q, double lo, double hi)
{
    constexpr int kGrid = 32; // the relative error grows smoothly away from tau = 0: the ends first
    for (int g = 2 * kGrid + 1; g >= 0; --g) {
        const double tau = (g & 1 ? lo : hi) * (g >> 1) / kGrid;
        if (tau == 0.0 && g > 0) continue;
        double top = 0.0; // largest exponent, taken out against overflow
        for (int j = 0; j < Q; ++j) top = std::max(top, tau * x[j]);
        double G = 0.0, Gr = 0.0;
        for (int j = 0; j < Q; ++j) G += W[j] * std::exp(tau * x[j] - top);
        for (int j = 0; j < q; ++j) Gr += Wr[j] * std::exp(tau * xr[j] - top);
        if (!(std::fabs(Gr - G) <= kRuleTol * G)) return false;
    }
    return true;
}

// A rule that stands for (x, W) by the two conditions above: of the node counts that
// the kernels process (4, 8, 12, 16, 20, 24 or 32, less than Qpad) the first that
// holds one, and in it the longest; lo <= 0 <= hi bound tau.
// Returns its node count, 0 if there is none (the given rule is then swept).
// *pad: the node count it is padded to.
int shorter_rule(const double *x, const double *W, int Q, int Qpad, double lo, double hi, double *xr, double *Wr,
                 int *pad)
{
    double spread = 0.0, nearest = std::fabs(x[0]), farthest = 0.0;
    for (int j = 0; j < Q; ++j) {
        if (!(W[j] > 0.0)) return 0; // a Gauss rule of the measure needs positive weights
        spread += W[j] / std::fabs(x[j]);
        nearest = std::min(nearest, std::fabs(x[j]));
        farthest = std::max(farthest, std::fabs(x[j]));
    }
    // With a node this close to 0 the rounding of c_j E_ij shows in the given rule's
    // prices (nearest 2e-5 of the farthest: 4e-5 of the prices against 64 bits).  A
    // shorter rule would not have it, but would move prices that a caller holds by as
    // much.  Such a rule is swept as given, at its full cost; the bound lies between
    // single rules (of 525 portfolio instances three lie below, at 2.5e-6, 1.9e-5 and
    // 3.8e-5, and the next at 8.2e-5).
    if (Q > 1 && nearest < 4e-5 * farthest) return 0;
    if (!std::isfinite(lo) || !std::isfinite(hi) || !std::isfinite(spread)) return 0;
    std::vector<double> y(x, x + Q), v(W, W + Q);
    const int most = std::min(Q, 32);
    Jacobi J(y, v);
    const int pads[] = {4, 8, 12, 16, 20, 24, 32};
    int below = 0;
    for (int p : pads) {
        if (p >= Qpad || J.extend(std::min(p, most)) != 0) break;
        for (int q = std::min(p, most); q > below; --q) {
            gauss_of_jacobi(J.al, J.bt, J.mu0, q, xr, Wr);
            if (!same_generating_function(x, W, Q, xr, Wr, q, lo, hi)) break; // fewer nodes are no nearer
            double s = 0.0;
            bool fine = true;
            for (int j = 0; j < q; ++j) {
                s += Wr[j] / std::fabs(xr[j]);
                fine = fine && Wr[j] > 0.0 && std::isfinite((float)(Wr[j] / (xr[j] * xr[j])));
            }
            if (!fine || !(s <= spread)) continue;
            *pad = p;
            return q;
        }
        below = p;
    }
    return 0;
}

}  // namespace lll
