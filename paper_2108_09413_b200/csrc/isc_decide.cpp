// Host side of Algorithm 1 (steps 2, 5-9) and Algorithm 2 (steps 2-6), and the cumulative
// table of the noise law (Def. 3.3, Eq. 2).  IEEE doubles, fixed evaluation order, compiled
// without contraction or fast-math so that the result is reproducible bit for bit.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "isc_internal.h"

namespace isc {

namespace {

// P[Binomial(n, p) >= k] for p <= k / n, its terms added for i = k, k+1, ..., n.  At such a p the terms fall from the
// first one on, so a term below 2^-60 of the sum so far is the last that has to be looked at: every later one, even
// with the rounding of its exponent (below 1e-3 for any n < 2^31), is less than half a unit in the sum's last place
// and would leave it as it is.  The sum is bit for bit the one over all n - k + 1 terms; near the bound's root
// that is about 6.5 standard deviations of terms instead of n - k + 1 (some 700 instead of 20,000 at n = 100,000,
// k = 80,000).  log_choose(n, i) does not depend on p and is kept from evaluation to evaluation.
class UpperTail {
public:
    UpperTail(int64_t k, int64_t n) : k_(k), n_(n), log_n_(std::lgamma((double)n + 1.0)) {}
    // `enough`: the sum may stop once it has reached it (it only grows)
    double operator()(double p, double enough = 1e300)
    {
        const double log_p = std::log(p);
        const double log_q = std::log1p(-p);
        double total = 0.0;
        for (int64_t i = k_; i <= n_ && total < enough; ++i) {
            const double e = choose(i) + (double)i * log_p + (double)(n_ - i) * log_q;
            if (e < -760.0) break;                       // this term and all later ones are zero
            const double term = std::exp(e);
            total += term;
            if (term < total * 0x1p-60) break;
        }
        return total;
    }
    // the same probability by the ratio of consecutive terms: not the same bits, but one division a term
    double estimate(double p)
    {
        const double odds = p / (1.0 - p);
        double term = 1.0, total = 1.0;
        for (int64_t i = k_; i < n_ && term >= total * 0x1p-60; ++i) {
            term *= odds * (double)(n_ - i) / (double)(i + 1);
            total += term;
        }
        return std::exp(choose(k_) + (double)k_ * std::log(p) + (double)(n_ - k_) * std::log1p(-p)) * total;
    }
    // Relative errors of the sum, from the roundings of its exponents (sums of numbers below `size` in magnitude) and
    // of its additions.  Against the true probability, at any p looked at (|log p|, |log q| < 50):
    double eps_any() const { return 0x1p-48 * (log_n_ + 50.0 * (double)n_); }
    // Against the same sum without the roundings that depend on p (its coefficients are what `choose` returns), near p:
    double eps_near(double p) const
    {
        const double size = -((double)(k_ + (int64_t)log_c_.size()) * std::log(p) + (double)(n_ - k_) * std::log1p(-p));
        return 0x1p-52 * (4.0 * size + (double)log_c_.size() + 512.0);
    }

private:
    double choose(int64_t i)
    {
        const size_t at = (size_t)(i - k_);
        if (at >= log_c_.size()) log_c_.push_back(log_n_ - std::lgamma((double)i + 1.0) - std::lgamma((double)(n_ - i) + 1.0));
        return log_c_[at];
    }
    int64_t k_, n_;
    double log_n_;
    std::vector<double> log_c_;
};

// The part of [0, k / n] where P[Binomial(n, p) >= k] has to be compared with alpha by the sum itself: at every p <= lo
// the sum is below alpha, at every hi <= p <= k / n it is not.  Both the probability and the sum with its coefficients
// as computed grow with p (each term does, p being at most k / n), and an evaluation of the sum differs from them by
// the factors above, so one value that clears alpha by four times the error decides for all p on its side.
struct RootBracket { double lo, hi; };

RootBracket bracket_root(UpperTail &tail, int64_t k, int64_t n, double alpha)
{
    const double top = (double)k / (double)n, target = std::log(alpha), eps = tail.eps_any();
    RootBracket b{0.0, 2.0};
    if (!(eps < 1e-2)) return b;
    // secant steps on log P, which is nearly a parabola in p, from about three standard deviations below k / n
    const double sd = std::sqrt(top * (1.0 - top) / (double)n);
    double p0 = top - 3.5 * sd, p1 = top - 3.0 * sd;
    if (!(p0 > 0.0)) { p0 = 0.25 * top; p1 = 0.5 * top; }
    double f0 = std::log(tail.estimate(p0)) - target, f1 = std::log(tail.estimate(p1)) - target, slope = 0.0;
    for (int step = 0; step < 16; ++step) {
        slope = (f1 - f0) / (p1 - p0);
        if (!(slope > 0.0) || !std::isfinite(slope)) return b;
        double p2 = p1 - f1 / slope;
        if (!(p2 > 0.25 * std::min(p0, p1))) p2 = 0.25 * std::min(p0, p1);
        if (!(p2 < top)) p2 = 0.5 * (std::max(p0, p1) + top);
        p0 = p1; f0 = f1;
        p1 = p2; f1 = std::log(tail.estimate(p1)) - target;
        if (std::fabs(f1) < eps) break;
    }
    const double wide = 8.0 * eps / slope;
    if (!(p1 - wide > 0.0 && p1 + wide < top)) return b;
    if (!(tail.estimate(p1 - wide) < alpha * (1.0 - 4.0 * eps) && tail.estimate(p1 + wide) > alpha * (1.0 + 4.0 * eps))) return b;
    b = {p1 - wide, p1 + wide};
    // within these ends the sum's own, smaller, error counts: a step to its root, then an interval around that
    p1 -= (std::log(tail(p1)) - target) / slope;
    const double near = tail.eps_near(p1), narrow = 6.0 * near / slope, lo = p1 - narrow, hi = p1 + narrow;
    if (lo > b.lo && hi < b.hi) {
        if (tail(lo) < alpha * (1.0 - 4.0 * near)) b.lo = lo;
        if (tail(hi) > alpha * (1.0 + 4.0 * near)) b.hi = hi;
    }
    return b;
}

inline int first_max(const int32_t *v, int n)
{
    int arg = 0;
    for (int i = 1; i < n; ++i)
        if (v[i] > v[arg]) arg = i;
    return arg;
}

}  // namespace

// One-sided (1 - alpha) Clopper-Pearson lower bound (Algorithm 1, step 5): the success
// probability at which seeing k or more successes in n trials has probability alpha.
// It follows the kernels on the call's path, on one host thread: what bounds it is calls of exp.  n = 100,000 and
// k = 86,099: 64 sums of 13,901 terms, 5.8 ms, became 17 sums of some 630, 0.08 ms; n = 1,000 and k = 929: 36 -> 17 us.
double lower_conf_bound(int64_t k, int64_t n, double alpha)
{
    if (k <= 0) return 0.0;
    if (k >= n) return std::exp(std::log(alpha) / (double)n);
    // Bisection on [0, k / n].  Points outside the bracket are decided without a sum, the others (about ten of 64) by the
    // sum; once the midpoint is one of the ends, no later step changes anything.
    UpperTail tail(k, n);
    const RootBracket root = bracket_root(tail, k, n, alpha);
    double left = 0.0, right = (double)k / (double)n;
    bool right_decided = false;
    for (int step = 0; step < 64; ++step) {
        const double mid = 0.5 * (left + right);
        if (mid == left || (mid == right && right_decided)) break;
        if (mid <= root.lo || (mid < root.hi && tail(mid, alpha) < alpha)) {
            left = mid;
        } else {
            right = mid;
            right_decided = true;
        }
    }
    return left;
}

// Phi^-1(p) for p >= 1/2 (Algorithm 1, step 7) by bisection of Phi(x) = erfc(-x/sqrt 2)/2 on [0, 9].
double normal_quantile(double p)
{
    double left = 0.0, right = 9.0;
    for (int step = 0; step < 64; ++step) {
        const double mid = 0.5 * (left + right);
        const double cdf = 0.5 * std::erfc(-mid / std::sqrt(2.0));
        if (cdf < p)
            left = mid;
        else
            right = mid;
    }
    return left;
}

// Two-sided exact binomial test of n_a successes out of m at probability 1/2 (Algorithm 2, step 3).  n_a >= m / 2, so
// the terms fall and the sum ends where a term no longer counts (see UpperTail).
double binom_pvalue_half(int64_t n_a, int64_t m)
{
    const double log_m = std::lgamma((double)m + 1.0), log_2 = std::log(2.0);
    double total = 0.0;
    for (int64_t i = n_a; i <= m; ++i) {
        const double log_c = log_m - std::lgamma((double)i + 1.0) - std::lgamma((double)(m - i) + 1.0);
        const double e = log_c - (double)m * log_2;
        if (2 * n_a >= m && e < -760.0) break;
        const double term = std::exp(e);
        total += term;
        if (2 * n_a >= m && term < total * 0x1p-60) break;
    }
    const double pv = 2.0 * total;
    return pv < 1.0 ? pv : 1.0;
}

int32_t decide_certify(const int32_t *counts0, const int32_t *counts, int n_classes, int64_t N,
                       double sigma, double alpha, double *radius, double *p_lower)
{
    const int c_a = first_max(counts0, n_classes);          // step 2: label with the most selection votes
    const int64_t n_a = counts[c_a];                        // step 4: its votes among the N fresh samples
    const double p_a = lower_conf_bound(n_a, N, alpha);     // step 5
    if (p_lower) *p_lower = p_a;
    if (p_a > 0.5) {                                        // steps 6-7
        *radius = sigma * normal_quantile(p_a);
        return c_a;
    }
    *radius = 0.0;                                          // step 8: ABSTAIN
    return -1;
}

namespace {

// floor(p * 2^32) as the table's fixed-point probability, saturated to 32 bits
uint32_t to_fixed32(double p)
{
    const double scaled = std::floor(p * 4294967296.0);
    if (scaled <= 0.0) return 0u;
    return scaled >= 4294967295.0 ? 4294967295u : (uint32_t)scaled;
}

// Theorem 3.2 step 2: the quantile of the discrete Gaussian by lookup, the first level whose cumulative entry reaches p
int32_t table_quantile(const std::vector<uint32_t> &cum, uint32_t p_fx)
{
    const int32_t T = (int32_t)(cum.size() - 1) / 2;
    const int32_t at = (int32_t)(std::lower_bound(cum.begin(), cum.end(), p_fx) - cum.begin());
    return at > 2 * T ? T : at - T;
}

}  // namespace

int32_t decide_certify_integer(const int32_t *counts0, const int32_t *counts, int n_classes, int64_t N, double sigma,
                               double alpha, bool two_sided, int32_t *q, int64_t *q_squared, const uint32_t *table, size_t n_table)
{
    *q = 0; *q_squared = 0;
    const int c_a = first_max(counts0, n_classes);           // Algorithm 1 steps 2, 4, 5, 6
    const double p_a = lower_conf_bound(counts[c_a], N, alpha);
    if (!(p_a > 0.5)) return -1;
    std::vector<uint32_t> cum;
    if (table) cum.assign(table, table + n_table);
    else noise_table(sigma, cum);
    const int32_t q_a = table_quantile(cum, to_fixed32(p_a));
    if (!two_sided) {                                         // Theorem 3.2 steps 2-3: radius and squared radius in pixel levels
        *q = q_a;
        *q_squared = (int64_t)q_a * q_a;
        return c_a;
    }
    // Theorem 3.1: the runner-up's upper bound enters as well; d = q_A - q_B is twice the radius
    int64_t n_b = 0;
    for (int c = 0; c < n_classes; ++c)
        if (c != c_a && counts[c] > n_b) n_b = counts[c];
    const double p_b = 1.0 - lower_conf_bound(N - n_b, N, alpha);
    if (p_a < p_b) return -1;
    const int32_t d = q_a - table_quantile(cum, to_fixed32(p_b));
    *q = d;
    *q_squared = (int64_t)d * d;
    return c_a;
}

int32_t decide_predict(const int32_t *counts, int n_classes, double alpha)
{
    const int c_a = first_max(counts, n_classes);
    const int64_t n_a = counts[c_a];
    int64_t n_b = 0;
    bool seen = false;
    for (int c = 0; c < n_classes; ++c) {
        if (c == c_a) continue;
        if (!seen || counts[c] > n_b) { n_b = counts[c]; seen = true; }
    }
    return binom_pvalue_half(n_a, n_a + n_b) <= alpha ? c_a : -1;
}

int noise_halfwidth(double sigma)
{
    return (int)std::ceil(7.0 * (255.0 * sigma));
}

// cum[z + T] = floor(2^32 * P[Z <= z]) for the discrete Gaussian of Eq. 2 on the integer pixel
// levels with std 255*sigma, support cut at +-T; the last entry is 2^32 - 1.  (One exponential for z and -z, and floors by
// conversion: 31 -> 21 us for sigma = 1, which every call with a new sigma pays.)
void noise_table(double sigma, std::vector<uint32_t> &cum)
{
    const double s = 255.0 * sigma;
    const int T = noise_halfwidth(sigma);
    const double two_var = 2.0 * s * s;
    std::vector<double> weight((size_t)(2 * T + 1));
    double norm = 0.0;
    for (int z = 0; z <= T; ++z) weight[(size_t)(T + z)] = weight[(size_t)(T - z)] = std::exp(-(double)((int64_t)z * z) / two_var);
    for (const double w : weight) norm += w;                                 // from -T on
    cum.resize((size_t)(2 * T + 1));
    double running = 0.0;
    for (int z = -T; z <= T; ++z) {
        running += weight[(size_t)(z + T)];
        const double scaled = running / norm * 4294967296.0;
        cum[(size_t)(z + T)] = scaled >= 4294967295.0 ? 4294967295u : (uint32_t)(int64_t)scaled;      // floor: not negative
    }
    cum[(size_t)(2 * T)] = 4294967295u;
}

// The same table form for the rounded continuous Gaussian: delta = round(255 sigma g), g ~ N(0, 1), the noise of the
// paper's comparison method that perturbs with continuous noise and then quantises (Sec. 4.1, comparison methods):
// cum[z + T] = floor(2^32 * Phi((z + 1/2) / (255 sigma))).
void noise_table_rounded(double sigma, std::vector<uint32_t> &cum)
{
    const double s = 255.0 * sigma;
    const int T = noise_halfwidth(sigma);
    cum.resize((size_t)(2 * T + 1));
    for (int z = -T; z <= T; ++z) {
        const double cdf = 0.5 * std::erfc(-(((double)z + 0.5) / s) / std::sqrt(2.0));
        const double scaled = cdf * 4294967296.0;
        cum[(size_t)(z + T)] = scaled >= 4294967295.0 ? 4294967295u : (uint32_t)(int64_t)scaled;
    }
    cum[(size_t)(2 * T)] = 4294967295u;
}

}  // namespace isc
