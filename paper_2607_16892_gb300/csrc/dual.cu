// The exact dual value of App. A (eq. app_kantorovich, gamma >= 0 not restricted to a grid):
//   cost(eta, eps) = min_{gamma >= 0} g(gamma),  g(gamma) = gamma eps + S(eta, gamma).
// g is convex and piecewise linear in gamma (each sample's supremum is a maximum of lines in
// gamma).  For gamma >= max(c_p, c_w) moving mass never pays and S is the empirical cost, so g
// rises with slope eps and the minimiser lies in [0, max(c_p, c_w)].  Every evaluation of S and of
// its derivative is O(1) from the class's cumulative counts and sums: with mu = min(gamma, c_p),
// nu = min(gamma, c_w), kappa = mu + nu and d = (c_p - mu) L - (c_p + c_w) eta, the samples with a
// positive excess kappa x + d (where U beats V) are x >= t for an integer threshold t, and
//   N S = c_w eta #{x < t} - nu sum_{x < t} x + c_p (L - eta) #{x >= t} - mu sum_{x >= t} (L - x),
//   N g' = N eps - nu' sum_{x < t} x - mu' sum_{x >= t} (L - x),  nu' = [gamma < c_w], mu' = [gamma < c_p].
// One thread per (regime, radius, class, reservation) closes a bracket on the sign of that right
// derivative down to two adjacent doubles, over the bit patterns of the nonnegative doubles (ordered
// as their values), so a kink at c_w = 1e-250 under c_p = 2 is found as surely as one near c_p.
//
// The derivative depends on gamma through t alone on each side of min(c_p, c_w), and t is monotone in
// gamma there, so the search runs over the integers t first (at most log2 L steps, no floating
// point), then gamma is where the excess at the last crossed value v vanishes, a quotient, and a few
// tests of the sign around it close the bracket.  Bisection on gamma alone takes 63 tests of some 30
// FP64-pipe instructions each: 33.3 ms for 8 classes x 200,000 samples x 2048 r x 16 radii x 32 regimes, where
// this takes 1.67 ms with the FP64 pipe 86 % busy.
#include <float.h>
#include <math.h>

#include "kvdro_internal.cuh"

namespace kvdro {
namespace {

constexpr int kDualThreads = 128;

// One (regime, class, reservation): the class's cumulative arrays and what the costs fix.
struct Cell {
    const int32_t* C;   // cumulative counts, L + 1 entries
    const int64_t* CS;  // cumulative sums
    long long N, sumx;
    int L, eta;
    double cp, cw, Ld;
    RowOffset row;
};

// count and sum of the samples below t, t in [0, L + 1]
__device__ __forceinline__ void below(const Cell& c, int t, long long& n, long long& s) {
    n = t >= 1 ? (long long)c.C[t - 1] : 0;
    s = t >= 1 ? (long long)c.CS[t - 1] : 0;
}

// The first active point at gamma, from which U beats V.
__device__ __forceinline__ int split_at(const Cell& c, double gam) {
    const double mu = dmin_nonneg(gam, c.cp);
    return first_active(__dadd_rn(mu, dmin_nonneg(gam, c.cw)), excess_offset(c.row, c.cp, mu, c.Ld), c.L);
}

// What the right derivative loses to the samples when the active ones start at t, times N, with nu' and
// mu' given: exact integers.
__device__ __forceinline__ long long drop_at(const Cell& c, int t, bool nu1, bool mu1) {
    long long n, s;
    below(c, t, n, s);
    return (nu1 ? s : 0) + (mu1 ? (long long)c.L * (c.N - n) - (c.sumx - s) : 0);
}

// g(gamma) = gamma eps + S(eta, gamma), every sample on its own branch of phi.
__device__ __forceinline__ double value_at(const Cell& c, double eps, double gam, double inv_n) {
    long long n, s;
    below(c, split_at(c, gam), n, s);
    const long long cnt = c.N - n;
    return fma(gam, eps, __dmul_rn(branch_sum(c.cp, c.cw, dmin_nonneg(gam, c.cp), dmin_nonneg(gam, c.cw), c.L, c.eta, c.N,
                                              cnt, s, (long long)c.L * cnt - (c.sumx - s)), inv_n));
}

// gamma at which the excess at the sample value v vanishes, on one side of min(c_p, c_w)
// (nu1, mu1: nu = gamma, mu = gamma there), about to the last bit: a difference of products over an
// integer, by two Newton corrections of the FP32 reciprocal's quotient.
__device__ __forceinline__ double crossing(const Cell& c, int v, bool nu1, bool mu1, int& den) {
    double num;
    if (nu1 && mu1) {  // gamma (2 v - L) = c_w eta - c_p (L - eta)
        num = diff_of_products(c.cw, to_double(c.eta), c.cp, to_double(c.L - c.eta));
        den = 2 * v - c.L;
    } else if (mu1) {  // gamma (L - v) = c_p (L - eta) - c_w (eta - v)
        const double s = to_double(abs(c.eta - v));
        num = diff_of_products(c.cp, to_double(c.L - c.eta), c.cw, c.eta < v ? -s : s);
        den = c.L - v;
    } else {  // gamma v = c_w eta - c_p (v - eta)
        const double s = to_double(abs(v - c.eta));
        num = diff_of_products(c.cw, to_double(c.eta), c.cp, v < c.eta ? -s : s);
        den = v;
    }
    if (den == 0) return 0.0;
    if (den < 0) num = -num;
    const double d = to_double(abs(den)), r = __longlong_as_double(((long long)__float_as_int(__frcp_rn((float)abs(den))) << 29) + (896ll << 52));
    double q = __dmul_rn(num, r);
    q = fma(fma(-d, q, num), r, q);
    return fma(fma(-d, q, num), r, q);
}

__global__ void __launch_bounds__(kDualThreads, 6) k_dual(const DualArgs a) {
    const int64_t i = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t total = (int64_t)a.M * a.E * a.K * a.R;
    const bool valid = i < total;
    int64_t t = valid ? i : total - 1;
    const int ri = (int)(t % a.R);
    t /= a.R;
    const int k = (int)(t % a.K);
    t /= a.K;
    const int e = (int)(t % a.E);
    const int m = (int)(t / a.E);
    Cell c;
    c.C = a.cdf + a.hist_off[k];
    c.CS = a.csum + a.hist_off[k];
    c.N = a.N[k];
    c.sumx = a.sumx[k];
    c.L = a.L[k];
    c.eta = a.r[ri] - a.L_in[k];
    c.cp = a.cp[m];
    c.cw = a.cw[m];
    c.Ld = to_double(c.L);
    c.row = row_offset(c.cp, c.cw, c.L, c.eta);
    const double eps = a.eps[e], inv_n = a.inv_n[k];
    // The derivative's sign is that of eps N - drop (eps N rounded once).  Drops are integers, at most
    // N L: below 2^53 they compare as integers with floor(eps N), above as doubles.
    const double eps_n = __dmul_rn(eps, to_double(c.N));
    const bool small_drops = c.N <= (1ll << 53) / c.L;
    const long long limit = eps_n >= 0x1p62 ? (1ll << 62) : __double2ll_rd(eps_n);
    auto enough = [&](long long drop) { return small_drops ? drop <= limit : eps_n >= (double)drop; };
    auto rising = [&](double gam, int at) {  // right derivative >= 0 at gamma, whose first active point is `at`
        return enough(drop_at(c, at, dbits(gam) < dbits(c.cw), dbits(gam) < dbits(c.cp)));
    };

    double lo = 0.0, hi = 0.0;
    const int t_zero = split_at(c, 0.0);
    if (dbits(c.cp) > 0 || dbits(c.cw) > 0) {
        if (!rising(0.0, t_zero)) {
            // g falls at `lo` and rises at `hi`: one side of min(c_p, c_w)
            const double c_min = dmin_nonneg(c.cp, c.cw);
            hi = dbits(c.cp) < dbits(c.cw) ? c.cw : c.cp;
            int t_lo = t_zero;
            if (dbits(c_min) > 0 && dbits(c_min) < dbits(hi)) {
                const int t_mid = split_at(c, c_min);
                if (rising(c_min, t_mid)) hi = c_min;
                else { lo = c_min; t_lo = t_mid; }
            }
            long long lb = dbits(lo), hb = dbits(hi);
            // the last double below hi: if g still falls there, the minimum is at hi
            if (hb - lb > 1) {
                const double last = __longlong_as_double(hb - 1);
                int t_hi = split_at(c, last);
                if (!rising(last, t_hi)) {
                    lb = hb - 1;
                } else {
                    hb = hb - 1;
                    // g falls at t_lo and rises at t_hi: halve between them
                    const bool nu1 = lb < dbits(c.cw), mu1 = lb < dbits(c.cp);
                    while (abs(t_hi - t_lo) > 1) {
                        const int mid = (t_lo + t_hi) / 2;
                        if (enough(drop_at(c, mid, nu1, mu1))) t_hi = mid;
                        else t_lo = mid;
                    }
                    // The first active point crosses v = min(t_lo, t_hi) where the excess at v changes sign,
                    // so g rises when v is active as it is at t_hi.  From the quotient the tests step
                    // outwards by what the offset's rounding is worth in gamma, then eight times as far,
                    // and halve between.
                    const int v = min(t_lo, t_hi);
                    const bool active_rises = t_hi <= v;
                    const double vd = to_double(v);
                    auto rises = [&](double g) {
                        const double mu = mu1 ? g : c.cp, nu = nu1 ? g : c.cw;
                        return dpos(fma(__dadd_rn(mu, nu), vd, excess_offset(c.row, c.cp, mu, c.Ld))) == active_rises;
                    };
                    int den;
                    long long x = dbits(crossing(c, v, nu1, mu1, den));
                    x = x < lb + 1 ? lb + 1 : (x > hb - 1 ? hb - 1 : x);
                    auto expo = [](double w) { return (int)(dbits(w) >> 52); };
                    const int unit = max(expo(c.row.cp_le), expo(c.row.cw_eta)) - (int)(x >> 52) - (31 - __clz(abs(den) | 1));
                    long long step = 1ll << min(max(unit, 0), 40);
                    bool out = true, first = true, up = false;
                    while (hb - lb > 1) {
                        const bool p = rises(__longlong_as_double(x));
                        if (p) hb = x;
                        else lb = x;
                        if (first) { up = p; first = false; }
                        else if (p != up) out = false;
                        if (out) {
                            x = up ? hb - step : lb + step;
                            step = min(step, 1ll << 57) << 3;  // at most 2^60
                            out = x > lb && x < hb;
                        }
                        if (!out) x = lb + (hb - lb) / 2;
                    }
                }
            }
            lo = __longlong_as_double(lb);
            hi = __longlong_as_double(hb);
        }
    }
    // g is linear between kinks: the better end of the final bracket is the minimum
    double best_g = value_at(c, eps, lo, inv_n), best_gam = lo;
    if (dbits(hi) > dbits(lo)) {
        const double g_hi = value_at(c, eps, hi, inv_n);
        if (order_key(g_hi) < order_key(best_g)) { best_g = g_hi; best_gam = hi; }
    }
    // Every g is at least the empirical cost (1/N) sum Q(eta, x_n): the empirical distribution
    // lies in the ball, and phi >= Q(eta, x) at every gamma.  That bound is exact from integer
    // sums, whereas g near a kink sums branches many orders above it when c_p or c_w is extreme;
    // at eps = 0 it is the value itself.
    {
        long long n, s;
        below(c, c.eta + 1, n, s);  // the samples up to eta
        const double emp = __dmul_rn(fma(c.cw, to_double((long long)c.eta * n - s),
                                         __dmul_rn(c.cp, to_double(c.sumx - s - (long long)c.eta * (c.N - n)))), inv_n);
        if (order_key(best_g) < order_key(emp)) best_g = emp;
    }
    const size_t row = ((size_t)m * a.E + e) * a.K + k;
    if (valid) {
        if (a.cost) a.cost[row * a.R + ri] = best_g;
        if (a.gamma) a.gamma[row * a.R + ri] = best_gam;
    }
    const long long gb = dbits(best_g);
    const bool above = gb > 0 && gb <= 0x7ff0000000000000ll;  // best_g > 0
    const unsigned long long key = ((unsigned long long)(above ? gb : 0ll) & ~0xFFFFFull) | (unsigned long long)ri;
    // one atomic per warp where its lanes hold one row of r values (a lane past the end repeats the last cell)
    if (__all_sync(0xffffffffu, row == __shfl_sync(0xffffffffu, row, 0))) {
        const unsigned long long low = warp_min(key);
        if ((threadIdx.x & 31) == 0) atomicMin(a.keys + row, low);
    } else {
        atomicMin(a.keys + row, key);
    }
}

}  // namespace

// Rows of 2^31 - 1 blocks; lanes of the last one past the cells repeat the last cell.
dim3 dual_grid(int64_t cells) {
    const int64_t blocks = (cells + kDualThreads - 1) / kDualThreads, x = blocks < 0x7fffffffLL ? blocks : 0x7fffffffLL;
    return dim3((unsigned)x, (unsigned)((blocks + x - 1) / x));
}

cudaError_t launch_dual(const DualArgs& a, cudaStream_t s) {
    const int64_t total = (int64_t)a.M * a.E * a.K * a.R;
    if (total <= 0) return cudaErrorInvalidConfiguration;
    k_dual<<<dual_grid(total), kDualThreads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace kvdro
