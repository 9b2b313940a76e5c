// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace kvdro {

// Samples of one class are staged for the grid kernel in regions of a multiple of kPadSamples, in one
// of two forms, the same for every class of a context.
//  - Quads, where every support is at most kExactMaxL: four samples a <= b <= c <= d (neighbours of the sorted
//    class) in 16 bytes as the integers {a + b + c + d, b + c, d - a, (c + d) - (a + b)}.  The class's last
//    quad starts with zeros where its samples are fewer, further quads are zeros; the exact kernel
//    subtracts their known |0 - c| per cell.
//  - (x, x) float pairs otherwise, so that one 128-bit shared-memory load yields the packed operands of two
//    samples, padded with NaN pairs, which contribute exactly zero to the per-term kernels' excess sums
//    (max(NaN, 0) = 0 in PTX max.f32 / max.f64).
constexpr int kPadSamples = 128;

// Error bits reported by kernels in ctx->d_err[1].
constexpr int kErrTimeout = 1;

struct SortArgs {
    const int32_t* lengths;     // caller samples (device), CSR by class
    const int64_t* offsets;     // [K+1]
    const int32_t* L;           // [K]
    const int64_t* hist_off;    // [K+1] start of class k's cumulative-count array (L_k + 1 entries)
    const int64_t* pair_off;    // [K+1] start of class k's padded region, in samples
    const int32_t* hist_blocks; // [K+1] prefix of histogram blocks per class
    const int32_t* exp_blocks;  // [K+1] prefix of expand blocks per class
    int32_t* hist;              // [hist_off[K]] counts, zero before the histogram
    int32_t* cum;               // [hist_off[K]] cumulative counts; may be `hist` (must, past scan_direct's tiles)
    int64_t* csum;              // [hist_off[K]] cumulative sums sum_{x <= v} x, or nullptr to skip
    int64_t* sumx;              // [K] sum of samples per class (written by the scan)
    int32_t* sorted;            // [offsets[K]]
    void* staged;               // pair_off[K] samples, 4 bytes each as quads or 8 as (x, x) pairs
    int32_t* err;               // [0] += out-of-range samples
    int64_t* tile_tot;          // [K][scan_tiles][2] scan tile totals (count, sum of v h[v])
    int32_t* tile_lo;           // [exp_blocks[K] + K] per class from exp_blocks[k] + k: the bin of the
                                // first position of each expansion tile, then the bin of position N - 1
    double* inv_n;              // [K] 1 / N written by the expansion, or nullptr to skip (may lie over
                                // tile_tot, which the expansion does not read)
    int32_t scan_tiles;         // scan tiles of the largest class: ceil((max L + 1) / scan tile bins)
    int32_t quads;          // the staged form
    int32_t K;
};

// Launchers (sort.cu)
// prefix[K + 1] of histogram blocks per class, sized to the current device (sort.cu)
cudaError_t hist_block_prefix(const int64_t* N, int32_t K, int32_t* prefix);
cudaError_t launch_histogram(const SortArgs& a, int32_t nblocks, cudaStream_t s);
cudaError_t launch_scan(const SortArgs& a, cudaStream_t s);
cudaError_t launch_expand(const SortArgs& a, int32_t nblocks, cudaStream_t s);
cudaError_t launch_gather_quantiles(const int32_t* sorted, const int64_t* offsets, const int32_t* rank, int32_t K,
                                    int32_t F, int32_t* out, cudaStream_t s);

// F32: per-term FP32 excess sums folded into FP64.  F64: per-term FP64.  EXACT: an exact integer
// threshold per cell, then an exact sum of |x - c| over the samples (four at a time), combined in FP64.
// ENVELOPE: the same sums in O(1) per cell from cumulative counts and sums (not per term).
enum class Prec { F32 = 0, F64 = 1, EXACT = 2, ENVELOPE = 3 };
constexpr int32_t kExactMaxL = 1 << 22;  // the exact kernel's integer sums need L <= 2^22

struct FinalizeArgs {
    const unsigned long long* keys;  // [M][E][K] argmin keys
    const void* cost;           // FP64: cost buffer to read min_cost from; FP32 unused
    const int32_t* r;
    const int32_t* L_in;
    const int64_t* N;
    const int32_t* cdf;
    const int64_t* hist_off;
    int32_t K, R, E, M;
    int32_t* r_idx;             // [M][E][K]
    void* min_cost;             // [M][E][K]
    double* fhat;               // [M][E][K]
};

struct GridArgs {
    const void* staged;         // the padded samples
    const int64_t* pair_off;    // [K+1] in samples
    int32_t quads;          // the staged form
    const int64_t* N;           // [K]
    const double* inv_n;        // [K] 1 / N
    const int64_t* sumx;        // [K]
    const int32_t* L;           // [K]
    const int32_t* L_in;        // [K]
    const int32_t* cdf;         // cumulative counts, class k at hist_off[k]
    const int64_t* csum;        // cumulative sample sums, same layout (envelope mode)
    const int64_t* hist_off;    // [K+1]
    const int32_t* r;           // [R]
    const double* lam;          // [NL]
    const double* eps;          // [E]
    const double* cp;           // [M]
    const double* cw;           // [M]
    int32_t K, R, NL, E, M;
    int32_t LT;                 // lam tiles per CTA (FP32 and FP64 kernels)
    int32_t RG;                 // r groups per CTA (FP32 and FP64 kernels)
    int32_t rows;               // r values per CTA
    int32_t passes;             // over the samples (exact kernel)
    int32_t chunk;              // samples per staged chunk (exact kernel)
    int32_t r_blocks;           // CTAs per (m, k)
    int32_t m0, m_count;        // regime range covered by this launch
    int32_t f32_out;            // exact kernel: write S, cost and the argmin keys as FP32 (FP32 mode)
    void* S_out;                // optional [M][K][R][NL]
    void* cost_out;             // [M][E][K][R] (caller's, or scratch for FP64 min_cost)
    int32_t* lam_idx_out;       // optional [M][E][K][R]
    unsigned long long* keys;   // [M][E][K] argmin keys (initialised to all ones)
    int32_t* err;               // [1] |= kErrTimeout
    // Bounded waits and their test hook, per launch: wait_ns bounds each wait on a staged chunk
    // (0: the default of about 2 s); test_skip_chunk >= 0 leaves that chunk's copy unissued, so
    // the waits on it run out (-1 in production).
    long long wait_ns;
    int32_t test_skip_chunk;
    // With `done` ([M][K] words, all ones before the launch) the last CTA of each (regime, class) finalises
    // its rows by `fin`; without, the caller launches the finalisation.
    uint32_t* done;
    FinalizeArgs fin;
};

// grid.cu
// Launch shape of the grid kernel for one (precision, grid) problem: which compiled variant, its
// r values and warps per CTA, CTAs per (regime, class), dynamic shared memory.
struct GridShape {
    int variant;       // index of the compiled kernel instantiation
    int LT, RG;        // lam tiles and r groups per CTA (FP32 and FP64 kernels: LT * RG warps)
    int rows;          // r values per CTA
    int passes = 1;    // over the samples, and samples per staged chunk (exact kernel)
    int chunk = 0;
    int threads;
    int r_blocks;      // CTAs per (m, k)
    size_t smem;
};
// K, M: classes and regimes that the request evaluates; sms: of the device
GridShape grid_shape(Prec p, int32_t R, int32_t NL, int32_t E, int32_t K, int32_t M, int sms);
cudaError_t sm_count(int* sms);  // of the current device (sort.cu)
cudaError_t grid_prepare(Prec p);  // per-device attributes of every variant of p, and F32's finalisation loaded
// Launches over regimes [a.m0, a.m0 + a.m_count); fills a.LT, a.RG, a.r_blocks from `sh`.
cudaError_t launch_grid(Prec p, const GridShape& sh, GridArgs a, cudaStream_t s);
cudaError_t launch_finalize(Prec p, const FinalizeArgs& a, cudaStream_t s);

// setup.cu: one launch that writes `bytes` of host parameters to dst (setup_fits) and fills two arrays of
// 32-bit words (16-byte aligned; 0 words to skip)
struct Fill {
    uint32_t* p;
    int64_t words;
    uint32_t value;
};
bool setup_fits(size_t bytes);
cudaError_t setup_prepare();  // loads every variant on the current device
cudaError_t launch_setup(const void* payload, size_t bytes, void* dst, const Fill& f0, const Fill& f1, cudaStream_t s);

// dual.cu: exact minimisation over gamma >= 0 per (regime, radius, class, reservation)
struct DualArgs {
    const int32_t* cdf;         // cumulative counts, class k at hist_off[k]
    const int64_t* csum;        // cumulative sums, same layout
    const int64_t* hist_off;    // [K+1]
    const int64_t* N;           // [K]
    const double* inv_n;        // [K] 1 / N
    const int64_t* sumx;        // [K]
    const int32_t* L;           // [K]
    const int32_t* L_in;        // [K]
    const int32_t* r;           // [R]
    const double* eps;          // [E]
    const double* cp;           // [M]
    const double* cw;           // [M]
    int32_t K, R, E, M;
    double* cost;               // [M][E][K][R] (needed for min_cost)
    double* gamma;              // optional [M][E][K][R]
    unsigned long long* keys;   // [M][E][K], initialised to all ones
};
dim3 dual_grid(int64_t cells);
cudaError_t launch_dual(const DualArgs& a, cudaStream_t s);

#ifdef __CUDACC__
// Every FP64-pipe instruction -- add, multiply, FMA, compare, minimum and each conversion from or to
// double -- runs at 1.6 to 1.9 lanes per clock per SM on this part, a warp's 32 lanes in about 64
// cycles of its scheduler's share, where an integer instruction takes 2.  The per-cell code
// therefore compares, converts and takes minima of doubles on their bit patterns and leaves to the
// FP64 pipe only the roundings that the results are made of.
__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ bool dpos(double v) { return dbits(v) > 0; }  // v > 0 (v not NaN)
// min(a, b) for a, b >= 0, not NaN
__device__ __forceinline__ double dmin_nonneg(double a, double b) { return dbits(a) < dbits(b) ? a : b; }

// (double)v, v >= 0: normalised by its leading zeros and packed, exact below 2^53 (every count and
// sum of ordinary problems); the conversion instruction rounds the larger ones.
__device__ __forceinline__ double to_double(long long v) {
    if (v >= (1ll << 53)) return (double)v;
    const int lz = __clzll(v);                                    // 64 for v = 0
    const unsigned long long m = (unsigned long long)v << (lz & 63);  // leading one at bit 63
    const unsigned long long b = ((unsigned long long)(1086 - lz) << 52) + ((m >> 11) & 0xFFFFFFFFFFFFFull);
    return __longlong_as_double(v == 0 ? 0ll : (long long)b);
}
__device__ __forceinline__ double to_double(int v) { return to_double((long long)v); }

// Magnitude of a double whose exponent lies in [-100, 100], cut to a float: relative error below 2^-23.
__device__ __forceinline__ bool narrowable(long long b) {
    const unsigned e = (unsigned)(b >> 52) & 0x7ff;
    return e - (1023u - 100u) <= 200u;
}
__device__ __forceinline__ float narrow(long long b) {
    return __uint_as_float((unsigned)((b & 0x7fffffffffffffffll) >> 29) - (896u << 23));
}

// Order key of a double: equal for equal values (-0 is taken as +0), ordered as the values are, and above them
// all for a NaN (a sum past the double range, whose own sign bit is set), which is no minimum.
__device__ __forceinline__ long long order_key(double v) {
    long long b = __double_as_longlong(v);
    if (b == (long long)0x8000000000000000ull) b = 0;
    if (((unsigned long long)b << 1) > 0xffe0000000000000ull) return 0x7fffffffffffffffll;
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// The smallest key of the warp, in every lane.
__device__ __forceinline__ unsigned long long warp_min(unsigned long long key) {
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o);
        key = other < key ? other : key;
    }
    return key;
}

// The offset d = (c_p - mu) L - (c_p + c_w) eta of a cell's excess kappa x + d, evaluated as
// c_p (L - eta) - (mu L + c_w eta): L - eta is an exact integer and every product is rounded once,
// so a large c_p never swallows a small mu or c_w (the first form cancels to 0 at eta = L when
// mu and c_w are far below c_p, though d is then -(mu + c_w) L).  At the saturated multiplier
// mu = c_p the L terms vanish exactly and d = -(c_p + c_w) eta.  Every rounding is spelled out
// (no contraction left to the compiler), so each call site gets the same d bit for bit: a
// kernel that classifies samples twice at one multiplier (the dual's slope and value) must see
// the same threshold both times.  What does not depend on mu is formed once per reservation.
struct RowOffset {
    double cw_eta, cp_le, d_sat;
};
__device__ __forceinline__ RowOffset row_offset(double cp, double cw, int L, int eta) {
    RowOffset r;
    const double e = to_double(eta);
    r.cw_eta = __dmul_rn(cw, e);
    r.cp_le = __dmul_rn(cp, to_double(L - eta));
    r.d_sat = -__fma_rn(cp, e, r.cw_eta);
    return r;
}
__device__ __forceinline__ double excess_offset(const RowOffset& r, double cp, double mu, double Ld) {
    return dbits(mu) == dbits(cp) ? r.d_sat : __dsub_rn(r.cp_le, __fma_rn(mu, Ld, r.cw_eta));
}

// The same excess about the reservation: kappa x + d = kappa (x - eta) + W(eta), with
//   W(eta) = (c_p - mu)(L - eta) - (c_w - nu) eta,
// for the per-term kernels, which add max(excess, 0) sample by sample.  x - eta is an exact
// integer; the two cost differences are exact or rounded once and each product is rounded once,
// so W(eta) is exactly 0 where the excess vanishes identically on one side of eta -- at the
// saturated multiplier (mu = c_p, nu = c_w), at eta = L with nu = c_w, at eta = 0 with mu = c_p --
// and a cell whose every term is zero sums to exactly zero.  (kappa x + d with the rounded d leaves
// the rounding error of mu L at x = L, which max(., 0) can pass on.)  The differences are at most
// the costs, so W(eta) is never less accurate than d.
__device__ __forceinline__ double excess_at_eta(double cp, double cw, double mu, double nu, double L, double eta) {
    return fma(__dsub_rn(cp, mu), L - eta, -__dmul_rn(__dsub_rn(cw, nu), eta));
}

// sum_n phi(x_n) with every sample on its own branch: V = c_w eta - nu x for the n - cnt samples
// below the cell's first active point, U = c_p (L - eta) - mu (L - x) for the cnt samples from it
// on.  The caller passes exact integer sums: sx_below = sum x below the point, dist_above =
// sum (L - x) from it on.  Nothing cancels beyond what each branch holds itself, whatever the
// ratios of c_p, c_w and the multiplier (V + max(U - V, 0) loses everything to cancellation
// when nu is many orders above the result).
// c i - m j for integers i, j held exactly in doubles: the rounding error of c i is recovered by
// one FMA, so the difference is rounded about once however closely the two products agree
// (forming both products first leaves only their rounding errors when they agree to 16 digits).
__device__ __forceinline__ double diff_of_products(double c, double i, double m, double j) {
    const double p = __dmul_rn(c, i);
    const double e = fma(c, i, -p);  // c i - p exactly, barring underflow
    return fma(-m, j, p) + e;
}

// A branch without samples is skipped: it would add exactly zero.
__device__ __forceinline__ double branch_sum(double cp, double cw, double mu, double nu, int L, int eta, long long n,
                                             long long cnt, long long sx_below, long long dist_above) {
    double v = 0.0;
    if (cnt < n) v = diff_of_products(cw, to_double((long long)eta * (n - cnt)), nu, to_double(sx_below));
    if (cnt > 0) {
        const double u = diff_of_products(cp, to_double((long long)(L - eta) * cnt), mu, to_double(dist_above));
        v = cnt < n ? __dadd_rn(v, u) : u;
    }
    return v;
}

// The per-term kernels sum phi as a base plus excesses: sum V + sum max(U - V, 0), or
// sum U + sum max(V - U, 0).  Each excess cancels, in the total, against the base's slope term
// (nu sum x, or mu sum (L - x)) on the samples it covers, so a cell takes the base whose slope
// is the smaller: U when nu > mu.  U - V = kappa x + d, so the U base negates kappa and d.
__device__ __forceinline__ bool use_u_split(double mu, double nu) { return nu > mu; }

// The first active support point of a cell: the smallest integer t in [0, L] with
// kappa * t + d > 0, or L + 1 when there is none (kappa >= 0, so the condition is monotone in
// t).  One FMA gives the sign of kappa * t + d exactly, so each test is exact.  settle_active finds
// t from the FP32 quotient -d / kappa (off by a few units at most for L <= 2^24), corrected by at
// most 8 tests each way; should that not settle it, the FP64 quotient is corrected the same way.
static __device__ __noinline__ int settle_active(double kappa, double d, int L) {
    if (!(fma(kappa, (double)L, d) > 0.0)) return L + 1;
    // here t is in [1, L]: kappa (t - 1) + d <= 0 < kappa t + d
    auto settle = [&](double q, int64_t& t) {
        const double e = floor(q) + 1.0;
        t = e < 1.0 ? 1 : (e > (double)L ? L : (int64_t)e);
        for (int i = 0; i < 8 && t > 1 && fma(kappa, (double)(t - 1), d) > 0.0; i++) t--;
        for (int i = 0; i < 8 && t < L && !(fma(kappa, (double)t, d) > 0.0); i++) t++;
        return (t == 1 || !(fma(kappa, (double)(t - 1), d) > 0.0)) && fma(kappa, (double)t, d) > 0.0;
    };
    int64_t t;
    if (settle((double)__fdiv_rn(-(float)d, (float)kappa), t)) return (int)t;
    (void)settle(-d / kappa, t);
    return (int)t;
}
// Almost every cell needs no FP64 instruction for it.  |d| and kappa cut to floats are at most 2^-23
// below their values and the quotient is within 2 ulp of theirs, so x0 = -d / kappa lies within
// q (1 +- 3 x 2^-23), inside q (1 +- 2^-21) after the rounding of the two ends.  Below 2^20 that
// interval is shorter than one and holds at most one integer n: with none, t is its floor plus one;
// with n, the sign at n decides.
__device__ __forceinline__ int first_active(double kappa, double d, int L) {
    const long long db = dbits(d), kb = dbits(kappa);
    if (db > 0) return db <= 0x7ff0000000000000ll ? 0 : L + 1;  // NaN is not positive
    if (kb <= 0) return L + 1;
    if ((db << 1) == 0) return 1;
    if (!narrowable(db) || !narrowable(kb)) return settle_active(kappa, d, L);
    const float q = __fdividef(narrow(db), narrow(kb));
    const float lo = fmaf(q, -0x1p-21f, q), hi = fmaf(q, 0x1p-21f, q);
    if (lo >= (float)L) return L + 1;  // (float)L is exact: L <= 2^24
    if (!(q < 0x1p20f)) return settle_active(kappa, d, L);
    const int n_lo = __float2int_rd(lo), n = __float2int_rd(hi);
    int t = n + 1;
    if (n_lo != n && dpos(fma(kappa, to_double(n), d))) t = n;
    return min(t, L + 1);
}
#endif

}  // namespace kvdro
