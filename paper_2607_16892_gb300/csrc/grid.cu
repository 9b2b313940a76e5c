// Grid evaluation of the worst-case reservation cost (the hot path) and its reductions.
//
// What is summed.  For class k (samples x_n in [0, L], count N), regime (c_p, c_w), reservation
// r with eta = r - L_in in [0, L], and multiplier lam >= 0, the per-sample supremum of App. A
// Step 4 is the maximum of four affine functions of x:
//   l1 = c_p (x - eta), l2 = c_w (eta - x)            (the two branches of Q(eta, x))
//   l3 = Q(eta, 0) - lam x = c_w eta - lam x          (sample moved to xi = 0)
//   l4 = Q(eta, L) - lam (L - x) = c_p (L - eta) - lam (L - x)   (moved to xi = L)
// Since l3 - l2 = (c_w - lam) x and l4 - l1 = (c_p - lam)(L - x), with x and L - x >= 0:
//   max(l2, l3) = V(x) = c_w eta - nu x,           nu = min(lam, c_w)
//   max(l1, l4) = U(x) = c_p (L - eta) - mu (L - x),  mu = min(lam, c_p)
// so phi = max(U, V) = V + max(W, 0) with W = U - V = kappa x + d,
//   kappa = mu + nu,   d = (c_p - mu) L - (c_p + c_w) eta.
// Summing over the class: sum_n phi_n = N c_w eta - nu sum_n x_n + sum_n max(kappa x_n + d, 0).
// Three forms of that sum:
//  - FP32 and FP64 per term: the excess max(kappa x + d, 0) term by term on the base V, or
//    max(-(kappa x + d), 0) on the base U when nu > mu, whichever cancels less (use_u_split).  The
//    excess is evaluated about the reservation, kappa (x - eta) + W(eta) (excess_at_eta), so that
//    it is exactly zero wherever it vanishes identically on one side of eta.  FP64: one fused
//    multiply-add, one max and one add per sample and cell.  FP32: one saturating fused
//    multiply-add on the excess scaled by a power of two (the clamp to [0, 1] is the max) and half
//    a packed add per sample and cell.
//  - EXACT (also FP32 and FP64 requests whose supports are all <= 2^22): each cell's integer threshold t
//    (x >= t exactly when kappa x + d > 0), then the exact sum of |x + 1 - t| over the samples, four at a
//    time (k_exact); the epilogue puts every sample on its own branch (branch_sum).
//  - ENVELOPE (k_envelope): the same branch sums from the cumulative counts and sums, O(1) per
//    cell, not per term.
//
// Work decomposition.  A CTA owns one (regime m, class k) and a block of consecutive r values for the whole
// lam grid.  A warp owns a few cells at a time -- a TR x TL tile of (r, lam) in k_grid, the next 16 of the
// CTA's rows laid end to end in k_exact -- and its 32 lanes split the class's samples, which stream
// through a ring of shared-memory chunks filled by TMA bulk copies (cp.async.bulk + mbarrier).  Packed
// f32x2 instructions serve two cells at once.  Periodically each lane's partial sums are transposed and
// reduced across the warp (fixed shuffle order) so that each lane then owns one cell, folded into an
// FP64 or int64 accumulator.  k_envelope has no samples to stream: its lanes lie along lam, its warps on rows.
// The epilogue forms S = (1/N) sum phi, then for every eps the minimum over lam (lowest index),
// and feeds the argmin over r through a 64-bit atomicMin on (cost, r index) keys.
#include <float.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "kvdro_internal.cuh"

namespace kvdro {
namespace {

typedef unsigned long long u64;

// Bound on any barrier wait: 2 s of the GPU's global nanosecond timer, and at least
// kWaitPollsPerNs polls per nanosecond of that bound spent polling (each poll suspends the
// thread for at most kPollSuspendNs).  The timer keeps running while a CTA is descheduled
// (time-slicing, preemption), but the poll count only grows while it runs, so a CTA that
// was switched out for longer than the bound does not give up on a copy that lands soon
// after it resumes.  kWaitPollCap bounds the loop even if the timer were to stop.
constexpr long long kWaitNs = 2000000000LL;
constexpr unsigned kPollSuspendNs = 1000;
constexpr long long kWaitNsPerPoll = 4096;   // polls required: limit_ns / 4096
constexpr unsigned kWaitPollCap = 1u << 28;

constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v / 2); }

// Shape of one instantiation of the FP32- or FP64-arithmetic kernel: precision, warp tile (TR
// reservations x TL multipliers, TR*TL a power of two <= 32), FP32 chunks between folds of the per-lane
// partial sums into FP64 (FP64 folds once at the end), the largest CTA and minimum CTAs per SM it is
// compiled for (these two bound its registers per thread), the staged chunk and ring depth, and the
// sample loop's unroll.
template <Prec P_, int TR_, int TL_, int FLUSH_, int MINB_, int MAXT_ = 512, int CHUNK_ = 2048, int STAGES_ = 3,
          int UNROLL_ = 2>
struct GridCfg {
    static constexpr Prec P = P_;
    static constexpr int TR = TR_, TL = TL_, V = TR_ * TL_, LOG2V = ilog2(TR_ * TL_), FLUSH = FLUSH_, MINB = MINB_;
    static constexpr int MAXT = MAXT_;
    static constexpr int CHUNK = CHUNK_;    // samples per staged chunk
    static constexpr int BYTES = 8;         // staged bytes per sample (native FP64 also reads quads, 4)
    static constexpr int STAGES = STAGES_;  // ring depth
    static constexpr int UNROLL = UNROLL_;  // unroll of the sample loop
    static_assert(P_ != Prec::EXACT && CHUNK_ % 128 == 0 && CHUNK_ * BYTES * STAGES_ <= 160 * 1024, "chunk ring must fit");
    static_assert((V & (V - 1)) == 0 && V >= 2 && V <= 32, "tile must hold a power of two <= 32 cells");
    static_assert(P_ == Prec::F64 || TL_ % 2 == 0, "the FP32 tiles pack lam values in pairs");
    static_assert(FLUSH >= 0 && UNROLL >= 1, "shape parameters out of range");
};
// FP32: 2 r x 8 lam tiles, up to 16 warps per CTA and two CTAs per SM (64 registers) for up to 128 lam
// values, 2 x 16 tiles above.  FP64: 2 x 8 tiles.  Both stage 32 KB chunks through a 2-deep ring; the FP32
// variants fold their partial sums every 2 chunks (256 samples per lane) and unroll the sample loop 4 times.
using CfgF32 = GridCfg<Prec::F32, 2, 8, 2, 2, 512, 4096, 2, 4>;
using CfgF32Wide = GridCfg<Prec::F32, 2, 16, 2, 1, 512, 4096, 2, 4>;
using CfgF64 = GridCfg<Prec::F64, 2, 8, 0, 1, 512, 4096, 2>;
constexpr int kWarpsTarget = 16;  // warps per CTA the r groups fill up to

// The exact kernel: kExactV cells per warp, up to kExactWarps warps per CTA and kExactBlocks CTAs per SM.  A
// CTA takes whole rows of lam values, laid over its warps without regard to rows (a warp needs kExactV
// thresholds, whatever cells they are), in one pass over the class's samples or several (exact_shape).
constexpr int kExactLog2V = 4;
constexpr int kExactV = 1 << kExactLog2V;
constexpr int kExactWarps = 16;
constexpr int kExactBlocks = 2;
constexpr int kExactMaxPasses = 4;
constexpr int kExactStages = 3;
constexpr int kExactChunk = 8192;  // samples per staged chunk at most
constexpr size_t kExactSmem = (228 * 1024 / kExactBlocks - 1024) - 256;  // an SM's 228 KB, 1 KB reserved for each CTA

// ---------------------------------------------------------------- PTX helpers

__device__ __forceinline__ u64 pk(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk(u64 r, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ u64 fadd2(u64 a, u64 b) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// a b + c rounded once, then clamped to [0, 1]; a NaN result becomes 0.  For |a b + c| <= 1 this is
// max(a b + c, 0) in one instruction on the FMA pipe.
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
    float d;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// max(|u|, |v| + p, d)
__device__ __forceinline__ float max3_abs(float u, float v, float p, float d) {
    float m;
    asm("{\n\t.reg .f32 q;\n\tabs.f32 q, %1;\n\tmax.f32 %0, %3, q, %2;\n\t}" : "=f"(m) : "f"(u), "f"(fabsf(v) + p), "f"(d));
    return m;
}
// max(w, 0); a NaN operand yields 0 (PTX max returns the non-NaN input).
__device__ __forceinline__ double relu(double w) {
    double d;
    asm("max.f64 %0, %1, 0d0000000000000000;" : "=d"(d) : "d"(w));
    return d;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// One bulk copy global -> shared, completing on `bar` (bytes and both addresses 16-byte aligned).
__device__ __forceinline__ void tma_bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// The same test, suspending the thread for at most about `ns` nanoseconds while the phase is
// incomplete.
__device__ __forceinline__ bool mbar_try_for(uint32_t bar, uint32_t parity, uint32_t ns) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(ns)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for phase `parity` of `bar`.  Gives up and returns false once limit_ns nanoseconds of
// the global timer have passed and the wait has polled at least limit_ns / kWaitNsPerPoll
// times (or after kWaitPollCap polls in any case).  limit_ns <= 0 selects kWaitNs.
__device__ __noinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, long long limit_ns) {
    if (mbar_try(bar, parity)) return true;
    if (limit_ns <= 0) limit_ns = kWaitNs;
    const unsigned long long t0 = global_ns();
    const unsigned min_polls = (unsigned)(limit_ns / kWaitNsPerPoll);
    unsigned polls = 0;
    while (!mbar_try_for(bar, parity, kPollSuspendNs)) {
        ++polls;
        if (polls >= kWaitPollCap) return false;
        if (polls >= min_polls && (long long)(global_ns() - t0) > limit_ns) return false;
    }
    return true;
}

// Reduce V per-lane values across the warp so that lane l ends with the warp-wide sum of value
// index l >> (5 - log2 V): recursive halving over lane bits 4, 3, ..., then butterflies over the
// remaining low bits.  The order of additions is fixed, so results are deterministic.
template <typename T, int V, int S>
struct TransposeStep {
    static __device__ __forceinline__ void run(T (&v)[V], int lane) {
        constexpr int n = V * S / 16;  // values still held per lane before this step
        if constexpr (n >= 2) {
            constexpr int h = n / 2;
            const bool up = (lane & S) != 0;
#pragma unroll
            for (int p = 0; p < h; p++) {
                const T send = up ? v[p] : v[p + h];
                const T keep = up ? v[p + h] : v[p];
                v[p] = keep + __shfl_xor_sync(0xffffffffu, send, S);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], S);
        }
        if constexpr (S > 1) TransposeStep<T, V, S / 2>::run(v, lane);
    }
};

template <typename T, int V>
__device__ __forceinline__ T transpose_reduce(T (&v)[V], int lane) {
    TransposeStep<T, V, 16>::run(v, lane);
    return v[0];
}

struct SmemLayout {
    size_t ring, full, lam, eps, S, lamf, Sf, total;
    int stride_f;
};

__host__ __device__ inline int four(int n) { return (n + 3) & ~3; }
// Floats per row of S cut to floats: read four at a time with lanes along the rows, so an odd number of fours.
__host__ __device__ inline int float_stride(int NL) { return 4 * ((NL + 3) / 4 | 1); }

__host__ __device__ inline SmemLayout smem_layout(int RG, int TR, int NLpad, int E, int chunk_bytes, int stages) {
    SmemLayout L;
    L.stride_f = float_stride(NLpad);
    L.ring = 0;
    L.full = (size_t)stages * chunk_bytes;
    L.lam = L.full + 8 * (size_t)stages;
    L.eps = L.lam + 8 * (size_t)NLpad;
    L.S = L.eps + 8 * (size_t)E;
    L.lamf = (L.S + 8 * (size_t)RG * TR * NLpad + 15) & ~(size_t)15;
    L.Sf = L.lamf + 4 * (size_t)four(NLpad);
    L.total = L.Sf + 4 * (size_t)RG * TR * L.stride_f;
    return L;
}

// The exact kernel's: `S` holds the cells' integer sums first, then their S, `t` their thresholds.
struct ExactSmem {
    size_t full, lam, eps, S, t, lamf, Sf, total;
    int stride_f;
};
__host__ __device__ inline ExactSmem exact_smem(int rows, int NL, int E, int tiles, int ring_bytes) {
    ExactSmem s;
    s.stride_f = float_stride(NL);
    s.full = ring_bytes;
    s.lam = s.full + 48;
    s.eps = s.lam + 8 * (size_t)NL;
    s.S = s.eps + 8 * (size_t)E;
    s.t = (s.S + 8 * (size_t)tiles * kExactV + 15) & ~(size_t)15;
    s.lamf = (s.t + 4 * (size_t)tiles * kExactV + 15) & ~(size_t)15;
    s.Sf = s.lamf + 4 * (size_t)four(NL);
    s.total = s.Sf + 4 * (size_t)rows * s.stride_f;
    return s;
}

// The minimum over lam of lam * eps + S for one (r, eps) pair: the value RN(RN(lam eps) + S) and the
// lowest index attaining it.
//
// FP32 first: with lam, eps and S cut to floats (each at most 2^-23 low) v' = fma(lam, eps, S) lies
// within [v (1 - 2.6 x 2^-23), v (1 + 2^-23)], so a lam attaining the minimum has v' at most
// (1 + 2^-20) times the smallest v', and only those values -- one as a rule -- are formed in FP64, in
// ascending order, except one whose lam and S are both no smaller than the best's, which cannot be
// below it.  Where the floats do not hold every value is formed: a negative S, magnitudes above 2^100, a
// nonzero lam or eps below 2^-100 (the other factor may be so large that their product decides), or
// a minimum below 2^-80, which an S cut to zero, below 2^-100, could matter to.
constexpr float kLamWindow = 1.f + 0x1p-19f;
constexpr float kLamFloor = 0x1p-80f;

// A value >= 0 cut to a float: 0 below 2^-100; `ok` is cleared above 2^100 and for negative values.
__device__ __forceinline__ float cut(double v, bool& ok) {
    const long long b = dbits(v);
    if ((b << 1) == 0) return 0.f;  // +-0
    const unsigned e = (unsigned)((unsigned long long)b >> 52);  // sign and exponent
    ok = ok && e <= 1023u + 100u;
    return e >= 1023u - 100u ? narrow(b) : 0.f;
}
// The same for a factor, lam or eps: `ok` is also cleared for a nonzero value below 2^-100.
__device__ __forceinline__ float cut_factor(double v, bool& ok) {
    const long long b = dbits(v);
    if ((b << 1) == 0) return 0.f;
    ok = ok && b > 0 && narrowable(b);
    return narrow(b);
}

struct LamMin {
    long long key = 0x7fffffffffffffffll;  // order key of v
    double v = DBL_MAX;
    int j = 0x7fffffff;
    // value j, in ascending order of j; `skip`: S >= 0 and finite floats (the window holds)
    __device__ __forceinline__ void take(double lam, double eps, double s, int at, bool skip, const double* L, const double* S) {
        if (skip && j != 0x7fffffff && dbits(lam) >= dbits(L[j]) && dbits(s) >= dbits(S[j])) return;
        const double w = __dadd_rn(__dmul_rn(lam, eps), s);
        const long long k = order_key(w);
        if (k < key) {
            key = k;
            v = w;
            j = at;
        }
    }
    // the lower of two lanes' results (ties: lower index), over groups of G lanes
    __device__ __forceinline__ void reduce(int G) {
        for (int o = 1; o < G; o <<= 1) {
            const long long ok = __shfl_xor_sync(0xffffffffu, key, o);
            const double ov = __shfl_xor_sync(0xffffffffu, v, o);
            const int oj = __shfl_xor_sync(0xffffffffu, j, o);
            if (ok < key || (ok == key && oj < j)) {
                key = ok;
                v = ov;
                j = oj;
            }
        }
    }
};

// One (r, eps) pair's results: the cost and lam index outputs and the argmin over r through a 64-bit
// key for atomicMin (FP32: cost bits and r index; otherwise the cost's double bits truncated to 44
// bits, order-preserving for non-negative values, with the r index in the low 20 bits).
template <bool F32OUT>
__device__ __forceinline__ u64 write_pair(const GridArgs& a, double best, int bj, int m, int k, int e, int ri) {
    const size_t o = (((size_t)m * a.E + e) * a.K + k) * a.R + ri;
    if (a.lam_idx_out) a.lam_idx_out[o] = bj;
    if constexpr (F32OUT) {
        const float cf = (float)best;
        if (a.cost_out) static_cast<float*>(a.cost_out)[o] = cf;
        return ((u64)__float_as_uint(cf > 0.f ? cf : 0.f) << 32) | (u64)(uint32_t)ri;
    } else {
        static_cast<double*>(a.cost_out)[o] = best;
        const bool above = dbits(best) > 0 && dbits(best) <= 0x7ff0000000000000ll;  // best > 0
        return ((u64)(above ? dbits(best) : 0ll) & ~0xFFFFFull) | (u64)ri;
    }
}

// Row i = (m, e, k) of the per-(regime, radius, class) outputs from its argmin key and, FP64, the cost there
// (past L1: other CTAs wrote them).
template <bool F32>
__device__ __forceinline__ void finalize_row(const FinalizeArgs& a, int64_t i, int k) {
    const u64 key = __ldcg(a.keys + i);
    if (key == ~0ull) {  // no r evaluated (cannot happen for R >= 1); report an invalid index
        if (a.r_idx) a.r_idx[i] = -1;
        return;
    }
    const int ri = (int)(F32 ? (key & 0xffffffffull) : (key & 0xFFFFFull));
    if (a.r_idx) a.r_idx[i] = ri;
    if (a.min_cost) {
        if constexpr (F32) static_cast<float*>(a.min_cost)[i] = __uint_as_float((uint32_t)(key >> 32));
        else static_cast<double*>(a.min_cost)[i] = __ldcg(static_cast<const double*>(a.cost) + i * a.R + ri);
    }
    if (a.fhat) {
        const int32_t v = a.r[ri] - a.L_in[k];
        a.fhat[i] = (double)a.cdf[a.hist_off[k] + v] / (double)a.N[k];
    }
}

// The last of the (regime, class)'s CTAs to get here finalises its rows: a launch of its own took 4 us of
// the smallest grids' 34.  Every CTA's outputs and keys are ordered before its count (barrier, fence,
// atomic), the last one's reads after.  A CTA that gave up a wait counts too, so rows are finalised whatever came of
// them.  Kept out of line: its registers are no concern of the sample loops.
template <bool F32>
__device__ __noinline__ void finish_rows(const GridArgs& a, int m, int k) {
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(a.done + (size_t)m * a.K + k, 1u) == (uint32_t)a.r_blocks - 2u;  // counts from all ones
        __threadfence();
    }
    __syncthreads();
    if (s_last)
        for (int e = threadIdx.x; e < a.E; e += blockDim.x) finalize_row<F32>(a.fin, ((int64_t)m * a.E + e) * a.K + k, k);
}

// The CTA's rows of S in shared memory, as doubles and cut to floats (INFINITY past NL up to a multiple of
// four), with the lam values likewise (0 past NL).
struct LamRows {
    const double *S, *lam, *eps;
    const float *Sf, *lamf;
    int stride, stride_f;
    int rows, NL;
    bool floats;  // every lam and S is >= 0 and its float holds
};

// The end of every grid kernel, by all threads of the CTA (whole warps): for each (r, eps) pair the minimum
// over lam, its outputs and the argmin over r.
//
// G lanes per pair, as many as keep every thread busy, groups along r first (outputs side by side, one
// atomic per warp and radius: one per pair held the envelope at 7.8 ms where it then took 3.7); each lane
// takes every G-th four lam values and keeps its smallest v', where it was, and its second smallest: with
// the second outside the window only that one value is formed in FP64, by all lanes at once.
template <bool F32OUT>
__device__ __forceinline__ void lam_min_epilogue(const GridArgs& a, const LamRows& x, int r_cta0, int m, int k) {
    const int tid = threadIdx.x, lane = tid & 31, threads = blockDim.x;
    const int pairs = x.rows * a.E, n4 = (x.NL + 3) / 4;
    int G = 1;
    while (G < 32 && G < n4 && 2 * G * pairs <= threads) G <<= 1;
    const int per_pass = threads / G, g = tid & (G - 1);
    for (int p0 = 0; p0 < pairs; p0 += per_pass) {  // the same trips for every lane: the group's shuffles are warp-wide
        const int p = p0 + tid / G;
        const bool active = p < pairs;
        const int e = active ? p / x.rows : 0, rl = active ? p % x.rows : 0;
        const double* S = x.S + rl * x.stride;
        const float* Sf = x.Sf + rl * x.stride_f;
        const double eps = x.eps[e];
        bool fast = x.floats;
        const float ef = cut_factor(eps, fast);
        float m1 = INFINITY, m2 = INFINITY;
        int j1 = 0;
        for (int q = g; q < n4; q += G) {
            const float4 l = reinterpret_cast<const float4*>(x.lamf)[q], s = reinterpret_cast<const float4*>(Sf)[q];
            const float v[4] = {fmaf(l.x, ef, s.x), fmaf(l.y, ef, s.y), fmaf(l.z, ef, s.z), fmaf(l.w, ef, s.w)};
#pragma unroll
            for (int i = 0; i < 4; i++) {
                m2 = fminf(m2, fmaxf(m1, v[i]));
                if (v[i] < m1) j1 = 4 * q + i;
                m1 = fminf(m1, v[i]);
            }
        }
        for (int o = 1; o < G; o <<= 1) {
            const float o1 = __shfl_xor_sync(0xffffffffu, m1, o), o2 = __shfl_xor_sync(0xffffffffu, m2, o);
            const int oj = __shfl_xor_sync(0xffffffffu, j1, o);
            m2 = fminf(fminf(m2, o2), fmaxf(m1, o1));
            if (o1 < m1 || (o1 == m1 && oj < j1)) j1 = oj;
            m1 = fminf(m1, o1);
        }
        fast = fast && m1 > kLamFloor;
        const float thr = m1 * kLamWindow;
        LamMin best;
        if (fast && m2 > thr) {
            best.v = __dadd_rn(__dmul_rn(x.lam[j1], eps), S[j1]);
            best.j = j1;
        }
        const bool several = active && best.j == 0x7fffffff;
        if (__any_sync(0xffffffffu, several)) {
            LamMin r;
            if (several)
                for (int j = g; j < x.NL; j += G)
                    if (!fast || fmaf(x.lamf[j], ef, Sf[j]) <= thr) r.take(x.lam[j], eps, S[j], j, fast, x.lam, S);
            r.reduce(G);
            if (several) best = r;
        }
        u64 key = ~0ull;
        if (active && g == 0) key = write_pair<F32OUT>(a, best.v, best.j, m, k, e, r_cta0 + rl);
        // the warp's minimum over each radius it holds, e0 (its first lane's) upwards
        const int e0 = __shfl_sync(0xffffffffu, e, 0), e1 = __reduce_max_sync(0xffffffffu, e);
        for (int ei = e0; ei <= e1; ei++) {
            const u64 low = warp_min(e == ei ? key : ~0ull);
            if (lane == 0 && low != ~0ull) atomicMin(a.keys + ((size_t)m * a.E + ei) * a.K + k, low);
        }
    }
    if (a.done) finish_rows<F32OUT>(a, m, k);
}

// ---------------------------------------------------------------- the FP32- and FP64-arithmetic kernels

template <class C>
__global__ void __launch_bounds__(C::MAXT, C::MINB) k_grid(const GridArgs a) {
    constexpr Prec P = C::P;
    constexpr int TR = C::TR, TL = C::TL, V = C::V, LOG2V = C::LOG2V;
    extern __shared__ __align__(128) unsigned char smem[];
    const int NLpad = a.LT * TL;
    const SmemLayout lay = smem_layout(a.RG, TR, NLpad, a.E, C::CHUNK * C::BYTES, C::STAGES);
    unsigned char* ring = smem + lay.ring;  // chunk c in stage c % STAGES
    constexpr size_t kStageBytes = (size_t)C::CHUNK * C::BYTES;
    u64* full = reinterpret_cast<u64*>(smem + lay.full);
    double* s_lam = reinterpret_cast<double*>(smem + lay.lam);
    double* s_eps = reinterpret_cast<double*>(smem + lay.eps);
    double* s_S = reinterpret_cast<double*>(smem + lay.S);
    float* s_lamf = reinterpret_cast<float*>(smem + lay.lamf);
    float* s_Sf = reinterpret_cast<float*>(smem + lay.Sf);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int b = blockIdx.x;
    const int rb = b % a.r_blocks;
    b /= a.r_blocks;
    const int k = b % a.K;
    const int m = a.m0 + b / a.K;
    const int lt = warp % a.LT, r_local0 = warp / a.LT * TR;
    const int r_cta0 = rb * a.RG * TR;

    for (int i = tid; i < NLpad; i += blockDim.x) s_lam[i] = i < a.NL ? a.lam[i] : 0.0;
    for (int i = tid; i < a.E; i += blockDim.x) s_eps[i] = a.eps[i];

    const int64_t pbase = a.pair_off[k];
    const int64_t np = a.pair_off[k + 1] - pbase;  // multiple of kPadSamples
    const int nchunks = (int)((np + C::CHUNK - 1) / C::CHUNK);
    // (native FP64 also serves contexts that stage quads)
    const int bytes = P == Prec::F64 && a.quads ? 4 : C::BYTES;
    const unsigned char* src = static_cast<const unsigned char*>(a.staged) + pbase * bytes;
    auto issue = [&](int c) {
        if (c == a.test_skip_chunk) return;  // test hook: nothing will complete this chunk's barrier
        const int s = c % C::STAGES;
        const int64_t cnt = min((int64_t)C::CHUNK, np - (int64_t)c * C::CHUNK);
        tma_bulk_load(smem_u32(ring + (size_t)s * kStageBytes), src + (int64_t)c * C::CHUNK * bytes, (uint32_t)(cnt * bytes),
                      smem_u32(&full[s]));
    };
    if (tid == 0) {
        for (int s = 0; s < C::STAGES; s++) mbar_init(smem_u32(&full[s]), 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0)
        for (int c = 0; c < C::STAGES && c < nchunks; c++) issue(c);
    int issued = min(C::STAGES, nchunks);  // chunks issued so far (tracked identically by every thread)
    int consumed = 0;                    // chunk at which the loop stopped

    // Per-cell constants of this warp's tile (identical across its lanes).
    const double cp = a.cp[m], cw = a.cw[m], Lk = (double)a.L[k];
    double eta[TR];
    bool rvalid[TR];
#pragma unroll
    for (int i = 0; i < TR; i++) {
        const int ri = r_cta0 + r_local0 + i;
        rvalid[i] = ri < a.R;
        eta[i] = rvalid[i] ? (double)a.r[ri] - (double)a.L_in[k] : 0.0;
    }

    bool timeout = false;
    double acc64 = 0.0;  // this lane's cell after the warp transposition

    if constexpr (P == Prec::F32) {
        // Each row's excess is taken about its reservation: kappa (x - eta) + W(eta) (excess_at_eta).
        // x - eta comes from the staged samples in one packed add per row and load (both samples of
        // the load); both are integers up to 2^24, so the add is exact.
        u64 noff[TR];
#pragma unroll
        for (int i = 0; i < TR; i++) {
            const float o = (float)-eta[i];
            noff[i] = pk(o, o);
        }
        u64 kap[TL / 2], dd[TR][TL / 2], acc[TR][TL / 2];
#pragma unroll
        for (int jp = 0; jp < TL / 2; jp++) {
            const int j0 = lt * TL + 2 * jp;
            const double l0 = s_lam[j0], l1 = s_lam[j0 + 1];
            const bool v0 = j0 < a.NL, v1 = j0 + 1 < a.NL;
            const double mu0 = fmin(l0, cp), mu1 = fmin(l1, cp), nu0 = fmin(l0, cw), nu1 = fmin(l1, cw);
            // the split of phi this column sums (see use_u_split): the sign of its excess
            const float s0 = use_u_split(mu0, nu0) ? -1.f : 1.f, s1 = use_u_split(mu1, nu1) ? -1.f : 1.f;
            kap[jp] = pk(v0 ? s0 * (float)(mu0 + nu0) : 0.f, v1 ? s1 * (float)(mu1 + nu1) : 0.f);
#pragma unroll
            for (int i = 0; i < TR; i++) {
                const double d0 = excess_at_eta(cp, cw, mu0, nu0, Lk, eta[i]);
                const double d1 = excess_at_eta(cp, cw, mu1, nu1, Lk, eta[i]);
                dd[i][jp] = pk(v0 && rvalid[i] ? s0 * (float)d0 : 0.f, v1 && rvalid[i] ? s1 * (float)d1 : 0.f);
                acc[i][jp] = 0ull;
            }
        }
        // One power of two S per warp tile with |kappa (x - eta) + W| <= S for every cell and every
        // x in [0, L].  The loop sums fma_sat(kappa / S, x - eta, W / S) = max(excess, 0) / S, and the
        // fold multiplies the reduced sums by S.  Scaling by a power of two changes no rounding, so
        // the sums equal those of a separate max per term, with the max folded into the FMA.
        double wmax = 1.0;
#pragma unroll
        for (int jp = 0; jp < TL / 2; jp++) {
            float k0, k1;
            upk(kap[jp], k0, k1);
#pragma unroll
            for (int i = 0; i < TR; i++) {
                float d0, d1;
                upk(dd[i][jp], d0, d1);
                const double xm = fmax(fabs(eta[i]), fabs(Lk - eta[i]));  // largest |x - eta|
                wmax = fmax(wmax, fmax(fabs((double)k0) * xm + fabs((double)d0), fabs((double)k1) * xm + fabs((double)d1)));
            }
        }
        int sexp;
        (void)frexp(wmax, &sexp);  // wmax < 2^sexp
        const float S = ldexpf(1.f, sexp), invS = ldexpf(1.f, -sexp);
#pragma unroll
        for (int jp = 0; jp < TL / 2; jp++) {
            float k0, k1;
            upk(kap[jp], k0, k1);
            kap[jp] = pk(k0 * invS, k1 * invS);
#pragma unroll
            for (int i = 0; i < TR; i++) {
                float d0, d1;
                upk(dd[i][jp], d0, d1);
                dd[i][jp] = pk(d0 * invS, d1 * invS);
            }
        }
        // one load: two samples' excesses for every cell of the tile.  The two samples' excesses are
        // added to each other before they join the running sum: the same number of adds, half as
        // many additions into the long sum.
        auto step = [&](const float4 v) {
#pragma unroll
            for (int i = 0; i < TR; i++) {
                // x - eta of the load's two samples in one packed add (v.x and v.z: one copy of each)
                const u64 xab = fadd2(pk(v.x, v.z), noff[i]);
                float xa0, xb0;
                upk(xab, xa0, xb0);
#pragma unroll
                for (int jp = 0; jp < TL / 2; jp++) {
                    float k0, k1, d0, d1;
                    upk(kap[jp], k0, k1);
                    upk(dd[i][jp], d0, d1);
                    const float a0 = fma_sat(k0, xa0, d0), a1 = fma_sat(k1, xa0, d1);
                    const float b0 = fma_sat(k0, xb0, d0), b1 = fma_sat(k1, xb0, d1);
                    acc[i][jp] = fadd2(acc[i][jp], fadd2(pk(a0, a1), pk(b0, b1)));
                }
            }
        };
        for (int c = 0; c < nchunks; c++) {
            const int s = c % C::STAGES;
            if (!mbar_wait_bounded(smem_u32(&full[s]), (uint32_t)((c / C::STAGES) & 1), a.wait_ns)) timeout = true;
            if (!timeout) {
                const int cnt = (int)min((int64_t)C::CHUNK, np - (int64_t)c * C::CHUNK);
                const float4* q = reinterpret_cast<const float4*>(ring + (size_t)s * kStageBytes);
                const int nq = cnt >> 6;  // float4 (two samples) per lane: (x, x) pairs
                if (nq == C::CHUNK / 64) {  // a full chunk: a fixed trip count, unrolled with no remainder
#pragma unroll(C::UNROLL)
                    for (int t = 0; t < C::CHUNK / 64; t++) step(q[lane + 32 * t]);
                } else {
#pragma unroll 1
                    for (int t = 0; t < nq; t++) step(q[lane + 32 * t]);
                }
                // Every C::FLUSH chunks (and after the last), fold the FP32 partials into the FP64
                // accumulator of the lane's cell.
                if ((c + 1) % C::FLUSH == 0 || c + 1 == nchunks) {
                    float vals[V];
#pragma unroll
                    for (int i = 0; i < TR; i++)
#pragma unroll
                        for (int jp = 0; jp < TL / 2; jp++) {
                            upk(acc[i][jp], vals[i * TL + 2 * jp], vals[i * TL + 2 * jp + 1]);
                            acc[i][jp] = 0ull;
                        }
                    acc64 += (double)transpose_reduce<float, V>(vals, lane) * (double)S;
                }
            }
            consumed = c;
            if (__syncthreads_or(timeout)) {
                timeout = true;
                break;
            }
            if (c + C::STAGES < nchunks) {
                if (tid == 0) {
                    fence_proxy_async();
                    issue(c + C::STAGES);
                }
                issued = c + C::STAGES + 1;
            }
        }
    } else if constexpr (P == Prec::F64) {
        // each row's excess about its reservation, as in the FP32 kernel: x - eta per sample and row
        double kap[TL], dd[TR][TL], acc[TR][TL];
#pragma unroll
        for (int j = 0; j < TL; j++) {
            const int lj = lt * TL + j;
            const double l = s_lam[lj];
            const bool v = lj < a.NL;
            const double mu = fmin(l, cp), nu = fmin(l, cw);
            const double sg = use_u_split(mu, nu) ? -1.0 : 1.0;  // the split of phi this column sums
            kap[j] = v ? sg * (mu + nu) : 0.0;
#pragma unroll
            for (int i = 0; i < TR; i++) {
                dd[i][j] = (v && rvalid[i]) ? sg * excess_at_eta(cp, cw, mu, nu, Lk, eta[i]) : 0.0;
                acc[i][j] = 0.0;
            }
        }
        for (int c = 0; c < nchunks; c++) {
            const int s = c % C::STAGES;
            if (!mbar_wait_bounded(smem_u32(&full[s]), (uint32_t)((c / C::STAGES) & 1), a.wait_ns)) timeout = true;
            if (!timeout) {
                const int cnt = (int)min((int64_t)C::CHUNK, np - (int64_t)c * C::CHUNK);
                const float4* q = reinterpret_cast<const float4*>(ring + (size_t)s * kStageBytes);
                auto two = [&](float x0, float x1) {  // two staged samples (NaN: none)
#pragma unroll
                    for (int i = 0; i < TR; i++) {
                        const double xa = (double)x0 - eta[i], xb = (double)x1 - eta[i];  // x - eta, exact
#pragma unroll
                        for (int j = 0; j < TL; j++) {
                            acc[i][j] += relu(fma(kap[j], xa, dd[i][j]));
                            acc[i][j] += relu(fma(kap[j], xb, dd[i][j]));
                        }
                    }
                };
                if (a.quads) {  // samples back from their quads, exactly; the class's last quad may start with padding
                    const int64_t left = a.N[k] - (int64_t)c * C::CHUNK;
                    for (int t = 0; t < cnt >> 7; t++) {
                        const int4 v = reinterpret_cast<const int4*>(q)[lane + 32 * t];
                        const int64_t first = max((int64_t)0, 4 * (int64_t)(lane + 32 * t) + 4 - left);  // of the four
                        const float nan = __int_as_float(0x7fc00000);
                        const int ends = v.x - v.y, gap = v.w - v.z;  // x0 + x3, x2 - x1
                        two(first < 1 ? (float)((ends - v.z) / 2) : nan, first < 2 ? (float)((v.y - gap) / 2) : nan);
                        two(first < 3 ? (float)((v.y + gap) / 2) : nan, first < 4 ? (float)((ends + v.z) / 2) : nan);
                    }
                } else {
                    for (int t = 0; t < cnt >> 6; t++) {
                        const float4 v = q[lane + 32 * t];
                        two(v.x, v.z);
                    }
                }
            }
            consumed = c;
            if (__syncthreads_or(timeout)) {
                timeout = true;
                break;
            }
            if (c + C::STAGES < nchunks) {
                if (tid == 0) {
                    fence_proxy_async();
                    issue(c + C::STAGES);
                }
                issued = c + C::STAGES + 1;
            }
        }
        if (!timeout) {
            double vals[V];
#pragma unroll
            for (int i = 0; i < TR; i++)
#pragma unroll
                for (int j = 0; j < TL; j++) vals[i * TL + j] = acc[i][j];
            acc64 = transpose_reduce<double, V>(vals, lane);
        }
    }

    if (timeout) {
        // Report, then let every copy this CTA issued land before the CTA's shared memory is released.
        if (tid == 0) {
            atomicOr(a.err + 1, kErrTimeout);
            for (int c = consumed; c < issued; c++)
                (void)mbar_wait_bounded(smem_u32(&full[c % C::STAGES]), (uint32_t)((c / C::STAGES) & 1), a.wait_ns);
        }
        __syncthreads();
        if (a.done) finish_rows<P == Prec::F32>(a, m, k);
        return;
    }

    // S for this lane's cell.
    bool ok = true;
    {
        const int cidx = lane >> (5 - LOG2V);
        const int i = cidx / TL, j = cidx % TL;
        const int ri = r_cta0 + r_local0 + i, lj = lt * TL + j;
        const bool owner = (lane & ((1 << (5 - LOG2V)) - 1)) == 0;
        if (owner && ri < a.R && lj < a.NL) {
            // the split's base plus its excess sum: sum V + sum max(kappa x + d, 0), or
            // sum U + sum max(-(kappa x + d), 0)
            const double mu = fmin(s_lam[lj], cp), nu = fmin(s_lam[lj], cw);
            const double Nk = (double)a.N[k];
            const double eta_i = (double)a.r[ri] - (double)a.L_in[k];
            const long long N64 = a.N[k], sx = a.sumx[k];
            const double base = use_u_split(mu, nu) ? cp * (Lk - eta_i) * Nk - mu * (double)((long long)a.L[k] * N64 - sx)
                                                    : cw * eta_i * Nk - nu * (double)sx;
            const double tot = base + acc64;
            const double S = __dmul_rn(tot, a.inv_n[k]);
            s_S[(r_local0 + i) * NLpad + lj] = S;
            s_Sf[(r_local0 + i) * lay.stride_f + lj] = cut(S, ok);
            if (a.S_out) {
                const size_t o = (((size_t)m * a.K + k) * a.R + ri) * a.NL + lj;
                if (P == Prec::F32) static_cast<float*>(a.S_out)[o] = (float)S;
                else static_cast<double*>(a.S_out)[o] = S;
            }
        }
    }
    // the floats past the last lam value; `ok` over the CTA
    for (int i = tid; i < a.RG * TR * 4; i += blockDim.x)
        if (a.NL + (i & 3) < four(a.NL)) s_Sf[(i >> 2) * lay.stride_f + a.NL + (i & 3)] = INFINITY;
    for (int j = tid; j < four(a.NL); j += blockDim.x) s_lamf[j] = j < a.NL ? cut_factor(s_lam[j], ok) : 0.f;
    const bool floats = __syncthreads_and(ok);
    const LamRows rows = {s_S, s_lam, s_eps, s_Sf, s_lamf, NLpad, lay.stride_f, min(a.RG * TR, a.R - r_cta0), a.NL, floats};
    lam_min_epilogue<P == Prec::F32>(a, rows, r_cta0, m, k);
}

// ---------------------------------------------------------------- the exact kernel
//
// Per cell the active samples are x >= t for an integer threshold t, and
// sum_n max(kappa x_n + d, 0) = kappa sum_{x >= t} x + d #{x >= t}.  With c = t - 1,
// max(x - c, 0) = (x - c + |x - c|) / 2 and sum_n (x - c) has a closed form, so the kernel streams
// sum_n |x - c| only, as integers.
//
// Quads: for sorted samples x0 <= x1 <= x2 <= x3 the sum over the four is the maximum of its linear pieces,
//   sum |x_i - c| = max(|S - 4c|, |Q - 2c| + P, D),
//   S = x0 + x1 + x2 + x3, Q = x1 + x2, P = x3 - x0, D = (x2 + x3) - (x0 + x1),
// so one load of {S, Q, P, D} serves four samples of every cell in two packed FP32 instructions for two cells
// (S - 4c; Q - 2c as one FMA from the same -4c), an add and a three-way max per cell, and half a
// three-input integer add: 3.5 instructions per cell for four samples, where pairs of samples,
// max(|a + b - 2c|, |a - b|), take 4.  FMA pipe (128 lanes a clock and SM) and ALU (64) carry 3 cycles each of
// those, so the issue slots bound it: 146 terms/clk/SM against the pairs' 128.
//
// The integers are the floats' bit patterns: an integer n <= 2^24 read as a float is n x 2^-149, a
// subnormal or one of the two smallest normal binades, where patterns are linear.  FP32 adds, fmas and
// maxima of such values are exact and full-rate, and their results are already integers: sums
// run on in 32-bit integer adds, on the pipe that has the room, and fold 256 times more rarely than
// FP32 sums below 2^24 would.  (The maths need subnormals kept: no flush-to-zero.)
//
// 8 classes x 100,000 samples x 4096 r x 128 lam: 13.64 ms, 98 terms/clk/SM (pairs 15.92); the loop alone runs at
// 97 to 99 in isolation, bound by register reads (23 operands for 8 terms) and their banks rather than by
// either pipe, so the order of operands counts: 13.65 to 14.05 over the six orders of the maximum's, 13.64
// with the second load's cells ahead of the first's.  Also measured, with the maximum's operands as written
// above (14.1 so): -2c kept beside -4c instead of the FMA 14.5 (80 registers, 12 warps); (S, Q) as one packed
// operand against (-4c, -2c) of one cell 16.1; 8, 10 and 12 cells a warp 15.6, 15.5, 14.8.
//
// The count #{x >= t} comes from the class's cumulative counts; every sample then goes on its branch of
// phi with these integer sums (branch_sum) in FP64.
__global__ void __launch_bounds__(32 * kExactWarps, kExactBlocks) k_exact(const GridArgs a) {
    constexpr int V = kExactV, kOwn = 5 - kExactLog2V;  // lane l owns cell l >> kOwn after the transposition
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_bad, s_timeout;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NL = a.NL;
    int b = blockIdx.x;
    const int r_cta0 = b % a.r_blocks * a.rows;
    b /= a.r_blocks;
    const int k = b % a.K;
    const int m = a.m0 + b / a.K;
    const int rows = min(a.rows, a.R - r_cta0), cells = rows * NL;
    const int chunk = a.chunk, stage_bytes = chunk * 4, nwarps = blockDim.x >> 5;
    const ExactSmem lay = exact_smem(a.rows, NL, a.E, nwarps * a.passes, kExactStages * stage_bytes);
    unsigned char* ring = smem;  // chunk c in stage c % stages
    u64* full = reinterpret_cast<u64*>(smem + lay.full);  // a chunk has landed in the stage
    u64* empty = full + kExactStages;                     // every warp is done with the stage's chunk
    double* s_lam = reinterpret_cast<double*>(smem + lay.lam);
    double* s_eps = reinterpret_cast<double*>(smem + lay.eps);
    double* s_S = reinterpret_cast<double*>(smem + lay.S);
    long long* sums = reinterpret_cast<long long*>(s_S);
    int* s_t = reinterpret_cast<int*>(smem + lay.t);
    float* s_lamf = reinterpret_cast<float*>(smem + lay.lamf);
    float* s_Sf = reinterpret_cast<float*>(smem + lay.Sf);

    const int64_t pbase = a.pair_off[k];
    const int64_t np = a.pair_off[k + 1] - pbase;  // multiple of kPadSamples
    const int nchunks = (int)((np + chunk - 1) / chunk), total = nchunks * a.passes;  // over all passes
    const unsigned char* src = static_cast<const unsigned char*>(a.staged) + pbase * 4;
    auto issue = [&](int c, int s) {  // the class's chunk c into stage s
        if (c == a.test_skip_chunk) return;  // test hook: nothing will complete this chunk's barrier
        const int64_t cnt = min((int64_t)chunk, np - (int64_t)c * chunk);
        tma_bulk_load(smem_u32(ring + (size_t)s * stage_bytes), src + (int64_t)c * stage_bytes, (uint32_t)(cnt * 4),
                      smem_u32(&full[s]));
    };
    // the chunk `ahead` places after the class's chunk c, passes wrapping
    auto chunk_after = [&](int c, int ahead) { return (c + ahead) % nchunks; };
    if (tid == 0) {  // no other thread touches a barrier before the __syncthreads below
        s_bad = s_timeout = 0;
        for (int s = 0; s < kExactStages; s++) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), nwarps);
        }
        fence_mbar_init();
        for (int i = 0; i < kExactStages && i < total; i++) issue(chunk_after(0, i), i);
    }
    for (int i = tid; i < NL; i += blockDim.x) s_lam[i] = a.lam[i];
    for (int i = tid; i < a.E; i += blockDim.x) s_eps[i] = a.eps[i];
    __syncthreads();

    // Each cell's threshold is one thread's work (its few FP64 instructions take the pipe as long for one
    // lane as for 32) and read back by its warp; a thread combines the cell's sums at the end, so
    // nothing of it stays in registers over the sample loop.
    const double cp = a.cp[m], cw = a.cw[m];
    for (int c = tid; c < nwarps * a.passes * V; c += blockDim.x) {
        int t = a.L[k] + 1;  // "none" (no sample exceeds L); t in [0, L + 1] keeps |x - c| <= L + 1
        if (c < cells) {
            const double lam = s_lam[c % NL], mu = dmin_nonneg(lam, cp);
            const RowOffset row = row_offset(cp, cw, a.L[k], a.r[r_cta0 + c / NL] - a.L_in[k]);
            t = first_active(__dadd_rn(mu, dmin_nonneg(lam, cw)), excess_offset(row, cp, mu, to_double(a.L[k])), a.L[k]);
        }
        s_t[c] = t;
        sums[c] = 0;
    }
    __syncthreads();
    u64 n4c[V / 2] = {};  // -4c for two cells
    unsigned acc[V] = {};
    const u64 half = pk(0.5f, 0.5f);
    const int* w_t = s_t + warp * V;  // the pass's thresholds
    // Fold after at most `fe` loads of 4 samples: 32 lanes' sums of at most 4 L a load then stay below 2^32.
    // The same for every thread of the CTA.
    const int fe = (int)((1u << 27) - 1) / (4 * max(a.L[k], 1)) & ~1;
    int pending = 0;  // loads since the last fold
    auto fold = [&]() {
        const unsigned sum = transpose_reduce<unsigned, V>(acc, lane);
        if ((lane & ((1 << kOwn) - 1)) == 0) sums[w_t - s_t + (lane >> kOwn)] += sum;
#pragma unroll
        for (int j = 0; j < V; j++) acc[j] = 0u;
        pending = 0;
    };
    // One load's sum for cells 2p and 2p + 1.
    auto quad = [&](const float4 v, int p, unsigned& s0, unsigned& s1) {
        float u0, u1, v0, v1;
        upk(ffma2(n4c[p], half, pk(v.y, v.y)), v0, v1);
        upk(fadd2(pk(v.x, v.x), n4c[p]), u0, u1);
        s0 = __float_as_uint(max3_abs(u0, v0, v.z, v.w));
        s1 = __float_as_uint(max3_abs(u1, v1, v.z, v.w));
    };
    auto two = [&](const float4 va, const float4 vb) {
#pragma unroll
        for (int p = 0; p < V / 2; p++) {
            unsigned a0, a1, b0, b1;
            quad(vb, p, b0, b1);
            quad(va, p, a0, a1);
            acc[2 * p] += a0 + b0;
            acc[2 * p + 1] += a1 + b1;
        }
    };
    // `loads` loads (a multiple of kSeg) in segments of a fixed trip count, two loads at a time.  64 with 8 loads
    // to an iteration run 13.65 ms on 8 classes x 100,000 samples x 4096 r x 128 lam, 4 or 16 14.1; segments of 16 with
    // 8 spill registers (15.1).
    auto segments = [&](const float4*& q, int loads, auto seg) {
        constexpr int kSeg = decltype(seg)::value, kUnroll = kSeg == 64 ? 8 : 4;
        const float4* stop = q + 32 * loads;
#pragma unroll 1
        for (; q < stop; q += 32 * kSeg) {
#pragma unroll kUnroll
            for (int t = 0; t < kSeg; t += 2) two(q[32 * t], q[32 * t + 32]);
        }
    };
    bool timeout = false;
    int issued = min(kExactStages, total);  // by thread 0
    int at = 0, c = 0, s = 0;  // chunk over all passes, of the class, its stage
    uint32_t phase = 0;
    for (; at < total; at++) {
        if (c == 0) {
#pragma unroll
            for (int p = 0; p < V / 2; p++) {
                const int c0 = max(w_t[2 * p], 1) - 1, c1 = max(w_t[2 * p + 1], 1) - 1;
                n4c[p] = pk(-__int_as_float(4 * c0), -__int_as_float(4 * c1));
            }
        }
        // The warps run on by themselves, up to a stage's reuse: a barrier of the CTA after each chunk costs 1 to 2 %.
        timeout = !__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&full[s]), phase, a.wait_ns));
        if (timeout) break;
        const float4* q = reinterpret_cast<const float4*>(ring + (size_t)s * stage_bytes) + lane;
        const float4* end = q + min((int64_t)chunk, np - (int64_t)c * chunk) / 4;
        while (q < end) {
            if (pending == fe) fold();
            const int loads = min((int)(end - q) / 32, fe - pending);
            pending += loads;
            segments(q, loads & ~63, std::integral_constant<int, 64>());
            segments(q, loads & 48, std::integral_constant<int, 16>());
            segments(q, loads & 14, std::integral_constant<int, 2>());
            if (loads & 1) {
#pragma unroll
                for (int p = 0; p < V / 2; p++) {
                    unsigned a0, a1;
                    quad(*q, p, a0, a1);
                    acc[2 * p] += a0;
                    acc[2 * p + 1] += a1;
                }
                q += 32;
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty[s]));
        // The first warp refills the stage before, which the others have mostly left by now.
        if (warp == 0 && at > 0 && at - 1 + kExactStages < total) {
            const int sp = s == 0 ? kExactStages - 1 : s - 1;
            const uint32_t done = s == 0 ? phase ^ 1 : phase;
            timeout = !__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&empty[sp]), done, a.wait_ns));
            if (timeout) break;
            if (lane == 0) {
                fence_proxy_async();
                issue(chunk_after(c, kExactStages - 1), sp);
                issued++;
            }
        }
        if (++s == kExactStages) {
            s = 0;
            phase ^= 1;
        }
        if (++c == nchunks) {  // the pass's sums
            c = 0;
            if (pending > 0) fold();
            w_t += nwarps * V;
        }
    }
    if (timeout) s_timeout = 1;
    __syncthreads();
    if (s_timeout) {
        // Report, then let every copy this CTA issued land before the CTA's shared memory is released.
        if (tid == 0) {
            atomicOr(a.err + 1, kErrTimeout);
            for (; at < issued; at++) {
                (void)mbar_wait_bounded(smem_u32(&full[s]), phase, a.wait_ns);
                if (++s == kExactStages) {
                    s = 0;
                    phase ^= 1;
                }
            }
        }
        __syncthreads();
        if (a.done && a.f32_out) finish_rows<true>(a, m, k);
        else if (a.done) finish_rows<false>(a, m, k);
        return;
    }
    bool ok = true;
    {
        const long long N = a.N[k], sumx = a.sumx[k], npad = np - N;
        const int L = a.L[k];
        for (int i = tid; i < cells; i += blockDim.x) {
            // the active count from the cumulative counts, then the branch sums
            const int ti = s_t[i], rl = i / NL, lj = i % NL;  // ti in [0, L + 1]
            const long long count = ti <= 0 ? N : (ti > L ? 0 : N - (long long)a.cdf[a.hist_off[k] + ti - 1]);
            // sum |x - c| over the samples and the padding zeros; with y = x - c, max(y, 0) = (y + |y|) / 2
            const long long c = max(ti, 1) - 1;  // x >= t exactly when x > c, or always for t = 0, where c = 0 serves too
            const long long sum_abs = sums[i] - npad * c;
            const long long sum_relu = (sumx - N * c + sum_abs) / 2;  // each sample adds y + |y| = 2 relu(y)
            const long long sum = sum_relu + c * count;               // sum_{x >= t} x
            // each sample on its own branch of phi (exact integer sums): V = c_w eta - nu x below t,
            // U = c_p (L - eta) - mu (L - x) from t on; no large term cancels another
            const double lam = s_lam[lj];
            const double tot = branch_sum(cp, cw, dmin_nonneg(lam, cp), dmin_nonneg(lam, cw), L,
                                          a.r[r_cta0 + rl] - a.L_in[k], N, count, sumx - sum, (long long)L * count - sum);
            const double S = __dmul_rn(tot, a.inv_n[k]);
            s_S[i] = S;  // in place of the sum, which only this thread reads
            s_Sf[rl * lay.stride_f + lj] = cut(S, ok);
            if (a.S_out) {
                const size_t o = (((size_t)m * a.K + k) * a.R + r_cta0 + rl) * NL + lj;
                if (a.f32_out) static_cast<float*>(a.S_out)[o] = (float)S;
                else static_cast<double*>(a.S_out)[o] = S;
            }
        }
        for (int i = tid; i < rows * 4; i += blockDim.x)
            if (NL + (i & 3) < four(NL)) s_Sf[(i >> 2) * lay.stride_f + NL + (i & 3)] = INFINITY;
        for (int j = tid; j < four(NL); j += blockDim.x) s_lamf[j] = j < NL ? cut_factor(s_lam[j], ok) : 0.f;
    }
    if (!ok) s_bad = 1;
    __syncthreads();
    const LamRows x = {s_S, s_lam, s_eps, s_Sf, s_lamf, NL, lay.stride_f, rows, NL, s_bad == 0};
    if (a.f32_out) lam_min_epilogue<true>(a, x, r_cta0, m, k);
    else lam_min_epilogue<false>(a, x, r_cta0, m, k);
}

// The same cells in O(1) each from the class's cumulative counts C[v] = #{x <= v} and sums
// CS[v] = sum_{x <= v} x: the samples with kappa x + d > 0 are exactly x >= t for the integer
// threshold t, so sum_n max(kappa x_n + d, 0) = kappa (sum - CS[t-1]) + d (N - C[t-1]).
//
// The FP64 pipe bounds it, so a cell whose samples all lie on one branch of phi -- an FP32 look at its
// offset settles most of those -- costs three FP64 instructions (one product less its row's
// rounded constant, and 1 / N) and the others about twelve; what depends on the reservation or on
// lam alone is formed once per CTA, and the minimum over lam leaves about one value per
// (r, eps) pair to FP64.
//
// A warp takes up to kEnvPasses passes of 32 / W rows, W lanes along lam each (W: NL rounded up to a power of
// two, at most 32), so small lam grids fill the warp with rows.  More passes share the CTA's start and end
// (128 regimes x 8 classes x 2048 r x 64 lam x 16 eps: 4 passes 3.33 ms, 3 3.58, 2 3.70); fewer where the
// grid leaves an SM fewer than eight CTAs, or rows so wide that two CTAs fill an SM's shared memory (more
// than 64 lam).  With 1, 4, 8, 16 and 64 CTAs in eight's place: 8 classes x 2048 r x 64 lam x 16 eps x 2 regimes 90.1, 90.0,
// 89.4, 96.6 and 96.7 us, 4 regimes 141.9, 141.9, 142.0, 145.0 and 168.2; one regime x 8 eps 57.0, 56.7, 59.6, 59.5 and 59.4.
constexpr int kEnvThreads = 256;
constexpr int kEnvPasses = 4;

__host__ __device__ inline int env_width(int NL) {
    int w = 1;
    while (w < NL && w < 32) w <<= 1;
    return w;
}
inline int env_rows(int NL, int64_t R, int64_t classes, int sms) {
    const int rows = kEnvThreads / env_width(NL);
    int passes = NL <= 64 ? kEnvPasses : 2;
    while (passes > 1 && classes * ((R + passes * rows - 1) / (passes * rows)) < 8 * (int64_t)sms) passes /= 2;
    return passes * rows;
}

struct EnvRow {
    RowOffset off;
    double pv, ev, pu, eu;  // c_w eta N and c_p (L - eta) N: rounded product and its error
    float cp_le, cw_eta;
    int eta;
};
struct EnvSmem {
    size_t kap, eps, S, row, muf, kapf, lamf, Sf, total;
    int stride, stride_f;  // elements per row of S and Sf
};
__host__ __device__ inline EnvSmem env_smem(int rows, int NL, int E) {
    EnvSmem s;
    const int n4 = four(NL);
    s.stride = NL | 1;  // odd: rows start in other banks
    s.stride_f = float_stride(NL);
    s.kap = 8 * (size_t)NL;
    s.eps = s.kap + 8 * (size_t)NL;
    s.S = s.eps + 8 * (size_t)E;
    s.row = s.S + 8 * (size_t)rows * s.stride;
    s.lamf = (s.row + sizeof(EnvRow) * rows + 15) & ~(size_t)15;
    s.Sf = s.lamf + 4 * (size_t)n4;
    s.muf = s.Sf + 4 * (size_t)rows * s.stride_f;
    s.kapf = s.muf + 4 * (size_t)NL;
    s.total = s.kapf + 4 * (size_t)NL;
    return s;
}

__global__ void __launch_bounds__(kEnvThreads) k_envelope(const GridArgs a) {
    extern __shared__ __align__(16) unsigned char esm[];
    __shared__ int s_bad[2];  // some magnitude the floats do not hold: in the inputs, in S
    __shared__ int s_first_sat, s_unsorted;
    const EnvSmem lay = env_smem(a.rows, a.NL, a.E);
    double* s_lam = reinterpret_cast<double*>(esm);
    double* s_kap = reinterpret_cast<double*>(esm + lay.kap);
    double* s_eps = reinterpret_cast<double*>(esm + lay.eps);
    double* s_S = reinterpret_cast<double*>(esm + lay.S);
    EnvRow* s_row = reinterpret_cast<EnvRow*>(esm + lay.row);
    float* s_lamf = reinterpret_cast<float*>(esm + lay.lamf);
    float* s_Sf = reinterpret_cast<float*>(esm + lay.Sf);
    float* s_muf = reinterpret_cast<float*>(esm + lay.muf);
    float* s_kapf = reinterpret_cast<float*>(esm + lay.kapf);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int b = blockIdx.x;
    const int rb = b % a.r_blocks;
    b /= a.r_blocks;
    const int k = b % a.K;
    const int m = a.m0 + b / a.K;
    const int NL = a.NL, W = env_width(NL);
    const int r_cta0 = rb * a.rows, rows = min(a.rows, a.R - r_cta0);
    const double cp = a.cp[m], cw = a.cw[m];
    const int L = a.L[k];
    const long long N = a.N[k], sumx = a.sumx[k];
    if (tid < 2) s_bad[tid] = 0;
    if (tid == 0) {
        s_first_sat = a.NL - 1;
        s_unsorted = 0;
    }
    __syncthreads();
    bool ok = true;
    for (int i = tid; i < rows; i += kEnvThreads) {
        const int eta = a.r[r_cta0 + i] - a.L_in[k];
        EnvRow w;
        w.off = row_offset(cp, cw, L, eta);
        const double iv = to_double((long long)eta * N), iu = to_double((long long)(L - eta) * N);
        w.pv = __dmul_rn(cw, iv);
        w.ev = fma(cw, iv, -w.pv);
        w.pu = __dmul_rn(cp, iu);
        w.eu = fma(cp, iu, -w.pu);
        w.cp_le = cut(w.off.cp_le, ok);
        w.cw_eta = cut(w.off.cw_eta, ok);
        w.eta = eta;
        s_row[i] = w;
    }
    for (int i = tid; i < NL; i += kEnvThreads) {
        const double l = a.lam[i], mu = dmin_nonneg(l, cp), nu = dmin_nonneg(l, cw), kap = __dadd_rn(mu, nu);
        s_lam[i] = l;
        s_kap[i] = kap;
        if (dbits(l) >= dbits(cp) && dbits(l) >= dbits(cw)) atomicMin(&s_first_sat, i);
        if (i > 0 && !(dbits(a.lam[i - 1]) <= dbits(l))) s_unsorted = 1;
        s_lamf[i] = cut_factor(l, ok);
        s_muf[i] = cut(mu, ok);
        s_kapf[i] = cut(kap, ok);
    }
    for (int i = tid; i < a.E; i += kEnvThreads) s_eps[i] = a.eps[i];
    if (!ok) s_bad[0] = 1;
    __syncthreads();
    const bool floats = s_bad[0] == 0;
    // Every lam from max(c_p, c_w) on gives the same S (mu = c_p, nu = c_w), and in an ascending grid the
    // first of them costs least at every radius, with the lowest index: the rest need no evaluation.
    const int NLs = s_unsorted ? NL : s_first_sat + 1;
    const double inv_n = a.inv_n[k], Ld = to_double(L), sumx_d = to_double(sumx);
    const long long dist_all = (long long)L * N - sumx;
    const double dist_d = to_double(dist_all);
    const float Lf = (float)L;
    const int32_t* C = a.cdf + a.hist_off[k];
    const int64_t* CS = a.csum + a.hist_off[k];
    for (int rl = warp * (32 / W) + lane / W; rl < rows; rl += kEnvThreads / W) {
        const EnvRow& w = s_row[rl];
        for (int j = lane & (W - 1); j < NLs; j += W) {
            const double lam = s_lam[j], mu = dmin_nonneg(lam, cp), nu = dmin_nonneg(lam, cw);
            // d in FP32, off by at most 2^-21 of the sum of its parts: far enough from zero, and kappa L + d
            // likewise, it tells that every sample is active (t = 0) or that none is (t = L + 1)
            const float part = fmaf(s_muf[j], Lf, w.cw_eta), d = w.cp_le - part, parts = w.cp_le + part;
            const float top = fmaf(s_kapf[j], Lf, d);
            int t;
            if (floats && parts > 0x1p-40f && d > 0x1p-20f * parts) t = 0;
            else if (floats && parts > 0x1p-40f && top < -0x1p-19f * parts) t = L + 1;
            else t = first_active(s_kap[j], excess_offset(w.off, cp, mu, Ld), L);
            const bool inside = t >= 1 && t <= L;
            const long long below_n = inside ? (long long)C[t - 1] : (t >= 1 ? N : 0);
            const long long cnt = N - below_n;  // samples from t on
            // sum phi: the branch sums (branch_sum) with the row's own products where one branch holds all
            double p = cnt == 0 ? w.pv : w.pu, e = cnt == 0 ? w.ev : w.eu, mul = cnt == 0 ? nu : mu;
            double by = cnt == 0 ? sumx_d : dist_d;
            long long below_s = 0;
            const bool both = cnt > 0 && cnt < N;
            if (both) {
                below_s = CS[t - 1];
                const double i = to_double((long long)w.eta * below_n);
                p = __dmul_rn(cw, i);
                e = fma(cw, i, -p);
                mul = nu;
                by = to_double(below_s);
            }
            double tot = __dadd_rn(fma(-mul, by, p), e);
            if (both)
                tot = __dadd_rn(tot, diff_of_products(cp, to_double((long long)(L - w.eta) * cnt), mu,
                                                      to_double((long long)L * cnt - (sumx - below_s))));
            const double S = __dmul_rn(tot, inv_n);
            s_S[rl * lay.stride + j] = S;
            s_Sf[rl * lay.stride_f + j] = cut(S, ok);
            if (a.S_out) {
                double* out = static_cast<double*>(a.S_out) + (((size_t)m * a.K + k) * a.R + r_cta0 + rl) * a.NL;
                out[j] = S;
                if (j == NLs - 1)
                    for (int i = NLs; i < NL; i++) out[i] = S;
            }
        }
        for (int j = NLs + (lane & (W - 1)); j < four(NLs); j += W) s_Sf[rl * lay.stride_f + j] = INFINITY;
    }
    for (int j = NL + tid; j < four(NL); j += kEnvThreads) s_lamf[j] = 0.f;
    if (!ok) s_bad[1] = 1;
    __syncthreads();
    const LamRows rows_of = {s_S, s_lam, s_eps, s_Sf, s_lamf, lay.stride, lay.stride_f, rows, NLs, floats && s_bad[1] == 0};
    lam_min_epilogue<false>(a, rows_of, r_cta0, m, k);
}

template <bool F32>
__global__ void k_finalize(const FinalizeArgs a) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (int64_t)a.M * a.E * a.K) finalize_row<F32>(a, i, (int)(i % a.K));
}

}  // namespace

template <class C>
GridShape shape_for(int variant, int32_t R, int32_t NL, int32_t E) {
    GridShape sh;
    sh.variant = variant;
    sh.LT = (NL + C::TL - 1) / C::TL;
    sh.RG = sh.LT >= kWarpsTarget ? 1 : kWarpsTarget / sh.LT;
    sh.threads = 32 * sh.LT * sh.RG;
    sh.rows = sh.RG * C::TR;
    sh.r_blocks = (R + sh.rows - 1) / sh.rows;
    sh.smem = smem_layout(sh.RG, C::TR, sh.LT * C::TL, E, C::CHUNK * C::BYTES, C::STAGES).total;
    return sh;
}

// Rows per CTA and passes over the samples.  A pass is 256 cells (16 warps); more passes lay a CTA's rows
// over more of them, so that fewer cells stand empty at the end, but leave fewer CTAs to fill the last wave.
// The choice maximises cells filled x waves filled.  A warp left out saves nothing while its scheduler still
// holds as many as the others (13 to 16 warps take the same time), and fewer per scheduler run at a lower
// rate: 5 classes x 1001 r x 200 lam x 3 regimes 2.27 ms in one pass of 13 warps, 1.90 in four passes of 16
// (2.09 in 2 r x 8 lam tiles with a second launch past 128 lam).  At 5 classes x 40,000 samples x 1001 r x 3 regimes and
// 13 lam counts from 1 to 250 the choice takes at most 3 % longer than the best of the four (33 lam: 769 us in one
// pass, 748 in two; 129: 2791 in three, 3145 in one).  In grids under two waves it can miss: one regime x 200 r, one
// pass against the choice, 129 lam 252 and 313 us, 150 lam 268 and 337 (366 in blocks of 128 lam, the form before);
// 72 lam 128 in two passes and 165.
GridShape exact_shape(int32_t R, int32_t NL, int32_t E, int32_t K, int64_t classes, int sms) {
    constexpr int kCells = kExactWarps * kExactV;
    GridShape best, sh;
    sh.variant = 3;
    sh.LT = sh.RG = 1;
    double best_score = -1.0;
    for (int passes = 1; passes <= kExactMaxPasses; passes++) {
        const int rows = std::min(R, passes * kCells / NL);
        if (rows < 1) continue;
        const int tiles = (rows * NL + kExactV - 1) / kExactV;
        sh.rows = rows;
        sh.passes = (tiles + kExactWarps - 1) / kExactWarps;
        const int warps = (tiles + sh.passes - 1) / sh.passes;
        sh.threads = 32 * warps;
        sh.r_blocks = (R + rows - 1) / rows;
        if ((int64_t)K * sh.r_blocks > 0x7fffffffLL) continue;  // a launch holds one regime's CTAs (four passes always do)
        // 96 KB of ring: three chunks of 8192 samples (6144 measured 1 % slower, 4096 3 %); smaller chunks where
        // the cells need the room
        sh.chunk = kExactChunk;
        do {
            sh.smem = exact_smem(rows, NL, E, warps * sh.passes, kExactStages * sh.chunk * 4).total;
        } while (sh.smem > kExactSmem && (sh.chunk -= 1024) > 0);
        const double slots = (double)kExactBlocks * sms, ctas = (double)classes * sh.r_blocks, waves = ctas / slots;
        const int held = (warps + 3) / 4 * 4;  // warps that the fullest of the four schedulers accounts for
        const double filled = (double)R * NL / ((double)sh.r_blocks * held * sh.passes * kExactV);
        const double rate = 0.55 + 0.45 * held / kExactWarps;
        const double score = filled * rate * waves / std::ceil(waves);
        if (score > best_score + 0.01) {
            best_score = score;
            best = sh;
        }
    }
    return best;
}

GridShape grid_shape(Prec p, int32_t R, int32_t NL, int32_t E, int32_t K, int32_t M, int sms) {
    const int64_t classes = (int64_t)M * K;
    if (p == Prec::ENVELOPE) {
        GridShape sh;
        sh.variant = 4;
        sh.LT = sh.RG = 1;
        sh.threads = kEnvThreads;
        sh.rows = env_rows(NL, R, classes, sms);
        sh.r_blocks = (R + sh.rows - 1) / sh.rows;
        sh.smem = env_smem(sh.rows, NL, E).total;
        return sh;
    }
    if (p == Prec::F64) return shape_for<CfgF64>(2, R, NL, E);
    if (p == Prec::EXACT) return exact_shape(R, NL, E, K, classes, sms);
    if (NL <= kWarpsTarget * CfgF32::TL) return shape_for<CfgF32>(0, R, NL, E);
    return shape_for<CfgF32Wide>(1, R, NL, E);
}

namespace {

cudaError_t allow_smem(const void* kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// The largest layout the kernel's shapes can have: all of its warps, 64 eps.
template <class C>
cudaError_t prepare() {
    const int warps = C::MAXT / 32;
    size_t most = 0;
    for (int lt = 1; lt <= warps; lt++)
        most = std::max(most, smem_layout(std::max(1, kWarpsTarget / lt), C::TR, lt * C::TL, 64, C::CHUNK * C::BYTES, C::STAGES).total);
    return allow_smem((const void*)k_grid<C>, most);
}

}  // namespace

cudaError_t grid_prepare(Prec p) {
    if (p == Prec::F64) return prepare<CfgF64>();
    if (p == Prec::EXACT) {
        return allow_smem((const void*)k_exact, kExactSmem);
    }
    if (p == Prec::ENVELOPE) {
        size_t most = 0;
        for (int nl = 1; nl <= 256; nl++) most = std::max(most, env_smem(env_rows(nl, 1 << 20, 1 << 20, 1), nl, 64).total);
        return allow_smem((const void*)k_envelope, most);
    }
    cudaFuncAttributes at;
    cudaError_t e = prepare<CfgF32>();
    if (e == cudaSuccess) e = prepare<CfgF32Wide>();
    return e == cudaSuccess ? cudaFuncGetAttributes(&at, (const void*)k_finalize<true>) : e;
}

cudaError_t launch_grid(Prec p, const GridShape& sh, GridArgs a, cudaStream_t s) {
    a.LT = sh.LT;
    a.RG = sh.RG;
    a.rows = sh.rows;
    a.passes = sh.passes;
    a.chunk = sh.chunk;
    a.r_blocks = sh.r_blocks;
    const int64_t nblocks = (int64_t)a.m_count * a.K * a.r_blocks;
    if (nblocks <= 0 || nblocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    if (p == Prec::ENVELOPE) k_envelope<<<(unsigned)nblocks, sh.threads, sh.smem, s>>>(a);
    else if (p == Prec::F64) k_grid<CfgF64><<<(unsigned)nblocks, sh.threads, sh.smem, s>>>(a);
    else if (p == Prec::EXACT) k_exact<<<(unsigned)nblocks, sh.threads, sh.smem, s>>>(a);
    else if (sh.variant == 0) k_grid<CfgF32><<<(unsigned)nblocks, sh.threads, sh.smem, s>>>(a);
    else k_grid<CfgF32Wide><<<(unsigned)nblocks, sh.threads, sh.smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_finalize(Prec p, const FinalizeArgs& a, cudaStream_t s) {
    const int64_t n = (int64_t)a.M * a.E * a.K;
    const int threads = 256;
    const unsigned blocks = (unsigned)((n + threads - 1) / threads);
    if (p == Prec::F32) k_finalize<true><<<blocks, threads, 0, s>>>(a);
    else k_finalize<false><<<blocks, threads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace kvdro
