// Segmented counting sort of bounded integer samples, per-class cumulative counts, and the
// quantile gather.  The samples are their own sort keys and are bounded by L_k, so class k's
// sorted order is fully determined by its histogram over [0, L_k]: histogram -> inclusive scan
// (the cumulative count C[v] = #{x <= v}, i.e. N times the empirical CDF) -> expansion of every
// output position p into the smallest v with C[v] > p.  The scan also records, for every tile of
// kExpandTile output positions, the bin its first position falls in; the expansion then searches the
// bins of its tile's range.  It also writes the samples in the form that the grid kernel streams
// (kvdro_internal.cuh), padded to a multiple of kPadSamples per class.
#include <math.h>

#include <algorithm>

#include "kvdro_internal.cuh"

namespace kvdro {
namespace {

constexpr int kHistThreads = 512;
constexpr int64_t kHistSlice = 65535;  // samples per histogram block: its counts fit 16 bits
// Bins [0, 2 kHistWords) are privatised in shared memory (66 KB, three blocks per SM), bin v in the low and
// v + kHistWords in the high half of word v: neighbouring values, the frequent ones, stay in words of their
// own.  A class whose support they cover counts without the global path, whose mere presence in the loop
// costs as much again: 32 M samples of support 32768 in 37 us (3.4 TB/s); 67 with the upper half counted in global memory.
// Three blocks of 66 KB are what an SM holds; the line shows no step (loading 32 M samples spread evenly over the
// support: 149 us at 32895, 152 at 32896), above it the share of samples past the bins counts: 188 us at 40000, 231 at 65535.
constexpr int kHistWords = 16448;
constexpr int kScanThreads = 512;
constexpr int kScanPer = 8;
constexpr int64_t kScanTile = (int64_t)kScanThreads * kScanPer;  // bins per scan block
constexpr int kExpandThreads = 256;
constexpr int64_t kExpandTile = 4096;  // sorted positions per expansion block
// Tiles whose positions lie among at least kSparseBins bins lay their runs out in shared memory instead of
// searching: 1.6 M samples of support 32768 in 24 us instead of 36 (search; 35 with a limit of 16384 bins), 3,000
// of support 8192 in 10 instead of 18, 32 M in 52 instead of 57.  From 256, 512 or 1024 bins on the same within
// 2 us.  Past kSparseMost the bins' loads outweigh the search (16 M of support 131072: 73 against 63).
constexpr int kSparseBins = 512;
constexpr int kSparseMost = 40960;
// Histogram slices get at least this many samples, so that counting outweighs clearing and
// flushing the block's shared bins.
constexpr int64_t kHistMinSlice = kHistWords;

__device__ __forceinline__ int find_segment(const int32_t* prefix, int K, int b) {
    // largest k with prefix[k] <= b; prefix is strictly increasing, prefix[0] = 0
    int lo = 0, hi = K;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (prefix[mid] <= b) lo = mid; else hi = mid;
    }
    return lo;
}

// Counts src[beg, end) into the block's bins; returns how many samples lie outside [0, L].  An unsigned
// comparison is the whole range check (a negative x wraps above L).
template <bool COVERED>
__device__ __forceinline__ int count_slice(const int32_t* src, int64_t beg, int64_t end, uint32_t L, uint32_t* bins,
                                           int32_t* gh) {
    int bad = 0;
    auto count = [&](int32_t x) {
        const uint32_t u = (uint32_t)x;
        const bool ok = u <= L;
        bad += ok ? 0 : 1;
        if (COVERED ? ok : ok && u < 2 * kHistWords) atomicAdd(bins + (u < kHistWords ? u : u - kHistWords), u < kHistWords ? 1u : 65536u);
        if (!COVERED && ok && u >= 2 * kHistWords) atomicAdd(gh + u, 1);
    };
    // 16-byte loads of four samples over the slice's aligned middle (alignment is taken from the
    // address: `lengths` is the caller's pointer): each thread loads its next two vectors before
    // it counts the current two, so four loads are in flight while the atomics run; the unaligned
    // head and the tail one sample at a time.
    const int64_t mis = (int64_t)((reinterpret_cast<uintptr_t>(src + beg) >> 2) & 3);
    const int64_t vbeg = min(end, beg + ((4 - mis) & 3));
    const int nvec = (int)((end - vbeg) >> 2);
    const int64_t vend = vbeg + 4 * (int64_t)nvec;
    for (int64_t i = beg + threadIdx.x; i < vbeg; i += kHistThreads) count(__ldg(src + i));
    const int4* v4 = reinterpret_cast<const int4*>(src + vbeg);
    auto four = [&](const int4 v) { count(v.x), count(v.y), count(v.z), count(v.w); };
    int q = threadIdx.x;
    int4 u = q < nvec ? __ldg(v4 + q) : int4(), w = q + kHistThreads < nvec ? __ldg(v4 + q + kHistThreads) : int4();
    for (; q + kHistThreads < nvec; q += 2 * kHistThreads) {
        const int n = q + 2 * kHistThreads;
        const int4 u2 = n < nvec ? __ldg(v4 + n) : int4(), w2 = n + kHistThreads < nvec ? __ldg(v4 + n + kHistThreads) : int4();
        four(u);
        four(w);
        u = u2;
        w = w2;
    }
    if (q < nvec) four(u);
    for (int64_t i = vend + threadIdx.x; i < end; i += kHistThreads) count(__ldg(src + i));
    return bad;
}

__global__ void __launch_bounds__(kHistThreads) k_histogram(SortArgs a) {
    extern __shared__ uint32_t sh_bins[];
    const int k = find_segment(a.hist_blocks, a.K, blockIdx.x);
    // the class's samples in equal slices, one per block (at most kHistSlice each)
    const int64_t nblk = a.hist_blocks[k + 1] - a.hist_blocks[k];
    const int64_t slice_len = (a.offsets[k + 1] - a.offsets[k] + nblk - 1) / nblk;
    const int64_t slice = blockIdx.x - a.hist_blocks[k];
    const int64_t beg = a.offsets[k] + slice * slice_len;
    const int64_t end = min(a.offsets[k + 1], beg + slice_len);
    const int32_t Lk = a.L[k];
    const int words = min(Lk + 1, kHistWords);
    int32_t* gh = a.hist + a.hist_off[k];
    for (int v = threadIdx.x; v < words; v += kHistThreads) sh_bins[v] = 0;
    __syncthreads();
    int bad = Lk < 2 * kHistWords ? count_slice<true>(a.lengths, beg, end, Lk, sh_bins, gh)
                                  : count_slice<false>(a.lengths, beg, end, Lk, sh_bins, gh);
    __syncthreads();
    for (int v = threadIdx.x; v < words; v += kHistThreads) {
        const uint32_t c = sh_bins[v];
        if (c & 0xffffu) atomicAdd(gh + v, (int32_t)(c & 0xffffu));
        if (c >> 16) atomicAdd(gh + v + kHistWords, (int32_t)(c >> 16));
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && bad) atomicAdd(a.err, bad);
}

// The cumulative counts and sums of every class over tiles of kScanTile bins, one block per (tile, class)
// so that every SM takes part: each tile's inclusive scan, offset by the class's earlier tiles, whose
// totals (count, sum of v h[v]) come from a pass before it.  Where the cumulative counts have an array of
// their own (up to 16 tiles a class) a block sums the earlier tiles' bins itself instead (they
// lie in L2), which saves the pass: 32 classes x 32769 bins took
// 6 + 15 us in two passes of 1024 threads with eleven barriers, 14 us now.
struct CountSum {
    int32_t c;
    long long v;
};
__device__ __forceinline__ CountSum operator+(CountSum x, CountSum y) { return {x.c + y.c, x.v + y.v}; }

__device__ __forceinline__ CountSum shfl_up(CountSum x, int o) {
    return {__shfl_up_sync(0xffffffffu, x.c, o), __shfl_up_sync(0xffffffffu, x.v, o)};
}
__device__ __forceinline__ CountSum warp_sum(CountSum x) {
#pragma unroll
    for (int o = 16; o; o >>= 1)
        x = x + CountSum{__shfl_xor_sync(0xffffffffu, x.c, o), __shfl_xor_sync(0xffffffffu, x.v, o)};
    return x;
}

// A lane's bins: kScanPer, 32 apart, from the warp's first (out of range: 0).
__device__ __forceinline__ void load_bins(const int32_t* h, int64_t first, int64_t n, CountSum (&t)[kScanPer]) {
#pragma unroll
    for (int j = 0; j < kScanPer; j++) {
        const int64_t i = first + 32 * j;
        const int32_t x = i < n ? h[i] : 0;
        t[j] = {x, i * x};
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_totals(SortArgs a) {
    __shared__ CountSum s_warp[kScanThreads / 32];
    const int k = blockIdx.y, lane = threadIdx.x & 31;
    const int64_t n = (int64_t)a.L[k] + 1, b0 = (int64_t)blockIdx.x * kScanTile;
    if (b0 >= n) return;  // the class has fewer tiles
    CountSum bins[kScanPer], t = {0, 0};
    load_bins(a.hist + a.hist_off[k], b0 + (threadIdx.x >> 5) * (32 * kScanPer) + lane, n, bins);
#pragma unroll
    for (int j = 0; j < kScanPer; j++) t = t + bins[j];
    t = warp_sum(t);
    if (lane == 0) s_warp[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x < 32) {
        const CountSum s = warp_sum(lane < kScanThreads / 32 ? s_warp[lane] : CountSum{0, 0});
        if (lane == 0) {
            const int64_t o = (int64_t)k * a.scan_tiles + blockIdx.x;
            a.tile_tot[2 * o] = s.c;
            a.tile_tot[2 * o + 1] = s.v;
        }
    }
}

__global__ void __launch_bounds__(kScanThreads, 2) k_scan_apply(SortArgs a) {
    __shared__ CountSum s_warp[kScanThreads / 32], s_carry[kScanThreads / 32];
    const int k = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = (int64_t)a.L[k] + 1, b0 = (int64_t)blockIdx.x * kScanTile;
    if (b0 >= n) return;
    const int32_t* h = a.hist + a.hist_off[k];
    // the thread's share of the class's earlier tiles
    CountSum carry = {0, 0};
    if (a.cum != a.hist) {
#pragma unroll 8
        for (int i = threadIdx.x; i < (int)b0; i += kScanThreads) {
            const int32_t x = h[i];
            carry = carry + CountSum{x, (long long)i * x};
        }
    } else {
        for (int u = threadIdx.x; u < (int)blockIdx.x; u += kScanThreads) {
            const int64_t o = (int64_t)k * a.scan_tiles + u;
            carry = carry + CountSum{(int32_t)a.tile_tot[2 * o], (long long)a.tile_tot[2 * o + 1]};
        }
    }
    // the warp's rows of 32 bins: a scan of each, offset by the rows before
    const int64_t i0 = b0 + warp * (32 * kScanPer) + lane;
    CountSum own[kScanPer], incl[kScanPer];
    load_bins(h, i0, n, own);
#pragma unroll
    for (int j = 0; j < kScanPer; j++) incl[j] = own[j];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int j = 0; j < kScanPer; j++) {
            const CountSum y = shfl_up(incl[j], o);
            if (lane >= o) incl[j] = incl[j] + y;
        }
    CountSum row = {0, 0};
#pragma unroll
    for (int j = 0; j < kScanPer; j++) {
        const CountSum total = {__shfl_sync(0xffffffffu, incl[j].c, 31), __shfl_sync(0xffffffffu, incl[j].v, 31)};
        incl[j] = incl[j] + row;
        row = row + total;
    }
    carry = warp_sum(carry);
    if (lane == 0) {
        s_warp[warp] = row;
        s_carry[warp] = carry;
    }
    __syncthreads();
    CountSum before = {0, 0};  // the earlier tiles, and the tile's earlier warps
    if (lane < kScanThreads / 32) {
        before = s_carry[lane];
        if (lane < warp) before = before + s_warp[lane];
    }
    before = warp_sum(before);
    // For the expansion: tile_lo[q] = the bin holding position q * kExpandTile for each tile q of
    // the class's sorted samples, and one more entry: the bin holding the last position, N - 1.
    // Every position lies in exactly one bin's run [C[v] - h[v], C[v]), so each entry is written once.
    const int64_t Nk = a.offsets[k + 1] - a.offsets[k];
    const int64_t tiles = (Nk + kExpandTile - 1) / kExpandTile;
    int32_t* tl = a.tile_lo + a.exp_blocks[k] + k;
    long long* cs = a.csum ? reinterpret_cast<long long*>(a.csum + a.hist_off[k]) : nullptr;
    int32_t* cum = a.cum + a.hist_off[k];
#pragma unroll
    for (int j = 0; j < kScanPer; j++) {
        const int64_t i = i0 + 32 * j;
        if (i >= n) break;
        const CountSum at = before + incl[j];
        const int64_t hi = at.c, lo = hi - own[j].c;
        cum[i] = (int32_t)hi;
        if (cs) cs[i] = at.v;
        if (i == n - 1) a.sumx[k] = at.v;
        if (lo < hi) {
            for (int64_t q = (lo + kExpandTile - 1) / kExpandTile; q * kExpandTile < hi && q < tiles; q++) tl[q] = (int32_t)i;
            if (lo <= Nk - 1 && Nk - 1 < hi) tl[tiles] = (int32_t)i;
        }
    }
}

// Smallest v in [lo, hi] with C[v] > p (C[hi] > p).
__device__ __forceinline__ int32_t value_at(const int32_t* C, int32_t lo, int32_t hi, int32_t p) {
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (__ldg(C + mid) > p) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// The sorted samples and their staged form, four consecutive positions per thread, 128 per warp and step.
// Where the tile's bins outnumber its runs (kSparseBins) the block lays the runs out in shared memory, eight
// bins' counts a thread and round, runs of more than eight positions by the whole warp.  Elsewhere
// a warp first searches the values at the ends of its steps, a lane each, among the bins of the tile's
// position range (recorded by the scan).  Where they are the same -- runs of equal samples are long where
// samples are many -- that is all; up to 31 bins apart each lane finds its first position among the run
// ends that the lanes hold, and otherwise by a search of its own: no shared memory, no
// barrier.  16-byte stores: 32 M samples in 52 us (4.9 TB/s of stores); a running maximum over run
// starts marked in shared memory took 86, a search per thread 75.
__global__ void __launch_bounds__(kExpandThreads) k_expand(SortArgs a) {
    constexpr int kWarps = kExpandThreads / 32, kSteps = (int)kExpandTile / 128 / kWarps;  // per warp
    const int k = find_segment(a.exp_blocks, a.K, blockIdx.x);
    const unsigned q = blockIdx.x - a.exp_blocks[k];
    // positions fit 32 bits: a class has at most 2^31 - 1 samples, padded to a multiple of 128
    const unsigned N = (unsigned)(a.offsets[k + 1] - a.offsets[k]), padk = (unsigned)(a.pair_off[k + 1] - a.pair_off[k]);
    const int32_t* C = a.cum + a.hist_off[k];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (a.inv_n && q == 0 && threadIdx.x == 0) a.inv_n[k] = 1.0 / (double)N;
    const unsigned p0 = q * (unsigned)kExpandTile;
    const int32_t* tl = a.tile_lo + a.exp_blocks[k] + k;
    // (samples out of range leave positions that no bin holds: entries not written by this load's scan)
    auto bin = [&](unsigned i) { return p0 < N ? min(max(tl[i], 0), a.L[k]) : 0; };
    const int32_t v_lo = bin(q), v_hi = bin(q + 1);
    __shared__ __align__(16) int32_t s_x[kExpandTile];  // a sparse tile's values
    const bool sparse = v_hi - v_lo >= kSparseBins && v_hi - v_lo < kSparseMost;
    if (sparse) {
        for (int i = threadIdx.x; i < (int)kExpandTile / 4; i += kExpandThreads)  // (positions no bin holds, as above)
            reinterpret_cast<int4*>(s_x)[i] = make_int4(v_hi, v_hi, v_hi, v_hi);
        __syncthreads();
        const int p1 = (int)min(N - p0, (unsigned)kExpandTile);
        constexpr int kPer = 8;
        for (int base = v_lo; base <= v_hi; base += kPer * kExpandThreads) {
            int from[kPer], to[kPer];  // positions in the tile of kPer bins' runs
#pragma unroll
            for (int j = 0; j < kPer; j++) {
                const int v = base + j * kExpandThreads + (int)threadIdx.x;
                from[j] = v <= v_hi && v > 0 ? __ldg(C + v - 1) : 0;
                to[j] = v <= v_hi ? __ldg(C + v) : 0;
            }
#pragma unroll
            for (int j = 0; j < kPer; j++) {
                const int v = base + j * kExpandThreads + (int)threadIdx.x;
                int f = max(from[j] - (int)p0, 0);
                const int e = min(to[j] - (int)p0, p1);
                for (unsigned wide = __ballot_sync(0xffffffffu, e - f > 8); wide; wide &= wide - 1) {  // by the warp
                    const int src = __ffs(wide) - 1, fv = __shfl_sync(0xffffffffu, f, src);
                    const int ev = __shfl_sync(0xffffffffu, e, src), vv = __shfl_sync(0xffffffffu, v, src);
                    for (int i = fv + lane; i < ev; i += 32) s_x[i] = vv;
                }
                if (e - f <= 8)
                    for (; f < e; f++) s_x[f] = v;
            }
        }
        __syncthreads();
    }
    // lanes 2i, 2i + 1: the values at the start of the warp's step i and just past its end
    int32_t ends = v_hi;
    if (!sparse) {
        const unsigned p = p0 + 128 * (warp + kWarps * (lane >> 1) + (lane & 1));
        if (lane < 2 * kSteps && p < N) ends = value_at(C, v_lo, v_hi, (int)p);
    }
    int32_t* sorted = a.sorted + a.offsets[k];
    float* staged = static_cast<float*>(a.staged) + a.pair_off[k] * (a.quads ? 1 : 2);
    const bool aligned = (a.offsets[k] & 3) == 0;
#pragma unroll 2
    for (int i = 0; i < kSteps; i++) {
        const unsigned first = p0 + 128 * (warp + kWarps * i), at = first + 4 * lane;
        if (first >= padk) break;  // warp-uniform; padk is a multiple of 128
        const int32_t vf = __shfl_sync(0xffffffffu, ends, 2 * i), vl = __shfl_sync(0xffffffffu, ends, 2 * i + 1);
        if (!sparse && vf == vl && first + 128 <= N && aligned && a.quads) {  // one run
            *reinterpret_cast<int4*>(sorted + at) = make_int4(vf, vf, vf, vf);
            *reinterpret_cast<int4*>(staged + at) = make_int4(4 * vf, 2 * vf, 0, 0);
            continue;
        }
        const int left = at < N ? (int)min(N - at, 4u) : 0;  // samples among the four
        const int pos = (int)min(at, N - 1);
        int32_t x[4] = {vf, vf, vf, vf};
        if (sparse) {
            const int4 y = reinterpret_cast<const int4*>(s_x)[(at - p0) / 4];
            x[0] = y.x, x[1] = y.y, x[2] = y.z, x[3] = y.w;
        } else if (vl - vf >= 32) {
            x[0] = value_at(C, vf, vl, pos);
            int32_t hi = __shfl_down_sync(0xffffffffu, x[0], 1);
            if (lane == 31) hi = vl;
#pragma unroll
            for (int j = 1; j < 4; j++) {
                x[j] = x[j - 1];
                if (j < left && x[j] < hi && __ldg(C + x[j]) <= pos + j) x[j] = value_at(C, x[j] + 1, hi, pos + j);
            }
        } else if (vl != vf) {  // the ends of the runs of bins vf, vf + 1, ... a lane each, searched through shuffles
            const int32_t end = vf + lane < vl ? __ldg(C + vf + lane) : 0x7fffffff;
            int n = 0;
#pragma unroll
            for (int s = 16; s; s >>= 1)
                if (__shfl_sync(0xffffffffu, end, n + s - 1) <= pos) n += s;
            const int32_t e0 = __shfl_sync(0xffffffffu, end, n), e1 = __shfl_sync(0xffffffffu, end, min(n + 1, 31));
            x[0] = vf + n;
#pragma unroll
            for (int j = 1; j < 4; j++) x[j] = x[0] + (pos + j >= e0);
            if (pos + 3 >= e1 && n < 31)  // a run of fewer than four samples
#pragma unroll
                for (int j = 1; j < 4; j++) x[j] = j < left ? value_at(C, x[j - 1], vl, pos + j) : x[j];
        }
        if (aligned && left == 4) {
            *reinterpret_cast<int4*>(sorted + at) = make_int4(x[0], x[1], x[2], x[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j < left) sorted[at + j] = x[j];
        }
        if (a.quads) {  // of the class's last samples and zeros before them
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j >= left) {
                    x[3] = x[2];
                    x[2] = x[1];
                    x[1] = x[0];
                    x[0] = 0;
                }
            const int low = x[0] + x[1], high = x[2] + x[3];
            *reinterpret_cast<int4*>(staged + at) = make_int4(low + high, x[1] + x[2], x[3] - x[0], high - low);
        } else {  // (x, x) pairs; NaN past the class's samples
            float f[4];
#pragma unroll
            for (int j = 0; j < 4; j++) f[j] = j < left ? (float)x[j] : __int_as_float(0x7fc00000);
            float4* out = reinterpret_cast<float4*>(staged + 2 * (size_t)at);
            out[0] = make_float4(f[0], f[0], f[1], f[1]);
            out[1] = make_float4(f[2], f[2], f[3], f[3]);
        }
    }
}

__global__ void k_gather_quantiles(const int32_t* sorted, const int64_t* offsets, const int32_t* rank, int32_t K,
                                   int32_t F, int32_t* out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)K * F) return;
    const int k = (int)(i / F);
    out[i] = sorted[offsets[k] + rank[i] - 1];
}

}  // namespace

cudaError_t sm_count(int* sms) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e == cudaSuccess ? cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) : e;
}

// Histogram blocks of each class (written as a prefix over the classes): slices of at most
// kHistSlice and at least kHistMinSlice samples, as many as fill whole waves of the device's
// resident histogram blocks -- a last wave only a little filled would leave most SMs idle.
cudaError_t hist_block_prefix(const int64_t* N, int32_t K, int32_t* prefix) {
    int sms = 0, per_sm = 0;
    cudaError_t e = sm_count(&sms);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_histogram, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kHistWords * (int)sizeof(int32_t));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_histogram, kHistThreads,
                                                          kHistWords * sizeof(int32_t));
    if (e != cudaSuccess) return e;
    const int64_t slots = std::max<int64_t>(1, (int64_t)sms * per_sm);
    int64_t total = 0, base = 0;
    for (int32_t k = 0; k < K; k++) {
        total += N[k];
        base += (N[k] + kHistSlice - 1) / kHistSlice;
    }
    const int64_t target = (base + slots - 1) / slots * slots;
    const int64_t slice = std::max<int64_t>(kHistMinSlice, (total + target - 1) / target);
    prefix[0] = 0;
    for (int32_t k = 0; k < K; k++) {
        const int64_t nb = std::max<int64_t>((N[k] + kHistSlice - 1) / kHistSlice, N[k] / slice);
        prefix[k + 1] = (int32_t)std::min<int64_t>(0x7fffffffLL, prefix[k] + std::max<int64_t>(1, nb));
    }
    return cudaSuccess;
}

cudaError_t launch_histogram(const SortArgs& a, int32_t nblocks, cudaStream_t s) {
    // per-device attribute; cheap enough to set on every launch
    cudaError_t e = cudaFuncSetAttribute(k_histogram, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kHistWords * (int)sizeof(int32_t));
    if (e != cudaSuccess) return e;
    k_histogram<<<nblocks, kHistThreads, kHistWords * sizeof(int32_t), s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_scan(const SortArgs& a, cudaStream_t s) {
    const dim3 grid((unsigned)a.scan_tiles, (unsigned)a.K);
    if (a.cum == a.hist) {
        k_scan_totals<<<grid, kScanThreads, 0, s>>>(a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    k_scan_apply<<<grid, kScanThreads, 0, s>>>(a);
    return cudaGetLastError();
}

int64_t scan_tile_bins() { return kScanTile; }
bool scan_direct(int64_t scan_tiles) { return scan_tiles <= 16; }

cudaError_t launch_expand(const SortArgs& a, int32_t nblocks, cudaStream_t s) {
    k_expand<<<nblocks, kExpandThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_gather_quantiles(const int32_t* sorted, const int64_t* offsets, const int32_t* rank, int32_t K,
                                    int32_t F, int32_t* out, cudaStream_t s) {
    const int64_t n = (int64_t)K * F;
    const int threads = 256;
    k_gather_quantiles<<<(unsigned)((n + threads - 1) / threads), threads, 0, s>>>(sorted, offsets, rank, K, F, out);
    return cudaGetLastError();
}

int64_t hist_slice_samples() { return kHistSlice; }
int64_t expand_tile_positions() { return kExpandTile; }

}  // namespace kvdro
