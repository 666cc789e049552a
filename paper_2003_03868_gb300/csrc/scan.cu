// Prefix sums and a deterministic FP64 sum, used by the stack builder and the
// filter compaction.
#include "common.cuh"

namespace dbg {
namespace {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kTile = kScanThreads * kScanItems;
constexpr int kScanOne = 4 * kTile;            // up to here one CTA takes the tiles one after the other

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ int64_t block_exclusive_scan(int64_t v, int64_t* warp_tot, int64_t& excl) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t t = (lane < (int)(blockDim.x >> 5)) ? warp_tot[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_tot[lane] = t;   // inclusive over warps
    }
    __syncthreads();
    int64_t before = (warp > 0) ? warp_tot[warp - 1] : 0;
    excl = before + x - v;
    int64_t total = warp_tot[(blockDim.x >> 5) - 1];
    __syncthreads();
    return total;
}

// A tile's word in the chain: its flag in the top two bits (0: nothing yet, 1: the tile's own sum, 2: the sum
// up to its end), the value below them (counts and sizes: never negative).
constexpr int kFlagShift = 62;
constexpr unsigned long long kValueMask = (1ull << kFlagShift) - 1;
constexpr int kPolls = 1 << 20;

template <class T>
struct ScanArgs {
    const T* in[kScanJobs];
    int64_t* out[kScanJobs];
    int64_t n, ntiles;
    unsigned long long* state;                 // per job: the tile counter, then a word per tile (zeroed)
};

// Sum of the tiles before `tile`, by one warp: 32 words at a time backwards until one holds a whole
// prefix.  Tiles are numbered in the order in which their CTAs start, so every word waited for is a
// running CTA's; should the polls run out all the same, the warp sums the input itself.
template <class T>
__device__ int64_t tiles_before(const T* __restrict__ in, const unsigned long long* words, int64_t tile) {
    const int lane = threadIdx.x & 31;
    int64_t sum = 0;
    for (int64_t last = tile - 1; last >= 0; last -= 32) {
        const int64_t idx = last - lane;
        unsigned long long w = 2ull << kFlagShift;
        if (idx >= 0) {
            const volatile unsigned long long* p = words + idx;
            int polls = 0;
            while (!((w = *p) >> kFlagShift) && ++polls < kPolls) {}
        }
        if (__any_sync(0xffffffffu, !(w >> kFlagShift))) {
            sum = 0;
            for (int64_t i = lane; i < tile * kTile; i += 32) sum += (int64_t)in[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            return sum;
        }
        const unsigned whole = __ballot_sync(0xffffffffu, (w >> kFlagShift) == 2ull);
        const int stop = whole ? __ffs(whole) - 1 : 31;
        int64_t v = lane <= stop ? (int64_t)(w & kValueMask) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        sum += v;
        if (whole) break;
    }
    return sum;
}

// Exclusive prefix sums, out[n] = the total, of up to kScanJobs arrays of one length (blockIdx.y), each in
// one pass over memory (single-pass scan with decoupled look-back; Merrill and Garland 2016): a CTA sums its
// tile, publishes the sum, adds up what lies before it and writes its tile.  Bound by launches at the sizes of a product's lists: scanning tiles, their sums and adding
// the offsets back took five to eight launches an array and 0.2 ms of a product on 512 waters; short
// arrays (ONE) are a single CTA's loop without a chain.
template <class T, bool ONE>
__global__ void __launch_bounds__(kScanThreads) k_scan(ScanArgs<T> A) {
    __shared__ int64_t warp_tot[32];
    __shared__ int64_t s_tile, s_before;
    const T* __restrict__ in = A.in[blockIdx.y];
    int64_t* __restrict__ out = A.out[blockIdx.y];
    unsigned long long* state = ONE ? nullptr : A.state + blockIdx.y * (A.ntiles + 1);
    int64_t before = 0, tile = 0;
    if (!ONE) {
        if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(state, 1ull);
        __syncthreads();
        tile = s_tile;
    }
    do {
        const int64_t base = tile * kTile + (int64_t)threadIdx.x * kScanItems;
        int64_t vals[kScanItems];
        int64_t local = 0;
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            vals[i] = base + i < A.n ? (int64_t)in[base + i] : 0;
            local += vals[i];
        }
        int64_t excl;
        const int64_t total = block_exclusive_scan(local, warp_tot, excl);
        if (!ONE) {
            volatile unsigned long long* word = state + 1 + tile;
            if (threadIdx.x == 0) *word = ((tile ? 1ull : 2ull) << kFlagShift) | (unsigned long long)total;
            if (tile && threadIdx.x < 32) {
                const int64_t b = tiles_before(in, state + 1, tile);
                if (threadIdx.x == 0) {
                    s_before = b;
                    *word = (2ull << kFlagShift) | (unsigned long long)(b + total);
                }
            }
            __syncthreads();
            if (tile) before = s_before;
        }
        int64_t run = before + excl;
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            if (base + i < A.n) out[base + i] = run;
            run += vals[i];
        }
        before += total;
        ++tile;
    } while (ONE && tile < A.ntiles);
    if (tile == A.ntiles && threadIdx.x == 0) out[A.n] = before;
}

template <class T>
void scan_impl(const T* const* in, int64_t* const* out, int jobs, int64_t n, cudaStream_t s) {
    if (n <= 0) {
        for (int j = 0; j < jobs; ++j) DBG_CK(cudaMemsetAsync(out[j], 0, sizeof(int64_t), s));
        return;
    }
    ScanArgs<T> a{};
    for (int j = 0; j < jobs; ++j) {
        a.in[j] = in[j];
        a.out[j] = out[j];
    }
    a.n = n;
    a.ntiles = ceil_div(n, kTile);
    if (n <= kScanOne) {
        k_scan<T, true><<<dim3(1, (unsigned)jobs), kScanThreads, 0, s>>>(a);
        DBG_LAUNCH_CK();
        return;
    }
    if (a.ntiles > 0x7fffffff) fail(DBCSR_ECAPACITY, "scan: too many elements");
    DBuf<unsigned long long> state;
    state.alloc((a.ntiles + 1) * jobs, s);
    state.zero();
    a.state = state.p;
    k_scan<T, false><<<dim3((unsigned)a.ntiles, (unsigned)jobs), kScanThreads, 0, s>>>(a);
    DBG_LAUNCH_CK();
}

constexpr int kSumThreads = 256;
constexpr int kSumBlocks = 1024;
static_assert(kSumBlocks == kDetSumPartials, "det_sum_into partial count");

// Each CTA sums a fixed contiguous chunk (thread-strided, then a fixed tree).
__global__ void k_sum_partials(const double* __restrict__ v, int64_t n, double* __restrict__ part) {
    __shared__ double sh[kSumThreads];
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = min(n, lo + chunk);
    double s = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) s += v[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = kSumThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_sum_final(const double* __restrict__ part, int np, double* __restrict__ out) {
    __shared__ double sh[kSumBlocks];
    for (int i = threadIdx.x; i < kSumBlocks; i += blockDim.x) sh[i] = (i < np) ? part[i] : 0.0;
    __syncthreads();
    for (int w = kSumBlocks / 2; w > 0; w >>= 1) {
        for (int i = threadIdx.x; i < w; i += blockDim.x) sh[i] += sh[i + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

}  // namespace

void scan_exclusive(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s) {
    scan_impl<int64_t>(&in, &out, 1, n, s);
}
void scan_exclusive(const int32_t* in, int64_t* out, int64_t n, cudaStream_t s) {
    scan_impl<int32_t>(&in, &out, 1, n, s);
}
void scan_exclusive(const int64_t* const* in, int64_t* const* out, int jobs, int64_t n, cudaStream_t s) {
    if (jobs < 1 || jobs > kScanJobs) fail(DBCSR_ECAPACITY, "scan: too many arrays");
    scan_impl<int64_t>(in, out, jobs, n, s);
}

void det_sum(const double* v, int64_t n, double* out, cudaStream_t s) {
    if (n <= 0) {
        DBG_CK(cudaMemsetAsync(out, 0, sizeof(double), s));
        return;
    }
    DBuf<double> part;
    part.alloc(kSumBlocks, s);
    k_sum_partials<<<kSumBlocks, kSumThreads, 0, s>>>(v, n, part.p);
    DBG_LAUNCH_CK();
    k_sum_final<<<1, 256, 0, s>>>(part.p, kSumBlocks, out);
    DBG_LAUNCH_CK();
}

void det_sum_into(const double* v, int64_t n, double* partials, double* out, cudaStream_t s) {
    if (n <= 0) {
        DBG_CK(cudaMemsetAsync(out, 0, sizeof(double), s));
        return;
    }
    k_sum_partials<<<kSumBlocks, kSumThreads, 0, s>>>(v, n, partials);
    DBG_LAUNCH_CK();
    k_sum_final<<<1, 256, 0, s>>>(partials, kSumBlocks, out);
    DBG_LAUNCH_CK();
}

}  // namespace dbg
