// The steps either side of the filter in a seed-and-extend mapper.
//
// Before (Sec. 1, Fig. 1 steps 2-3): the read's seeds are looked up in a
// table of reference locations; each location is a potential mapping, and
// the filter checks the bins that hold one (Sec. 3.3).
//   - grim_seed_index_build: a CSR table of the start positions of every
//     k-mer of the reference (count, prefix sum, fill; the order of the
//     positions of one k-mer is not specified);
//   - grim_seed_candidates: non-overlapping k-mer seeds per read; every
//     location p of the seed at offset o votes for the bin whose core holds
//     max(0, p - o); distinct bins are kept, the `cap` most voted when
//     there are more (equal votes: the lower bin), ascending.  Per batch of
//     reads: hits per read (warp per read) -> prefix sum -> seed_fast_kernel:
//     a group of threads per read fetches its seeds' locations, sorts the
//     voted bins in shared memory and keeps the distinct ones; the few reads
//     it cannot take (too many votes, votes piled into one region, more bins
//     than the cap) are listed and go through votes in scratch -> one CTA per
//     read that sorts them (bucket or stable LSD radix sort), finds the runs,
//     applies the cap (binary search on the vote threshold) and compacts ->
//     prefix sum of the kept counts -> copy into the CSR output.
// After (Sec. 3.3, Fig. 4 steps 2-3): the Seed Location Checker turns the
// filter's bitmask into the list of passing locations and the reference
// segments the aligner receives.
//   - grim_locate: tile counts of passing bytes -> prefix sum -> ordered
//     write of (read, bin, span); optional segment bases copied out of the
//     2-bit reference (one warp per segment).
#include <type_traits>

#include "grim_internal.cuh"

struct grim_seed_index {
    int64_t len;
    int k;
    int device;
    uint32_t* offsets;    // device, 4^k + 1 entries
    uint32_t* positions;  // device, len - k + 1 entries
    // the most candidates per read (x 16, rounded up) that a call has
    // produced: a sizing hint for callers that allocate per batch
    mutable std::atomic<int64_t> per_read_x16{0};
};

namespace grim {

int64_t seed_candidates_hint(const grim_seed_index* idx, int64_t n_reads) {
    return idx->per_read_x16.load() * n_reads / 16;
}

namespace {

// ------------------------------------------------------------ prefix sums

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int64_t kScanTile = (int64_t)kScanThreads * kScanItems;

// Block-wide exclusive scan of one value per thread (all threads call it);
// *total receives the block's sum.
template <typename T>
__device__ T block_exclusive_scan(T v, T* warp_sums, T* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? warp_sums[lane] : T(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T y = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) warp_sums[lane] = w;
    }
    __syncthreads();
    const T before = warp == 0 ? T(0) : warp_sums[warp - 1];
    *total = warp_sums[nw - 1];
    __syncthreads();
    return before + x - v;
}

template <typename T>
__global__ void set_value_kernel(T* p, T v, const T* v_dev) {
    *p = v_dev ? *v_dev : v;
}

// tile sums over the same index sets scan_tiles_kernel uses
template <typename T>
__global__ void tile_sums_kernel(const T* __restrict__ in, int64_t n, T* __restrict__ sums) {
    __shared__ T ws[32];
    const int64_t t0 = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++)
        if (t0 + i < n) s += in[t0 + i];
    T total;
    block_exclusive_scan<T>(s, ws, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// one block of 1024 threads: sums[b] <- init + sum of sums[0..b), init
// read from init_dev when that is not null
template <typename T>
__global__ void scan_sums_kernel(T* __restrict__ sums, int64_t n_tiles, T init, const T* init_dev) {
    __shared__ T ws[32];
    T carry = init_dev ? *init_dev : init;
    for (int64_t b = 0; b < n_tiles; b += blockDim.x) {
        const int64_t j = b + threadIdx.x;
        const T v = j < n_tiles ? sums[j] : T(0);
        T total;
        const T ex = block_exclusive_scan<T>(v, ws, &total);
        if (j < n_tiles) sums[j] = carry + ex;
        carry += total;
    }
}

// out[i] = tile base + sum of in[tile start .. i); out[n] = the grand total.
// Each thread reads its own items before writing them, so in == out works.
template <typename T>
__global__ void scan_tiles_kernel(const T* in, T* out, int64_t n, const T* __restrict__ sums) {
    __shared__ T ws[32];
    const int64_t t0 = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T v[kScanItems];
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        v[i] = t0 + i < n ? in[t0 + i] : T(0);
        s += v[i];
    }
    T total;
    T run = sums[blockIdx.x] + block_exclusive_scan<T>(s, ws, &total);
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        if (t0 + i < n) out[t0 + i] = run;
        run += v[i];
        if (t0 + i == n - 1) out[n] = run;
    }
}

}  // namespace

// out[0..n]: out[i] = init + in[0] + ... + in[i-1]; in == out is allowed.
// init_dev (nullable) supplies init from device memory (it may be out[0]).
template <typename T>
int exclusive_scan(const T* in, T* out, int64_t n, T init, cudaStream_t s, const T* init_dev = nullptr) {
    if (n == 0) {
        set_value_kernel<T><<<grim::fault_grid(1), 1, 0, s>>>(out, init, init_dev);
        GRIM_CUDA_TRY(cudaGetLastError());
        return GRIM_OK;
    }
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    T* sums = nullptr;
    GRIM_CUDA_TRY(grim::scratch_alloc((void**)&sums, (size_t)tiles * sizeof(T), s));
    tile_sums_kernel<T><<<grim::fault_grid((unsigned)tiles), kScanThreads, 0, s>>>(in, n, sums);
    scan_sums_kernel<T><<<grim::fault_grid(1), 1024, 0, s>>>(sums, tiles, init, init_dev);
    scan_tiles_kernel<T><<<grim::fault_grid((unsigned)tiles), kScanThreads, 0, s>>>(in, out, n, sums);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(sums, s);
    if (e != cudaSuccess) {
        set_last_cuda_error(e);
        return GRIM_ECUDA;
    }
    return GRIM_OK;
}

namespace {

__device__ __forceinline__ uint32_t ref_base(const uint8_t* __restrict__ ref2bit, int64_t i) {
    return (__ldg(ref2bit + (i >> 2)) >> (2 * (i & 3))) & 3u;
}

// ------------------------------------------------------------- seed index

constexpr int kIndexChunk = 64;  // consecutive positions per thread (rolling key)

// FILL = false: counts[key]++ for every position; true: positions[cursor[key]++] = p.
template <bool FILL>
__global__ void seed_index_kernel(const uint8_t* __restrict__ ref2bit, int64_t npos, int k,
                                  uint32_t* __restrict__ table, uint32_t* __restrict__ positions) {
    const uint32_t mask = (k >= 16) ? 0xFFFFFFFFu : ((1u << (2 * k)) - 1u);
    const int64_t chunks = (npos + kIndexChunk - 1) / kIndexChunk;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p0 = c * kIndexChunk;
        const int64_t p1 = p0 + kIndexChunk < npos ? p0 + kIndexChunk : npos;
        uint32_t key = 0;
        for (int j = 0; j < k - 1; j++) key = (key << 2) | ref_base(ref2bit, p0 + j);
        for (int64_t p = p0; p < p1; p++) {
            key = ((key << 2) | ref_base(ref2bit, p + k - 1)) & mask;
            if (FILL) {
                const uint32_t slot = atomicAdd(&table[key], 1u);
                positions[slot] = (uint32_t)p;
            } else {
                atomicAdd(&table[key], 1u);
            }
        }
    }
}

// ------------------------------------------------------- seed candidates

// Key of the k bases at s (first base most significant); false if one of
// them is not a base code.
__device__ __forceinline__ bool seed_key(const uint8_t* __restrict__ s, int k, uint32_t* key) {
    uint32_t v = 0;
    bool ok = true;
    for (int j = 0; j < k; j++) {
        const uint32_t c = __ldg(s + j);
        ok &= c <= 3u;
        v = (v << 2) | (c & 3u);
    }
    *key = v;
    return ok;
}

__device__ __forceinline__ int64_t n_seeds_of(int64_t L, int k) { return L >= k ? L / k : 0; }

// hits[r] = number of reference locations of read r's seeds (warp per read)
__global__ void seed_hits_kernel(const uint32_t* __restrict__ idx_off, int k, const uint8_t* __restrict__ reads,
                                 const int64_t* __restrict__ read_offsets, int64_t n, int64_t* __restrict__ hits) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
        const int64_t ro = read_offsets[r], L = read_offsets[r + 1] - ro;
        const int64_t ns = n_seeds_of(L, k);
        int64_t h = 0;
        for (int64_t sd = lane; sd < ns; sd += 32) {
            uint32_t key;
            if (seed_key(reads + ro + sd * k, k, &key)) h += (int64_t)(idx_off[key + 1] - idx_off[key]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(kFull, h, o);
        if (lane == 0) hits[r] = h;
    }
}

// Quotient of any 32-bit n by a fixed divisor (Granlund and Montgomery,
// "Division by invariant integers using multiplication", 1994, fig. 4.1).
struct FastDiv {
    uint32_t mul;
    int sh1, sh2;
    explicit FastDiv(uint32_t d) {
        int l = 0;
        while (l < 32 && (uint64_t(1) << l) < d) l++;
        mul = (uint32_t)(((uint64_t(1) << 32) * ((uint64_t(1) << l) - d)) / d + 1);
        sh1 = l < 1 ? l : 1;
        sh2 = l > 1 ? l - 1 : 0;
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t n) const {
        const uint32_t t = __umulhi(mul, n);
        return (t + ((n - t) >> sh1)) >> sh2;
    }
};

// ---- the common case: a group of T threads per read, in shared memory
//
// The distinct bins come from a bitmap of the bin ids scaled to 32 V T bits
// (T = 128, V = 24: 98,304): a vote that finds its bit clear is its cell's first and
// takes the place the bit's rank gives; a vote that finds it set is a repeat
// of the first vote's bin, or (rarely: 1,700 votes over 98,304 cells share
// about 15) another bin of the same cell, which goes to a short list that is
// sorted by itself and merged on the way out.  Two passes over the votes and
// one over the bitmap, whatever the order the votes come in.
// Bound: issue slots and latency together (half of each SM's threads, ~52%
// issue; the per-thread cost of the bitmap pass is paid whatever the votes, so
// small groups go with few votes).  500,000 reads of 100 bases on 3.1 Gbp
// (1,700 votes a read): 14.9 -> 10.0 ms for the whole call; 500,000 of 150 on
// 100 Mbp 3.77 -> 1.15, on 1 Mbp 3.01 -> 0.83; 200,000 on 800 Mbp, cap 100,
// 3.27 -> 2.03.  What it replaced wrote every vote to memory, read it back and
// sorted it by buckets with 256 threads a read; the same buckets sorted by
// insertion here, without the trip through memory, took 17.5 ms.
constexpr int kFewSeeds = 64;     // seeds per read, unless the group is built for more (MANY)
constexpr int kStoredSeeds = 16;  // of which seed_lookup_kernel leaves the location ranges of the first
constexpr int kFastExtra = 128;   // bins beside the first of their cell
constexpr int kFastLoads = 4;     // locations in flight per thread
constexpr int kSmallSeedReads = 32;  // reads per SM of a small batch, at most
constexpr int kFastHist = 64;     // the cap's vote threshold lies below this

// T threads per read, each holding up to V votes in registers; CAP: reads may
// have more bins than the cap keeps; MANY: reads may have more than kFewSeeds
// seeds (a vote's seed is then searched for, not walked to).
template <int T, int V, bool CAP, bool MANY>
struct FastGeo {
    static_assert(V % 8 == 0 && V <= 32, "whole 16-byte groups of ranks, one bit per vote");
    static constexpr int kVotes = V * T;
    static constexpr int kWords = V * T;             // bitmap words: V per thread
    static constexpr int kSeeds = MANY ? kWords / 4 : kFewSeeds;
    static constexpr int kGroups = T == 32 ? 4 : 1;  // reads side by side in a CTA
    // CTAs an SM should hold (registers): as many as the shared memory allows
    static constexpr int kMinCtas = T == 32 ? 8 : T == 512 ? (V <= 16 ? 2 : 1) : (V <= 16 ? 1280 : 896) / T;
};

template <int T, int V, bool CAP, bool MANY>
struct alignas(16) FastSmem {
    using F = FastGeo<T, V, CAP, MANY>;
    uint32_t map[F::kWords];                // (with a cap: then every bin, in order)
    // the first vote's bin of every set cell, in order; from the back: the
    // votes that found their bit set
    uint32_t bin[F::kVotes];
    union {
        struct {  // until the votes are read
            uint32_t seed_at[F::kSeeds];    // vote i of the seed lies at seed_at + i
            uint32_t seed_end[F::kSeeds];   // votes up to and with this seed
        };
        alignas(16) uint16_t rank[F::kWords];  // set cells before each bitmap word (then every bin's votes)
    };
    uint32_t votes2[CAP ? F::kVotes / 2 : 4];  // with a cap: votes of bin[], two 16-bit counts a word
    uint32_t extra[kFastExtra];             // as found, then without repeats
    uint32_t sorted[kFastExtra];
    uint32_t extra_votes[CAP ? kFastExtra : 1];
    uint32_t hist[CAP ? kFastHist : 1];     // bins by votes (the last: and more)
    uint32_t warp_sum[32];
    uint32_t n_set, n_extra, n_sorted;
};

// The seeds of each read of the batch, 16 lanes per read: (at, end) with vote
// i < end of the seed at location at + i, as FastSmem holds them.  Done here,
// a read's group starts its loads of locations two dependent loads after its
// offsets instead of four (reads with more seeds, and those of small batches,
// look theirs up themselves).
__global__ void seed_lookup_kernel(const uint32_t* __restrict__ idx_off, int k, const uint8_t* __restrict__ reads,
                                   const int64_t* __restrict__ read_offsets, int64_t n, uint2* __restrict__ seeds) {
    const int lane = threadIdx.x & 15;
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x >> 4);
    const int64_t first = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
    const int64_t rounds = (n + groups - 1) / groups;
    for (int64_t i = 0; i < rounds; i++) {  // the same for both halves of a warp
        const int64_t r = first + i * groups;
        int64_t ns = 0, ro = 0;
        if (r < n) {
            ro = read_offsets[r];
            ns = n_seeds_of(read_offsets[r + 1] - ro, k);
        }
        uint32_t at = 0, m = 0, key;
        if (ns <= kStoredSeeds && lane < ns && seed_key(reads + ro + (int64_t)lane * k, k, &key)) {
            at = idx_off[key];
            m = idx_off[key + 1] - at;
        }
        uint32_t x = m;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, x, o, 16);
            if (lane >= o) x += y;
        }
        if (r < n) seeds[r * kStoredSeeds + lane] = make_uint2(at - (x - m), x);
    }
}

template <int T>
__device__ __forceinline__ void group_sync() {
    if constexpr (T == 32) __syncwarp();
    else __syncthreads();
}

// Exclusive prefix sum over the group's T threads; *total: the group's sum.
template <int T>
__device__ __forceinline__ uint32_t group_scan(uint32_t v, uint32_t* warp_sum, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = (threadIdx.x % T) >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if constexpr (T == 32) {
        *total = __shfl_sync(kFull, x, 31);
        return x - v;
    } else {
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        uint32_t before = 0, sum = 0;
#pragma unroll
        for (int w = 0; w < T / 32; w++) {
            const uint32_t y = warp_sum[w];
            if (w < warp) before += y;
            sum += y;
        }
        *total = sum;
        __syncthreads();  // warp_sum may be used again
        return before + x - v;
    }
}

// Read r's kept bins (ascending) to H[hit_off[r] - h0 ...], their number to
// kept[r]; false (nothing written) for a read this path cannot take.
// cell_mul: floor(2^32 cells / n_bins), so that bin * cell_mul >> 32 spreads
// the bin ids evenly and in order over the bitmap.  The whole group; ends
// with the shared memory free for another read.
template <int T, int V, bool CAP, bool MANY>
__device__ __forceinline__ bool fast_read(FastSmem<T, V, CAP, MANY>& sm, int64_t r, const uint32_t* __restrict__ idx_off,
                                          const uint32_t* __restrict__ idx_pos, int k,
                                          const uint8_t* __restrict__ reads,
                                          const int64_t* __restrict__ read_offsets, const uint2* __restrict__ seeds,
                                          const int64_t* __restrict__ hit_off, int64_t h0, FastDiv bin_div,
                                          uint32_t last_bin, uint32_t cell_mul, int cap, uint32_t* __restrict__ H,
                                          int64_t* __restrict__ kept) {
    using F = FastGeo<T, V, CAP, MANY>;
    const int t = threadIdx.x % T, lane = threadIdx.x & 31;
    const int64_t base = hit_off[r] - h0, votes = hit_off[r + 1] - hit_off[r];
    if (votes <= 0) {
        if (t == 0) kept[r] = 0;
        return true;
    }
    const int64_t ro = read_offsets[r];
    const int64_t ns = n_seeds_of(read_offsets[r + 1] - ro, k);
    if (votes > F::kVotes || ns > F::kSeeds) return false;
    const int n = (int)votes;

    // the seeds' location ranges (first warp), an empty bitmap
#pragma unroll
    for (int i = 0; i < F::kWords / 4 / T; i++)
        reinterpret_cast<uint4*>(sm.map)[i * T + t] = make_uint4(0, 0, 0, 0);
    if (seeds && ns <= kStoredSeeds) {
        if (t < kStoredSeeds) {
            const uint2 v = __ldg(seeds + r * kStoredSeeds + t);
            sm.seed_at[t] = v.x;
            sm.seed_end[t] = v.y;
        }
    } else if constexpr (MANY) {
        static_assert(F::kSeeds % T == 0, "whole rounds of the group");
        uint32_t before = 0;
        for (int g = 0; g < (int)ns; g += T) {
            uint32_t at = 0, m = 0, key, total;
            if (g + t < ns && seed_key(reads + ro + (int64_t)(g + t) * k, k, &key)) {
                at = idx_off[key];
                m = idx_off[key + 1] - at;
            }
            const uint32_t o = before + group_scan<T>(m, sm.warp_sum, &total);
            sm.seed_at[g + t] = at - o;
            sm.seed_end[g + t] = o + m;
            before += total;
        }
    } else if (t < 32) {
        uint32_t before = 0;
        for (int g = 0; g < (int)ns; g += 32) {
            uint32_t at = 0, m = 0, key;
            if (g + lane < ns && seed_key(reads + ro + (int64_t)(g + lane) * k, k, &key)) {
                at = idx_off[key];
                m = idx_off[key + 1] - at;
            }
            uint32_t x = m;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, x, o);
                if (lane >= o) x += y;
            }
            sm.seed_at[g + lane] = at - (before + x - m);
            sm.seed_end[g + lane] = before + x;
            before += __shfl_sync(kFull, x, 31);
        }
    }
    if (t == 0) sm.n_set = sm.n_extra = 0;
    group_sync<T>();

    // the votes' bins, in registers; a clear bit makes a vote its cell's first
    uint32_t bin[V];
    uint32_t is_first = 0;
    int sd = 0;
    uint32_t end = sm.seed_end[0], at = sm.seed_at[0];  // of seed sd
#pragma unroll
    for (int u0 = 0; u0 < V; u0 += kFastLoads) {
        if (u0 * T >= n) break;  // the whole group
        uint32_t off[kFastLoads];
#pragma unroll
        for (int u = 0; u < kFastLoads; u++) {
            const int i = (u0 + u) * T + t;
            if (i < n) {
                if constexpr (MANY) {
                    if ((uint32_t)i >= end) {  // the first seed that ends after i
                        int hi = (int)ns - 1;
                        sd++;
                        while (sd < hi) {
                            const int mid = (sd + hi) >> 1;
                            if ((uint32_t)i < sm.seed_end[mid]) hi = mid;
                            else sd = mid + 1;
                        }
                        at = sm.seed_at[sd];
                        end = sm.seed_end[sd];
                    }
                } else {
                    while ((uint32_t)i >= end) {  // i < n = the last seed's end
                        at = sm.seed_at[++sd];
                        end = sm.seed_end[sd];
                    }
                }
                bin[u0 + u] = __ldg(idx_pos + (at + (uint32_t)i));
                off[u] = (uint32_t)(sd * k);
            }
        }
#pragma unroll
        for (int u = 0; u < kFastLoads; u++) {
            const int i = (u0 + u) * T + t;
            if (i < n) {
                const uint32_t pos = bin[u0 + u];
                uint32_t b = bin_div(pos > off[u] ? pos - off[u] : 0u);
                b = b < last_bin ? b : last_bin;
                bin[u0 + u] = b;
                const uint32_t cell = __umulhi(b, cell_mul), m = 1u << (cell & 31);
                if (!(atomicOr(&sm.map[cell >> 5], m) & m)) is_first |= 1u << (u0 + u);
                else sm.bin[F::kVotes - 1 - atomicAdd(&sm.n_set, 1u)] = b;
            }
        }
    }
    group_sync<T>();

    // set cells before each word: thread t owns words V t .. V t + V - 1
    uint32_t n_first;
    {
        uint32_t c[V], sum = 0;
#pragma unroll
        for (int i = 0; i < V / 4; i++) {
            const uint4 w = reinterpret_cast<const uint4*>(sm.map)[V / 4 * t + i];
            c[4 * i] = __popc(w.x);
            c[4 * i + 1] = __popc(w.y);
            c[4 * i + 2] = __popc(w.z);
            c[4 * i + 3] = __popc(w.w);
        }
#pragma unroll
        for (int i = 0; i < V; i++) sum += c[i];
        uint32_t o = group_scan<T>(sum, sm.warp_sum, &n_first);
        uint4* dst = reinterpret_cast<uint4*>(sm.rank) + V / 8 * t;
#pragma unroll
        for (int g = 0; g < V / 8; g++) {
            uint32_t pk[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                pk[i] = o | ((o + c[8 * g + 2 * i]) << 16);
                o += c[8 * g + 2 * i] + c[8 * g + 2 * i + 1];
            }
            dst[g] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
    }
    group_sync<T>();
    auto place = [&](uint32_t cell) {
        return (uint32_t)sm.rank[cell >> 5] + __popc(sm.map[cell >> 5] & ((1u << (cell & 31)) - 1u));
    };
#pragma unroll
    for (int u = 0; u < V; u++) {
        if (u * T >= n) break;
        if ((is_first >> u) & 1u) sm.bin[place(__umulhi(bin[u], cell_mul))] = bin[u];
    }
    group_sync<T>();
    for (uint32_t i = t; i < sm.n_set; i += T) {
        const uint32_t b = sm.bin[F::kVotes - 1 - i];
        if (sm.bin[place(__umulhi(b, cell_mul))] != b) {
            const uint32_t e = atomicAdd(&sm.n_extra, 1u);
            if (e < kFastExtra) sm.extra[e] = b;
        }
    }
    group_sync<T>();
    const int n_extra = (int)sm.n_extra;
    if (n_extra > kFastExtra) return false;
    int n_sorted = 0;
    if (n_extra > 0) {  // sort the extras, without repeats
        constexpr uint32_t kNone = 0xFFFFFFFFu;  // no bin id
        constexpr int kPer = (kFastExtra + T - 1) / T;
        uint32_t x[kPer];
        if (t == 0) sm.n_sorted = 0;
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const int e = q * T + t;
            x[q] = e < n_extra ? sm.extra[e] : kNone;
            bool repeat = false;
            if (e < n_extra)
                for (int j = 0; j < e; j++) repeat |= sm.extra[j] == x[q];
            if (repeat) x[q] = kNone;
        }
        group_sync<T>();
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const int e = q * T + t;
            if (e < n_extra) {
                sm.extra[e] = x[q];
                if (x[q] != kNone) atomicAdd(&sm.n_sorted, 1u);
            }
        }
        group_sync<T>();
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            if (x[q] != kNone) {
                int rank = 0;
                for (int j = 0; j < n_extra; j++) rank += sm.extra[j] < x[q];
                sm.sorted[rank] = x[q];
            }
        }
        group_sync<T>();
        n_sorted = (int)sm.n_sorted;
    }
    const uint32_t total = n_first + (uint32_t)n_sorted;
    uint32_t* out = H + base;
    auto extras_below = [&](uint32_t b) {
        int lo = 0, hi = n_sorted;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (sm.sorted[mid] < b) lo = mid + 1;
            else hi = mid;
        }
        return lo;
    };
    if (CAP && total > (uint32_t)cap) {
        // the cap: the votes of every bin, the threshold v that leaves at
        // least `cap` bins, then all bins above it and the first ones at it
        for (int i = t; i < F::kVotes / 8; i += T)
            reinterpret_cast<uint4*>(sm.votes2)[i] = make_uint4(0, 0, 0, 0);
        for (int e = t; e < kFastExtra; e += T) sm.extra_votes[e] = 0;
        for (int e = t; e < kFastHist; e += T) sm.hist[e] = 0;
        group_sync<T>();
#pragma unroll
        for (int u = 0; u < V; u++) {
            if (u * T >= n) break;
            if (u * T + t < n) {
                const uint32_t p = place(__umulhi(bin[u], cell_mul));
                if (sm.bin[p] == bin[u]) atomicAdd(&sm.votes2[p >> 1], 1u << (16 * (p & 1)));
                else atomicAdd(&sm.extra_votes[extras_below(bin[u])], 1u);
            }
        }
        group_sync<T>();
        auto votes_of = [&](uint32_t j) { return (sm.votes2[j >> 1] >> (16 * (j & 1))) & 0xFFFFu; };
        uint32_t ones = 0;  // most bins: counted apart, without atomics on one word
        for (uint32_t j = t; j < n_first; j += T) {
            const uint32_t v = votes_of(j);
            if (v == 1) ones++;
            else atomicAdd(&sm.hist[v < kFastHist - 1 ? v : kFastHist - 1], 1u);
        }
        constexpr int kPerE = (kFastExtra + T - 1) / T;
        uint32_t e_bin[kPerE], e_votes[kPerE], e_at[kPerE];
#pragma unroll
        for (int q = 0; q < kPerE; q++) {
            const int e = q * T + t;
            if (e < n_sorted) {
                e_bin[q] = sm.sorted[e];
                e_votes[q] = sm.extra_votes[e];
                const uint32_t p = place(__umulhi(e_bin[q], cell_mul));
                e_at[q] = p + (sm.bin[p] < e_bin[q]) + e;
                atomicAdd(&sm.hist[e_votes[q] < kFastHist - 1 ? e_votes[q] : kFastHist - 1], 1u);
            }
        }
        ones = __reduce_add_sync(kFull, ones);
        if (lane == 0 && ones) atomicAdd(&sm.hist[1], ones);
        group_sync<T>();  // the bitmap and the ranks are free
        const uint32_t h0v = sm.hist[2 * lane], h1v = sm.hist[2 * lane + 1];
        uint32_t ge = h0v + h1v;  // bins of at least 2 lane votes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kFull, ge, o);
            if (lane + o < 32) ge += y;
        }
        const uint32_t c32 = (uint32_t)cap;
        const uint32_t v_lane = ge - h0v >= c32 ? 2 * lane + 1 : ge >= c32 ? 2 * lane : 0;
        const uint32_t v_star = __reduce_max_sync(kFull, v_lane);
        if (v_star == kFastHist - 1) return false;
        // bins above the threshold: ge at v_star + 1
        const uint32_t above_even = __shfl_sync(kFull, ge, ((v_star + 1) >> 1) & 31);
        const uint32_t above_odd = __shfl_sync(kFull, ge - h0v, ((v_star + 1) >> 1) & 31);
        const uint32_t need = c32 - ((v_star + 1) & 1 ? above_odd : above_even);
        for (uint32_t j = t; j < n_first; j += T) {
            const uint32_t b = sm.bin[j], to = j + extras_below(b);
            sm.map[to] = b;
            sm.rank[to] = (uint16_t)votes_of(j);
        }
#pragma unroll
        for (int q = 0; q < kPerE; q++)
            if (q * T + t < n_sorted) {
                sm.map[e_at[q]] = e_bin[q];
                sm.rank[e_at[q]] = (uint16_t)e_votes[q];
            }
        group_sync<T>();
        uint32_t n_gt = 0, n_eq = 0;  // before this chunk of 4 T bins
        for (uint32_t c0 = 0; c0 < total; c0 += 4 * T) {
            uint32_t gt = 0, eq = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const uint32_t j = c0 + 4 * t + q;
                const uint32_t v = j < total ? sm.rank[j] : 0u;
                gt |= (uint32_t)(v > v_star) << q;
                eq |= (uint32_t)(v == v_star) << q;  // v_star >= 1
            }
            uint32_t both;
            const uint32_t o =
                group_scan<T>((uint32_t)__popc(gt) | ((uint32_t)__popc(eq) << 16), sm.warp_sum, &both);
            uint32_t g = n_gt + (o & 0xFFFFu), q_eq = n_eq + (o >> 16);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if ((gt >> q) & 1u) {
                    out[g + (q_eq < need ? q_eq : need)] = sm.map[c0 + 4 * t + q];
                    g++;
                } else if ((eq >> q) & 1u) {
                    if (q_eq < need) out[g + q_eq] = sm.map[c0 + 4 * t + q];
                    q_eq++;
                }
            }
            n_gt += both & 0xFFFFu;
            n_eq += both >> 16;
        }
        if (t == 0) kept[r] = cap;
        return true;
    }

    // extra e goes in before first vote number cut_e (its bin's rank among
    // them): a warp's 32 consecutive first votes are mostly between two cuts
    constexpr int kPerCut = kFastExtra / 32;
    uint32_t cut[kPerCut];  // of extras 32 q + lane, in every warp
    const int cuts = (n_sorted + 31) >> 5;
#pragma unroll
    for (int q = 0; q < kPerCut; q++) {
        cut[q] = 0xFFFFFFFFu;
        const int e = 32 * q + lane;
        if (q < cuts && e < n_sorted) {
            const uint32_t b = sm.sorted[e];
            const uint32_t p = place(__umulhi(b, cell_mul));  // its cell's first vote
            cut[q] = p + (sm.bin[p] < b);
            if (t < 32) out[cut[q] + e] = b;
        }
    }
    for (uint32_t j0 = t - lane; j0 < n_first; j0 += T) {
        const uint32_t j = j0 + lane;
        uint32_t shift = 0;
        bool split = false;
#pragma unroll
        for (int q = 0; q < kPerCut; q++)
            if (q < cuts) {
                shift += __popc(__ballot_sync(kFull, cut[q] <= j0));
                split |= __ballot_sync(kFull, cut[q] > j0 && cut[q] <= j0 + 31) != 0;
            }
        if (j < n_first) {
            const uint32_t b = sm.bin[j];
            out[j + (split ? (uint32_t)extras_below(b) : shift)] = b;
        }
    }
    if (t == 0) kept[r] = total;
    return true;
}

// Every read of the batch (list == null) or the listed ones, a group of T
// threads each; those that fast_read does not take are appended to
// slow[0 .. *n_slow).
template <int T, int V, bool CAP, bool MANY>
__global__ void __launch_bounds__(T * FastGeo<T, V, CAP, MANY>::kGroups, FastGeo<T, V, CAP, MANY>::kMinCtas)
seed_fast_kernel(const uint32_t* __restrict__ idx_off, const uint32_t* __restrict__ idx_pos, int k,
                 const uint8_t* __restrict__ reads, const int64_t* __restrict__ read_offsets,
                 const uint2* __restrict__ seeds, int64_t n_reads, const uint32_t* __restrict__ list,
                 const uint32_t* __restrict__ n_list, const int64_t* __restrict__ hit_off, int64_t h0,
                 FastDiv bin_div, uint32_t last_bin,
                 uint32_t cell_mul, int cap, uint32_t* __restrict__ H, int64_t* __restrict__ kept,
                 uint32_t* __restrict__ slow, uint32_t* __restrict__ n_slow) {
    using F = FastGeo<T, V, CAP, MANY>;
    extern __shared__ __align__(16) uint8_t fast_smem_raw[];
    const int group = threadIdx.x / T;
    FastSmem<T, V, CAP, MANY>& sm = reinterpret_cast<FastSmem<T, V, CAP, MANY>*>(fast_smem_raw)[group];
    const int64_t n = list ? (int64_t)*n_list : n_reads;
    for (int64_t i = (int64_t)blockIdx.x * F::kGroups + group; i < n; i += (int64_t)gridDim.x * F::kGroups) {
        const int64_t r = list ? (int64_t)list[i] : i;
        const bool taken = fast_read<T, V, CAP, MANY>(sm, r, idx_off, idx_pos, k, reads, read_offsets, seeds, hit_off, h0,
                                        bin_div, last_bin, cell_mul, cap, H, kept);
        if (!taken && threadIdx.x % T == 0) slow[atomicAdd(n_slow, 1u)] = (uint32_t)r;
        group_sync<T>();
    }
}

// The votes of the listed reads list[0 .. *n_list) of the batch: read r's
// bins at H[hit_off[r] - h0 ...].  A short list is of reads with thousands of
// locations per seed: one CTA per read, its warps taking the seeds in turn.  A
// long one (reads of thousands of seeds of few locations) gives each read as
// many of its warps as there are to go round.
__global__ void seed_expand_kernel(const uint32_t* __restrict__ idx_off, const uint32_t* __restrict__ idx_pos, int k,
                                   const uint8_t* __restrict__ reads, const int64_t* __restrict__ read_offsets,
                                   const uint32_t* __restrict__ list, const uint32_t* __restrict__ n_list,
                                   const int64_t* __restrict__ hit_off, int64_t h0, uint32_t bin_len,
                                   uint32_t last_bin, uint32_t* __restrict__ H) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int64_t n = *n_list;
    int team = warps;  // warps per read: 1, 2, 4 or 8
    while (team > 1 && n * team > (int64_t)gridDim.x * warps) team >>= 1;
    const int64_t stride = (int64_t)gridDim.x * warps / team;
    for (int64_t i = ((int64_t)blockIdx.x * warps + warp) / team; i < n; i += stride) {
        const int64_t r = list[i];
        const int64_t ro = read_offsets[r], L = read_offsets[r + 1] - ro;
        const int64_t ns = n_seeds_of(L, k);
        int64_t w = hit_off[r] - h0;  // first vote of this group of 32 seeds
        for (int64_t g = 0; g < ns; g += 32) {
            // lane sd of every warp looks up seed g + sd
            uint32_t a = 0, m = 0, key;
            if (g + lane < ns && seed_key(reads + ro + (g + lane) * k, k, &key)) {
                a = idx_off[key];
                m = idx_off[key + 1] - a;
            }
            int64_t x = m;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(kFull, x, o);
                if (lane >= o) x += y;
            }
            const int cnt = ns - g < 32 ? (int)(ns - g) : 32;
            for (int sd = warp % team; sd < cnt; sd += team) {
                const uint32_t sa = __shfl_sync(kFull, a, sd), sm = __shfl_sync(kFull, m, sd);
                const int64_t to = w + __shfl_sync(kFull, x, sd) - sm;
                const uint32_t o = (uint32_t)((g + sd) * k);
                for (uint32_t j = lane; j < sm; j += 32) {
                    const uint32_t p = __ldg(idx_pos + sa + j);
                    const uint32_t start = p > o ? p - o : 0u;
                    const uint32_t bin = start / bin_len;
                    H[to + j] = bin < last_bin ? bin : last_bin;
                }
            }
            w += __shfl_sync(kFull, x, 31);
        }
    }
}

constexpr int kDedupThreads = 256;
constexpr int kDedupSmem = 4096;  // votes sorted in shared memory up to this many
constexpr int kDedupItems = 8;    // consecutive entries per thread in the run and cap passes
constexpr int64_t kDedupChunk = (int64_t)kDedupThreads * kDedupItems;
constexpr int kRadixBits = 4;
constexpr int kRadixBuckets = 1 << kRadixBits;
constexpr int kDedupPadded = kDedupSmem + kDedupSmem / 32;
constexpr int kCountWords = kRadixBuckets * kDedupThreads + kRadixBuckets * kDedupThreads / 16;
constexpr size_t kDedupSmemBytes = (2 * (size_t)kDedupPadded + (size_t)kCountWords) * 4;

// Counter (bucket d, thread t) lives at word l + l / 16 for l = d * 256 + t:
// a thread's column (fixed t) and the scan's 16 consecutive counters of a
// thread (l = 16 t' + k, at word 17 t' + k) both spread over the banks.
__device__ __forceinline__ int cnt_at(int l) { return l + (l >> 4); }

// Shared-memory key arrays get one pad word per 32 so that threads reading
// consecutive blocks of keys do not collide on a bank.
template <bool SMEM, typename I>
__device__ __forceinline__ I rx_at(I i) {
    return SMEM ? i + (i >> 5) : i;
}

// Stable ascending LSD radix sort of A[0..n) on `passes` (even) digits of
// kRadixBits, with B as the second buffer; the result ends in A.  Thread t
// owns the contiguous keys [t * ipt, (t + 1) * ipt) and column t of the
// bucket-major counters, so counting and scattering need no atomics and
// keep equal digits in their original order.  I: index type (32-bit for
// the shared-memory case).
template <bool SMEM, typename I>
__device__ __forceinline__ void radix_sort(uint32_t* A, uint32_t* B, I n, int passes, uint32_t* cnt, uint32_t* ws) {
    const int t = threadIdx.x;
    const I ipt = (n + kDedupThreads - 1) / kDedupThreads;
    const I i0 = (I)t * ipt < n ? (I)t * ipt : n;
    const I i1 = i0 + ipt < n ? i0 + ipt : n;
    for (int ps = 0; ps < passes; ps++) {
        const int shift = ps * kRadixBits;
        uint32_t* src = (ps & 1) ? B : A;
        uint32_t* dst = (ps & 1) ? A : B;
#pragma unroll
        for (int b = 0; b < kRadixBuckets; b++) cnt[cnt_at(b * kDedupThreads + t)] = 0;
        for (I i = i0; i < i1; i++)
            cnt[cnt_at((int)((src[rx_at<SMEM>(i)] >> shift) & (kRadixBuckets - 1)) * kDedupThreads + t)]++;
        __syncthreads();
        // exclusive scan of the counters in bucket-major order: thread t owns
        // counters 16 t .. 16 t + 15 of that order (words 17 t .. 17 t + 15)
        uint32_t* mine = cnt + 17 * t;
        uint32_t v[kRadixBuckets];
        uint32_t sum = 0;
#pragma unroll
        for (int k = 0; k < kRadixBuckets; k++) {
            v[k] = mine[k];
            sum += v[k];
        }
        uint32_t tot;
        uint32_t run = block_exclusive_scan<uint32_t>(sum, ws, &tot);
#pragma unroll
        for (int k = 0; k < kRadixBuckets; k++) {
            mine[k] = run;
            run += v[k];
        }
        __syncthreads();
        for (I i = i0; i < i1; i++) {
            const uint32_t key = src[rx_at<SMEM>(i)];
            const uint32_t pos = cnt[cnt_at((int)((key >> shift) & (kRadixBuckets - 1)) * kDedupThreads + t)]++;
            dst[rx_at<SMEM>((I)pos)] = key;
        }
        __syncthreads();
    }
}

constexpr int kBucketBits = 10;  // the shared-memory sort's buckets: the keys' top 10 bits
constexpr int kBuckets = 1 << kBucketBits;
constexpr int kMaxBucket = 256;  // a fuller bucket hands the votes to the radix sort

// Ascending sort of the shared-memory keys A[0..n) (padded layout), all
// below 2^key_bits, into A, with B as the second buffer: the keys go to
// kBuckets buckets by their top bits (one counting pass, one scatter with
// shared atomics), then every key takes its final place in its bucket by
// counting the bucket's keys below it, ties broken by position.  The order
// of equal keys is immaterial here (only the sorted values and their run
// lengths are used).  Returns false, with A unchanged, when a bucket holds
// more than kMaxBucket keys.  cnt: 2 * kBuckets words.
__device__ bool bucket_sort_smem(uint32_t* A, uint32_t* B, int n, int key_bits, uint32_t* cnt, uint32_t* ws32) {
    constexpr int kPer = kBuckets / kDedupThreads;  // buckets per thread
    const int t = threadIdx.x;
    const int shift = key_bits > kBucketBits ? key_bits - kBucketBits : 0;
    uint32_t* start = cnt;              // first slot of each bucket
    uint32_t* cursor = cnt + kBuckets;  // counts, then scatter cursors, then bucket ends
    for (int b = t; b < kBuckets; b += kDedupThreads) cursor[b] = 0;
    __syncthreads();
    for (int i = t; i < n; i += kDedupThreads) atomicAdd(&cursor[A[rx_at<true>(i)] >> shift], 1u);
    __syncthreads();
    uint32_t c[kPer], sum = 0, mx = 0;
#pragma unroll
    for (int k = 0; k < kPer; k++) {
        c[k] = cursor[kPer * t + k];
        sum += c[k];
        mx = c[k] > mx ? c[k] : mx;
    }
    uint32_t tot;
    uint32_t run = block_exclusive_scan<uint32_t>(sum, ws32, &tot);
    if (__syncthreads_or(mx > (uint32_t)kMaxBucket)) return false;
#pragma unroll
    for (int k = 0; k < kPer; k++) {
        start[kPer * t + k] = run;
        cursor[kPer * t + k] = run;
        run += c[k];
    }
    __syncthreads();
    for (int i = t; i < n; i += kDedupThreads) {
        const uint32_t key = A[rx_at<true>(i)];
        B[rx_at<true>((int)atomicAdd(&cursor[key >> shift], 1u))] = key;
    }
    __syncthreads();
    for (int i = t; i < n; i += kDedupThreads) {
        const uint32_t key = B[rx_at<true>(i)];
        const uint32_t bk = key >> shift;
        const int s0 = (int)start[bk], s1 = (int)cursor[bk];
        int rank = s0;
        for (int j = s0; j < s1; j++) {
            const uint32_t o = B[rx_at<true>(j)];
            rank += (o < key) | ((o == key) & (j < i));
        }
        A[rx_at<true>(rank)] = key;
    }
    __syncthreads();
    return true;
}

// Votes of run j of the sorted votes: starts st[0..u), n votes in all.
template <typename I>
__device__ __forceinline__ uint32_t run_votes(const uint32_t* st, I u, I n, I j) {
    return (uint32_t)((j + 1 < u ? (I)st[j + 1] : n) - (I)st[j]);
}

// Block-wide count of runs with at least v votes.
template <typename I>
__device__ int64_t count_votes_at_least(const uint32_t* st, I u, I n, uint32_t v, int64_t* ws) {
    int64_t c = 0;
    for (I j = threadIdx.x; j < u; j += blockDim.x) c += run_votes<I>(st, u, n, j) >= v;
    int64_t total;
    block_exclusive_scan<int64_t>(c, ws, &total);
    return total;
}

// One read's votes A[0..n) (B: second buffer): sort, runs, cap, and the
// kept bins (ascending) to out[0..); returns their number.  st: scratch of
// n u32 for the run starts.  The shared-memory case (SMEM, 32-bit
// indices) reads A through the padded layout; the other case is global
// memory throughout.
template <bool SMEM, typename I>
__device__ __forceinline__ int64_t dedupe_read(uint32_t* A, uint32_t* B, I n, int cap, int passes, int bits,
                                               uint32_t* cnt,
                                               uint32_t* st, uint32_t* out, uint32_t* ws32, int64_t* ws,
                                               unsigned int* max_votes) {
    if (!SMEM || !bucket_sort_smem(A, B, (int)n, bits, cnt, ws32))
        radix_sort<SMEM, I>(A, B, n, passes, cnt, ws32);
    // run starts -> st[0..u), kDedupItems consecutive votes per thread
    I u = 0;
    for (I c0 = 0; c0 < n; c0 += (I)kDedupChunk) {
        const I i0 = c0 + (I)threadIdx.x * kDedupItems;
        uint32_t fl = 0;
#pragma unroll
        for (int k = 0; k < kDedupItems; k++) {
            const I i = i0 + k;
            if (i < n && (i == 0 || A[rx_at<SMEM>(i)] != A[rx_at<SMEM>((I)(i - 1))])) fl |= 1u << k;
        }
        uint32_t tot;
        I o = u + (I)block_exclusive_scan<uint32_t>((uint32_t)__popc(fl), ws32, &tot);
#pragma unroll
        for (int k = 0; k < kDedupItems; k++)
            if ((fl >> k) & 1u) st[o++] = (uint32_t)(i0 + k);
        u += (I)tot;
    }
    __syncthreads();
    int64_t n_keep = 0;
    if (u <= (I)cap) {
        for (I j = threadIdx.x; j < u; j += blockDim.x) out[j] = A[rx_at<SMEM>((I)st[j])];
        n_keep = u;
    } else {
        // the cap: keep votes > v_star, and the first `need` (lowest bins) at v_star
        if (threadIdx.x == 0) *max_votes = 0;
        __syncthreads();
        for (I j = threadIdx.x; j < u; j += blockDim.x) atomicMax(max_votes, run_votes<I>(st, u, n, j));
        __syncthreads();
        uint32_t lo = 1, hi = *max_votes;  // count(votes >= lo) >= cap always holds
        while (lo < hi) {
            const uint32_t mid = lo + (hi - lo + 1) / 2;
            if (count_votes_at_least<I>(st, u, n, mid, ws) >= cap) lo = mid;
            else hi = mid - 1;
        }
        const uint32_t v_star = lo;
        const int64_t need = cap - count_votes_at_least<I>(st, u, n, v_star + 1, ws);
        int64_t n_eq = 0;
        for (I c0 = 0; c0 < u; c0 += (I)kDedupChunk) {
            const I j0 = c0 + (I)threadIdx.x * kDedupItems;
            uint32_t gt = 0, eq = 0;
#pragma unroll
            for (int k = 0; k < kDedupItems; k++) {
                const I j = j0 + k;
                if (j < u) {
                    const uint32_t v = run_votes<I>(st, u, n, j);
                    if (v > v_star) gt |= 1u << k;
                    else if (v == v_star) eq |= 1u << k;
                }
            }
            int64_t tot_eq;
            int64_t e = n_eq + block_exclusive_scan<int64_t>(__popc(eq), ws, &tot_eq);
            uint32_t keep = gt;
#pragma unroll
            for (int k = 0; k < kDedupItems; k++)
                if ((eq >> k) & 1u) {
                    if (e < need) keep |= 1u << k;
                    e++;
                }
            int64_t tot_keep;
            int64_t o = n_keep + block_exclusive_scan<int64_t>(__popc(keep), ws, &tot_keep);
#pragma unroll
            for (int k = 0; k < kDedupItems; k++)
                if ((keep >> k) & 1u) out[o++] = A[rx_at<SMEM>((I)st[j0 + k])];
            n_eq += tot_eq;
            n_keep += tot_keep;
        }
    }
    return n_keep;
}

// The listed reads list[0 .. *n_list) of the batch, one CTA at a time: votes
// sorted, runs found, the cap applied and the kept bins (ascending) written to
// H[hit_off[r] - h0 ...], their number to kept[r].  Reads of up to kDedupSmem
// votes work in shared memory (bucket sort, else radix sort; run starts in the
// sort's second buffer).  Longer reads use S, scratch of 8 bytes per vote, as
// 2n u32: run starts from the front, the back half as the radix sort's second
// buffer, then their list after the starts before it is copied to H.
// `passes`: radix digits covering every bin id (even); `bits`: bits of the
// largest bin id.
__global__ void __launch_bounds__(kDedupThreads)
seed_dedupe_kernel(const uint32_t* __restrict__ read_list, const uint32_t* __restrict__ n_list,
                   const int64_t* __restrict__ hit_off, int64_t h0, int cap, int passes, int bits,
                   uint32_t* __restrict__ H,
                   unsigned long long* __restrict__ S, int64_t* __restrict__ kept) {
    extern __shared__ uint32_t dedupe_smem[];
    __shared__ int64_t ws[32];
    __shared__ uint32_t ws32[32];
    __shared__ unsigned int max_votes;
    const uint32_t n_reads = *n_list;
    for (uint32_t i_list = blockIdx.x; i_list < n_reads; i_list += gridDim.x) {
        const int64_t r = read_list[i_list];
        const int64_t base = hit_off[r] - h0, n = hit_off[r + 1] - hit_off[r];  // n > 0
        uint32_t* st = reinterpret_cast<uint32_t*>(S + base);  // 2n u32 of scratch
        int64_t n_keep;
        if (n <= kDedupSmem) {
            uint32_t* A_s = dedupe_smem;
            uint32_t* B_s = dedupe_smem + kDedupPadded;
            uint32_t* cnt = dedupe_smem + 2 * kDedupPadded;
            const int ni = (int)n;
            for (int i = threadIdx.x; i < ni; i += blockDim.x) A_s[rx_at<true>(i)] = H[base + i];
            __syncthreads();
            // the run starts go to B_s, free once A_s is sorted
            n_keep = dedupe_read<true, int>(A_s, B_s, ni, cap, passes, bits, cnt, B_s, H + base, ws32, ws,
                                            &max_votes);
        } else {
            uint32_t* cnt = dedupe_smem + 2 * kDedupPadded;
            // the list is built after the starts (st + n: the sort's buffer, free by then)
            uint32_t* list = st + n;
            n_keep = dedupe_read<false, int64_t>(H + base, st + n, n, cap, passes, bits, cnt, st, list, ws32, ws,
                                                 &max_votes);
            __syncthreads();
            for (int64_t j = threadIdx.x; j < n_keep; j += blockDim.x) H[base + j] = list[j];
        }
        if (threadIdx.x == 0) kept[r] = n_keep;
        __syncthreads();  // the shared arrays are free for the next read
    }
}

struct FastArgs {
    const grim_seed_index* idx;
    const uint8_t* reads;
    const int64_t* read_offsets;
    const uint2* seeds;
    int64_t nb;
    const int64_t* hit_off;
    int64_t h0;
    int bin_len;
    int64_t n_bins;
    int cap;
    uint32_t* H;
    int64_t* kept;
};

template <int T, int V, bool CAP, bool MANY>
cudaError_t launch_fast(const FastArgs& a, const uint32_t* list, const uint32_t* n_list, uint32_t* slow,
                        uint32_t* n_slow, cudaStream_t s) {
    using F = FastGeo<T, V, CAP, MANY>;
    constexpr size_t smem = sizeof(FastSmem<T, V, CAP, MANY>) * F::kGroups;
    static DeviceCache attr[64];  // per device
    const int dev = a.idx->device;
    if (smem > 48 * 1024 && dev >= 0 && dev < 64 && !attr[dev].load()) {
        const cudaError_t e = cudaFuncSetAttribute(seed_fast_kernel<T, V, CAP, MANY>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr[dev].store(1);
    }
    const uint64_t mul = ((uint64_t)(32 * F::kWords) << 32) / (uint64_t)a.n_bins;
    int64_t blocks = (a.nb + F::kGroups - 1) / F::kGroups;
    if (list && blocks > 4 * sm_count()) blocks = 4 * sm_count();  // few, taken in turn
    seed_fast_kernel<T, V, CAP, MANY><<<grim::fault_grid((unsigned)blocks), T * F::kGroups, smem, s>>>(
        a.idx->offsets, a.idx->positions, a.idx->k, a.reads, a.read_offsets, a.seeds, a.nb, list, n_list, a.hit_off, a.h0,
        FastDiv((uint32_t)a.bin_len), (uint32_t)(a.n_bins - 1),
        (uint32_t)(mul < 0xFFFFFFFFull ? mul : 0xFFFFFFFFull), a.cap, a.H, a.kept, slow, n_slow);
    return cudaGetLastError();
}

// A cap that no read the kernel takes can exceed needs no votes per bin.
template <int T, int V, bool MANY = false>
cudaError_t launch_seed_fast(const FastArgs& a, const uint32_t* list, const uint32_t* n_list, uint32_t* slow,
                             uint32_t* n_slow, cudaStream_t s) {
    return a.cap >= FastGeo<T, V, true, MANY>::kVotes ? launch_fast<T, V, false, MANY>(a, list, n_list, slow, n_slow, s)
                                                : launch_fast<T, V, true, MANY>(a, list, n_list, slow, n_slow, s);
}

// The reads that a first kernel left to list0 by the larger groups, by both or
// by the largest alone; what these leave: list2.  n_list: the lists' lengths.
template <bool MANY>
cudaError_t launch_larger(const FastArgs& a, bool both, uint32_t* list0, uint32_t* list1, uint32_t* list2,
                          uint32_t* n_list, cudaStream_t s) {
    if (!both) return launch_seed_fast<512, 24, MANY>(a, list0, n_list, list2, n_list + 2, s);
    const cudaError_t e = launch_seed_fast<256, 24, MANY>(a, list0, n_list, list1, n_list + 1, s);
    if (e != cudaSuccess) return e;
    return launch_seed_fast<512, 24, MANY>(a, list1, n_list + 1, list2, n_list + 2, s);
}

// cand_bins[cand_off[r] ...] <- the kept bins of read r (warp per read),
// entries at or beyond `capacity` dropped.
__global__ void seed_copy_kernel(const uint32_t* __restrict__ H, const int64_t* __restrict__ hit_off, int64_t h0,
                                 const int64_t* __restrict__ cand_off, int64_t n, uint32_t* __restrict__ cand_bins,
                                 int64_t capacity) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
        const uint32_t* src = H + (hit_off[r] - h0);
        const int64_t d = cand_off[r], m = cand_off[r + 1] - d;
        const int64_t room = capacity - d < m ? capacity - d : m;
        int64_t j = lane;
        for (; j + 7 * 32 < room; j += 8 * 32) {  // eight loads in flight per lane
            uint32_t v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) v[u] = src[j + 32 * u];
#pragma unroll
            for (int u = 0; u < 8; u++) cand_bins[d + j + 32 * u] = v[u];
        }
        for (; j < room; j += 32) cand_bins[d + j] = src[j];
    }
}

// next batch [r0, r1): the most reads after r0 whose votes fit `budget`
// (at least one read), at most max_reads.
// out = {hit_off[r0], r1, hit_off[r1], hit_off[n], bases of the batch}; also
// empties the batch's lists (n_list[0 .. 3)) and starts the first batch's
// candidate offsets.
__global__ void batch_end_kernel(const int64_t* __restrict__ hit_off, const int64_t* __restrict__ read_offsets,
                                 int64_t n, int64_t r0, int64_t budget, int64_t max_reads, int64_t* __restrict__ out,
                                 uint32_t* __restrict__ n_list, int64_t* __restrict__ cand_off) {
    n_list[0] = n_list[1] = n_list[2] = 0;
    if (r0 == 0) cand_off[0] = 0;
    const int64_t h0 = hit_off[r0];
    int64_t lo = r0 + 1, hi = (n - r0) < max_reads ? n : r0 + max_reads;
    while (lo < hi) {  // largest r1 in [r0 + 1, hi] with hit_off[r1] - h0 <= budget (or r0 + 1)
        const int64_t mid = lo + (hi - lo + 1) / 2;
        if (hit_off[mid] - h0 <= budget) lo = mid;
        else hi = mid - 1;
    }
    out[0] = h0;
    out[1] = lo;
    out[2] = hit_off[lo];
    out[3] = hit_off[n];
    out[4] = read_offsets[lo] - read_offsets[r0];
}

// ------------------------------------------------------ seed location checker

// Candidates per thread: 16 (VECS = 1) while the tiles of these fill the GPU
// once at most, else 64, four 16-byte loads in flight: both kernels are bound by
// the latency of a CTA's few dependent loads and barriers, so fewer CTAs of more
// bytes each are faster once there are enough (us a call, 1% passing, by 16 / by
// 64: 1,000 bytes 25 / 29, 3M 31 / 32, 10M 44 / 35, 200M 366 / 188).
template <int VECS>
struct LocGeo {
    static_assert(VECS == 1 || VECS == 4, "one bit per candidate of a thread");
    using Mask = typename std::conditional<VECS == 1, uint32_t, uint64_t>::type;
    static constexpr int kItems = 16 * VECS;
    static constexpr int kTile = kScanThreads * kItems;
    // A tile with more passing candidates than this is written in VECS rounds of 16
    // candidates a thread: a thread that writes its own 64 leaves a warp's stores
    // four times as far apart (200M bytes, us at once / in
    // rounds: 8% passing 449 / 430, 30% 2,757 / 1,248).
    static constexpr int kDense = VECS == 1 ? kTile : kTile / 16;
};

// Nonzero pass bytes among this thread's (bit i = byte t0 + i), by 16-byte
// loads from the 16-byte boundary at or before the first of them (`shift` bytes
// before it) where these lie among the n bytes: the masks are shifted into
// place, not the bytes.
template <int VECS>
__device__ __forceinline__ typename LocGeo<VECS>::Mask pass_mask(const uint8_t* __restrict__ pass, int64_t t0, int64_t n,
                                                                 int shift) {
    using Mask = typename LocGeo<VECS>::Mask;
    constexpr int kItems = LocGeo<VECS>::kItems;
    Mask m = 0;
    const int64_t a0 = t0 - shift;
    if (a0 >= 0 && a0 + kItems + (shift ? 16 : 0) <= n) {
        const uint4* p = reinterpret_cast<const uint4*>(pass + a0);
        uint4 v[VECS];
#pragma unroll
        for (int u = 0; u < VECS; u++) v[u] = __ldg(p + u);
        Mask above = 0;
        if (shift) above = nonzero_bytes16(__ldg(p + VECS));  // the same for the whole call
#pragma unroll
        for (int u = 0; u < VECS; u++) m |= (Mask)nonzero_bytes16(v[u]) << (16 * u);
        if (shift) {
            m = (m >> shift) | (above << (kItems - shift));
            if (VECS == 1) m &= 0xFFFFu;
        }
        return m;
    }
    for (int i = 0; i < kItems; i++)
        if (t0 + i < n && pass[t0 + i]) m |= (Mask)1 << i;
    return m;
}

template <int VECS>
__global__ void locate_count_kernel(const uint8_t* __restrict__ pass, int64_t n_cands, int shift,
                                    int64_t* __restrict__ counts) {
    __shared__ int warp_sum[kScanThreads / 32];
    const int64_t t0 = (int64_t)blockIdx.x * LocGeo<VECS>::kTile + (int64_t)threadIdx.x * LocGeo<VECS>::kItems;
    const int c = __reduce_add_sync(kFull, (unsigned)__popcll(pass_mask<VECS>(pass, t0, n_cands, shift)));
    if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t total = 0;
        for (int w = 0; w < kScanThreads / 32; w++) total += warp_sum[w];
        counts[blockIdx.x] = total;
    }
}

// Reads holding candidates c0 (lanes 0-15) and c1 (lanes 16-31): the last
// r in [0, n_reads - 1] with cand_offsets[r] <= c, by a 16-ary search per
// half-warp (about log16(n_reads) rounds of parallel loads).  Whole warp.
__device__ int64_t reads_of_half_warps(const int64_t* __restrict__ co, int64_t n_reads, int64_t c0, int64_t c1,
                                       int lane) {
    const int j = lane & 15;
    const int64_t c = lane < 16 ? c0 : c1;
    int64_t lo = 0, hi = n_reads - 1;  // the answer lies in [lo, hi]; co[0] <= c
    while (__any_sync(kFull, hi - lo > 15)) {  // then 16 lanes cover [lo, hi]
        const int64_t p = lo + 1 + (hi - lo - 1 > 0 ? (hi - lo - 1) * j / 15 : 0);  // samples in (lo, hi]
        const bool le = p <= hi && __ldg(co + p) <= c;
        const unsigned b = __ballot_sync(kFull, le);
        const unsigned half = lane < 16 ? b & 0xFFFFu : b >> 16;
        const int k = __popc(half);  // the samples at or below c are a prefix
        const int64_t p_last = __shfl_sync(kFull, p, (lane & 16) + (k > 0 ? k - 1 : 0));
        const int64_t p_next = __shfl_sync(kFull, p, (lane & 16) + (k < 16 ? k : 15));
        if (k > 0) lo = p_last;
        if (k < 16 && p_next - 1 < hi) hi = p_next - 1;
        if (hi < lo) hi = lo;  // only with decreasing (invalid) offsets
    }
    const int64_t p = lo + j;
    const unsigned b = __ballot_sync(kFull, p <= hi && __ldg(co + p) <= c);
    const int cnt = __popc(lane < 16 ? b & 0xFFFFu : b >> 16);
    return cnt > 0 ? lo + cnt - 1 : lo;
}

// read holding candidate c: the last r in [lo, hi] with cand_offsets[r] <= c
__device__ __forceinline__ int64_t read_of(const int64_t* __restrict__ co, int64_t lo, int64_t hi, int64_t c) {
    while (lo < hi) {
        const int64_t mid = lo + (hi - lo + 1) / 2;
        if (co[mid] <= c) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <int VECS>
__global__ void __launch_bounds__(kScanThreads)
locate_write_kernel(const uint8_t* __restrict__ pass, int shift, const uint32_t* __restrict__ cand_bins,
                    const int64_t* __restrict__ cand_offsets, int64_t n_reads, int64_t n_cands,
                    const int64_t* __restrict__ tile_base, int64_t len, int64_t n_bins, int bin_len, int overlap,
                    int64_t capacity, uint32_t* __restrict__ loc_read, uint32_t* __restrict__ loc_bin,
                    int64_t* __restrict__ loc_begin, int64_t* __restrict__ loc_end, uint32_t* __restrict__ status) {
    using G = LocGeo<VECS>;
    __shared__ int64_t ws[32];
    __shared__ int64_t tile_reads[2];
    const int64_t tile0 = (int64_t)blockIdx.x * G::kTile;
    const int64_t t0 = tile0 + (int64_t)threadIdx.x * G::kItems;
    typename G::Mask m = pass_mask<VECS>(pass, t0, n_cands, shift);
    uint32_t flags = 0;
    if (threadIdx.x == 0 && blockIdx.x == 0 && cand_offsets[n_reads] != n_cands) flags |= GRIM_FLAG_BAD_OFFSETS;
    int64_t total;
    int64_t base = tile_base[blockIdx.x];
    int64_t o = base + block_exclusive_scan<int64_t>(__popcll(m), ws, &total);
    if (total == 0) {  // nothing passes in this tile (block-uniform)
        if (flags) atomicOr(status, flags);
        return;
    }
    if (threadIdx.x < 32) {  // the reads of the tile's first and last candidates
        const int64_t last = (tile0 + G::kTile < n_cands ? tile0 + G::kTile : n_cands) - 1;
        const int64_t rr = reads_of_half_warps(cand_offsets, n_reads, tile0, last, threadIdx.x);
        if (threadIdx.x == 0) tile_reads[0] = rr;
        if (threadIdx.x == 16) tile_reads[1] = rr;
    }
    __syncthreads();
    const int64_t tr0 = tile_reads[0], tr1 = tile_reads[1] > tile_reads[0] ? tile_reads[1] : tile_reads[0];
    const bool dense = VECS > 1 && total > G::kDense;  // block-uniform
    __shared__ uint64_t masks[VECS > 1 ? kScanThreads : 1];
    if (dense) {
        masks[threadIdx.x] = m;
        __syncthreads();
    }
    for (int round = 0; round < (dense ? VECS : 1); round++) {
        int64_t c0 = t0;
        if (dense) {  // 16 candidates, tile0 + 16 * place on
            const int place = round * kScanThreads + threadIdx.x;
            m = (typename G::Mask)((masks[place / VECS] >> (16 * (place % VECS))) & 0xFFFFu);
            c0 = tile0 + 16 * place;
            int64_t in_round;
            const int64_t before = block_exclusive_scan<int64_t>(__popcll(m), ws, &in_round);
            o = base + before;
            base += in_round;
        }
        int64_t r = -1;
        while (m && o < capacity) {
            const int i = __ffsll((long long)m) - 1;
            m &= m - 1;
            const int64_t c = c0 + i;
            // the read: one search within the tile's reads, then forward
            if (r < 0) r = read_of(cand_offsets, tr0, tr1, c);
            while (r + 1 < n_reads && cand_offsets[r + 1] <= c) r++;
            const uint32_t b = cand_bins[c];
            int64_t begin = 0, end = 0;
            if ((int64_t)b < n_bins) {
                begin = (int64_t)b * bin_len;
                end = begin + bin_len + overlap < len ? begin + bin_len + overlap : len;
            } else {
                flags |= GRIM_FLAG_BAD_BIN;
            }
            loc_read[o] = (uint32_t)r;
            loc_bin[o] = b;
            if (loc_begin) loc_begin[o] = begin;
            if (loc_end) loc_end[o] = end;
            o++;
        }
    }
    if (flags) atomicOr(status, flags);
}

// segment rows: the span's base codes, then 4 up to the stride (warp per row)
__global__ void locate_segments_kernel(const uint8_t* __restrict__ ref2bit, const int64_t* __restrict__ n_loc,
                                       int64_t capacity, const int64_t* __restrict__ loc_begin,
                                       const int64_t* __restrict__ loc_end, uint8_t* __restrict__ seg,
                                       int64_t stride) {
    const int lane = threadIdx.x & 31;
    const int64_t rows = *n_loc < capacity ? *n_loc : capacity;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < rows; i += warps) {
        const int64_t b = loc_begin[i], e = loc_end[i];
        uint8_t* row = seg + i * stride;
        for (int64_t j = lane; j < stride; j += 32) row[j] = b + j < e ? (uint8_t)ref_base(ref2bit, b + j) : 4;
    }
}

}  // namespace
}  // namespace grim

extern "C" {

int grim_seed_index_build(const uint8_t* ref2bit, int64_t len, int k, void* stream, grim_seed_index** out) {
    if (!out) return GRIM_EINVAL;
    *out = nullptr;
    if (!ref2bit || k < 1 || k > 15 || len < k || len > (int64_t)0xFFFFFFFFll) return GRIM_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t nk = int64_t(1) << (2 * k);
    const int64_t npos = len - k + 1;
    grim_seed_index* idx = new grim_seed_index();
    idx->len = len;
    idx->k = k;
    if (cudaGetDevice(&idx->device) != cudaSuccess) {
        delete idx;
        return GRIM_ECUDA;
    }
    uint32_t* cursor = nullptr;
    cudaError_t e = grim::fault_alloc_now() ? cudaErrorMemoryAllocation
                                            : cudaMalloc((void**)&idx->offsets, (size_t)(nk + 1) * 4);
    if (e == cudaSuccess)
        e = grim::fault_alloc_now() ? cudaErrorMemoryAllocation
                                    : cudaMalloc((void**)&idx->positions, (size_t)npos * 4);
    if (e == cudaSuccess) e = grim::scratch_alloc((void**)&cursor, (size_t)nk * 4, s);
    int rc = GRIM_OK;
    if (e == cudaSuccess) e = cudaMemsetAsync(cursor, 0, (size_t)nk * 4, s);
    if (e == cudaSuccess) {
        const int blocks = grim::sm_count() * 8;
        grim::seed_index_kernel<false><<<grim::fault_grid(blocks), 256, 0, s>>>(ref2bit, npos, k, cursor, nullptr);
        e = cudaGetLastError();
        if (e == cudaSuccess) rc = grim::exclusive_scan<uint32_t>(cursor, idx->offsets, nk, 0u, s);
        if (e == cudaSuccess && rc == GRIM_OK)
            e = cudaMemcpyAsync(cursor, idx->offsets, (size_t)nk * 4, cudaMemcpyDeviceToDevice, s);
        if (e == cudaSuccess && rc == GRIM_OK) {
            grim::seed_index_kernel<true><<<grim::fault_grid(blocks), 256, 0, s>>>(
                    ref2bit, npos, k, cursor, idx->positions);
            e = cudaGetLastError();
        }
    }
    if (cursor) cudaFreeAsync(cursor, s);
    if (e != cudaSuccess || rc != GRIM_OK) {
        if (e != cudaSuccess) {
            grim::set_last_cuda_error(e);
            rc = e == cudaErrorMemoryAllocation ? GRIM_ENOMEM : GRIM_ECUDA;
        }
        cudaStreamSynchronize(s);
        cudaFree(idx->offsets);
        cudaFree(idx->positions);
        delete idx;
        return rc;
    }
    *out = idx;
    return GRIM_OK;
}

int grim_seed_index_info(const grim_seed_index* idx, int64_t* len, int* k, const uint32_t** offsets,
                         const uint32_t** positions) {
    if (!idx) return GRIM_EINVAL;
    if (len) *len = idx->len;
    if (k) *k = idx->k;
    if (offsets) *offsets = idx->offsets;
    if (positions) *positions = idx->positions;
    return GRIM_OK;
}

int grim_seed_index_free(grim_seed_index* idx) {
    if (!idx) return GRIM_OK;
    cudaDeviceSynchronize();
    cudaFree(idx->offsets);
    cudaFree(idx->positions);
    delete idx;
    return GRIM_OK;
}

int grim_seed_candidates(const grim_seed_index* idx, const uint8_t* reads, const int64_t* read_offsets,
                         int64_t n_reads, int bin_len, int64_t n_bins, int cap, uint32_t* cand_bins,
                         int64_t capacity, int64_t* cand_offsets, int64_t* n_cands, void* stream) {
    if (!idx || n_reads < 0 || bin_len < 1 || n_bins < 1 || n_bins > (int64_t)0xFFFFFFFFll || cap < 1 ||
        capacity < 0 || !cand_offsets || !n_cands || (capacity > 0 && !cand_bins))
        return GRIM_EINVAL;
    *n_cands = 0;
    if (n_reads > 0 && (!reads || !read_offsets)) return GRIM_EINVAL;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != idx->device) return GRIM_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (n_reads == 0) return grim::exclusive_scan<int64_t>(nullptr, cand_offsets, 0, 0, s);

    const int threads = 256;
    const int64_t warp_blocks = (n_reads * 32 + threads - 1) / threads;
    const unsigned blocks = (unsigned)(warp_blocks < 65535 ? warp_blocks : 65535);
    const int64_t kBudget = int64_t(1) << 28;     // votes per batch
    const int64_t kMaxReads = int64_t(1) << 20;   // reads per batch
    // the call's fixed working memory, in one piece: every allocation and its
    // release costs a short call 1-2 us
    const int64_t max_nb = n_reads < kMaxReads ? n_reads : kMaxReads;
    const int64_t small_reads = grim::kSmallSeedReads * (int64_t)grim::sm_count();
    const size_t seeds_bytes = n_reads > small_reads ? (size_t)max_nb * grim::kStoredSeeds * sizeof(uint2) : 0;
    int64_t* info = nullptr;  // batch bounds
    GRIM_CUDA_TRY(grim::scratch_alloc(
        (void**)&info, 64 + seeds_bytes + (size_t)(n_reads + 1 + max_nb) * 8 + (size_t)(3 * max_nb + 4) * 4, s));
    // location ranges of the batch's seeds
    uint2* seeds = seeds_bytes ? reinterpret_cast<uint2*>(info + 8) : nullptr;
    int64_t* hit_off = info + 8 + seeds_bytes / 8;
    int64_t* kept = hit_off + n_reads + 1;
    uint32_t* slow = reinterpret_cast<uint32_t*>(kept + max_nb);  // lists of the reads the fast path leaves
    int rc = GRIM_OK;
    grim::seed_hits_kernel<<<grim::fault_grid(blocks), threads, 0, s>>>(
            idx->offsets, idx->k, reads, read_offsets, n_reads, hit_off);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) rc = grim::exclusive_scan<int64_t>(hit_off, hit_off, n_reads, 0, s);

    // radix digits covering bin ids 0 .. n_bins - 1, rounded up to even
    int bits = 0;
    while (bits < 32 && ((n_bins - 1) >> bits) != 0) bits++;
    const int passes = 2 * ((bits + 2 * grim::kRadixBits - 1) / (2 * grim::kRadixBits));
    static grim::DeviceCache smem_set[64];
    if (dev >= 0 && dev < 64 && !smem_set[dev].load()) {
        GRIM_CUDA_TRY(cudaFuncSetAttribute(grim::seed_dedupe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)grim::kDedupSmemBytes));
        smem_set[dev].store(1);
    }
    // scratch kept across batches (freeing it would hand it back to the
    // pool at every synchronisation): votes as u32 (H) and 2 u32 per vote (S)
    uint32_t* H = nullptr;
    unsigned long long* S = nullptr;
    int64_t cap_votes = 0;
    for (int64_t r0 = 0; r0 < n_reads && e == cudaSuccess && rc == GRIM_OK;) {
        int64_t b[5];
        grim::batch_end_kernel<<<grim::fault_grid(1), 1, 0, s>>>(hit_off, read_offsets, n_reads, r0, kBudget, kMaxReads,
                                                                 info, slow, cand_offsets);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(b, info, sizeof(b), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) break;
        const int64_t h0 = b[0], r1 = b[1], votes = b[2] - b[0], nb = r1 - r0;
        if (votes > cap_votes) {
            // the first batch sizes it for the largest regular batch
            const int64_t want = votes > kBudget ? votes : (b[3] - h0 < kBudget ? b[3] - h0 : kBudget);
            if (H) cudaFreeAsync(H, s);
            if (S) cudaFreeAsync(S, s);
            H = nullptr;
            S = nullptr;
            e = grim::scratch_alloc((void**)&H, (size_t)(want > 0 ? want : 1) * 4, s);
            if (e == cudaSuccess) e = grim::scratch_alloc((void**)&S, (size_t)(want > 0 ? want : 1) * 8, s);
            if (e != cudaSuccess) break;
            cap_votes = want;
        }
        const int64_t wb = (nb * 32 + threads - 1) / threads;
        const unsigned bb = (unsigned)(wb < 65535 ? wb : 65535);
        // three lists and their lengths: reads of more votes than the batch's
        // group size takes (tried again with larger groups), and the rest
        uint32_t *n_list = slow, *list0 = slow + 4, *list1 = list0 + nb, *list2 = list1 + nb;
        // threads per read by the batch's mean votes, with room for about three
        // times it (at 1,700 votes: 256 x 16 10.0 ms a call, 128 x 24 11.1,
        // whose reads of over 3,072 votes then take the larger groups); a small
        // batch does not fill the GPU, and a larger group has its read sooner
        // (1,000 reads on 1 Gbp, 540 votes: 137 us by 64 x 24, 118 by 256 x 16)
        const int64_t mean = votes / nb;
        // a small batch is a chain of launches of a few us each: the seeds are
        // looked up by the reads' groups and what these leave goes straight to the
        // last kernels (800 reads of 2.6 Mbp: 120 -> 101 us a call; 2,500 of 20 Mbp
        // 122 -> 110; 4,000 of 400 Mbp 147 -> 131).  Only while these leave next to
        // none: the last kernels are slow (2,000 reads of 300 bases on 3.1 Gbp, 5,000
        // votes each: 1,231 us that way, 590 by the larger groups; 1,000 of 100, 1,700
        // votes each: 213 and 150).
        const bool small = nb <= small_reads && mean <= 800;
        if (!small && seeds) {
            const int64_t lookup_blocks = (nb * 16 + threads - 1) / threads;
            grim::seed_lookup_kernel<<<grim::fault_grid((unsigned)(lookup_blocks < 65535 ? lookup_blocks : 65535)),
                                       threads, 0, s>>>(idx->offsets, idx->k, reads, read_offsets + r0, nb, seeds);
            e = cudaGetLastError();
            if (e != cudaSuccess) break;
        }
        const grim::FastArgs fa{idx,     reads,  read_offsets + r0, small ? nullptr : seeds, nb, hit_off + r0, h0,
                                bin_len, n_bins, cap,               H,                       kept};
        uint32_t *left = small ? list2 : list0, *n_left = small ? n_list + 2 : n_list;
        // batches with reads of more seeds than most groups take (769 bases and more
        // at k = 12), by their mean length: the groups for many seeds cost the others
        // a search per vote (20,000 reads of 300 bases on 3.1 Gbp, 25 seeds: 2.73 ms
        // for 2.58)
        const int64_t mean_seeds = b[4] / nb / idx->k;
        const bool many = mean_seeds > grim::kFewSeeds / 2;
        if (many) {
            if (mean <= 800 && mean_seeds <= 300)
                e = grim::launch_seed_fast<64, 24, true>(fa, nullptr, nullptr, left, n_left, s);
            else
                e = grim::launch_seed_fast<256, 24, true>(fa, nullptr, nullptr, left, n_left, s);
        } else if (small && mean > 500) e = grim::launch_seed_fast<256, 16>(fa, nullptr, nullptr, left, n_left, s);
        else if (mean <= 160) e = grim::launch_seed_fast<32, 16>(fa, nullptr, nullptr, left, n_left, s);
        else if (mean <= 400) e = grim::launch_seed_fast<64, 16>(fa, nullptr, nullptr, left, n_left, s);
        else if (mean <= 800) e = grim::launch_seed_fast<64, 24>(fa, nullptr, nullptr, left, n_left, s);
        else if (mean <= 1200) e = grim::launch_seed_fast<128, 24>(fa, nullptr, nullptr, left, n_left, s);
        else e = grim::launch_seed_fast<256, 16>(fa, nullptr, nullptr, left, n_left, s);
        if (!small && e == cudaSuccess) {
            // both larger groups where the list is long enough for the smaller one to
            // pay (a launch with a few reads takes 10-18 us: 2,500 reads on 3.1 Gbp
            // 229 us by both, 204 by the largest alone; 5,000 303 and 280; 40,000 on
            // 1 Gbp 453 either way; 2,000 of 5,000 votes each 587 and 600)
            const bool both = nb > 200 * (int64_t)grim::sm_count() || mean > 2000;
            e = many ? grim::launch_larger<true>(fa, both, list0, list1, list2, n_list, s)
                     : grim::launch_larger<false>(fa, both, list0, list1, list2, n_list, s);
        }
        if (e != cudaSuccess) break;
        const unsigned few = (unsigned)(nb < 4 * grim::sm_count() ? nb : 4 * grim::sm_count());
        const int64_t all = 8 * (int64_t)grim::sm_count();  // CTAs the GPU holds
        grim::seed_expand_kernel<<<grim::fault_grid((unsigned)(nb < all ? nb : all)), threads, 0, s>>>(
                idx->offsets, idx->positions, idx->k, reads, read_offsets + r0, list2, n_list + 2, hit_off + r0, h0,
                (uint32_t)bin_len, (uint32_t)(n_bins - 1), H);
        grim::seed_dedupe_kernel<<<grim::fault_grid(few), grim::kDedupThreads, grim::kDedupSmemBytes, s>>>(
            list2, n_list + 2, hit_off + r0, h0, cap, passes, bits, H, S, kept);
        e = cudaGetLastError();
        // offsets continue from the previous batch's total in cand_offsets[r0]
        if (e == cudaSuccess) rc = grim::exclusive_scan<int64_t>(kept, cand_offsets + r0, nb, 0, s, cand_offsets + r0);
        if (e == cudaSuccess && rc == GRIM_OK) {
            grim::seed_copy_kernel<<<grim::fault_grid(bb), threads, 0, s>>>(
                    H, hit_off + r0, h0, cand_offsets + r0, nb, cand_bins, capacity);
            e = cudaGetLastError();
        }
        r0 = r1;
    }
    int64_t total = 0;
    if (e == cudaSuccess && rc == GRIM_OK)
        e = cudaMemcpyAsync(&total, cand_offsets + n_reads, 8, cudaMemcpyDeviceToHost, s);
    if (H) cudaFreeAsync(H, s);
    if (S) cudaFreeAsync(S, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFreeAsync(info, s);
    if (e != cudaSuccess) {
        grim::set_last_cuda_error(e);
        return e == cudaErrorMemoryAllocation ? GRIM_ENOMEM : GRIM_ECUDA;
    }
    if (rc != GRIM_OK) return rc;
    *n_cands = total;
    const int64_t x16 = (total * 16 + n_reads - 1) / n_reads;
    int64_t seen = idx->per_read_x16.load();
    while (x16 > seen && !idx->per_read_x16.compare_exchange_weak(seen, x16)) {
    }
    return total > capacity ? GRIM_EOVERFLOW : GRIM_OK;
}

int grim_locate(const grim_bank* bank, const uint8_t* ref2bit, const uint32_t* cand_bins,
                const int64_t* cand_offsets, int64_t n_reads, int64_t n_cands, const uint8_t* pass,
                uint32_t* loc_read, uint32_t* loc_bin, int64_t* loc_begin, int64_t* loc_end, uint8_t* segments,
                int64_t seg_stride, int64_t capacity, int64_t* n_loc, void* stream) {
    if (!bank || n_reads < 0 || n_cands < 0 || capacity < 0 || !n_loc || !cand_offsets) return GRIM_EINVAL;
    if (n_cands > 0 && (!cand_bins || !pass)) return GRIM_EINVAL;
    if (capacity > 0 && (!loc_read || !loc_bin)) return GRIM_EINVAL;
    if (segments && (seg_stride <= 0 || !ref2bit || !loc_begin || !loc_end)) return GRIM_EINVAL;
    if (n_cands > 0 && n_reads == 0) return GRIM_EINVAL;
    int rc = grim::check_device(bank);
    if (rc != GRIM_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    if (n_cands == 0) return grim::exclusive_scan<int64_t>(nullptr, n_loc, 0, 0, s);
    // tiles of 16 candidates a thread where these fill the GPU once at most
    const bool small = n_cands <= 8 * (int64_t)grim::sm_count() * grim::LocGeo<1>::kTile;
    const int64_t tile = small ? grim::LocGeo<1>::kTile : grim::LocGeo<4>::kTile;
    const int64_t tiles = (n_cands + tile - 1) / tile;
    int64_t* counts = nullptr;
    GRIM_CUDA_TRY(grim::scratch_alloc((void**)&counts, (size_t)(tiles + 1) * 8, s));
    const int shift = (int)((uintptr_t)pass & 15);
    const unsigned blocks = grim::fault_grid((unsigned)tiles);
    if (small) grim::locate_count_kernel<1><<<blocks, grim::kScanThreads, 0, s>>>(pass, n_cands, shift, counts);
    else grim::locate_count_kernel<4><<<blocks, grim::kScanThreads, 0, s>>>(pass, n_cands, shift, counts);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) rc = grim::exclusive_scan<int64_t>(counts, counts, tiles, 0, s);
    if (e == cudaSuccess && rc == GRIM_OK)
        e = cudaMemcpyAsync(n_loc, counts + tiles, 8, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess && rc == GRIM_OK) {
        auto write = small ? grim::locate_write_kernel<1> : grim::locate_write_kernel<4>;
        write<<<grim::fault_grid((unsigned)tiles), grim::kScanThreads, 0, s>>>(
            pass, shift, cand_bins, cand_offsets, n_reads, n_cands, counts, bank->len, bank->n_bins, bank->bin_len,
            bank->overlap, capacity, loc_read, loc_bin, loc_begin, loc_end, bank->status);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && rc == GRIM_OK && segments && capacity > 0) {
        grim::locate_segments_kernel<<<grim::fault_grid(grim::sm_count() * 8), 256, 0, s>>>(
                ref2bit, n_loc, capacity, loc_begin, loc_end, segments, seg_stride);
        e = cudaGetLastError();
    }
    cudaFreeAsync(counts, s);
    if (e != cudaSuccess) {
        grim::set_last_cuda_error(e);
        return GRIM_ECUDA;
    }
    return rc;
}

}  // extern "C"
