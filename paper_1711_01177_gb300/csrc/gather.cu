// Gather-form filter (Sec. 3.2 steps 1-5 for every (read, candidate bin)).
//
// The accumulation sum of read r in bin b is the number of r's token
// positions whose existence bit is set in b.  Grouping equal tokens, it is
// sum_t count_r(t) * bit_b(t): a dot product of the read's token-count
// vector with the bin's bitvector.  Writing the counts in binary,
// count_r(t) = sum_p 2^p * plane_p(t), turns it into
//     Sum(r, b) = sum_p 2^p * popcount(plane_p AND row_b),
// exact integer arithmetic over whole 32-bit words instead of one bit test
// per token.  Reads of 100-150 bases need two or three planes.
//
// One warp per read (warps claim reads; the launch at the end of the file):
//   0. the first candidate rows are requested before anything else, so
//      their latency hides behind the token work;
//   1. each lane packs 5 consecutive bases of a 160-base block (2 bits per
//      base, first base highest), a shuffle brings it the next 5, and its
//      5 tokens are shifts and masks of that 10-base window (the q-gram
//      window of Sec. 3.2 step 1);
//   2. each token is counted in a byte counter in shared memory (one
//      atomic add), and the count planes are cut out of the counters with
//      masks and shifts; for q = 6 and for reads of more than 1,024 tokens it
//      is added to the bit-sliced planes by a carry chain of atomicXor;
//   3. every lane keeps its slice of the planes in registers (reads with up
//      to three planes, two for q = 6) or reads it from shared memory (more
//      planes);
//   4. candidate rows stream through the warp as 16-byte vectors,
//      lanes_per_row lanes per row (4 lanes x 32 bytes for q=5: 8 rows per
//      warp step); each row is requested one step (q <= 5, with 4 CTAs of
//      64 registers per SM) or three steps (q = 6) before it is scored,
//      its id taken from a prefetched window of 32 candidate ids; rows are
//      ANDed with the planes and popcounted, and the lanes' shares of the
//      window's 32 rows are combined by shuffles as the steps finish
//      (steps 3-4);
//   5. every lane then holds one whole sum of the window, compares it with
//      the threshold and stores its pass byte (and sum): 32 bytes of one
//      window land together (step 5).
#include <type_traits>

#include "grim_internal.cuh"
#include "tokens.cuh"

namespace grim {

constexpr int kGatherWarps = 8;
constexpr int kPlanes = 16;  // sums and counts stay below 2^16

template <int Q>
struct GatherGeo {
    static constexpr int kRowWords = Geo<Q>::kRowWords;
    static constexpr int kRowVecs = kRowWords / 4;             // 16-byte vectors per row
    static constexpr int kVPL = kRowWords >= 32 ? 2 : 1;        // vectors per lane per row
    static constexpr int kLPB = kRowVecs / kVPL;               // lanes per row
    static constexpr int kBPS = 32 / kLPB;                     // rows per warp step
    static constexpr int kPlaneWords = kPlanes * kRowWords;    // per warp
    static_assert(kLPB >= 1 && kLPB <= 32 && 32 % kBPS == 0, "bad gather geometry");
};

template <int Q>
constexpr size_t gather_smem_bytes(int warps = kGatherWarps) {
    return 4 * (size_t)warps * GatherGeo<Q>::kPlaneWords;
}

__device__ __forceinline__ uint32_t and_popc(const uint4& a, const uint4& b) {
    return __popc(a.x & b.x) + __popc(a.y & b.y) + __popc(a.z & b.z) + __popc(a.w & b.w);
}

// Carry-save adder over words: bitwise, a + b + c = lo + 2 hi.
__device__ __forceinline__ void csa(uint32_t& hi, uint32_t& lo, uint32_t a, uint32_t b, uint32_t c) {
    const uint32_t u = a ^ b;
    hi = (a & b) | (u & c);
    lo = u ^ c;
}

// A lane's weighted count of one row slice: sum_p 2^p popcount(x AND plane_p)
// over its 8 words x (two 16-byte vectors), for reads of NP count planes.
//
// POPC runs at 16 lanes a clock and SM, a quarter of the logic rate, so
// counting every ANDed word by itself is bound by that pipe (q = 5 with two
// planes: 16 POPC = 128 cycles of a scheduler per warp step against 48 of
// logic).  Two things take POPCs out:
//  - full adders over words of equal weight (Harley-Seal): 2 three-input
//    logic ops in place of one POPC and its add;
//  - the top plane of a read is nearly empty (150 bases, q = 5: ~9 of 1,024
//    tokens occur twice).  When no two of the four words of a vector share
//    a bit in it (`kSparse`, checked once per read by sparse_plane), their
//    ANDed words are simply ORed together - one three-input op per word -
//    and counted once per vector.
// kSparse: the upper of two planes is folded that way.
// 1M reads of 150 bases, 75 candidates each, bank in L2: 1.55 -> 1.49 ms;
// 200,000 reads of 1,000 candidates 3.20 -> 2.78; q = 6, 290M checks, 18.2 ->
// 16.6 (there the bank is read from HBM, and the adders were in use before).
template <int NP, bool kSparse>
__device__ __forceinline__ uint32_t row_sum8(const uint4 (&v)[2], const uint4 (&p)[NP][2]) {
    static_assert(NP == 2 || (NP == 1 && !kSparse), "one or two planes");
    uint32_t sum = 0;
    if constexpr (kSparse) {
        const uint4(&t)[2] = p[1];
        uint32_t o0 = v[0].x & t[0].x, o1 = v[1].x & t[1].x;
        o0 |= v[0].y & t[0].y;
        o1 |= v[1].y & t[1].y;
        o0 |= v[0].z & t[0].z;
        o1 |= v[1].z & t[1].z;
        o0 |= v[0].w & t[0].w;
        o1 |= v[1].w & t[1].w;
        sum = 2 * (__popc(o0) + __popc(o1));
    }
    const uint32_t a0 = v[0].x & p[0][0].x, a1 = v[0].y & p[0][0].y, a2 = v[0].z & p[0][0].z,
                   a3 = v[0].w & p[0][0].w, a4 = v[1].x & p[0][1].x, a5 = v[1].y & p[0][1].y,
                   a6 = v[1].z & p[0][1].z, a7 = v[1].w & p[0][1].w;
    uint32_t c1, s1, c2, s2, c3, s3, d1, s4;
    csa(c1, s1, a0, a1, a2);
    csa(c2, s2, a3, a4, a5);
    csa(c3, s3, s1, s2, a6);
    csa(d1, s4, c1, c2, c3);
    sum += __popc(s3) + __popc(a7);
    if constexpr (NP == 1 || kSparse) {
        return sum + 2 * __popc(s4) + 4 * __popc(d1);
    } else {
        const uint32_t b0 = v[0].x & p[1][0].x, b1 = v[0].y & p[1][0].y, b2 = v[0].z & p[1][0].z,
                       b3 = v[0].w & p[1][0].w, b4 = v[1].x & p[1][1].x, b5 = v[1].y & p[1][1].y,
                       b6 = v[1].z & p[1][1].z, b7 = v[1].w & p[1][1].w;
        uint32_t d2, s5, d3, s6, d4, s7;  // weight 2: s4 b0..b7
        csa(d2, s5, b0, b1, b2);
        csa(d3, s6, b3, b4, b5);
        csa(d4, s7, s4, s5, s6);
        return sum + 2 * (__popc(s7) + __popc(b6) + __popc(b7)) +
               4 * (__popc(d1) + __popc(d2) + __popc(d3) + __popc(d4));
    }
}

// Whether no two words of each of the lane's vectors share a bit, over the
// whole warp (see row_sum8).  `t`: the lane's two vectors of the plane.
__device__ __forceinline__ bool sparse_plane(const uint4& t0, const uint4& t1) {
    auto shared_bits = [](const uint4& m) {
        return (m.x & m.y) | ((m.x | m.y) & m.z) | ((m.x | m.y | m.z) & m.w);
    };
    return !__any_sync(kFull, (shared_bits(t0) | shared_bits(t1)) != 0);
}

// The candidate stream of one read.  Step k scores rows k*BPS .. k*BPS+BPS-1
// (lane group g = lane / LPB takes row k*BPS + g).  Candidate ids arrive in
// windows of 32 (one per lane, the next window prefetched); rows are
// requested kAhead steps before they are scored, into kBufs rotating
// register buffers.  A past-the-end or out-of-range id fetches row 0, which
// is scored but never stored.
template <int Q, bool DEEP>
struct Stream {
    using G = GatherGeo<Q>;
    static constexpr int kWinSteps = 32 / G::kBPS;       // steps per id window
    // row buffers (a divisor of kWinSteps): two for q <= 5 with the bank in
    // L2, whose smaller register budget lets 4 CTAs share an SM; four for
    // q = 6 and for banks read from HBM (DEEP: three steps of rows in flight
    // per warp cover the longer latency)
    static constexpr int kBufs =
        (Q <= 5 && !DEEP && kWinSteps >= 2) ? 2 : (kWinSteps >= 4 ? 4 : kWinSteps);
    static constexpr int kAhead = kBufs - 1;                      // steps a row is requested early
    // q = 6: rows are also prefetched into L2 this many steps ahead (within
    // the two id windows held), which covers more of the DRAM latency than
    // the register buffers alone
    static constexpr int kPrefetch = Q >= 6 ? 8 : 0;
    static_assert(kPrefetch < kWinSteps, "a prefetched id must lie in the next window at most");
    static_assert(kWinSteps % kBufs == 0, "buffer rotation must repeat every window");
    uint32_t win_cur, win_next;  // candidate ids c = base + lane, base + 32 + lane
    uint4 r[kBufs][G::kVPL];
};

__device__ __forceinline__ uint32_t window_id(const uint32_t* __restrict__ cands, int c, int n) {
    return c < n ? __ldcs(cands + c) : 0xFFFFFFFFu;
}

// Asks the L2 for the 128-byte lines of a row that will be scored later
// (no register holds it meanwhile): lane s of the row group covers the
// lines holding its vectors when s is a multiple of 8 (8 x 16 bytes).
template <int Q>
__device__ __forceinline__ void prefetch_row(uint32_t id, const uint32_t* __restrict__ bank, uint32_t n_bins32,
                                             int s) {
    using G = GatherGeo<Q>;
    // past the read's end (or an invalid id) there is nothing to fetch; a
    // stand-in row would send every warp's requests to the same lines
    if ((s & 7) != 0 || id >= n_bins32) return;
    const uint4* row = reinterpret_cast<const uint4*>(bank) + (size_t)id * G::kRowVecs + s;
#pragma unroll
    for (int u = 0; u < G::kVPL; u++) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + u * G::kLPB));
}

template <int Q>
__device__ __forceinline__ void fetch_row(uint4 (&r)[GatherGeo<Q>::kVPL], uint32_t id,
                                          const uint32_t* __restrict__ bank, uint32_t n_bins32, int s) {
    using G = GatherGeo<Q>;
    const uint32_t b = id < n_bins32 ? id : 0u;
    const uint4* row = reinterpret_cast<const uint4*>(bank) + (size_t)b * G::kRowVecs + s;
#pragma unroll
    for (int u = 0; u < G::kVPL; u++) r[u] = __ldg(row + u * G::kLPB);
}

// Before the token work: the first two id windows and the first kAhead steps' rows.
template <int Q, bool DEEP>
__device__ __forceinline__ void stream_start(Stream<Q, DEEP>& st, const uint32_t* __restrict__ cands, int n,
                                             const uint32_t* __restrict__ bank, uint32_t n_bins32, int lane) {
    using G = GatherGeo<Q>;
    using S = Stream<Q, DEEP>;
    st.win_cur = window_id(cands, lane, n);
    st.win_next = window_id(cands, 32 + lane, n);
    const int s = lane % G::kLPB, g = lane / G::kLPB;
#pragma unroll
    for (int k = 0; k < S::kAhead; k++) {
        const int idx = k * G::kBPS + g;  // < 64: within the two windows
        const uint32_t id = __shfl_sync(kFull, idx < 32 ? st.win_cur : st.win_next, idx & 31);
        fetch_row<Q>(st.r[k], id, bank, n_bins32, s);
    }
}

// Partial sums of one id window: lane s of a row group holds, for every
// step t of the window, its share of row (t, g); the kLPB lanes of a group
// together hold the kLPB steps.  Steps are combined pairwise as they finish,
// like a binary counter: two step groups that differ in bit l of the step
// index meet across lane bit l, the lane with that bit clear keeping the
// lower group and the other the upper, each adding its partner's share.
// After the last step, lane s holds the whole sum of step s: one shuffle
// per step instead of log2(kLPB), and one row per lane to store.
template <int N>
struct StepReducer {
    static constexpr int kLevels = N >= 16 ? 4 : N >= 8 ? 3 : N >= 4 ? 2 : N >= 2 ? 1 : 0;
    static_assert((1 << kLevels) == N, "steps per window must be a power of two");
    uint32_t stk[kLevels > 0 ? kLevels : 1];
    uint32_t total = 0;
    // T: the step index (a constant once the window loop is unrolled)
    __device__ __forceinline__ void add(int T, uint32_t v, int s) {
#pragma unroll
        for (int l = 0; l < kLevels; l++) {
            if (((T >> l) & 1) == 0) {
                stk[l] = v;
                return;
            }
            const uint32_t lo = stk[l], hi = v;
            const bool upper = (s >> l) & 1;
            const uint32_t send = upper ? lo : hi;
            v = (upper ? hi : lo) + __shfl_xor_sync(kFull, send, 1 << l);
        }
        total = v;
    }
    // The same for a window run as passes of P unrolled steps: step
    // h * P + tl, tl a constant, h the pass (only the levels above log2 P
    // look at it, and only at a pass's last step).
    template <int P>
    __device__ __forceinline__ void add_split(int tl, int h, uint32_t v, int s) {
        constexpr int kPassLevels = P >= 16 ? 4 : P >= 8 ? 3 : P >= 4 ? 2 : P >= 2 ? 1 : 0;
#pragma unroll
        for (int l = 0; l < kLevels; l++) {
            const int bit = l < kPassLevels ? ((tl >> l) & 1) : ((h >> (l - kPassLevels)) & 1);
            if (bit == 0) {
                stk[l] = v;
                return;
            }
            const uint32_t lo = stk[l], hi = v;
            const bool upper = (s >> l) & 1;
            const uint32_t send = upper ? lo : hi;
            v = (upper ? hi : lo) + __shfl_xor_sync(kFull, send, 1 << l);
        }
        total = v;
    }
};

// Score the read's candidates.  NP > 0: NP planes held in registers (SPARSE:
// the top one folded, see row_sum8); NP == 0: P planes read from shared
// memory.  cands / pass / sums point at the read's first candidate.
template <int Q, int NP, bool DEEP, bool SPARSE = false>
__device__ __forceinline__ void score_read(Stream<Q, DEEP>& st, const uint4* __restrict__ planes, int P, int T,
                                           int n, const uint32_t* __restrict__ cands,
                                           const uint32_t* __restrict__ bank, uint32_t n_bins32,
                                           uint8_t* __restrict__ pass, uint16_t* __restrict__ sums, int lane,
                                           uint32_t& flags) {
    using G = GatherGeo<Q>;
    using S = Stream<Q, DEEP>;
    const int s = lane % G::kLPB, g = lane / G::kLPB;
    uint4 pl[NP > 0 ? NP : 1][G::kVPL];
    if (NP > 0) {
#pragma unroll
        for (int p = 0; p < (NP > 0 ? NP : 1); p++)
#pragma unroll
            for (int u = 0; u < G::kVPL; u++) pl[p][u] = planes[p * G::kRowVecs + s + u * G::kLPB];
    }
    static_assert(S::kWinSteps == G::kLPB, "one step of the window per lane of a row group");
    // full: all 32 rows of the window exist, so its steps are one straight piece
    // of code whose loads, logic and shuffles interleave; the read's last rows
    // test before each step.  Only for the folded planes that nearly every read
    // has (SPARSE): with a second loop for every number of planes the code no
    // longer fits the instruction cache.  Tests everywhere / straight for SPARSE /
    // straight for all: 1M reads of 75 candidates, bank in L2, 1.490 / 1.373 /
    // 1.524 ms; 200,000 of 1,000 2.62 / 2.25 / 2.26; q = 6, 290M checks, 16.6 /
    // 15.9-16.1 / 15.9; 3.1 Gbp by segment 25.2 / 23.0 / 27.5, read from HBM (100,000
    // reads) 4.12 / 3.7 / 4.13.
    auto window = [&](auto full_window, int w0) {
        constexpr bool full = decltype(full_window)::value;
        const uint32_t win_after = window_id(cands, w0 + 64 + lane, n);  // two windows ahead
        StepReducer<S::kWinSteps> red;
        // 16-step windows (q = 6) run as two passes of one unrolled 8-step
        // body: half the code of the scoring loop, for the instruction cache
        constexpr int kPass = S::kWinSteps >= 16 ? 8 : S::kWinSteps;
        static_assert(kPass % S::kBufs == 0, "register buffers must rotate within a pass");
#pragma unroll 1
        for (int h = 0; h < S::kWinSteps / kPass; h++) {
#pragma unroll
        for (int tl = 0; tl < kPass; tl++) {
            const int t = h * kPass + tl;
            const int c0 = w0 + t * G::kBPS;
            uint32_t part = 0;
            if (full || c0 < n) {  // warp-uniform
                // request the rows kAhead steps ahead (window position t + kAhead)
                {
                    const int ahead = t + S::kAhead;
                    const int idx = (ahead % S::kWinSteps) * G::kBPS + g;
                    const uint32_t src = ahead < S::kWinSteps ? st.win_cur : st.win_next;
                    const uint32_t id = __shfl_sync(kFull, src, idx);
                    fetch_row<Q>(st.r[(tl + S::kAhead) % S::kBufs], id, bank, n_bins32, s);
                }
                if constexpr (S::kPrefetch > 0) {
                    const int ahead = t + S::kPrefetch;
                    const int idx = (ahead % S::kWinSteps) * G::kBPS + g;
                    const uint32_t src = ahead < S::kWinSteps ? st.win_cur : st.win_next;
                    const uint32_t id = __shfl_sync(kFull, src, idx);
                    prefetch_row<Q>(id, bank, n_bins32, s);
                }
                // score this step's rows
                const uint4 (&v)[G::kVPL] = st.r[tl % S::kBufs];
                if constexpr (NP > 0 && NP <= 2 && G::kVPL == 2) {
                    part = row_sum8<NP, SPARSE>(v, pl);
                } else if (NP > 0) {
#pragma unroll
                    for (int p = 0; p < (NP > 0 ? NP : 1); p++) {
                        uint32_t q = 0;
#pragma unroll
                        for (int u = 0; u < G::kVPL; u++) q += and_popc(v[u], pl[p][u]);
                        part += q << p;
                    }
                } else {
                    for (int p = 0; p < P; p++) {
                        uint32_t q = 0;
#pragma unroll
                        for (int u = 0; u < G::kVPL; u++)
                            q += and_popc(v[u], planes[p * G::kRowVecs + s + u * G::kLPB]);
                        part += q << p;
                    }
                }
            }
            if constexpr (kPass == S::kWinSteps) red.add(t, part, s);
            else red.template add_split<kPass>(tl, h, part, s);
        }
        }
        // this lane's row: step s, group g
        const int j = s * G::kBPS + g;
        const int c = w0 + j;
        const uint32_t id = __shfl_sync(kFull, st.win_cur, j);
        if (full || c < n) {
            const bool in_range = id < n_bins32;
            if (!in_range) flags |= GRIM_FLAG_BAD_BIN;
            const uint32_t sum = in_range ? red.total : 0u;
            __stcs(pass + c, (uint8_t)((in_range && (int)sum >= T) ? 1 : 0));
            if (sums) sums[c] = (uint16_t)sum;
        }
        st.win_cur = st.win_next;
        st.win_next = win_after;
    };
    int w = 0;
    if constexpr (SPARSE && NP == 2)
        for (; w + 32 <= n; w += 32) window(std::true_type{}, w);
    for (; w < n; w += 32) window(std::false_type{}, w);
}

// Outputs of a read whose sum is 0 for every candidate (no tokens, or a
// read rejected for bad data: then nothing passes).
__device__ __forceinline__ void write_constant(int64_t co, int64_t ce, const uint32_t* __restrict__ cand_bins,
                                               int64_t n_bins, bool pass0, uint8_t* __restrict__ pass,
                                               uint16_t* __restrict__ sums, int lane, uint32_t& flags) {
    for (int64_t c = co + lane; c < ce; c += 32) {
        const bool in_range = (int64_t)__ldg(cand_bins + c) < n_bins;
        if (!in_range) flags |= GRIM_FLAG_BAD_BIN;
        pass[c] = (in_range && pass0) ? 1 : 0;
        if (sums) sums[c] = 0;
    }
}

// Reads of up to 1,024 token positions (q <= 5) count their tokens in bytes: one
// shared atomic add per token, no carries.  The counters sit in the upper
// half of the warp's plane area (planes 8-15, which such reads never use)
// in a transposed order: the counter of token t is byte (t / 8) % 4 of
// counter word k = t % 8 of group w = t / 32, and word k of group w lies at
// 16-byte vector (k / 4) * RW + w, slot k % 4.  Bit 8 b + k of plane word w
// then is bit p of byte b of counter word k, so a plane word is eight
// masked shifts of the group's counter words, with no bit shuffling.
template <int Q>
__device__ __forceinline__ uint32_t counter_word(uint32_t tok) {
    constexpr uint32_t RW = GatherGeo<Q>::kRowWords;
    return 8 * RW + (tok & 4u) * RW + ((tok >> 5) << 2) + (tok & 3u);
}

// Count planes 0 .. used-1 from the byte counters of the warp's reads, which
// are zeroed on the way; returns used (the bit length of the largest count).
// Whole warp, after a __syncwarp that follows the counting.
template <int Q>
__device__ __forceinline__ int planes_from_counters(uint32_t* __restrict__ planes, int lane) {
    constexpr int RW = GatherGeo<Q>::kRowWords;
    uint4* cnt = reinterpret_cast<uint4*>(planes + 8 * RW);
    uint32_t any = 0;  // OR of every count: its bit length is the largest count's
    for (int w = lane; w < RW; w += 32) {
        const uint4 a = cnt[w], b = cnt[RW + w];
        any |= a.x | a.y | a.z | a.w | b.x | b.y | b.z | b.w;
    }
    any |= any >> 16;
    any |= any >> 8;
    const int used = 32 - __clz((int)__reduce_or_sync(kFull, any & 0xFFu));
    for (int w = lane; w < RW; w += 32) {
        const uint4 a = cnt[w], b = cnt[RW + w];
        cnt[w] = make_uint4(0u, 0u, 0u, 0u);
        cnt[RW + w] = make_uint4(0u, 0u, 0u, 0u);
        const uint32_t c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int p = 0; p < 8; p++) {
            if (p >= used) break;  // warp-uniform
            uint32_t u = 0;
#pragma unroll
            for (int k = 0; k < 8; k++) u |= ((c[k] >> p) & 0x01010101u) << k;
            planes[p * RW + w] = u;
        }
    }
    return used;
}

// First word of a warp's plane area that must be zero between reads: all but
// four planes for q <= 5 (the byte counters, and planes few reads have; the
// lowest are written whole from the counters, or zeroed before a carry chain),
// all of it for q = 6 (planes only ever built by carries).
template <int Q>
constexpr int kCleanFrom = Q <= 5 ? 4 * GatherGeo<Q>::kRowWords : 0;

// Shared-memory set-up of a gather warp.
template <int Q>
__device__ __forceinline__ void gather_warp_setup(uint32_t* planes, int lane) {
    for (int i = kCleanFrom<Q> + lane; i < GatherGeo<Q>::kPlaneWords; i += 32) planes[i] = 0;
    __syncwarp();
}

// Reads of up to this many tokens are counted in bytes (q <= 5), whose sum
// tells whether one ran over (137,000 reads of 270-300 bases with few
// candidates: 164 us by carry chains, 146 so).
constexpr int kCountedTokens = 1024;

// Steps 1-2: the count planes of a read of n_tok token positions; returns how
// many there are.  Whole warp; bad_base collects codes > 3.
template <int Q>
__device__ __forceinline__ int build_planes(const uint8_t* __restrict__ rd, int L, int n_tok,
                                            uint32_t* __restrict__ planes, int lane, uint32_t& bad_base) {
    constexpr int RW = GatherGeo<Q>::kRowWords;
    // byte counters, then the planes from them (q <= 5); for q = 6 the 4096
    // counters cost more to cut into planes than the carries they save
    if (Q <= 5 && n_tok <= kCountedTokens) {
        for_each_token5<Q>(rd, L, lane, bad_base,
                           [&](uint32_t tok) { atomicAdd(&planes[counter_word<Q>(tok)], 1u << (tok & 0x18u)); });
        __syncwarp();
        bool fits = n_tok <= 255;
        if (!fits) {  // a byte that ran over took 255 or 256 from the bytes' sum
            uint32_t sum = 0;
            for (int i = 8 * RW + lane; i < 16 * RW; i += 32) sum = __dp4a(planes[i], 0x01010101u, sum);
            fits = __reduce_add_sync(kFull, sum) == (uint32_t)n_tok;
        }
        if (fits) return planes_from_counters<Q>(planes, lane);
        for (int i = 8 * RW + lane; i < 16 * RW; i += 32) planes[i] = 0;
    }
    // q = 6, longer reads and a token of more than 255 times: a carry chain of
    // atomicXor per token
    for (int i = lane; i < kCleanFrom<Q>; i += 32) planes[i] = 0;
    __syncwarp();
    int top = -1;  // highest plane this lane set
    for_each_token5<Q>(rd, L, lane, bad_base, [&](uint32_t tok) {
        const uint32_t w = tok >> 5, m = 1u << (tok & 31);
        int p = 0;
        while (p < kPlanes) {
            const uint32_t old = atomicXor(&planes[p * RW + w], m);
            if (!(old & m)) break;
            ++p;
        }
        top = p > top ? p : top;
    });
    return (int)__reduce_max_sync(kFull, (unsigned)(top + 1));
}

// The plane area clean again after a read of `used` planes.
template <int Q>
__device__ __forceinline__ void clean_planes(uint32_t* __restrict__ planes, int used, int lane) {
    __syncwarp();
    if (used * GatherGeo<Q>::kRowWords > kCleanFrom<Q>) {
        for (int i = kCleanFrom<Q> + lane; i < used * GatherGeo<Q>::kRowWords; i += 32) planes[i] = 0;
        __syncwarp();
    }
}

// The whole filter for read r, by one warp (steps 0-5 above).  The warp's
// plane area is zero from kCleanFrom on at entry, and left so.
// ro, re: the read's bases; co, ce: its candidates; e: its edit budget.
template <int Q, bool DEEP>
__device__ __forceinline__ void gather_read(int64_t ro, int64_t re, int64_t co, int64_t ce, int e,
                                            const uint32_t* __restrict__ bank, int64_t n_bins,
                                            const uint8_t* __restrict__ reads,
                                            const uint32_t* __restrict__ cand_bins, uint8_t* __restrict__ pass,
                                            uint16_t* __restrict__ sums, uint32_t* __restrict__ planes, int lane,
                                            uint32_t& flags) {
    using G = GatherGeo<Q>;
    const uint4* planes4 = reinterpret_cast<const uint4*>(planes);
    if (ce < co) {  // nothing sensible to write for this read
        flags |= GRIM_FLAG_BAD_OFFSETS;
        return;
    }
    // 0. the first candidate rows in flight while the tokens are built
    const uint32_t n_bins32 = (uint32_t)n_bins;  // n_bins < 2^32 (checked when the bank is built)
    const int n_c = (int)(ce - co);
    const uint32_t* cands = cand_bins + co;
    Stream<Q, DEEP> st;
    if (n_c > 0) stream_start<Q, DEEP>(st, cands, n_c, bank, n_bins32, lane);

    bool bad_read = false;
    int L = 0;
    if (re < ro) {
        flags |= GRIM_FLAG_BAD_OFFSETS;
        bad_read = true;
    } else if (re - ro > GRIM_MAX_READ_LEN) {
        flags |= GRIM_FLAG_LONG_READ;
        bad_read = true;
    } else {
        L = (int)(re - ro);
    }
    const uint8_t* rd = reads + ro;

    // 1-2. tokens into bit-sliced count planes
    uint32_t bad_base = 0;
    const int n_tok = L - Q + 1 > 0 ? L - Q + 1 : 0;
    int used = build_planes<Q>(rd, L, n_tok, planes, lane, bad_base);
    if (__any_sync(kFull, bad_base)) {
        flags |= GRIM_FLAG_BAD_BASE;
        bad_read = true;
    }
    __syncwarp();
    const int T = n_tok - Q * e;

    // 3-5. score the candidates
    if (co < ce) {
        if (bad_read || used == 0)
            write_constant(co, ce, cand_bins, n_bins, !bad_read && T <= 0, pass, sums, lane, flags);
        else {
            // the read's planes: one, two or three in registers, the upper of two
            // folded when it is sparse enough; anything else from shared memory
            // q = 6: a read of one plane and a short list goes the way of two, the second
            // empty (the area is clean past `used`): short and long reads side by side
            // then share one loop's code (not where a warp has one read only: 2-4%
            // slower so).  150,000 reads of 50-300 bases, 8 candidates
            // each, 228 -> 203 us (32: 362 -> 331); long lists are faster by one plane.
            if (Q >= 6 && !DEEP && used == 1 && n_c <= 96) used = 2;
            bool sparse = false;
            if (G::kVPL == 2 && used == 2) {
                const uint4* top = planes4 + G::kRowVecs + lane % G::kLPB;
                sparse = sparse_plane(top[0], top[G::kLPB * (G::kVPL - 1)]);
            }
            uint16_t* sums_r = sums ? sums + co : nullptr;
            if (used == 1)
                score_read<Q, 1, DEEP>(st, planes4, used, T, n_c, cands, bank, n_bins32, pass + co, sums_r, lane, flags);
            else if (used == 2 && sparse)
                score_read<Q, 2, DEEP, true>(st, planes4, used, T, n_c, cands, bank, n_bins32, pass + co, sums_r, lane,
                                             flags);
            else if (used == 2)
                score_read<Q, 2, DEEP>(st, planes4, used, T, n_c, cands, bank, n_bins32, pass + co, sums_r, lane, flags);
            else if (Q <= 5 && used == 3)  // for q = 6 three planes stay in shared memory
                score_read<Q, 3, DEEP>(st, planes4, used, T, n_c, cands, bank, n_bins32, pass + co,
                                                     sums_r, lane, flags);
            else
                score_read<Q, 0, DEEP>(st, planes4, used, T, n_c, cands, bank, n_bins32, pass + co, sums_r, lane, flags);
        }
    }

    clean_planes<Q>(planes, used, lane);  // for the warp's next read
}

// Modelled cost of the reads before r: 8 per candidate, 1 per base, 64 per
// read.  Strictly increasing in r for valid offsets, so equal cost shares
// are contiguous, disjoint read ranges that cover every read.
__device__ __forceinline__ int64_t cost_before(const int64_t* __restrict__ read_offsets,
                                               const int64_t* __restrict__ cand_offsets, int64_t r) {
    return 8 * (__ldg(cand_offsets + r) - __ldg(cand_offsets)) + (__ldg(read_offsets + r) - __ldg(read_offsets)) +
           64 * r;
}

// Smallest r in [0, n] with cost_before(r) >= target, found by a half-warp
// 16-ary search: lanes 0-15 search target0, lanes 16-31 target1.  Every
// lane returns its own half's answer.
__device__ int64_t split_search(const int64_t* __restrict__ read_offsets, const int64_t* __restrict__ cand_offsets,
                                int64_t n, int64_t target0, int64_t target1, int lane) {
    const int j = lane & 15;
    const int64_t target = lane < 16 ? target0 : target1;
    int64_t lo = 0, hi = n;  // the answer lies in [lo, hi]
    while (__any_sync(kFull, hi - lo > 16)) {
        const int64_t p = lo + (hi - lo) * (j + 1) / 17;  // sorted samples inside [lo, hi)
        const unsigned below = __ballot_sync(kFull, cost_before(read_offsets, cand_offsets, p) < target);
        const unsigned half = lane < 16 ? below & 0xFFFFu : below >> 16;
        const int k = __popc(half);  // the samples below target are a prefix
        const int64_t p_last = __shfl_sync(kFull, p, (lane & 16) + (k > 0 ? k - 1 : 0));
        const int64_t p_next = __shfl_sync(kFull, p, (lane & 16) + (k < 16 ? k : 15));
        if (k > 0) lo = p_last + 1;
        if (k < 16) hi = p_next;
        if (lo > hi) lo = hi;  // only with a non-monotone cost (invalid offsets)
    }
    const int64_t p = lo + j;
    const bool below = p < hi && cost_before(read_offsets, cand_offsets, p) < target;
    const unsigned b = __ballot_sync(kFull, below);
    return lo + __popc(lane < 16 ? b & 0xFFFFu : b >> 16);
}

// floor(total * i / n) without overflow, for 0 <= i <= n.
__device__ __forceinline__ int64_t cost_share(int64_t total, int64_t i, int64_t n) {
    return total / n * i + total % n * i / n;
}

// The gather launch: one wave of CTAs of WARPS warps whose warps claim
// `claim` reads at a time, in one of two ways.
//  - counter == nullptr: each CTA owns the contiguous read range of an equal
//    share of the modelled cost and claims from a shared-memory counter.  No
//    device state, so concurrent launches on different streams stay
//    independent (the one-launch filter).
//  - counter != nullptr: every warp claims from that zeroed device counter,
//    which also absorbs speed differences between SMs; the batched filter
//    resets it before each launch of its graph.
template <int Q, int WARPS, bool DEEP>
__global__ void __launch_bounds__(WARPS * 32, (Q >= 6 || DEEP ? 24 : 32) / WARPS)
gather_kernel(const uint32_t* __restrict__ bank, int64_t n_bins, const uint8_t* __restrict__ reads,
              const int64_t* __restrict__ read_offsets, int64_t n_reads, const uint32_t* __restrict__ cand_bins,
              const int64_t* __restrict__ cand_offsets, const uint16_t* __restrict__ E,
              uint8_t* __restrict__ pass, uint16_t* __restrict__ sums, uint32_t* __restrict__ status, int claim,
              unsigned long long* __restrict__ counter) {
    using G = GatherGeo<Q>;
    extern __shared__ uint4 gather_smem[];
    __shared__ unsigned long long next_read;
    __shared__ long long end_read;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    uint32_t* planes = reinterpret_cast<uint32_t*>(gather_smem) + warp * G::kPlaneWords;
    if (counter == nullptr && warp == 0) {
        const int64_t n_ctas = gridDim.x, b = blockIdx.x;
        const int64_t total = cost_before(read_offsets, cand_offsets, n_reads);
        const int64_t split = split_search(read_offsets, cand_offsets, n_reads, cost_share(total, b, n_ctas),
                                           cost_share(total, b + 1, n_ctas), lane);
        const int64_t r_begin = __shfl_sync(kFull, split, 0);
        const int64_t r_end = __shfl_sync(kFull, split, 16);
        // The ends are pinned so that every read lies in some CTA's range even
        // when decreasing (invalid) offsets break the monotone cost; such
        // reads are then flagged by whichever warp visits them.
        if (lane == 0) {
            next_read = b == 0 ? 0 : (unsigned long long)r_begin;
            end_read = b == n_ctas - 1 ? n_reads : r_end;
        }
    }
    gather_warp_setup<Q>(planes, lane);
    __syncthreads();  // next_read; kept for counter launches too, whose code spilled 60-200 bytes without it
    const int64_t r_end = counter ? n_reads : end_read;
    unsigned long long* next = counter ? counter : &next_read;

    uint32_t flags = 0;
    while (true) {
        unsigned long long r0 = 0;
        if (lane == 0) r0 = atomicAdd(next, (unsigned long long)claim);
        r0 = __shfl_sync(kFull, r0, 0);
        if ((int64_t)r0 >= r_end) break;
        const int64_t r1 = (int64_t)r0 + claim < r_end ? (int64_t)r0 + claim : r_end;
        for (int64_t r = (int64_t)r0; r < r1; r++)
            gather_read<Q, DEEP>(read_offsets[r], read_offsets[r + 1], cand_offsets[r], cand_offsets[r + 1], E[r],
                                 bank, n_bins, reads, cand_bins, pass, sums, planes, lane, flags);
    }
    flags = __reduce_or_sync(kFull, flags);
    if (lane == 0 && flags) atomicOr(status, flags);
}

// A batch of no more reads than the GPU holds warps: one read per warp, no
// shares to work out and no counter, spread over every SM (1,000 reads of 32
// candidates: 32 CTAs of the kernel above, claiming four reads a warp, took
// 9.2 us of device time).
constexpr int kSmallWarps = 4;

template <int Q>
__global__ void __launch_bounds__(kSmallWarps * 32)
gather_small_kernel(const uint32_t* __restrict__ bank, int64_t n_bins, const uint8_t* __restrict__ reads,
                    const int64_t* __restrict__ read_offsets, int64_t n_reads,
                    const uint32_t* __restrict__ cand_bins, const int64_t* __restrict__ cand_offsets,
                    const uint16_t* __restrict__ E, uint8_t* __restrict__ pass, uint16_t* __restrict__ sums,
                    uint32_t* __restrict__ status) {
    extern __shared__ uint4 gather_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * kSmallWarps + warp;
    if (r >= n_reads) return;
    const int64_t ro = read_offsets[r], re = read_offsets[r + 1], co = cand_offsets[r], ce = cand_offsets[r + 1];
    uint32_t* planes = reinterpret_cast<uint32_t*>(gather_smem) + warp * GatherGeo<Q>::kPlaneWords;
    gather_warp_setup<Q>(planes, lane);
    uint32_t flags = 0;
    gather_read<Q, true>(ro, re, co, ce, E[r], bank, n_bins, reads, cand_bins, pass, sums, planes, lane, flags);
    flags = __reduce_or_sync(kFull, flags);
    if (lane == 0 && flags) atomicOr(status, flags);
}

template <int Q>
static int launch_small(const grim_bank* bank, const GatherArgs& a, int64_t r0, int64_t n, cudaStream_t s) {
    constexpr size_t smem = gather_smem_bytes<Q>(kSmallWarps);
    static_assert(smem <= 48 * 1024, "no attribute needed");
    gather_small_kernel<Q><<<grim::fault_grid((unsigned)((n + kSmallWarps - 1) / kSmallWarps)), kSmallWarps * 32, smem,
                             s>>>(bank->bits, bank->n_bins, a.reads, a.read_offsets + r0, n, a.cand_bins,
                                  a.cand_offsets + r0, a.E + r0, a.pass, a.sums, bank->status);
    GRIM_CUDA_TRY(cudaGetLastError());
    return GRIM_OK;
}

// Up to 16 reads an SM take gather_small_kernel: as many warps as it holds at
// once (96 registers), and no more reads than the claiming kernel would give
// each warp one of.  1,000 reads of 32 candidates: 12.3 -> 11.5 us a call, 47
// -> 38 us for a first call on new buffers.
constexpr int kSmallReadsPerSm = 16;

// Banks larger than this are read from HBM rather than L2: the gather then
// keeps three steps of rows in flight per warp (the DEEP form).
constexpr double kDeepBankBytes = 96e6;

// One launch over reads [r0, r0 + n) with `per_sm` CTAs per SM (0 = as many
// as fit).
template <int Q, int WARPS, bool DEEP>
static int launch_range(const grim_bank* bank, const GatherArgs& a, int64_t r0, int64_t n, int per_sm, int claim,
                        unsigned long long* counter, cudaStream_t s) {
    constexpr size_t smem = gather_smem_bytes<Q>(WARPS);
    static DeviceCache max_blocks_of[64];  // per device, like the attribute
    const int slot = device_slot();
    if (slot < 0) return GRIM_ENOTSUP;
    if (max_blocks_of[slot].load() == 0) {
        if (smem > 48 * 1024)
            GRIM_CUDA_TRY(cudaFuncSetAttribute(gather_kernel<Q, WARPS, DEEP>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        int b = 0;
        GRIM_CUDA_TRY(
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, gather_kernel<Q, WARPS, DEEP>, WARPS * 32, smem));
        max_blocks_of[slot].store(b > 0 ? b : 1);
    }
    const int max_blocks = max_blocks_of[slot].load();
    if (per_sm <= 0 || per_sm > max_blocks) per_sm = max_blocks;
    if (claim <= 0) claim = 1;
    int64_t blocks = (int64_t)sm_count() * per_sm;
    // fewer claims than warps: one read to a claim, to occupy every SM
    if (n < blocks * WARPS * claim) claim = 1;
    const int64_t need = (n + (int64_t)WARPS * claim - 1) / ((int64_t)WARPS * claim);  // a claim per warp at least
    if (need < blocks) blocks = need;
    if (counter) GRIM_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s));
    gather_kernel<Q, WARPS, DEEP><<<grim::fault_grid((unsigned)blocks), WARPS * 32, smem, s>>>(
        bank->bits, bank->n_bins, a.reads, a.read_offsets + r0, n, a.cand_bins, a.cand_offsets + r0, a.E + r0,
        a.pass, a.sums, bank->status, claim, counter);
    GRIM_CUDA_TRY(cudaGetLastError());
    return GRIM_OK;
}

// ------------------------------------------------------------ by bank segment

// A bank beyond the L2 whose rows are scored many times over (3.1 Gbp, 1M
// reads of ~1,700 candidates: 138 checks a row) is read from HBM once per
// check by the kernels above.  Here the checks go segment by segment of the
// bank (72 MB, about half the L2), all reads' candidates in one segment before
// the next, so that a segment comes from HBM once and its rows from the L2:
//   1. blocked_prep_kernel (warp per read): the read's count planes and
//      threshold to memory, and where each segment's candidates start in its
//      list.  Lists ascend as seed tables give them; one that does not is cut
//      at other places and only loses the order (every candidate is scored by
//      its own id whatever segment it was counted to).  A read that is
//      invalid or has no or more than four planes is listed for step 3 (one
//      such read is a serial tail of 0.2 ms: its rows come from HBM);
//   2. blocked_kernel: warps claim (segment, 32 reads) in segment order; the
//      next read's planes (cp.async) and candidate ids come in while one is
//      scored;
//   3. blocked_direct_kernel: the listed reads as in gather_kernel.
// 3.1 Gbp, 1M reads, 1.67e9 checks: 38.2 -> 23.0 ms, of which the ordering
// (step 1) is 1.25.  Bound: issue, and the breaks between the short runs of two
// reads (rows from the L2 at 9.8 TB/s; loads that do nothing else reach 15).
// When it took 25.3: segments of 32 MB 29.9 (half as many candidates per read
// and segment), of 128 MB 27.9; 3 CTAs of 8 warps 26.4; two row buffers and 4
// CTAs 27.3.
constexpr size_t kSegmentBytes = size_t(72) << 20;
// Where the line lies (q = 5, reads of 100 bases unless said; by segment
// against the claiming kernel, ms): rows of 8 GB read in all - 3.1 Gbp 30,000
// reads (6.4 GB) 1.18 / 1.18, 60,000 1.95 / 2.23, 120,000 3.28 / 4.35, 1M 25.3
// / 37.9; 1 Gbp 60,000 (4 GB) 0.71 / 0.69, 200,000 1.77 / 2.14; 600 Mbp 400,000
// 2.13 / 2.42.  Banks of 200 MB are half in the L2 already: 0.50 / 0.42.  At
// least 20 candidates of a read in a segment, or the switches between reads
// cost more: 24 (reads of 36 bases) 3.84 / 4.20, 16 (24 bases) 4.27 / 3.78.
// q = 6 rows are slower this way (100 Mbp: 11.4 / 9.7) and are left as above.
constexpr double kBlockedBankBytes = 256e6;
constexpr double kBlockedRowBytes = 8e9;
constexpr int64_t kBlockedChecksPerItem = 20;
constexpr int kMaxSegments = 256;
constexpr int64_t kBlockedReads = int64_t(1) << 20;  // reads per round over the bank

struct BlockedRead {
    int T;
    // 0: two planes, the upper one folded (row_sum8); 1: two planes; 2 + 2 i: three, 3 + 2 i: four, the last two in extra[i]
    int mode;
};
// One read in so many may have three or four planes: one in 5 of reads of 300
// bases does, and those left over are a serial tail from HBM (3.1 Gbp, 20,000
// reads of 300 bases, 2.60 ms at one in 16, 2.17 so; the one launch 2.30).
constexpr int kExtraShare = 4;

template <int Q>
__global__ void __launch_bounds__(kSmallWarps * 32)
blocked_prep_kernel(const uint8_t* __restrict__ reads, const int64_t* __restrict__ read_offsets, int64_t n_reads,
                    const uint32_t* __restrict__ cand_bins, const int64_t* __restrict__ cand_offsets,
                    const uint16_t* __restrict__ E, uint32_t seg_bins, int n_seg,
                    uint4* __restrict__ planes_out, uint4* __restrict__ extra, uint32_t n_extra,
                    BlockedRead* __restrict__ info, uint32_t* __restrict__ starts, uint32_t* __restrict__ list,
                    uint32_t* __restrict__ counts) {  // counts[0]: list's length, counts[2]: extra's
    using G = GatherGeo<Q>;
    extern __shared__ uint4 gather_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* planes = reinterpret_cast<uint32_t*>(gather_smem) + warp * G::kPlaneWords;
    const uint4* planes4 = reinterpret_cast<const uint4*>(planes);
    gather_warp_setup<Q>(planes, lane);
    for (int64_t r = (int64_t)blockIdx.x * kSmallWarps + warp; r < n_reads; r += (int64_t)gridDim.x * kSmallWarps) {
        const int64_t ro = read_offsets[r], re = read_offsets[r + 1], co = cand_offsets[r], ce = cand_offsets[r + 1];
        bool direct = ce < co || ce - co > 0x7fffffff || re < ro || re - ro > GRIM_MAX_READ_LEN;
        const int n_c = direct ? 0 : (int)(ce - co);
        if (!direct) {
            const int L = (int)(re - ro), n_tok = L - Q + 1 > 0 ? L - Q + 1 : 0;
            uint32_t bad_base = 0;
            const int used = build_planes<Q>(reads + ro, L, n_tok, planes, lane, bad_base);
            direct = __any_sync(kFull, bad_base) || (n_c > 0 && (used < 1 || used > 4));
            __syncwarp();
            if (!direct && n_c > 0) {
                int mode = 0;
                if (used > 2) {
                    uint32_t x = 0;
                    if (lane == 0) x = atomicAdd(counts + 2, 1u);
                    x = __shfl_sync(kFull, x, 0);
                    direct = x >= n_extra;
                    mode = 2 + 2 * (int)x + (used == 4 ? 1 : 0);
                    if (!direct)
                        for (int v = lane; v < 2 * G::kRowVecs; v += 32)  // planes 2 and 3
                            extra[(size_t)x * 2 * G::kRowVecs + v] =
                                v < G::kRowVecs || used == 4 ? planes4[2 * G::kRowVecs + v] : make_uint4(0, 0, 0, 0);
                } else {
                    const uint4* top = planes4 + G::kRowVecs + lane % G::kLPB;
                    mode = used == 1 || sparse_plane(top[0], top[G::kLPB * (G::kVPL - 1)]) ? 0 : 1;
                }
                for (int v = lane; v < 2 * G::kRowVecs; v += 32)
                    planes_out[r * 2 * G::kRowVecs + v] =
                        v < G::kRowVecs || used >= 2 ? planes4[v] : make_uint4(0, 0, 0, 0);
                if (lane == 0) info[r] = BlockedRead{n_tok - Q * (int)E[r], mode};
            }
            clean_planes<Q>(planes, used, lane);
        }
        // where each segment's candidates start: a search among 32 samples of
        // the list, then in the stretch between two of them
        const uint32_t* cands = cand_bins + co;
        const uint32_t sample = n_c > 0 ? __ldg(cands + (int)((int64_t)lane * n_c >> 5)) : 0u;
        uint32_t before = 0;
        for (int s0 = 0; s0 <= n_seg; s0 += 32) {
            const int sg = s0 + lane;
            const uint32_t key = (uint32_t)sg * seg_bins;  // sg < n_seg: below n_bins
            int lo = 0, hi = 32;  // samples below key: a prefix of an ascending list
#pragma unroll
            for (int step = 0; step < 5; step++) {
                const int mid = (lo + hi) >> 1;
                if (__shfl_sync(kFull, sample, mid) < key) lo = mid;
                else hi = mid;
            }
            uint32_t at = 0;
            if (sg >= n_seg) {
                at = (uint32_t)n_c;
            } else if (sg > 0 && n_c > 0) {
                int a = (int)((int64_t)lo * n_c >> 5), z = hi < 32 ? (int)((int64_t)hi * n_c >> 5) : n_c;
                while (a < z) {
                    const int mid = (a + z) >> 1;
                    if (__ldg(cands + mid) < key) a = mid + 1;
                    else z = mid;
                }
                at = (uint32_t)a;
            }
            // in an unordered list the places found need not ascend
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, at, o);
                if (lane >= o) at = y > at ? y : at;
            }
            at = before > at ? before : at;
            before = __shfl_sync(kFull, at, 31);
            if (sg <= n_seg) starts[(int64_t)sg * n_reads + r] = direct ? 0u : at;
        }
        if (direct && lane == 0) list[atomicAdd(counts, 1u)] = (uint32_t)r;
        __syncwarp();
    }
}

constexpr int kBlockedWarps = 4;
constexpr int kBlockedCtas = 6;  // per SM (80 registers); 7 of 72 24.7 ms for 23.0, 5 of 96 23.6

template <int Q>
__global__ void __launch_bounds__(kBlockedWarps * 32, kBlockedCtas)
blocked_kernel(const uint32_t* __restrict__ bank, uint32_t n_bins32, const uint32_t* __restrict__ cand_bins,
               const int64_t* __restrict__ cand_offsets, int64_t n_reads, int n_seg,
               const uint4* __restrict__ planes_in, const uint4* __restrict__ extra, const BlockedRead* __restrict__ info,
               const uint32_t* __restrict__ starts, uint8_t* __restrict__ pass, uint32_t* __restrict__ status,
               unsigned long long* __restrict__ counter) {
    using G = GatherGeo<Q>;
    using S = Stream<Q, true>;
    constexpr int kVecs = 2 * G::kRowVecs;  // two planes
    __shared__ uint4 planes_s[kBlockedWarps][2][2 * kVecs];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = lane % G::kLPB, g = lane / G::kLPB;
    const int64_t groups = (n_reads + 31) >> 5, total = groups * n_seg;
    uint32_t flags = 0;
    while (true) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(counter, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if ((int64_t)item >= total) break;
        const int64_t sg = (int64_t)item / groups, r0 = ((int64_t)item - sg * groups) << 5;
        // lane i: read r0 + i's candidates in this segment
        int64_t first = 0;
        int n_l = 0;
        BlockedRead rd{0, 0};
        if (r0 + lane < n_reads) {
            const uint32_t lo = __ldg(starts + sg * n_reads + r0 + lane);
            n_l = (int)(__ldg(starts + (sg + 1) * n_reads + r0 + lane) - lo);
            if (n_l > 0) {
                first = __ldg(cand_offsets + r0 + lane) + lo;
                rd = info[r0 + lane];
            }
        }
        uint32_t todo = __ballot_sync(kFull, n_l > 0);
        if (todo == 0) continue;
        int i = __ffs(todo) - 1, buf = 0;
        auto ask = [&](uint4* dst, const uint4* src) {
#pragma unroll
            for (int v = lane; v < kVecs; v += 32)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(dst + v)),
                             "l"(src + v)
                             : "memory");
        };
        auto ask_planes = [&](int which, int b) {
            ask(planes_s[warp][b], planes_in + (r0 + which) * kVecs);
            const int mode = __shfl_sync(kFull, rd.mode, which);
            if (mode >= 2) ask(planes_s[warp][b] + kVecs, extra + (size_t)((mode - 2) >> 1) * kVecs);
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        ask_planes(i, 0);
        int64_t at = __shfl_sync(kFull, first, i);
        int n = __shfl_sync(kFull, n_l, i);
        uint32_t id0 = window_id(cand_bins + at, lane, n), id1 = window_id(cand_bins + at, 32 + lane, n);
        while (true) {
            const int64_t at_now = at;
            const int n_now = n, i_now = i;
            S st;
            st.win_cur = id0;
            st.win_next = id1;
#pragma unroll
            for (int k = 0; k < S::kAhead; k++) {
                const int idx = k * G::kBPS + g;
                const uint32_t id = __shfl_sync(kFull, idx < 32 ? st.win_cur : st.win_next, idx & 31);
                fetch_row<Q>(st.r[k], id, bank, n_bins32, s);
            }
            todo &= todo - 1;
            if (todo) {  // the next read's planes and ids
                i = __ffs(todo) - 1;
                ask_planes(i, buf ^ 1);
                at = __shfl_sync(kFull, first, i);
                n = __shfl_sync(kFull, n_l, i);
                id0 = window_id(cand_bins + at, lane, n);
                id1 = window_id(cand_bins + at, 32 + lane, n);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncwarp();
            const int T = __shfl_sync(kFull, rd.T, i_now);
            const int mode = __shfl_sync(kFull, rd.mode, i_now);
            if (mode == 0)
                score_read<Q, 2, true, true>(st, planes_s[warp][buf], 2, T, n_now, cand_bins + at_now, bank, n_bins32,
                                             pass + at_now, nullptr, lane, flags);
            else if (mode == 1)
                score_read<Q, 2, true>(st, planes_s[warp][buf], 2, T, n_now, cand_bins + at_now, bank, n_bins32,
                                       pass + at_now, nullptr, lane, flags);
            else
                score_read<Q, 0, true>(st, planes_s[warp][buf], 3 + (mode & 1), T, n_now, cand_bins + at_now, bank, n_bins32,
                                       pass + at_now, nullptr, lane, flags);
            __syncwarp();
            if (!todo) break;
            buf ^= 1;
        }
    }
    flags = __reduce_or_sync(kFull, flags);
    if (lane == 0 && flags) atomicOr(status, flags);
}

template <int Q>
__global__ void __launch_bounds__(kSmallWarps * 32, 5)
blocked_direct_kernel(const uint32_t* __restrict__ bank, int64_t n_bins, const uint8_t* __restrict__ reads,
                      const int64_t* __restrict__ read_offsets, const uint32_t* __restrict__ cand_bins,
                      const int64_t* __restrict__ cand_offsets, const uint16_t* __restrict__ E,
                      uint8_t* __restrict__ pass, uint32_t* __restrict__ status, const uint32_t* __restrict__ list,
                      const uint32_t* __restrict__ n_list, uint32_t* __restrict__ next) {
    extern __shared__ uint4 gather_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* planes = reinterpret_cast<uint32_t*>(gather_smem) + warp * GatherGeo<Q>::kPlaneWords;
    gather_warp_setup<Q>(planes, lane);
    const uint32_t n = *n_list;
    uint32_t flags = 0;
    while (true) {
        uint32_t i = 0;
        if (lane == 0) i = atomicAdd(next, 1u);
        i = __shfl_sync(kFull, i, 0);
        if (i >= n) break;
        const uint32_t r = list[i];
        gather_read<Q, true>(read_offsets[r], read_offsets[r + 1], cand_offsets[r], cand_offsets[r + 1], E[r], bank,
                             n_bins, reads, cand_bins, pass, nullptr, planes, lane, flags);
    }
    flags = __reduce_or_sync(kFull, flags);
    if (lane == 0 && flags) atomicOr(status, flags);
}

template <int Q>
static int launch_blocked(const grim_bank* bank, const GatherArgs& a, uint32_t seg_bins, int n_seg, cudaStream_t s) {
    using G = GatherGeo<Q>;
    const int64_t most = a.n_reads < kBlockedReads ? a.n_reads : kBlockedReads;
    const size_t planes_bytes = (size_t)most * 2 * G::kRowVecs * 16, info_bytes = (size_t)most * sizeof(BlockedRead);
    const uint32_t n_extra = (uint32_t)(most / kExtraShare + 32);
    const size_t extra_bytes = (size_t)n_extra * 2 * G::kRowVecs * 16;
    const size_t starts_bytes = ((size_t)(n_seg + 1) * most * 4 + 15) & ~(size_t)15;
    uint8_t* mem = nullptr;
    const cudaError_t ea = scratch_alloc((void**)&mem, 64 + planes_bytes + extra_bytes + info_bytes + starts_bytes + most * 4, s);
    if (ea != cudaSuccess) {
        cudaGetLastError();
        return kBlockedNoMemory;
    }
    unsigned long long* counter = reinterpret_cast<unsigned long long*>(mem);
    uint32_t *counts = reinterpret_cast<uint32_t*>(mem + 8), *next = counts + 1;  // counts[0], next, counts[2]
    uint8_t* p = mem + 64;
    uint4* planes = reinterpret_cast<uint4*>(p);
    uint4* extra = reinterpret_cast<uint4*>(p += planes_bytes);
    BlockedRead* info = reinterpret_cast<BlockedRead*>(p += extra_bytes);
    uint32_t* starts = reinterpret_cast<uint32_t*>(p += info_bytes);
    uint32_t* list = reinterpret_cast<uint32_t*>(p += starts_bytes);
    constexpr size_t smem = gather_smem_bytes<Q>(kSmallWarps);
    cudaError_t e = cudaSuccess;
    for (int64_t r0 = 0; r0 < a.n_reads && e == cudaSuccess; r0 += most) {
        const int64_t n = a.n_reads - r0 < most ? a.n_reads - r0 : most;
        e = cudaMemsetAsync(mem, 0, 64, s);
        if (e != cudaSuccess) break;
        const int64_t need = (n + kSmallWarps - 1) / kSmallWarps, wave = (int64_t)sm_count() * 12;
        blocked_prep_kernel<Q><<<fault_grid((unsigned)(need < wave ? need : wave)), kSmallWarps * 32, smem, s>>>(
            a.reads, a.read_offsets + r0, n, a.cand_bins, a.cand_offsets + r0, a.E + r0,
            seg_bins, n_seg, planes, extra, n_extra, info, starts, list, counts);
        e = cudaGetLastError();
        if (e != cudaSuccess) break;
        blocked_kernel<Q><<<fault_grid((unsigned)(sm_count() * kBlockedCtas)), kBlockedWarps * 32, 0, s>>>(
            bank->bits, (uint32_t)bank->n_bins, a.cand_bins, a.cand_offsets + r0, n, n_seg, planes, extra, info, starts,
            a.pass, bank->status, counter);
        e = cudaGetLastError();
        if (e != cudaSuccess) break;
        blocked_direct_kernel<Q><<<fault_grid((unsigned)(sm_count() * 4)), kSmallWarps * 32, smem, s>>>(
            bank->bits, bank->n_bins, a.reads, a.read_offsets + r0, a.cand_bins, a.cand_offsets + r0, a.E + r0, a.pass,
            bank->status, list, counts, next);
        e = cudaGetLastError();
    }
    cudaFreeAsync(mem, s);
    if (e != cudaSuccess) {
        set_last_cuda_error(e);
        return GRIM_ECUDA;
    }
    return GRIM_OK;
}

int launch_gather_blocked(const grim_bank* bank, const GatherArgs& a, int64_t n_checks, cudaStream_t s) {
    const int64_t row_bytes = bank->row_words * 4;
    if (bank->q != 5 || a.sums || (double)bank->n_bins * (double)row_bytes < kBlockedBankBytes)
        return kBlockedNotBetter;
    const int64_t n_seg = (bank->n_bins * row_bytes + (int64_t)kSegmentBytes - 1) / (int64_t)kSegmentBytes;
    const int64_t seg_bins = (bank->n_bins + n_seg - 1) / n_seg;  // equal segments
    if (n_seg > kMaxSegments || (double)n_checks * (double)row_bytes < kBlockedRowBytes ||
        n_checks < kBlockedChecksPerItem * n_seg * a.n_reads)
        return kBlockedNotBetter;
    return launch_blocked<5>(bank, a, (uint32_t)seg_bins, (int)n_seg, s);
}

template <int Q>
static int launch_batches(const grim_bank* bank, const GatherArgs& a, const grim_tune& t,
                          unsigned long long* counter, cudaStream_t s) {
    const int64_t batch = t.batch_reads > 0 ? t.batch_reads : a.n_reads;
    const bool deep = Q <= 5 && (double)bank->n_bins * (double)bank->row_words * 4.0 > kDeepBankBytes;
    constexpr bool kDeepForm = Q <= 5;  // q = 6 keeps its rows three steps ahead in either form
    for (int64_t r0 = 0; r0 < a.n_reads; r0 += batch) {
        const int64_t n = (a.n_reads - r0) < batch ? (a.n_reads - r0) : batch;
        const int pc = t.ctas_per_sm, rc_ = t.reads_per_claim;
        int rc;
        if (n <= kSmallReadsPerSm * (int64_t)sm_count())
            rc = launch_small<Q>(bank, a, r0, n, s);
        else if (deep)
            rc = t.warps_per_cta == 4 ? launch_range<Q, 4, kDeepForm>(bank, a, r0, n, pc, rc_, counter, s)
                                      : launch_range<Q, 8, kDeepForm>(bank, a, r0, n, pc, rc_, counter, s);
        else
            rc = t.warps_per_cta == 4 ? launch_range<Q, 4, false>(bank, a, r0, n, pc, rc_, counter, s)
                                      : launch_range<Q, 8, false>(bank, a, r0, n, pc, rc_, counter, s);
        if (rc != GRIM_OK) return rc;
    }
    return GRIM_OK;
}

int launch_gather_batches(const grim_bank* bank, const GatherArgs& a, const grim_tune& t,
                          unsigned long long* counter, cudaStream_t s) {
    switch (bank->q) {
        case 1: return launch_batches<1>(bank, a, t, counter, s);
        case 2: return launch_batches<2>(bank, a, t, counter, s);
        case 3: return launch_batches<3>(bank, a, t, counter, s);
        case 4: return launch_batches<4>(bank, a, t, counter, s);
        case 5: return launch_batches<5>(bank, a, t, counter, s);
        case 6: return launch_batches<6>(bank, a, t, counter, s);
        default: return GRIM_ENOTSUP;
    }
}

int launch_gather(const grim_bank* bank, const uint8_t* reads, const int64_t* read_offsets, int64_t n_reads,
                  const uint32_t* cand_bins, const int64_t* cand_offsets, const uint16_t* E, uint8_t* pass,
                  uint16_t* sums, cudaStream_t s) {
    const GatherArgs a{reads, read_offsets, n_reads, cand_bins, cand_offsets, E, pass, sums};
    const grim_tune t = {kGatherWarps, 4, 0, 0, 0};  // one launch over every read, 4 reads per claim
    return launch_gather_batches(bank, a, t, nullptr, s);
}

}  // namespace grim
