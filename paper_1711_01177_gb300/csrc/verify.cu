// Verification side of the filter (the aligner's check and the paper's
// quality metrics, Sec. 5 and 6.1).
//
// grim_verify: for each location (read r, bin b), the semi-global edit
// distance of r against b's span - the fewest edits that turn r into some
// substring of the span (Sellers' recurrence: free start and end in the
// text).  A location "results in a mapping" when that distance is <= E.
// One thread per location runs Myers' bit-vector form of the recurrence
// (Myers, 1999, "A fast bit-vector algorithm for approximate string matching
// based on dynamic programming"): the vertical differences of one column of
// the table, 32 or 64 rows per machine word, advance by a handful of word
// operations per column.  Spans of up to 1,024 bases are the rows, the read's
// bases the columns (verify_rows_kernel); for longer spans the read's bases
// are the rows, in 64-row blocks that exchange only the horizontal difference
// at their boundary row (Myers, Sec. 4; verify_kernel).
//
// grim_verify_stats: counts of passing / rejected locations with and
// without a mapping, from which the paper's "false negative rate" (passing
// locations without a mapping over all passing locations) and the zero-miss
// property (no rejected location with a mapping) follow.
#include "grim_internal.cuh"

namespace grim {
namespace {

constexpr int kVerifyMaxBlocks = 8;  // reads up to 512 bases

__device__ __forceinline__ uint32_t ref_code(const uint8_t* __restrict__ ref2bit, int64_t i) {
    return (__ldg(ref2bit + (i >> 2)) >> (2 * (i & 3))) & 3u;
}

// One text column for one 64-row block: updates the block's vertical
// differences (Pv: +1 rows, Mv: -1 rows) given the horizontal difference
// hin entering at its top row; returns the horizontal difference at the row
// marked by `top` (the block's last read row).
__device__ __forceinline__ int myers_step(uint64_t& Pv, uint64_t& Mv, uint64_t Eq, int hin, uint64_t top) {
    const uint64_t Xv = Eq | Mv;
    if (hin < 0) Eq |= 1ull;
    const uint64_t Xh = (((Eq & Pv) + Pv) ^ Pv) | Eq;
    uint64_t Ph = Mv | ~(Xh | Pv);
    uint64_t Mh = Pv & Xh;
    const int hout = (Ph & top) ? 1 : ((Mh & top) ? -1 : 0);
    Ph <<= 1;
    Mh <<= 1;
    if (hin < 0) Mh |= 1ull;
    else if (hin > 0) Ph |= 1ull;
    Pv = Mh | ~(Xv | Ph);
    Mv = Ph & Xv;
    return hout;
}

// Semi-global distance of read[0..L) (64 (B-1) < L <= 64 B) against the
// text ref[begin..end).
template <int B>
__device__ uint32_t sellers_distance(const uint8_t* __restrict__ read, int L, const uint8_t* __restrict__ ref2bit,
                                     int64_t begin, int64_t end) {
    uint64_t peq[4][B];
#pragma unroll
    for (int b = 0; b < B; b++) {
        uint64_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;
        const int lo = 64 * b, hi = L < 64 * (b + 1) ? L : 64 * (b + 1);
        for (int i = lo; i < hi; i++) {
            const uint32_t c = __ldg(read + i);
            const uint64_t m = 1ull << (i - lo);
            p0 |= c == 0 ? m : 0ull;
            p1 |= c == 1 ? m : 0ull;
            p2 |= c == 2 ? m : 0ull;
            p3 |= c == 3 ? m : 0ull;  // codes > 3 match nothing
        }
        peq[0][b] = p0;
        peq[1][b] = p1;
        peq[2][b] = p2;
        peq[3][b] = p3;
    }
    uint64_t Pv[B], Mv[B];
#pragma unroll
    for (int b = 0; b < B; b++) {
        Pv[b] = ~0ull;  // column 0: D[i][0] = i, every vertical difference +1
        Mv[b] = 0ull;
    }
    const uint64_t top_last = 1ull << ((L - 1) & 63);
    uint32_t score = (uint32_t)L, best = (uint32_t)L;
    for (int64_t j = begin; j < end; j++) {
        const uint32_t t = ref_code(ref2bit, j);
        int h = 0;  // row 0 of the semi-global table is all zeros
#pragma unroll
        for (int b = 0; b < B; b++) {
            const uint64_t eq = t == 0 ? peq[0][b] : t == 1 ? peq[1][b] : t == 2 ? peq[2][b] : peq[3][b];
            h = myers_step(Pv[b], Mv[b], eq, h, b == B - 1 ? top_last : (1ull << 63));
        }
        score += h;
        best = score < best ? score : best;
    }
    return best;
}

// sellers_distance for a read of nb blocks, K <= nb <= MAXB (0 for nb = 0).
template <int K, int MAXB>
__device__ __forceinline__ uint32_t distance_blocks(int nb, const uint8_t* __restrict__ read, int L,
                                                   const uint8_t* __restrict__ ref2bit, int64_t begin, int64_t end) {
    if constexpr (K > MAXB) {
        return 0;
    } else {
        if (nb == K) return sellers_distance<K>(read, L, ref2bit, begin, end);
        return distance_blocks<K + 1, MAXB>(nb, read, L, ref2bit, begin, end);
    }
}

// Locations whose read spans MINB..MAXB blocks of 64 bases; the MINB == 0
// launch also writes every location it cannot score (bad ids, decreasing
// offsets, reads longer than the largest class).  Splitting by length keeps
// the register budget of short reads small.
template <int MINB, int MAXB>
__global__ void __launch_bounds__(256)
verify_kernel(const uint8_t* __restrict__ ref2bit, int64_t len, int64_t n_bins, int bin_len, int overlap,
              const uint8_t* __restrict__ reads, const int64_t* __restrict__ read_offsets, int64_t n_reads,
              const uint32_t* __restrict__ loc_read, const uint32_t* __restrict__ loc_bin, int64_t n_loc,
              uint16_t* __restrict__ dist, uint32_t* __restrict__ status) {
    uint32_t flags = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_loc; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = loc_read[i], b = loc_bin[i];
        int64_t L = -1;
        if ((int64_t)r < n_reads && (int64_t)b < n_bins) {
            const int64_t ro = read_offsets[r], re = read_offsets[r + 1];
            L = re >= ro ? re - ro : -1;
        }
        const int nb = L <= 0 ? 0 : (int)((L + 63) / 64);
        if (L < 0 || L > 64 * kVerifyMaxBlocks) {
            if (MINB == 0) {
                flags |= (int64_t)b >= n_bins ? GRIM_FLAG_BAD_BIN
                         : L > 64 * kVerifyMaxBlocks ? GRIM_FLAG_LONG_READ : GRIM_FLAG_BAD_OFFSETS;
                dist[i] = 0xFFFF;
            }
            continue;
        }
        if (nb < MINB || nb > MAXB) continue;
        const int64_t begin = (int64_t)b * bin_len;
        const int64_t end = begin + bin_len + overlap < len ? begin + bin_len + overlap : len;
        const uint32_t d = distance_blocks<(MINB > 0 ? MINB : 1), MAXB>(nb, reads + read_offsets[r], (int)L, ref2bit,
                                                                        begin, end);
        dist[i] = (uint16_t)(d < 0xFFFF ? d : 0xFFFF);
    }
    if (flags) atomicOr(status, flags);
}

// ------------------------------------------------------------ rows = the span

// The same distances with the roles swapped: the rows of the table are the
// span's bases (W 32-bit words, W fixed by the bank's geometry), its columns
// the read's.  Every lane then runs the same code whatever its read's length,
// a column's fixed costs are paid once per read base instead of once per span
// base, and reads of different lengths share a warp with no divergence but
// their trip counts, which the CTA evens out by sorting its locations by
// length.  Boundary: D[i][0] = 0 (free start in the span), D[0][j] = j (the
// horizontal difference entering the top row is always +1); the answer is the
// minimum of the last column, found once from its vertical differences.
//
// Bound: the integer (ALU) pipe, at 10 operations per word and read base.
// The match mask of a word is one shared-memory load instead of two logic
// operations: the four masks of every word lie in the CTA's shared memory,
// word-major with one column per thread (no bank conflicts).
// 1M locations, reads of 50-300 bases, spans of 556 bases: 2.07 ms, where the
// read-as-rows kernels took 14.9 ms (three launches, each with the lanes of
// the other lengths idle, and 24 selects and logic operations a word).
constexpr int kRowThreads = 128;
constexpr int kRowMaxTile = 512;  // locations sorted together

// Bits 0, 2, .. 30 of x packed into the low 16.
__device__ __forceinline__ uint32_t even_bits(uint32_t x) {
    x &= 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0F0F0F0Fu;
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return (x | (x >> 8)) & 0xFFFFu;
}

// 32-bit word k of the packed reference (16 bases); bytes past its end read 0.
__device__ __forceinline__ uint32_t packed_word(const uint8_t* __restrict__ ref2bit, int64_t nbytes, bool aligned,
                                                int64_t k) {
    const int64_t b = 4 * k;
    if (aligned && b + 4 <= nbytes) return __ldg(reinterpret_cast<const uint32_t*>(ref2bit + b));
    uint32_t v = 0;
    for (int i = 0; i < 4; i++)
        if (b + i < nbytes) v |= (uint32_t)__ldg(ref2bit + b + i) << (8 * i);
    return v;
}

// s + p over N words, low word first: s becomes the sum.  The condition code
// lives within one asm statement; from one statement to the next the carry is
// a value (kIn: `carry` goes in; kOut: it comes out).
template <int N, bool kIn, bool kOut>
__device__ __forceinline__ void add_words(uint32_t* s, const uint32_t* p, uint32_t& carry) {
    static_assert(N == 1 || N == 2 || N == 3 || N == 8, "the group sizes below");
#define GRIM_ADD(words, ...)                                                                               \
    if constexpr (kIn && kOut) asm("add.cc.u32 %0, %0, 0xffffffff;\n\taddc" words "addc.u32 %0, 0, 0;" __VA_ARGS__); \
    else if constexpr (kIn) asm("add.cc.u32 %0, %0, 0xffffffff;\n\taddc" words __VA_ARGS__);               \
    else if constexpr (kOut) asm("add" words "addc.u32 %0, 0, 0;" __VA_ARGS__);                            \
    else asm("add" words __VA_ARGS__)
    if constexpr (N == 1) {
        GRIM_ADD(".cc.u32 %1, %1, %2;\n\t", : "+r"(carry), "+r"(s[0]) : "r"(p[0]));
    } else if constexpr (N == 2) {
        GRIM_ADD(".cc.u32 %1, %1, %3;\n\taddc.cc.u32 %2, %2, %4;\n\t",
                 : "+r"(carry), "+r"(s[0]), "+r"(s[1]) : "r"(p[0]), "r"(p[1]));
    } else if constexpr (N == 3) {
        GRIM_ADD(".cc.u32 %1, %1, %4;\n\taddc.cc.u32 %2, %2, %5;\n\taddc.cc.u32 %3, %3, %6;\n\t",
                 : "+r"(carry), "+r"(s[0]), "+r"(s[1]), "+r"(s[2]) : "r"(p[0]), "r"(p[1]), "r"(p[2]));
    } else {
        GRIM_ADD(".cc.u32 %1, %1, %9;\n\taddc.cc.u32 %2, %2, %10;\n\taddc.cc.u32 %3, %3, %11;\n\t"
                 "addc.cc.u32 %4, %4, %12;\n\taddc.cc.u32 %5, %5, %13;\n\taddc.cc.u32 %6, %6, %14;\n\t"
                 "addc.cc.u32 %7, %7, %15;\n\taddc.cc.u32 %8, %8, %16;\n\t",
                 : "+r"(carry), "+r"(s[0]), "+r"(s[1]), "+r"(s[2]), "+r"(s[3]), "+r"(s[4]), "+r"(s[5]), "+r"(s[6]),
                   "+r"(s[7])
                 : "r"(p[0]), "r"(p[1]), "r"(p[2]), "r"(p[3]), "r"(p[4]), "r"(p[5]), "r"(p[6]), "r"(p[7]));
    }
#undef GRIM_ADD
}

// Words of one addition at most.  Two operations a column pass the carry over
// each boundary, which hardly shows while the GPU is full (18 words, 1M
// locations: 2.07 ms in groups of 2 to 18); a call of few locations waits for
// each column's chain, and what that takes turns on the order the groups give
// the code.  500 locations, us, for groups of 2, 3, 6 and one statement a word
// whose carry the next one took from the condition code: 15 words 57.4, 63.5,
// 63.9, 58; 18 words 71.6, 67.6, 73.3, 67.6; 26 words -, 88, 82, 99; 32 words
// -, 113, 103 (8: 103), 108.
template <int W>
constexpr int kAddWords = W == 15 ? 2 : W == 8 || W == 32 ? 8 : 3;

// Up to this many words a column's masks are asked for while the one before is
// worked on: with few words the wait for them shows (spans of 178 bases, reads of
// 100-150, 500 / 100,000 locations: 38.9 / 117.9 us without, 31.6 / 95.9 so).
constexpr int kAheadWords = 8;

// Words of the next group when `left` are still to be added: groups as equal
// as they can be.
template <int W>
__host__ __device__ constexpr int add_group(int left) {
    const int groups = (left + kAddWords<W> - 1) / kAddWords<W>;
    return groups > 0 ? (left + groups - 1) / groups : 0;
}

// Words W0 .. W - 1 of one read base's step, a group at a time; e: the match
// masks of the first group.  The next group's are asked for before this one is
// worked on.
template <int W, int W0, int N, typename Eq>
__device__ __forceinline__ void rows_words(uint32_t (&Pv)[W], uint32_t (&Mv)[W], const uint32_t (&e)[N], Eq&& eq,
                                           uint32_t carry, uint32_t ph_below, uint32_t mh_below) {
    constexpr int kNext = add_group<W>(W - W0 - N);
    uint32_t e_next[kNext > 0 ? kNext : 1], s[N];
#pragma unroll
    for (int i = 0; i < kNext; i++) e_next[i] = eq(W0 + N + i);
#pragma unroll
    for (int i = 0; i < N; i++) s[i] = e[i] & Pv[W0 + i];
    add_words<N, (W0 > 0), (kNext > 0)>(s, Pv + W0, carry);
#pragma unroll
    for (int i = 0; i < N; i++) {
        const uint32_t pv = Pv[W0 + i], mv = Mv[W0 + i];
        const uint32_t xv = e[i] | mv;
        const uint32_t xh = (s[i] ^ pv) | e[i];
        const uint32_t ph = mv | ~(xh | pv);
        const uint32_t mh = pv & xh;
        const uint32_t phs = __funnelshift_l(ph_below, ph, 1);
        const uint32_t mhs = __funnelshift_l(mh_below, mh, 1);
        ph_below = ph;
        mh_below = mh;
        Pv[W0 + i] = mhs | ~(xv | phs);
        Mv[W0 + i] = phs & xv;
    }
    if constexpr (kNext > 0) rows_words<W, W0 + N>(Pv, Mv, e_next, eq, carry, ph_below, mh_below);
}

// One read base: Pv / Mv (rows whose vertical difference is +1 / -1) advance
// by a column.  eq(w): match mask of word w.
template <int W, typename Eq>
__device__ __forceinline__ void rows_step(uint32_t (&Pv)[W], uint32_t (&Mv)[W], Eq&& eq) {
    constexpr int kFirst = add_group<W>(W);
    uint32_t e[kFirst];
#pragma unroll
    for (int i = 0; i < kFirst; i++) e[i] = eq(i);
    rows_words<W, 0>(Pv, Mv, e, eq, 0u, 0x80000000u, 0u);  // D[0][j] - D[0][j-1] = +1
}

template <int W>
struct RowsSmem {
    uint32_t eq[4][W][kRowThreads];  // match masks per base code, one column per thread
    int16_t walk[256];               // four vertical differences (P nibble | M nibble << 4): min prefix << 8 | sum
    uint16_t order[kRowMaxTile];     // the tile's locations, longest reads first
    uint32_t count[64];              // by length class
    int next;                        // first chunk of `order` not yet taken
};

// Locations [tile * blockIdx.x, ...): `tile` of them per CTA.  SPANs of at
// most 32 W bases, reads of at most 64 kVerifyMaxBlocks.
template <int W>
__global__ void __launch_bounds__(kRowThreads)
verify_rows_kernel(const uint8_t* __restrict__ ref2bit, int64_t len, int64_t n_bins, int bin_len, int overlap,
                   const uint8_t* __restrict__ reads, const int64_t* __restrict__ read_offsets, int64_t n_reads,
                   const uint32_t* __restrict__ loc_read, const uint32_t* __restrict__ loc_bin, int64_t n_loc,
                   int tile, uint16_t* __restrict__ dist, uint32_t* __restrict__ status) {
    extern __shared__ __align__(16) uint8_t rows_smem_raw[];
    RowsSmem<W>& sm = *reinterpret_cast<RowsSmem<W>*>(rows_smem_raw);
    const int t = threadIdx.x, lane = t & 31;
    const int64_t i0 = (int64_t)blockIdx.x * tile;
    const int n = (int)(n_loc - i0 < tile ? n_loc - i0 : tile);
    if (t < 64) sm.count[t] = 0;
    if (t == 0) sm.next = 0;
    for (int x = t; x < 256; x += kRowThreads) {
        int d = 0, mn = 0;
        for (int k = 0; k < 4; k++) {
            d += ((x >> k) & 1) - ((x >> (4 + k)) & 1);
            mn = d < mn ? d : mn;
        }
        sm.walk[x] = (int16_t)((mn << 8) | (d & 0xFF));
    }
    __syncthreads();

    // the tile's locations by read length (64 classes of 8 bases, longest
    // first); one that cannot be scored is answered here
    uint32_t flags = 0;
    int cls[kRowMaxTile / kRowThreads];
#pragma unroll
    for (int k = 0; k < kRowMaxTile / kRowThreads; k++) {
        const int i = k * kRowThreads + t;
        cls[k] = -1;
        if (i >= n) continue;
        const uint32_t r = loc_read[i0 + i], b = loc_bin[i0 + i];
        int64_t L = -1;
        if ((int64_t)r < n_reads && (int64_t)b < n_bins) {
            const int64_t ro = read_offsets[r], re = read_offsets[r + 1];
            L = re >= ro ? re - ro : -1;
        }
        if (L < 0 || L > 64 * kVerifyMaxBlocks) {
            flags |= (int64_t)b >= n_bins ? GRIM_FLAG_BAD_BIN
                     : L > 64 * kVerifyMaxBlocks ? GRIM_FLAG_LONG_READ : GRIM_FLAG_BAD_OFFSETS;
            dist[i0 + i] = 0xFFFF;
            continue;
        }
        cls[k] = 63 - (int)(L > 0 ? (L - 1) >> 3 : 0);
        atomicAdd(&sm.count[cls[k]], 1u);
    }
    __syncthreads();
    if (t < 32) {  // counts -> first places
        const uint32_t c0 = sm.count[2 * lane], c1 = sm.count[2 * lane + 1];
        uint32_t x = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        sm.count[2 * lane] = x - c0 - c1;
        sm.count[2 * lane + 1] = x - c1;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRowMaxTile / kRowThreads; k++)
        if (cls[k] >= 0) sm.order[atomicAdd(&sm.count[cls[k]], 1u)] = (uint16_t)(k * kRowThreads + t);
    __syncthreads();
    const int n_ok = (int)sm.count[63];  // every place handed out

    const int64_t nbytes = (len + 3) >> 2;
    const bool aligned = ((uintptr_t)ref2bit & 3) == 0;
    while (true) {  // warps take 32 locations at a time
        int c = 0;
        if (lane == 0) c = atomicAdd(&sm.next, 32);
        c = __shfl_sync(kFull, c, 0);
        if (c >= n_ok) break;
        if (c + lane < n_ok) {
            const int64_t i = i0 + sm.order[c + lane];
            const uint32_t r = loc_read[i];
            const int64_t begin = (int64_t)loc_bin[i] * bin_len;
            const int64_t end = begin + bin_len + overlap < len ? begin + bin_len + overlap : len;
            const int S = (int)(end - begin);  // rows
            const int64_t ro = read_offsets[r];
            const int L = (int)(read_offsets[r + 1] - ro);

            // the span's match masks
            const int sh = 2 * (int)(begin & 15);
            const int64_t k0 = begin >> 4;
            uint32_t lo = packed_word(ref2bit, nbytes, aligned, k0);
#pragma unroll
            for (int w = 0; w < W; w++) {
                const uint32_t mid = packed_word(ref2bit, nbytes, aligned, k0 + 2 * w + 1);
                const uint32_t hi = packed_word(ref2bit, nbytes, aligned, k0 + 2 * w + 2);
                const uint32_t x0 = __funnelshift_r(lo, mid, sh), x1 = __funnelshift_r(mid, hi, sh);
                lo = hi;
                const uint32_t b0 = even_bits(x0) | (even_bits(x1) << 16);
                const uint32_t b1 = even_bits(x0 >> 1) | (even_bits(x1 >> 1) << 16);
                sm.eq[0][w][t] = ~(b0 | b1);
                sm.eq[1][w][t] = b0 & ~b1;
                sm.eq[2][w][t] = ~b0 & b1;
                sm.eq[3][w][t] = b0 & b1;
            }

            uint32_t Pv[W], Mv[W];
#pragma unroll
            for (int w = 0; w < W; w++) Pv[w] = Mv[w] = 0;  // D[i][0] = 0
            const uint8_t* rd = reads + ro;
            uint32_t next = L > 0 ? __ldg(rd) : 0u;
            if constexpr (W <= kAheadWords) {
                uint32_t e[W];  // the next column's masks
                auto ask = [&](uint32_t code) {
                    const uint32_t* eq = &sm.eq[code & 3u][0][t];
#pragma unroll
                    for (int w = 0; w < W; w++) e[w] = code <= 3u ? eq[w * kRowThreads] : 0u;  // others match nothing
                };
                ask(next);
                if (L > 1) next = __ldg(rd + 1);
                for (int j = 0; j < L; j++) {
                    uint32_t now[W];
#pragma unroll
                    for (int w = 0; w < W; w++) now[w] = e[w];
                    ask(next);
                    if (j + 2 < L) next = __ldg(rd + j + 2);
                    rows_step<W>(Pv, Mv, [&](int w) { return now[w]; });
                }
            } else {
                for (int j = 0; j < L; j++) {
                    const uint32_t code = next;
                    if (j + 1 < L) next = __ldg(rd + j + 1);
                    if (code <= 3u) {
                        const uint32_t* eq = &sm.eq[code][0][t];
                        rows_step<W>(Pv, Mv, [&](int w) { return eq[w * kRowThreads]; });
                    } else {
                        rows_step<W>(Pv, Mv, [](int) { return 0u; });  // matches nothing
                    }
                }
            }

            // minimum of D[0..S][L]: rows past the span only go up
            int cur = L, best = L;
#pragma unroll
            for (int w = 0; w < W; w++) {
                const int rows = S - 32 * w;
                const uint32_t in = rows >= 32 ? 0xFFFFFFFFu : rows <= 0 ? 0u : (1u << rows) - 1u;
                const uint32_t p = Pv[w] | ~in, m = Mv[w] & in;
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const uint32_t x = ((p >> (4 * q)) & 15u) | (((m >> (4 * q)) & 15u) << 4);
                    const int step = sm.walk[x];
                    const int low = cur + (step >> 8);
                    best = low < best ? low : best;
                    cur += (int)(int8_t)step;
                }
            }
            dist[i] = (uint16_t)best;  // <= L <= 512
        }
        __syncwarp();
    }
    flags = __reduce_or_sync(kFull, flags);
    if (lane == 0 && flags) atomicOr(status, flags);
}

// counts: [0] passing, [1] passing without a mapping (dist > E),
//         [2] rejected, [3] rejected with a mapping (a miss)
__global__ void verify_stats_kernel(const uint8_t* __restrict__ pass, const uint16_t* __restrict__ dist,
                                    const uint32_t* __restrict__ loc_read, const uint16_t* __restrict__ E,
                                    int64_t n_reads, int64_t n, unsigned long long* __restrict__ counts) {
    unsigned long long c[4] = {0, 0, 0, 0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = loc_read[i];
        const bool mapped = (int64_t)r < n_reads && dist[i] <= E[r];
        if (!pass || pass[i]) {
            c[0]++;
            c[1] += !mapped;
        } else {
            c[2]++;
            c[3] += mapped;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
        unsigned long long v = c[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&counts[k], v);
    }
}

struct VerifyArgs {
    const uint8_t* ref2bit;
    const uint8_t* reads;
    const int64_t* read_offsets;
    int64_t n_reads;
    const uint32_t* loc_read;
    const uint32_t* loc_bin;
    int64_t n_loc;
    uint16_t* dist;
};

template <int W>
int launch_verify_rows(const grim_bank* bank, const VerifyArgs& a, cudaStream_t s) {
    constexpr size_t smem = sizeof(RowsSmem<W>);
    static DeviceCache per_sm_of[64];  // per device, like the attribute
    const int slot = device_slot();
    if (slot < 0) return GRIM_ENOTSUP;
    if (per_sm_of[slot].load() == 0) {
        if (smem > 48 * 1024)
            GRIM_CUDA_TRY(cudaFuncSetAttribute(verify_rows_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem));
        int b = 0;
        GRIM_CUDA_TRY(
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, verify_rows_kernel<W>, kRowThreads, smem));
        per_sm_of[slot].store(b > 0 ? b : 1);
    }
    // the largest tile that still gives every resident CTA several: a larger
    // tile sorts better, more tiles leave a shorter last wave
    const int64_t want = 4 * (int64_t)sm_count() * per_sm_of[slot].load();
    int tile = kRowMaxTile;
    while (tile > kRowThreads && a.n_loc < want * tile) tile >>= 1;
    const int64_t blocks = (a.n_loc + tile - 1) / tile;
    if (blocks > 0x7fffffff) return GRIM_ENOTSUP;
    verify_rows_kernel<W><<<grim::fault_grid((unsigned)blocks), kRowThreads, smem, s>>>(
        a.ref2bit, bank->len, bank->n_bins, bank->bin_len, bank->overlap, a.reads, a.read_offsets, a.n_reads,
        a.loc_read, a.loc_bin, a.n_loc, tile, a.dist, bank->status);
    GRIM_CUDA_TRY(cudaGetLastError());
    return GRIM_OK;
}

}  // namespace
}  // namespace grim

extern "C" {

int grim_verify(const grim_bank* bank, const uint8_t* ref2bit, const uint8_t* reads, const int64_t* read_offsets,
                int64_t n_reads, const uint32_t* loc_read, const uint32_t* loc_bin, int64_t n_loc, uint16_t* dist,
                void* stream) {
    if (!bank || n_reads < 0 || n_loc < 0) return GRIM_EINVAL;
    if (n_loc == 0) return GRIM_OK;
    if (!ref2bit || !reads || !read_offsets || !loc_read || !loc_bin || !dist) return GRIM_EINVAL;
    int rc = grim::check_device(bank);
    if (rc != GRIM_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const grim::VerifyArgs a{ref2bit, reads, read_offsets, n_reads, loc_read, loc_bin, n_loc, dist};
    // the span as rows, W words of 32: spans of up to 1,024 bases (8 to 65 KB
    // of match masks per CTA; W rounded up to the next of a few sizes, at most
    // a quarter more work than the span needs above 256 bases); longer spans
    // the read as rows
    const int64_t words = ((int64_t)bank->bin_len + bank->overlap + 31) / 32;
    if (words <= 8) return grim::launch_verify_rows<8>(bank, a, s);
    if (words <= 10) return grim::launch_verify_rows<10>(bank, a, s);
    if (words <= 12) return grim::launch_verify_rows<12>(bank, a, s);
    if (words <= 13) return grim::launch_verify_rows<13>(bank, a, s);
    if (words <= 15) return grim::launch_verify_rows<15>(bank, a, s);
    if (words <= 18) return grim::launch_verify_rows<18>(bank, a, s);
    if (words <= 21) return grim::launch_verify_rows<21>(bank, a, s);
    if (words <= 26) return grim::launch_verify_rows<26>(bank, a, s);
    if (words <= 32) return grim::launch_verify_rows<32>(bank, a, s);
    const int64_t need = (n_loc + 255) / 256;
    const int64_t cap = (int64_t)grim::sm_count() * 16;
    const unsigned blocks = (unsigned)(need < cap ? need : cap);
    // reads of up to 128, 129-256 and 257-512 bases
    grim::verify_kernel<0, 2><<<grim::fault_grid(blocks), 256, 0, s>>>(
            ref2bit, bank->len, bank->n_bins, bank->bin_len, bank->overlap, reads, read_offsets, n_reads, loc_read,
            loc_bin, n_loc, dist, bank->status);
    grim::verify_kernel<3, 4><<<grim::fault_grid(blocks), 256, 0, s>>>(
            ref2bit, bank->len, bank->n_bins, bank->bin_len, bank->overlap, reads, read_offsets, n_reads, loc_read,
            loc_bin, n_loc, dist, bank->status);
    grim::verify_kernel<5, 8><<<grim::fault_grid(blocks), 256, 0, s>>>(
            ref2bit, bank->len, bank->n_bins, bank->bin_len, bank->overlap, reads, read_offsets, n_reads, loc_read,
            loc_bin, n_loc, dist, bank->status);
    GRIM_CUDA_TRY(cudaGetLastError());
    return GRIM_OK;
}

int grim_verify_stats(const uint8_t* pass, const uint16_t* dist, const uint32_t* loc_read, const uint16_t* E,
                      int64_t n_reads, int64_t n, unsigned long long* counts, void* stream) {
    if (n < 0 || n_reads < 0 || !counts) return GRIM_EINVAL;
    if (n > 0 && (!dist || !loc_read || !E)) return GRIM_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    GRIM_CUDA_TRY(cudaMemsetAsync(counts, 0, 4 * sizeof(unsigned long long), s));
    if (n == 0) return GRIM_OK;
    const int64_t need = (n + 255) / 256;
    const int64_t cap = (int64_t)grim::sm_count() * 8;
    grim::verify_stats_kernel<<<grim::fault_grid((unsigned)(need < cap ? need : cap)), 256, 0, s>>>(
            pass, dist, loc_read, E, n_reads, n, counts);
    GRIM_CUDA_TRY(cudaGetLastError());
    return GRIM_OK;
}

}  // extern "C"
