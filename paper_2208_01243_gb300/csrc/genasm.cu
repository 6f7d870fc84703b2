// GenASM (Section 2.4.3): windowed bit-parallel edit distance with a
// forward traceback, under a threshold of k edits.  One thread aligns one pair.
//
// Window.  At read position i and target position j a window holds
// wp = min(W, n-i) read bases and wt = min(W, m-j) target bases (W <= 64).  The
// read ends inside it when n-i <= W, the target when m-j <= W.  f(a, c) is the
// least number of edits of a path from (a, c) to the window's far edge; an edge
// whose sequence goes on past the window is free (cost 0 there), an edge whose
// sequence ends inside it charges one edit per base left on the other side.
//
// Difference vectors.  Neighbouring values of f differ by at most one, so a column t is held by the signs of its
// differences, one bit per read base (bit 0 the last read base of the window, bit wp-1 the first):
//   P, N   f(a, t) - f(a+1, t) is +1, is -1
//   H+, H- f(a, t) - f(a, t+1) is +1, is -1
//   Z      f(a, t) - f(a+1, t+1) is 0
// and one column follows from the next with a dozen word operations and one carry chain, whatever the distance
// (Myers, "A fast bit-vector algorithm for approximate string matching based on dynamic programming", 1999, over the
// reversed window).  With EQ the bits whose read base equals T[t] and h the difference along the empty read suffix (1 where
// the read ends in the window, 0 where its edge is free):
//   Z  = (((EQ & P) + P) ^ P) | EQ | N
//   H+ = N | ~(Z | P),   H- = P & Z
//   P' = (H- << 1) | ~(EQ | N | (H+ << 1 | h)),   N' = (H+ << 1 | h) & (EQ | N)
// (Z, in H+ and H-, without its last term, which changes neither).  The column past the window starts all +1 where the
// target ends in it, all 0 where its edge is free.  The window distance is f(wp, 0) plus the differences of column 0.
// A bitap's status vectors say the same level by level: [f <= d] for d up to the distance, eight words a column for
// windows of up to seven edits.  A window whose distance exceeds the edits left ends the pair: any way the alignment
// goes on crosses the window's far edge, so the count only grows.
//
// Traceback, forward from (0, 0): after an I, I first; after a D, D first; then M, X, I, D, each only when the rest
// still fits the window's distance.  The edits left always equal f(a, c), so an I fits where f(a, c) - f(a+1, c) is 1
// (P of column c), a D where f(a, c) - f(a, c+1) is 1 (H+ of column c), an X where f(a, c) - f(a+1, c+1) is not 0 (Z of
// column c; the bases differ), and a match always.  Match runs are taken with 32-base XOR compares.  A non-final window
// stops once W-O read or W-O target bases have been consumed in it; the final window runs to its corner.  So the three
// words are kept for the columns the traceback can reach, as the 32 bits from 16 below the diagonal position wp-1-t (or
// from bit 0): a path with d edits never strays more than d diagonals, and a window that turns out to need more than 14
// is computed again with whole words.
//
// Scratch per warp, lane-interleaved (32 lanes of a step store one contiguous row): W columns of three rows of 32 words.
//
// What bounds it: the integer pipe, 81-84 % busy, on the columns' word operations (150 bp at 5 %: 587 warp instructions
// a pair where status vectors level by level took 1,637).  1M pairs of 150 bp at 5 % in 0.82 ms (2.20 before), of 250 bp
// at 5 % in 1.30 (4.93), of 100 bp at 1 % in 0.45 (0.62); 200k of 1,000 bp at 5 % in 1.16 ms (5.31; 1.93 with whole
// words always kept, where the waits for them in the traceback led); 2,700 of 1,000 bp in 0.19 (0.58).
#include <algorithm>
#include <type_traits>

#include "aim_internal.cuh"

namespace aim {
namespace {

constexpr int kBandEdits = 14;         // widest window distance a 32-bit band serves

struct GenasmArgs {
    PairsView P;
    LimitView L;
    OutView O;
    uint8_t* scratch;
    size_t warp_bytes;              // stored columns of one warp
    int W, overlap;
    int64_t max_limit;              // the call's largest threshold, which a pair without one of its own gets
    uint32_t nwarps;
    uint32_t* counter;
};

constexpr uint32_t kNoOp = 0;

// The stored copy of a word of column t: the whole word, or the 32 bits from band_start(wp, t) up, which hold every bit
// the traceback can ask for (within 16 of the diagonal position wp-1-t, never below bit 0).
__device__ __forceinline__ int band_start(int wp, int t) { return max(wp - 17 - t, 0); }
template <typename Band>
__device__ __forceinline__ Band band_of(uint64_t v, int s);
template <>
__device__ __forceinline__ uint64_t band_of<uint64_t>(uint64_t v, int) { return v; }
template <>
__device__ __forceinline__ uint32_t band_of<uint32_t>(uint64_t v, int s) {   // bits s..s+31, s in [0, 47]
    const uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
    return s < 32 ? __funnelshift_r(lo, hi, (uint32_t)s) : (hi >> (s - 32));
}
// bit b of a stored copy whose band starts at bit s
__device__ __forceinline__ bool band_bit(uint64_t x, int b, int) { return (x >> b) & 1ull; }
__device__ __forceinline__ bool band_bit(uint32_t x, int b, int s) { return (x >> (b - s)) & 1u; }

// 32 even bits (bit 2s) of x -> bits s of the result
__device__ __forceinline__ uint32_t even_bits(uint64_t x) {
    x &= 0x5555555555555555ull;
    x = (x | (x >> 1)) & 0x3333333333333333ull;
    x = (x | (x >> 2)) & 0x0F0F0F0F0F0F0F0Full;
    x = (x | (x >> 4)) & 0x00FF00FF00FF00FFull;
    x = (x | (x >> 8)) & 0x0000FFFF0000FFFFull;
    x = (x | (x >> 16)) & 0x00000000FFFFFFFFull;
    return (uint32_t)x;
}

// one bit per base of a 32-base window word (first base in the top bits): 1 where the base is `code`
__device__ __forceinline__ uint32_t match_bits(uint64_t w, uint32_t code) {
    const uint64_t x = w ^ (0x5555555555555555ull * code);
    return even_bits(~(x | (x >> 1)));
}

// 32 bases from place p (0..63) of a window of two words
__device__ __forceinline__ uint64_t from_place(uint64_t w0, uint64_t w1, int p) {
    return p < 32 ? join_window(w0, w1, 2 * p) : w1 << (2 * (p - 32));
}

struct Window {
    uint64_t eq[4];     // read bases of the window, one mask per base code
    uint64_t r0, r1;    // read bases 0..31 and 32..63 of the window
    uint64_t t0, t1;    // target bases
    int wp, wt;
    int tmax;           // last column the traceback can read
    bool end_r, end_t;
};

// The window's distance; columns 0 .. tmax stored at lv (three words of 32 lanes each).
template <typename Band>
__device__ __forceinline__ int window_distance(const Window& w, Band* lv) {
    uint64_t P = w.end_t ? ~0ull : 0ull, N = 0ull;
    const uint64_t h = w.end_r ? 1ull : 0ull;
    auto column = [&](const int t, auto keep) {
        const uint64_t tword = t < 32 ? w.t0 : w.t1;
        const uint32_t code = (uint32_t)(tword >> (62 - 2 * (t & 31))) & 3u;
        const uint64_t e01 = (code & 1) ? w.eq[1] : w.eq[0], e23 = (code & 1) ? w.eq[3] : w.eq[2];
        const uint64_t eq = (code & 2) ? e23 : e01;
        const uint64_t z = (((eq & P) + P) ^ P) | eq;
        const uint64_t hp = N | ~(z | P), hn = P & z;
        const uint64_t x = eq | N, hs = (hp << 1) | h;
        const uint64_t zero = z | N;
        P = (hn << 1) | ~(x | hs);
        N = hs & x;
        if constexpr (decltype(keep)::value) {
            const int s = band_start(w.wp, t);
            Band* at = lv + (size_t)t * 96;
            at[0] = band_of<Band>(P, s);
            at[32] = band_of<Band>(hp, s);
            at[64] = band_of<Band>(zero, s);
        }
    };
    int t = w.wt - 1;
    for (; t > w.tmax; --t) column(t, std::false_type{});
    for (; t >= 0; --t) column(t, std::true_type{});
    const uint64_t rows = w.wp >= 64 ? ~0ull : (1ull << w.wp) - 1ull;
    return (w.end_r ? w.wt : 0) + __popcll(P & rows) - __popcll(N & rows);
}

// WIDE: some window may need more than kBandEdits edits: its columns are then computed again and kept whole
template <bool WIDE>
__global__ void __launch_bounds__(128) genasm_kernel(GenasmArgs a) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gwarp >= a.nwarps) return;
    const int W = a.W, stop = a.W - a.overlap;
    uint8_t* slot = a.scratch + (size_t)gwarp * a.warp_bytes;
    unsigned long long st_cells = 0, st_pairs = 0;

    for (;;) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(a.counter, 32u);
        base = __shfl_sync(kFull, base, 0);
        if (base >= a.P.num_pairs) break;
        const uint32_t pi = base + lane;
        if (pi >= a.P.num_pairs) continue;
        ++st_pairs;

        const uint32_t n = a.P.read_len[pi], m = a.P.target_len[pi];
        const int64_t k = min((long long)pair_limit(a.L, pi), (long long)a.max_limit);
        if (pair_bad(a.P, pi) || n > a.P.max_length || m > a.P.max_length || k == -2) {
            write_header(a.O, pi, -1, AIM_F_BAD_PAIR, 0);
            continue;
        }
        const uint64_t* rw = read_words(a.P, pi);
        const uint64_t* tw = target_words(a.P, pi);
        const uint32_t nrw = (n + 31) >> 5, ntw = (m + 31) >> 5;
        RunWriter out;
        uint32_t cap = 0;
        uint32_t* runs = nullptr;
        if (a.O.cigars && a.O.cigar_off) {
            const uint64_t off = a.O.cigar_off[pi];
            runs = a.O.cigars + off;
            cap = (uint32_t)(a.O.cigar_off[pi + 1] - off);
        }
        out.init(runs, cap);

        uint32_t i = 0, j = 0, prev = kNoOp;
        int64_t used = 0;
        bool rejected = false;
        while (i < n && j < m) {
            Window w;
            w.wp = (int)min(n - i, (uint32_t)W);
            w.wt = (int)min(m - j, (uint32_t)W);
            w.end_r = n - i <= (uint32_t)W;
            w.end_t = m - j <= (uint32_t)W;
            const bool fin = w.end_r && w.end_t;
            const int wp = w.wp, wt = w.wt;
            w.tmax = (fin ? wt : min(stop, wt)) - 1;
            // read window masks: bit wp-1-a is read base i+a
            w.r0 = window32(rw, nrw, i);
            w.r1 = window32(rw, nrw, i + 32);
#pragma unroll
            for (uint32_t c = 0; c < 4; ++c)
                w.eq[c] = (((uint64_t)match_bits(w.r0, c) << 32) | match_bits(w.r1, c)) >> (64 - wp);
            w.t0 = window32(tw, ntw, j);
            w.t1 = window32(tw, ntw, j + 32);

            const int64_t left = k - used;
            const int dist = window_distance<uint32_t>(w, reinterpret_cast<uint32_t*>(slot) + lane);
            const bool over = dist > left;
            // work of a bitap: levels 0..d (0..left when the window is over the budget) at every position
            st_cells += (unsigned long long)((over ? left : (int64_t)dist) + 1) * wt;
            if (over) { rejected = true; break; }

            // traceback
            int ta = 0, tc = 0;
            auto trace = [&](auto lv) {   // pointer to this lane's stored columns
                using Band = typename std::remove_pointer<decltype(lv)>::type;
                for (;;) {
                    if (!fin && (ta >= stop || tc >= stop)) break;
                    if (ta == wp && tc == wt) break;
                    uint32_t op;
                    int len = 1;
                    if (ta == wp) {
                        op = kOpDel;
                    } else if (tc == wt) {
                        op = kOpIns;
                    } else {
                        const Band* at = lv + (size_t)tc * 96;
                        const int b = wp - 1 - ta, from = sizeof(Band) == 4 ? band_start(wp, tc) : 0;
                        const bool fI = band_bit(at[0], b, from), fD = band_bit(at[32], b, from);
                        const bool fX = !band_bit(at[64], b, from);
                        // equal bases from here on, as far as 32 bases of the window's words show
                        const uint64_t x = from_place(w.r0, w.r1, ta) ^ from_place(w.t0, w.t1, tc);
                        const int same = __clzll((long long)x) >> 1;   // __clzll(0) = 64
                        if (prev == kOpIns && fI) op = kOpIns;
                        else if (prev == kOpDel && fD) op = kOpDel;
                        else if (same) {
                            op = kOpMatch;
                            int lim = min(wp - ta, wt - tc);
                            if (!fin) lim = min(lim, min(stop - ta, stop - tc));
                            len = min(same, lim);
                        } else if (fX) op = kOpMismatch;
                        else if (fI) op = kOpIns;
                        else op = kOpDel;
                    }
                    out.put(op, (uint32_t)len);
                    prev = op;
                    if (op != kOpMatch) ++used;
                    if (op == kOpMatch || op == kOpMismatch) { ta += len; tc += len; }
                    else if (op == kOpIns) ++ta;
                    else ++tc;
                }
            };
            if (WIDE && dist > kBandEdits) {
                uint64_t* whole = reinterpret_cast<uint64_t*>(slot) + lane;
                window_distance<uint64_t>(w, whole);
                trace(whole);
            } else {
                trace(reinterpret_cast<uint32_t*>(slot) + lane);
            }
            i += (uint32_t)ta;
            j += (uint32_t)tc;
            if (used > k) { rejected = true; break; }
        }
        if (!rejected) {
            // one sequence is used up: the rest of the other is one gap
            if (i < n) { out.put(kOpIns, n - i); used += n - i; }
            if (j < m) { out.put(kOpDel, m - j); used += m - j; }
            if (used > k) rejected = true;
        }
        if (rejected) {
            write_header(a.O, pi, -1, AIM_F_REJECTED, 0);
            continue;
        }
        out.finish();
        const uint8_t flags = (runs && out.n > cap) ? AIM_F_CIGAR_OVERFLOW : 0;
        write_header(a.O, pi, (int32_t)used, flags, out.n);
    }
    warp_stat_add(a.O.stats, 4, st_cells, lane);
    warp_stat_add(a.O.stats, 3, st_pairs, lane);
}

bool banded(int W, int64_t max_limit) { return (max_limit < W ? max_limit : W) <= kBandEdits; }

// a warp's stored columns
size_t column_bytes(int W, int64_t max_limit) {
    return align_up((size_t)W * 96 * (banded(W, max_limit) ? sizeof(uint32_t) : sizeof(uint64_t)), 256);
}

}  // namespace

// The scratch a call has to bring for one warp (the entry points' limit, kept from the form that stored a word per
// distance level: a row of W + 1 words, then levels in blocks of 4, or 8 where the threshold allows about two or more
// edits per window).  Never less than column_bytes.
size_t genasm_warp_bytes(int W, int64_t max_limit, uint32_t max_length) {
    const int64_t len = std::max<int64_t>(max_length, W), top = std::min<int64_t>(max_limit, W);
    const int block = max_limit >= 4 && max_limit * W >= 2 * len ? 8 : 4;
    const size_t levels = (size_t)((top + block) / block * block);
    const size_t word = banded(W, max_limit) ? sizeof(uint32_t) : sizeof(uint64_t);
    return align_up((size_t)(W + 1) * 32 * sizeof(uint64_t), 256) + align_up(levels * (W + 1) * 32 * word, 256);
}

cudaError_t launch_genasm(int W, int O, const PairsView& P, const LimitView& L, const OutView& Ov, int64_t max_limit,
                          uint8_t* scratch, size_t scratch_bytes, uint32_t* counter, int num_sms, cudaStream_t st,
                          int* warps_used) {
    *warps_used = 0;
    if (P.num_pairs == 0) return cudaSuccess;
    GenasmArgs a;
    a.P = P; a.L = L; a.O = Ov;
    a.W = W; a.overlap = O;
    a.max_limit = max_limit;
    a.counter = counter;
    a.warp_bytes = column_bytes(W, max_limit);
    // warp slots start on 256-byte boundaries so that every stored row is one aligned segment
    uint8_t* base = reinterpret_cast<uint8_t*>(align_up(reinterpret_cast<size_t>(scratch), 256));
    const size_t skip = (size_t)(base - scratch);
    if (skip >= scratch_bytes) return cudaSuccess;
    a.scratch = base;
    void (*kernel)(GenasmArgs) = banded(W, max_limit) ? genasm_kernel<false> : genasm_kernel<true>;
    int bps = 0;
    cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, 128, 0);
    if (err != cudaSuccess) return err;
    if (bps < 1) bps = 1;
    size_t warps = (size_t)num_sms * bps * 4;
    const size_t fit = (scratch_bytes - skip) / a.warp_bytes;
    if (warps > fit) warps = fit;
    const size_t need = ((size_t)P.num_pairs + 31) / 32;
    if (warps > need) warps = need;
    if (warps == 0) return cudaSuccess;
    a.nwarps = (uint32_t)warps;
    const unsigned blocks = (unsigned)((warps + 3) / 4);
    kernel<<<blocks, 128, 0, st>>>(a);
    *warps_used = (int)warps;
    return cudaGetLastError();
}

}  // namespace aim
