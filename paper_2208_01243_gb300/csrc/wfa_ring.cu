// Gap-affine wavefront alignment with the running state in shared memory: the form for thresholds whose wavefronts
// are narrow enough to hold a pair's last few wavefronts beside its sequences (see ring_ok).
//
// G lanes align one pair and a warp runs P = 32 / G pairs in lockstep, G = 1 being one pair per lane.  Lane
// l = gl * P + g is lane gl of pair g, and every per-pair array in shared memory is interleaved by pair (element j of
// pair g at [j * P + g]), so whatever the diagonal, the 32 lanes of an access touch 32 consecutive words.
//
// Scores are scaled as in wfa.cu (X, OE = O + E, and E == 1 here).  Instead of reading M~[s-OE] and I~[s-E] from
// stored wavefronts, the pass carries, per diagonal k,
//   mh[k]  M~[s-1..s-4, k], four 16-bit values in one 64-bit word that shifts by one value per score,
//   jd[k]  J = max(M~[s-O, k], I~[s, k]) and K = max(M~[s-O, k], D~[s, k]), two 16-bit values,
// so that   I~[s, k] = J[s-1, k+1],   D~[s, k] = K[s-1, k-1] + 1   and M~[s-X, k], M~[s-O, k] come out of mh by one
// byte permute each: three shared loads and two stores per entry, with no test against any wavefront's range.
// An invalid value is -1; a candidate is dropped when it would leave the matrix, as in wfa.cu.
//
// Ranges.  Row s covers the diagonals that can lie on an alignment within the limit S: at most s - O from diagonal
// 0, at most S - s from the end diagonal kend, and inside the window [kmin, kmax] outside which even a gap out and a
// gap back cost more than S (2 O + |k| + |k - kend| > S).  The ranges are arithmetic in s, so no per-score record is
// read or reduced.  Dropping the other diagonals changes no result: a value that would have come from outside lies on
// no alignment of cost <= S, and the traceback reads entries on optimal paths only.  Every pair walks its own row; the
// warp walks as many entries as its widest row.  The positions just outside a row read as invalid in the next one.
//
// History for the traceback, written 32 (or G) consecutive entries at a time.  Reads up to 1,022 bp: M~, I~ and D~,
// each + 1 in 10 bits of a word.  Longer ones: M~ + 1 and two source bits in 16 bits (up to 16,382 bp) or 32, set when
// J or K came from the extension (I~ > M~[s-O], D~ > M~[s-O]); the traceback follows them back to the gap's opening.
// Row s starts at a fixed distance from row s-1, or, for a longer read alone in its unit, where row s-1 ends, and the
// traceback computes where that is (RowMap).  A round of P pairs leaves its history in its unit's arena; after
// 32 pairs (or when the arena may not hold another round) a lane each traces them back, by the tests of wfa.cu.
//
// What bounds it: instruction issue at short reads.  150 bp at 6 edits take 931 warp instructions a pair, 22 of 32 lanes
// at work, 95 thread instructions for each of some 217 entries, at 2.2 per cycle (100k pairs; wfa.cu's 4-lane groups 1,790);
// 250 bp, band 25, 4 lanes, 9,480 at 2.8.  1M pairs of the first in 1.03 ms against 2.43 ms, of the second in 9.6 ms against
// 21.4 ms (all on one launch, packing apart).  Wide windows leave shared memory for few warps (10-13 % of an SM's at 16 and
// 32 lanes: 1.6-1.9 per cycle), and a block per pair waits at its barrier (4.0 of 7.8 stalls an issue at 5 kbp, 1.7).
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "ring_rows.h"
#include "wfa_common.cuh"

namespace aim {
namespace {

constexpr int kWarpsPerBlock = 4;
constexpr int kMhDepth = 4;               // scores of M~ held per diagonal
constexpr uint32_t kNarrowLength = 1022;  // longest read whose offsets + 1 fit 10 bits

struct RingArgs {
    WfaArgs w;
    uint32_t width;          // diagonals per pair in shared memory, two of them padding
    uint32_t seq_words;      // 32-bit words per sequence in shared memory
    uint32_t seq_rounds;     // rounds whose copies are kept: G, or 1 and the traceback reads the packed sequences
    uint32_t smem_warp;      // bytes of shared memory per warp
    uint32_t stage_shared;   // runs are staged in shared memory
    uint32_t sel_x, sel_o;   // byte permute selectors of M~[s-X], M~[s-O] in mh
};

// history forms
enum : int { kWhole = 0, kBits16 = 1, kBits32 = 2 };
template <int FMT>
struct Entry {   // kBits16, kBits32
    using T = typename std::conditional<FMT == kBits16, uint16_t, uint32_t>::type;
    static constexpr int kBits = FMT == kBits16 ? 14 : 30;
    static __device__ __forceinline__ T make(int m, int i, int d, int mo) {
        return (T)((uint32_t)(m + 1) | ((uint32_t)(i > mo) << kBits) | ((uint32_t)(d > mo) << (kBits + 1)));
    }
    static __device__ __forceinline__ T none() { return 0; }
    static __device__ __forceinline__ int m(T e) { return (int)((uint32_t)e & ((1u << kBits) - 1)) - 1; }
    static __device__ __forceinline__ bool from_ins(T e) { return ((uint32_t)e >> kBits) & 1u; }
    static __device__ __forceinline__ bool from_del(T e) { return ((uint32_t)e >> (kBits + 1)) & 1u; }
};
template <>
struct Entry<kWhole> {
    using T = uint32_t;
    static constexpr uint32_t kBias = 1u | (1u << 10) | (1u << 20);
    static __device__ __forceinline__ T make(int m, int i, int d, int) {
        return (uint32_t)m + ((uint32_t)i << 10) + ((uint32_t)d << 20);   // each value + 1 once kBias is added
    }
    static __device__ __forceinline__ T none() { return 0u - kBias; }
    static __device__ __forceinline__ int m(T e) { return (int)((e + kBias) & 1023u) - 1; }
    static __device__ __forceinline__ int i(T e) { return (int)(((e + kBias) >> 10) & 1023u) - 1; }
    static __device__ __forceinline__ int d(T e) { return (int)((e + kBias) >> 20) - 1; }
    static __device__ __forceinline__ bool from_ins(T) { return false; }
    static __device__ __forceinline__ bool from_del(T) { return false; }
};

// What the traceback of a lane's pair needs.
struct Pending {
    uint32_t pi;
    int final_s;             // < 0: none
    int koff, last, S;       // its Window
    uint32_t base, stride;   // its round's history: 256-byte units from the arena's rounds, entries per row
    int round;
};

// Where entry (c, j) of a finished pair lies: row c at c * stride, or, with kDense, rows end to end.
template <int P, bool kDense>
struct RowMap {
    Window w;
    int O;
    uint32_t stride;
    DenseRows dense;
    __device__ __forceinline__ RowMap(const Window& win, int o, uint32_t st) : w(win), O(o), stride(st), dense(win, o) {}
    __device__ __forceinline__ uint32_t start(int c) const {
        if constexpr (kDense) return dense.start(c);
        return (uint32_t)c * stride;
    }
    template <typename H>
    __device__ __forceinline__ typename H::T get(const typename H::T* hist, int c, int j) const {
        const int lo = w.lo(c, O);
        if (c < 0 || j < lo || j > w.hi(c, O)) return H::none();
        return hist[(size_t)start(c) + (uint32_t)((j - lo) * P)];
    }
};

template <int P, int FMT>
constexpr bool kDenseRows = P == 1 && FMT != kWhole;

// Canonical traceback of one finished pair by one lane (the tests of wfa.cu's traceback).  Every step issues its loads
// at once: the entries of its tests and both sequences' windows ending at (v, h), whose XOR gives the match run.
// seqs_kept: the pair's copies in shared memory (words [i * P]); otherwise the packed sequences are read.
template <int P, int FMT>
__device__ uint32_t ring_traceback(const WfaArgs& a, const uint8_t* rounds, const Pending& q, int g, bool seqs_kept,
                                   const uint32_t* sp, const uint32_t* st, RunStage& wr, bool& ok) {
    using H = Entry<FMT>;
    const typename H::T* hist = reinterpret_cast<const typename H::T*>(rounds + ((size_t)q.base << 8)) + g;
    const int n = (int)a.P.read_len[q.pi], m = (int)a.P.target_len[q.pi];
    const uint64_t* Pg = read_words(a.P, q.pi);
    const uint64_t* Tg = target_words(a.P, q.pi);
    const uint32_t nwP = (uint32_t)(n + 31) >> 5, nwT = (uint32_t)(m + 31) >> 5;
    const int X = a.X, OE = a.OE, O = OE - 1;
    const RowMap<P, kDenseRows<P, FMT>> rows(Window{q.koff, q.last, -q.koff, m - n - q.koff, q.S}, O, q.stride);
    auto entry = [&](int c, int j) { return rows.template get<H>(hist, c, j); };
    // source-bit forms: I~[c, j] from the bit of (c-1, j+1) and M~ of (c-OE, j+1), loaded together, or further back
    // along the gap; D~ likewise
    auto ins_of = [&](int c, int j, typename H::T src, typename H::T opening) -> int {
        const int hmax = min(m, n + j + q.koff);
        for (int guard = n + m; H::from_ins(src) && guard > 0; --guard) {
            --c; ++j;
            src = entry(c - 1, j + 1);
            opening = entry(c - OE, j + 1);
        }
        const int at = H::m(opening);
        return at <= hmax ? at : -1;
    };
    auto del_of = [&](int c, int j, typename H::T src, typename H::T opening) -> int {
        const int hmax = min(m, n + j + q.koff);
        int more = 1;
        for (int guard = n + m; H::from_del(src) && guard > 0; --guard) {
            --c; --j; ++more;
            src = entry(c - 1, j - 1);
            opening = entry(c - OE, j - 1);
        }
        const int at = H::m(opening);
        return at >= 0 && at + more <= hmax ? at + more : -1;
    };
    // matching bases back from (v, h), as far as one window shows
    auto match_back = [&](int v, int h) -> int {
        if (seqs_kept) {   // 16 bases back; before the start the window's earlier bases are not looked at
            const int back = min(min(v, h), 16);
            const uint32_t x = window16<P>(sp, max(v - 16, 0)) >> (v < 16 ? 2 * (16 - v) & 31 : 0);
            const uint32_t y = window16<P>(st, max(h - 16, 0)) >> (h < 16 ? 2 * (16 - h) & 31 : 0);
            const uint32_t d = x ^ y;
            return min(d ? (__ffs((int)d) - 1) >> 1 : 16, back);
        }
        const int back = min(min(v, h), 32);
        const uint64_t d = back ? window_ending(Pg, nwP, v - 1) ^ window_ending(Tg, nwT, h - 1) : 1ull;
        return min(d ? (__ffsll((long long)d) - 1) >> 1 : 32, back);
    };
    int v = n, h = m, cM = q.final_s, cI = q.final_s, cD = q.final_s;
    while ((v > 0 || h > 0) && ok) {
        const int j = h - v - q.koff;
        const auto eX = entry(cM - X, j), eM = entry(cM, j);
        typename H::T eI, eD, oI, oD;
        if constexpr (FMT == kWhole) {
            eI = entry(cI, j); eD = entry(cD, j);
        } else {
            eI = entry(cI - 1, j + 1); oI = entry(cI - OE, j + 1);
            eD = entry(cD - 1, j - 1); oD = entry(cD - OE, j - 1);
        }
        int same = match_back(v, h);
        const int mX = H::m(eX), mM = H::m(eM);
        int vI, vD;
        if constexpr (FMT == kWhole) { vI = H::i(eI); vD = H::d(eD); }
        else { vI = ins_of(cI, j, eI, oI); vD = del_of(cD, j, eD, oD); }
        // A run of matches leaves the diagonal and the score, and so the entries, as they are: the edit before it is
        // decided from the same loads.
        for (;;) {
            const bool diag = v > 0 && h > 0, match = same > 0;
            if (diag && !match && mX >= h - 1) {
                cM = cI = cD = cM - X; --v; --h;
                wr.put(kOpMismatch, 1);
                break;
            }
            if (v > 0 && vI >= h) {
                const int c = cI;
                cM = cD = c - OE; cI = c - 1; --v;
                wr.put(kOpIns, 1);
                break;
            }
            if (h > 0 && vD >= h) {
                const int c = cD;
                cM = cI = c - OE; cD = c - 1; --h;
                wr.put(kOpDel, 1);
                break;
            }
            if (!match || mM < h - 1) { ok = false; break; }
            if (cI != cM || cD != cM) {   // I~ and D~ of M~'s own score from here on
                if constexpr (FMT == kWhole) { vI = H::i(eM); vD = H::d(eM); }
                else {
                    if (cI != cM) vI = ins_of(cM, j, entry(cM - 1, j + 1), entry(cM - OE, j + 1));
                    if (cD != cM) vD = del_of(cM, j, entry(cM - 1, j - 1), entry(cM - OE, j - 1));
                }
                cI = cD = cM;
            }
            // to where a gap may end or the window does: a longer run is taken window by window
            const int run = min(same, h - max(vI, vD));
            if (run < 1) { ok = false; break; }
            v -= run; h -= run;
            wr.put(kOpMatch, (uint32_t)run);
            if (v == 0 && h == 0) break;
            same = match_back(v, h);
        }
    }
    wr.flush();
    ok = ok && wr.n <= wr.cap;
    return wr.n;
}

extern __shared__ __align__(16) uint8_t s_ring[];

// threads of a block: four warps on their own, or, for G > 32, one group of G threads on one pair
template <int G>
constexpr int kBlockThreads = G > 32 ? G : 32 * kWarpsPerBlock;

template <int G, int FMT>
__global__ void __launch_bounds__(kBlockThreads<G>) wfa_ring_kernel(RingArgs r) {
    using E = typename Entry<FMT>::T;
    constexpr bool kBlock = G > 32;
    constexpr int P = kBlock ? 1 : 32 / G;
    constexpr bool kDense = kDenseRows<P, FMT>;
    constexpr int kRounds = 32 / P;          // rounds of P pairs until 32 tracebacks are due
    constexpr int kRows = G == 1 ? 1 : 2;   // jd rows: one lane per pair updates its row in place
    const WfaArgs& a = r.w;
    // lane of the unit (a warp, or the block), this thread's pair and its place among the pair's lanes
    const int lane = kBlock ? (int)threadIdx.x : (int)(threadIdx.x & 31);
    const int g = lane % P, gl = lane / P;
    const uint32_t unit = kBlock ? blockIdx.x : (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (unit >= a.nwarps) return;
    auto sync = [] {
        if constexpr (kBlock) __syncthreads();
        else __syncwarp();
    };
    const uint32_t W = r.width;
    uint8_t* sm = s_ring + (kBlock ? 0 : (size_t)(threadIdx.x >> 5) * r.smem_warp);
    uint2* mh = reinterpret_cast<uint2*>(sm);                            // [W][P]
    uint32_t* jd = reinterpret_cast<uint32_t*>(sm + (size_t)W * P * 8);  // [kRows][W][P]
    // copies of a round's reads, then of its targets, [seq_words][P] each; of every round awaiting its traceback
    // when seq_rounds says so
    uint32_t* seq = jd + (size_t)kRows * W * P;
    const uint32_t seq_round = 2 * r.seq_words * P;
    const bool seqs_kept = r.seq_rounds == (uint32_t)kRounds;
    uint8_t* arena = a.scratch + (size_t)unit * a.warp_bytes;
    uint8_t* rounds = arena + 32 * a.runs_bytes;
    const size_t rounds_bytes = a.warp_bytes - 32 * a.runs_bytes;
    const int O = a.OE - 1;
    const uint32_t begin = a.bounds ? a.bounds[0] : 0;
    const uint32_t end = a.bounds ? a.bounds[1] : a.P.num_pairs;
    unsigned long long st_cells = 0, st_windows = 0;
    uint32_t st_pairs = 0;

    __shared__ int s_end[2];
    Pending pend{0, -1, 0, 0, 0, 0, 0, 0};
    int round = 0;
    size_t used = 0;   // arena bytes of the rounds awaiting their traceback
    // the lane that traces pair g of round i: 32 in a warp, spread over the warps of a block
    auto tracer = [&](int i) { return kBlock ? (i % (G / 32)) * 32 + i / (G / 32) : i * P + g; };
    auto finish = [&]() {
        sync();
        // runs staged where the forward pass kept its state, lane l's i-th run at [33 i + l], or in the arena
        const int slot = kBlock ? pend.round : lane;
        uint32_t* stage = r.stage_shared ? reinterpret_cast<uint32_t*>(sm) + slot
                                         : reinterpret_cast<uint32_t*>(arena + (size_t)slot * a.runs_bytes);
        RunStage wr{stage, r.stage_shared ? 33u : 1u, a.runs_cap, 0, 0, 0};
        bool ok = pend.final_s >= 0;
        uint64_t off = 0;
        uint32_t copy = 0;
        if (ok) {
            const uint32_t* sp = seq + (seqs_kept ? (uint32_t)pend.round * seq_round : 0u) + g;
            const uint32_t nruns = ring_traceback<P, FMT>(a, rounds, pend, g, seqs_kept, sp, sp + r.seq_words * P, wr, ok);
            uint8_t flags = ok ? 0 : AIM_F_STEP_CAP;
            if (ok && a.O.cigars) {
                off = a.O.cigar_off[pend.pi];
                if (nruns <= a.O.cigar_off[pend.pi + 1] - off) copy = nruns;
                else flags = AIM_F_CIGAR_OVERFLOW;
            }
            write_header(a.O, pend.pi, ok ? pend.final_s * a.g : -1, flags, nruns);
        }
        __syncwarp();
        if (a.O.cigars)
            copy_runs(a.O, copy, off,
                      r.stage_shared ? reinterpret_cast<const uint32_t*>(sm) : reinterpret_cast<const uint32_t*>(arena),
                      r.stage_shared ? 1u : (uint32_t)(a.runs_bytes / 4), r.stage_shared ? 33u : 1u, slot);
        sync();
        pend.final_s = -1;
        round = 0;
        used = 0;
    };

    for (;;) {
        uint32_t pos = 0;
        if constexpr (kBlock) {
            __shared__ uint32_t s_pos;
            if (lane == 0) s_pos = atomicAdd(a.counters, 1u);
            __syncthreads();
            pos = s_pos;
            __syncthreads();
        } else {
            if (lane == 0) pos = atomicAdd(a.counters, (uint32_t)P);
            pos = __shfl_sync(kFull, pos, 0);
        }
        if (pos >= end - begin || end <= begin) break;

        // ---- the round's pairs
        const uint32_t q = begin + pos + (uint32_t)g;
        int status = kIdle, n = 0, m = 0, S = 0, kend = 0;
        uint32_t pi = 0;
        if (q < end) {
            pi = a.order ? a.order[q] : q;
            n = (int)a.P.read_len[pi];
            m = (int)a.P.target_len[pi];
            kend = m - n;
            const int64_t lim = pair_limit(a.L, pi);
            if (gl == 0) ++st_pairs;
            if (pair_bad(a.P, pi) || (uint32_t)n > a.P.max_length || (uint32_t)m > a.P.max_length || lim == -2) {
                status = kBad;
            } else {
                const int64_t S64 = lim / a.g;
                S = (int)(S64 > a.smax ? a.smax : S64);
                if (a.bound) {   // a bound pass found an alignment of this score: the optimum is at most that
                    const int ub = a.bound[pi];
                    if (ub >= 0 && ub < S) S = ub;
                }
                // rejected at once: the end diagonal outside the band, or its gap alone above the limit
                const bool far = a.band >= 0 && (kend > a.band || -kend > a.band);
                status = far || S < 0 || (kend != 0 && abs(kend) + O > S) ? kRejected : kRun;
            }
        }
        bool run = status == kRun;
        Window win{0, 0, 0, 0, S};
        if (run) {
            const int right = reach(kend, m, S, O, a.band), left = reach(-kend, n, S, O, a.band);
            win = Window{-left - 1, left + right + 1, left + 1, kend + left + 1, S};
        }
        const int wide = P == 1 ? win.last : __reduce_max_sync(kFull, win.last);   // 0: no pair to run
        // entry (s, t-th of its row) of the history at [s * stride + t * P]
        const uint32_t stride = ((uint32_t)wide * P + 31u) & ~31u;
        // what rows 0 .. S take, from the pairs' own limits and windows: the arena holds more rounds than of the worst case
        size_t need = 0;
        if constexpr (kDense) {
            if (run) need = (size_t)DenseRows(win, O).start(S + 1) * sizeof(E);
        } else {
            const int rows = P == 1 ? S : __reduce_max_sync(kFull, run ? S : 0);
            if (wide) need = (size_t)(rows + 1) * stride * sizeof(E);
        }
        if (round == kRounds || rounds_bytes - used < need) finish();
        int final_s = -1, s = 0;
        uint32_t entries = 0;   // of the round's history
        if (wide) {
            uint32_t* dp = seq + (seqs_kept ? (uint32_t)round * seq_round : 0u) + g;
            uint32_t* dt = dp + r.seq_words * P;
            const uint32_t* sp = dp;
            const uint32_t* st = dt;
            // nothing is reachable yet
            for (int i = lane; i < (wide + 2) * P; i += kBlock ? G : 32) {
                mh[i] = make_uint2(~0u, ~0u);
                jd[i] = ~0u;
                if (kRows == 2) jd[i + W * P] = ~0u;
            }
            if (run) {
                const uint64_t* Pw = read_words(a.P, pi);
                const uint64_t* Tw = target_words(a.P, pi);
                for (int w = gl; w < (n + 31) >> 5; w += G) {
                    const uint64_t x = __ldg(Pw + w);
                    dp[2 * w * P] = (uint32_t)(x >> 32); dp[(2 * w + 1) * P] = (uint32_t)x;
                }
                for (int w = gl; w < (m + 31) >> 5; w += G) {
                    const uint64_t x = __ldg(Tw + w);
                    dt[2 * w * P] = (uint32_t)(x >> 32); dt[(2 * w + 1) * P] = (uint32_t)x;
                }
            }
            sync();
            uint32_t cells = 0, windows = 0;
            E* hrow = reinterpret_cast<E*>(rounds + used) + lane;   // row s, this lane's first entry
            uint32_t filled = 1;                                    // kDense: entries of the rows so far
            // row 0: diagonal 0 from offset 0
            if (run && gl == 0) {
                const int m0 = match_on<P>(sp, st, 0, 0, min(n, m));
                mh[win.zero * P + g] = make_uint2((uint32_t)m0 | 0xffff0000u, ~0u);
                hrow[0] = Entry<FMT>::make(m0, -1, -1, -1);
                if constexpr (kBlock) s_end[0] = win.zero == win.end ? m0 : -1;
                ++cells; ++windows;
            }
            for (;;) {
                // the row just computed ends the pair if it reaches the end of the end diagonal
                if (G > 1) sync();
                int reached;   // M~ on the end diagonal
                if constexpr (kBlock) reached = s_end[s & 1];
                else reached = (int)(mh[win.end * P + g].x & 0xffffu);
                if (G == 32) __syncwarp();   // every lane has read it before the next row is written (P > 1: the vote below)
                if (run && reached == m) { status = kDone; final_s = s; run = false; }
                ++s;
                if (run && s > S) { status = kRejected; run = false; }
                if (P == 1 ? !run : !__any_sync(kFull, run)) break;
                const int jlo = win.lo(s, O), jhi = win.hi(s, O);
                const int w = run ? max(jhi - jlo + 1, 0) : 0;
                const int rows = P == 1 ? w : __reduce_max_sync(kFull, w);
                if constexpr (kDense) {
                    hrow = reinterpret_cast<E*>(rounds + used) + filled + lane;
                    filled += (uint32_t)w;
                } else {
                    hrow += stride;
                }
                const uint32_t odd = (uint32_t)(s & 1);
                const uint32_t at = (uint32_t)(jlo * P + g);       // the row's first position
                uint2* mhr = mh + at;
                uint32_t* jw = (kRows == 2 ? jd + odd * (W * P) : jd) + at;                // this row
                const uint32_t* jr = (kRows == 2 ? jd + (odd ^ 1u) * (W * P) : jd) + at;   // row s-1
                const int kb = jlo + win.koff;                     // the row's first diagonal
                uint32_t before = 0, here = 0;   // G == 1: jd of positions j-1 and j in row s-1
                // U entries of every lane at a time: the loads and the first 16 bases of each overlap
                auto step = [&](const int tb, auto count) {
                    constexpr int U = decltype(count)::value;
                    int mv[U], ins[U], del[U], mo[U], hmax[U];
                    uint32_t x[U];
                    uint2 h4[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int t = min(tb + u * G + (G > 1 ? gl : 0), w - 1);   // a lane past its row repeats the last
                        uint32_t left, right;
                        if (G == 1) {
                            left = before;
                            right = jr[(t + 1) * P];
                            before = here;
                            here = right;
                        } else {
                            left = jr[(t - 1) * P]; right = jr[(t + 1) * P];
                        }
                        h4[u] = mhr[t * P];
                        const int k = kb + t;
                        hmax[u] = min(m, n + k);   // >= 0 inside the window
                        mo[u] = prmt(h4[u].x, h4[u].y, r.sel_o);
                        int mis = prmt(h4[u].x, h4[u].y, r.sel_x);
                        ins[u] = prmt(right, 0u, 0x9910u);
                        del[u] = prmt(left, 0u, 0xbb32u);
                        mis = (unsigned)mis < (unsigned)hmax[u] ? mis + 1 : -1;
                        del[u] = (unsigned)del[u] < (unsigned)hmax[u] ? del[u] + 1 : -1;
                        ins[u] = ins[u] <= hmax[u] ? ins[u] : -1;   // (an invalid -1 stays)
                        mv[u] = max(mis, max(ins[u], del[u]));
                        // an invalid entry reads words before its copies, inside the warp's shared memory, and
                        // matches nothing
                        x[u] = (window16<P>(sp, mv[u] - k) ^ window16<P>(st, mv[u])) | (uint32_t)(mv[u] >> 31);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int t = tb + u * G + (G > 1 ? gl : 0);
                        const int rem = hmax[u] - mv[u];   // bases left on both sequences
                        int len = min(__clz((int)x[u]) >> 1, rem);
                        if (t < w) windows += 1 + (mv[u] >> 31);
                        if (x[u] == 0 && rem > 16) {
                            len = 16 + match_on<P>(sp, st, mv[u] - kb - min(t, w - 1) + 16, mv[u] + 16, rem - 16);
                            if (t < w) windows += (uint32_t)len >> 5;
                        }
                        mv[u] += len;
                        if (t < w) {
                            mhr[t * P] =
                                make_uint2((uint32_t)prmt((uint32_t)mv[u], h4[u].x, 0x5410u),
                                           (uint32_t)prmt(h4[u].x, h4[u].y, 0x5432u));
                            jw[t * P] = (uint32_t)prmt((uint32_t)max(mo[u], ins[u]), (uint32_t)max(mo[u], del[u]), 0x5410u);
                            hrow[(tb + u * G) * P] = Entry<FMT>::make(mv[u], ins[u], del[u], mo[u]);
                        }
                    }
                };
                if (w > 0) {   // lanes whose pair has ended have no row
                    if (G == 1) { before = jr[-P]; here = jr[0]; }
                    int t = 0;
                    for (; t + G < rows; t += 2 * G) step(t, std::integral_constant<int, 2>{});
                    if (t < rows) step(t, std::integral_constant<int, 1>{});
                }
                if constexpr (kBlock) {   // the end diagonal's M~ for the check above, in a place of the row's parity
                    const int te = win.end - jlo;
                    const bool in_row = te >= 0 && te < w;
                    if (gl == (in_row ? te % G : 0)) s_end[odd] = in_row ? (int)(mhr[te].x & 0xffffu) : -1;
                }
                if (gl == 0 && w > 0) {   // just outside the row: invalid
                    jw[-P] = ~0u;
                    jw[w * P] = ~0u;
                    cells += (uint32_t)w;
                }
            }
            st_cells += cells;
            st_windows += windows;
            entries = kDense ? filled : (uint32_t)s * stride;
        }
        if (gl == 0 && (status == kRejected || status == kBad)) emit_failed(a, pi, status);
        // the pair's tracer takes what it needs (P == 1: every lane has it)
        if constexpr (P == 1) {
            if (lane == tracer(round))
                pend = Pending{pi, final_s, win.koff, win.last, S, (uint32_t)(used >> 8), stride, round};
        } else {
            const int src = lane % P;
            const uint32_t p_pi = __shfl_sync(kFull, pi, src);
            const int p_s = __shfl_sync(kFull, final_s, src), p_koff = __shfl_sync(kFull, win.koff, src);
            const int p_last = __shfl_sync(kFull, win.last, src), p_S = __shfl_sync(kFull, S, src);
            if (lane == tracer(round)) pend = Pending{p_pi, p_s, p_koff, p_last, p_S, (uint32_t)(used >> 8), stride, round};
        }
        if (wide && (P > 1 || final_s >= 0)) {   // (a single pair that was rejected leaves nothing to trace)
            used += ((size_t)entries * sizeof(E) + 255) & ~(size_t)255;
            ++round;
        }
    }
    finish();
    const uint32_t wl = threadIdx.x & 31;
    warp_stat_add(a.O.stats, 0, st_cells, wl);
    warp_stat_add(a.O.stats, 1, st_windows, wl);
    warp_stat_add(a.O.stats, 3, st_pairs, wl);
}

template <int FMT>
void (*ring_kernel_for(int G))(RingArgs) {
    switch (G) {
        case 1: return wfa_ring_kernel<1, FMT>;
        case 2: return wfa_ring_kernel<2, FMT>;
        case 4: return wfa_ring_kernel<4, FMT>;
        case 8: return wfa_ring_kernel<8, FMT>;
        case 16: return wfa_ring_kernel<16, FMT>;
        case 32: return wfa_ring_kernel<32, FMT>;
        default: return wfa_ring_kernel<256, FMT>;
    }
}

// Lanes per pair: the fewest whose warps fit an SM at least 16 at a time (14 KB of shared memory each), since one lane
// per pair wastes no lane on a row's end and shares a row's fixed work between the most pairs; more when the batch, or
// the pairs that the scratch holds at once, would otherwise give the device less than 8 warps per SM, where the pair's
// own serial chain is what counts, up to the lanes that the widest row gives work to (1,270 pairs, 2 edits: 18.0 us with 8
// lanes, 18.1 with 32).
// Measured, ms at 1 / 2 / 4 / 8 / 16 lanes: 1M x 150 bp, 6 edits (12 KB at 1 lane) 1.15 / 1.24 / 1.50 / 1.99 / 2.89;
// 1M x 250 bp, 25 edits, band 25 (12 KB at 4) 13.4 / 10.7 / 9.8 / 10.4 / 12.8; 300k x 300 bp, 30 edits (11 KB at 8)
// 12.6 / 12.2 / 5.7 / 4.6 / 4.9; 10k x 150 bp 0.080 / 0.067 / 0.060 / 0.064 / 0.073; 61 x 150 bp 0.072 / 0.056 /
// 0.045 / 0.039 / 0.037.
constexpr size_t kGoodSmem = 14u << 10;
// Short of scratch, ms at 8 / 16 / 32 / 256 lanes: 10k x 1,000 bp, 50 edits, 16 MB 25.0 / 16.9 / 11.8 / 9.1, 256 MB 1.79 /
// 1.25 / 0.92 / 1.54, 1 GB 0.71 / 0.59 / 0.57 / 1.40; at 32 / 256: 500 x 5 kbp, 250 edits, 64 MB 12.4 / 6.5, 1 GB 1.55 / 1.26;
// 5,000 of them, 1 GB 8.9 / 8.3, 2 GB 6.4 / 7.7.  (wfa.cu: 500 x 5 kbp, 64 MB, 11.1; the rule had taken 32 there.)  A batch
// plan's classes run side by side and share scratch and device, so there the scratch has no say.
constexpr int kGoodWarps = 8;
constexpr int kThinWarps = 4;              // a block per pair below so many warps an SM for want of scratch
constexpr int64_t kBlockWidth = 128;       // narrower rows leave half a block without work
constexpr size_t kBlockSmem = 20u << 10;   // a whole block per pair where a warp's state takes more
constexpr size_t kMaxSmem = 226u << 10;   // dynamic shared memory a block may use (227 KB, less its static few bytes)
constexpr size_t kPlainSmem = 47u << 10;  // ... and without asking for it (48 KB, less the same)

int entry_form(uint32_t max_length) {
    return max_length <= kNarrowLength ? kWhole : max_length <= kMaxWfaLength16c ? kBits16 : kBits32;
}
size_t entry_bytes(uint32_t max_length) { return entry_form(max_length) == kBits16 ? 2 : 4; }

// pairs of a warp, or 1 where a block works on one
size_t pairs_of(int G) { return G > 32 ? 1 : 32 / G; }

// diagonals per pair: the widest window (2 O + 2 k - kend <= S on both sides, or just 0 .. kend: S - O + 1), the
// band's or the matrix's, or what the caller knows of its pairs, and the two padding positions
int64_t ring_width(const WfaPlan& p, uint32_t max_length) {
    const int64_t O = p.oe - p.e;
    int64_t w = p.smax - O + 1;
    if (p.band >= 0) w = std::min<int64_t>(w, 2 * (int64_t)p.band + 1);
    if (p.ring_diagonals) w = std::min<int64_t>(w, p.ring_diagonals);
    return std::max<int64_t>(std::min<int64_t>(w, 2 * (int64_t)max_length + 1), 1) + 2;
}

// rows 0 .. S of a pair
size_t ring_rows(const WfaPlan& p) {
    return (size_t)(p.ring_scores ? std::min(p.ring_scores, p.smax) : p.smax) + 1;
}

uint32_t seq_words(uint32_t max_length) { return 2 * ((max_length + 31) / 32) + 2; }

}  // namespace

namespace {

// bytes of the copies of `pairs` pairs' sequences
size_t seq_bytes(uint32_t max_length, size_t pairs) { return pairs * 2 * seq_words(max_length) * 4; }

// the copies of every round are kept for the traceback while they take no more than this
constexpr size_t kKeepBytes = 5u << 10;

}  // namespace

size_t ring_smem_per_warp(const WfaPlan& p, int G, uint32_t max_length) {
    const size_t P = pairs_of(G), W = (size_t)ring_width(p, max_length);
    const size_t kept = seq_bytes(max_length, 32) <= kKeepBytes ? 32 : P;
    return align_up(P * W * (8 + (G == 1 ? 4 : 8)) + seq_bytes(max_length, kept), 16);
}

size_t ring_warp_bytes(const WfaPlan& p, int G, uint32_t max_length) {
    const size_t P = pairs_of(G), W = (size_t)ring_width(p, max_length);
    size_t entries = 0;
    if (P > 1 || entry_form(max_length) == kWhole) {
        entries = ring_rows(p) * ((W * P + 31) / 32 * 32);
    } else {
        entries = dense_entries((int64_t)ring_rows(p) - 1, p.oe - p.e, (int64_t)W);
    }
    return align_up(32 * p.runs_bytes + entries * entry_bytes(max_length) + 512, 256);
}

bool ring_ok(const WfaPlan& p, uint32_t max_length) {
    const int O = p.oe - p.e;
    return p.adapt_min_len < 0 && !p.bound_pass && p.e == 1 && O >= 1 && O <= kMhDepth && p.x <= kMhDepth &&
           max_length <= kMaxWfaLength16 && ring_width(p, max_length) < 32768 && p.smax < (1 << 20);
}

// units (warps, or blocks for G > 32) of a block
static size_t units_of(int G) { return G > 32 ? 1 : kWarpsPerBlock; }

bool ring_fits(const WfaPlan& p, int G, uint32_t max_length, size_t scratch_bytes) {
    return ring_ok(p, max_length) && units_of(G) * ring_smem_per_warp(p, G, max_length) <= kMaxSmem &&
           units_of(G) * ring_warp_bytes(p, G, max_length) <= scratch_bytes;
}

int ring_group(const WfaPlan& p, uint32_t max_length, uint32_t num_pairs, int num_sms, size_t scratch_bytes, bool alone) {
    const int64_t widest = ring_width(p, max_length) - 2;
    auto held = [&](int G) -> uint64_t {   // pairs that the scratch holds at once
        return alone ? scratch_bytes / ring_warp_bytes(p, G, max_length) * pairs_of(G) : UINT32_MAX;
    };
    auto thin = [&](int G) {   // the pairs at work leave SMs short of warps
        return std::min<uint64_t>(num_pairs, held(G)) * G < (uint64_t)num_sms * kGoodWarps * 32;
    };
    int G = 1;
    while (G < 32 && (ring_smem_per_warp(p, G, max_length) > kGoodSmem || (G < widest && thin(G)))) G *= 2;
    while (G <= 32 && !ring_fits(p, G, max_length, scratch_bytes)) G *= 2;
    if (G > 32 || (G == 32 && (ring_smem_per_warp(p, G, max_length) > kBlockSmem ||
                              (widest > kBlockWidth && held(G) < (uint64_t)num_sms * kThinWarps))))
        G = 256;
    return ring_fits(p, G, max_length, scratch_bytes) ? G : 0;
}

namespace {

using RingKernel = void (*)(RingArgs);
RingKernel ring_kernel(int G, uint32_t max_length) {
    const int form = entry_form(max_length);
    return form == kWhole ? ring_kernel_for<kWhole>(G) : form == kBits16 ? ring_kernel_for<kBits16>(G) : ring_kernel_for<kBits32>(G);
}

// units of a grid that fills the device (0: none fits)
cudaError_t ring_grid(const WfaPlan& p, int G, uint32_t max_length, int num_sms, size_t* n) {
    const RingKernel kernel = ring_kernel(G, max_length);
    const size_t smem = units_of(G) * ring_smem_per_warp(p, G, max_length);
    cudaError_t e = cudaSuccess;
    if (smem > kPlainSmem)   // small calls are short enough for the call to count
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    if (e != cudaSuccess) return e;
    int bps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, G > 32 ? G : 32 * kWarpsPerBlock, smem);
    *n = (size_t)num_sms * (size_t)std::max(bps, 0) * units_of(G);
    return e;
}

}  // namespace

size_t ring_full_scratch(const WfaPlan& p, int G, uint32_t max_length, int num_sms) {
    size_t n = 0;
    if (ring_grid(p, G, max_length, num_sms, &n) != cudaSuccess) return 0;
    return n * ring_warp_bytes(p, G, max_length);
}

cudaError_t launch_wfa_ring(const WfaPlan& plan, int G, const PairsView& P, const LimitView& L, const OutView& O,
                            const uint32_t* order, const uint32_t* bounds, uint8_t* scratch, size_t scratch_bytes,
                            uint32_t* counters, int num_sms, cudaStream_t st, int* warps_used) {
    *warps_used = 0;
    if (P.num_pairs == 0) return cudaSuccess;
    RingArgs r{};
    WfaArgs& a = r.w;
    a.X = plan.x; a.OE = plan.oe; a.E = plan.e; a.g = plan.g; a.smax = plan.smax; a.band = plan.band;
    a.P = P; a.L = L; a.O = O;
    a.scratch = scratch;
    a.runs_bytes = plan.runs_bytes; a.runs_cap = (uint32_t)plan.runs_cap;
    a.order = order; a.bounds = bounds; a.counters = counters; a.nbuckets = 1;
    a.bound = plan.bound;
    const uint32_t len = P.max_length;
    r.width = (uint32_t)ring_width(plan, len);
    r.seq_words = seq_words(len);
    r.smem_warp = (uint32_t)ring_smem_per_warp(plan, G, len);
    r.seq_rounds = seq_bytes(len, 32) <= kKeepBytes ? (uint32_t)(32 / pairs_of(G)) : 1u;
    r.stage_shared = (size_t)plan.runs_cap * 33 * 4 <= (size_t)r.width * pairs_of(G) * (8 + (G == 1 ? 4 : 8));
    const size_t min_warp = ring_warp_bytes(plan, G, len);
    // value d scores back: bytes 2 (d - 1) and 2 (d - 1) + 1 of mh, the sign replicated above them
    auto sel = [](int d) { const uint32_t b = 2u * (uint32_t)(d - 1); return b | ((b + 1) << 4) | ((b + 9) << 8) | ((b + 9) << 12); };
    r.sel_x = sel(plan.x);
    r.sel_o = sel(plan.oe - plan.e);
    const size_t units = units_of(G), smem = units * r.smem_warp;
    const int threads = G > 32 ? G : 32 * kWarpsPerBlock;
    size_t n = 0;
    cudaError_t e = ring_grid(plan, G, len, num_sms, &n);
    if (e != cudaSuccess || n == 0) return e;
    n = std::min(n, scratch_bytes / min_warp);
    if (!bounds) n = std::min(n, ((size_t)P.num_pairs + pairs_of(G) - 1) / pairs_of(G));
    if (n == 0) return cudaSuccess;
    a.nwarps = (uint32_t)n;
    // a unit's arena: its share of the scratch, up to as many worst-case rounds as it defers
    a.warp_bytes = std::min(scratch_bytes / n & ~(size_t)255,
                            min_warp + (32 / pairs_of(G) - 1) * (min_warp - 32 * plan.runs_bytes));
    ring_kernel(G, len)<<<(unsigned)((n + units - 1) / units), threads, smem, st>>>(r);
    e = cudaGetLastError();
    if (e == cudaSuccess) *warps_used = (int)n;
    return e;
}

}  // namespace aim
