// Banded global DP with one pair per lane: NW edit distance (unit costs) and gap-affine Gotoh, the same alignments as
// dp_banded.cu's, for bands and costs that fit (dp_lane_evenness).
//
// Values carry their traceback.  The canonical traceback takes, in each cell, the first of X < I < D < M among the
// states that meet the cost the rest must have.  Values are 4 * cost + rank, where the rank says which op the state
// stands for in that cell: 0 M on a mismatch, 1 I, 2 D, 3 M on a match.  A minimum over predecessors then picks the
// least cost and, among equal costs, the first op in one instruction, and the two low bits of the result are the
// traceback's next op: nothing is compared for equality and no base is read again.
//   M(v,h) = [B(v-1,h-1)] + (mismatch ? 4 x : 3)      [.]: the cost without its rank
//   I(v,h) = [I'(v-1,h)] + 1,   D(v,h) = [D'(v,h-1)] + 2
//   B = min(M, I, D),   I' = min(M + 4 oe, D + 4 oe, I + 4 e),   D' = min(M + 4 oe, I + 4 oe, D + 4 e)
// A cell's trace is the ranks of its B, I' and D': the op before an M, an I or a D that leads on from it.  Costs are
// kept relative to 4 e (v + h), so that extending a gap adds nothing: I' = min(M + 4 o, D + 4 o, I), and M takes 8 e
// off.  What the next cells read is kept with the rank they want: B | 3, [I'] + 1, [D'] + 2.  With unit costs there is
// one state: H = min((H(v-1,h-1) | 3) + (mismatch ? 1 : 0), (H(v-1,h) | 3) + 2, (H(v,h-1) | 3) + 3), its rank the
// cell's own op.  Ranks go into the trace word by one funnel shift each.
//
// A lane sweeps its pair row by row over the 2b+1 diagonals, four cells at a time: B and I' of the row before in
// shared memory (four diagonals of a lane in one 16-byte access, lanes side by side), D' in a register, 16 cells'
// mismatch bits from one XOR of the target's window with the row's base.  The warp writes three 128-byte segments of
// trace per 16 cells (one with unit costs).  No lane waits for another, none is idle at the band's edge, and no value
// is shuffled; a batch of 32 pairs costs as many instructions as its longest pair.
//
// Cells outside the matrix: left of column 0 everything comes from infinite values; right of column m values are
// computed but nothing at or left of column m reads them; the diagonal after the last one is set infinite.  Infinity
// is 2^30 + 2^29, and the host checks that four times the costs along a path stay below 2^28, so infinite values,
// which move by as much, stay apart from others.
// What bounds it: the integer pipe and issue (59 % and 1.8 per cycle over 50k pairs, whose second wave is a third full),
// 24 lane instructions a cell of which the three 3-input minima, three shifts into the trace and three ranks are most.  1M
// pairs of 250 bp, band 25: 13.4 ms, 9,700 warp instructions a pair (dp_banded.cu: 51.3 ms and 55,400); edit distance, 1M x 100 bp, band 10: 1.45 ms (9.3 ms).  With ranks compared
// by equality and six bits assembled per cell it took 15.3 ms, with costs not relative to 4 e (v + h) 15.1 ms.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "wfa_common.cuh"

namespace aim {
namespace {

constexpr int kInf4 = (1 << 30) + (1 << 29);
constexpr int kLaneWarps = 2;   // per block

struct LaneArgs {
    Costs c;
    PairsView P;
    LimitView L;
    OutView O;
    int band;
    int groups;               // of four diagonals
    uint32_t row_words;       // trace words per row and lane
    uint32_t t_words;         // 32-bit words of a target copy, padding included
    uint32_t t_pad;           // words before its first base
    uint32_t smem_warp;
    uint8_t* scratch;
    size_t warp_bytes, trace_bytes;   // a warp's scratch: trace rows, then 32 lanes' runs
    uint32_t runs_cap;
    uint32_t nwarps;
    uint32_t evenness;        // reads of an EVEN instance
    uint32_t* counter;
};

extern __shared__ __align__(16) uint8_t s_lane[];

// the two low bits of v pushed into the top of a trace word
__device__ __forceinline__ void push(uint32_t& word, int v) { word = __funnelshift_r(word, (uint32_t)v, 2); }

// EVEN: only batches of reads at least a.evenness even (an instance of its own: the test alone cost unit costs 12 %)
template <bool UNIT, bool EVEN>
__global__ void __launch_bounds__(32 * kLaneWarps) dp_lane_kernel(LaneArgs a) {
    if (EVEN && !reads_even(a.P, a.evenness)) return;
    const int lane = (int)(threadIdx.x & 31);
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gwarp >= a.nwarps) return;
    const int b = a.band, NG = a.groups;
    uint8_t* sm = s_lane + (size_t)(threadIdx.x >> 5) * a.smem_warp;
    int4* sB = reinterpret_cast<int4*>(sm) + lane;             // [groups][32]: B (H with unit costs)
    int4* sI = sB + (UNIT ? 0 : (NG + 1) * 32);                // [groups][32]: I' (each a group longer than the band)
    uint32_t* sT = reinterpret_cast<uint32_t*>(sm + (size_t)(UNIT ? 1 : 2) * (NG + 1) * 512) + lane;   // [t_words][32]
    uint32_t* trace = reinterpret_cast<uint32_t*>(a.scratch + (size_t)gwarp * a.warp_bytes) + lane;   // [row][word][32]
    uint32_t* staged = reinterpret_cast<uint32_t*>(a.scratch + (size_t)gwarp * a.warp_bytes + a.trace_bytes);
    const int e4 = UNIT ? 0 : 4 * a.c.e, o4 = 4 * a.c.o;
    const int on_match = -2 * e4, on_mismatch = 4 * a.c.x - 3 - 2 * e4;   // what M adds to B | 3
    unsigned long long st_cells = 0;
    uint32_t st_pairs = 0;

    for (;;) {
        uint32_t p0 = 0;
        if (lane == 0) p0 = atomicAdd(a.counter, 32u);
        p0 = __shfl_sync(kFull, p0, 0);
        if (p0 >= a.P.num_pairs) break;
        const bool have = (uint32_t)lane < a.P.num_pairs - p0;
        const uint32_t pi = p0 + (have ? (uint32_t)lane : 0u);
        int n = 0, m = 0, kend = 0, lim4 = 0, fail = -1;   // fail >= 0: the flags of a pair without an alignment
        const uint64_t* Pw = nullptr;
        bool live = have;
        if (have) {
            ++st_pairs;
            n = (int)a.P.read_len[pi]; m = (int)a.P.target_len[pi];
            const int64_t lim = pair_limit(a.L, pi);
            if (pair_bad(a.P, pi) || (uint32_t)n > a.P.max_length || (uint32_t)m > a.P.max_length || lim == -2) {
                fail = AIM_F_BAD_PAIR;
            } else {
                kend = m - n;
                if (kend > b || -kend > b) fail = AIM_F_REJECTED;
                lim4 = lim >= (int64_t)kInf ? (1 << 30) - 1 : (int)lim * 4 + 3;
            }
            live = fail < 0;
        }
        if (!live) n = m = 0;
        // the target's copy, its first base after t_pad words
        if (live) {
            Pw = read_words(a.P, pi);
            const uint64_t* Tw = target_words(a.P, pi);
            for (int w = 0; w < (m + 31) >> 5; ++w) {
                const uint64_t x = __ldg(Tw + w);
                sT[(a.t_pad + 2 * w) * 32] = (uint32_t)(x >> 32);
                sT[(a.t_pad + 2 * w + 1) * 32] = (uint32_t)x;
            }
        }
        // row 0: offset 0 on diagonal 0, a deletion of h bases on diagonal h
        for (int g = 0; g <= NG; ++g) {
            int B[4], I[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int h = 4 * g + c - b;
                if (UNIT) {
                    B[c] = h < 0 || h > b ? kInf4 : (4 * h) | 3;
                } else {
                    B[c] = h < 0 ? kInf4 : (h == 0 ? 0 : o4) | 3;                      // D: o + h e
                    I[c] = h < 0 || h > b ? kInf4 : (h == 0 ? 0 : o4) + o4 + 1;
                }
            }
            sB[g * 32] = make_int4(B[0], B[1], B[2], B[3]);
            if (!UNIT) sI[g * 32] = make_int4(I[0], I[1], I[2], I[3]);
        }
        for (uint32_t w = 0; w < a.row_words; ++w) trace[(size_t)w * 32] = 0xaaaaaaaau;   // from D throughout
        const int qend = kend + b;
        const int* lane_B = reinterpret_cast<const int*>(sB + (qend >> 2) * 32) + (qend & 3);
        int* past = reinterpret_cast<int*>((UNIT ? sB : sI) + ((2 * b + 1) >> 2) * 32) + ((2 * b + 1) & 3);
        int end_val = live && n == 0 ? *lane_B + e4 * m : kInf4;
        uint32_t cells = live ? (uint32_t)min(m, b) + 1 : 0;

        const int rows = __reduce_max_sync(kFull, n);
        uint64_t pword = 0;
        for (int v = 1; v <= rows; ++v) {
            if (((v - 1) & 31) == 0 && v <= n) pword = __ldg(Pw + ((v - 1) >> 5));
            const uint32_t base = (uint32_t)(pword >> 62) * 0x55555555u;   // the row's base in every place
            pword <<= 2;
            uint32_t* trow = trace + (size_t)v * a.row_words * 32;
            const int t0 = v - 1 - b + 16 * (int)a.t_pad;   // place of the first cell's target base in the copy
            int D = kInf4;               // [D'] + 2 (H | 3 with unit costs) of the cell to the left
            int4 up = UNIT ? sB[0] : sI[0];   // of the row before: this group's
            int4 B = UNIT ? up : sB[0];
            auto sixteen = [&](const int g0, const int left, auto full) {   // `left` groups of the row from g0 on
                // mismatch bits of 16 cells, the first cell's in bit 0
                const uint32_t* tw = sT + ((t0 + 4 * g0) >> 4) * 32;
                const uint32_t z = __brev(__funnelshift_l(tw[32], tw[0], 2 * (t0 + 4 * g0)) ^ base);
                const uint32_t y = (z | (z >> 1)) & 0x55555555u;
                uint32_t wB = 0, wI = 0, wD = 0;
                int4* pB = sB + g0 * 32;
                int4* pI = sI + g0 * 32;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (decltype(full)::value || u < left) {
                        const int4 up_next = UNIT ? pB[(u + 1) * 32] : pI[(u + 1) * 32];
                        const int4 B_next = UNIT ? up_next : pB[(u + 1) * 32];
                        const int upv[5] = {up.x, up.y, up.z, up.w, up_next.x};
                        const int Bv[4] = {B.x, B.y, B.z, B.w};
                        int Bn[4], In[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const bool mm = (y & (1u << (8 * u + 2 * c))) != 0;
                            if (UNIT) {
                                const int H = __vimin3_s32(D + 3, upv[c + 1] + 2, Bv[c] + (mm ? 1 : 0));
                                push(wB, H);
                                D = Bn[c] = H | 3;
                            } else {
                                const int M = Bv[c] + (mm ? on_mismatch : on_match), I = upv[c + 1];
                                const int Mo = M + o4;
                                const int Bc = __vimin3_s32(M, I, D);
                                const int Ic = __vimin3_s32(Mo, D + o4, I);
                                const int Dc = __vimin3_s32(Mo, I + o4, D);
                                push(wB, Bc); push(wI, Ic); push(wD, Dc);
                                Bn[c] = Bc | 3;
                                In[c] = (Ic & ~3) | 1;
                                D = (Dc & ~3) | 2;
                            }
                        }
                        pB[u * 32] = make_int4(Bn[0], Bn[1], Bn[2], Bn[3]);
                        if (!UNIT) pI[u * 32] = make_int4(In[0], In[1], In[2], In[3]);
                        up = up_next;
                        B = B_next;
                    }
                }
                const int rest = 32 - 8 * left;   // a short word's bits move down to its low end
                uint32_t* t = trow + (size_t)(g0 >> 2) * (UNIT ? 32 : 96);
                t[0] = wB >> rest;
                if (!UNIT) { t[32] = wI >> rest; t[64] = wD >> rest; }
            };
            int g0 = 0;
            for (; g0 + 4 <= NG; g0 += 4) sixteen(g0, 4, std::true_type{});
            if (g0 < NG) sixteen(g0, NG - g0, std::false_type{});
            *past = kInf4;   // the diagonal after the last one, to the row below
            if (v <= n) {
                cells += (uint32_t)max(min(m, v + b) - max(v - b, 0) + 1, 0);
                if (v == n) end_val = *lane_B + e4 * (n + m);
            }
            // every path crosses every row and costs never fall along it: a lane whose row lies above its limit is
            // done, and the warp once all its lanes are
            if ((v & 15) == 0) {
                bool over = true;
                if (v < n) {
                    int least = kInf4;
                    for (int g = 0; g < NG; ++g) {
                        const int4 q = sB[g * 32];
                        const int rel = e4 * (2 * v + 4 * g - b);   // the first cell's 4 e (v + h)
                        least = min(least, min(min(q.x, q.y + e4), min(q.z + 2 * e4, q.w + 3 * e4)) + rel);
                    }
                    over = least > lim4;
                    if (over) n = 0;   // rejected: end_val stays infinite
                }
                if (__all_sync(kFull, over)) break;
            }
        }

        // ---- results
        __syncwarp();
        if (live && end_val > lim4) { live = false; fail = AIM_F_REJECTED; }
        RunStage wr{staged + (size_t)lane * a.runs_cap, 1, a.runs_cap, 0, 0, 0};
        uint64_t off = 0;
        uint32_t copy = 0;
        if (live) {
            int v = (int)a.P.read_len[pi], h = m;
            bool ok_path = true;
            // the trace words of the next rows at once: paths mostly stay on their diagonal, and a step then costs a
            // fraction of a memory round trip
            constexpr int kAhead = UNIT ? 8 : 4;
            uint32_t op = 0;   // affine: the op at (v, h); from the end cell's B at first
            uint32_t from = 0; // which of the cell's three words says it: 0 B, 1 I', 2 D'
            while ((v > 0 || h > 0) && ok_path) {
                const int top = v, col = (h - v + b) >> 4;
                uint32_t w[kAhead][UNIT ? 1 : 3];
#pragma unroll
                for (int i = 0; i < kAhead; ++i)
#pragma unroll
                    for (int k = 0; k < (UNIT ? 1 : 3); ++k)
                        w[i][k] = trace[((size_t)max(top - i, 0) * a.row_words + col * (UNIT ? 1 : 3) + k) * 32];
#pragma unroll
                for (int i = 0; i < kAhead; ++i) {
                    while (v == top - i && (v > 0 || h > 0)) {
                        const int q = h - v + b;
                        if (q >> 4 != col) break;
                        const uint32_t word = UNIT ? w[i][0] : from == 0 ? w[i][0] : from == 1 ? w[i][UNIT ? 0 : 1] : w[i][UNIT ? 0 : 2];
                        op = (word >> (2 * (q & 15))) & 3u;
                        if (op == 1) { wr.put(kOpIns, 1); --v; from = 1; }
                        else if (op == 2) { wr.put(kOpDel, 1); --h; from = 2; }
                        else { wr.put(op == 0 ? kOpMismatch : kOpMatch, 1); --v; --h; from = 0; }
                        if (v < 0 || h < 0) { ok_path = false; break; }   // (not expected)
                    }
                }
            }
            wr.flush();
            const bool ok = v == 0 && h == 0 && wr.n <= wr.cap;   // (not expected otherwise)
            uint8_t flags = ok ? 0 : AIM_F_STEP_CAP;
            if (ok && a.O.cigars) {
                off = a.O.cigar_off[pi];
                if (wr.n <= a.O.cigar_off[pi + 1] - off) copy = wr.n;
                else flags = AIM_F_CIGAR_OVERFLOW;
            }
            write_header(a.O, pi, ok ? end_val >> 2 : -1, flags, wr.n);
        } else if (have) {
            write_header(a.O, pi, -1, (uint8_t)fail, 0);
        }
        __syncwarp();
        if (a.O.cigars) copy_runs(a.O, copy, off, staged, a.runs_cap, 1, lane);
        __syncwarp();
        st_cells += cells;
    }
    warp_stat_add(a.O.stats, 2, st_cells, (uint32_t)lane);
    warp_stat_add(a.O.stats, 3, st_pairs, (uint32_t)lane);
}

int groups_of(int band) { return (2 * band + 1 + 3) / 4; }
uint32_t row_words_of(bool unit, int band) { return (unit ? 1u : 3u) * ((uint32_t)(groups_of(band) + 3) / 4); }
uint32_t t_pad_of(int band) { return (uint32_t)band / 16 + 1; }
uint32_t t_words_of(int band, uint32_t max_length) {
    return t_pad_of(band) + 2 * ((max_length + 31) / 32) + (uint32_t)band / 16 + 3;
}
size_t lane_smem(bool unit, int band, uint32_t max_length) {
    return (size_t)(unit ? 1 : 2) * (groups_of(band) + 1) * 512 + (size_t)t_words_of(band, max_length) * 128;
}
size_t lane_trace(bool unit, int band, uint32_t max_length) {
    return align_up(((size_t)max_length + 1) * row_words_of(unit, band) * 128, 256);
}
uint32_t lane_runs(bool unit, const Costs& c, uint32_t max_length, int64_t max_limit) {
    const int64_t minc = unit ? 1 : std::min(c.x, c.o + c.e);
    int64_t cap = 2 * (int64_t)max_length + 1;
    if (max_limit < kUnbounded) cap = std::min(cap, 2 * (max_limit / minc) + 1);
    return (uint32_t)cap;
}
size_t lane_warp(bool unit, int band, const Costs& c, uint32_t max_length, int64_t max_limit) {
    return lane_trace(unit, band, max_length) + align_up((size_t)lane_runs(unit, c, max_length, max_limit) * 128, 256);
}

constexpr size_t kLaneSmem = 226u << 10;   // dynamic shared memory a block may use

}  // namespace

// Where this form is the faster one.  A warp takes as long for one pair as for 32, rho times a lone pair's warp in
// dp_banded.cu, and runs in waves of the pairs that shared memory and scratch hold.  dp_banded.cu's time grows with the
// pairs' own lengths: of y = pairs * mean / longest, as many as the scratch holds are at work, and sat of them on every SM
// double the time of each.  In a lone pair's times:
//   here rho * waves,   there max(1, y / held) (1 + min(y, held) / (sat * SMs)).
// The two are equal at the share of the mean in the longest that this returns; the launches look at the lengths.  Fitted to
// (ms, dp_banded.cu / here, 1 GB unless stated) 250 bp, band 25: 2,500 pairs 0.37 / 0.46, 5,000 0.53 / 0.46; 1,000 bp, 8,000
// pairs, 64 MB: band 25 13.8 / 10.3, band 60 40.3 / 36.6, band 120 121 / 128, at 256 MB 33.5 / 36.1, 1 GB 15.1 / 10.6; 3,000
// bp, band 25, 8,000 pairs 12.1 / 9.1; 50-1,000 bp, band 25: 4,200 pairs 1.19 / 1.54, 8,000 1.45 / 1.58, 10,000 1.59 / 1.56;
// band 60: 4,200 1.73 / 2.94, 16,000 3.82 / 2.98; band 120: 8,000 5.19 / 5.22, 16,000 8.97 / 10.1; edit distance, 100 bp, band
// 10: 2,500 0.100 / 0.101, 5,000 0.139 / 0.101; 50-1,000 bp, band 12: 4,200 0.567 / 0.587, 6,000 0.706 / 0.594.
// Below 27 pairs an SM it has not been measured throughout.  A share below a quarter counts as none, such batches being
// rare, and so does any below 1 with unit costs, where little is lost, or where the second launch's 4 us would show (250
// rows of band 25 take 0.41 ms).
uint32_t dp_lane_evenness(const DpPlan& plan, const Costs& c, uint32_t max_length, int64_t max_limit, uint32_t num_pairs,
                          int num_sms, size_t scratch_bytes) {
    const bool unit = plan.unit;
    const int band = plan.band;
    if (num_pairs < 27u * (uint32_t)num_sms) return kNeverEven;
    const int64_t maxc = unit ? 1 : std::max<int64_t>(c.x, (int64_t)c.o + c.e);
    const size_t smem = kLaneWarps * lane_smem(unit, band, max_length), warp = lane_warp(unit, band, c, max_length, max_limit);
    if ((2 * (int64_t)max_length + 2 * (int64_t)band + 8) * maxc >= (int64_t)1 << 26 || smem > kLaneSmem ||
        kLaneWarps * warp > scratch_bytes)
        return kNeverEven;
    const size_t held = scratch_bytes / dp_slot_bytes(plan, c, max_length, max_limit);   // pairs at once in dp_banded.cu
    if (held < (size_t)plan.pairs_per_warp) return 0;   // it has room for none
    const int r = plan.blocks == 1 ? 0 : plan.blocks == 2 ? 1 : 2;
    const double rho = unit ? (r == 0 ? 1.7 : r == 1 ? 2.2 : 2.7) : (r == 0 ? 2.0 : r == 1 ? 2.3 : 3.0);
    const double sat = (unit ? 13.0 : r == 0 ? 27.0 : r == 1 ? 19.0 : 10.0) * num_sms;
    const size_t warps = std::min((size_t)num_sms * std::min<size_t>(kLaneSmem / smem * kLaneWarps, 16), scratch_bytes / warp);
    const size_t waves = ((size_t)num_pairs + 32 * warps - 1) / (32 * warps);
    const double here = rho * (double)waves;
    double y = (here - 1.0) * sat;
    if (y > (double)held) y = here / (1.0 / (double)held + 1.0 / sat);
    const double share = y / (double)num_pairs;
    if (share >= 1.0) return kNeverEven;
    return unit || share <= 0.25 || (uint64_t)max_length * (2 * band + 1) < 250 * 51 ? 0 : (uint32_t)(share * 256.0);
}

cudaError_t launch_dp_lane(bool unit, int band, const Costs& c, const PairsView& P, const LimitView& L, const OutView& O,
                           int64_t max_limit, uint32_t evenness, uint8_t* scratch, size_t scratch_bytes,
                           uint32_t* counter, int num_sms, cudaStream_t st, int* warps_used) {
    *warps_used = 0;
    if (P.num_pairs == 0) return cudaSuccess;
    LaneArgs a{};
    a.c = c; a.P = P; a.L = L; a.O = O;
    a.evenness = evenness;
    a.band = band;
    a.groups = groups_of(band);
    a.row_words = row_words_of(unit, band);
    a.t_words = t_words_of(band, P.max_length);
    a.t_pad = t_pad_of(band);
    a.smem_warp = (uint32_t)lane_smem(unit, band, P.max_length);
    a.scratch = scratch;
    a.trace_bytes = lane_trace(unit, band, P.max_length);
    a.warp_bytes = lane_warp(unit, band, c, P.max_length, max_limit);
    a.runs_cap = lane_runs(unit, c, P.max_length, max_limit);
    a.counter = counter;
    void (*kernel)(LaneArgs) = unit ? dp_lane_kernel<true, false>
                               : evenness ? dp_lane_kernel<false, true> : dp_lane_kernel<false, false>;
    const size_t smem = (size_t)kLaneWarps * a.smem_warp;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLaneSmem);
    if (e != cudaSuccess) return e;
    int bps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, 32 * kLaneWarps, smem);
    if (e != cudaSuccess) return e;
    if (bps < 1) return cudaSuccess;
    size_t warps = std::min((size_t)num_sms * bps * kLaneWarps, scratch_bytes / a.warp_bytes);
    warps = std::min(warps, ((size_t)P.num_pairs + 31) / 32);
    if (warps == 0) return cudaSuccess;
    a.nwarps = (uint32_t)warps;
    kernel<<<(unsigned)((warps + kLaneWarps - 1) / kLaneWarps), 32 * kLaneWarps, smem, st>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess) *warps_used = (int)warps;
    return e;
}

}  // namespace aim
