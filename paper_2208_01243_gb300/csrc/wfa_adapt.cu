// WFA-adaptive with the running state in shared memory: wfa_ring.cu's recurrences and layout (G lanes per pair, P =
// 32 / G pairs per warp, arrays interleaved by pair, M~ of the last four scores and J, K per diagonal; E == 1, X and
// O up to 4) under the pruning rule, which decides every wavefront's range from its entries.
//
// Ranges.  A score's range is the union of its sources' recorded ranges, the gap sources' one diagonal wider, and its
// record is the part of it that holds valid entries, with the outer diagonals too far behind dropped.  Row s also
// covers the diagonals of the last four records that its own range leaves out: there M~, I~ and D~ are invalid, and J
// and K become M~[s-O], which the next score may open a gap from.  Diagonals sit at k mod W, W a power of two; a pair
// whose row and its two neighbours do not fit W, or whose history outgrows its warp's arena, is flagged AIM_F_STEP_CAP
// and aligned again by wfa.cu's kernel, as are the pairs that outgrow that kernel's first pass.
//
// A dropped entry must not feed later scores: its newest M~ and its history word are cleared, and J and K go back to
// M~[s-O], kept for that in an array of its own.
//
// Pairs end at scores far apart, so a group whose pair has ended takes its next one while the others of its warp go on.
// Each group has places of its own for the tables and histories of the pair under way and of those that await their
// traceback; when one has no place left, the whole warp traces back what waits, a lane each, and goes on.
//
// History: per entry M~ in 16 bits, which candidate gave the offset that M~ extends (mismatch, I or D, in that order),
// and whether J and K came from the extension (on ties they do: the traceback takes an extension before an opening).
// Following these bits is the source-following traceback: at each step the word of one entry says where to go, and a
// gap's offset is the M~ at its opening.  A table holds each row's place and each pair's first diagonal in it.
//
// What bounds it: issue and the integer pipe (2.4 per cycle, 53-58 % busy) with 20 to 23 of 32 lanes at work: 56,600 warp
// instructions a pair of 1,000 bp at 5 % and 8 lanes, two reductions of three shuffles and the votes in every score.
#include <algorithm>
#include <cstdint>

#include "wfa_common.cuh"

namespace aim {
namespace {

constexpr int kAdaptWarps = 2;   // per block
constexpr int kFarLo = 1 << 29, kFarHi = -(1 << 29);

struct AdaptArgs {
    WfaArgs w;
    uint32_t width;          // W
    uint32_t seq_words;      // 32-bit words per sequence copy
    uint32_t smem_warp;
    uint32_t table_rows;     // rows a pair's table holds
    size_t table_bytes;
    uint32_t hist_entries;   // entries a pair's history holds
    uint32_t place_units;    // 256-byte units of a pair's table and history
    uint32_t sel_x, sel_o;
};

extern __shared__ __align__(16) uint8_t s_adapt[];

// history words
__device__ __forceinline__ uint32_t word_of(int mv, uint32_t src, bool ins_ext, bool del_ext) {
    return ((uint32_t)mv & 0xffffu) | (src << 16) | ((uint32_t)ins_ext << 18) | ((uint32_t)del_ext << 19);
}
constexpr uint32_t kNoWord = 0xffffu;
__device__ __forceinline__ int m_of(uint32_t e) { return (int16_t)(uint16_t)e; }

// Source-following traceback of one finished pair by one lane.
__device__ void adapt_traceback(const WfaArgs& a, const uint8_t* place, size_t table_bytes, uint32_t pi, int final_s,
                                RunStage& wr, bool& ok) {
    const int2* table = reinterpret_cast<const int2*>(place);
    const uint32_t* hist = reinterpret_cast<const uint32_t*>(place + table_bytes);
    const int n = (int)a.P.read_len[pi], m = (int)a.P.target_len[pi];
    const int X = a.X, OE = a.OE;
    auto entry = [&](int c, int k) -> uint32_t {   // only entries that a row holds are asked for
        const int2 t = table[c];
        return hist[(uint32_t)(t.y + (k - t.x))];
    };
    int c = final_s, k = m - n, h = m;
    for (int guard = n + m + 2; ok; --guard) {
        if (c == 0) { ok = k == 0; if (h > 0) wr.put(kOpMatch, (uint32_t)h); break; }
        if (guard <= 0 || c < 0) { ok = false; break; }
        const uint32_t e = entry(c, k);
        const uint32_t src = (e >> 16) & 3u;
        if (src == 0) {
            if (c < X) { ok = false; break; }
            const int f0 = m_of(entry(c - X, k)) + 1;
            if (f0 <= 0 || f0 > h) { ok = false; break; }
            if (h > f0) wr.put(kOpMatch, (uint32_t)(h - f0));
            wr.put(kOpMismatch, 1);
            h = f0 - 1;
            c -= X;
        } else {
            // the gap back to its opening: `len` bases, then M~ there is the offset an insertion leaves unchanged
            const int step = src == 1 ? 1 : -1;
            const uint32_t bit = src == 1 ? 18 : 19;
            int len = 0;
            for (;;) {
                ++len;
                if (c < 1 || len > n + m) { ok = false; break; }
                k += step;
                if (!((entry(c - 1, k) >> bit) & 1u)) break;
                --c;
            }
            c -= OE;
            if (!ok || c < 0) { ok = false; break; }
            const int at = m_of(entry(c, k)), f0 = src == 1 ? at : at + len;
            if (at < 0 || f0 > h) { ok = false; break; }
            if (h > f0) wr.put(kOpMatch, (uint32_t)(h - f0));
            wr.put(src == 1 ? kOpIns : kOpDel, (uint32_t)len);
            h = at;
        }
    }
    wr.flush();
    ok = ok && wr.n <= wr.cap;
}

template <int G>
__global__ void __launch_bounds__(32 * kAdaptWarps) wfa_adapt_kernel(AdaptArgs r) {
    constexpr int P = 32 / G;
    const WfaArgs& a = r.w;
    const int lane = (int)(threadIdx.x & 31), g = lane % P, gl = lane / P;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gwarp >= a.nwarps) return;
    const int W = (int)r.width, wm = W - 1;
    uint8_t* sm = s_adapt + (size_t)(threadIdx.x >> 5) * r.smem_warp;
    uint2* mh = reinterpret_cast<uint2*>(sm) + g;                             // [W][P] M~ of the last four scores
    uint32_t* jd = reinterpret_cast<uint32_t*>(sm + (size_t)W * P * 8) + g;   // [2][W][P] J, K
    uint32_t* sp = reinterpret_cast<uint32_t*>(sm + (size_t)W * P * 16) + g;
    uint32_t* st = sp + r.seq_words * P;
    uint16_t* smo = reinterpret_cast<uint16_t*>(sm + (size_t)W * P * 16 + (size_t)r.seq_words * P * 8) + g;   // [W][P] M~[s-O]
    uint8_t* arena = a.scratch + (size_t)gwarp * a.warp_bytes;
    // a group's places for tables and histories, in 256-byte units
    const uint32_t group_units = (uint32_t)((a.warp_bytes - 32 * a.runs_bytes) / P >> 8);
    uint8_t* places = arena + 32 * a.runs_bytes + ((size_t)g * group_units << 8);
    const int X = a.X, OE = a.OE, O = OE - 1;
    const uint32_t pair_lanes = G == 32 ? kFull : (uint32_t)(0xffffffffull / ((1ull << P) - 1ull)) << g;
    unsigned long long st_cells = 0, st_windows = 0;
    uint32_t st_pairs = 0;
    // finished pairs awaiting their traceback: the group's j-th with its lane j * P + g
    uint32_t p_pi = 0, p_at = 0;
    int p_s = -1, waiting = 0;
    // the next place starts at `next`, and ends before `last`; nothing live lies below `low`
    uint32_t next = 0, last = group_units, low = 0;

    auto least2 = [&](uint32_t v) {   // the smaller of each 16-bit half over the pair's lanes
#pragma unroll
        for (int o = P; o < 32; o <<= 1) v = __vminu2(v, __shfl_xor_sync(kFull, v, o));
        return v;
    };
    bool run = false;    // this group's pair is under way, at `next`
    auto finish = [&]() {
        __syncwarp();
        RunStage wr{reinterpret_cast<uint32_t*>(arena + (size_t)lane * a.runs_bytes), 1u, a.runs_cap, 0, 0, 0};
        bool ok = p_s >= 0;
        uint64_t off = 0;
        uint32_t copy = 0;
        if (ok) {
            adapt_traceback(a, places + ((size_t)p_at << 8), r.table_bytes, p_pi, p_s, wr, ok);
            uint8_t flags = ok ? 0 : AIM_F_STEP_CAP;
            if (ok && a.O.cigars) {
                off = a.O.cigar_off[p_pi];
                if (wr.n <= a.O.cigar_off[p_pi + 1] - off) copy = wr.n;
                else flags = AIM_F_CIGAR_OVERFLOW;
            }
            write_header(a.O, p_pi, ok ? p_s * a.g : -1, flags, wr.n);
        }
        __syncwarp();
        if (a.O.cigars) copy_runs(a.O, copy, off, reinterpret_cast<const uint32_t*>(arena), (uint32_t)(a.runs_bytes / 4), 1u, lane);
        __syncwarp();
        p_s = -1;
        waiting = 0;
        if (!run) next = 0;   // only the pair under way is left
        low = next;
        last = group_units;
    };

    uint32_t pi = 0;
    int status = kIdle, n = 0, m = 0, S = 0, kend = 0, klo = 0, khi = 0, s = 0;
    uint32_t filled = 0, cells = 0, windows = 0;
    int2* table = nullptr;
    uint32_t* hist = nullptr;
    int2 rc[5];          // the records of the last five scores, the newest first
    int zlo = 0, zhi = 0;   // diagonals whose places hold this pair's values (or invalid ones)
    bool hit = false;
    bool more = true;    // the queue may hold pairs

    // what is left of a pair that has ended
    auto settle = [&]() {
        if (status == kDone) {
            if (gl == waiting) { p_pi = pi; p_s = s; p_at = next; }
            ++waiting;
            next += (uint32_t)((r.table_bytes + (size_t)filled * sizeof(uint32_t) + 255) >> 8);
        } else if (gl == 0) {
            emit_failed(a, pi, status);
        }
        st_cells += cells;
        st_windows += windows;
        cells = windows = 0;
    };

    for (;;) {
        // groups whose pair has ended take their next one while the others go on
        const uint32_t idle = __ballot_sync(kFull, !run) & ((1u << P) - 1u);   // a bit per group
        if (more && idle) {
            auto room = [&]() {
                if (last - next < r.place_units && last == group_units && low >= r.place_units) { next = 0; last = low; }
                return waiting < G && last - next >= r.place_units;
            };
            if (__any_sync(kFull, !run && !room())) finish();
            uint32_t pos = 0;
            if (lane == 0) pos = atomicAdd(a.counters, (uint32_t)__popc(idle));
            pos = __shfl_sync(kFull, pos, 0);
            more = pos < a.P.num_pairs && a.P.num_pairs - pos > (uint32_t)__popc(idle);
            const uint32_t ahead = (uint32_t)__popc(idle & ((1u << g) - 1u));
            const bool fresh = !run && pos < a.P.num_pairs && ahead < a.P.num_pairs - pos;
            if (fresh) {
                pi = pos + ahead;
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
                    const bool far = a.band >= 0 && (kend > a.band || -kend > a.band);
                    status = far || S < 0 || (kend != 0 && abs(kend) + O > S) ? kRejected : kRun;
                }
                klo = a.band >= 0 ? max(-n, -a.band) : -n;
                khi = a.band >= 0 ? min(m, a.band) : m;
                run = status == kRun;
                if (!run) settle();
            }
            const bool begins = fresh && run;
            __syncwarp();   // the last pair's copies have been read
            if (begins) {
                const uint64_t* Pw = read_words(a.P, pi);
                const uint64_t* Tw = target_words(a.P, pi);
                for (int w = gl; w < (n + 31) >> 5; w += G) {
                    const uint64_t x = __ldg(Pw + w);
                    sp[2 * w * P] = (uint32_t)(x >> 32); sp[(2 * w + 1) * P] = (uint32_t)x;
                }
                for (int w = gl; w < (m + 31) >> 5; w += G) {
                    const uint64_t x = __ldg(Tw + w);
                    st[2 * w * P] = (uint32_t)(x >> 32); st[(2 * w + 1) * P] = (uint32_t)x;
                }
                if (gl < 3) {   // diagonals -1, 0, 1
                    const int at = ((gl - 1) & wm) * P;
                    mh[at] = make_uint2(~0u, ~0u);
                    jd[at] = ~0u;
                    jd[W * P + at] = ~0u;
                }
            }
            __syncwarp();
            if (begins) {
                table = reinterpret_cast<int2*>(places + ((size_t)next << 8));
                hist = reinterpret_cast<uint32_t*>(places + ((size_t)next << 8) + r.table_bytes);
                rc[0] = make_int2(0, 0);
                rc[1] = rc[2] = rc[3] = rc[4] = make_int2(kFarLo, kFarHi);
                zlo = -1; zhi = 1;
                s = 0;
                filled = 1;
                hit = false;
                if (gl == 0) {
                    const int m0 = match_on<P>(sp, st, 0, 0, min(n, m));
                    mh[0] = make_uint2((uint32_t)m0 | 0xffff0000u, ~0u);
                    table[0] = make_int2(0, 0);
                    hist[0] = word_of(m0, 0, false, false);
                    hit = kend == 0 && m0 >= m;
                    ++cells; ++windows;
                }
            }
            const bool at_once = (__ballot_sync(kFull, begins && hit) & pair_lanes) != 0;
            if (begins && at_once) { status = kDone; run = false; settle(); }
            __syncwarp();
        }
        if (!__any_sync(kFull, run)) {
            if (more) continue;
            break;
        }
        // scores of every pair under way, until one ends
        bool over = false;
        auto end_as = [&](int how) { status = how; over = true; run = false; };
        do {
            if (run && ++s > S) end_as(kRejected);
            int lo = kFarLo, hi = kFarHi, elo = kFarLo, ehi = kFarHi;
            if (run) {
                const int2 r1 = rc[0], r2 = rc[1], r3 = rc[2], r4 = rc[3];
                const int2 rx = X == 1 ? r1 : X == 2 ? r2 : X == 3 ? r3 : r4;
                const int2 ro = OE == 2 ? r2 : OE == 3 ? r3 : OE == 4 ? r4 : rc[4];
                lo = max(min(rx.x, min(ro.x, r1.x) - 1), klo);
                hi = min(max(rx.y, max(ro.y, r1.y) + 1), khi);
                if (lo > hi) { lo = kFarLo; hi = kFarHi; }
                elo = min(min(lo, min(r1.x, r2.x)), min(r3.x, r4.x));
                ehi = max(max(hi, max(r1.y, r2.y)), max(r3.y, r4.y));
                if (elo > ehi) end_as(kRejected);   // no source left: the end cell is lost
                else if (ehi - elo + 3 > W) end_as(kCap);
            }
            int w = run ? ehi - elo + 1 : 0;
            if (run && (filled + (uint32_t)w > r.hist_entries || (uint32_t)s >= r.table_rows)) { end_as(kCap); w = 0; }
            const int rows = G == 32 ? w : __reduce_max_sync(kFull, w);
            if (P == 1 ? !run : rows == 0) break;
            const uint32_t odd = (uint32_t)(s & 1);
            uint32_t* jw = jd + odd * (W * P);
            uint32_t* jr = jd + (odd ^ 1u) * (W * P);
            if (run) {   // diagonals that come in: nothing there yet
                const int below = max(zlo - (elo - 1), 0), come = below + max(ehi + 1 - zhi, 0);
                for (int i = gl; i < come; i += G) {
                    const int at = ((i < below ? elo - 1 + i : ehi + 1 - (i - below)) & wm) * P;
                    mh[at] = make_uint2(~0u, ~0u);
                    jr[at] = ~0u;
                }
                zlo = elo - 1; zhi = ehi + 1;
                if (gl == 0) table[s] = make_int2(elo, (int)filled);
            }
            __syncwarp();
            int vlo = 1 << 30, vhi = -(1 << 30), dmin = 1 << 30, dmax = -(1 << 30);
            hit = false;
            uint32_t* hrow = hist + filled;
            for (int tb = 0; tb < rows; tb += G) {
                const int t = tb + gl;
                if (t < w) {
                    const int k = elo + t, at = (k & wm) * P;
                    const uint32_t left = jr[((k - 1) & wm) * P], right = jr[((k + 1) & wm) * P];
                    const uint2 h4 = mh[at];
                    const bool in = k >= lo && k <= hi;
                    const int hmax = min(m, n + k);   // >= 0: rows stay inside the matrix
                    const int mo = prmt(h4.x, h4.y, r.sel_o);
                    int mis = prmt(h4.x, h4.y, r.sel_x);
                    int ins = prmt(right, 0u, 0x9910u), del = prmt(left, 0u, 0xbb32u);
                    mis = in && (unsigned)mis < (unsigned)hmax ? mis + 1 : -1;
                    del = in && (unsigned)del < (unsigned)hmax ? del + 1 : -1;
                    ins = in && ins <= hmax ? ins : -1;
                    int mv = max(mis, max(ins, del));
                    const uint32_t src = mis == mv ? 0u : ins == mv ? 1u : 2u;
                    cells += in;
                    if (mv >= 0) {
                        const int rem = hmax - mv;
                        const uint32_t x = window16<P>(sp, mv - k) ^ window16<P>(st, mv);
                        int len = min(__clz((int)x) >> 1, rem);
                        ++windows;
                        if (x == 0 && rem > 16) {
                            len = 16 + match_on<P>(sp, st, mv - k + 16, mv + 16, rem - 16);
                            windows += (uint32_t)len >> 5;
                        }
                        mv += len;
                        vlo = min(vlo, k);
                        vhi = max(vhi, k);
                        const int dist = max(n + k, m) - mv;   // max(n - v, m - h)
                        dmin = min(dmin, dist);
                        dmax = max(dmax, dist);
                        hit |= k == kend && mv >= m;
                    }
                    mh[at] = make_uint2((uint32_t)prmt((uint32_t)mv, h4.x, 0x5410u), (uint32_t)prmt(h4.x, h4.y, 0x5432u));
                    jw[at] = (uint32_t)prmt((uint32_t)max(mo, ins), (uint32_t)max(mo, del), 0x5410u);
                    smo[at] = (uint16_t)mo;
                    hrow[t] = word_of(mv, src, ins >= max(mo, 0), del >= max(mo, 0));
                }
            }
            // the range of valid entries from both ends of the row, and the distances from both ends of 0 .. 65,535
            // (reads and targets are at most 32,000)
            const uint32_t ends = least2(vlo <= vhi ? (uint32_t)(vlo - elo) | ((uint32_t)(ehi - vhi) << 16) : 0xffffffffu);
            const uint32_t dist = least2(vlo <= vhi ? (uint32_t)dmin | ((uint32_t)(0xffff - dmax) << 16) : 0xffffffffu);
            hit = (__ballot_sync(kFull, hit) & pair_lanes) != 0;
            const bool any = (ends & 0xffffu) != 0xffffu;   // the row holds a valid entry
            vlo = elo + (int)(ends & 0xffffu);
            vhi = any ? ehi - (int)(ends >> 16) : vlo - 1;
            dmin = (int)(dist & 0xffffu);
            dmax = 0xffff - (int)(dist >> 16);
            bool prune = run && !hit && any && vhi - vlo + 1 >= a.adapt_min_len && dmax - dmin > a.adapt_max_dist;
            __syncwarp();
            // from each end, G diagonals at a time, up to the first one kept: the others lose their M~, and their J
            // and K are as if there were no I~, D~
            for (int side = 0; side < 2; ++side) {
                bool look = prune;
                while (__any_sync(kFull, look)) {
                    const int k = side == 0 ? vlo + gl : vhi - gl;
                    const int at = (k & wm) * P;
                    bool keep = false;
                    const bool mine = look && k >= vlo && k <= vhi;
                    if (mine) {
                        const int mv = (int16_t)(uint16_t)mh[at].x;
                        keep = mv >= 0 && max(n + k, m) - mv - dmin <= a.adapt_max_dist;
                    }
                    const uint32_t kept = __ballot_sync(kFull, keep) & pair_lanes;
                    const int first = kept ? (__ffs((int)kept) - 1) / P : G;   // lanes before the first one kept
                    if (mine && gl < first) {
                        mh[at].x |= 0xffffu;
                        const uint32_t mo = smo[at];
                        jw[at] = mo | (mo << 16);
                        hist[filled + (uint32_t)(k - elo)] = kNoWord;
                    }
                    if (look) {
                        if (side == 0) vlo += first;
                        else vhi -= first;
                        look = !kept && vlo <= vhi;
                    }
                }
            }
            __syncwarp();
            if (run) {
                rc[4] = rc[3]; rc[3] = rc[2]; rc[2] = rc[1]; rc[1] = rc[0];
                rc[0] = vlo <= vhi ? make_int2(vlo, vhi) : make_int2(kFarLo, kFarHi);
                if (gl == 0) {
                    const int at = ((elo - 1) & wm) * P;
                    mh[at] = make_uint2(~0u, ~0u);
                    jw[at] = ~0u;
                }
                if (gl == 1 % G) {
                    const int at = ((ehi + 1) & wm) * P;
                    mh[at] = make_uint2(~0u, ~0u);
                    jw[at] = ~0u;
                }
                filled += (uint32_t)w;
                if (hit) end_as(kDone);
            }
            __syncwarp();
        } while (P == 1 ? run : !__any_sync(kFull, over));
        if (over) settle();
    }
    finish();
    warp_stat_add(a.O.stats, 0, st_cells, (uint32_t)lane);
    warp_stat_add(a.O.stats, 1, st_windows, (uint32_t)lane);
    warp_stat_add(a.O.stats, 3, st_pairs, (uint32_t)lane);
}

constexpr size_t kAdaptSmem = 226u << 10;    // dynamic shared memory a block may use
constexpr int kAdaptDiagonals = 48;          // history: diagonals per score that a pair has room for on average

uint32_t adapt_seq_words(uint32_t max_length) { return 2 * ((max_length + 31) / 32) + 2; }

// W: room for diagonals as far behind as the rule keeps, on both sides, unless the limit keeps wavefronts narrower.  At
// distance 50 none of 200,000 pairs of 1,000 bp, 5 %, outgrows 128; 4.7 % outgrow 64, and over half at 10 kbp.
uint32_t adapt_width(const WfaPlan& p) {
    const int64_t need = std::min<int64_t>(2 * (int64_t)p.adapt_max_dist + 28, 2 * std::max<int64_t>(p.smax - (p.oe - p.e), 0) + 8);
    uint32_t w = 16;
    while (w < need && w < 4096) w *= 2;
    return w;
}

size_t adapt_smem(const WfaPlan& p, int G, uint32_t max_length) {
    const size_t P = 32 / G, W = adapt_width(p);
    return align_up(P * (W * 18 + 8 * (size_t)adapt_seq_words(max_length)), 16);
}
size_t adapt_entries(const WfaPlan& p) { return ((size_t)p.smax + 1) * std::min<size_t>(adapt_width(p), kAdaptDiagonals) + adapt_width(p); }
size_t adapt_table(const WfaPlan& p) { return align_up(((size_t)p.smax + 1) * 8, 256); }
size_t adapt_place(const WfaPlan& p) { return align_up(adapt_table(p) + adapt_entries(p) * 4, 256); }
size_t adapt_warp(const WfaPlan& p, int G) { return align_up(32 * p.runs_bytes + adapt_place(p) * (32 / G) + 1024, 256); }

bool adapt_fits(const WfaPlan& p, int G, uint32_t max_length, size_t scratch_bytes) {
    return kAdaptWarps * adapt_smem(p, G, max_length) <= kAdaptSmem && kAdaptWarps * adapt_warp(p, G) <= scratch_bytes;
}

}  // namespace

// Lanes per pair, and where this kernel may be used (api.cu says where it is).  Ranges vary from pair to pair, and rows of
// one warp's pairs wait for the widest, so fewer lanes than 8 lose more than they save; beyond 2,048 bp a pair has its warp
// to itself, and its history in 4 bytes an entry instead of 8 lets more of them run.  Measured, ms, wfa.cu / here: 200k x
// 1,000 bp, 5 %, 14.6 / 13.9 (pairs of a warp in step 13.5; 4 lanes so 20.2, 32 lanes 20.6), 200-1,000 bp 7.49 / 7.36 (in
// step 8.95), on 1 GiB 23.4 / 15.8 (14.6); 4k x 10 kbp 13.3 / 6.3.  wfa.cu's warp per pair stays ahead on short reads (1M x
// 150 bp, 5 %, 7.3 / 8.1) and where the pairs do not fill the device (3,000 x 1,000 bp 0.40 / 0.47; 246 x 4,905 bp 1.06 /
// 1.30).  Refills once two of four groups wait, and rows that start on sectors, measured worse (14.15, 13.9).
int adapt_group(const WfaPlan& p, uint32_t max_length, uint32_t num_pairs, int num_sms, size_t scratch_bytes) {
    const int O = p.oe - p.e;
    if (p.e != 1 || O < 1 || O > 4 || p.x > 4 || max_length > kMaxWfaLength16 || p.smax >= (1 << 20)) return 0;
    const int G = max_length <= 2048 ? 8 : 32;
    const uint64_t enough = (uint64_t)num_sms * (G == 8 ? 128 : 16);
    return max_length >= 768 && num_pairs >= enough && adapt_fits(p, G, max_length, scratch_bytes) ? G : 0;
}

bool adapt_group_fits(const WfaPlan& p, int G, uint32_t max_length, size_t scratch_bytes) {
    return (G == 8 || G == 32) && adapt_fits(p, G, max_length, scratch_bytes);
}

cudaError_t launch_wfa_adapt(const WfaPlan& plan, int G, const PairsView& P, const LimitView& L, const OutView& O,
                             uint8_t* scratch, size_t scratch_bytes, uint32_t* counter, int num_sms, cudaStream_t st,
                             int* warps_used) {
    *warps_used = 0;
    if (P.num_pairs == 0) return cudaSuccess;
    AdaptArgs r{};
    WfaArgs& a = r.w;
    a.X = plan.x; a.OE = plan.oe; a.E = plan.e; a.g = plan.g; a.smax = plan.smax; a.band = plan.band;
    a.P = P; a.L = L; a.O = O;
    a.scratch = scratch;
    a.runs_bytes = plan.runs_bytes; a.runs_cap = (uint32_t)plan.runs_cap;
    a.counters = counter; a.nbuckets = 1;
    a.adapt_min_len = plan.adapt_min_len; a.adapt_max_dist = plan.adapt_max_dist;
    r.width = adapt_width(plan);
    r.seq_words = adapt_seq_words(P.max_length);
    r.smem_warp = (uint32_t)adapt_smem(plan, G, P.max_length);
    r.table_rows = (uint32_t)plan.smax + 1;
    r.table_bytes = adapt_table(plan);
    r.hist_entries = (uint32_t)adapt_entries(plan);
    r.place_units = (uint32_t)(adapt_place(plan) >> 8);
    auto sel = [](int d) { const uint32_t b = 2u * (uint32_t)(d - 1); return b | ((b + 1) << 4) | ((b + 9) << 8) | ((b + 9) << 12); };
    r.sel_x = sel(plan.x);
    r.sel_o = sel(plan.oe - plan.e);
    void (*kernel)(AdaptArgs) = G == 8 ? wfa_adapt_kernel<8> : wfa_adapt_kernel<32>;
    const size_t smem = (size_t)kAdaptWarps * r.smem_warp, min_warp = adapt_warp(plan, G);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAdaptSmem);
    if (e != cudaSuccess) return e;
    int bps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, 32 * kAdaptWarps, smem);
    if (e != cudaSuccess) return e;
    if (bps < 1) return cudaSuccess;
    size_t warps = std::min((size_t)num_sms * bps * kAdaptWarps, scratch_bytes / min_warp);
    warps = std::min(warps, ((size_t)P.num_pairs * G + 31) / 32);
    if (warps == 0) return cudaSuccess;
    a.nwarps = (uint32_t)warps;
    a.warp_bytes = std::min(scratch_bytes / warps & ~(size_t)255, min_warp + (size_t)(G - 1) * (32 / G) * adapt_place(plan));
    kernel<<<(unsigned)((warps + kAdaptWarps - 1) / kAdaptWarps), 32 * kAdaptWarps, smem, st>>>(r);
    e = cudaGetLastError();
    if (e == cudaSuccess) *warps_used = (int)warps;
    return e;
}

}  // namespace aim
