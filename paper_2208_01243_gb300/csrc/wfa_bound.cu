// Bound passes: a pruned forward pass whose end score bounds a pair's optimum from above (see wfa.cu), with one pair
// per lane where the batch fills the device that way and a warp's 32 pairs keep their sequences in shared memory, else
// with one pair per warp.
//
// The pass follows the best alignment with a window of nine diagonals kept whole in registers, in wfa_ring.cu's form
// (M~ of the last four scores, J and K per diagonal; E == 1, X and O up to 4): no range, record or reduction, and
// neighbours are the lane's own registers.  After a score the window moves one diagonal towards the entry closest to
// the end, by max(n - v, m - h), once that entry is two diagonals off its centre.  What leaves the window is lost and
// what enters it starts invalid, so every value is an offset that some alignment of that cost reaches, and the score
// at which the closest entry has nothing left is the cost of an alignment.  A pair whose window loses the end by its
// limit gets no bound (-1), and its exact pass runs under the limit alone.
// Pairs end at scores far apart, so idle lanes take new pairs while the others carry on (kRefill).  1M pairs of
// 100-1,000 bp, 1-10 %: 3.8 ms in step with the slowest lane (16 of 32 lanes at work), 2.3 ms with refills; wfa.cu's
// groups of four lanes took about 11 ms over the same pairs.  That form runs 400 instructions a score for 32 pairs with the
// few warps that their copies leave room for (1.3 per cycle, 14 of 32 lanes at work over 50k pairs); a warp per pair is
// bound by one score's chain of loads and shuffles, about 0.15 us (0.66 per cycle): 4,000 pairs of 1-10 kbp in
// 11.0 ms all told (14.3 with wfa.cu's 32-lane groups, 14.2 without a bound pass; 16 lanes a pair and a window of 16
// diagonals, which loses the end more often, 11.8), a server's burst of 24 requests in 31 ms (36).
#include <algorithm>
#include <cstdint>

#include "wfa_common.cuh"

namespace aim {
namespace {

constexpr int kBoundWarps = 2;    // per block
constexpr int kWin = 9, kMid = kWin / 2;
constexpr int kRefill = 8;        // idle lanes that call for a refill

struct BoundArgs {
    WfaArgs w;
    uint32_t seq_words;
    uint32_t smem_warp;
    uint32_t sel_x, sel_o;
};

extern __shared__ __align__(16) uint8_t s_bound[];

__global__ void __launch_bounds__(32 * kBoundWarps) wfa_bound_kernel(BoundArgs r) {
    const WfaArgs& a = r.w;
    const int lane = (int)(threadIdx.x & 31);
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gwarp >= a.nwarps) return;
    uint32_t* sp = reinterpret_cast<uint32_t*>(s_bound + (size_t)(threadIdx.x >> 5) * r.smem_warp) + 32 + lane;
    uint32_t* st = sp + r.seq_words * 32;
    const int O = a.OE - 1;
    const uint32_t begin = a.bounds ? a.bounds[0] : 0;
    const uint32_t end = a.bounds ? a.bounds[1] : a.P.num_pairs;
    uint32_t ml[kWin], mu[kWin], jk[kWin];   // M~ of scores s-1, s-2 and s-3, s-4; J, K
#pragma unroll
    for (int i = 0; i < kWin; ++i) ml[i] = mu[i] = jk[i] = ~0u;
    uint32_t pi = 0, cells = 0, windows = 0;
    int n = 0, m = 0, S = 0, klo = 0, khi = 0, s = 0;
    int mid = 0;        // the window's middle diagonal
    bool run = false;   // this lane's pair is under way
    bool more = true;   // the queue may hold pairs
    unsigned long long st_cells = 0, st_windows = 0;

    for (;;) {
        // new pairs for the idle lanes once there are eight of them: pairs end at very different scores, and a refill
        // costs the warp as much for one lane as for many
        const uint32_t idle = __ballot_sync(kFull, !run);
        if (more && __popc(idle) >= kRefill) {
            uint32_t pos = 0;
            if (lane == 0) pos = atomicAdd(a.counters, (uint32_t)__popc(idle));
            pos = __shfl_sync(kFull, pos, 0);
            more = begin < end && pos + (uint32_t)__popc(idle) < end - begin;
            const uint32_t q = pos + (uint32_t)__popc(idle & ((1u << lane) - 1u));
            bool fresh = !run && begin < end && q < end - begin;
            if (fresh) {
                pi = a.order ? a.order[begin + q] : begin + q;
                n = (int)a.P.read_len[pi];
                m = (int)a.P.target_len[pi];
                const int kend = m - n;
                const int64_t lim = pair_limit(a.L, pi);
                const int64_t S64 = lim / a.g;
                S = (int)(S64 > a.smax ? a.smax : S64);
                klo = a.band >= 0 ? max(-n, -a.band) : -n;
                khi = a.band >= 0 ? min(m, a.band) : m;
                // (the exact pass reports the others)
                fresh = !pair_bad(a.P, pi) && (uint32_t)n <= a.P.max_length && (uint32_t)m <= a.P.max_length && lim != -2 &&
                        kend >= klo && kend <= khi && (kend == 0 || abs(kend) + O <= S);
                if (!fresh) a.bound[pi] = -1;
            }
            if (fresh) {
                const uint64_t* Pw = read_words(a.P, pi);
                const uint64_t* Tw = target_words(a.P, pi);
#pragma unroll 4
                for (int w = 0; w < (n + 31) >> 5; ++w) {
                    const uint64_t x = __ldg(Pw + w);
                    sp[2 * w * 32] = (uint32_t)(x >> 32); sp[(2 * w + 1) * 32] = (uint32_t)x;
                }
#pragma unroll 4
                for (int w = 0; w < (m + 31) >> 5; ++w) {
                    const uint64_t x = __ldg(Tw + w);
                    st[2 * w * 32] = (uint32_t)(x >> 32); st[(2 * w + 1) * 32] = (uint32_t)x;
                }
                const int m0 = match_on<32>(sp, st, 0, 0, min(n, m));
#pragma unroll
                for (int i = 0; i < kWin; ++i) ml[i] = mu[i] = jk[i] = ~0u;
                ml[kMid] = (uint32_t)m0 | 0xffff0000u;
                mid = 0;
                s = 0;
                ++cells; ++windows;
                run = true;
                if (n == m && m0 == m) { a.bound[pi] = 0; run = false; }
            }
            __syncwarp();
        }
        if (!__any_sync(kFull, run)) {
            if (more) continue;
            break;
        }
        // one score of every pair under way
        int move = 0;
        if (run) {
            ++s;
            if (s > S) { a.bound[pi] = -1; run = false; }
        }
        if (run) {
            uint32_t before = ~0u;   // J, K of the diagonal below, from score s-1
            int best = 1 << 30;      // (distance to the end) * 16 + place
#pragma unroll
            for (int i = 0; i < kWin; ++i) {
                const int k = mid - kMid + i;
                const uint32_t left = before, right = i + 1 < kWin ? jk[i + 1] : ~0u;
                before = jk[i];
                const bool in = k >= klo && k <= khi;
                const int hmax = in ? min(m, n + k) : -1, room = max(hmax, 0);
                const int mo = prmt(ml[i], mu[i], r.sel_o);
                int mis = prmt(ml[i], mu[i], r.sel_x);
                int ins = prmt(right, 0u, 0x9910u), del = prmt(left, 0u, 0xbb32u);
                mis = (unsigned)mis < (unsigned)room ? mis + 1 : -1;
                del = (unsigned)del < (unsigned)room ? del + 1 : -1;
                ins = ins <= hmax ? ins : -1;
                int mv = max(mis, max(ins, del));
                if (mv >= 0) {
                    const int rem = hmax - mv;
                    const uint32_t x = window16<32>(sp, mv - k) ^ window16<32>(st, mv);
                    int len = min(__clz((int)x) >> 1, rem);
                    ++windows;
                    if (x == 0 && rem > 16) {
                        len = 16 + match_on<32>(sp, st, mv - k + 16, mv + 16, rem - 16);
                        windows += (uint32_t)len >> 5;
                    }
                    mv += len;
                    best = min(best, (max(n + k, m) - mv) * 16 + i);
                }
                mu[i] = (uint32_t)prmt(ml[i], mu[i], 0x5432u);
                ml[i] = (uint32_t)prmt((uint32_t)mv, ml[i], 0x5410u);
                jk[i] = (uint32_t)prmt((uint32_t)max(mo, ins), (uint32_t)max(mo, del), 0x5410u);
            }
            cells += kWin;
            if (best < 16) { a.bound[pi] = s; run = false; }   // nothing left on either sequence
            else if (best < (1 << 30)) move = (best & 15) >= kMid + 2 ? 1 : (best & 15) <= kMid - 2 ? -1 : 0;
        }
        if (__any_sync(kFull, move != 0)) {
            mid += move;
            uint32_t l = ~0u, u = ~0u, j = ~0u;   // the place below, before it moved
#pragma unroll
            for (int i = 0; i < kWin; ++i) {
                const uint32_t nl = i + 1 < kWin ? ml[i + 1] : ~0u, nu = i + 1 < kWin ? mu[i + 1] : ~0u,
                               nj = i + 1 < kWin ? jk[i + 1] : ~0u;
                const uint32_t cl = ml[i], cu = mu[i], cj = jk[i];
                ml[i] = move > 0 ? nl : move < 0 ? l : cl;
                mu[i] = move > 0 ? nu : move < 0 ? u : cu;
                jk[i] = move > 0 ? nj : move < 0 ? j : cj;
                l = cl; u = cu; j = cj;
            }
        }
        if (cells >= 1u << 30) { st_cells += cells; st_windows += windows; cells = windows = 0; }
    }
    st_cells += cells;
    st_windows += windows;
    warp_stat_add(a.O.stats, 0, st_cells, (uint32_t)lane);
    warp_stat_add(a.O.stats, 1, st_windows, (uint32_t)lane);
}

// The same with a warp per pair, one diagonal of the window in each lane: neighbours come by shuffles, and a score costs
// a pair 32 lanes' instructions but one entry's latency.  The window moves every kLook scores, to have the entry closest
// to the end in its middle.
constexpr int kLook = 4;

__global__ void __launch_bounds__(32 * kBoundWarps) wfa_bound_group_kernel(BoundArgs r) {
    const WfaArgs& a = r.w;
    const int lane = (int)(threadIdx.x & 31);
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gwarp >= a.nwarps) return;
    uint32_t* sp = reinterpret_cast<uint32_t*>(s_bound + (size_t)(threadIdx.x >> 5) * r.smem_warp);
    uint32_t* st = sp + r.seq_words;
    const int O = a.OE - 1;
    const uint32_t begin = a.bounds ? a.bounds[0] : 0;
    const uint32_t end = a.bounds ? a.bounds[1] : a.P.num_pairs;
    uint32_t ml = ~0u, mu = ~0u, jk = ~0u;   // as above
    uint32_t pi = 0, cells = 0, windows = 0;
    int n = 0, m = 0, S = 0, klo = 0, khi = 0, s = 0;
    int k = 0;          // this lane's diagonal
    bool run = false;   // the warp's pair is under way
    bool more = true;   // the queue may hold pairs
    unsigned long long st_cells = 0, st_windows = 0;

    for (;;) {
        if (!run) {
            uint32_t q = 0;
            if (lane == 0) q = atomicAdd(a.counters, 1u);
            q = __shfl_sync(kFull, q, 0);
            more = begin < end && q + 1 < end - begin;
            bool fresh = begin < end && q < end - begin;
            if (fresh) {
                pi = a.order ? a.order[begin + q] : begin + q;
                n = (int)a.P.read_len[pi];
                m = (int)a.P.target_len[pi];
                const int kend = m - n;
                const int64_t lim = pair_limit(a.L, pi);
                const int64_t S64 = lim / a.g;
                S = (int)(S64 > a.smax ? a.smax : S64);
                klo = a.band >= 0 ? max(-n, -a.band) : -n;
                khi = a.band >= 0 ? min(m, a.band) : m;
                // (the exact pass reports the others)
                fresh = !pair_bad(a.P, pi) && (uint32_t)n <= a.P.max_length && (uint32_t)m <= a.P.max_length && lim != -2 &&
                        kend >= klo && kend <= khi && (kend == 0 || abs(kend) + O <= S);
                if (!fresh && lane == 0) a.bound[pi] = -1;
            }
            __syncwarp();   // the last pair's copies have been read
            if (fresh) {
                const uint64_t* Pw = read_words(a.P, pi);
                const uint64_t* Tw = target_words(a.P, pi);
                for (int w = lane; w < (n + 31) >> 5; w += 32) {
                    const uint64_t x = __ldg(Pw + w);
                    sp[2 * w] = (uint32_t)(x >> 32); sp[2 * w + 1] = (uint32_t)x;
                }
                for (int w = lane; w < (m + 31) >> 5; w += 32) {
                    const uint64_t x = __ldg(Tw + w);
                    st[2 * w] = (uint32_t)(x >> 32); st[2 * w + 1] = (uint32_t)x;
                }
            }
            __syncwarp();
            if (fresh) {
                const int m0 = match_on<1>(sp, st, 0, 0, min(n, m));
                ml = mu = jk = ~0u;
                k = lane - 16;
                if (k == 0) ml = (uint32_t)m0 | 0xffff0000u;
                s = 0;
                ++cells; ++windows;
                run = true;
                if (n == m && m0 == m) {
                    if (lane == 0) a.bound[pi] = 0;
                    run = false;
                }
            }
        }
        if (!run) {
            if (more) continue;
            break;
        }
        if (++s > S) {
            if (lane == 0) a.bound[pi] = -1;
            run = false;
            continue;
        }
        uint32_t left = __shfl_up_sync(kFull, jk, 1), right = __shfl_down_sync(kFull, jk, 1);
        if (lane == 0) left = ~0u;
        if (lane == 31) right = ~0u;
        bool hit = false;
        int dist = 1 << 30;
        {
            const bool in = k >= klo && k <= khi;
            const int hmax = in ? min(m, n + k) : -1, room = max(hmax, 0);
            const int mo = prmt(ml, mu, r.sel_o);
            int mis = prmt(ml, mu, r.sel_x);
            int ins = prmt(right, 0u, 0x9910u), del = prmt(left, 0u, 0xbb32u);
            mis = (unsigned)mis < (unsigned)room ? mis + 1 : -1;
            del = (unsigned)del < (unsigned)room ? del + 1 : -1;
            ins = ins <= hmax ? ins : -1;
            int mv = max(mis, max(ins, del));
            if (mv >= 0) {
                const int rem = hmax - mv;
                const uint32_t x = window16<1>(sp, mv - k) ^ window16<1>(st, mv);
                int len = min(__clz((int)x) >> 1, rem);
                ++windows;
                if (x == 0 && rem > 16) {
                    len = 16 + match_on<1>(sp, st, mv - k + 16, mv + 16, rem - 16);
                    windows += (uint32_t)len >> 5;
                }
                mv += len;
                dist = max(n + k, m) - mv;   // max(n - v, m - h)
                hit = dist == 0;             // nothing left on either sequence
            }
            mu = (uint32_t)prmt(ml, mu, 0x5432u);
            ml = (uint32_t)prmt((uint32_t)mv, ml, 0x5410u);
            jk = (uint32_t)prmt((uint32_t)max(mo, ins), (uint32_t)max(mo, del), 0x5410u);
            ++cells;
        }
        if (__any_sync(kFull, hit)) {
            if (hit) a.bound[pi] = s;
            run = false;
        } else if (s % kLook == 0) {
            const int best = __reduce_min_sync(kFull, dist < (1 << 30) ? dist * 32 + lane : INT32_MAX);   // (dist <= 32,000)
            const int move = best == INT32_MAX ? 0 : (best & 31) - 16;
            const int from = lane + move;
            const bool have = from >= 0 && from < 32;
            const int src = have ? from : lane;
            const uint32_t l = __shfl_sync(kFull, ml, src), u = __shfl_sync(kFull, mu, src), j = __shfl_sync(kFull, jk, src);
            ml = have ? l : ~0u;
            mu = have ? u : ~0u;
            jk = have ? j : ~0u;
            k += move;
        }
        if (cells >= 1u << 30) { st_cells += cells; st_windows += windows; cells = windows = 0; }
    }
    st_cells += cells;
    st_windows += windows;
    warp_stat_add(a.O.stats, 0, st_cells, (uint32_t)lane);
    warp_stat_add(a.O.stats, 1, st_windows, (uint32_t)lane);
}

uint32_t bound_seq_words(uint32_t max_length) { return 2 * ((max_length + 31) / 32) + 2; }
// (a word of room before the copies: nothing reads there, an index below them would)
size_t bound_smem(uint32_t max_length) { return 128 + (size_t)bound_seq_words(max_length) * 256; }

// pairs per SM from which a lane per pair is the faster form: five warps, what 1,000 bp reads leave room for
constexpr uint32_t kLanePairs = 160;
constexpr size_t kLaneBoundSmem = 40u << 10;   // shared memory per warp: 5 warps on an SM

}  // namespace

bool bound_ok(const WfaPlan& p, uint32_t max_length) {
    const int O = p.oe - p.e;
    return p.e == 1 && O >= 1 && O <= 4 && p.x <= 4 && max_length <= kMaxWfaLength16 && p.smax < (1 << 26);
}

cudaError_t launch_wfa_bound(const WfaPlan& plan, const PairsView& P, const LimitView& L, const OutView& O,
                             const uint32_t* order, const uint32_t* bounds, uint32_t* counters, int num_sms,
                             cudaStream_t st) {
    if (P.num_pairs == 0) return cudaSuccess;
    const bool lanes = bound_smem(P.max_length) <= kLaneBoundSmem && P.num_pairs >= (uint32_t)num_sms * kLanePairs;
    BoundArgs r{};
    WfaArgs& a = r.w;
    a.X = plan.x; a.OE = plan.oe; a.E = plan.e; a.g = plan.g; a.smax = plan.smax; a.band = plan.band;
    a.P = P; a.L = L; a.O = O;
    a.order = order; a.bounds = bounds; a.counters = counters; a.nbuckets = 1;
    a.bound = plan.bound;
    r.seq_words = bound_seq_words(P.max_length);
    auto sel = [](int d) { const uint32_t b = 2u * (uint32_t)(d - 1); return b | ((b + 1) << 4) | ((b + 9) << 8) | ((b + 9) << 12); };
    r.sel_x = sel(plan.x);
    r.sel_o = sel(plan.oe - plan.e);
    const int per_warp = lanes ? 32 : 1;
    r.smem_warp = (uint32_t)(lanes ? bound_smem(P.max_length) : (size_t)r.seq_words * 8 * per_warp);
    void (*kernel)(BoundArgs) = lanes ? wfa_bound_kernel : wfa_bound_group_kernel;
    const size_t smem = (size_t)kBoundWarps * r.smem_warp;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kBoundWarps * kLaneBoundSmem));
    if (e != cudaSuccess) return e;
    int bps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, 32 * kBoundWarps, smem);
    if (e != cudaSuccess) return e;
    size_t warps = (size_t)num_sms * std::max(bps, 1) * kBoundWarps;
    warps = std::min(warps, ((size_t)P.num_pairs + per_warp - 1) / per_warp);
    a.nwarps = (uint32_t)warps;
    kernel<<<(unsigned)((warps + kBoundWarps - 1) / kBoundWarps), 32 * kBoundWarps, smem, st>>>(r);
    return cudaGetLastError();
}

}  // namespace aim
