// Device code shared by the wavefront kernels: backward match runs, pair states, and a pair's result.
#pragma once

#include "aim_internal.cuh"

namespace aim {

// 32 bases ending at base p (inclusive) with base p in the low two bits; for
// p < 31 only bases 0..p are present (in the low bits).
__device__ __forceinline__ uint64_t window_ending(const uint64_t* w, uint32_t nwords, int p) {
    if (p >= 31) return window32(w, nwords, (uint32_t)(p - 31));
    return window32(w, nwords, 0) >> (2 * (31 - p));
}

// number of consecutive matches P[v-1-i] == T[h-1-i], i = 0, 1, ... (at most min(v, h))
__device__ __forceinline__ int match_run_back(const uint64_t* Pw, uint32_t nwP, int v, const uint64_t* Tw,
                                              uint32_t nwT, int h) {
    int run = 0;
    for (;;) {
        const int pv = v - 1 - run, ph = h - 1 - run;
        if (pv < 0 || ph < 0) break;
        const uint64_t d = window_ending(Pw, nwP, pv) ^ window_ending(Tw, nwT, ph);
        const int avail = min(min(pv, ph) + 1, 32);
        int z = d ? ((__ffsll((long long)d) - 1) >> 1) : 32;
        if (z > avail) z = avail;
        run += z;
        if (z < 32) break;
    }
    return run;
}

enum : int { kRun = 0, kDone = 1, kRejected = 2, kCap = 3, kBad = 4, kIdle = 5 };

// Result of a finished pair: score, flags, run count, and its runs (staged end-first) copied start-first by
// lanes gl, gl + G, ... of its group; every lane of the group calls this with the same values.
__device__ __forceinline__ void emit_done(const WfaArgs& a, uint32_t pi, int final_s, uint32_t nruns, bool ok,
                                          const uint32_t* staged, int gl, int G) {
    const int32_t score = final_s * a.g;
    uint8_t flags = ok ? 0 : AIM_F_STEP_CAP;
    if (ok && a.O.cigars && a.O.cigar_off) {
        const uint64_t off = a.O.cigar_off[pi];
        const uint64_t cap = a.O.cigar_off[pi + 1] - off;
        if (nruns <= cap) {
            for (uint32_t j = (uint32_t)gl; j < nruns; j += (uint32_t)G) a.O.cigars[off + j] = staged[nruns - 1 - j];
        } else {
            flags |= AIM_F_CIGAR_OVERFLOW;
        }
    }
    if (gl == 0) write_header(a.O, pi, ok ? score : -1, flags, nruns);
}

// One lane: result of a pair that ended without an alignment.
__device__ __forceinline__ void emit_failed(const WfaArgs& a, uint32_t pi, int status) {
    const uint8_t f = status == kBad ? AIM_F_BAD_PAIR : status == kRejected ? AIM_F_REJECTED : AIM_F_STEP_CAP;
    write_header(a.O, pi, -1, f, 0);
}

__device__ __forceinline__ int prmt(uint32_t a, uint32_t b, uint32_t sel) {   // sign-replicating byte permute
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return (int)r;
}

// 16 bases from position pos of a sequence copy (32-bit word i of the pair at [i * P])
template <int P>
__device__ __forceinline__ uint32_t window16(const uint32_t* s, int pos) {
    const uint32_t* w = s + (pos >> 4) * P;
    return __funnelshift_l(w[P], w[0], 2 * pos);   // the shift is taken modulo 32
}

// the match run from (v, h) on, 32 bases a turn: at most rem
template <int P>
__device__ __forceinline__ int match_on(const uint32_t* sp, const uint32_t* st, int v, int h, int rem) {
    int run = 0;
    const uint32_t* p = sp + (v >> 4) * P;
    const uint32_t* t = st + (h >> 4) * P;
    uint32_t a = p[0], c = t[0];
    do {
        const uint32_t b = p[P], d = t[P];
        const uint32_t x = __funnelshift_l(b, a, 2 * v) ^ __funnelshift_l(d, c, 2 * h);
        if (x || run + 16 >= rem) { run += __clz((int)x) >> 1; break; }   // __clz(0) = 32
        a = p[2 * P]; c = t[2 * P];
        const uint32_t y = __funnelshift_l(a, b, 2 * v) ^ __funnelshift_l(c, d, 2 * h);
        run += 16 + (__clz((int)y) >> 1);
        if (y) break;
        p += 2 * P; t += 2 * P;
    } while (run < rem);
    return min(run, rem);
}

// runs in end-first order, every `stride` words
struct RunStage {
    uint32_t* runs;
    uint32_t stride, cap, n, op, len;
    __device__ __forceinline__ void flush() {
        if (len) {
            if (n < cap) runs[n * stride] = (len << 4) | op;
            ++n;
        }
    }
    __device__ __forceinline__ void put(uint32_t o, uint32_t l) {
        if (o == op) { len += l; return; }
        flush();
        op = o; len = l;
    }
};

// Whole warp: copies each lane's `count` runs, staged end first in slot `slot` (its i-th run at slot * between + i *
// stride of staged), to its pair's place `at` in the CIGAR array, start first; half a warp takes one pair at a time.
__device__ __forceinline__ void copy_runs(const OutView& O, uint32_t count, uint64_t at, const uint32_t* staged,
                                          uint32_t between, uint32_t stride, int slot) {
    const uint32_t wl = threadIdx.x & 31, hl = wl & 15;
    for (int q = (int)(wl >> 4); q < 32; q += 2) {
        const uint32_t cnt = __shfl_sync(kFull, count, q);
        const uint64_t to = __shfl_sync(kFull, at, q);
        const uint32_t* from = staged + (size_t)(uint32_t)__shfl_sync(kFull, slot, q) * between;
        for (uint32_t i = hl; i < cnt; i += 16) O.cigars[to + i] = from[(size_t)(cnt - 1 - i) * stride];
    }
}

}  // namespace aim
