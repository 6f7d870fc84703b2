// Rows of a wavefront history: which positions row s of a pair covers, and where it starts when rows lie end to end.
// Plain arithmetic for the host and the device (and for a test without either's compiler).
#pragma once

#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define AIM_ROWS __host__ __device__ __forceinline__
#else
#define AIM_ROWS inline
#endif

namespace aim {

AIM_ROWS int least_of(int a, int b) { return a < b ? a : b; }
AIM_ROWS int most_of(int a, int b) { return a > b ? a : b; }

// A pair's ring: diagonal k at position k - koff, position 1 the window's first diagonal and `last` its last one;
// diagonal 0 at `zero`, the end diagonal at `end`.  Row s covers lo(s) .. hi(s).
struct Window {
    int koff, last, zero, end, S;
    AIM_ROWS int lo(int s, int O) const { return most_of(most_of(zero - most_of(s - O, 0), end - (S - s)), 1); }
    AIM_ROWS int hi(int s, int O) const { return least_of(least_of(zero + most_of(s - O, 0), end + (S - s)), last); }
};

// The window of a pair of n read and m target bases under scaled limit S (|m - n| no wider than the band or the limit
// allows): 2 O + k + (k - kend) <= S beyond both 0 and kend = m - n, and likewise on the other side.
AIM_ROWS Window window_of(int n, int m, int S, int O, int band) {
    const int kend = m - n;
    int right = least_of(most_of(most_of(0, kend), (S - 2 * O + kend) >> 1), m);
    int left = least_of(most_of(most_of(0, -kend), (S - 2 * O - kend) >> 1), n);
    if (band >= 0) { right = least_of(right, band); left = least_of(left, band); }
    return Window{-left - 1, left + right + 1, left + 1, kend + left + 1, S};
}

// Rows end to end: row c at the sum of hi(i) - lo(i) + 1 over i < c.  lo(i) is zero - min(g, zero - 1), g = max(i - O, 0),
// up to row turn_lo and the line end - S + i from there on (the first does not grow with i, the second does); hi(i)
// likewise.  The sums are taken modulo 2^32: a unit's history holds fewer entries (rows of a window times the largest
// limit, 13,461 x 160,005), and the halved products stay below that too: 2 rows up to 2 S, a line of at most a window's rows.
struct DenseRows {
    int O, turn_lo, turn_hi;
    uint32_t zero, last, end, S, sum_lo, sum_hi;   // the sums of lo, hi up to those rows
    // sum of min(t, a) over t = 1 .. u
    static AIM_ROWS uint32_t ramp(int u, uint32_t a) {
        const uint32_t v = u > 0 ? (uint32_t)u : 0u, q = v < a ? v : a;
        return q * (q + 1) / 2 + (v - q) * a;
    }
    AIM_ROWS uint32_t early_lo(int c) const { return (uint32_t)c * zero - ramp(c - 1 - O, zero - 1); }
    AIM_ROWS uint32_t early_hi(int c) const { return (uint32_t)c * zero + ramp(c - 1 - O, last - zero); }
    AIM_ROWS DenseRows(const Window& w, int o)
        : O(o), zero((uint32_t)w.zero), last((uint32_t)w.last), end((uint32_t)w.end), S((uint32_t)w.S) {
        turn_lo = most_of(least_of(w.zero + w.S - w.end, (w.zero + o + w.S - w.end) >> 1), 1 - w.end + w.S);
        turn_hi = most_of(least_of(w.end + w.S - w.zero, (w.end + w.S - w.zero + o) >> 1), w.end + w.S - w.last);
        sum_lo = early_lo(turn_lo + 1);
        sum_hi = early_hi(turn_hi + 1);
    }
    AIM_ROWS uint32_t start(int c) const {
        const int dl = c - 1 - turn_lo, dh = c - 1 - turn_hi;
        const uint32_t ul = (uint32_t)dl, uh = (uint32_t)dh;
        const uint32_t lo = dl <= 0 ? early_lo(c) : sum_lo + ul * (end - S) + ((uint32_t)(c + turn_lo) * ul >> 1);
        const uint32_t hi = dh <= 0 ? early_hi(c) : sum_hi + uh * (end + S) - ((uint32_t)(c + turn_hi) * uh >> 1);
        return hi - lo + (uint32_t)c;
    }
};

// entries of rows 0 .. S of any pair whose ring takes `width` positions, two of them padding: row s has at most s - O
// diagonals on either side of 0 and S - s of the end diagonal, inside the window
inline size_t dense_entries(int64_t S, int64_t O, int64_t width) {
    size_t n = 0;
    for (int64_t s = 0; s <= S; ++s) {
        const int64_t up = 2 * (s > O ? s - O : 0), down = 2 * (S - s);
        const int64_t w = (up < down ? up : down) + 1;
        n += (size_t)(w < width - 2 ? w : width - 2);
    }
    return n;
}

}  // namespace aim

#undef AIM_ROWS
