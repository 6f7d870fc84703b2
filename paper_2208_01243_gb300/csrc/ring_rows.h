// What wfa_ring.cu's memory is sized by: the window and rows of a pair, where a row starts when rows lie end to end, and
// the work and width classes of batch plans with what each says of its pairs.  The kernel does not check its rows against
// its memory again (checks in its loop over rounds cost 2 % by the registers they took), so this is plain arithmetic, kept
// apart for a test that takes it through every kind of pair without a GPU.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define AIM_ROWS __host__ __device__ __forceinline__
#else
#define AIM_ROWS inline
#endif

namespace aim {

#ifdef __CUDACC__
AIM_ROWS int least_of(int a, int b) { return min(a, b); }
AIM_ROWS int most_of(int a, int b) { return max(a, b); }
#else
AIM_ROWS int least_of(int a, int b) { return a < b ? a : b; }
AIM_ROWS int most_of(int a, int b) { return a > b ? a : b; }
#endif

// A pair's ring: diagonal k at position k - koff, position 1 the window's first diagonal and `last` its last one;
// diagonal 0 at `zero`, the end diagonal at `end`.  Row s covers lo(s) .. hi(s).
struct Window {
    int koff, last, zero, end, S;
    AIM_ROWS int lo(int s, int O) const { return most_of(most_of(zero - most_of(s - O, 0), end - (S - s)), 1); }
    AIM_ROWS int hi(int s, int O) const { return least_of(least_of(zero + most_of(s - O, 0), end + (S - s)), last); }
};

// Diagonals beyond 0 and `end` on the end's side that can lie on an alignment within scaled limit S, of `most` that the
// matrix has: 2 O + k + (k - end) <= S, and no fewer than reach the end.
AIM_ROWS int reach(int end, int most, int S, int O, int band) {
    const int k = least_of(most_of(most_of(0, end), (S - 2 * O + end) >> 1), most);
    return band >= 0 ? least_of(k, band) : k;
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
    const int64_t n = S - O, c = width - 3, a = c / 2;   // t = s - O rises to n; beside the middle one, 2 t or 2 (n - t), at most c
    const auto half = [&](int64_t k) -> int64_t {        // sum of min(2 t, c) over t = 0 .. k
        return k < 0 ? 0 : k <= a ? k * (k + 1) : a * (a + 1) + (k - a) * c;
    };
    return (size_t)(S + 1 + (n > 0 ? half(n / 2) + half(n - n / 2 - 1) : 0));
}

// Buckets of batch plans: with W = min(2 S / E + 3, n + m + 1, 2 band + 1) and C = (S + 1) W, bucket
// (kWorkClasses - 1 - kc) kWidthClasses + kWidthClasses - 1 - wc holds the pairs of work class kc = log2(C + 1) / 3 and width
// class wc, W <= 64, 128, 256 or more.
constexpr int kWidthClasses = 4;
constexpr int kWorkClasses = 8;

AIM_ROWS int work_bucket(int64_t n, int64_t m, int64_t S, int E, int band) {
    int64_t W = 2 * (S / E) + 3;
    if (n + m + 1 < W) W = n + m + 1;
    if (band >= 0 && 2 * (int64_t)band + 1 < W) W = 2 * (int64_t)band + 1;
    const uint64_t C = (uint64_t)(S + 1) * (uint64_t)W;
    const int wc = W <= 64 ? 0 : W <= 128 ? 1 : W <= 256 ? 2 : 3;
#ifdef __CUDA_ARCH__
    const int zeros = __clzll((long long)(C + 1));
#else
    const int zeros = __builtin_clzll(C + 1);
#endif
    const int kc = (63 - zeros) / 3;
    return (kWorkClasses - 1 - least_of(kc, kWorkClasses - 1)) * kWidthClasses + (kWidthClasses - 1 - wc);
}

// No pair of bucket b has a window of more diagonals, or a larger scaled limit (0: the bucket says nothing).  With
// C = (S + 1) W < 2^(3 (kc + 1)) - 1 and the window at most W: W is at most 64 / 128 / 256 in the narrower width classes, and
// at most sqrt(2 C) + 1 in the widest (W <= 2 S + 3, so C >= W (W - 1) / 2); S + 1 is C over the class's least W.
inline void bucket_limits(int b, int64_t* diagonals, int64_t* scores) {
    const int kc = kWorkClasses - 1 - b / kWidthClasses;
    const int wc = kWidthClasses - 1 - b % kWidthClasses;
    const int64_t cmax = ((int64_t)1 << (3 * (kc + 1))) - 2;
    *diagonals = *scores = 0;
    if (wc < kWidthClasses - 1) *diagonals = (int64_t)64 << wc;
    else if (kc < kWorkClasses - 1) *diagonals = (int64_t)std::sqrt(2.0 * (double)cmax) + 2;
    const int64_t wmin = wc == 0 ? 1 : ((int64_t)32 << wc) + 1;
    if (kc < kWorkClasses - 1) *scores = cmax / wmin > 1 ? cmax / wmin : 1;
}

}  // namespace aim

#undef AIM_ROWS
