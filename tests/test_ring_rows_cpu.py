"""Where the ring kernel's history rows lie (ring_rows.h), compiled for the CPU with overflow checks: row starts in closed
form against the sum of the rows' widths, every pair's rows within the entries that the host reserves, and its window
within the ring's width, over limits, bands, gap openings and end diagonals up to the largest that a launch can hold; the
same by what a batch plan's bucket says of its pairs."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <algorithm>
#include "ring_rows.h"
using namespace aim;
static Window window_of(int n, int m, int kend, int S, int O, int band) {
    const int right = reach(kend, m, S, O, band), left = reach(-kend, n, S, O, band);
    return Window{-left - 1, left + right + 1, left + 1, kend + left + 1, S};
}
static int64_t width_of(int64_t smax, int64_t O, int64_t band, int64_t len) {   // the host's ring width
    int64_t w = smax - O + 1;
    if (band >= 0) w = std::min<int64_t>(w, 2 * band + 1);
    return std::max<int64_t>(std::min<int64_t>(w, 2 * len + 1), 1) + 2;
}
static void check(int n, int m, int S, int O, int band, int64_t smax, int64_t len, size_t reserved) {
    const int kend = m - n;
    if ((band >= 0 && std::abs(kend) > band) || (kend && std::abs(kend) + O > S)) return;   // rejected at once
    const Window w = window_of(n, m, kend, S, O, band);
    const DenseRows d(w, O);
    uint64_t sum = 0;
    const int step = S > 20000 ? 97 : 1;
    for (int s = 0; s <= S; ++s) {
        if (s % step == 0 && d.start(s) != sum) { std::printf("start %d %d %d %d %d: row %d\n", n, m, S, O, band, s); std::exit(1); }
        const int lo = w.lo(s, O), hi = w.hi(s, O);
        if (lo < 1 || hi > w.last) { std::printf("window %d %d %d %d %d\n", n, m, S, O, band); std::exit(1); }
        sum += hi >= lo ? (uint64_t)(hi - lo + 1) : 0;
        if (hi < lo - 1) { std::printf("gap %d %d %d %d %d: row %d\n", n, m, S, O, band, s); std::exit(1); }
    }
    if (d.start(S + 1) != sum || sum >> 32 || sum > reserved || w.last + 2 > width_of(smax, O, band, len)) {
        std::printf("total %d %d %d %d %d: %llu %u of %zu, last %d\n", n, m, S, O, band, (unsigned long long)sum, d.start(S + 1),
                    reserved, w.last);
        std::exit(1);
    }
}
static void check_bucket(int n, int m, int S, int O, int band) {
    const int kend = m - n;
    if ((band >= 0 && std::abs(kend) > band) || (kend && std::abs(kend) + O > S)) return;
    int64_t diagonals, scores;
    const int b = work_bucket(n, m, S, 1, band);
    bucket_limits(b, &diagonals, &scores);
    const Window w = window_of(n, m, kend, S, O, band);
    if (b < 0 || b >= kWorkClasses * kWidthClasses || (diagonals && w.last > diagonals) || (scores && S > scores)) {
        std::printf("bucket %d of %d %d %d %d %d: %d of %lld, %d of %lld\n", b, n, m, S, O, band, w.last, (long long)diagonals, S,
                    (long long)scores);
        std::exit(1);
    }
}
static size_t counted(int64_t S, int64_t O, int64_t width) {
    size_t n = 0;
    for (int64_t s = 0; s <= S; ++s)
        n += (size_t)std::min(std::min(2 * std::max<int64_t>(s - O, 0), 2 * (S - s)) + 1, width - 2);
    return n;
}
int main() {
    for (int S = 0; S < 70; ++S)
        for (int O = 1; O <= 4; ++O)
            for (int width = 3; width < 90; ++width)
                if (dense_entries(S, O, width) != counted(S, O, width)) { std::printf("entries %d %d %d\n", S, O, width); return 1; }
    for (int O = 1; O <= 4; ++O)
        for (int band : {-1, 0, 1, 3, 9})
            for (int n = 0; n <= 12; ++n)
                for (int m = 0; m <= 12; ++m)
                    for (int smax : {0, 1, 2, 5, 9, 14, 30, 61}) {
                        const size_t reserved = dense_entries(smax, O, width_of(smax, O, band, 12));
                        for (int S = 0; S <= smax; S += 1 + S / 7) check(n, m, S, O, band, smax, 12, reserved);
                    }
    unsigned x = 7;
    auto rnd = [&](int k) { x = x * 1664525u + 1013904223u; return (int)((x >> 8) % (unsigned)k); };
    for (int i = 0; i < 400; ++i) {
        const int len = 1 + rnd(2000), smax = rnd(3000), O = 1 + rnd(4), band = rnd(3) ? -1 : rnd(300);
        const size_t reserved = dense_entries(smax, O, width_of(smax, O, band, len));
        for (int j = 0; j < 8; ++j) check(rnd(len + 1), rnd(len + 1), rnd(smax + 1), O, band, smax, len, reserved);
    }
    for (int S = 0; S < 4000; ++S)   // across every line between classes
        for (int len : {0, 1, 31, 32, 63, 64, 127, 128, 300, 3000})
            for (int band : {-1, 0, 31, 32, 63, 64, 127, 128, 1000}) check_bucket(len, len + (S & 1), S, 1 + (S & 3), band);
    for (int i = 0; i < 2000000; ++i) {
        const int len = 1 + rnd(1 << (1 + rnd(15))), S = rnd(1 << (1 + rnd(18)));
        check_bucket(rnd(len + 1), rnd(len + 1), S, 1 + rnd(4), rnd(2) ? -1 : rnd(1 << (1 + rnd(14))));
    }
    // the most a launch can hold: 32,000 bp without a threshold at mismatch 4, opening 4 (scaled), the widest band whose
    // ring fits 226 KB, and the widest limit without a band
    for (int kend : {0, 1, -1, 500, 6730, -6730}) {
        const int smax = 4 * 32000 + 4 + 32000, n = kend > 0 ? 32000 - kend : 32000, m = n + kend;
        const size_t reserved = dense_entries(smax, 4, width_of(smax, 4, 6730, 32000));
        check(n, m, smax, 4, 6730, smax, 32000, reserved);
        check(n, m, smax - 1, 4, 6730, smax, 32000, reserved);
        const int wide = 13464;
        check(n, m, wide, 4, -1, wide, 32000, dense_entries(wide, 4, width_of(wide, 4, -1, 32000)));
    }
    std::puts("ok");
}
"""


def test_row_starts_and_reserved_entries(tmp_path):
    src, exe = tmp_path / "rows.cc", tmp_path / "rows"
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all",
                           "-I", os.path.join(ROOT, "paper_2208_01243_gb300", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.stdout + r.stderr)[-2000:]
