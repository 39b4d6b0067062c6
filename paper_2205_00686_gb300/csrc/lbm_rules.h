// Host rules that pick launch shapes.  Plain C++, so that they can be compiled
// and checked without CUDA.
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace lbm {

// Segment height of a batch without a tuned tile: the domains' strips are cut
// into segments of at most R rows, even within a domain, and the CTAs take them
// from one list, longest first, so a launch lasts about w (R + 8) iterations
// where w rounds of resident CTAs (`slots`) take all segments (a segment's sweep
// runs 6 iterations beyond its rows and starts up in about 2).  For each of 12
// round counts from the fewest that hold the uncut strips, the smallest R that
// fits; then the one that gives the shortest launch, or 64 rows where those are
// shorter (many strips next to a few tall ones: the rounds above then start far
// below what cutting the tall ones needs).  FP32 open domains, us per step: 64
// of sides 64-512, 64 rows on the register tile 222, this (73 rows, staged) 203,
// the tuner's best fixed height 208; 20 of sides 64-300 45 (19 rows), 8 of sides
// 64-200 30 (8 rows).  Iterations by the model: 10 000 of 64 x 64 with one 64 x
// 4096, 608 CTAs, 1224 (64 rows; uncut 4104).
//
// The rule runs on the host at every attach and detach.  Each round count is first
// asked whether the tallest height that would still be shorter fits, and searched
// only if so: some 30 passes over the members at most instead of 110 (512 domains
// attached one by one 100 -> 39 ms, 55 with a fixed height).  passes, if given,
// counts them.
inline int batch_rows(const int* nx, const int* ny, size_t n, int threads, long long slots, int* passes = nullptr) {
    const int W = threads - 8;
    long long strip_rows = 0;
    int most = 1;
    std::vector<int> strips(n);
    for (size_t i = 0; i < n; ++i) {
        strips[i] = (nx[i] + W - 1) / W;
        strip_rows += (long long)strips[i] * ny[i];
        most = std::max(most, ny[i]);
    }
    auto segments = [&](int R) {
        if (passes) ++*passes;
        // ceil(ny / R) by a multiplication: heights are below 2^20, so the half row
        // keeps the product off the integers by far more than its rounding
        const double inv = 1.0 / R, up = R - 0.5;
        long long s = 0;
        for (size_t i = 0; i < n; ++i) s += strips[i] * (int)((ny[i] + up) * inv);
        return s;
    };
    auto rounds = [&](long long segs) { return std::max<long long>(1, (segs + slots - 1) / slots); };
    int rows = std::min(64, most);
    long long best = rounds(segments(rows)) * (rows + 8);
    // w rounds hold the uncut strips, and w rounds of the tallest all rows
    const long long w0 = std::max(rounds(segments(most)), (strip_rows + slots * most - 1) / (slots * most));
    for (long long w = w0; w < w0 + 12; ++w) {
        // heights from the least that could fit to the last that would be shorter
        int lo = (int)std::max<long long>(std::min(8, most), (strip_rows + w * slots - 1) / (w * slots));
        int hi = (int)std::min<long long>(most, (best - 1) / w - 8);
        if (hi < lo || segments(hi) > w * slots) continue;
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (segments(mid) <= w * slots) hi = mid;
            else lo = mid + 1;
        }
        best = w * (lo + 8);
        rows = lo;
    }
    return rows;
}

}  // namespace lbm
