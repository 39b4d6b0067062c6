// Host rules that pick launch shapes.  Plain C++, so that they can be compiled
// and checked without CUDA.
#pragma once

#include <algorithm>
#include <cstddef>

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
inline int batch_rows(const int* nx, const int* ny, size_t n, int threads, long long slots) {
    const int W = threads - 8;
    long long strip_rows = 0;
    int most = 1;
    for (size_t i = 0; i < n; ++i) {
        strip_rows += (long long)((nx[i] + W - 1) / W) * ny[i];
        most = std::max(most, ny[i]);
    }
    auto segments = [&](int R) {
        long long s = 0;
        for (size_t i = 0; i < n; ++i) s += (long long)((nx[i] + W - 1) / W) * ((ny[i] + R - 1) / R);
        return s;
    };
    auto rounds = [&](long long segs) { return std::max<long long>(1, (segs + slots - 1) / slots); };
    int rows = std::min(64, most);
    long long best = rounds(segments(rows)) * (rows + 8);
    // w rounds hold the uncut strips, and w rounds of the tallest all rows
    const long long w0 = std::max(rounds(segments(most)), (strip_rows + slots * most - 1) / (slots * most));
    for (long long w = w0; w < w0 + 12; ++w) {
        int lo = std::min(8, most), hi = most;
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (segments(mid) <= w * slots) hi = mid;
            else lo = mid + 1;
        }
        const long long t = w * (lo + 8);
        if (t < best) {
            best = t;
            rows = lo;
        }
    }
    return rows;
}

}  // namespace lbm
