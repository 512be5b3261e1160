// How knn_exact samples the rows and sizes its candidate lists: arithmetic on the host alone.
#ifndef DEG_KNN_SAMPLE_H
#define DEG_KNN_SAMPLE_H

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace deg {

constexpr int64_t kSampleMax = 65536;   // sampled rows per query, where every stride-th row is enough
constexpr int64_t kGroupsMax = 49152;   // group minima per query, at most (192 KB of shared memory)
constexpr int kCandCapMax = 8192;       // candidates per query, at most

struct SamplePlan {
    int64_t stride, ns, ng;             // every stride-th row is sampled; the sampled rows; their groups
    int32_t group, cap;                 // sampled rows per group, 16 or 64; candidates a list holds
    double expected;                    // rows at or below the threshold, on average over rows in random order
    bool filter;                        // false: the CUDA-core path takes the call
};

// The threshold of a query is the k-th smallest group minimum. With ng groups of g sampled rows, a row is below it
// with the probability F at which k of the ng groups hold one: (1 - F)^g = 1 - (k - 1/2) / ng.
//   stride  about k * stride rows fall below the threshold and the list holds twice that: every stride-th row is
//           sampled, about 65,536 of them, or more where k * stride would outgrow the longest list (at k = 1,001
//           every fourth of 1M rows);
//   group   64 (a quarter of the stores and of the selection) where 16 k groups leave the threshold as tight, or
//           where groups of 16 are too many for the selection; else 16;
//   cap     room for twice k * stride, and for the expected rows and three standard deviations;
//   filter  not where the expected rows outgrow the longest list (at k = 1,001 from 25M rows on): nearly every query
//           would be computed a second time, on the CUDA cores. With fewer groups than k every row is a candidate.
// Nor where the CUDA cores are as fast (times in us, CUDA cores | filter, 128 columns where none are given):
//   more than a quarter of the rows expected (lists of up to 1,024 stay with the filter up to k = 256):
//           16,384 rows, k = 1,024 (38%): 310 | 456 for 200 queries, 1,002 | 1,533 for 2,000; k = 800 (9%): 309 | 225,
//           1,002 | 650; 8,192 rows, k = 500 (21%): 268 | 220, 654 | 564; k = 800 (all): 274 | 505, 693 | 1,415;
//   k above 256 and at most 65,536 distances, a buffer that takes no fresh memory: 72 and 10 for each million of
//           n * dim, 1 query, k = 500: 8,192 rows 82 | 134; 20,000 96 | 138; 40,000 122 | 148; 60,000 x 32 121 | 140;
//           20,000 x 960 250 | 332; but 60,000 x 960 659 | 427. (With more distances the allocation alone is 160: 16
//           queries x 9,000, k = 500: 236 | 161.)
inline SamplePlan sample_plan(int64_t n, int64_t nq, int32_t dim, int32_t k) {
    SamplePlan p{};
    p.stride = std::min<int64_t>((n + kSampleMax - 1) / kSampleMax, std::max(1, kCandCapMax / (2 * k)));
    for (;;) {
        p.ns = (n + p.stride - 1) / p.stride;
        p.group = (p.ns + 63) / 64 >= 16 * (int64_t)k || (p.ns + 15) / 16 > kGroupsMax ? 64 : 16;
        p.ng = (p.ns + p.group - 1) / p.group;
        if (p.ng <= kGroupsMax) break;
        p.stride = (n + 64 * kGroupsMax - 1) / (64 * kGroupsMax);
    }
    double deviation = 0.0;
    p.expected = (double)n;
    if (p.ng >= k) {
        const double hit = (k - 0.5) / (double)p.ng, miss = std::pow(1.0 - hit, 1.0 / p.group);
        p.expected = (double)n * (1.0 - miss);
        deviation = (double)n * std::sqrt((double)p.ng * hit * (1.0 - hit)) / ((double)p.ng * p.group * std::pow(miss, p.group - 1));
    }
    const double room = std::max(2.0 * k * (double)p.stride, std::min((double)n, p.expected + 3.0 * deviation));
    p.cap = 1024;
    while (p.cap < kCandCapMax && p.cap < room) p.cap <<= 1;
    const bool many = p.expected > 0.25 * (double)n && (n > 1024 || k > 256);
    const bool small = k > 256 && nq * n <= 65536 && (n <= 20480 || n * dim <= (1 << 23));
    p.filter = p.expected <= kCandCapMax && !many && !small;
    return p;
}

}  // namespace deg

#endif
