// Which kernels a page demand call takes, and in how many CTAs (page_demand.cu).  Host code without CUDA.
#pragma once

#include <stdint.h>

namespace janus {

constexpr int PD_THREADS = 1024;
constexpr int PD_MAX_CLUSTER = 16;
constexpr int PD_PORTABLE_CLUSTER = 8;
constexpr int PD_SMEM_WORDS = PD_PORTABLE_CLUSTER * PD_THREADS;      // private bitmap of a marking CTA: up to 32 KB, 262144 pages
constexpr int PD_MAX_CLUSTERS = 64;
constexpr int PD_FEW_WORDS = 256;

// One launch of one cluster while it reads the indices as fast as clearing, chip-wide marking and lists would: 128 K indices of 142 pages
// 5.7 us against 5.8, of 2112 pages 7.0 both, of 16384 pages 10.4 against 13.3, 32 K of 2112 pages 5.3 against 6.9; 64 rows with tables of their
// own over 131136 pages 16.6 against 22.0; and while its lists are as fast as those of several clusters: 131072 indices of 524288 pages
// 38.0 us in one launch, 20.4 without.
constexpr int64_t PD_ONE_LAUNCH_INDICES = 1 << 17;

struct PdPlan {
    bool few;             // the lists by one CTA, of one cluster that marks as well or alone
    bool one_launch;      // marking and lists by one cluster; otherwise the whole chip marks first
    int cluster;          // CTAs of a cluster (few lists alone need one CTA)
    int clusters;         // of the lists
};

// `largest`: CTAs of the largest cluster that the device takes (8 always, 16 on a whole B200).
inline PdPlan page_demand_plan(int64_t n_idx, int n_words, int largest) {
    // A CTA's slice of the set is one chunk, PD_THREADS words, and up to PD_FEW_WORDS words one CTA makes the lists (2048 indices of 513 pages
    // 6.8 -> 5.0 us, 19 x 2048 of 142 pages 7.7 -> 4.9, 256 x 256 of 68 pages 7.8 -> 5.0, twelve rows of 2048 over 6000 pages 8.4 -> 6.7; at 256 words
    // 7.7 -> 6.7, and 1.7 us more with every 240 words, so that the lists of a whole cluster catch up at 512).  Four CTAs for few indices in
    // such a pool (four and eight alike up to three rows of 2048; nineteen rows 7.1 with four, 5.2 with eight, 4.9 with sixteen), all the
    // device takes beyond: 2048 indices of 16384 pages 8.2 against 9.6 with four, of 131072 pages 11.8 against 19.1.
    if (n_idx <= PD_ONE_LAUNCH_INDICES && n_words <= PD_SMEM_WORDS)
        return {n_words <= PD_FEW_WORDS, true, n_idx <= 8192 && n_words <= PD_FEW_WORDS ? 4 : largest, 1};
    // Lists alone: one CTA for a small pool (whole call of 4096 x 2048 indices of 2112 pages 26.3 us with a cluster of 8, 22.7 with one CTA;
    // 2048 x 2048 of 544 pages 18.5 and 14.6); larger pools are shared by clusters, which count what lies before them: up to four while
    // each CTA has 256 words, then as many as give each one chunk.  524288 indices of 500000 pages 43.2 us with one cluster, 30.0 with
    // four; 131072 of 1048576 pages 55.6, 31.8, 23.5 and 29.3 with one, two, four and eight; of 2097152 pages 88 with one, 29.3 with four
    // and 35.7 with eight.
    if (n_words <= PD_FEW_WORDS) return {true, false, PD_PORTABLE_CLUSTER, 1};
    const auto shares = [&](int64_t words) { return (n_words + words * largest - 1) / (words * largest); };
    int64_t n = shares(256) < 4 ? shares(256) : 4;
    if (n < shares(PD_THREADS)) n = shares(PD_THREADS);
    return {false, false, largest, n < PD_MAX_CLUSTERS ? static_cast<int>(n) : PD_MAX_CLUSTERS};
}

}  // namespace janus
