// Which kernels a page demand call takes, and in how many CTAs (page_demand.cu).  Host code without CUDA.
#pragma once

#include <stdint.h>

namespace janus {

constexpr int PD_THREADS = 1024;
constexpr int PD_MAX_CLUSTER = 16;
constexpr int PD_PORTABLE_CLUSTER = 8;
constexpr int PD_SMEM_WORDS = PD_MAX_CLUSTER * PD_THREADS;      // private bitmap of a CTA: up to 64 KB, half a million pages

// One launch of one cluster while it reads the indices as fast as memset, chip-wide marking and lists would (12.4 us up to 512 K
// indices): 128 K indices in 9.6 us, 256 K in 12.3, 512 K in 17.4.
constexpr int64_t PD_ONE_LAUNCH_INDICES = 1 << 17;

struct PdPlan {
    bool one_launch;      // marking and lists by one cluster; otherwise the whole chip marks first
    int cluster;          // CTAs of the cluster of page_demand_kernel
};

// `largest`: CTAs of the largest cluster that the device takes (8 always, 16 on a whole B200).
inline PdPlan page_demand_plan(int64_t n_idx, int n_words, int largest) {
    // Four CTAs up to 8 K indices (7.1 us; eight and sixteen cost 0.1 and 0.3 us more), sixteen beyond (256 x 256 8.0 us against 10.7 with
    // four and 8.6 with eight, 12 decode rows 8.4, 10.5 and 9.1, 64 rows of a 131136-page pool 17.1, 26.4 and 26.4).
    if (n_idx <= PD_ONE_LAUNCH_INDICES && n_words <= largest * PD_THREADS) {
        int cluster = n_idx <= 8192 ? 4 : largest;
        while (n_words > cluster * PD_THREADS) cluster *= 2;      // a slice is one chunk
        return {true, cluster};
    }
    return {false, n_words <= PD_PORTABLE_CLUSTER * PD_THREADS ? PD_PORTABLE_CLUSTER : largest};      // 2112 pages: 14.4 us with 8, 16.5 with 16
}

}  // namespace janus
