// How many CTAs share a row of top-k.  Plain C++, so that it can be tested without a device.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define JANUS_PLAN_FN __host__ __device__ inline
#else
#define JANUS_PLAN_FN inline
#endif

namespace janus {

// CTAs that share one of `rows` rows of up to `n` elements (n < 0: the lengths are on the device).  One CTA takes 7.5 us and 0.08 us
// per thousand elements; a cluster streams its share only, but its start and its four cluster-wide barriers cost about a
// microsecond, and more once the clusters leave few SMs free.  With 1, 2, 4 and 8 CTAs, k = 2048 (us): 8 rows of 16 K 8.2, 8.7, 9.4, 9.1;
// of 24 K 9.5, 9.3, 9.3, 9.2; of 50 K 11.7, 10.7, 10.1, 9.2; of 131 K 18.2, 13.6, 11.5, 10.1; 12 rows of 33 K 10.4, 10.1, 10.0, 10.9; of 50 K
// 11.7, 10.8, 10.3, 11.0; of 131 K 17.9, 13.6, 12.1, 12.0; 24 rows of 33 K 10.4, 10.1, 12.1, 11.7; of 96 K 15.5, 12.4, 13.9, 12.8; of 131 K 18.3, 13.9, 14.2,
// 12.9; 64 rows of 50 K 12.4, 13.7, 14.5, 22.5; of 96 K 19.4, 17.2, 16.6, 25.1; 74 rows of 64 K 14.2, 11.6, 21.3, 28.9.  Rows whose length only
// the device knows get a cluster, which takes its row whole or splits it.
inline int topk_cluster_size(int64_t rows, double n) {
    const bool unknown = n < 0;
    if (rows <= 8 && (unknown || n >= 22e3)) return 8;
    if (rows <= 14 && (unknown || n >= 36e3)) return 4;
    if (rows > 14 && rows <= 30 && n >= 112e3) return 8;
    if (rows <= 37 && n >= 32e3) return 2;
    if (rows <= 74 && (unknown || n >= 64e3)) return 2;
    return 1;
}

// Elements from which a cluster of n_cta CTAs splits a row; a shorter one is taken by its first CTA as if it were alone.  The lines lie where
// that is no slower for any number of rows: 12 rows (four CTAs) of 9 K 9.6 us split and 7.9 alone, of 20 K 10.0 and 9.4, of 24 K 9.8 both; 64
// rows (two) of 9 K 10.9 and 9.9, of 16 K 11.2 both, of 20 K 12.1 and 12.4; 8 rows (eight) of 9 K 9.1 and 8.3, of 16 K 9.4 and 9.3.
JANUS_PLAN_FN int topk_split_from(int n_cta) { return n_cta == 4 ? 24000 : 18000; }

}  // namespace janus
