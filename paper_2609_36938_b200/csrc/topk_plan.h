// How many CTAs share a row of top-k.  Plain C++, so that it can be tested without a device.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define JANUS_PLAN_FN __host__ __device__ inline
#else
#define JANUS_PLAN_FN inline
#endif

namespace janus {

// One CTA takes 7.5 us and 0.08 us per thousand elements; a cluster streams its share only, but its start and its four cluster-wide barriers
// cost about a microsecond, and more once the clusters leave few SMs free.  Microseconds with 1, 2, 4 and 8 CTAs, k = 2048:
//    8 rows of 18 K  9.0  9.4  9.4  9.3    of 24 K   9.7  9.5  9.5  9.2    of 50 K  11.8 10.8 10.2  9.3    of 131 K 18.2 13.7 11.5 10.2
//    9 rows of 24 K  9.8  9.6  9.7 10.3    of 40 K  11.1 10.2 10.4 10.3    of 50 K  11.8 10.9 10.3 10.2    of 131 K 18.1 13.7 11.5 11.5
//   14 rows of 24 K  9.9  9.7  9.6 11.0    of 40 K  11.1 10.2 10.3 11.0    of 50 K  12.2 11.1 10.4 11.1    of 131 K 18.4 13.9 11.8 12.2
//   15 rows of 28 K 10.1  9.6 10.7 10.8    of 50 K  11.9 11.0 11.5 10.9    of 96 K  15.4 12.4 12.8 11.9    of 112 K 16.8 13.5 12.9 11.9
//   24 rows of 32 K 10.4  9.7 11.5 11.8    of 50 K  12.0 10.9 12.7 11.8    of 96 K  15.7 12.6 14.0 12.9    of 112 K 16.8 13.5 14.2 13.0
//   30 rows of 32 K 10.6 10.2 12.2 11.9    of 50 K  12.2 11.2 13.4 11.9    of 96 K  15.7 12.7 14.8 13.0    of 112 K 17.0 14.0 15.2 13.1
//   31 rows of 32 K 10.2 10.9 12.2 12.0    of 50 K  12.0 11.9 13.3 12.0    of 64 K  13.0 12.0 13.3 12.0    of 112 K 17.0 15.3 15.2 13.2
//   33 rows of 64 K 13.2 12.8 13.1 12.2    of 112 K 16.9 15.7 15.1 13.5;   34 rows of 64 K 13.0 13.1 13.1 17.3    of 112 K 17.0 15.7 15.1 19.2
//   74 rows of 64 K 13.1 11.5 21.3 29.0    of 131 K 18.7 14.2 24.6 32.4;   75 rows of 64 K 14.7 14.5 21.3 29.1    of 131 K 21.5 19.0 24.7 32.5
// (31 to 36 rows lose by pairs below 64 K, 37, half of the SMs with two CTAs each, would gain.)

// CTAs that share one of `rows` rows of up to `n` elements; n < 0: only the device knows the lengths, and a cluster takes its row whole or splits
// it (topk_split_from).
inline int topk_cluster_size(int64_t rows, double n) {
    const bool unknown = n < 0;
    if (rows <= 8 && (unknown || n >= 22e3)) return 8;
    if (rows <= 14 && (unknown || n >= 45e3)) return 4;
    if (rows > 14 && rows <= 33 && n >= 112e3) return 8;
    if (rows <= 30 && n >= 32e3) return 2;
    if (rows <= 74 && (unknown || n >= 64e3)) return 2;
    return 1;
}

// Elements from which a cluster of n_cta CTAs splits a row; a shorter one is taken by its first CTA as if it were alone.  The lines lie where
// that is no slower for any number of rows: 12 rows (four CTAs) of 9 K 9.6 us split and 7.9 alone, of 20 K 10.0 and 9.4, of 24 K 9.8 both; 64
// rows (two) of 9 K 10.9 and 9.9, of 16 K 11.2 both, of 20 K 12.1 and 12.4; 8 rows (eight) of 9 K 9.1 and 8.3, of 16 K 9.4 and 9.3.
JANUS_PLAN_FN int topk_split_from(int n_cta) { return n_cta == 4 ? 24000 : 18000; }

}  // namespace janus
