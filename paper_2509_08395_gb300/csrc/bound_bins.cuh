// The bins of a query's histogram H of the candidates its windows emitted.
// Plain functions of integers, so that the host tests run the same code.
//
// H bounds what can still enter a query's answer (g candidates lie at or above
// some bin), so its bins decide how many slots below the true bound a window
// still emits: bins on 12 bits of the order key, 8 an octave, let a query of
// the 1M-document workload emit about 3 times what it has to, and had to be
// read whole by every block (16 KiB). Most bins of such a full-range table
// never fill. Here the bins hang from the largest score the query can have:
// M = its largest product bound max_j |w_j| vmax_j (a maximum, so every block
// and kernel gets the same one, in any order of the terms) times its number of
// terms, rounded up to a power of two (8 at least). Below that, non-negative
// scores have 12 octaves of 64 bins, 14 of 8 and 32 of one; bin kHRest holds the
// rest of them and zero, and the bins under it negative scores, 8 an octave of
// their magnitude. (With the top bin at 8 M for any number of terms, all answers
// over data of many similar products, as uniform or binary vectors have, lay in
// the top bin, and with one bin for zero and all negative scores answers below
// zero had no bound: 200 queries of 20 terms over 1M binary documents of 60
// entries, 500 candidates, took 3.52 ms one by one and 1.93 batched, now 1.70 and
// 0.91; with 8 bins an octave everywhere 2.04 and 1.37.)
#pragma once

#include <stdint.h>

#include "checks.cuh"  // SINDI_HD

namespace sindi {

constexpr int kHBins = 1024;  // bins of H
constexpr int kHFine = 768;   // of which from the top: 64 an octave,
constexpr int kHMid = 112;    // then 8 an octave,
constexpr int kHLow = 32;     // then one an octave
constexpr int kHRest = kHBins - 1 - (kHFine + kHMid + kHLow);  // other scores >= 0; the bins below it: scores < 0

// The top bin's place, from the order bits (float_order_bits) of M and the query's number of terms.
SINDI_HD int32_t hbin_top(uint32_t order_bits, int terms = 8) {
#ifdef __CUDA_ARCH__
    const int octaves = terms > 8 ? 32 - __clz(terms - 1) : 3;
#else
    int octaves = 3;
    while (octaves < 31 && (int64_t)terms > (int64_t)1 << octaves) octaves++;
#endif
    return (int32_t)(order_bits >> 17) + octaves * 64;
}

// Bin of the score with order bits ob.
SINDI_HD uint32_t hbin(uint32_t ob, int32_t top) {
    if (ob < 0x80000000u) {  // negative: the complement is the magnitude's order bits
        const int32_t under = top - (int32_t)(~ob >> 17);
        const int32_t b = under > 0 ? under >> 3 : 0;
        return (uint32_t)(b < kHRest - 1 ? b : kHRest - 1);
    }
    const int32_t under = top - (int32_t)(ob >> 17);
    const int32_t d = under > 0 ? under : 0;
    if (d < kHFine) return (uint32_t)(kHBins - 1 - d);
    const int32_t mid = (d - kHFine) >> 3, low = kHMid + ((d - kHFine - 8 * kHMid) >> 6);
    const int32_t e = mid < kHMid ? mid : low;
    return (uint32_t)(e < kHMid + kHLow ? kHBins - 1 - kHFine - e : kHRest);
}

// Least order bits of bin b: a score lies in bin b or above exactly when its order bits are at least these.
SINDI_HD uint32_t hbin_floor(uint32_t b, int32_t top) {
    if (b == 0) return 0;
    if ((int)b < kHRest) {
        const int32_t t = top - 8 * (int32_t)b;  // the largest magnitude's place
        return t >= 0x7FFF ? 0u : t < 0x4000 ? 0x80000000u : ~(((uint32_t)t << 17) | 0x1FFFFu);
    }
    const int32_t e = kHBins - 1 - (int32_t)b;
    const int32_t d = e < kHFine ? e
                      : e < kHFine + kHMid ? kHFine + ((e - kHFine) << 3) + 7
                                           : kHFine + 8 * kHMid + ((e - kHFine - kHMid) << 6) + 63;
    const int32_t t = top - d;
    if ((int)b == kHRest || t <= 0x4000) return 0x80000000u;  // every score >= 0
    return t > 0x7FFF ? 0xFFFFFFFFu : (uint32_t)t << 17;      // (above every score: M near FP32's largest)
}

}  // namespace sindi
