// The bins of a query's histogram H of the candidates its windows emitted.
// Plain functions of integers, so that the host tests run the same code.
//
// H bounds what can still enter a query's answer (g candidates lie at or above
// some bin), so its bins decide how many slots below the true bound a window
// still emits: bins on 12 bits of the order key, 8 an octave, let a query of
// the 1M-document workload emit about 3 times what it has to, and had to be
// read whole by every block (16 KiB). Most bins of such a full-range table
// never fill. Here the top bin holds every score of 8 M and more, M = the
// query's largest product bound max_j |w_j| vmax_j (a maximum, so every block
// and kernel gets the same one, in any order of the terms); below it 12
// octaves have 64 bins each and 32 more octaves 8 each; bin 0 holds the rest.
#pragma once

#include <stdint.h>

#include "checks.cuh"  // SINDI_HD

namespace sindi {

constexpr int kHBins = 1024;  // bins of H
constexpr int kHFine = 768;   // of which from the top: 64 an octave; the rest: 8 an octave

// The top bin's place, from the order bits (float_order_bits) of M.
SINDI_HD int32_t hbin_top(uint32_t order_bits) { return (int32_t)(order_bits >> 17) + 3 * 64; }

// Bin of the score with order bits ob.
SINDI_HD uint32_t hbin(uint32_t ob, int32_t top) {
    const int32_t under = top - (int32_t)(ob >> 17);
    const int32_t d = under > 0 ? under : 0;
    const int32_t e = d < kHFine ? d : kHFine + ((d - kHFine) >> 3);
    return e < kHBins ? (uint32_t)(kHBins - 1 - e) : 0u;
}

// Least order bits of bin b: a score lies in bin b or above exactly when its order bits are at least these.
SINDI_HD uint32_t hbin_floor(uint32_t b, int32_t top) {
    if (b == 0) return 0;
    int32_t d = kHBins - 1 - (int32_t)b;
    if (d >= kHFine) d = kHFine + ((d - kHFine) << 3) + 7;
    const int32_t t = top - d;
    if (t > 0x7FFF) return 0xFFFFFFFFu;  // above every score (M near FP32's largest)
    return t > 0 ? (uint32_t)t << 17 : 0u;
}

}  // namespace sindi
