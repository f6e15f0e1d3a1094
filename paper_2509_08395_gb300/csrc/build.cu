// Index construction on the device: Algorithm 3 (alpha-mass of every
// document, Sec. 4.1) followed by Algorithm 1 (value-storing inverted lists,
// Sec. 3.1) with the lists cut into windows of lambda ids (Sec. 3.3.1).
//
// Pipeline (one stream):
//   validate_indptr  -> prune_select (warp per row) [+ prune_rows, prune_long_rows: rows that need a sort]
//   -> exclusive scan of kept counts -> compact
//   -> stable radix sort of kept entries by dim (input is in document order, so
//      equal dims stay in ascending document id: the order is (dim, doc))
//   -> (dim, window) counts -> scan = seg -> [List Pruning] -> [E4M3 per-list scales]
//   -> order_pack (bank-aware order, uint16 window-local id + value, vmax, signs).
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "index.cuh"
#include "mass.cuh"
#include "primitives.cuh"

namespace sindi {

constexpr int kPruneWarps = 4;                 // warps per block in prune_rows (32 KiB static smem)
constexpr int kPruneRowCap = 1024;             // longest row a warp sorts (smem 8 KB / warp)

__global__ void validate_indptr_kernel(const int64_t* indptr, int64_t n, uint32_t* err) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && indptr[0] != 0) atomicOr(err, kErrDocIndptr);
    if (i < n && indptr[i + 1] < indptr[i]) atomicOr(err, kErrDocIndptr);
}

void launch_validate_indptr(const int64_t* indptr, int64_t n, uint32_t* err, cudaStream_t stream) {
    const int64_t threads = n + 1;
    const unsigned blocks = (unsigned)((threads + 255) / 256);
    validate_indptr_kernel<<<blocks, 256, 0, stream>>>(indptr, n, err);
    SINDI_CUDA(cudaGetLastError());
}

// The kept set of a row is a bit mask: entry t of row i (indptr b) is bit t & 31 of word keep_words(b, i) + t / 32.
// A row's words follow those of the row before it (ceil(m / 32) <= floor((b + m) / 32) - floor(b / 32) + 1), so the
// whole mask takes nnz / 32 + n words: 1/64 of the kept entries' worst case.
__host__ __device__ __forceinline__ int64_t keep_words(int64_t b, int64_t i) { return (b >> 5) + i; }

struct PruneArgs {
    const int64_t* indptr;
    const int32_t* indices;
    const float* values;
    int64_t n;
    int32_t dim;
    double alpha;
    uint32_t vn;           // > 0: Vector Number Pruning
    uint32_t* kept;        // [n]
    uint32_t* mask;        // kept set, see keep_words
    uint32_t* sort_rows;   // rows left to prune_rows_kernel, and their count
    uint32_t* n_sort;
    uint32_t* long_rows;   // rows left to prune_long_rows_kernel, and their count
    uint32_t* n_long;
    uint32_t* next_long;   // rows of that list that a block has taken
    uint32_t* err;
};

// ---------------------------------------------------------------------------
// Pruning without a sort: one warp per row of up to 32 * I entries, I entries
// per lane in registers. The kept set is a prefix of the pi order (|x|
// descending, equal |x| by lower dim), so only its last |x|, K, is needed:
// the largest K whose entries of |x| >= K reach alpha * mass (or vn entries).
// K is found by bisecting the bit patterns of |x|, the end that moves pulled to
// the nearest |x| of the row (about 6 steps for 128 entries). The steps compare
// 32-bit sums (the shares' top 31 bits: one warp reduction a step); the K they
// end at is then checked with the whole sums, and moved when it is not the one.
//
// The rule sums FP64 values one after another in pi order. The values are
// FP32, so unless their magnitudes spread over 2^20 or more, every such sum
// is exact and does not depend on the order: with the least |x|'s last place
// as the unit and the sum below 2^53 units, the sums are taken here as whole
// numbers of units, and the kept count is bit-identical. Rows for
// which this does not hold, rows whose dims do not ascend (their duplicates
// need a sort to be found) and rows of more than 512 entries go to
// prune_rows_kernel.
//
// What bounds it: issue, and the chain of warp reductions. The row lengths are
// split over three launches (up to 128, 256, 512 entries): with all of them in
// one kernel the unrolled paths did not fit the instruction cache, and warps
// waited 6.5 of 14 cycles per instruction for it. Sorting a row instead takes
// 28 compare-exchange passes over shared memory and 2 * nnz dependent FP64 adds
// by one lane (20.1 ms for 1M documents of 120 entries, alpha 0.5; now 1.48).
// ---------------------------------------------------------------------------
constexpr int kSelectWarps = 8;
constexpr int kSelectRowCap = 512;

// Sum over the warp of one 53-bit share per lane (the total below 2^53): two 32-bit reductions.
__device__ __forceinline__ uint64_t warp_sum53(uint64_t v) {
    const uint32_t lo = __reduce_add_sync(kFull, (uint32_t)v & 0x3FFFFFFu);
    const uint32_t hi = __reduce_add_sync(kFull, (uint32_t)(v >> 26));
    return ((uint64_t)hi << 26) + lo;
}

// One row b .. b + m - 1 of at most 32 * I entries. False: the row is not for this path.
template <int I>
__device__ __forceinline__ bool prune_row_select(const PruneArgs& p, int64_t i, int64_t b, int m, int lane) {
    uint32_t a[I];  // bits of |x|; 0: an explicit zero (not an entry) or past the row
    bool bad_dim = false, bad_value = false, ascending = true;
#pragma unroll
    for (int u = 0; u < I; u++) {
        const int t = lane + 32 * u;
        a[u] = 0;
        if (t < m) {
            const int32_t j = __ldg(p.indices + b + t);
            const int32_t before = t > 0 ? __ldg(p.indices + b + t - 1) : -1;
            a[u] = __float_as_uint(__ldg(p.values + b + t)) & 0x7FFFFFFFu;
            bad_dim |= j < 0 || j >= p.dim;
            bad_value |= a[u] >= 0x7F800000u;
            ascending &= before < j;
        }
    }
    if (__any_sync(kFull, bad_dim || bad_value)) {
        if (bad_dim) atomicOr(p.err, kErrDocDim);
        if (bad_value) atomicOr(p.err, kErrDocValue);
        if (lane == 0) p.kept[i] = 0;
        return true;
    }
    if (!__all_sync(kFull, ascending)) return false;
    uint32_t nz_l = 0, top_l = 0, least_l = 0xFFFFFFFFu;
#pragma unroll
    for (int u = 0; u < I; u++) {
        nz_l += a[u] ? 1u : 0u;
        top_l = max(top_l, a[u]);
        least_l = a[u] ? min(least_l, a[u]) : least_l;
    }
    const uint32_t nz = __reduce_add_sync(kFull, nz_l);
    uint32_t K = 1, ties = 0xFFFFFFFFu;  // kept: |x| > K, and the first `ties` entries of |x| == K
    const bool by_mass = p.vn == 0;
    if (nz && (by_mass ? p.alpha < 1.0 : p.vn < nz)) {
        const uint32_t top = __reduce_max_sync(kFull, top_l);
        const uint32_t least = __reduce_min_sync(kFull, least_l);
        // every |x| is a whole number of units 2^(low - 150), below 2^(Etop + 24 - low) of them
        const int low = max(1, (int)(least >> 23));
        if (by_mass && max(1, (int)(top >> 23)) + 24 + (32 - __clz((int)(nz - 1) | 1)) - low > 53) return false;
        // an entry's share: |x| in units (the shift is at most 29), or 1 when entries are counted
        auto share = [&](uint32_t x) -> uint64_t {
            if (!by_mass) return x ? 1u : 0u;
            const uint32_t mant = x >= 0x800000u ? (x & 0x7FFFFFu) | 0x800000u : x;
            const int sh = x ? max(1, (int)(x >> 23)) - low : 0;
            return ((uint64_t)__funnelshift_l(mant, 0u, sh) << 32) | (mant << sh);
        };
        uint64_t mine = 0;
#pragma unroll
        for (int u = 0; u < I; u++) mine += share(a[u]);
        const uint64_t mass = warp_sum53(mine);
        uint64_t target = p.vn;
        if (by_mass) {
            target = (uint64_t)ceil(__dmul_rn(p.alpha, (double)mass));  // prefix >= alpha * mass, for whole prefixes
            if (target == 0) target = 1;
        }
        const int cutoff = max(0, 33 - __clzll((long long)mass));  // at most 22; mass >> cutoff below 2^31
        const uint32_t target32 = (uint32_t)(target >> cutoff);
        uint32_t s32[I];
#pragma unroll
        for (int u = 0; u < I; u++) {
            const uint64_t f = share(a[u]);
            s32[u] = __funnelshift_r((uint32_t)f, (uint32_t)(f >> 32), cutoff);
        }
        // lo: the least |x| whose entries and those above it reach the target; hi: K < hi (both by the short sums)
        uint32_t lo = least, hi = top + 1;
        uint32_t s_lo = (uint32_t)(mass >> cutoff), s_hi = 0;  // about the sums at and above lo and hi
        bool half = false;
        while (lo + 1 < hi) {
            // by turns where the target lies between the two sums, and halfway
            uint32_t off = (hi - lo) / 2;
            if (!half && s_lo > s_hi && s_lo > target32)
                off = (uint32_t)(__fdividef((float)(s_lo - target32), (float)(s_lo - s_hi)) * (float)(hi - lo));
            half = !half;
            const uint32_t mid = lo + min(max(off, 1u), hi - lo - 1u);  // lo < mid < hi
            uint32_t sum = 0;
#pragma unroll
            for (int u = 0; u < I; u++) sum += a[u] >= mid ? s32[u] : 0u;
            sum = __reduce_add_sync(kFull, sum);
            if (sum >= target32) {
                s_lo = sum;
                uint32_t up = 0xFFFFFFFFu;  // the nearest |x| of the row at or above mid
#pragma unroll
                for (int u = 0; u < I; u++) up = a[u] >= mid ? min(up, a[u]) : up;
                lo = __reduce_min_sync(kFull, up);
            } else {
                s_hi = sum;
                uint32_t down = 0;  // and below it
#pragma unroll
                for (int u = 0; u < I; u++) down = a[u] < mid ? max(down, a[u]) : down;
                hi = __reduce_max_sync(kFull, down) + 1;
            }
        }
        K = lo;
        while (true) {
            uint64_t above_l = 0;
            uint32_t eq_l = 0;
#pragma unroll
            for (int u = 0; u < I; u++) {
                above_l += share(a[u] > K ? a[u] : 0u);
                eq_l += a[u] == K ? 1u : 0u;
            }
            const uint64_t above = warp_sum53(above_l);
            const uint32_t eq = __reduce_add_sync(kFull, eq_l);
            const uint64_t fk = share(K);
            if (above >= target) {  // K lies higher
                uint32_t up = 0xFFFFFFFFu;
#pragma unroll
                for (int u = 0; u < I; u++) up = a[u] > K ? min(up, a[u]) : up;
                K = __reduce_min_sync(kFull, up);
            } else if (above + eq * fk < target) {  // lower (some |x| does reach the target: alpha < 1, vn < nz)
                uint32_t down = 0;
#pragma unroll
                for (int u = 0; u < I; u++) down = a[u] < K ? max(down, a[u]) : down;
                K = __reduce_max_sync(kFull, down);
            } else {
                // most rows: one entry of |x| == K, needed whole
                ties = target - above <= fk ? 1u : (uint32_t)((target - above + fk - 1) / fk);
                break;
            }
        }
    }
    uint32_t r = 0, tied = 0;
    uint32_t* words = p.mask + keep_words(b, i);
#pragma unroll
    for (int u = 0; u < I; u++) {
        if (32 * u < m) {
            const unsigned eq = __ballot_sync(kFull, a[u] == K);
            const bool keep = a[u] > K || (a[u] == K && tied + (uint32_t)__popc(eq & ((1u << lane) - 1u)) < ties);
            tied += (uint32_t)__popc(eq);
            const unsigned kw = __ballot_sync(kFull, keep);
            r += (uint32_t)__popc(kw);
            if (lane == 0) words[u] = kw;
        }
    }
    if (lane == 0) p.kept[i] = r;
    return true;
}

// Rows of more than `over` and at most 32 * I entries: a warp takes `rows` (<= 32) consecutive ones. The first launch
// (over < 0) also lists the rows that no launch takes.
template <int I>
__global__ void __launch_bounds__(kSelectWarps * 32, I <= 8 ? 4 : 2) prune_select_kernel(PruneArgs p, int over, int rows) {
    const int lane = threadIdx.x & 31;
    const int64_t i0 = ((int64_t)blockIdx.x * kSelectWarps + (threadIdx.x >> 5)) * rows;
    int64_t b_l = 0, m_l = -1;  // lane l: row i0 + l
    if (lane < rows && i0 + lane < p.n) {
        b_l = p.indptr[i0 + lane];
        m_l = p.indptr[i0 + lane + 1] - b_l;
    }
    if (over < 0 && m_l > kSelectRowCap) {
        if (m_l > kMaxRowNnz) {
            atomicOr(p.err, kErrDocTooLong);
            p.kept[i0 + lane] = 0;
        } else if (m_l > kPruneRowCap) {
            p.long_rows[atomicAdd(p.n_long, 1u)] = (uint32_t)(i0 + lane);
        } else {
            p.sort_rows[atomicAdd(p.n_sort, 1u)] = (uint32_t)(i0 + lane);
        }
    }
    unsigned todo = __ballot_sync(kFull, m_l > over && m_l >= 0 && m_l <= 32 * I);
    while (todo) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int64_t b = __shfl_sync(kFull, b_l, l);
        const int m = (int)__shfl_sync(kFull, m_l, l);
        if (!prune_row_select<I>(p, i0 + l, b, m, lane) && lane == 0)
            p.sort_rows[atomicAdd(p.n_sort, 1u)] = (uint32_t)(i0 + l);
    }
}

// The mask words of a row whose pi order is in s (kept: its first r entries).
// The row's threads t0, t0 + stride, ... (whole warps) call it.
__device__ __forceinline__ void write_row_mask(const PruneArgs& p, int64_t i, int64_t b, int m, const uint64_t* s, int r,
                                               int t0, int stride) {
    const uint64_t last = r > 0 ? s[r - 1] : 0;
    uint32_t* words = p.mask + keep_words(b, i);
    for (int t = t0; t - (t0 & 31) < m; t += stride) {
        bool keep = false;
        if (t < m && r > 0) {
            const float v = p.values[b + t];
            keep = v != 0.0f && mass_key(p.indices[b + t], v) <= last;
        }
        const unsigned kw = __ballot_sync(kFull, keep);
        if ((t & 31) == 0) words[t >> 5] = kw;
    }
}

// One warp per listed row (rows prune_select_kernel leaves, at most kPruneRowCap
// entries). Validates the row (dims in range, finite values, no duplicate dim)
// and computes r_i = |alpha-mass(x_i)| (or, when vn > 0, r_i = min(vn, nnz):
// Vector Number Pruning) from the sorted row.
__global__ void __launch_bounds__(kPruneWarps * 32) prune_rows_kernel(PruneArgs p) {
    __shared__ uint64_t sm[kPruneWarps][kPruneRowCap];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t* s = sm[warp];
    const uint32_t n_rows = *p.n_sort;
    for (uint32_t row = blockIdx.x * kPruneWarps + warp; row < n_rows; row += gridDim.x * kPruneWarps) {
        const int64_t i = p.sort_rows[row];
        const int64_t b = p.indptr[i];
        const int mm = (int)(p.indptr[i + 1] - b);
        int p2 = 32;
        while (p2 < mm) p2 <<= 1;
        // 1) dims: range check, and duplicates unless the row is strictly ascending
        bool bad = false, ascending = true;
        for (int t = lane; t < p2; t += 32) {
            if (t < mm) {
                int32_t j = p.indices[b + t];
                float v = p.values[b + t];
                if (j < 0 || j >= p.dim) { bad = true; atomicOr(p.err, kErrDocDim); }
                if (!isfinite(v)) { bad = true; atomicOr(p.err, kErrDocValue); }
                if (t + 1 < mm && p.indices[b + t + 1] <= j) ascending = false;
                s[t] = ((uint64_t)(uint32_t)j << 32) | (uint32_t)t;
            } else {
                s[t] = ~0ull;
            }
        }
        bad = __any_sync(kFull, bad);
        ascending = __all_sync(kFull, ascending);
        __syncwarp();
        if (bad) {
            if (lane == 0) p.kept[i] = 0;
            continue;
        }
        if (!ascending) {
            warp_bitonic_sort_asc(s, p2);
            bool dup = false;
            for (int t = lane + 1; t < mm; t += 32)
                if ((s[t] >> 32) == (s[t - 1] >> 32)) dup = true;
            dup = __any_sync(kFull, dup);
            __syncwarp();
            if (dup) {
                if (lane == 0) {
                    atomicOr(p.err, kErrDocDup);
                    p.kept[i] = 0;
                }
                continue;
            }
        }
        // 2) the pi order; explicit zeros are not entries (Definition 1) and sort last
        int nz = 0;
        for (int t = lane; t < p2; t += 32) {
            uint64_t key = ~0ull;
            if (t < mm) {
                float v = p.values[b + t];
                if (v != 0.0f) {
                    key = mass_key(p.indices[b + t], v);
                    nz++;
                }
            }
            s[t] = key;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nz += __shfl_xor_sync(kFull, nz, o);
        __syncwarp();
        warp_bitonic_sort_asc(s, p2);
        int r = 0;
        if (lane == 0) r = p.vn ? (nz < (int)p.vn ? nz : (int)p.vn) : alpha_mass_count(s, nz, p.alpha);
        r = __shfl_sync(kFull, r, 0);
        write_row_mask(p, i, b, mm, s, r, lane, 32);
        if (lane == 0) p.kept[i] = (uint32_t)r;
        __syncwarp();
    }
}

// One block per listed long row (kPruneRowCap < m <= kMaxRowNnz); same rules. A block takes the next row when it is done
// with one: rows of 2,000 to 6,000 entries differ by four in their sorts, and shared out beforehand they left SMs idle.
constexpr int kLongBlock = 512;
__global__ void __launch_bounds__(kLongBlock) prune_long_rows_kernel(PruneArgs p) {
    extern __shared__ uint64_t s[];
    __shared__ int flags[2];
    __shared__ int s_r, s_nz;
    __shared__ uint32_t s_row;
    const uint32_t n_rows = *p.n_long;
    while (true) {
        __syncthreads();  // the previous row is done with the shared arrays
        if (threadIdx.x == 0) s_row = atomicAdd(p.next_long, 1u);
        __syncthreads();
        const uint32_t row = s_row;
        if (row >= n_rows) break;
        const int64_t i = p.long_rows[row];
        const int64_t b = p.indptr[i];
        const int mm = (int)(p.indptr[i + 1] - b);
        int p2 = 32;
        while (p2 < mm) p2 <<= 1;
        if (threadIdx.x == 0) { flags[0] = 0; flags[1] = 0; s_nz = 0; }
        __syncthreads();
        for (int t = threadIdx.x; t < p2; t += kLongBlock) {
            if (t < mm) {
                int32_t j = p.indices[b + t];
                float v = p.values[b + t];
                if (j < 0 || j >= p.dim) { flags[0] = 1; atomicOr(p.err, kErrDocDim); }
                if (!isfinite(v)) { flags[0] = 1; atomicOr(p.err, kErrDocValue); }
                s[t] = ((uint64_t)(uint32_t)j << 32) | (uint32_t)t;
            } else {
                s[t] = ~0ull;
            }
        }
        __syncthreads();
        if (flags[0]) {
            if (threadIdx.x == 0) p.kept[i] = 0;
            continue;
        }
        // ascending sort of dims: reuse the descending sort on inverted keys
        for (int t = threadIdx.x; t < p2; t += kLongBlock) s[t] = ~s[t];
        __syncthreads();
        block_bitonic_sort_desc<kLongBlock>(s, p2);
        for (int t = threadIdx.x + 1; t < mm; t += kLongBlock)
            if (((~s[t]) >> 32) == ((~s[t - 1]) >> 32)) flags[1] = 1;
        __syncthreads();
        if (flags[1]) {
            if (threadIdx.x == 0) {
                atomicOr(p.err, kErrDocDup);
                p.kept[i] = 0;
            }
            continue;
        }
        for (int t = threadIdx.x; t < p2; t += kLongBlock) {
            uint64_t key = ~0ull;
            if (t < mm) {
                float v = p.values[b + t];
                if (v != 0.0f) {
                    key = mass_key(p.indices[b + t], v);
                    atomicAdd(&s_nz, 1);
                }
            }
            s[t] = ~key;  // descending sort of inverted keys = ascending mass_key
        }
        __syncthreads();
        block_bitonic_sort_desc<kLongBlock>(s, p2);
        for (int t = threadIdx.x; t < p2; t += kLongBlock) s[t] = ~s[t];
        __syncthreads();
        if (threadIdx.x == 0) s_r = p.vn ? (s_nz < (int)p.vn ? s_nz : (int)p.vn) : alpha_mass_count(s, s_nz, p.alpha);
        __syncthreads();
        const int r = s_r;
        write_row_mask(p, i, b, mm, s, r, (int)threadIdx.x, kLongBlock);
        if (threadIdx.x == 0) p.kept[i] = (uint32_t)r;
    }
}

// Kept entries of every row -> compact arrays in document order: a warp per row, the row's mask words read at once.
// Bound by HBM: the rows are read again, at 32-byte sectors (1M documents of 120 entries, 26 of them kept: 0.9 GB).
constexpr int kCompactWarps = 8;
__global__ void __launch_bounds__(kCompactWarps * 32) compact_kernel(const int64_t* indptr, const int32_t* indices,
                                                                     const float* values, const uint32_t* mask,
                                                                     const int64_t* kept_off, int64_t n, uint32_t* sdim,
                                                                     uint32_t* sdoc, uint32_t* sval) {
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * kCompactWarps + (threadIdx.x >> 5);
    if (i >= n) return;
    const int64_t b = indptr[i], m = indptr[i + 1] - b;
    const uint32_t* words = mask + keep_words(b, i);
    int64_t o = kept_off[i];
    const unsigned lt = (1u << lane) - 1u;
    for (int64_t t0 = 0; t0 < m; t0 += 1024) {
        const uint32_t mine = t0 + 32 * lane < m ? words[(t0 >> 5) + lane] : 0u;
        const int nw = (int)(m - t0 < 1024 ? (m - t0 + 31) >> 5 : 32);
        for (int u0 = 0; u0 < nw; u0 += 4) {  // four words' loads in flight
            uint32_t kw[4], jj[4], xx[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                kw[u] = __shfl_sync(kFull, mine, u0 + u);  // (0 past the row)
                const int64_t from = b + t0 + 32 * (u0 + u) + lane;
                jj[u] = xx[u] = 0;
                if ((kw[u] >> lane) & 1u) {
                    jj[u] = (uint32_t)__ldg(indices + from);
                    xx[u] = __float_as_uint(__ldg(values + from));
                }
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                if ((kw[u] >> lane) & 1u) {
                    const int64_t at = o + __popc(kw[u] & lt);
                    sdim[at] = jj[u];
                    sdoc[at] = (uint32_t)i;
                    sval[at] = xx[u];
                }
                o += __popc(kw[u]);
            }
        }
    }
}

// Postings of every list I_{j,w}, cnt[j * sigma + w], from the sorted order (cnt zero on entry): a posting that starts
// a list takes its place off the list's count, and adds it to the list that ends there (mod 2^32; the last list ends
// at P). Two atomics a list instead of one a posting, whose head lists met on few addresses (26M: 574 -> 108 us).
__global__ void list_count_kernel(const uint32_t* sdim, const uint32_t* sdoc, int64_t P, uint32_t lambda, uint32_t sigma,
                                  uint32_t* cnt) {
    auto list_of = [&](int64_t p) { return (uint64_t)sdim[p] * sigma + sdoc[p] / lambda; };
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t here = list_of(p);
        if (p == P - 1) atomicAdd(&cnt[here], (uint32_t)P);
        if (p > 0) {
            const uint64_t before = list_of(p - 1);
            if (before == here) continue;
            atomicAdd(&cnt[before], (uint32_t)p);
        }
        atomicSub(&cnt[here], (uint32_t)p);
    }
}

// amax[j] = the largest |x| of list I_j over all its windows, as the bits of a non-negative float (zero on entry):
// a warp per list I_{j,w}.
__global__ void list_amax_kernel(const uint32_t* seg, const uint32_t* sval, int64_t S, uint32_t sigma, uint32_t* amax) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t sg = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); sg < S; sg += warps) {
        const uint32_t lo = seg[sg], hi = seg[sg + 1];
        if (lo == hi) continue;
        uint32_t m = 0;
        for (uint32_t p = lo + lane; p < hi; p += 32) m = max(m, sval[p] & 0x7FFFFFFFu);
        m = __reduce_max_sync(kFull, m);
        if (lane == 0 && m > __ldcg(&amax[sg / sigma])) atomicMax(&amax[sg / sigma], m);
    }
}

// Per-list E4M3 scale: max |x| over the list I_j (all windows) / 448.
__global__ void list_scale_kernel(const uint32_t* amax, int32_t dim, float* scale) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < dim; j += (int64_t)gridDim.x * blockDim.x) {
        const float sc = __fdiv_rn(__uint_as_float(amax[j]), 448.0f);
        scale[j] = sc > 0.0f ? sc : 1.0f;
    }
}

// A stored value: its code, and the value the scan reads back for it (without an E4M3 list's scale).
template <int DT>
__device__ __forceinline__ float store_value(float v, float scale, void* pval, uint32_t p) {
    if (DT == SINDI_F32) {
        static_cast<float*>(pval)[p] = v;
        return v;
    } else if (DT == SINDI_F16) {
        const __half h = __float2half_rn(v);
        static_cast<__half*>(pval)[p] = h;
        return __half2float(h);
    } else {
        const __nv_fp8_storage_t c = __nv_cvt_float_to_fp8(__fdiv_rn(v, scale), __NV_SATFINITE, __NV_E4M3);
        static_cast<__nv_fp8_storage_t*>(pval)[p] = c;
        return __half2float(__half(__nv_cvt_fp8_to_halfraw(c, __NV_E4M3)));
    }
}

// List Pruning (Sec. 4.1): every list I_j keeps its `lp` entries of largest
// |x|, equal |x| by lower document id. Postings are in (dim, doc) order, so a
// list is one range and its order of documents the order of positions: a block
// per list that is longer than lp selects the lp largest (|x|, position) keys.
// A dropped entry leaves its document's count. A stable sort of every posting
// by |x| and dim ranks them all in up to eight radix passes; it is kept for
// postings of which one list holds a large part (lp_by_sort).
constexpr int kLpBlock = 512;
__global__ void __launch_bounds__(kLpBlock) lp_select_kernel(const uint32_t* seg, const uint32_t* sval, int32_t dim,
                                                             uint32_t sigma, uint32_t lp, const uint32_t* sdoc,
                                                             uint32_t* keep, uint32_t* kept) {
    __shared__ uint32_t hist[256];
    __shared__ uint32_t st[4];
    for (int64_t j = blockIdx.x; j < dim; j += gridDim.x) {
        const uint32_t lo = seg[(uint64_t)j * sigma], L = seg[(uint64_t)(j + 1) * sigma] - lo;
        uint64_t T = 0;
        auto key_of = [&](int64_t i) -> uint64_t {
            return ((uint64_t)(sval[lo + i] & 0x7FFFFFFFu) << 32) | (0xFFFFFFFFu - (uint32_t)i);
        };
        if (L > lp) T = group_select_threshold<SyncBlock<kLpBlock>>(key_of, (int64_t)L, (int64_t)lp, hist, st);
        for (int64_t i = threadIdx.x; i < L; i += kLpBlock) {
            const bool k = key_of(i) >= T;
            keep[lo + i] = k ? 1u : 0u;
            if (!k) atomicSub(&kept[sdoc[lo + i]], 1u);
        }
        __syncthreads();
    }
}

// Whether the lists are pruned by a sort: a block selects from a list of its own at about 2.9 ns an entry, all blocks
// at once, so the longest list decides; the sort takes about 0.0065 ns a posting and pass on the whole device. Builds
// with one or the other, ms: 4M documents of one dim 14.3 selected, 2.5 sorted; 4M of 2 to 8 entries in 16 dims 8.3
// and 4.4; 6M of 20 to 60 entries, Zipf dims, the longest list 1/40 of the postings: 53.1 and 48.9. (1M of 60 to 180,
// the longest list 1/120 of them, are selected: 15.2.)
static bool lp_by_sort(uint32_t longest, int64_t P, int passes) { return (int64_t)longest > P * passes / 450; }

__global__ void longest_list_kernel(const uint32_t* seg, int32_t dim, uint32_t sigma, uint32_t* longest) {
    uint32_t m = 0;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < dim; j += (int64_t)gridDim.x * blockDim.x)
        m = max(m, seg[(uint64_t)(j + 1) * sigma] - seg[(uint64_t)j * sigma]);
    m = __reduce_max_sync(kFull, m);
    if ((threadIdx.x & 31) == 0) atomicMax(longest, m);
}

// Sort keys: 0x7FFFFFFF - |x| bits (ascending = |x| descending), and the entry's position.
__global__ void lp_keys_kernel(const uint32_t* sval, int64_t P, uint32_t* inv, uint32_t* pos) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (int64_t)gridDim.x * blockDim.x) {
        inv[p] = 0x7FFFFFFFu - (sval[p] & 0x7FFFFFFFu);
        pos[p] = (uint32_t)p;
    }
}

// Entry t of the (dim, |x| descending, document) order has rank t - start(list) in its list.
__global__ void lp_mark_kernel(const uint32_t* dim_sorted, const uint32_t* pos_sorted, int64_t P, const uint32_t* seg,
                               uint32_t sigma, uint32_t lp, const uint32_t* sdoc, uint32_t* keep, uint32_t* kept) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < P; t += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = pos_sorted[t];
        const bool k = (uint64_t)t - seg[(uint64_t)dim_sorted[t] * sigma] < lp;
        keep[p] = k ? 1u : 0u;
        if (!k) atomicSub(&kept[sdoc[p]], 1u);
    }
}

// Entries with keep[p] = 1 move to off[p] (exclusive scan of keep); the
// (dim, doc) order is kept.
__global__ void lp_compact_kernel(const uint32_t* keep, const uint32_t* off, int64_t P, const uint32_t* sdim,
                                  const uint32_t* sdoc, const uint32_t* sval, uint32_t* odim, uint32_t* odoc,
                                  uint32_t* oval) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (int64_t)gridDim.x * blockDim.x) {
        if (keep[p]) {
            const uint32_t o = off[p];
            odim[o] = sdim[p];
            odoc[o] = sdoc[p];
            oval[o] = sval[p];
        }
    }
}

// The lists' final arrays: window ids and stored values of every segment I_{j,w}, in the order of the window scan's
// shared-memory scatter-add: the 32 postings one add instruction of a warp
// takes should sit in 32 different shared-memory banks (window slot mod 32),
// which makes the shared-memory atomicAdd conflict-free where a chunk is one
// whole piece of the segment (the pipelined and query-group scans). The default
// scan's chunks begin at any group of 8 and may hold two terms, so it meets
// fewer conflicts than in document order, but some: 2.3 wavefronts an add
// instruction on the 1M-document workload. One warp per segment:
//   1. every posting gets its bank b and a rank r among the segment's
//      postings of bank b; ordering the postings by (r, b) visits the banks
//      round robin, so any 32 consecutive ones hold 32 banks while every bank
//      still has postings. Its place is T[r] + the banks below b that hold
//      more than r postings, T[r] = the postings of rank below r: one table
//      row (T[r], the banks that hold more than r) per rank;
//   2. that order is laid out over the positions of the segment in the order
//      the scan's add instructions visit them (see kVecMin), so each
//      instruction takes 32 consecutive ones.
// Any order of a segment gives the same scores up to FP32 rounding; this one
// only changes which bank each add of an instruction meets.
// The same pass packs the postings (uint16 id, stored value), raises the
// list's largest |stored value| vmax[j] (bits; zero on entry) and sets *neg
// when a stored value's sign bit is set. With those as passes of their own (a
// warp per whole list for vmax) and 32 counts read per posting for its place,
// 26M postings took 1.35 ms, now 0.50.
// scratch: uint32[P], for segments longer than kOrderStage.
constexpr int kOrderWarps = 8;
static_assert(kVecMin <= 33, "segments of more than 32 postings are tiled on 8-aligned groups");
constexpr uint32_t kOrderStage = 1024;  // postings of a segment whose order stays in shared memory
constexpr uint32_t kOrderRanks = 256;   // ranks in the table; a segment with a fuller bank counts again per posting
template <int DT>
__global__ void __launch_bounds__(kOrderWarps * 32) order_pack_kernel(const uint32_t* seg, int64_t S, uint32_t sigma,
                                                                     const uint32_t* __restrict__ sdoc,
                                                                     const uint32_t* __restrict__ sval,
                                                                     uint32_t lambda, const float* scale,
                                                                     uint32_t* scratch, uint16_t* pid, void* pval,
                                                                     uint32_t* vmax, uint32_t* neg) {
    __shared__ uint32_t s_cnt[kOrderWarps][32];
    __shared__ uint32_t s_rnk[kOrderWarps][32];
    __shared__ uint2 s_row[kOrderWarps][kOrderRanks];
    __shared__ uint16_t s_perm[kOrderWarps][kOrderStage];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *cnt = s_cnt[warp], *rnk = s_rnk[warp];
    uint2* row = s_row[warp];
    uint16_t* perm = s_perm[warp];
    const unsigned lt = (1u << lane) - 1u;
    const int64_t warps = (int64_t)gridDim.x * kOrderWarps;
    uint32_t negative = 0;
    for (int64_t sg = (int64_t)blockIdx.x * kOrderWarps + warp; sg < S; sg += warps) {
        const uint32_t s = seg[sg], e = seg[sg + 1], L = e - s;
        if (L == 0) continue;
        const uint32_t j = (uint32_t)(sg / sigma);
        const float sc = DT == SINDI_F8E4M3 ? scale[j] : 1.0f;
        float top = 0.0f;
        auto put = [&](uint32_t p, uint32_t doc, uint32_t val) {
            pid[p] = (uint16_t)(doc % lambda);
            const float v = store_value<DT>(__uint_as_float(val), sc, pval, p);
            top = fmaxf(top, fabsf(v));
            negative |= __float_as_uint(v) >> 31;
        };
        if (L <= 32) {
            // one add instruction takes the whole segment: nothing to gain
            if (lane < (int)L) put(s + lane, __ldg(sdoc + s + lane), __ldg(sval + s + lane));
        } else {
            cnt[lane] = 0;
            rnk[lane] = 0;
            __syncwarp();
#pragma unroll 4
            for (uint32_t i = lane; i < L; i += 32) atomicAdd(&cnt[(__ldg(sdoc + s + i) % lambda) & 31u], 1u);
            __syncwarp();
            const uint32_t mine = cnt[lane];
            const uint32_t most = __reduce_max_sync(kFull, mine);
            const bool table = most <= kOrderRanks;
            if (table) {
                uint32_t below = 0;
                for (uint32_t r = 0; r < most; r++) {
                    const unsigned more = __ballot_sync(kFull, mine > r);
                    if (lane == 0) row[r] = make_uint2(below, more);
                    below += (uint32_t)__popc(more);
                }
                __syncwarp();
            }
            const bool staged = L <= kOrderStage;
            uint32_t next = __ldg(sdoc + s + lane);  // (L > 32)
            for (uint32_t i0 = 0; i0 < L; i0 += 32) {
                // rank = earlier postings of the same bank, in segment order (deterministic)
                const uint32_t i = i0 + (uint32_t)lane;
                const bool ok = i < L;
                const uint32_t b = (next % lambda) & 31u;
                if (i + 32 < L) next = __ldg(sdoc + s + i + 32);
                const unsigned peers = warp_match<5>(b) & __ballot_sync(kFull, ok);
                const uint32_t r = ok ? rnk[b] + (uint32_t)__popc(peers & lt) : 0u;
                __syncwarp();
                if (ok && (peers & lt) == 0) rnk[b] += (uint32_t)__popc(peers);
                __syncwarp();
                if (ok) {
                    // place of (r, b) in the (rank, bank) order
                    uint32_t q = 0;
                    if (table) {
                        const uint2 t = row[r];
                        q = t.x + (uint32_t)__popc(t.y & ((1u << b) - 1u));
                    } else {
                        for (uint32_t bb = 0; bb < 32; bb++) {
                            const uint32_t c = cnt[bb];
                            q += c < r ? c : r;
                            q += (bb < b && c > r) ? 1u : 0u;
                        }
                    }
                    if (staged) perm[q] = (uint16_t)i;
                    else scratch[s + q] = i;
                }
            }
            __syncwarp();
            // the positions in the order the scan's add instructions take them
            uint32_t run = 0;
            {
                const uint32_t g0 = s & ~7u, e8 = (e + 7u) & ~7u;
                for (uint32_t base = g0; base < e8; base += (uint32_t)kChunkLen) {
                    // the chunk's eight gathers in flight
                    const uint32_t p0 = base + 8u * (uint32_t)lane;
                    uint32_t src[kChunkU], doc[kChunkU], val[kChunkU];
#pragma unroll
                    for (int u = 0; u < kChunkU; u++) {
                        const bool ok = p0 + u >= s && p0 + u < e;
                        const unsigned bal = __ballot_sync(kFull, ok);
                        const uint32_t q = run + (uint32_t)__popc(bal & lt);
                        src[u] = ok ? s + (staged ? (uint32_t)perm[q] : scratch[s + q]) : 0xFFFFFFFFu;
                        run += (uint32_t)__popc(bal);
                    }
#pragma unroll
                    for (int u = 0; u < kChunkU; u++) {
                        doc[u] = val[u] = 0;
                        if (src[u] != 0xFFFFFFFFu) {
                            doc[u] = __ldg(sdoc + src[u]);
                            val[u] = __ldg(sval + src[u]);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kChunkU; u++)
                        if (src[u] != 0xFFFFFFFFu) put(p0 + u, doc[u], val[u]);
                }
            }
            __syncwarp();
        }
        const uint32_t m = __reduce_max_sync(kFull, __float_as_uint(top));
        if (lane == 0 && m > __ldcg(&vmax[j])) atomicMax(&vmax[j], m);
    }
    if (__any_sync(kFull, negative != 0) && lane == 0) atomicOr(neg, 1u);
}

__global__ void fill_u32_kernel(float* p, int64_t n, float v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

static int grid_for(int64_t n, int block, int cap = 152 * 16) {
    int64_t g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

static uint32_t read_u32(const uint32_t* d, cudaStream_t s) {
    uint32_t h = 0;
    SINDI_CUDA(cudaMemcpyAsync(&h, d, 4, cudaMemcpyDeviceToHost, s));
    SINDI_CUDA(cudaStreamSynchronize(s));
    return h;
}

static std::string doc_error_text(uint32_t e) {
    std::string m;
    if (e & kErrDocIndptr) m += "indptr[0] != 0 or decreasing; ";
    if (e & kErrDocDim) m += "a document dim outside [0, dim); ";
    if (e & kErrDocValue) m += "a non-finite document value; ";
    if (e & kErrDocDup) m += "a dim repeated within a document; ";
    if (e & kErrDocTooLong) m += "a document row longer than 16384 entries; ";
    return m;
}

// Builds the lists of `ix`. Its documents are on the device and indptr has
// been validated (indptr[0] = 0, non-decreasing). Allocates the index arrays
// (seg, pid, pval, scale, kept) from the library pool; they belong to `ix`.
// Returns SINDI_OK or an error status with the message set.
sindi_status build_lists(IndexImpl& ix, cudaStream_t stream) {
    Pool P{ix.pool, stream};
    const int64_t n = ix.n_docs;
    const int32_t d = ix.dim;
    const uint32_t lambda = ix.lambda;
    const uint32_t sigma = ix.sigma;
    uint32_t e = 0;
    // the document stage: Vector Number Pruning keeps vn entries per row,
    // otherwise alpha-mass (alpha = 1 keeps every entry)
    const uint32_t vn = ix.prune == SINDI_PRUNE_VECTOR_NUMBER ? ix.prune_n : 0u;
    const uint32_t lp = (ix.prune == SINDI_PRUNE_LIST || ix.prune == SINDI_PRUNE_MASS_LIST) ? ix.prune_n : 0u;
    SINDI_TRACE_MSG("build_lists: enter");
    ix.kept = P.alloc<uint32_t>(n > 0 ? n : 1);
    ix.scale = P.alloc<float>(d);
    ix.seg = P.alloc<uint32_t>((size_t)d * sigma + 1);
    const int64_t nnz = ix.doc_nnz;
    uint32_t* kept = ix.kept;
    const size_t mask_words = (size_t)keep_words(nnz, n) + 1;
    uint32_t* mask = P.alloc<uint32_t>(mask_words);
    uint32_t* left_rows = P.alloc<uint32_t>(2 * (size_t)n + 3);  // rows to sort, long rows, their counts, rows taken
    uint32_t* n_left = left_rows + 2 * n;
    SINDI_CUDA(cudaMemsetAsync(n_left, 0, 12, stream));
    SINDI_TRACE_MSG("build_lists: launching the pruning kernels");
    int64_t* kept_off = P.alloc<int64_t>(n + 1);
    if (n > 0) {
        const PruneArgs pa{ix.indptr, ix.indices, ix.values, n,         d,          ix.alpha,      vn,
                           kept,      mask,       left_rows, n_left,    left_rows + n, n_left + 1, n_left + 2,
                           ix.err};
        // rows per warp: as many as leave four waves of warps
        const int rows = (int)std::min<int64_t>(32, std::max<int64_t>(1, n / (152 * 32 * 4)));
        const unsigned blocks = (unsigned)((n + (int64_t)rows * kSelectWarps - 1) / ((int64_t)rows * kSelectWarps));
        prune_select_kernel<4><<<blocks, kSelectWarps * 32, 0, stream>>>(pa, -1, rows);
        SINDI_CUDA(cudaGetLastError());
        prune_select_kernel<8><<<blocks, kSelectWarps * 32, 0, stream>>>(pa, 128, rows);
        SINDI_CUDA(cudaGetLastError());
        prune_select_kernel<16><<<blocks, kSelectWarps * 32, 0, stream>>>(pa, 256, rows);
        SINDI_CUDA(cudaGetLastError());
        // the listed rows; their counts stay on the device
        prune_rows_kernel<<<grid_for(n, kPruneWarps, 152 * 6), kPruneWarps * 32, 0, stream>>>(pa);
        SINDI_CUDA(cudaGetLastError());
        const size_t sm = (size_t)kMaxRowNnz * sizeof(uint64_t);
        SINDI_CUDA(cudaFuncSetAttribute(prune_long_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        prune_long_rows_kernel<<<grid_for(n, 1, 152), kLongBlock, sm, stream>>>(pa);
        SINDI_CUDA(cudaGetLastError());
    }
    exclusive_scan<uint32_t, int64_t>(kept, kept_off, n, P);
    int64_t Pn0 = 0;
    SINDI_CUDA(cudaMemcpyAsync(&Pn0, kept_off + n, 8, cudaMemcpyDeviceToHost, stream));
    e = read_u32(ix.err, stream);
    P.free(left_rows);
    if (e) {
        P.free(mask); P.free(kept_off);
        set_last_error("malformed documents: " + doc_error_text(e));
        return (e & kErrDocTooLong) && !(e & ~kErrDocTooLong) ? SINDI_ERR_UNSUPPORTED : SINDI_ERR_INVALID_DATA;
    }

    SINDI_TRACE_MSG("build_lists: pruning done");
    // --- compact kept entries (document order)
    if (Pn0 > kMaxPostings) {
        P.free(mask); P.free(kept_off);
        set_last_error("more than 2^32 - 4096 kept entries");
        return SINDI_ERR_UNSUPPORTED;
    }
    int64_t Pn = Pn0;
    uint32_t* sdim = P.alloc<uint32_t>(Pn);
    uint32_t* sdoc = P.alloc<uint32_t>(Pn);
    uint32_t* sval = P.alloc<uint32_t>(Pn);
    if (n > 0) {
        compact_kernel<<<(unsigned)((n + kCompactWarps - 1) / kCompactWarps), kCompactWarps * 32, 0, stream>>>(
            ix.indptr, ix.indices, ix.values, mask, kept_off, n, sdim, sdoc, sval);
        SINDI_CUDA(cudaGetLastError());
    }
    P.free(mask);
    P.free(kept_off);

    SINDI_TRACE_MSG("build_lists: compacted %lld kept entries", (long long)Pn);
    // --- stable sort by dim: (dim, doc) order
    const int64_t S = (int64_t)d * sigma;
    int dim_bits = 0;
    while (dim_bits < 32 && ((uint64_t)1 << dim_bits) < (uint64_t)d) dim_bits++;
    {
        uint32_t* kb = P.alloc<uint32_t>(Pn);
        uint32_t* db = P.alloc<uint32_t>(Pn);
        uint32_t* vb = P.alloc<uint32_t>(Pn);
        radix_sort_triples(sdim, sdoc, sval, kb, db, vb, Pn, dim_bits, P);
        P.free(kb); P.free(db); P.free(vb);
    }
    SINDI_TRACE_MSG("build_lists: sort done");
    // --- offsets of every list I_{j,w}
    auto list_offsets = [&]() {
        uint32_t* cnt = P.alloc<uint32_t>(S > 0 ? S : 1);
        SINDI_CUDA(cudaMemsetAsync(cnt, 0, sizeof(uint32_t) * (size_t)(S > 0 ? S : 1), stream));
        if (Pn > 0) {
            list_count_kernel<<<grid_for(Pn, 256), 256, 0, stream>>>(sdim, sdoc, Pn, lambda, sigma, cnt);
            SINDI_CUDA(cudaGetLastError());
        }
        exclusive_scan<uint32_t, uint32_t>(cnt, ix.seg, S, P);
        P.free(cnt);
    };
    list_offsets();
    SINDI_TRACE_MSG("build_lists: list offsets done");

    if (lp > 0 && Pn > 0) {
        // --- List Pruning on the lists built so far, then their offsets again
        uint32_t* keep = P.alloc<uint32_t>(Pn);
        uint32_t* off = P.alloc<uint32_t>(Pn + 1);
        uint32_t* longest = off;  // (read before the scan below writes it)
        SINDI_CUDA(cudaMemsetAsync(longest, 0, 4, stream));
        longest_list_kernel<<<grid_for(d, 256), 256, 0, stream>>>(ix.seg, d, sigma, longest);
        SINDI_CUDA(cudaGetLastError());
        // (the sort's arrays take 20 bytes a posting; without room for them the lists are selected)
        uint32_t* inv = nullptr;
        if (lp_by_sort(read_u32(longest, stream), Pn, 4 + (dim_bits + 7) / 8)) inv = P.try_alloc<uint32_t>(5 * Pn);
        if (inv) {
            uint32_t *dcp = inv + Pn, *pos = dcp + Pn, *kb = pos + Pn, *db = kb + Pn;
            lp_keys_kernel<<<grid_for(Pn, 256), 256, 0, stream>>>(sval, Pn, inv, pos);
            SINDI_CUDA(cudaGetLastError());
            SINDI_CUDA(cudaMemcpyAsync(dcp, sdim, sizeof(uint32_t) * (size_t)Pn, cudaMemcpyDeviceToDevice, stream));
            radix_sort_triples(inv, dcp, pos, kb, db, keep, Pn, 31, P);        // by |x| descending (stable)
            radix_sort_triples(dcp, inv, pos, kb, db, keep, Pn, dim_bits, P);  // then by dim (stable)
            lp_mark_kernel<<<grid_for(Pn, 256), 256, 0, stream>>>(dcp, pos, Pn, ix.seg, sigma, lp, sdoc, keep, kept);
            SINDI_CUDA(cudaGetLastError());
            P.free(inv);
        } else {
            lp_select_kernel<<<grid_for(d, 1, 152 * 4), kLpBlock, 0, stream>>>(ix.seg, sval, d, sigma, lp, sdoc, keep,
                                                                               kept);
            SINDI_CUDA(cudaGetLastError());
        }
        exclusive_scan<uint32_t, uint32_t>(keep, off, Pn, P);
        const int64_t Pk = read_u32(off + Pn, stream);
        uint32_t* odim = P.alloc<uint32_t>(Pk > 0 ? Pk : 1);
        uint32_t* odoc = P.alloc<uint32_t>(Pk > 0 ? Pk : 1);
        uint32_t* oval = P.alloc<uint32_t>(Pk > 0 ? Pk : 1);
        lp_compact_kernel<<<grid_for(Pn, 256), 256, 0, stream>>>(keep, off, Pn, sdim, sdoc, sval, odim, odoc, oval);
        SINDI_CUDA(cudaGetLastError());
        P.free(keep); P.free(off);
        P.free(sdim); P.free(sdoc); P.free(sval);
        sdim = odim;
        sdoc = odoc;
        sval = oval;
        Pn = Pk;
        list_offsets();
        SINDI_TRACE_MSG("build_lists: list pruning kept %lld postings", (long long)Pn);
    }
    ix.postings = Pn;
    // posting arrays padded to a multiple of 8 entries: the scan reads aligned groups of 8
    const int64_t Pp = (Pn + 7) & ~(int64_t)7;
    ix.pid = P.alloc<uint16_t>(Pp);
    ix.pval = P.alloc<uint8_t>((size_t)Pp * ix.value_bytes());
    if ((reinterpret_cast<uintptr_t>(ix.pid) | reinterpret_cast<uintptr_t>(ix.pval)) & 31)
        throw CudaError{cudaErrorMisalignedAddress, "posting arrays are not 32-byte aligned"};
    if (Pp > Pn) {
        SINDI_CUDA(cudaMemsetAsync(ix.pid + Pn, 0, sizeof(uint16_t) * (size_t)(Pp - Pn), stream));
        SINDI_CUDA(cudaMemsetAsync(static_cast<uint8_t*>(ix.pval) + (size_t)Pn * ix.value_bytes(), 0,
                                   (size_t)(Pp - Pn) * ix.value_bytes(), stream));
    }
    // --- the lists: order, window-local ids, stored values, their bounds
    ix.vmax = P.alloc<float>(d);
    uint32_t* flags = P.alloc<uint32_t>((size_t)d + 1);  // largest |x| of every list; a stored value is negative
    uint32_t* neg = flags + d;
    SINDI_CUDA(cudaMemsetAsync(ix.vmax, 0, sizeof(float) * (size_t)d, stream));
    SINDI_CUDA(cudaMemsetAsync(flags, 0, sizeof(uint32_t) * ((size_t)d + 1), stream));
    if (ix.dtype == SINDI_F8E4M3) {
        list_amax_kernel<<<grid_for(S, 8, 152 * 32), 256, 0, stream>>>(ix.seg, sval, S, sigma, flags);
        SINDI_CUDA(cudaGetLastError());
        list_scale_kernel<<<grid_for(d, 256), 256, 0, stream>>>(flags, d, ix.scale);
        SINDI_CUDA(cudaGetLastError());
    } else {
        fill_u32_kernel<<<grid_for(d, 256), 256, 0, stream>>>(ix.scale, d, 1.0f);
        SINDI_CUDA(cudaGetLastError());
    }
    if (Pn > 0) {
        uint32_t* scratch = P.alloc<uint32_t>(Pn);
        const unsigned blocks = (unsigned)grid_for(S, kOrderWarps, 152 * 32);
        uint32_t* vmax = reinterpret_cast<uint32_t*>(ix.vmax);
        auto launch = [&](auto kern) {
            kern<<<blocks, kOrderWarps * 32, 0, stream>>>(ix.seg, S, sigma, sdoc, sval, lambda, ix.scale, scratch, ix.pid,
                                                          ix.pval, vmax, neg);
            SINDI_CUDA(cudaGetLastError());
        };
        if (ix.dtype == SINDI_F32) launch(order_pack_kernel<SINDI_F32>);
        else if (ix.dtype == SINDI_F16) launch(order_pack_kernel<SINDI_F16>);
        else launch(order_pack_kernel<SINDI_F8E4M3>);
        P.free(scratch);
    }
    P.free(sdim);
    P.free(sdoc);
    P.free(sval);
    ix.nonneg = read_u32(neg, stream) == 0;  // synchronises the stream
    P.free(flags);
    return SINDI_OK;
}

// Sets *flag when a stored posting value has its sign bit set (FP32, binary16
// or E4M3 alike: the top bit of the stored word).
__global__ void negative_values_kernel(const unsigned char* pval, int64_t P, int vbytes, uint32_t* flag) {
    bool neg = false;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P && !neg;
         p += (int64_t)gridDim.x * blockDim.x)
        neg = (pval[p * vbytes + vbytes - 1] & 0x80u) != 0;  // little-endian: the sign is in the last byte
    if (__syncthreads_or(neg) && threadIdx.x == 0) atomicOr(flag, 1u);
}

bool postings_nonnegative(const IndexImpl& ix, cudaStream_t stream) {
    Pool P{ix.pool, stream};
    uint32_t* flag = P.alloc<uint32_t>(1);
    SINDI_CUDA(cudaMemsetAsync(flag, 0, 4, stream));
    if (ix.postings > 0) {
        negative_values_kernel<<<grid_for(ix.postings, 256), 256, 0, stream>>>(
            static_cast<const unsigned char*>(ix.pval), ix.postings, (int)ix.value_bytes(), flag);
        SINDI_CUDA(cudaGetLastError());
    }
    uint32_t h = 0;
    SINDI_CUDA(cudaMemcpyAsync(&h, flag, 4, cudaMemcpyDeviceToHost, stream));
    P.free(flag);
    SINDI_CUDA(cudaStreamSynchronize(stream));
    return h == 0;
}

}  // namespace sindi
