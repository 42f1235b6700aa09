// Two queries of a batch scanned together (pair.cu prepares, scan.cu scans, merge.cu reads).
//
// The scan is bound by its table look-ups: one 4-byte shared-memory load per code byte and QUERY.  Where queries of a batch
// probe the same long lists, a look-up can serve two of them: a table entry then holds, in its two 16-bit halves, a lower
// bound of each query's 32-bit entry, and one 32-bit addition advances both sums.
//
// The bound.  For a query, sub-space m and code j the 32-bit table holds the integer T(j, m).  With
// low(m) = min_j T(j, m) and a shift s of the query's own,
//     e(j, m) = (T(j, m) - low(m)) >> s,       sum_m max_j e(j, m) <= 65 535,
//     L = sum_m low(m) + (sum_m e) * 2^s  <=  sum_m T  <=  L + M (2^s - 1).
// The score is a monotone function of the sum (conversion, multiplication by a positive number, additions: each rounds
// monotonically), so the score of L, formed by the same operations, is never above the score of the vector.  A vector
// whose bound does not pass the query's threshold could not have passed it; the bounds that do pass are collected, and before
// anything is handed on the few that remain are scored with the 32-bit table, exactly as the scan of one query does.
// What is returned, and every comparison that orders two results, rests on those scores: the answers are the same bits.
#pragma once
#include "common.cuh"

namespace rago {

constexpr int PAIR_MIN_NQ = 65;    // smaller batches are planned by the selection kernel and merged by a kernel of their own
// Queries of a batch: their keys fit a CTA's static shared memory (every CTA of pair_rank_kernel holds all of them) and carry the query's
// number in 12 bits, and their tables are built ahead.
constexpr int PAIR_MAX_NQ = 4096;
static_assert(PAIR_MAX_NQ * 8 <= 48 * 1024 && PAIR_MAX_NQ <= 1 << 12 && PAIR_MAX_NQ <= PREBUILT_MAX_NQ, "limits of a batch with pairs");
constexpr int PAIR_MAX_K = 512;

struct PairParams {   // of a pair of queries
    int32_t q[2];     // the queries
    int32_t base[2];  // sum_m low(m)
    int32_t shift[2];
    float inv[2];     // fp32 value of one unit of the 32-bit tables
};

// Entries: (list, term) pairs of the whole batch in the order in which they are scanned, nq * nprobe of them.  The first
// 2 * nprobe * head[0] belong to the pairs, 2 * nprobe each: the lists both queries probe, then those of the first, then those
// of the second; what is left of the 2 * nprobe is -1.  The others are the single queries', nprobe each.
struct PairView {
    const int32_t* head;        // [0]: number of pairs
    const int32_t* order;       // [nq]: the queries of pair u at 2u and 2u + 1, after the last pair the single ones
    const float* term_b;        // [entries] the second query's term (pairs)
    const int32_t* mask;        // [entries] bit 0, 1: the first, the second query probes the list
    const uint2* range;         // [2][entries] of either query: storage positions of the list, from, to (1, 0: it does not probe it)
    const PairParams* params;   // [pairs]
    const uint8_t* img;         // [pairs] table images
    int tile_vecs;              // vectors per tile of the pairs' scan
};

// Where a query's entries and slots are (see the scan's slot numbering): position i of the order.
struct PairPlace {
    int e0, per_unit, e_base, e_end;   // first entry, entries; entries of the launch that scanned it
    int slot_base, slot_stride, unit;  // slot of CTA b: slot_base + (unit + b) * slot_stride
};
__host__ __device__ inline PairPlace pair_place(int i, int npairs_q, int nq, int nprobe, int ctas) {
    PairPlace p;
    if (i < 2 * npairs_q) {
        p.unit = i >> 1; p.per_unit = 2 * nprobe; p.e_base = 0; p.e_end = 2 * nprobe * npairs_q;
        p.slot_base = i & 1; p.slot_stride = 2;
    } else {
        p.unit = i - 2 * npairs_q; p.per_unit = nprobe; p.e_base = 2 * nprobe * npairs_q; p.e_end = nq * nprobe;
        p.slot_base = 2 * (npairs_q + ctas); p.slot_stride = 1;
    }
    p.e0 = p.e_base + p.unit * p.per_unit;
    return p;
}
inline size_t pair_slots(int nq, int ctas) { return (size_t)nq + 3 * (size_t)ctas; }

// Workspace of the preparation (offsets from its start).
struct PairLayout {
    size_t head, order, state, entry_list, entry_term, term_b, mask, range, params, img, ok, total;
};
PairLayout pair_layout(int nq, int nprobe, int lut_bytes);
// Whether a batch of these sizes is looked through for pairs.
bool pair_applies(const IndexImpl* ix, int nq, int nprobe, int k);
bool pair_reserves(const IndexImpl* ix, int nq, int nprobe);
void pair_list_stats(IndexImpl* ix, const int64_t* offsets);
cudaError_t launch_pair_queries(const IndexImpl* ix, const int32_t* probe_list, const float* probe_term, int nq, int nprobe,
                                int k, const uint8_t* lut_img, const float* lut_inv, uint8_t* ws, const PairLayout& L, PairView* view,
                                cudaStream_t s);

}  // namespace rago
