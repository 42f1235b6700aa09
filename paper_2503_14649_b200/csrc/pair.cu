// Pairs of queries: which queries of a batch are scanned together, their entries, and their two-in-one tables (pair.cuh).
//
// A pair is two queries whose nearest list is the same one (neighbours after sorting by nearest, then second nearest list)
// and that share enough of their work.  All of it is decided on the device, from the probe lists.
#include <algorithm>
#include <cmath>

#include "pair.cuh"
#include "plan.cuh"
#include "topk.cuh"

namespace rago {

constexpr int PR_THREADS = 256, PR_WARPS = PR_THREADS / 32;
constexpr int PU_THREADS = 128, PU_WARPS = PU_THREADS / 32;  // one warp per query of the sorted order
static_assert(PU_WARPS == 4, "states are counted a word, four positions, at a time");
constexpr uint8_t ST_SINGLE = 0, ST_FIRST = 1, ST_SECOND = 2, ST_NONE = 0xFF;
// A pair shares at least one vector in so many of both queries' work (its tiles cost 10 to 15% more than a query's), and codes of at least so many
// bytes: sharing 2 MB saves a CTA about 30 us, what closing a pair costs beyond closing two queries.  (4 000 queries over 1 024
// lists of 2 150, 8 probes, 64 bytes, every batch looked through: 1 395 us per call without pairs, with all that share 0.2 MB
// 1 802, 1 MB 1 531, 2 MB 1 485; with lists of 30 000 vectors all of them 2 135 to 2 167.)
constexpr int PAIR_SHARE = 8, PAIR_MIN_BYTES = 2 << 20;

// The queries ranked by nearest, then second nearest list; runs of equal nearest lists are split into neighbours.  state[i]: what
// the query at position i of sorted[] is.  A query whose table is not bounded (ok = 0) has no partner.  Every warp counts, for
// its queries, the keys below theirs and the keys of their run (one CTA sorting 1 024 keys took 14 us).
__global__ void __launch_bounds__(PR_THREADS) pair_rank_kernel(const int32_t* __restrict__ probe_list, const int32_t* __restrict__ ok,
                                                               int nq, int nprobe, int32_t* __restrict__ sorted,
                                                               uint8_t* __restrict__ state) {
    __shared__ unsigned long long keys[PAIR_MAX_NQ];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    grid_dependency_wait();
    grid_dependents_may_launch();
    for (int i = tid; i < nq; i += PR_THREADS) {
        const uint32_t l0 = (uint32_t)probe_list[(size_t)i * nprobe];
        const uint32_t l1 = nprobe > 1 ? (uint32_t)probe_list[(size_t)i * nprobe + 1] : 0u;
        const uint32_t run = ok[i] ? l0 : 0x80000000u | (uint32_t)i;  // list numbers have 31 bits, query numbers here 12
        keys[i] = ((unsigned long long)run << 32) | ((l1 & 0xFFFFFu) << 12) | (uint32_t)i;
    }
    __syncthreads();
    for (int i = blockIdx.x * PR_WARPS + warp; i < nq; i += gridDim.x * PR_WARPS) {  // uniform within the warp
        const unsigned long long mine = keys[i];
        int below = 0, run_below = 0, run = 0;
#pragma unroll 4
        for (int j = lane; j < nq; j += 32) {
            const unsigned long long x = keys[j];
            const int less = x < mine ? 1 : 0, same = (uint32_t)(x >> 32) == (uint32_t)(mine >> 32) ? 1 : 0;
            below += less;
            run_below += less & same;
            run += same;
        }
        below = __reduce_add_sync(0xffffffffu, below);
        run_below = __reduce_add_sync(0xffffffffu, run_below);
        run = __reduce_add_sync(0xffffffffu, run);
        if (lane == 0) {
            sorted[below] = i;
            state[below] = (run_below & 1) ? ST_SECOND : (run_below + 1 < run ? ST_FIRST : ST_SINGLE);
        }
    }
    if (blockIdx.x == 0 && tid < 4 && nq + tid < ((nq + 3) & ~3)) state[nq + tid] = ST_NONE;  // the rest of the last word
}

// Whether list x of lane `lane`s query is among the n lists at other: index there, or -1.
__device__ __forceinline__ int index_in(int x, const int32_t* __restrict__ other, int n, int lane) {
    int at = -1;
    for (int b0 = 0; b0 < n; b0 += 32) {
        const int y = b0 + lane < n ? other[b0 + lane] : -2;
        for (int j = 0; j < 32; ++j)
            if (__shfl_sync(0xffffffffu, y, j) == x) at = b0 + j;
    }
    return at;
}

// One warp per position: pairs that share too little are taken apart.
__global__ void __launch_bounds__(PU_THREADS) pair_judge_kernel(const int32_t* __restrict__ probe_list, const int64_t* __restrict__ offsets,
                                                                int nq, int nprobe, long long min_shared,
                                                                const int32_t* __restrict__ sorted, uint8_t* __restrict__ state) {
    const int i = blockIdx.x * PU_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    grid_dependency_wait();
    grid_dependents_may_launch();
    if (i >= nq || state[i] != ST_FIRST) return;
    const int32_t* la = probe_list + (size_t)sorted[i] * nprobe;
    const int32_t* lb = probe_list + (size_t)sorted[i + 1] * nprobe;
    long long shared = 0, total = 0;
    for (int a0 = 0; a0 < nprobe; a0 += 32) {
        const int x = a0 + lane < nprobe ? la[a0 + lane] : -1, y = a0 + lane < nprobe ? lb[a0 + lane] : -1;
        const long long lx = x >= 0 ? offsets[x + 1] - offsets[x] : 0, ly = y >= 0 ? offsets[y + 1] - offsets[y] : 0;
        if (index_in(x, lb, nprobe, lane) >= 0) shared += lx;
        total += lx + ly;
    }
    for (int o = 16; o; o >>= 1) {
        shared += __shfl_xor_sync(0xffffffffu, shared, o);
        total += __shfl_xor_sync(0xffffffffu, total, o);
    }
    if (lane < 2 && (shared < min_shared || shared * PAIR_SHARE < total)) state[i + lane] = ST_SINGLE;
}

// One warp per position: order and entries.
__global__ void __launch_bounds__(PU_THREADS) pair_entries_kernel(const int32_t* __restrict__ probe_list, const float* __restrict__ probe_term,
                                                                  int nq, int nprobe, const int32_t* __restrict__ sorted,
                                                                  const uint8_t* __restrict__ state, int32_t* __restrict__ head,
                                                                  int32_t* __restrict__ order, int32_t* __restrict__ entry_list,
                                                                  float* __restrict__ entry_term, float* __restrict__ term_b,
                                                                  int32_t* __restrict__ mask, const int64_t* __restrict__ offsets,
                                                                  uint2* __restrict__ range) {
    __shared__ int s_before[PU_WARPS][2], s_total[PU_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    grid_dependency_wait();
    grid_dependents_may_launch();
    // pairs in all, pairs and single queries before this CTA's positions
    int total = 0, firsts = 0, singles = 0;
    for (int w = tid; w < (nq + 3) / 4; w += PU_THREADS) {
        const uint32_t st = reinterpret_cast<const uint32_t*>(state)[w];
        const int f = __popc(__vcmpeq4(st, 0x01010101u)) >> 3, g = __popc(__vcmpeq4(st, 0u)) >> 3;
        total += f;
        if (w < (int)blockIdx.x) { firsts += f; singles += g; }
    }
    total = __reduce_add_sync(0xffffffffu, total);
    firsts = __reduce_add_sync(0xffffffffu, firsts);
    singles = __reduce_add_sync(0xffffffffu, singles);
    if (lane == 0) { s_total[warp] = total; s_before[warp][0] = firsts; s_before[warp][1] = singles; }
    __syncthreads();
    total = firsts = singles = 0;
    for (int w = 0; w < PU_WARPS; ++w) { total += s_total[w]; firsts += s_before[w][0]; singles += s_before[w][1]; }
    if (blockIdx.x == 0 && tid == 0) head[0] = total;
    const int i = blockIdx.x * PU_WARPS + warp;
    if (i >= nq) return;
    for (int w = 0; w < warp; ++w) {
        const uint8_t st = state[blockIdx.x * PU_WARPS + w];
        firsts += st == ST_FIRST ? 1 : 0;
        singles += st == ST_SINGLE ? 1 : 0;
    }
    const uint8_t st = state[i];
    if (st == ST_SECOND) return;
    const int qa = sorted[i];
    const int32_t* la = probe_list + (size_t)qa * nprobe;
    const float* ta = probe_term + (size_t)qa * nprobe;
    if (st == ST_SINGLE) {
        const size_t e0 = (size_t)2 * nprobe * total + (size_t)singles * nprobe;
        if (lane == 0) order[2 * total + singles] = qa;
        for (int e = lane; e < nprobe; e += 32) { entry_list[e0 + e] = la[e]; entry_term[e0 + e] = ta[e]; }
        return;
    }
    const int qb = sorted[i + 1];
    const int32_t* lb = probe_list + (size_t)qb * nprobe;
    const float* tb = probe_term + (size_t)qb * nprobe;
    const size_t e0 = (size_t)2 * nprobe * firsts;
    if (lane == 0) { order[2 * firsts] = qa; order[2 * firsts + 1] = qb; }
    const uint32_t lt = (1u << lane) - 1u;
    int n = 0;
    auto put = [&](bool take, int list, float t0, float t1, int m) {
        const uint32_t b = __ballot_sync(0xffffffffu, take);
        if (take) {
            const size_t e = e0 + n + __popc(b & lt);
            entry_list[e] = list; entry_term[e] = t0; term_b[e] = t1; mask[e] = m;
            const uint2 r = make_uint2((uint32_t)offsets[list], (uint32_t)offsets[list + 1]), none = make_uint2(1u, 0u);
            range[e] = m & 1 ? r : none;
            range[(size_t)nq * nprobe + e] = m & 2 ? r : none;
        }
        n += __popc(b);
    };
    for (int part = 0; part < 3; ++part) {  // lists of both, of the first only, of the second only
        const int32_t* mine = part < 2 ? la : lb;
        const float* tm = part < 2 ? ta : tb;
        for (int c0 = 0; c0 < nprobe; c0 += 32) {
            const int c = c0 + lane;
            const int x = c < nprobe ? mine[c] : -1;
            const int at = index_in(x, part < 2 ? lb : la, nprobe, lane);
            const float t = c < nprobe ? tm[c] : 0.f;
            put(x >= 0 && (at >= 0) == (part == 0), x, part < 2 ? t : 0.f, part == 0 ? (at >= 0 ? tb[at] : 0.f) : t, part == 0 ? 3 : (part == 1 ? 1 : 2));
        }
    }
    for (int e = n + lane; e < 2 * nprobe; e += 32) {
        entry_list[e0 + e] = -1; entry_term[e0 + e] = 0.f; term_b[e0 + e] = 0.f; mask[e0 + e] = 0;
        range[e0 + e] = range[(size_t)nq * nprobe + e0 + e] = make_uint2(1u, 0u);
    }
}

// The two 32-bit table images of a pair -> one image of 16-bit halves, and the pair's parameters.  A cluster of PI_CTAS CTAs
// per pair, each with a share of the columns: thread (g, c) keeps four neighbouring columns of every G-th code value in
// registers, so the images are read once, with all of a thread's loads in flight together (one CTA per pair, reading
// them twice: 64 us for 512 pairs of 96 columns, 45 for 38).  The CTAs exchange what the shift and the base are made of.
constexpr int PI_CTAS = 4, PI_THREADS = 256, PI_SHIFTS = 17;
template <int M>
__global__ void __cluster_dims__(PI_CTAS, 1, 1) __launch_bounds__(PI_THREADS) pair_tables_kernel(
    const int32_t* __restrict__ head, const int32_t* __restrict__ order, const uint8_t* __restrict__ lut_img,
    const float* __restrict__ lut_inv, int lut_bytes, int kind, PairParams* __restrict__ params, uint8_t* __restrict__ img) {
    constexpr int COLS = M / PI_CTAS, C4 = COLS / 4, G = PI_THREADS / C4, ROWS = (KSUB + G - 1) / G;
    static_assert(M % (4 * PI_CTAS) == 0, "whole groups of four columns");
    __shared__ alignas(16) int s_mn[2][G][COLS], s_mx[2][G][COLS], low[2][COLS];  // read and written as int4 too
    __shared__ uint32_t range[2][COLS];
    __shared__ int part[2][PI_SHIFTS + 1];  // sums of the ranges >> s over this CTA's columns, and of the lows
    grid_dependency_wait();
    grid_dependents_may_launch();
    const int u = blockIdx.x / PI_CTAS, rank = blockIdx.x % PI_CTAS, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (u >= head[0]) return;  // uniform over the cluster
    const int c = tid % C4, g = tid / C4, col = rank * COLS + c * 4;
    const int q[2] = {order[2 * u], order[2 * u + 1]};
    const uint32_t off0 = lut_offset(kind, 0, col);  // four neighbouring columns lie in one row
    int4 v[2][ROWS];
#pragma unroll
    for (int side = 0; side < 2; ++side)
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int j = g + r * G;
            if (g < G && j < KSUB) v[side][r] = __ldg(reinterpret_cast<const int4*>(lut_img + (size_t)q[side] * lut_bytes + off0 + (uint32_t)j * lut_row(kind)));
        }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        int4 mn = make_int4(0x7FFFFFFF, 0x7FFFFFFF, 0x7FFFFFFF, 0x7FFFFFFF), mx = make_int4(-0x7FFFFFFF, -0x7FFFFFFF, -0x7FFFFFFF, -0x7FFFFFFF);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            if (!(g < G && g + r * G < KSUB)) continue;
            const int4 x = v[side][r];
            mn = make_int4(min(mn.x, x.x), min(mn.y, x.y), min(mn.z, x.z), min(mn.w, x.w));
            mx = make_int4(max(mx.x, x.x), max(mx.y, x.y), max(mx.z, x.z), max(mx.w, x.w));
        }
        if (g < G) {
            *reinterpret_cast<int4*>(&s_mn[side][g][c * 4]) = mn;
            *reinterpret_cast<int4*>(&s_mx[side][g][c * 4]) = mx;
        }
    }
    __syncthreads();
    for (int i = warp; i < 2 * COLS; i += PI_THREADS / 32) {  // uniform within the warp
        const int side = i / COLS, k = i % COLS;
        int mn = 0x7FFFFFFF, mx = -0x7FFFFFFF;
        for (int r = lane; r < G; r += 32) { mn = min(mn, s_mn[side][r][k]); mx = max(mx, s_mx[side][r][k]); }
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) {
            low[side][k] = mn;
            range[side][k] = (uint32_t)mx - (uint32_t)mn;  // |entries| < 2^30 / M + 1: no overflow, here or in the sums
        }
    }
    __syncthreads();
    if (tid < 2 * (PI_SHIFTS + 1)) {
        const int side = tid / (PI_SHIFTS + 1), s = tid % (PI_SHIFTS + 1);
        int sum = 0;
        for (int k = 0; k < COLS; ++k) sum += s < PI_SHIFTS ? (int)(range[side][k] >> s) : low[side][k];
        part[side][s] = sum;
    }
    cluster_sync_all();
    int shift[2], base[2];
#pragma unroll
    for (int side = 0; side < 2; ++side) {  // lane s of every warp: the sum for shift s, lane PI_SHIFTS the base
        int sum = 0;
        if (lane <= PI_SHIFTS)
            for (int r = 0; r < PI_CTAS; ++r) sum += (int)lds_cluster_u32(mapa_shared(smem_u32(&part[side][lane]), (uint32_t)r));
        // the smallest shift with a sum of at most 65 535: the ranges sum to less than 2^31 + M, so 16 is always one
        const uint32_t fits = __ballot_sync(0xffffffffu, lane < PI_SHIFTS && (uint32_t)sum <= 65535u);
        shift[side] = fits ? __ffs(fits) - 1 : PI_SHIFTS - 1;
        base[side] = __shfl_sync(0xffffffffu, sum, PI_SHIFTS);
    }
    cluster_sync_all();  // nobody's sums go away while another CTA reads them
    uint8_t* out = img + (size_t)u * lut_bytes;
    if (g < G) {
        const int4 la = *reinterpret_cast<const int4*>(&low[0][c * 4]), lb = *reinterpret_cast<const int4*>(&low[1][c * 4]);
        auto half2 = [&](int x, int lx, int y, int ly) { return ((uint32_t)(x - lx) >> shift[0]) | (((uint32_t)(y - ly) >> shift[1]) << 16); };
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int j = g + r * G;
            if (j >= KSUB) continue;
            const int4 x = v[0][r], y = v[1][r];
            const uint4 e = make_uint4(half2(x.x, la.x, y.x, lb.x), half2(x.y, la.y, y.y, lb.y), half2(x.z, la.z, y.z, lb.z), half2(x.w, la.w, y.w, lb.w));
            *reinterpret_cast<uint4*>(out + off0 + (uint32_t)j * lut_row(kind)) = e;
            if (kind == LUT_DOT2) *reinterpret_cast<uint4*>(out + off0 + (uint32_t)j * lut_row(kind) + LUT_COPY) = e;
        }
    }
    if (rank == 0 && tid < 2) {
        PairParams* p = params + u;
        p->q[tid] = tid ? q[1] : q[0]; p->base[tid] = tid ? base[1] : base[0]; p->shift[tid] = tid ? shift[1] : shift[0];
        p->inv[tid] = lut_inv[tid ? q[1] : q[0]];
    }
}

// ---- host side ----------------------------------------------------------------------------------
// Lists by the bits of their length: what is needed of the list lengths to guess how much of a batch is shared.
void pair_list_stats(IndexImpl* ix, const int64_t* offsets) {
    double w[33] = {}, w2[33] = {};
    for (int l = 0; l < ix->nlist; ++l) {
        const int64_t n = offsets[l + 1] - offsets[l];
        if (n <= 0) continue;
        int b = 0;
        while (b < 32 && (n >> b) > 1) ++b;
        const double x = (double)n / (double)ix->N;
        w[b] += x;
        w2[b] += x * x;
    }
    for (int b = 0; b <= 32; ++b) { ix->list_weight[b] = (float)w[b]; ix->list_square[b] = (float)w2[b]; }
}

// Vectors a query scans, how many of them it is expected to share with a partner, and the share of queries that have one, if queries come as
// the stored vectors do: a query's nearest list has weight w with probability w, then nq w others have the same one, and the share of them that
// finds a partner is 1 - (1 - e^-2x) / 2x for x = nq w (an odd number leaves one over).  Partners share their nearest list and,
// since it is where they both lie, about half of the others.
static void pair_expect(const IndexImpl* ix, int nq, int nprobe, double* scanned, double* shared, double* paired_share) {
    double own = 0.0, own_shared = 0.0, paired = 0.0;
    for (int b = 0; b <= 32; ++b) {
        if (!(ix->list_weight[b] > 0.f)) continue;
        const double x = (double)nq * ix->list_square[b] / ix->list_weight[b];
        const double f = x > 1e-6 ? 1.0 - (1.0 - std::exp(-2.0 * x)) / (2.0 * x) : 0.0;
        own += ix->list_square[b];
        own_shared += f * ix->list_square[b];
        paired += f * ix->list_weight[b];
    }
    const double others = (double)(nprobe - 1) / (double)ix->nlist;
    *scanned = (double)ix->N * (own + others);
    *shared = (double)ix->N * (own_shared + 0.5 * paired * others);
    *paired_share = paired;
}

static bool pair_possible(const IndexImpl* ix, int nq, int k) {
    const int ds = ix->dsub;
    return nq >= PAIR_MIN_NQ && nq <= PAIR_MAX_NQ && k <= PAIR_MAX_K && ix->plan.pairs && ix->N > 0 &&
           (ds == 4 || ds == 8 || ds == 12 || ds == 16);  // those whose table kernel checks the tables' bound
}
// What of a batch is shared saves less than half of its look-ups.  Against that stand, in us: the preparation, 20 to 50 and, where every list
// of a query is looked for among its partner's, 1 000 for 1 024 probes (more than about 1 200 queries queue for the SMs); and closing a pair on
// each CTA that scans part of it, 40 and more with k beyond closing two queries (4 000 queries over 1 024 lists of 2 150, whose CTAs
// close 13 pairs each: 64 bytes, 4 probes, without / with pairs 973 / 1 426 us per call, 96 bytes, 8 probes 1 803 / 2 032).
// Below PAIR_MIN_US the two sides could not be told apart.  Where the rule says yes, without / with: 1 024 queries, 87% of their work in
// lists that others share, 96 bytes 8 460 / 5 610; 300 queries, 48 bytes 1 466 / 1 192; 77 queries, 96 bytes (expected saving 290 us)
// 683 / 670; 500 queries, 256 of 512 lists of 1 950, 96 bytes 4 935 / 4 222; 1 000 queries, 1 024 lists of 1 950, all probed 40 100 / 31 160.
constexpr double PAIR_MIN_SHARE = 0.2, PAIR_MIN_US = 120.0, PAIR_BYTES_PER_US = 4.7e6;
constexpr double PAIR_PREPARE_US = 60.0, PAIR_MATCH_US = 1000.0, PAIR_CLOSE_US = 40.0, PAIR_CLOSE_K_US = 0.08;
static bool pair_worth(const IndexImpl* ix, int nq, int nprobe, int k) {
    double scanned, shared, paired;
    pair_expect(ix, nq, nprobe, &scanned, &shared, &paired);
    const double p = nprobe / 1024.0, closed = 0.5 * nq * paired / ix->plan.ctas + 1.0;  // pairs that a CTA closes
    const double cost = PAIR_PREPARE_US + PAIR_MATCH_US * p * p * (1.0 + nq / 1200.0) + closed * (PAIR_CLOSE_US + PAIR_CLOSE_K_US * k);
    return shared >= PAIR_MIN_SHARE * scanned && 0.5 * shared * nq * ix->M >= std::max(cost, PAIR_MIN_US) * PAIR_BYTES_PER_US;
}
bool pair_applies(const IndexImpl* ix, int nq, int nprobe, int k) { return pair_possible(ix, nq, k) && pair_worth(ix, nq, nprobe, k); }
// Workspace is set aside where any k, and any number of probes up to nprobe, takes pairs: the shared part is a ratio of two
// linear functions of it, so largest at one end, and the amount grows with it (what it has to exceed is at least PAIR_MIN_US).
bool pair_reserves(const IndexImpl* ix, int nq, int nprobe) {
    if (!pair_possible(ix, nq, 1)) return false;
    double s1, h1, s2, h2, paired;
    pair_expect(ix, nq, 1, &s1, &h1, &paired);
    pair_expect(ix, nq, nprobe, &s2, &h2, &paired);
    return (h1 >= PAIR_MIN_SHARE * s1 || h2 >= PAIR_MIN_SHARE * s2) && 0.5 * h2 * nq * ix->M >= PAIR_MIN_US * PAIR_BYTES_PER_US;
}

PairLayout pair_layout(int nq, int nprobe, int lut_bytes) {
    PairLayout L;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += align_up(bytes ? bytes : 1, 256);
        return at;
    };
    const size_t e = (size_t)nq * nprobe * 4;
    L.head = take(4);
    L.ok = take((size_t)nq * 4);
    L.order = take((size_t)nq * 8);  // sorted, then the final order
    L.state = take((size_t)nq + 4);
    L.entry_list = take(e); L.entry_term = take(e); L.term_b = take(e); L.mask = take(e); L.range = take(4 * e);
    L.params = take((size_t)(nq / 2) * sizeof(PairParams));
    L.img = take((size_t)(nq / 2) * lut_bytes);
    L.total = o;
    return L;
}

cudaError_t launch_pair_queries(const IndexImpl* ix, const int32_t* probe_list, const float* probe_term, int nq, int nprobe,
                                int k, const uint8_t* lut_img, const float* lut_inv, uint8_t* ws, const PairLayout& L, PairView* view,
                                cudaStream_t s) {
    int32_t* head = reinterpret_cast<int32_t*>(ws + L.head);
    const int32_t* ok = reinterpret_cast<const int32_t*>(ws + L.ok);
    int32_t* sorted = reinterpret_cast<int32_t*>(ws + L.order);
    int32_t* order = sorted + nq;
    uint8_t* state = ws + L.state;
    int32_t* entry_list = reinterpret_cast<int32_t*>(ws + L.entry_list);
    float* entry_term = reinterpret_cast<float*>(ws + L.entry_term);
    float* term_b = reinterpret_cast<float*>(ws + L.term_b);
    int32_t* mask = reinterpret_cast<int32_t*>(ws + L.mask);
    PairParams* params = reinterpret_cast<PairParams*>(ws + L.params);
    uint2* range = reinterpret_cast<uint2*>(ws + L.range);
    uint8_t* img = ws + L.img;
    const ScanPlan& pl = ix->plan;
    const dim3 grid((nq + PU_WARPS - 1) / PU_WARPS);
    const int rank_ctas = (nq + PR_WARPS - 1) / PR_WARPS;
    cudaError_t e = launch_overlapped(pair_rank_kernel, dim3(rank_ctas < ix->num_sms ? rank_ctas : ix->num_sms), dim3(PR_THREADS), 0, s,
                                      probe_list, ok, nq, nprobe, sorted, state);
    if (e == cudaSuccess)
        e = launch_overlapped(pair_judge_kernel, grid, dim3(PU_THREADS), 0, s, probe_list, ix->list_offsets, nq, nprobe,
                              (long long)(PAIR_MIN_BYTES / ix->M), sorted, state);
    if (e == cudaSuccess)
        e = launch_overlapped(pair_entries_kernel, grid, dim3(PU_THREADS), 0, s, probe_list, probe_term, nq, nprobe, sorted, state, head,
                              order, entry_list, entry_term, term_b, mask, ix->list_offsets, range);
    if (e != cudaSuccess) return e;
    auto tables = [&](auto kernel) {
        return launch_overlapped(kernel, dim3(PI_CTAS * (nq / 2)), dim3(PI_THREADS), 0, s, head, order, lut_img, lut_inv, pl.lut_bytes,
                                 pl.lut_kind, params, img);
    };
    switch (ix->M) {
        case 16: e = tables(pair_tables_kernel<16>); break;
        case 32: e = tables(pair_tables_kernel<32>); break;
        case 48: e = tables(pair_tables_kernel<48>); break;
        case 64: e = tables(pair_tables_kernel<64>); break;
        case 96: e = tables(pair_tables_kernel<96>); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    count_launch(4);
    view->head = head; view->order = order; view->term_b = term_b; view->mask = mask; view->range = range; view->params = params; view->img = img;
    view->tile_vecs = scan_pair_tile_vecs(ix, k);
    return cudaGetLastError();
}

}  // namespace rago
