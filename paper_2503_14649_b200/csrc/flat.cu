// Exact flat search: score = <q, y_i> over bf16 inputs, fp32 accumulation, k largest per query.
//
// Main path (k <= 960): the tensor-core kernel of gemm_select.cu with rows = queries and columns =
// database rows; every CTA streams its own share of the database once (both 128-query row tiles are
// multiplied against a database tile while it is hot) and keeps each query's k best of that range;
// flat_merge_kernel merges the ranges.  No score is ever written to memory.
// Fallback (larger k): the database is processed in panels of PANEL rows on the fp32 pipes: scores of
// a panel go to scratch, each (query, 64K-row chunk) keeps its k best, and the same merge finishes.
#include "topk.cuh"

namespace rago {

constexpr int FBM = 64, FBN = 64, FBK = 16;
constexpr int FLAT_CHUNK = 1 << 16;   // rows per selection chunk
constexpr int FLAT_PANEL = 1 << 20;   // rows scored per pass

__global__ void __launch_bounds__(256) flat_scores_kernel(const __nv_bfloat16* __restrict__ Q,
                                                          const __nv_bfloat16* __restrict__ Y, int nq,
                                                          long long row_begin, int nrows, int d,
                                                          float* __restrict__ scores) {
    __shared__ __align__(16) float As[FBK][FBM + 4];
    __shared__ __align__(16) float Bs[FBK][FBN + 4];
    const int tid = threadIdx.x;
    const int row0 = blockIdx.y * FBM, col0 = blockIdx.x * FBN;
    const int lr = tid >> 2, lk = (tid & 3) * 4;
    const int ty = tid >> 4, tx = tid & 15;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < d; k0 += FBK) {
        float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
        if (row0 + lr < nq) {
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = __bfloat162float(Q[(size_t)(row0 + lr) * d + k0 + lk + i]);
        }
        if (col0 + lr < nrows) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                b[i] = __bfloat162float(Y[(size_t)(row_begin + col0 + lr) * d + k0 + lk + i]);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            As[lk + i][lr] = a[i];
            Bs[lk + i][lr] = b[i];
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < FBK; ++kk) {
            const float4 av = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
            const float4 bv = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
            const float ar[4] = {av.x, av.y, av.z, av.w}, br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = row0 + ty * 4 + i;
        if (r >= nq) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = col0 + tx * 4 + j;
            if (c < nrows) scores[(size_t)r * FLAT_PANEL + c] = -acc[i][j];  // smaller = better
        }
    }
}

constexpr int FSEL_THREADS = 256;

// grid (chunks in panel, nq): k best of one chunk of one query -> slot (q, global chunk).
__global__ void __launch_bounds__(FSEL_THREADS) flat_select_kernel(const float* __restrict__ scores,
                                                                   long long row_begin, int nrows, int k,
                                                                   int chunk_begin, int nchunks_total,
                                                                   int32_t* __restrict__ slot_cnt,
                                                                   unsigned long long* __restrict__ slot_keys) {
    __shared__ unsigned long long keys[TOPK_CAP];
    __shared__ int cnt;
    const int tid = threadIdx.x, q = blockIdx.y, ch = blockIdx.x;
    auto sync = [] { __syncthreads(); };
    if (tid == 0) cnt = 0;
    __syncthreads();
    const int c0 = ch * FLAT_CHUNK;
    int c1 = c0 + FLAT_CHUNK;
    if (c1 > nrows) c1 = nrows;
    const float* srow = scores + (size_t)q * FLAT_PANEL;
    unsigned long long tau = KEY_MAX;
    int ub = 0;
    for (int i0 = c0; i0 < c1; i0 += FSEL_THREADS) {
        const int i = i0 + tid;
        unsigned long long key = KEY_MAX;
        if (i < c1) key = make_key(srow[i], (uint32_t)(row_begin + i));
        warp_push(keys, &cnt, i < c1 && key < tau, key);
        ub += FSEL_THREADS;
        if (ub + FSEL_THREADS > TOPK_CAP) {
            __syncthreads();
            const int kept = block_select(keys, &cnt, k, tid, FSEL_THREADS, sync);
            if (kept == k) tau = keys[k - 1];
            ub = kept;
            __syncthreads();
        }
    }
    __syncthreads();
    const int kept = block_select(keys, &cnt, k, tid, FSEL_THREADS, sync);
    const size_t slot = (size_t)q * nchunks_total + chunk_begin + ch;
    for (int i = tid; i < kept; i += FSEL_THREADS) slot_keys[slot * k + i] = keys[i];
    if (tid == 0) slot_cnt[slot] = kept;
}

// Final selection of a query: the k best of its candidate lists, best first.
//
// List l of query q holds slot_cnt entries at slot_keys[(q * nlists + l) * stride ...]; with `raw` they are the raw
// candidate entries of the tensor-core kernel (cand_key turns them into keys).  Latency is what counts here: a query
// has a few hundred short lists (one per share of the columns and half tile), and walking them one after the other cost
// about a microsecond per list (290 us for one query over 100 000 rows, 264 us for 37 over a million, 308 us for 256
// over ten million).  So the counts of up to FM_LISTS lists are fetched at once and summed, the entries are numbered
// through, and every thread fetches FM_KPT of them side by side; a counting bisection on the keys (distinct, so it
// always ends) finds a cut with between k and k + k/4 + 8 keys at or below it, and only those are ranked.  More
// entries than one round holds go through further rounds against the cut of the rounds before.
//
// nq * parts CTAs.  Without starting thresholds a list keeps what it saw up to its capacity, and one CTA would pull a hundred
// thousand entries through one SM; a small batch then splits a query's lists into parts.  Each part leaves its keys in
// the storage of its own first list (read by nobody else), and the part that finishes last (a ticket per query, zero
// before the launch) selects among what the parts left.
constexpr int FM_THREADS = 512, FM_KPT = 8, FM_LISTS = 512;
constexpr int FM_ENTRIES = FM_THREADS * FM_KPT;  // entries of one round
constexpr int FM_MAX_PARTS = 32;
constexpr int FM_OLD = 4;                        // keys of earlier rounds a thread takes back: at most MAX_K * 5 / 4 + 8 in all
static_assert(FM_OLD * FM_THREADS >= TOPK_CAP && MAX_K + MAX_K / 4 + 8 <= TOPK_CAP, "a round's survivors fit the buffer");
constexpr int FM_TICKET_WORD = 32;               // tickets lie in the error block, one word per query
constexpr int FM_TICKETS = 64 - FM_TICKET_WORD;

struct FlatMergeState {
    unsigned long long keys[TOPK_CAP];
    int pre[FM_LISTS + 1];
    int wsum[FM_THREADS / 32];
    unsigned long long mn, mx;
    uint32_t nv, round[3];
    int cnt, last;
};

// Most keys a part leaves; the short selection ranks WARP_SORT_MAX as fast as fewer.
__host__ __device__ inline int flat_merge_most(int k) { return k + (k >> 2) + 8 > WARP_SORT_MAX ? k + (k >> 2) + 8 : WARP_SORT_MAX; }

// Adds the entries of lists slot_of(l), l0 <= l < l1 (count cnts[slot], entries at entries[slot * stride ...]), to the
// keys the buffer holds and leaves there the min(k, all) smallest and a few more: at most flat_merge_most(k), in the last pass
// (`last`) what sorts as fast, or up to TOPK_CAP where the last FM_LISTS lists turn out to be empty.
template <class SlotOf>
__device__ __forceinline__ void flat_merge_lists(FlatMergeState& S, const int32_t* cnts, const unsigned long long* entries,
                                                 int l0, int l1, SlotOf slot_of, int stride, int raw, uint32_t raw_sign,
                                                 int k, bool last) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t want_max = (uint32_t)flat_merge_most(k);
    if (last && k > RANK_MAX) {  // sorted, not ranked: up to the next power of two costs the same, beyond it twice as much
        const uint32_t pow2 = 1u << (32 - __clz(k - 1));
        if (pow2 >= (uint32_t)(k + (k >> 6) + 4)) want_max = pow2;
    }
    // Of n_all entries, n_seen seen and n_held of those at or below the bound: would the rest pass into the buffer?
    auto rest_fits = [](int n_held, int n_seen, int n_all) {
        const float rest = (float)n_held * (float)(n_all - n_seen) / (float)n_seen;
        return rest + 4.f * sqrtf(rest) + (float)n_held <= (float)TOPK_CAP;
    };
    unsigned long long bound = KEY_MAX - 1;  // nothing above it can be a result
    for (int g0 = l0; g0 < l1; g0 += FM_LISTS) {
        const int ng = l1 - g0 < FM_LISTS ? l1 - g0 : FM_LISTS;
        {   // exclusive prefix of the counts (FM_LISTS <= FM_THREADS: one list per thread)
            const int c = tid < ng ? list_count(__ldcg(cnts + slot_of(g0 + tid)), stride) : 0;
            int incl = c;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) S.wsum[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                int w = lane < FM_THREADS / 32 ? S.wsum[lane] : 0;
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, w, o);
                    if (lane >= o) w += y;
                }
                if (lane < FM_THREADS / 32) S.wsum[lane] = w;
            }
            __syncthreads();
            if (tid < ng) S.pre[tid + 1] = (warp ? S.wsum[warp - 1] : 0) + incl;
            if (tid == 0) S.pre[0] = 0;
        }
        __syncthreads();
        const int nitems = S.pre[ng];
        // Many entries: once the bound of the rounds taken leaves so few of the rest that they fit the buffer (after one
        // round for k = 10; 17 of 65 for k = 400), the rest is streamed past it, a warp per list and with no numbering, at a
        // tenth of the instructions of a round.  If it does not fit after all (rows in an order of their own), the
        // pass counts for nothing and the other rounds are taken.  Streaming after the first round whatever k threw the
        // pass away for large k: 33 queries over 250 001 rows, k = 400, 644 us, this 272.
        bool tried = false;
        for (int r0 = 0; r0 < nitems; r0 += FM_ENTRIES) {  // uniform
            if (!tried && nitems - r0 > FM_ENTRIES && bound != KEY_MAX - 1 && r0 > 0 && rest_fits(S.cnt, r0, nitems)) {
                tried = true;
                const int before = S.cnt;
                __syncthreads();
                const uint32_t bound32 = (uint32_t)(bound >> 32);
                for (int l = warp; l < ng; l += FM_THREADS / 32) {
                    const int skip = r0 - S.pre[l], n = S.pre[l + 1] - S.pre[l];  // entries the rounds have seen
                    const unsigned long long* src = entries + (size_t)slot_of(g0 + l) * stride;
                    for (int i0 = skip > 0 ? skip : 0; i0 < n; i0 += 32 * FM_KPT) {
                        unsigned long long e[FM_KPT];
                        bool any = false;
#pragma unroll
                        for (int j = 0; j < FM_KPT; ++j) {
                            const int i = i0 + 32 * j + lane;
                            e[j] = i < n ? __ldcg(src + i) : KEY_MAX;
                        }
#pragma unroll
                        for (int j = 0; j < FM_KPT; ++j) {
                            if (i0 + 32 * j + lane < n && raw) e[j] = cand_key(e[j], raw_sign);
                            any = any || (uint32_t)(e[j] >> 32) <= bound32;
                        }
                        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
                        for (int j = 0; j < FM_KPT; ++j) warp_push(S.keys, &S.cnt, e[j] <= bound, e[j]);
                    }
                }
                __syncthreads();
                if (S.cnt <= TOPK_CAP) {  // uniform
                    r0 = nitems;  // one last round with no new entries, which cuts the buffer
                } else {
                    __syncthreads();
                    if (tid == 0) S.cnt = before;  // the rounds' keys are intact; the pushes that fitted lie behind them
                    __syncthreads();
                }
            }
            unsigned long long mine[FM_KPT + FM_OLD];
            unsigned long long mn = KEY_MAX, mx = 0ull;
            uint32_t nv = 0;
#pragma unroll
            for (int j = 0; j < FM_KPT; ++j) {
                const int e = r0 + j * FM_THREADS + tid;
                mine[j] = KEY_MAX;
                if (e < nitems) {
                    int lo = 0, hi = ng;  // pre[lo] <= e < pre[hi]
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (S.pre[mid] <= e) lo = mid; else hi = mid;
                    }
                    mine[j] = __ldcg(entries + (size_t)slot_of(g0 + lo) * stride + (e - S.pre[lo]));
                }
            }
#pragma unroll
            for (int j = 0; j < FM_KPT; ++j) {
                if (r0 + j * FM_THREADS + tid >= nitems) continue;
                if (raw) mine[j] = cand_key(mine[j], raw_sign);
                if (mine[j] > bound) mine[j] = KEY_MAX;
            }
            const int old = S.cnt;
#pragma unroll
            for (int j = 0; j < FM_OLD; ++j) {
                const int i = tid + j * FM_THREADS;
                mine[FM_KPT + j] = i < old ? S.keys[i] : KEY_MAX;
            }
#pragma unroll
            for (int j = 0; j < FM_KPT + FM_OLD; ++j) {
                if (mine[j] == KEY_MAX) continue;
                mn = mine[j] < mn ? mine[j] : mn;
                mx = mine[j] > mx ? mine[j] : mx;
                ++nv;
            }
            if (tid == 0) { S.mn = KEY_MAX; S.mx = 0ull; S.nv = 0u; S.round[0] = S.round[1] = S.round[2] = 0u; }
            __syncthreads();  // the old keys and their count have been read, the shared words are initialised
            if (tid == 0) S.cnt = 0;
            nv = __reduce_add_sync(0xffffffffu, nv);
            if (nv) {  // uniform within the warp
                for (int o = 16; o; o >>= 1) {
                    const unsigned long long a = shfl_xor_u64(mn, o), b = shfl_xor_u64(mx, o);
                    mn = a < mn ? a : mn;
                    mx = b > mx ? b : mx;
                }
                if (lane == 0) { atomicMin(&S.mn, mn); atomicMax(&S.mx, mx); atomicAdd(&S.nv, nv); }
            }
            __syncthreads();
            uint32_t c_hi = S.nv;
            // First on the score words alone (half the instructions of a 64-bit compare), then, if a group of equal
            // scores is still too large, on whole keys: #(key <= lo) <= k and #(key <= hi) >= k throughout.
            long long lo32 = (long long)(S.mn >> 32) - 1, hi32 = (long long)(S.mx >> 32);
            int round = 0;
            auto count = [&](auto below) {
                uint32_t c = 0;
#pragma unroll
                for (int j = 0; j < FM_KPT + FM_OLD; ++j) c += below(mine[j]) ? 1u : 0u;  // never true of an empty slot
                c = __reduce_add_sync(0xffffffffu, c);
                const int slot = round % 3;
                if (lane == 0 && c) atomicAdd(&S.round[slot], c);
                if (tid == 0) S.round[(slot + 1) % 3] = 0u;  // next round's word; its last readers passed two barriers ago
                __syncthreads();
                ++round;
                return S.round[slot];
            };
            // more entries follow and all survivors fit the buffer: no cut yet, the next rounds go by the old bound, unless
            // a cut now lets the rest be streamed
            const bool more = r0 + FM_ENTRIES < nitems || g0 + FM_LISTS < l1;
            const bool cut_to_stream = !tried && nitems - r0 > 2 * FM_ENTRIES && rest_fits((int)want_max, r0 + FM_ENTRIES, nitems);
            unsigned long long hi = KEY_MAX - 1;
            if (c_hi > (more && !cut_to_stream ? (uint32_t)TOPK_CAP : want_max)) {  // uniform
                while (hi32 - lo32 > 1 && c_hi > want_max) {
                    const uint32_t mid = bisect_mid(lo32, hi32, round);
                    const uint32_t c = count([&](unsigned long long x) { return (uint32_t)(x >> 32) <= mid; });
                    if (c < (uint32_t)k) lo32 = mid; else { hi32 = mid; c_hi = c; }
                }
                hi = ((unsigned long long)hi32 << 32) | 0xFFFFFFFFull;
                unsigned long long lo = (unsigned long long)hi32 << 32;
                while (hi - lo > 1 && c_hi > want_max) {  // only when the scores left are all equal
                    const unsigned long long mid = lo + (hi - lo) / 2;
                    const uint32_t c = count([&](unsigned long long x) { return x <= mid; });
                    if (c < (uint32_t)k) lo = mid; else { hi = mid; c_hi = c; }
                }
                bound = hi;  // at least k keys lie at or below it
            }
#pragma unroll
            for (int j = 0; j < FM_KPT + FM_OLD; ++j) warp_push(S.keys, &S.cnt, mine[j] <= hi && mine[j] != KEY_MAX, mine[j]);
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(FM_THREADS, 2) flat_merge_kernel(int nlists, int parts, int k, int stride, int raw, uint32_t raw_sign,
                                                                int32_t* __restrict__ slot_cnt,
                                                                unsigned long long* __restrict__ slot_keys,
                                                                uint32_t* __restrict__ tickets,
                                                                int64_t* __restrict__ out_ids,
                                                                float* __restrict__ out_scores) {
    __shared__ FlatMergeState S;
    grid_dependency_wait();
    grid_dependents_may_launch();
    const int tid = threadIdx.x, q = blockIdx.x / parts, part = blockIdx.x % parts;
    if (!raw && nlists == 1) {  // uniform: one chunk of at most k keys, which flat_select_kernel left in order
        const int n = list_count(slot_cnt[q], k);
        for (int i = tid; i < k; i += FM_THREADS) {
            const unsigned long long key = i < n ? slot_keys[(size_t)q * stride + i] : KEY_MAX;
            out_ids[(size_t)q * k + i] = i < n ? (int64_t)(uint32_t)(key & 0xFFFFFFFFull) : -1;
            out_scores[(size_t)q * k + i] = i < n ? -orderable_f32((uint32_t)(key >> 32)) : __int_as_float(0xff800000);
        }
        return;
    }
    auto sync = [] { __syncthreads(); };
    if (tid == 0) S.cnt = 0;
    __syncthreads();
    int32_t* cnts = slot_cnt + (size_t)q * nlists;
    unsigned long long* entries = slot_keys + (size_t)q * nlists * stride;
    int l0 = (int)((long long)part * nlists / parts), l1 = (int)((long long)(part + 1) * nlists / parts);
    const int first = l0;
    for (int pass = 0;; ++pass) {
        // second pass: the first lists of all parts
        auto slot_of = [&](int l) { return pass ? (int)((long long)l * nlists / parts) : l; };
        flat_merge_lists(S, cnts, entries, l0, l1, slot_of, stride, pass ? 0 : raw, raw_sign, k, pass || parts == 1);
        if (pass || parts == 1) break;  // uniform
        const int n = S.cnt;  // at most flat_merge_most(k) <= stride: the launcher checked (a part has at most FM_LISTS lists)
        for (int i = tid; i < n; i += FM_THREADS) entries[(size_t)first * stride + i] = S.keys[i];
        if (tid == 0) cnts[first] = n;
        __syncthreads();  // the part's keys and count are written ...
        if (tid == 0) {
            __threadfence();  // ... and ordered before the ticket
            S.last = atomicAdd(tickets + q, 1u) == (uint32_t)(parts - 1) ? 1 : 0;
            __threadfence();
            S.cnt = 0;
        }
        __syncthreads();
        if (!S.last) return;  // uniform
        l0 = 0;
        l1 = parts;
    }
    const int kept = block_select_short(S.keys, &S.cnt, k, tid, FM_THREADS, sync);
    for (int i = tid; i < k; i += FM_THREADS) {
        int64_t id = -1;
        float sc = __int_as_float(0xff800000);
        if (i < kept) {
            id = (int64_t)(uint32_t)(S.keys[i] & 0xFFFFFFFFull);
            sc = -orderable_f32((uint32_t)(S.keys[i] >> 32));
        }
        out_ids[(size_t)q * k + i] = id;
        out_scores[(size_t)q * k + i] = sc;
    }
}

static int sm_count() {
    static int sms = 0;
    if (!sms) {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0)
            sms = n;
        else {
            cudaGetLastError();
            return 148;  // no device yet (size queries on a host without one): the B200 count
        }
    }
    return sms;
}

static bool flat_on_tensor_cores(int d, int k) { return gemm_cand_cap(k) != 0 && d % 8 == 0; }

// Pilot pass of the flat search: worth it for large databases; the sample must hold 4 k rows.  Whole column tiles: the
// score matrix then has 16-byte aligned rows and takes 16-byte stores (with 32 679 columns, stored one float at a
// time, the pilot of 256 queries took 88 us).
static int flat_pilot_cols(int64_t N, int k) {
    if (N < (1 << 18)) return 0;
    const int64_t np = N / gemm_pilot_stride(N) / 256 * 256;
    return np >= 4LL * k ? (int)np : 0;
}

// Workspace, tensor-core path: [err 256 B][cand nq*nlists*cap u64][cand_cnt nq*nlists i32][pilot scores nq*np f32][row_tau nq f32]
//            (nlists = shares of the grid x GEMM_COL_HALVES candidate lists per query)
//            fallback:         [err 256 B][scores nq*PANEL f32][slot_cnt nq*nchunks i32][slot_keys nq*nchunks*k u64]
size_t flat_workspace_bytes(int64_t N, int d, int nq, int k) {
    if (flat_on_tensor_cores(d, k)) {
        int mg, nsplit, mgroups;
        gemm_grid(nq > 0 ? nq : 1, N > 0 ? N : 1, d, sm_count(), &mg, &nsplit, &mgroups);
        const size_t nlists = (size_t)nsplit * GEMM_COL_HALVES;
        return 256 + align_up((size_t)nq * nlists * gemm_cand_cap(k) * 8, 256) + align_up((size_t)nq * nlists * 4, 256) +
               align_up((size_t)nq * flat_pilot_cols(N, k) * 4, 256) + align_up((size_t)nq * 4, 256);
    }
    const size_t nchunks = (size_t)((N + FLAT_CHUNK - 1) / FLAT_CHUNK);
    size_t b = 256;
    b += align_up((size_t)nq * FLAT_PANEL * 4, 256);
    b += align_up((size_t)nq * (nchunks ? nchunks : 1) * 4, 256);
    b += align_up((size_t)nq * (nchunks ? nchunks : 1) * k * 8, 256);
    return b;
}

cudaError_t launch_flat_search(const void* db, int64_t N, int d, const void* queries, int nq, int k, int64_t* out_ids,
                               float* out_scores, void* workspace, cudaStream_t s) {
    if (flat_on_tensor_cores(d, k) && N > 0) {
        cudaError_t e = gemm_select_init();
        if (e != cudaSuccess) return e;
        int mg, nsplit, mgroups;
        gemm_grid(nq, N, d, sm_count(), &mg, &nsplit, &mgroups);
        const int cap = gemm_cand_cap(k);
        const int nlists = nsplit * GEMM_COL_HALVES;
        uint8_t* w = static_cast<uint8_t*>(workspace) + 256;
        unsigned long long* cand = reinterpret_cast<unsigned long long*>(w);
        w += align_up((size_t)nq * nlists * cap * 8, 256);
        int32_t* cand_cnt = reinterpret_cast<int32_t*>(w);
        w += align_up((size_t)nq * nlists * 4, 256);
        const int np = flat_pilot_cols(N, k);
        float* pilot_scores = reinterpret_cast<float*>(w);
        w += align_up((size_t)nq * np * 4, 256);
        float* row_tau = reinterpret_cast<float*>(w);
        alignas(64) unsigned char tmap_a[128], tmap_b[128], tmap_bh[128];
        e = make_tmap_bf16(tmap_a, queries, (uint64_t)nq, (uint64_t)d, 128);
        if (e == cudaSuccess) e = make_tmap_bf16(tmap_b, db, (uint64_t)N, (uint64_t)d, 256);
        if (e == cudaSuccess) e = make_tmap_bf16(tmap_bh, db, (uint64_t)N, (uint64_t)d, 128);
        if (e != cudaSuccess) return e;
        GemmLaunch G;
        G.tmap_a = tmap_a; G.tmap_b = tmap_b; G.tmap_b_half = tmap_bh;
        G.nrows = nq; G.ncols = N; G.d = d;
        G.a_part_rows = nq; G.b_part_rows = N;
        G.nterms = 1;
        for (int t = 0; t < 6; ++t) G.term_a[t] = G.term_b[t] = 0;
        G.mg = mg; G.nsplit = nsplit;
        G.alpha = -1.f;  // smaller = better
        G.colterm = nullptr; G.colterm_stride = 1;
        G.row_tau = nullptr;
        G.mode = 0; G.nsel = k < N ? k : (int)N; G.cap = cap;
        G.cand = cand; G.cand_cnt = cand_cnt; G.scores = nullptr;
        G.err = static_cast<uint32_t*>(workspace);
        G.clear_block = np ? nullptr : G.err;  // the first launch clears the error block and the tickets in it
        if (np) {
            // pilot pass over every stride-th row: each query starts from the k-th best score of that sample
            alignas(64) unsigned char tmap_p[128], tmap_ph[128];
            const int ps = gemm_pilot_stride(N);
            e = make_tmap_bf16(tmap_p, db, (uint64_t)np, (uint64_t)d, 256, (uint64_t)ps * d);
            if (e == cudaSuccess) e = make_tmap_bf16(tmap_ph, db, (uint64_t)np, (uint64_t)d, 128, (uint64_t)ps * d);
            if (e != cudaSuccess) return e;
            GemmLaunch P = G;
            int pg = 1;
            P.tmap_b = tmap_p; P.tmap_b_half = tmap_ph;
            P.ncols = np; P.b_part_rows = np;
            gemm_grid(nq, np, d, sm_count(), &P.mg, &P.nsplit, &pg);
            P.mode = 1; P.scores = pilot_scores;
            P.clear_block = G.err;
            e = launch_gemm_select(P, s);
            if (e == cudaSuccess) e = launch_row_tau(pilot_scores, nq, np, G.nsel, row_tau, s);
            if (e != cudaSuccess) return e;
            G.row_tau = row_tau;
        }
        e = launch_gemm_select(G, s);
        if (e != cudaSuccess) return e;
        // Parts per query: a starting threshold leaves a few thousand entries per query, one round of one CTA; without
        // one, parts of half a round each while the batch alone does not fill the GPU.
        int parts = 1;
        if (!np && nq <= FM_TICKETS && flat_merge_most(k) <= cap && nlists <= FM_LISTS) {
            const int64_t tiles = (N + 255) / 256, cols = (tiles + nsplit - 1) / nsplit * (256 / GEMM_COL_HALVES);
            const int64_t most = (int64_t)nlists * (cols < cap ? cols : cap);
            parts = (int)((most + FM_ENTRIES / 2 - 1) / (FM_ENTRIES / 2));
            const int room = sm_count() / nq;
            if (parts > room) parts = room;
            if (parts > FM_MAX_PARTS) parts = FM_MAX_PARTS;
            if (parts > nlists) parts = nlists;
            if (parts < 1) parts = 1;
        }
        e = launch_overlapped(flat_merge_kernel, dim3(nq * parts), dim3(FM_THREADS), 0, s, nlists, parts, k, cap, 1,
                              gemm_cand_sign(G.alpha, G.colterm), cand_cnt, cand, G.err + FM_TICKET_WORD, out_ids, out_scores);
        count_launch();
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    const cudaError_t ec = cudaMemsetAsync(workspace, 0, 256, s);
    if (ec != cudaSuccess) return ec;
    const int nchunks = (int)((N + FLAT_CHUNK - 1) / FLAT_CHUNK);
    uint8_t* w = static_cast<uint8_t*>(workspace) + 256;
    float* scores = reinterpret_cast<float*>(w);
    w += align_up((size_t)nq * FLAT_PANEL * 4, 256);
    int32_t* slot_cnt = reinterpret_cast<int32_t*>(w);
    w += align_up((size_t)nq * (nchunks ? nchunks : 1) * 4, 256);
    unsigned long long* slot_keys = reinterpret_cast<unsigned long long*>(w);
    for (int64_t r0 = 0; r0 < N; r0 += FLAT_PANEL) {
        const int nrows = (int)((N - r0) < FLAT_PANEL ? (N - r0) : FLAT_PANEL);
        dim3 g((nrows + FBN - 1) / FBN, (nq + FBM - 1) / FBM);
        flat_scores_kernel<<<g, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(queries),
                                             static_cast<const __nv_bfloat16*>(db), nq, r0, nrows, d, scores);
        dim3 gs((nrows + FLAT_CHUNK - 1) / FLAT_CHUNK, nq);
        flat_select_kernel<<<gs, FSEL_THREADS, 0, s>>>(scores, r0, nrows, k, (int)(r0 / FLAT_CHUNK), nchunks,
                                                       slot_cnt, slot_keys);
        count_launch(2);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    flat_merge_kernel<<<nq, FM_THREADS, 0, s>>>(nchunks, 1, k, k, 0, 0u, slot_cnt, slot_keys, nullptr, out_ids, out_scores);
    count_launch();
    return cudaGetLastError();
}

// The final selection alone, over the caller's raw lists (test hook).
cudaError_t launch_selftest_final_selection(int32_t* counts, unsigned long long* entries, int nlists, int stride, int nq, int k,
                                            int64_t* out_ids, float* out_scores, cudaStream_t s) {
    flat_merge_kernel<<<nq, FM_THREADS, 0, s>>>(nlists, 1, k, stride, 1, gemm_cand_sign(-1.f, nullptr), counts, entries, nullptr,
                                                out_ids, out_scores);
    count_launch();
    return cudaGetLastError();
}

}  // namespace rago
