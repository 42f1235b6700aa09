// Lookup-table construction + asymmetric-distance scan of the probed inverted lists.
//
// One persistent CTA per SM walks a contiguous share of the batch's code tiles (pairs (query, probed list) in probe
// order, each list cut into equal tiles of at most TV vectors); shares hold the same number of tiles, the start of a
// query counting as several (scan_query_lead).  A producer
// warp streams code tiles global -> shared with 1-D bulk copies (cp.async.bulk + mbarrier, a ring of
// S tiles in flight, where it pays the tiles two steps further down the list prefetched into L2); consumer warps
// build the lookup table of the current QUERY in shared memory (or, for small batches, fetch the
// image a kernel before the scan has built), then every lane owns one (virtual) code row of the tile
// and sums table entries.
//
// Score, smaller is better for both metrics:
//   inner product:  -<q, c_p>  +  sum_m -<q_m, cw_m>
//   squared L2:     ||q - c_p||^2  +  (||r||^2 + 2<c_p, r>)  +  sum_m -2<q_m, cw_m>      (r = decoded residual)
// i.e. bias(q, list) + term(vector) + sum of entries of a table that depends on the query only, so a
// table is rebuilt when the query changes, not at every probed list.  The expansion costs a few ulps
// of the largest term (see vector_terms_kernel); results agree with the direct form to ~1e-6 relative
// on data whose residuals are not tiny against the centroid distances.  The per-vector terms of a tile
// travel with it (a second bulk copy on the same barrier).
//
// Shared-memory access pattern.  A code row is read as 32-bit words; at step (blk, il, t) lane L
// reads word  blk*G + (il ^ a(L))  and uses byte  t ^ b(L)  of it, so that within any one
// instruction the 32 lanes touch 32 different banks both for the code words (rows are M bytes
// apart) and for the table (bank = table column mod 32).  Rows wider than 32*odd bytes are split
// into R "virtual rows" handled by adjacent lanes and summed with a shuffle; sub-space counts that
// are 16 mod 32 keep two table copies so lanes L and L^4 never collide.
//
// Table addressing.  Per code byte the inner loop spends one instruction on the address, one shared load and half an add.
// LUT_DOT (16, 48, 80, 96, 128 bytes): rows of 128 bytes; a byte dot product of the code word with 128 in the byte's place,
// plus the lane's address of the column in row 0, is the address.  It runs on the multiplier pipe, while byte permutations
// share theirs with everything else of the loop, the rows need no padding and the table may lie anywhere.  LUT_PERM (32 and 64 bytes): rows of 256 bytes from a multiple of 64 KB on, the address
// (place << 16) | (code << 8) | column*4  is one PRMT of the code word and a lane constant for every two bytes, half as many
// registers.  us per call, permutation / dot product: 96 bytes (400 queries, lists of 2 200) 710 / 667, 80 bytes 358 / 335, 16 bytes
// 569 / 548, 128 bytes 437 / 432; 64 bytes 483 / 494, 32 bytes 592 / 621, 48 bytes 499 / 512 (pairs 1 188 / 1 174).
//
// Fixed-point table.  Entries are stored as 32-bit integers scaled by a per-query power of two chosen
// so that a sum of M entries cannot overflow (|sum| < 2^30): the scan then adds two entries per
// instruction (a three-input integer add) and the sum is exact, so it does not depend on the order of
// the additions; it is converted back to fp32 once per vector.  The quantisation step is
// max|entry| * M / 2^30, i.e. an absolute error below max|entry| * M^2 / 2^31 per vector (2e-5 for
// M = 96 and entries of size 5), far inside the 1e-4 relative bar.
//
// Candidates better than the running threshold go to a shared buffer (topk.cuh).  The producer warp
// watches the buffer count and marks a tile "cut first" when the tiles in flight could overflow it; a
// cut is a CTA-wide bisection on the keys (ordered score bits, then position) that keeps the k best and a few
// more (one barrier per step), and the exact k best are sorted once, when the CTA leaves the query.  The
// threshold of a query is shared between CTAs through global memory, which only ever removes keys that
// cannot be among the k best, so the result does not depend on timing.
//
// Batches whose queries share long lists are scanned two queries at a time (SCAN_PAIRS; pair.cuh says how the answers stay the same
// bits): one look-up then serves both, and the kernel below is the same but for what happens to the sums.
//
// A warp works on RGW row groups of 32 (virtual) rows per tile, unrolled, so that several independent
// chains code word -> address -> table entry are in flight per warp; with R lanes per vector one
// epilogue (term, bias, key, push) serves R row groups.
#include <cstring>
#include <type_traits>

#include "topk.cuh"
#include "plan.cuh"
#include "pair.cuh"

namespace rago {

constexpr int MAX_STAGES = 4;
constexpr int SCAN_PF = 2;                  // tiles ahead of the one being copied that are prefetched into L2 (measured: 1-2 best)
// Prefetch of a contiguous global range into L2 (16-byte aligned start, size a multiple of 16 bytes).
__device__ __forceinline__ void l2_prefetch(const void* g, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(g), "r"(bytes) : "memory");
}
constexpr int SMEM_OPTIN = 227 * 1024;          // dynamic shared memory asked for (the sm_100 per-block limit)
constexpr uint32_t SMEM_BASE_EXPECTED = 1024;   // shared-window address of dynamic shared memory when the kernel has no static part
constexpr int CTRL_BYTES = 1024;

struct alignas(16) TileDesc {
    int32_t flags;       // bit 0: first tile of this pair inside this CTA; bit 1: cut the candidate buffer before this tile; bit 2: last tile of the CTA;
                         // two queries at a time: bit 3: cut the second query's buffer; bits 4, 5: the first, the second query probes this list
                         // from bit 8: vectors in this tile; negative: the CTA has no tile
    uint32_t pos0;       // storage position of the tile's first vector
    uint32_t tile_addr;  // shared address of the stage's code tile
    float term_b;        // two queries at a time: the second query's term
    uint32_t vt_addr;    // shared address of the first vector's term
    int32_t pair;        // index into probe_list (query * nprobe + rank)
    float term;          // the pair's (query, list) term of the score
    int32_t unused;
};

struct ScanArgs {
    const uint8_t* codes;
    const int64_t* list_offsets;
    const int32_t* probe_list;
    const float* probe_term;
    const float* queries;
    const float* cbT;
    const float* vterm;  // [N + 4] per-vector term (L2), null for inner product
    const int64_t* work_prefix;
    unsigned long long* qthresh;
    int32_t* slot_cnt;
    unsigned long long* slot_keys;
    uint32_t* err;
    const uint8_t* lut_img;  // [nq][LUT_BYTES] tables built ahead of the scan (small batches), or null
    const float* lut_inv;    // [nq] fp32 value of one integer unit of each such table
    int32_t npairs, nprobe, d, dsub, metric, k, stages;
    int32_t lead;            // work units in front of a query's first tile (scan_query_lead)
    int32_t stream_once;     // the batch is small: code tiles are fetched with an evict-first hint, so that the centroid
                             // table the next search's coarse step reads stays in L2
    int32_t prefetch;        // pull tiles into L2 ahead of their copies
    int32_t tile_vecs;       // vectors per tile of this launch (scan_tile_vecs)
    uint32_t dyn_bytes;
    PairView pv;             // batches in which queries are scanned two at a time (pair.cuh)
};

template <int WV, int G, int R, int NCW_, int RGW_, bool DUAL_>
struct Cfg {
    static constexpr bool DUAL = DUAL_;                 // two queries at a time
    static constexpr int NCW = NCW_;                    // consumer warps
    static constexpr int NCT = NCW * 32;                // consumer threads
    static constexpr int THREADS = NCT + 32;            // + one producer warp
    static constexpr int MV = WV * 4;                   // bytes per virtual row
    static constexpr int M = MV * R;                    // code bytes per vector
    static constexpr int NBLK = WV / G;                 // blocks of G words per virtual row
    static constexpr int KIND = G == 4 ? LUT_DOT2 : (M == 32 || M == 64 ? LUT_PERM : LUT_DOT);
    static constexpr int LUT_BYTES = lut_image_bytes(M, KIND);
    static constexpr int RGW = RGW_;                    // 32-row groups per warp per tile (unrolled: independent work in flight)
    // Row group g of warp w is g * NCW + w where a tile is longer than lists often are (48 bytes, 960 vectors), so that short lists occupy
    // all warps, and w * RGW + g elsewhere.  us per call side by side / dealt (with one row group per warp and a 128 KB table): 200 queries,
    // 512 of 1 024 lists of 390 vectors 827 / 731 (694), of 980 1 420 / 1 322 (1 413); 400 queries, lists of 2 200 404 / 407 (461).
    static constexpr bool DEALT = M == 48 && !DUAL;
    static constexpr int TILE_VROWS = NCW * 32 * RGW;
    static constexpr int TV = TILE_VROWS / R;           // vectors per tile
    static constexpr int TILE_BYTES = TILE_VROWS * MV;
    static constexpr bool CUT_SMALLER = !DUAL && TILE_BYTES > 40 * 1024 && TILE_BYTES <= 48 * 1024;  // scan_tile_vecs
    static constexpr int VT_BYTES = (TV + 4) * 4;       // staged per-vector terms (start rounded down to 16 bytes)
    // Keys of a candidate buffer (two queries at a time: two buffers): as many as fit beside two tiles.  Few keys mean a cut
    // before every tile: 96 bytes, 400 queries over lists of 2 200, k = 500, 2 048 / 4 096 keys 1 305 / 726 us, k = 1 024 1 590 / 800.
    static constexpr int KCAP = LUT_BYTES + 2 * (TILE_BYTES + VT_BYTES) + (DUAL ? 2 : 1) * 2 * TOPK_CAP * 8 + CTRL_BYTES <= SMEM_OPTIN ? 2 * TOPK_CAP : TOPK_CAP;
    // Tables of the kind LUT_PERM start at this absolute shared address (a multiple of 64 KB).  Two tiles of more than 48 KB do not
    // fit above a table at 64 KB, so configurations with such tiles keep their tiles below a table at 128 KB.
    static constexpr uint32_t LUT_WINDOW = TILE_BYTES > 48 * 1024 ? 0x20000u : 0x10000u;
    static_assert(WV % G == 0, "virtual rows are whole blocks");
    static_assert(TILE_VROWS % R == 0, "tile must hold whole vectors");
    static_assert(RGW % (R < RGW ? R : RGW) == 0, "row groups are taken min(R, RGW) at a time");
    static_assert(!DEALT || R == 1, "row groups taken together lie side by side");
    // The producer asks for a cut of the candidate buffer when the count it sees plus everything the tiles in
    // flight can still push would not fit.  It reads the count while a cut may be rewriting it, and may see less than the cut
    // keeps: the tiles in flight are then pushed behind that without another cut, so both must fit.  SMAX bounds the ring depth
    // accordingly, and so that half the buffer is left to work in.
    static constexpr int CUT_KEEPS = DUAL ? PAIR_MAX_K + TV : MAX_K + MAX_K / 4 + 8;  // of pairs at most KCAP - (S + 1) * TV
    static constexpr int SFIT = (KCAP - CUT_KEEPS) / TV, SHALF = KCAP / TV / 2;
    static constexpr int SMAX = SFIT < SHALF ? (SFIT < MAX_STAGES ? SFIT : MAX_STAGES) : (SHALF < MAX_STAGES ? SHALF : MAX_STAGES);
    static_assert(SMAX >= 2, "two tiles in flight must fit the candidate buffer twice over, and behind what a cut keeps");
    static_assert(VT_BYTES % 16 == 0 && TILE_BYTES % 16 == 0, "bulk-copy destinations are 16-byte granular");
    static_assert(KIND == LUT_DOT2 ? G == 4 && R == 1 : MV % 32 == 0, "a lane's columns of a block of words lie in one 32-column part of the table");
    static_assert(KIND != LUT_PERM || NBLK == 1, "one block of words to a (virtual) row");
};

// Absolute shared-memory addresses of everything the kernel keeps there.  The same function runs on
// the host (to choose the number of stages, with the expected window base) and in the kernel (with
// the real base); a plan that does not fit makes the kernel report an error and return.
struct SmemPlan {
    uint32_t lut, ctrl, keys, rT, vt[MAX_STAGES], tile[MAX_STAGES];
    int ok;
};

template <class C>
__host__ __device__ inline SmemPlan plan_smem(uint32_t base, uint32_t dyn_bytes, int d, int stages, bool need_vt) {
    SmemPlan p;
    p.ok = 1;
    const uint32_t end = base + dyn_bytes;
    uint32_t lo_cur = base, lo_end = base, hi_cur;
    if (C::KIND == LUT_PERM) {
        p.lut = lo_end = C::LUT_WINDOW;
        if (base > C::LUT_WINDOW) p.ok = 0;
    } else {
        p.lut = (base + 127u) & ~127u;  // rows of 128 bytes: bank = column
    }
    hi_cur = p.lut + C::LUT_BYTES;
    if (hi_cur > end) p.ok = 0;
    auto take = [&](uint32_t bytes, uint32_t align) -> uint32_t {  // below the table if it fits there, else above
        uint32_t a = (lo_cur + align - 1) & ~(align - 1);
        if (a + bytes <= lo_end) { lo_cur = a + bytes; return a; }
        a = (hi_cur + align - 1) & ~(align - 1);
        if (a + bytes <= end) { hi_cur = a + bytes; return a; }
        p.ok = 0;
        return base;
    };
    // largest pieces first
    for (int s = 0; s < MAX_STAGES; ++s) p.tile[s] = s < stages ? take(C::TILE_BYTES, 128) : base;
    p.keys = take(C::KCAP * (C::DUAL ? 16 : 8), 16);  // two queries at a time: two buffers
    for (int s = 0; s < MAX_STAGES; ++s) p.vt[s] = (s < stages && need_vt) ? take(C::VT_BYTES, 16) : base;
    // The scaled, transposed query is only alive while a table is built, when the candidate buffer is empty: it
    // shares the buffer's space when it fits there.
    p.rT = C::DUAL ? base : (uint32_t)d * 4 <= (uint32_t)C::KCAP * 8 ? p.keys : take((uint32_t)d * 4, 16);
    p.ctrl = take(CTRL_BYTES, 16);
    return p;
}

// Control block.
constexpr int WARP_CUT_MAX = 1024;  // buffer cuts of at most this many keys, for k of at most WARP_CUT_K, are made by one warp
constexpr int WARP_CUT_K = 32;      // (a larger k needs bisection rounds, which the whole CTA does faster)
struct Ctrl {
    unsigned long long full[MAX_STAGES];
    unsigned long long empty[MAX_STAGES];
    unsigned long long cbar;  // consumer barrier
    unsigned long long lutbar;  // a prebuilt table has landed
    uint32_t tile[MAX_STAGES], vt[MAX_STAGES];  // the stages' places (SmemPlan's, which would go to local memory to be indexed)
    TileDesc desc[MAX_STAGES];
    int cnt;
    int cnt_b;  // two queries at a time: keys in the second query's buffer
    uint32_t abort_flag;
    float red[32];  // per-warp maxima of the table build
    uint32_t redu[2][32];  // per-warp minima / maxima / counts of the buffer cut
};
static_assert(sizeof(Ctrl) <= CTRL_BYTES, "control block too large");

template <int IMM>
__device__ __forceinline__ float lds_f32_imm(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(addr), "n"(IMM));
    return v;
}
template <int IMM>
__device__ __forceinline__ uint32_t lds_u32_imm(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(IMM));
    return v;
}
__device__ __forceinline__ void sts_f32(uint32_t addr, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// Table construction by the consumer threads.  Entry e = j * M + m of the transposed codebook is
// DSUB contiguous floats; consecutive threads take consecutive entries (coalesced loads, and table
// stores that walk the banks).  UNR entries per thread are loaded before any is used so that enough
// requests are in flight to cover the L2 latency.
template <class C, int D4>
__device__ __forceinline__ float build_table(const float* __restrict__ cbT, const float* rT, uint32_t lut, int ctid) {
    float mx = 0.f;
    constexpr int UNR = D4 >= 3 ? 4 : 8;
    constexpr int TOTAL = KSUB * C::M;
    for (int e0 = ctid; e0 < TOTAL; e0 += C::NCT * UNR) {
        float4 cv[UNR][D4];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int e = e0 + u * C::NCT;
#pragma unroll
            for (int i = 0; i < D4; ++i)
                cv[u][i] = e < TOTAL ? __ldg(reinterpret_cast<const float4*>(cbT + (size_t)e * (D4 * 4)) + i)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int e = e0 + u * C::NCT;
            if (e >= TOTAL) break;
            const int j = e / C::M, m = e - j * C::M;
            float acc = 0.f;
#pragma unroll
            for (int i = 0; i < D4; ++i) {
                acc = fmaf(rT[(4 * i + 0) * C::M + m], cv[u][i].x, acc);
                acc = fmaf(rT[(4 * i + 1) * C::M + m], cv[u][i].y, acc);
                acc = fmaf(rT[(4 * i + 2) * C::M + m], cv[u][i].z, acc);
                acc = fmaf(rT[(4 * i + 3) * C::M + m], cv[u][i].w, acc);
            }
            sts_f32(lut + lut_offset(C::KIND, j, m), acc);
            mx = fmaxf(mx, fabsf(acc));
        }
    }
    return mx;
}
template <class C>
__device__ __forceinline__ float build_table_any(const float* __restrict__ cbT, const float* rT, uint32_t lut,
                                                int ctid, int dsub) {
    float mx = 0.f;
    for (int e = ctid; e < KSUB * C::M; e += C::NCT) {
        const int j = e / C::M, m = e - j * C::M;
        float acc = 0.f;
        for (int t = 0; t < dsub; ++t) acc = fmaf(rT[t * C::M + m], __ldg(cbT + (size_t)e * dsub + t), acc);
        sts_f32(lut + lut_offset(C::KIND, j, m), acc);
        mx = fmaxf(mx, fabsf(acc));
    }
    return mx;
}
// Second pass of the table build: every thread turns the fp32 entries it wrote itself into scaled
// integers (and fills the second copy where the layout keeps one).
template <class C>
__device__ __forceinline__ void quantise_table(uint32_t lut, int ctid, float scale) {
    for (int e = ctid; e < KSUB * C::M; e += C::NCT) {
        const int j = e / C::M, m = e - j * C::M;
        const uint32_t addr = lut + lut_offset(C::KIND, j, m);
        const int q = __float2int_rn(lds_f32(addr) * scale);
        sts_f32(addr, __int_as_float(q));
        if (C::KIND == LUT_DOT2) sts_f32(addr + LUT_COPY, __int_as_float(q));
    }
}

// Code words of one virtual row, all loaded before the first look-up (look-up addresses depend on them,
// so loading block by block would expose the shared-memory latency once per block).
// wa[il] is the lane's address of word (il ^ a(L)) of its row in the tile's first row group of this warp; OFF is
// the byte offset of the row group being read, a compile-time constant that ends up in the load's immediate.
template <class C, int G, int BLK, int OFF>
struct LoadWords {
    __device__ __forceinline__ static void run(const uint32_t (&wa)[G], uint32_t (&x)[C::NBLK][G]) {
#pragma unroll
        for (int il = 0; il < G; ++il) x[BLK][il] = lds_u32_imm<OFF + BLK * G * 4>(wa[il]);
        if constexpr (BLK + 1 < C::NBLK) LoadWords<C, G, BLK + 1, OFF>::run(wa, x);
    }
};

// One block (G code words = 4G sub-spaces) of one virtual row: 4G look-ups, written as three passes over
// half a block (all addresses, all loads, all adds).
template <class C, int G, int BLK>
__device__ __forceinline__ void scan_block(const uint32_t (&x)[G], const uint32_t (&at)[G][4], const uint32_t (&pick)[4], int (&acc)[4]) {
    constexpr int H = G / 2;
#pragma unroll
    for (int h0 = 0; h0 < G; h0 += H) {
        uint32_t ad[H][4];
        uint32_t vv[H][4];
#pragma unroll
        for (int i = 0; i < H; ++i)
#pragma unroll
            for (int t = 0; t < 4; ++t)
                ad[i][t] = C::KIND == LUT_PERM ? __byte_perm(x[h0 + i], at[h0 + i][t >> 1], pick[t]) : __dp4a(x[h0 + i], pick[t], at[h0 + i][t]);
#pragma unroll
        for (int i = 0; i < H; ++i)
#pragma unroll
            for (int t = 0; t < 4; ++t) vv[i][t] = lds_u32_imm<BLK * (int)LUT_PART>(ad[i][t]);
#pragma unroll
        for (int i = 0; i < H; i += 2)  // two entries per add
#pragma unroll
            for (int t = 0; t < 4; ++t) acc[t] = acc[t] + (int)vv[i][t] + (int)vv[i + 1][t];
    }
}
template <class C, int G, int BLK>
struct ScanBlocks {
    __device__ __forceinline__ static void run(const uint32_t (&x)[C::NBLK][G], const uint32_t (&at)[G][4], const uint32_t (&pick)[4],
                                               int (&acc)[4]) {
        scan_block<C, G, BLK>(x[BLK], at, pick, acc);
        if constexpr (BLK + 1 < C::NBLK) ScanBlocks<C, G, BLK + 1>::run(x, at, pick, acc);
    }
};

// ---- making a buffer of bounds exact (pairs of queries) ----
// Both steps are written for few registers: what they hold beside the tile loop's values goes to local memory, which, with
// nearly all of the SM's cache being shared memory, means trips to L2 (with 100 to 200 bytes of it the loop took twice as long).
// First step, a thread per key: the bound in the upper word of a key is replaced by the sum of the terms of its list (found among
// the unit's entries by the vector's position) and of the vector.
template <class C>
__device__ __forceinline__ void dual_terms(unsigned long long* kb, int kept, const float* terms, const uint2* ranges, int per_unit,
                                           const float* vterm, bool ip, int ctid) {
#pragma unroll 1
    for (int i = ctid; i < kept; i += C::NCT) {
        const uint32_t pos = (uint32_t)kb[i];
        int at = 0;
#pragma unroll 8
        for (int e = 0; e < per_unit; ++e) {
            const uint2 r = __ldg(ranges + e);
            if (pos >= r.x && pos < r.y) at = e;
        }
        const float t = __ldg(terms + at), vt = vterm != nullptr ? __ldg(vterm + pos) : 0.f;
        kb[i] = ((unsigned long long)__float_as_uint((ip ? -t : t) + vt) << 32) | pos;
    }
}
// Second step, a warp to a few keys, lanes over sub-spaces: the entries of the query's own 32-bit table at `lut`, summed and scored as
// the scan of one query does.
template <class C>
__device__ __forceinline__ void dual_exact(unsigned long long* kb, int kept, const uint8_t* codes, uint32_t lut, float inv, int ctid) {
    constexpr int MP = (C::M + 31) / 32, UN = C::THREADS > 512 ? 4 : 8;
    const int lane = ctid & 31;
#pragma unroll 1
    for (int i0 = ctid >> 5; i0 < kept; i0 += C::NCW * UN) {  // keys i0, i0 + NCW, ...
        uint32_t code[UN];  // a lane's codes, one byte each
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            const uint32_t pos = (uint32_t)kb[i0 + u * C::NCW < kept ? i0 + u * C::NCW : i0];
            code[u] = 0u;
#pragma unroll
            for (int j = 0; j < MP; ++j)
                if (lane + 32 * j < C::M) code[u] |= (uint32_t)__ldg(codes + (size_t)pos * C::M + lane + 32 * j) << (8 * j);
        }
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            int sum = 0;
#pragma unroll
            for (int j = 0; j < MP; ++j)  // bank = lane (of two copies the upper half of the lanes read the second)
                if (lane + 32 * j < C::M)
                    sum += (int)lds_u32(lut + lut_offset(C::KIND, (int)((code[u] >> (8 * j)) & 0xFFu), lane + 32 * j) + (C::KIND == LUT_DOT2 && lane >= 16 ? LUT_COPY : 0u));
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (lane == 0 && i0 + u * C::NCW < kept) {
                const unsigned long long key = kb[i0 + u * C::NCW];
                kb[i0 + u * C::NCW] = make_key(__uint_as_float((uint32_t)(key >> 32)) + (float)sum * inv, (uint32_t)key);
            }
        }
    }
}

// SCAN_PAIRS: every unit of work is a pair of queries (pair.cuh).  SCAN_BESIDE: the single queries of a batch with pairs.  SCAN_ALONE: every
// query of a batch without.  (One kernel for the latter two, which found the entries of its launch at run time, was 1 to 6% slower on
// batches without pairs: us per call, 200 queries, 512 of 1 024 lists of 980 vectors, 32 bytes 1 250 / 1 226, 128 bytes 3 240 / 3 047.)
enum ScanMode { SCAN_ALONE, SCAN_BESIDE, SCAN_PAIRS };
template <int WV, int G, int R, int NCW_, int RGW_, ScanMode MODE>
__global__ void __launch_bounds__(Cfg<WV, G, R, NCW_, RGW_, MODE == SCAN_PAIRS>::THREADS, 1) scan_kernel(const ScanArgs a) {
    constexpr bool DUAL = MODE == SCAN_PAIRS;
    using C = Cfg<WV, G, R, NCW_, RGW_, DUAL>;
    constexpr int NCW = C::NCW, NCT = C::NCT;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int S = a.stages;
    const uint32_t base = smem_u32(smem);
    const SmemPlan P = plan_smem<C>(base, a.dyn_bytes, a.d, S, a.vterm != nullptr);
    if (!P.ok) {  // uniform: every thread sees the same plan
        grid_dependency_wait();  // a CTA that exits lets the next kernel go on as one that has waited does
        if (tid == 0) atomicExch(a.err, (uint32_t)ERR_SMEM_LAYOUT);
        return;
    }
    Ctrl* ctrl = reinterpret_cast<Ctrl*>(smem + (P.ctrl - base));
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem + (P.keys - base));
    float* rT = reinterpret_cast<float*>(smem + (P.rT - base));
    volatile uint32_t* abort_flag = &ctrl->abort_flag;

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < MAX_STAGES; ++s) { ctrl->tile[s] = P.tile[s]; ctrl->vt[s] = P.vt[s]; }
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&ctrl->full[s]), 1);
            mbar_init(smem_u32(&ctrl->empty[s]), NCW);
        }
        mbar_init(smem_u32(&ctrl->cbar), NCW);
        mbar_init(smem_u32(&ctrl->lutbar), 1);
        ctrl->cnt = 0;
        ctrl->cnt_b = 0;
        ctrl->abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async();
    }
    __syncthreads();

    // Everything above touched shared memory and kernel arguments only; from here on the kernel reads what the
    // kernels before it wrote.  That holds for the launch for the single queries of a batch with pairs too, although it reads nothing
    // of the pairs' launch in front of it: that one's wait says nothing about what this one sees.
    grid_dependency_wait();
    grid_dependents_may_launch();
    // A batch of a few queries is latency-bound, and most of a CTA's start-up would be a chain of dependent reads
    // (total, binary search for the first pair, the pair's list, the list's offset) before its first tile can be
    // asked for.  With at most 32 pairs lane i of every warp reads pair i's first unit beside the total, so the
    // first pair follows from one vote; the producer warp reads the rest of every pair's description in the same
    // round trip (the offsets in a second one), and the consumers know their first query without the producer.
    // (Not where the entries of the batch are divided between pairs and single queries.)
    const bool few_pairs = MODE == SCAN_ALONE && a.npairs <= 32;
    // the entries this launch scans, and how many of them make a unit: a query, or a pair of queries
    const int npairs_q = MODE == SCAN_ALONE ? 0 : a.pv.head[0];
    const int per_unit = DUAL ? 2 * a.nprobe : a.nprobe;
    const int e_base = DUAL ? 0 : 2 * a.nprobe * npairs_q, e_end = DUAL ? 2 * a.nprobe * npairs_q : a.npairs;
    const long long pw = few_pairs ? a.work_prefix[lane < a.npairs ? lane : a.npairs] : 0;  // >= npairs: the total
    int c_list = 0; long long c_off = 0, c_len = 0, c_ws = 0, c_we = 0; float c_term = 0.f; int c_tv = C::CUT_SMALLER ? a.tile_vecs : C::TV;  // producer: lane i's cached pair
    if (few_pairs && warp == NCW && lane < a.npairs) {
        c_list = a.probe_list[lane];
        c_term = a.probe_term[lane];
        c_we = a.work_prefix[lane + 1];
        c_off = a.list_offsets[c_list];
        c_len = a.list_offsets[c_list + 1] - c_off;
    }
    // This CTA's share of the work units: the tiles whose place on the line of units lies in [u_begin, u_end).
    const long long W0 = e_base ? a.work_prefix[e_base] : 0, W = a.work_prefix[e_end];
    const long long u_begin = W0 + (long long)blockIdx.x * (W - W0) / gridDim.x;
    const long long u_end = W0 + (long long)(blockIdx.x + 1) * (W - W0) / gridDim.x;
    if (u_end <= u_begin) return;
    // few pairs: the pair whose range contains u_begin = the largest p with work_prefix[p] <= u_begin
    const int first_pair = few_pairs ? __popc(__ballot_sync(0xffffffffu, pw <= u_begin)) - 1 : -1;

    if (warp == NCW) {
        // ================= producer warp =================
        // first pair whose range contains u_begin: largest p with work_prefix[p] <= u_begin
        int lo = e_base, hi = e_end;  // invariant: work_prefix[lo] <= u_begin < work_prefix[hi]
        while (!few_pairs && hi - lo > 1) {  // 32 probes per step, evenly spaced: lane i looks at lo + (i + 1) * step
            const int step = (hi - lo + 31) / 32;
            const int pp = lo + (lane + 1) * step;
            const bool le = pp < hi && a.work_prefix[pp] <= u_begin;
            const int c = __popc(__ballot_sync(0xffffffffu, le));  // the prefix is monotone: the first c probes pass
            const int nhi = lo + (c + 1) * step;
            lo += c * step;
            hi = nhi < hi ? nhi : hi;
        }
        int cache_base = few_pairs ? 0 : lo;  // lane i caches pair cache_base + i
        if (few_pairs) {
            c_ws = pw + pair_lead(lane, a.nprobe, a.lead);
            if (lane >= a.npairs) { c_ws = c_we = W; }
        }
        // A list of several tiles is cut into tiles of one size (whole groups of 32 vectors) instead of full tiles and a
        // remainder: with two or three tiles in flight, a short tile leaves too little time for the copy behind it.
        // (Not for a few pairs, where a CTA has a tile or two and the division would stand before its first copy.)
        auto tile_size = [&]() {
            const uint32_t nt = (uint32_t)(c_we - c_ws), n = (uint32_t)c_len;  // positions are 32-bit
            c_tv = C::CUT_SMALLER ? a.tile_vecs : C::TV;
            if (nt > 1u) {
                const uint32_t share = n / nt;
                c_tv = (int)((share + (share * nt != n ? 32u : 31u)) & ~31u);
            }
        };
        static_assert(C::TV % 32 == 0, "a rounded-up tile must not exceed the tile it was cut from");
        float c_term_b = 0.f; int c_mask = 0;
        auto fill = [&]() {
            const int p = cache_base + lane;
            if (p < e_end) {
                c_list = a.probe_list[p];
                if (DUAL && c_list < 0) c_list = 0;  // an unused entry: no tiles
                c_off = a.list_offsets[c_list];
                c_len = a.list_offsets[c_list + 1] - c_off;
                c_ws = a.work_prefix[p] + pair_lead(p - e_base, per_unit, a.lead);  // place of its first tile
                c_we = a.work_prefix[p + 1];
                c_term = a.probe_term[p];
                if (DUAL) { c_term_b = a.pv.term_b[p]; c_mask = a.pv.mask[p]; }
            } else {
                c_list = 0; c_off = 0; c_len = 0; c_ws = c_we = W; c_term = 0.f;
            }
            tile_size();
        };
        if (!few_pairs) fill();
        int cur = few_pairs ? first_pair : 0;
        const uint64_t once_policy = l2_policy_evict_first();
        long long u = u_begin;
        bool dead = false;
        int issued = 0;
        int pst = 0;          // n % S, kept by counting (S is a run-time value: no division per tile)
        uint32_t pround = 0;  // n / S
        // Moves to the first tile at or after unit u (skips empty pairs and leads); false: there is none in the share.
        auto advance = [&]() -> bool {
            for (;;) {
                const long long first = __shfl_sync(0xffffffffu, c_ws, cur), we = __shfl_sync(0xffffffffu, c_we, cur);
                if (u < first) u = first;
                if (u >= u_end) return false;
                if (u < we) return true;
                if (++cur == 32) { cache_base += 32; fill(); cur = 0; }
            }
        };
        bool more = advance();
        if (!more && lane == 0) {  // a share without a tile: a descriptor with no copy says so
            ctrl->desc[0].flags = -1;
            mbar_arrive(smem_u32(&ctrl->full[0]));
        }
        for (int n = 0; more; ++n) {
            const int st = pst;
            const uint32_t round = pround;
            if (++pst == S) { pst = 0; ++pround; }
            const long long ws = __shfl_sync(0xffffffffu, c_ws, cur);
            const long long off = __shfl_sync(0xffffffffu, c_off, cur);
            const long long len = __shfl_sync(0xffffffffu, c_len, cur);
            const float term = __shfl_sync(0xffffffffu, c_term, cur);
            const float term_b = DUAL ? __shfl_sync(0xffffffffu, c_term_b, cur) : 0.f;
            const int mask = DUAL ? __shfl_sync(0xffffffffu, c_mask, cur) : 0;
            const int tv = __shfl_sync(0xffffffffu, c_tv, cur);
            const int pair = cache_base + cur;
            const long long t_in_pair = u - ws;
            const long long v0 = t_in_pair * tv;
            const int nvec = (int)(len - v0 < tv ? len - v0 : tv);
            const uint32_t pos0 = (uint32_t)(off + v0);
            const uint32_t bytes = (uint32_t)nvec * C::M;
            // per-vector terms: start rounded down to a 16-byte boundary, length rounded up
            const uint32_t vbytes = a.vterm ? (((pos0 & 3u) + (uint32_t)nvec) * 4u + 15u) & ~15u : 0u;
            const uint32_t bar = smem_u32(&ctrl->full[st]);
            const long long u_this = u++;
            more = advance();
            // All of the above stands before the wait for the stage, so that as little as possible lies between its coming
            // free and its refill (looking for the next tile after the wait: 48-byte codes, 300 queries 1 588 us, before it 1 500).
            const uint32_t tile_at = ctrl->tile[st], vt_at = ctrl->vt[st];
            const uint8_t* src = a.codes + (size_t)pos0 * C::M;
            if (round > 0) dead = !mbar_wait(smem_u32(&ctrl->empty[st]), (round - 1) & 1, abort_flag, a.err);
            if (dead) break;
            if (lane == 0) {
                // The copies first, then the descriptor, then the arrival: the barrier's count of bytes may run ahead of what it is
                // told to expect, and its phase cannot end without the arrival, which also makes the descriptor visible.
                if (a.stream_once) {  // small batch: the codes are read once and should leave L2 first
                    bulk_g2s_hint(tile_at, src, bytes, bar, once_policy);
                    if (vbytes) bulk_g2s_hint(vt_at, a.vterm + (pos0 & ~3u), vbytes, bar, once_policy);
                } else {
                    bulk_g2s(tile_at, src, bytes, bar);
                    if (vbytes) bulk_g2s(vt_at, a.vterm + (pos0 & ~3u), vbytes, bar);
                }
                TileDesc& D = ctrl->desc[st];
                // everything tiles n-S+1 .. n can still push must fit behind what is in the buffer now
                const int cnt_seen = *reinterpret_cast<volatile int*>(&ctrl->cnt);
                int flags = ((n == 0 || t_in_pair == 0) ? 1 : 0) | (cnt_seen + (S + 1) * C::TV > C::KCAP ? 2 : 0) | (more ? 0 : 4) | (nvec << 8);
                if (DUAL) {
                    const int seen_b = *reinterpret_cast<volatile int*>(&ctrl->cnt_b);
                    flags |= (seen_b + (S + 1) * C::TV > C::KCAP ? 8 : 0) | (mask << 4);
                    D.term_b = term_b;
                }
                D.flags = flags;
                D.pos0 = pos0;
                D.tile_addr = tile_at;
                D.vt_addr = vt_at + (pos0 & 3u) * 4u;
                D.pair = pair;
                D.term = term;
                mbar_arrive_expect_tx(bar, bytes + vbytes);
                // pull the tiles a few steps ahead in this list into L2, with their terms, so that their copies find them there
                if (a.prefetch) {
                    for (int ahead = (t_in_pair == 0 ? 1 : SCAN_PF); ahead <= SCAN_PF && u_this + ahead < u_end; ++ahead) {
                        const long long vp = v0 + (long long)ahead * tv;
                        if (vp >= len) break;
                        long long np = len - vp;
                        if (np > tv) np = tv;
                        const long long first = off + vp;
                        l2_prefetch(a.codes + (size_t)first * C::M, (uint32_t)np * C::M);
                        if (a.vterm) l2_prefetch(a.vterm + (first & ~3ll), (uint32_t)(((first & 3) + np) * 4 + 15) & ~15u);
                    }
                }
            }
            issued = n + 1;
        }
        if (dead && lane == 0) {
            // let copies already in flight land before the CTA's shared memory goes away
            for (int n = issued > S ? issued - S : 0; n < issued; ++n) {
                const uint32_t bar = smem_u32(&ctrl->full[n % S]);
                for (int it = 0; it < (1 << 16) && !mbar_try_wait(bar, (n / S) & 1); ++it) __nanosleep(64);
            }
        }
        return;
    }

    // ================= consumer warps =================
    const int ctid = tid;  // 0 .. NCT-1
    uint32_t cphase = 0, lphase = 0;
    bool dead = false;
    auto csync = [&]() {
        if (dead) return;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctrl->cbar));
        dead = !mbar_wait(smem_u32(&ctrl->cbar), cphase, abort_flag, a.err);
        cphase ^= 1;
    };

    // lane constants of the access pattern
    const int xa = G == 8 ? (lane >> 2) : (lane >> 3);  // word xor
    const int xb = lane & 3;                            // byte xor
    const int copy = G == 4 ? ((lane >> 2) & 1) : 0;
    const int sr = lane % R;                            // which slice of the vector this lane sums
    // xo: offset in a tile of the lane's word il of the warp's first row group.  An address of the table from a word's byte t:
    // LUT_DOT   at: the column in row 0 of the first part; pick: the rows' distance in the byte's place, so that the dot product of
    //           word and pick, plus at, is the address
    // LUT_PERM  at[0, 1]: bytes  column * 4 of t = 2h, of t = 2h + 1, the table's place / 64 KB; pick: selects the column's
    //           byte, the word's byte and the place into (place << 16) | (byte << 8) | column * 4
    uint32_t xo[G], at[G][4], pick[4];
#pragma unroll
    for (int il = 0; il < G; ++il) {
        xo[il] = (uint32_t)(warp * (C::DEALT ? 1 : C::RGW) * 32 + lane) * C::MV + 4u * (uint32_t)(il ^ xa);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t col = 16u * (uint32_t)(il ^ xa);
            if (C::KIND == LUT_PERM)
                at[il][t] = (uint32_t)sr * C::MV * 4u + col + 4u * (uint32_t)((2 * (t & 1)) ^ xb)
                          | ((uint32_t)sr * C::MV * 4u + col + 4u * (uint32_t)((2 * (t & 1) + 1) ^ xb)) << 8 | P.lut;
            else
                at[il][t] = P.lut + (uint32_t)(sr * (C::MV / 32)) * LUT_PART + (copy ? LUT_COPY : 0u) + col + 4u * (uint32_t)(t ^ xb);
        }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t)
        pick[t] = C::KIND == LUT_PERM ? (uint32_t)(4 + (t & 1)) | ((uint32_t)(t ^ xb) << 4) | 0x7600u : LUT_ROW << (8 * (t ^ xb));

    int cur_u = -1, cur_q = -1;  // the unit the CTA is working on, and its query
    unsigned long long tau = KEY_MAX;
    float bias = 0.f;
    const int k = a.k;
    const bool ip = a.metric == RAGO_IP;
    const float lut_scale = ip ? -1.f : -2.f;
    float inv_scale = 1.f;  // fp32 value of one unit of the current query's integer table

    // Cut the candidate buffer (more than k keys, count stable, called by all consumer threads after a csync and
    // followed by another before the buffer or its count is used again):
    // every thread takes its share of the keys into registers, the CTA bisects for a key with between k and
    // k + k/4 keys at or below it (one barrier per step instead of the ~66 of a full sort), and the keys up to
    // it are pushed back.  All keys of the k best are kept; that key bounds the k-th best.
    auto cut_buffer = [&]() {
        constexpr int KPT = (C::KCAP + NCT - 1) / NCT;
        const int n = ctrl->cnt < C::KCAP ? ctrl->cnt : C::KCAP;
        if (n <= WARP_CUT_MAX && k <= WARP_CUT_K) {  // uniform
            // A short buffer and a small k (small batches, mostly): warp 0 alone finds the cut and compacts the buffer in place,
            // with no barrier and no atomic on the way; the others wait once.  For k <= 32 the cut is the k-th
            // smallest of the 32 lanes' minima: at least k keys lie at or below it, about 1.5 k on keys in no
            // particular order.  Otherwise (or if ties leave too many) it is bisected, the score words re-read from
            // shared memory in every round.
            if (warp == 0) {
                const uint32_t* kw = reinterpret_cast<const uint32_t*>(keys);  // score word of key i: kw[2 i + 1]
                uint32_t lmn = 0xFFFFFFFFu, wmx = 0u;  // this lane's smallest score word, the largest of all
#pragma unroll 4
                for (int i = lane; i < n; i += 32) {
                    const uint32_t o = kw[2 * i + 1];
                    lmn = o < lmn ? o : lmn;
                    wmx = o > wmx ? o : wmx;
                }
                const uint32_t wmn = __reduce_min_sync(0xffffffffu, lmn);
                wmx = __reduce_max_sync(0xffffffffu, wmx);
                long long lo = (long long)wmn - 1, hi = wmx;  // #(score <= lo) < k <= #(score <= hi)
                uint32_t want_max = (uint32_t)(k + (k >> 2) + 8);
                if (want_max < (uint32_t)WARP_SORT_MAX) want_max = WARP_SORT_MAX;  // what one warp sorts afterwards
                const bool quick = k <= 32 && n >= 32;
                uint32_t c_hi = (uint32_t)n;
                if (quick) {  // the count at the quick cut comes out of the compaction
                    hi = __shfl_sync(0xffffffffu, warp_sort_u32(lmn, lane), k - 1);
                    c_hi = 0;
                }
                const uint32_t lt_mask = (1u << lane) - 1u;
                int nn = n;
                for (int attempt = 0; attempt < 2; ++attempt) {
                    while (hi - lo > 1 && c_hi > want_max) {
                        const uint32_t mid = (uint32_t)(lo + (hi - lo) / 2);
                        uint32_t c = 0;
#pragma unroll 4
                        for (int i = lane; i < nn; i += 32) c += kw[2 * i + 1] <= mid ? 1u : 0u;
                        c = __reduce_add_sync(0xffffffffu, c);
                        if (c < (uint32_t)k) lo = mid; else { hi = mid; c_hi = c; }
                    }
                    const uint32_t Tw = (uint32_t)hi;
                    int base = 0;
                    for (int i0 = 0; i0 < nn; i0 += 128) {  // four rows of 32 keys at a time: their loads overlap
                        unsigned long long key[4];
                        uint32_t m[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int i = i0 + 32 * u + lane;
                            key[u] = i < nn ? keys[i] : KEY_MAX;
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            m[u] = __ballot_sync(0xffffffffu, i0 + 32 * u + lane < nn && (uint32_t)(key[u] >> 32) <= Tw);
                        __syncwarp();  // a key moves to a position at or before its own, and these 128 have been read
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if ((m[u] >> lane) & 1u) keys[base + __popc(m[u] & lt_mask)] = key[u];
                            base += __popc(m[u]);
                        }
                    }
                    __syncwarp();
                    nn = base;
                    c_hi = (uint32_t)base;
                    if (!quick || attempt == 1 || c_hi <= want_max) break;
                }
                if (lane == 0) { ctrl->redu[0][1] = (uint32_t)nn; ctrl->redu[0][0] = (uint32_t)hi; }
            }
            csync();
            if (dead) return;
            // the count changes only now that every thread has taken this branch on the old one; nobody reads or
            // adds to it before the barrier the callers follow this call with
            if (ctid == 0) ctrl->cnt = (int)ctrl->redu[0][1];
            const unsigned long long bound = ((unsigned long long)ctrl->redu[0][0] << 32) | 0xFFFFFFFFull;  // >= the k-th best key
            if (bound < tau) tau = bound;
            if (ctid == 0) atomicMin(&a.qthresh[cur_q], bound);
            return;
        }
        unsigned long long mine[KPT];
        uint32_t mn = 0xFFFFFFFFu, mx = 0u;
#pragma unroll
        for (int j = 0; j < KPT; ++j) {
            const int i = ctid + j * NCT;
            mine[j] = i < n ? keys[i] : KEY_MAX;
            if (i < n) {
                const uint32_t o = (uint32_t)(mine[j] >> 32);
                mn = o < mn ? o : mn;
                mx = o > mx ? o : mx;
            }
        }
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) { ctrl->redu[0][warp] = mn; ctrl->redu[1][warp] = mx; }
        csync();
        if (dead) return;
        for (int w = 0; w < NCW; ++w) {
            mn = ctrl->redu[0][w] < mn ? ctrl->redu[0][w] : mn;
            mx = ctrl->redu[1][w] > mx ? ctrl->redu[1][w] : mx;
        }
        csync();  // the minima / maxima have been read; redu is free for the counts
        if (dead) return;
        // Whole keys are bisected, not scores: of a group of equal scores larger than the buffer (duplicates among the vectors) the
        // first by position are kept, and room remains for what is better than all of them.  #(key <= lo) < k <= #(key <= hi)
        unsigned long long lo = mn ? ((unsigned long long)mn << 32) - 1 : 0ull, hi = ((unsigned long long)mx << 32) | 0xFFFFFFFFull;
        uint32_t c_hi = (uint32_t)n;
        const uint32_t want_max = (uint32_t)(k + (k >> 2) + 8);
        int round = 0;
        while (hi - lo > 1 && c_hi > want_max) {  // uniform across the CTA
            const unsigned long long mid = lo + (hi - lo) / 2;
            uint32_t c = 0;
#pragma unroll
            for (int j = 0; j < KPT; ++j) c += mine[j] <= mid ? 1u : 0u;  // (mid < KEY_MAX, the value of a slot without a key)
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0) ctrl->redu[round & 1][warp] = c;
            csync();
            if (dead) return;
            c = 0;
            for (int w = 0; w < NCW; ++w) c += ctrl->redu[round & 1][w];
            if (c < (uint32_t)k) lo = mid; else { hi = mid; c_hi = c; }
            ++round;
        }
        if (ctid == 0) ctrl->cnt = 0;  // every thread holds its keys in registers since the first barrier above
        csync();
        if (dead) return;
#pragma unroll
        for (int j = 0; j < KPT; ++j)
            warp_push(keys, &ctrl->cnt, mine[j] != KEY_MAX && mine[j] <= hi, mine[j], C::KCAP);
        if (hi < tau) tau = hi;  // >= the k-th best key
        if (ctid == 0) atomicMin(&a.qthresh[cur_q], hi);
    };

    // Close the current query's candidate buffer: keep at most k keys and park them in this CTA's slot.
    auto finalize = [&]() {
        csync();
        if (dead) return;
        int kept = ctrl->cnt;
        // a long buffer: bisect down to about k keys first, then sort only those.  A cut pays when it makes the sort
        // smaller: for small k down to what one warp sorts, otherwise below the next power of two.
        if (k <= 32 ? kept > WARP_SORT_MAX : kept > 2 * k + 64) {
            cut_buffer();
            if (dead) return;
            csync();
            if (dead) return;
            kept = ctrl->cnt;
        }
        if (kept > 1) {  // the slot is left in ascending order, which the merge relies on
            kept = block_select_short(keys, &ctrl->cnt, k, ctid, NCT, csync, C::KCAP);  // few keys: one warp, one barrier
            if (dead) return;
        }
        if (kept == k && ctid == 0) atomicMin(&a.qthresh[cur_q], keys[k - 1]);
        const size_t slot = (MODE == SCAN_BESIDE ? 2 * ((size_t)npairs_q + gridDim.x) : 0) + cur_u + blockIdx.x;
        for (int i = ctid; i < kept; i += NCT) a.slot_keys[slot * k + i] = keys[i];
        if (ctid == 0) a.slot_cnt[slot] = kept;
        csync();
    };

    // Table of a query: entry (j, m) = lut_scale * <q_m, codeword j of sub-space m>.
    // Small k: once the first tiles of a query have put a hundred-odd keys into the buffer it is cut at once (cheap at
    // that length), so that the tiles that follow are pushed against a threshold instead of in full.
    bool early = false;
    auto begin_query = [&](int unit) {
        const int q = MODE == SCAN_BESIDE ? a.pv.order[2 * npairs_q + unit] : unit;
        cur_u = unit;
        cur_q = q;
        early = k <= 32;
        if (a.lut_img != nullptr) {  // the table was built ahead of the scan: fetch its shared-memory image
            // One thread asks the copy engine for the image (bulk copies, completion counted on a barrier): the 32
            // to 160 KB arrive at the rate of the L2 -> shared-memory path instead of a few 16-byte loads per thread
            // and round trip.  Every consumer is past its last look-up in the old table (the barrier that ended the
            // previous query); the fence orders those reads before the copies' writes.
            if (ctid == 0) {
                ctrl->cnt = 0;
                fence_proxy_async();
                const uint8_t* src = a.lut_img + (size_t)q * C::LUT_BYTES;
                const uint32_t bar = smem_u32(&ctrl->lutbar);
                mbar_arrive_expect_tx(bar, (uint32_t)C::LUT_BYTES);
                constexpr uint32_t PIECE = 32768;
                for (uint32_t o = 0; o < (uint32_t)C::LUT_BYTES; o += PIECE)
                    bulk_g2s(P.lut + o, src + o, (uint32_t)C::LUT_BYTES - o < PIECE ? (uint32_t)C::LUT_BYTES - o : PIECE, bar);
            }
            inv_scale = __ldg(a.lut_inv + q);
            tau = *reinterpret_cast<volatile unsigned long long*>(&a.qthresh[q]);
            dead = dead || !mbar_wait(smem_u32(&ctrl->lutbar), lphase, abort_flag, a.err);
            lphase ^= 1u;
            csync();
            return;
        }
        const float* qrow = a.queries + (size_t)q * a.d;
        for (int j = ctid; j < a.d; j += NCT) rT[(j % a.dsub) * C::M + j / a.dsub] = lut_scale * qrow[j];
        if (ctid == 0) ctrl->cnt = 0;
        csync();
        if (dead) return;
        float mx;
        switch (a.dsub) {
            case 4: mx = build_table<C, 1>(a.cbT, rT, P.lut, ctid); break;
            case 8: mx = build_table<C, 2>(a.cbT, rT, P.lut, ctid); break;
            case 12: mx = build_table<C, 3>(a.cbT, rT, P.lut, ctid); break;
            case 16: mx = build_table<C, 4>(a.cbT, rT, P.lut, ctid); break;
            default: mx = build_table_any<C>(a.cbT, rT, P.lut, ctid, a.dsub); break;
        }
        // per-query scale: the largest power of two that keeps a sum of M entries below 2^30
        mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));  // non-negative floats order like their bits
        if (lane == 0) ctrl->red[warp] = mx;
        csync();
        if (dead) return;
        for (int w = 0; w < NCW; ++w) mx = fmaxf(mx, ctrl->red[w]);
        int ex = 0;
        if (mx > 0.f && mx < 3.0e38f) frexpf(mx * (float)C::M, &ex);  // mx * M < 2^ex
        ex = ex < -90 ? -90 : (ex > 120 ? 120 : ex);
        quantise_table<C>(P.lut, ctid, ldexpf(1.f, 30 - ex));
        inv_scale = ldexpf(1.f, ex - 30);
        tau = *reinterpret_cast<volatile unsigned long long*>(&a.qthresh[q]);
        csync();
    };

    // ---- two queries at a time (pair.cuh): their buffers hold keys of lower bounds until a query is closed ----
    int dq[2] = {0, 0}, dbase[2] = {0, 0}, dshift[2] = {0, 0};
    float dinv[2] = {1.f, 1.f}, dunit[2] = {1.f, 1.f}, dbias[2] = {0.f, 0.f}, dlimit[2];
    unsigned long long dtau[2] = {KEY_MAX, KEY_MAX};
    bool duse[2] = {false, false};
    dlimit[0] = dlimit[1] = 0.f;
    auto dual_keys = [&](int side) { return keys + (side ? C::KCAP : 0); };
    // A table image takes the place of the one in use (every consumer is past its last look-up); ends with it there for this thread.
    auto fetch_table = [&](const uint8_t* src) {
        if (ctid == 0) {
            fence_proxy_async();
            const uint32_t bar = smem_u32(&ctrl->lutbar);
            mbar_arrive_expect_tx(bar, (uint32_t)C::LUT_BYTES);
            constexpr uint32_t PIECE = 32768;
            for (uint32_t o = 0; o < (uint32_t)C::LUT_BYTES; o += PIECE)
                bulk_g2s(P.lut + o, src + o, (uint32_t)C::LUT_BYTES - o < PIECE ? (uint32_t)C::LUT_BYTES - o : PIECE, bar);
        }
        dead = dead || !mbar_wait(smem_u32(&ctrl->lutbar), lphase, abort_flag, a.err);
        lphase ^= 1u;
    };
    // Limits of the scan's first test.  A bound is  bias + vt + (base + half * 2^s) * inv  up to its roundings, the test's left side
    // is  x = (2^23 + half) * unit + vt  with unit = 2^s * inv, so a bound at or below the threshold's score t has
    // x <= t - bias - base * inv + 2^23 * unit, up to roundings of both that lie below 2^-20 of the sum of all magnitudes (that
    // of vt is at most that of the others together where the two sides are close).  No threshold yet: t is NaN, and so is the
    // limit, which nothing is above.  A list that the query does not probe: nothing passes.
    auto dual_limits = [&]() {
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const double t = (double)orderable_f32((uint32_t)(dtau[side] >> 32)), b = (double)dbias[side];
            const double base = (double)dbase[side] * (double)dinv[side], top = 8388608.0 * (double)dunit[side];
            const double lim = t - b - base + top;
            dlimit[side] = duse[side] ? __double2float_ru(lim + (fabs(t) + fabs(b) + fabs(base) + 2.0 * top) * 0x1p-20) : -__int_as_float(0x7f800000);
        }
    };
    // Cuts the buffers of the sides in `sides` (bits), or closes both.  One body for both, called from one place: its size counts.
    //
    // A cut is that of cut_buffer on the bounds.  The k-th smallest bound T does not bound the k-th best score, but the score
    // of a vector whose bound is at most T is at most T + M (2^s - 1) units and the roundings of the three operations, all of
    // which lie below 2^-22 of the value and 128 units: everything up to that is kept, and it is the new threshold.  If
    // that is more than the buffer can hold beside the tiles in flight (coarse shifts, equal codes), or the query is closed,
    // the keys are replaced by those of the exact scores - entries of the query's own 32-bit table, which takes the place of
    // the pair's, summed and scored as the scan of one query does, a few keys to a warp at a time, lanes over sub-spaces - and
    // cut to k.  (Gathered from the table in global memory, which the codes have pushed out of L2 by then, the entries
    // of about 250 keys took 75 us a query.)
    auto dual_settle = [&](int sides, bool close) {
        constexpr int KPT = (C::KCAP + NCT - 1) / NCT;
        csync();
        if (dead) return;
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            if (!((sides >> side) & 1)) continue;
            unsigned long long* kb = dual_keys(side);
            int* cn = side ? &ctrl->cnt_b : &ctrl->cnt;
            const int q = side ? dq[1] : dq[0];
            const float inv = side ? dinv[1] : dinv[0];
            const int n = *cn < C::KCAP ? *cn : C::KCAP;
            // closing: cutting first costs less than the exact scores it saves
            const bool cut = n > (close ? k + (k >> 2) + WARP_SORT_MAX : k);
            unsigned long long bound = KEY_MAX;
            if (cut) {  // uniform
                unsigned long long mine[KPT];
                uint32_t mn = 0xFFFFFFFFu, mx = 0u;
#pragma unroll
                for (int j = 0; j < KPT; ++j) {
                    const int i = ctid + j * NCT;
                    mine[j] = i < n ? kb[i] : KEY_MAX;
                    if (i < n) {
                        const uint32_t o = (uint32_t)(mine[j] >> 32);
                        mn = o < mn ? o : mn;
                        mx = o > mx ? o : mx;
                    }
                }
                mn = __reduce_min_sync(0xffffffffu, mn);
                mx = __reduce_max_sync(0xffffffffu, mx);
                if (lane == 0) { ctrl->redu[0][warp] = mn; ctrl->redu[1][warp] = mx; }
                csync();
                if (dead) return;
                for (int w = 0; w < NCW; ++w) {
                    mn = ctrl->redu[0][w] < mn ? ctrl->redu[0][w] : mn;
                    mx = ctrl->redu[1][w] > mx ? ctrl->redu[1][w] : mx;
                }
                if (ctid == 0) *cn = 0;  // every thread holds its keys in registers
                csync();
                if (dead) return;
                long long lo = (long long)mn - 1, hi = mx;  // #(score <= lo) < k <= #(score <= hi)
                uint32_t c_hi = (uint32_t)n;
                const uint32_t want_max = (uint32_t)(k + (close ? k >> 3 : k >> 1) + 8);
                int round = 0;
                while (hi - lo > 1 && c_hi > want_max) {  // uniform across the CTA
                    const uint32_t mid = bisect_mid(lo, hi, round);
                    uint32_t c = 0;
#pragma unroll
                    for (int j = 0; j < KPT; ++j) c += (mine[j] != KEY_MAX && (uint32_t)(mine[j] >> 32) <= mid) ? 1u : 0u;
                    c = __reduce_add_sync(0xffffffffu, c);
                    if (lane == 0) ctrl->redu[round & 1][warp] = c;
                    csync();
                    if (dead) return;
                    c = 0;
                    for (int w = 0; w < NCW; ++w) c += ctrl->redu[round & 1][w];
                    if (c < (uint32_t)k) lo = mid; else { hi = mid; c_hi = c; }
                    ++round;
                }
                const double t = (double)orderable_f32((uint32_t)hi);
                const double slack = ((double)C::M * (double)((1u << (side ? dshift[1] : dshift[0])) - 1u) + 128.0) * (double)inv;
                const uint32_t T = f32_orderable(__double2float_ru(t + slack + (fabs(t) + slack) * 0x1p-22));
#pragma unroll
                for (int j = 0; j < KPT; ++j)
                    warp_push(kb, cn, mine[j] != KEY_MAX && (uint32_t)(mine[j] >> 32) <= T, mine[j], C::KCAP);
                bound = ((unsigned long long)T << 32) | 0xFFFFFFFFull;  // >= the k-th best key
                csync();
                if (dead) return;
            }
            int kept = *cn;
            if (close || kept > C::KCAP - (S + 1) * C::TV) {  // uniform
                const size_t eb = (size_t)e_base + (size_t)cur_u * per_unit;
                dual_terms<C>(kb, kept, (side ? a.pv.term_b : a.probe_term) + eb, a.pv.range + (side ? (size_t)a.npairs : 0) + eb, per_unit, a.vterm, ip, ctid);
                fetch_table(a.lut_img + (size_t)q * C::LUT_BYTES);  // in the place of the pair's
                csync();
                if (dead) return;
                dual_exact<C>(kb, kept, a.codes, P.lut, inv, ctid);
                csync();
                if (dead) return;
                if (kept > 1) {
                    kept = block_select_short<2 * RANK_MAX>(kb, cn, k, ctid, NCT, csync, C::KCAP);
                    if (dead) return;
                }
                if (kept == k) bound = kb[k - 1];
                if (!close) {
                    fetch_table(a.pv.img + (size_t)cur_u * C::LUT_BYTES);
                }
                if (close) {
                    const size_t slot = 2 * ((size_t)cur_u + blockIdx.x) + side;
                    for (int i = ctid; i < kept; i += NCT) a.slot_keys[slot * k + i] = kb[i];
                    if (ctid == 0) a.slot_cnt[slot] = kept;
                }
            }
            if (ctid == 0 && bound != KEY_MAX) atomicMin(&a.qthresh[q], bound);
            if (side) { if (bound < dtau[1]) dtau[1] = bound; } else { if (bound < dtau[0]) dtau[0] = bound; }
        }
        if (!close) {
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const unsigned long long g = *reinterpret_cast<volatile unsigned long long*>(&a.qthresh[dq[side]]);
                if (g < dtau[side]) dtau[side] = g;
            }
        }
        csync();
    };
    auto dual_begin = [&](int unit) {
        cur_u = unit;
        if (ctid == 0) { ctrl->cnt = 0; ctrl->cnt_b = 0; }
        const PairParams* pp = a.pv.params + unit;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            dq[side] = pp->q[side]; dbase[side] = pp->base[side]; dshift[side] = pp->shift[side]; dinv[side] = pp->inv[side];
            dunit[side] = dinv[side] * (float)(1u << dshift[side]);
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) dtau[side] = *reinterpret_cast<volatile unsigned long long*>(&a.qthresh[dq[side]]);
        fetch_table(a.pv.img + (size_t)unit * C::LUT_BYTES);
        csync();
    };

    // few pairs: the first query is known without the producer, so its table is fetched while the first tile is
    // still on its way (the tile loop finds cur_q set and goes straight to the scan)
    if (few_pairs) begin_query(first_pair / a.nprobe);
    int cst = 0;            // n % S and the parity of n / S, kept by counting
    uint32_t cparity = 0;
    for (bool last = false; (DUAL || !last) && !dead;) {
        const int st = cst;
        const bool end = DUAL && last;  // pairs: one more round closes the last one
        TileDesc D;
        if (!end) {
            const uint32_t parity = cparity;
            if (++cst == S) { cst = 0; cparity ^= 1u; }
            dead = dead || !mbar_wait(smem_u32(&ctrl->full[st]), parity, abort_flag, a.err);
            if (dead) break;
            D = ctrl->desc[st];
            if (D.flags < 0) break;
            last = (D.flags & 4) != 0;
        }
        if constexpr (DUAL) {
            int unit = cur_u;
            if (!end && (D.flags & 1)) {
                unit = (D.pair - e_base) / per_unit;
                dbias[0] = ip ? -D.term : D.term;
                dbias[1] = ip ? -D.term_b : D.term_b;
                duse[0] = (D.flags & 16) != 0;
                duse[1] = (D.flags & 32) != 0;
            }
            const bool close = cur_u >= 0 && (end || unit != cur_u);
            const int sides = close ? 3 : (end || unit != cur_u ? 0 : ((D.flags >> 1) & 1) | ((D.flags >> 2) & 2));
            if (sides) dual_settle(sides, close);
            if (dead || end) break;
            if (unit != cur_u) {
                dual_begin(unit);
                if (dead) break;
            }
            if (sides || (D.flags & 1)) dual_limits();
        } else if (D.flags & 1) {
            const int unit = (D.pair - e_base) / per_unit;
            if (unit != cur_u) {
                if (cur_u >= 0) finalize();
                if (dead) break;
                begin_query(unit);
                if (dead) break;
            }
            bias = ip ? -D.term : D.term;
        }
        // the producer saw the buffer filling up, or (small k) this is the query's second tile in this CTA: keep the
        // best k (or a few more), lower the threshold.  One site for both, so that the cut is in the loop once.
        const bool full_cut = (D.flags & 2) != 0;
        if (!DUAL && (full_cut || (early && !(D.flags & 1)))) {
            csync();
            if (dead) break;
            if (ctrl->cnt > (full_cut ? k : 2 * WARP_SORT_MAX)) {  // uniform: nothing is pushed between the two barriers
                cut_buffer();
                early = false;
            }
            if (dead) break;
            const unsigned long long g = *reinterpret_cast<volatile unsigned long long*>(&a.qthresh[cur_q]);
            if (g < tau) tau = g;
            csync();
            if (dead) break;
        }

        // ---- scan this tile: a warp owns RGW row groups (Cfg::DEALT says which) ----
        const int nvr = (D.flags >> 8) * R;
        const uint32_t tile_base = D.tile_addr;
        const uint32_t vt_base = D.vt_addr;
        // Row groups are taken MERGE at a time: with R lanes per vector every lane of an R-group ends up with
        // the vector's sum, so lane slice g finishes row group g and one epilogue serves MERGE row groups.
        constexpr int MERGE = R < C::RGW ? R : C::RGW;
        bool released = false;
        uint32_t wa[G];  // this lane's word addresses in the warp's first row group of the tile
#pragma unroll
        for (int il = 0; il < G; ++il) wa[il] = tile_base + xo[il];
        // One pass: MERGE row groups and their shared epilogue.  RG is a type carrying the first row group's index,
        // so that every shared-memory offset below is a compile-time constant.  Returns false when the tile ended.
        auto pass = [&](auto RG) -> bool {
            constexpr int rg = decltype(RG)::value;
            const int vr0 = C::DEALT ? (rg * NCW + warp) * 32 : (warp * C::RGW + rg) * 32;
            if (vr0 >= nvr) return false;
            int mine = 0;
            auto group = [&](auto GI) {
                constexpr int g = decltype(GI)::value;
                int acc[4] = {0, 0, 0, 0};
                uint32_t x[C::NBLK][G];
                LoadWords<C, G, 0, (rg + g) * (C::DEALT ? NCW : 1) * 32 * C::MV>::run(wa, x);
                ScanBlocks<C, G, 0>::run(x, at, pick, acc);
                int si = (acc[0] + acc[1]) + (acc[2] + acc[3]);
                if (R >= 2) si += __shfl_xor_sync(0xffffffffu, si, 1);
                if (R >= 4) si += __shfl_xor_sync(0xffffffffu, si, 2);
                if (MERGE == 1 || sr == g) mine = si;
            };
            group(std::integral_constant<int, 0>{});
            if constexpr (MERGE >= 2) group(std::integral_constant<int, 1>{});
            if constexpr (MERGE >= 3) group(std::integral_constant<int, 2>{});
            if constexpr (MERGE >= 4) group(std::integral_constant<int, 3>{});
            const int vr = vr0 + (MERGE == 1 ? 0 : sr * 32) + lane;  // the virtual row whose vector this lane finishes
            // per-vector term of the L2 expansion (0 for inner product); rows past the tile's end read
            // stale but in-bounds shared memory and are never pushed
            const float vt = a.vterm != nullptr ? lds_f32(vt_base + (uint32_t)(vr / R) * 4u) : 0.f;
            // In the last pass over the tile that was this warp's last read of the stage: hand the stage back
            // before the rest of the epilogue, so that the refill starts that much earlier (M = 96: -1%).
            if (rg + MERGE >= C::RGW || (C::DEALT && vr0 + NCW * 32 >= nvr)) {
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctrl->empty[st]));
                released = true;
            }
            const bool owner = MERGE == 1 ? sr == 0 : sr < MERGE;
            const uint32_t pos = D.pos0 + (uint32_t)(vr / R);
            if constexpr (DUAL) {
                // The two halves of the sum are lower bounds.  Most are above the threshold's score, which this shows in three
                // instructions a side: 2^23 + half as a float (its bits are 0x4B00 and the half), times the unit, plus the
                // vector's term, against the limit that dual_limits has made of all the rest.
                const float xa = fmaf(__uint_as_float(__byte_perm((uint32_t)mine, 0x4B00u, 0x5410u)), dunit[0], vt);
                const float xb = fmaf(__uint_as_float(__byte_perm((uint32_t)mine, 0x4B00u, 0x5432u)), dunit[1], vt);
                const bool live = vr < nvr && owner;
                const bool pa = live && !(xa > dlimit[0]), pb = live && !(xb > dlimit[1]);
                if (__any_sync(0xffffffffu, pa || pb)) {
                    const float sa = (float)(dbase[0] + (int)(((uint32_t)mine & 0xFFFFu) << dshift[0])) * dinv[0];
                    const float sb = (float)(dbase[1] + (int)(((uint32_t)mine >> 16) << dshift[1])) * dinv[1];
                    const unsigned long long key_a = make_key((dbias[0] + vt) + sa, pos), key_b = make_key((dbias[1] + vt) + sb, pos);
                    warp_push(dual_keys(0), &ctrl->cnt, pa && duse[0] && key_a < dtau[0], key_a, C::KCAP);
                    warp_push(dual_keys(1), &ctrl->cnt_b, pb && duse[1] && key_b < dtau[1], key_b, C::KCAP);
                }
            } else {
                const float s = (float)mine * inv_scale;
                const float score = (bias + vt) + s;  // smaller is better for both metrics
                const unsigned long long key = make_key(score, pos);
                warp_push(keys, &ctrl->cnt, vr < nvr && owner && key < tau, key, C::KCAP);
            }
            return true;
        };
        static_assert(C::RGW / MERGE <= 4, "passes are written out below");
        bool more = pass(std::integral_constant<int, 0>{});
        if constexpr (C::RGW > MERGE) more = more && pass(std::integral_constant<int, MERGE>{});
        if constexpr (C::RGW > 2 * MERGE) more = more && pass(std::integral_constant<int, 2 * MERGE>{});
        if constexpr (C::RGW > 3 * MERGE) more = more && pass(std::integral_constant<int, 3 * MERGE>{});
        if (!released) {  // a warp that left the loop early: no rows of this tile are its own
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctrl->empty[st]));
        }
    }
    if constexpr (!DUAL) { if (!dead && cur_u >= 0) finalize(); }
}

// ---- host side ----------------------------------------------------------------------------------
struct Variant {
    int M;
    void (*kernel)(const ScanArgs);
    void (*beside)(const ScanArgs);  // the same for the single queries of a batch with pairs, null where there are none
    int threads, tile_vecs;
    int (*stages_for)(int d, bool need_vt);
    int lut_bytes, lut_kind, buffer_keys;
};
template <class C>
static int stages_for(int d, bool need_vt) {
    for (int s = C::SMAX; s >= 2; --s)
        if (plan_smem<C>(SMEM_BASE_EXPECTED, SMEM_OPTIN, d, s, need_vt).ok) return s;
    return 0;
}
#define RAGO_VARIANT(WV, G, R, NCW, RGW, MODE, BESIDE) \
    { Cfg<WV, G, R, NCW, RGW, MODE == SCAN_PAIRS>::M, scan_kernel<WV, G, R, NCW, RGW, MODE>, BESIDE, \
      Cfg<WV, G, R, NCW, RGW, MODE == SCAN_PAIRS>::THREADS, Cfg<WV, G, R, NCW, RGW, MODE == SCAN_PAIRS>::TV, \
      stages_for<Cfg<WV, G, R, NCW, RGW, MODE == SCAN_PAIRS>>, Cfg<WV, G, R, NCW, RGW, MODE == SCAN_PAIRS>::LUT_BYTES, \
      Cfg<WV, G, R, NCW, RGW, MODE == SCAN_PAIRS>::KIND, Cfg<WV, G, R, NCW, RGW, MODE == SCAN_PAIRS>::KCAP }
#define RAGO_SINGLE(WV, G, R, NCW, RGW) RAGO_VARIANT(WV, G, R, NCW, RGW, SCAN_ALONE, (scan_kernel<WV, G, R, NCW, RGW, SCAN_BESIDE>))
#define RAGO_ALONE(WV, G, R, NCW, RGW) RAGO_VARIANT(WV, G, R, NCW, RGW, SCAN_ALONE, nullptr)
#define RAGO_PAIR(WV, G, R, NCW, RGW) RAGO_VARIANT(WV, G, R, NCW, RGW, SCAN_PAIRS, nullptr)
// Warps x unrolled row groups per warp were chosen by measurement: independent row groups in flight inside a warp
// hide the look-up latency better than more warps do (M = 64: 16 x 2 -> 12 x 4 gave +30%; M = 48: 15 x 1 -> 15 x 2 +13 to 17%, for
// pairs 15 x 1 -> 10 x 2 +6%, 8 x 2 -6%; M = 96: 15 x 1 -> 8 x 2 -4%, for pairs 15 x 1 -> 7 x 2 -11%), and 15 consumer warps
// (four warps on every scheduler, the producer included) beat 12, 14 and 16 wherever their tiles fit (M = 32: +3%,
// M = 64: +4.5%).  Where a code size has two entries the first one whose shared-memory plan fits the
// index (dimension, metric) is taken (of the pairs': find_pair_variant).
static const Variant kVariants[] = {
    RAGO_SINGLE(4, 4, 1, 16, 2),   // M = 16
    RAGO_SINGLE(8, 8, 1, 15, 2),   // M = 32
    RAGO_SINGLE(12, 4, 1, 15, 2),  // M = 48: two 46 KB tiles beside the 96 KB table
    RAGO_SINGLE(8, 8, 2, 15, 4),   // M = 64: two 60 KB tiles below the table
    RAGO_SINGLE(8, 8, 2, 12, 4),   // M = 64 where those do not fit
    RAGO_ALONE(20, 4, 1, 8, 1),   // M = 80
    RAGO_SINGLE(24, 8, 1, 15, 1),  // M = 96
    RAGO_ALONE(8, 8, 4, 12, 3),   // M = 128
};
// The same table layouts for pairs of queries (the tables of 80 and 128 bytes leave no room for two buffers).
static const Variant kPairVariants[] = {
    RAGO_PAIR(4, 4, 1, 15, 2),    // M = 16: 16 warps and the producer would leave 96 registers a thread, too few
    RAGO_PAIR(8, 8, 1, 15, 2),
    RAGO_PAIR(12, 4, 1, 10, 2),   // M = 48: two row groups for as many warps as the two buffers leave room for
    RAGO_PAIR(8, 8, 2, 15, 2),    // M = 64: the tiles in flight have to fit each buffer twice over
    RAGO_PAIR(24, 8, 1, 15, 1),
    RAGO_PAIR(24, 8, 1, 12, 1),    // M = 96 for larger k (find_pair_variant)
};

static const Variant* find_variant(int M, int d, bool need_vt) {
    for (const Variant& v : kVariants)
        if (v.M == M && v.stages_for(d, need_vt) >= 2) return &v;
    return nullptr;
}
// A cut of a buffer of bounds keeps up to k * 3 / 2 keys and a few; beyond what the tiles in flight leave room for, the next cut follows at
// once.  Of two entries the first is taken whose buffer leaves that room and a quarter more.  96 bytes, 15 / 12 warps (without
// pairs), us per call, 200 queries over 32 of 300 lists of 30 000: k = 100 3 142 / 3 193 (3 704), 300 3 475 / 3 401, 350 3 606 / 3 486, 400
// 3 834 / 3 610 (3 832), 512 4 592 / 3 867 (3 877); 1 000 queries: 200 13 650 / 13 960, 300 14 170 / 14 290, 350 14 570 / 14 460.
static const Variant* find_pair_variant(int M, int d, bool need_vt, int k) {
    const Variant* found = nullptr;
    for (const Variant& v : kPairVariants) {
        if (v.M != M) continue;
        const int stages = v.stages_for(d, need_vt);
        if (stages < 2) continue;
        found = &v;
        if (v.buffer_keys - (stages + 1) * v.tile_vecs >= 2 * k) break;
    }
    return found;
}

bool scan_supported(int M) {
    for (const Variant& v : kVariants)
        if (v.M == M) return true;
    return false;
}

cudaError_t scan_plan(const IndexImpl* ix, ScanPlan* plan) {
    const Variant* v = find_variant(ix->M, ix->d, ix->metric != RAGO_IP);
    if (!v) return cudaErrorInvalidValue;
    const int stages = v->stages_for(ix->d, ix->metric != RAGO_IP);
    plan->tile_vecs = v->tile_vecs;
    plan->stages = stages;
    plan->buffer_keys = v->buffer_keys;
    plan->ctas = ix->num_sms;
    plan->smem_bytes = SMEM_OPTIN;
    plan->lut_bytes = v->lut_bytes; plan->lut_kind = v->lut_kind;
    plan->pairs = 0;
    for (const Variant& pv : kPairVariants) {
        if (pv.M != ix->M || pv.stages_for(ix->d, ix->metric != RAGO_IP) < 2) continue;
        plan->pairs = 1;
        for (auto kernel : {pv.kernel, v->beside}) {
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_OPTIN);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaFuncSetAttribute(v->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_OPTIN);
}

// Vectors per tile of a batch's scan.  Tiles of 46 KB (48 and 96 bytes) are smaller where whole ones would leave half of the CTAs without one: the
// lists are then spread over more CTAs, each of which waits for less.  Lists of 1 216 vectors, us per call with 480 / 256 vectors (384 before the
// tiles grew), 96 bytes: one query, 16 probes 43.0 / 36.3 (38.4), 4 probes 40.0 / 36.6 (38.6); 48 bytes with 960 / 256: 39.6 / 35.1, 36.8 /
// 34.2; but 8 queries, 8 probes (192 tiles) 43.3 / 48.0, 16 queries, 32 probes 67.3 / 69.6.
int scan_tile_vecs(const IndexImpl* ix, int nq, int nprobe) {
    const int whole = ix->plan.tile_vecs, tile_bytes = whole * ix->M;  // bounds: Cfg::CUT_SMALLER, a constant of the kernels (32 bytes 1% slower with a run-time size)
    const int64_t tiles = (int64_t)nq * nprobe * ((ix->N / ix->nlist + whole) / whole);
    return tile_bytes > 40 * 1024 && tile_bytes <= 48 * 1024 && 2 * tiles <= ix->plan.ctas ? 256 : whole;
}

// Work units (tiles) that stand for the start of a query on the line that is cut into one share per CTA.  Every CTA opens
// the query its share begins with; one that meets the start of another query closes the first (cut, rank), fetches
// the second's table and fills its candidate buffer without a threshold, which takes as long as scanning several tiles: in
// shares of equal tile counts the CTAs with the most query starts finished last (48-byte codes, 300 queries: 17 us per
// start, last CTA at 1 595 us against a mean of 1 457; 32 bytes, 16 queries: 5.5 us, 36 against 26).  Per start: k <= 32
// about 5.5 us; more with a 4 096-key buffer 7 us, with a 2 048-key buffer (more cuts) 17; per tile 1 us for 36 KB, no
// less than 0.8 us.  Where a share is shorter than the start of a query the tiles are short or few, no CTA waits long
// for another, and leads only leave CTAs without work (64 queries over 100 000 vectors 64.8 -> 67.1 us per call): none.
// 7 and 17 were measured with 64 bytes and with 48 in their former buffer of 2 048 keys; the other sizes take them by their
// buffer, and the tile count is that of average lists.  With 7 / 17 for the buffers of 4 096 keys beside 96 KB tables, us per call: 48 bytes,
// lists of 2 200, 40 queries 95.0 / 98.8, 100 queries 170.2 / 169.1, 200 over lists of 10 000 686 / 682; 96 bytes the same 126.6 / 127.8,
// 230.4 / 234.2, 1 158 / 1 156.  All of them only move work between CTAs: no result depends on them.
int scan_query_lead(const IndexImpl* ix, int nq, int nprobe, int k) {
    if (nq < 2 || ix->nlist < 1) return 0;
    const float start_us = k <= 32 ? 5.5f : (ix->plan.buffer_keys > TOPK_CAP ? 7.f : 17.f);
    const int tile_vecs = scan_tile_vecs(ix, nq, nprobe);
    const float tile_us = (float)(tile_vecs * ix->M) / 36000.f;
    const int lead = (int)(start_us / (tile_us > 0.8f ? tile_us : 0.8f) + 0.5f);
    const int64_t tiles_per_list = (ix->N / ix->nlist + tile_vecs) / tile_vecs;  // of a list of average length
    return (int64_t)nq * nprobe * tiles_per_list >= (int64_t)lead * ix->plan.ctas ? lead : 0;
}

// The start of a pair of queries: two buffers are closed (cut, made exact, ranked: about 90 000 cycles in all) and filled again.
// (1 024 queries, 96 bytes: with 30 us the CTAs of the short lists, 18 closes each, ended 12% after the others.)
int scan_pair_lead(const IndexImpl* ix, int pair_tile_vecs) {
    const float tile_us = (float)(pair_tile_vecs * ix->M) / 36000.f;
    return (int)(60.f / tile_us + 0.5f);
}

int scan_pair_tile_vecs(const IndexImpl* ix, int k) { return find_pair_variant(ix->M, ix->d, ix->metric != RAGO_IP, k)->tile_vecs; }

// Prefetching into L2 pays where the tiles in flight are small (a copy from DRAM takes longer than the tile in front
// of it is scanned) and the batch does not meet each list several times, which brings most tiles from L2 anyway and
// makes the prefetches only extra traffic.  Without / with, us per call: 64 bytes (60 KB tiles), 4 096 queries 14 560 / 14 730, 33
// queries 226.9 / 233.8.  Tiles of 46 KB (48 and 96 bytes) lose by it where a batch meets few of the lists: lists of 2 200, 0.47 probes per
// list 96 bytes 157.5 / 162.8 (inner product 154.7 / 164.4), 48 bytes 114.5 / 115.7, 0.23 probes 106.1 / 110.3; lists of 15 000, 0.53 probes
// 143.0 / 155.2, 0.96 220.9 / 230.4; from one probe on they gain a little: 2.1 412.5 / 411.7, 1.0 272.6 / 271.6, 1.6 374.8 / 372.6, 2.3
// 516 / 513 (inner product 530 / 518).
// Long lists of a database beyond L2 come from DRAM however often they are met, which shows where a tile is scanned in a
// short time: 80 bytes (20 KB tiles), 64 lists of 47 000 vectors, 600 queries with 32 probes, without / with 19 490 / 18 950, and 48 bytes,
// whose tiles took as long while they were as small (9 520 / 8 940) and gain less now: lists of 30 000 1 794 / 1 767, 20 000 1 246 /
// 1 239, 9 000 638 / 633, 47 000 1 274 / 1 267.  Lists below 640 KB, inside L2, and the other sizes (16 bytes 3%, 64 bytes 3%
// more): the other way round or equal.
bool scan_prefetches(const IndexImpl* ix, int64_t npairs) {
    const int tile_bytes = ix->plan.tile_vecs * ix->M;
    const bool few = npairs <= 4ll * ix->nlist && (tile_bytes <= 40 * 1024 || (tile_bytes <= 48 * 1024 && npairs >= ix->nlist));
    const bool long_lists = ix->N / ix->nlist * ix->M >= 640 * 1024 && ix->N * ix->M > (128ll << 20);
    return few || (ix->M >= 48 && ix->plan.lut_kind == LUT_DOT2 && long_lists);
}

// view (may be null): the batch's pairs of queries, scanned by a launch of their own in front of that of the single ones.
cudaError_t launch_scan(const IndexImpl* ix, const ScanPlan& plan, const float* queries, const int32_t* probe_list,
                        const float* probe_term, const int64_t* work_prefix, int nq, int nprobe, int k,
                        unsigned long long* qthresh, int32_t* slot_cnt, unsigned long long* slot_keys,
                        uint32_t* err_word, const uint8_t* lut_img, const float* lut_inv, const PairView* view, cudaStream_t s) {
    const bool need_vt = ix->metric != RAGO_IP;
    const Variant* v = find_variant(ix->M, ix->d, need_vt);
    if (!v) return cudaErrorInvalidValue;
    ScanArgs a;
    a.codes = ix->codes; a.list_offsets = ix->list_offsets; a.probe_list = probe_list; a.probe_term = probe_term;
    a.queries = queries; a.cbT = ix->cbT; a.work_prefix = work_prefix;
    a.vterm = ix->vterm;
    a.qthresh = qthresh; a.slot_cnt = slot_cnt; a.slot_keys = slot_keys; a.err = err_word;
    a.lut_img = lut_img; a.lut_inv = lut_inv;
    a.npairs = nq * nprobe; a.nprobe = nprobe; a.d = ix->d; a.dsub = ix->dsub;
    a.lead = scan_query_lead(ix, nq, nprobe, k);
    a.metric = ix->metric; a.k = k; a.stages = plan.stages; a.dyn_bytes = (uint32_t)plan.smem_bytes;
    a.stream_once = nq <= 64 ? 1 : 0;
    a.prefetch = scan_prefetches(ix, a.npairs) ? 1 : 0;
    a.tile_vecs = scan_tile_vecs(ix, nq, nprobe);
    std::memset(&a.pv, 0, sizeof(a.pv));
    if (view) {
        const Variant* p = find_pair_variant(ix->M, ix->d, need_vt, k);
        if (!p) return cudaErrorInvalidValue;
        ScanArgs b = a;
        b.pv = a.pv = *view;
        b.lead = a.lead ? scan_pair_lead(ix, p->tile_vecs) : 0;
        b.stages = p->stages_for(ix->d, need_vt);
        const cudaError_t e = launch_overlapped(p->kernel, dim3(plan.ctas), dim3(p->threads), plan.smem_bytes, s, b);
        if (e != cudaSuccess) return e;
        count_launch();
    }
    const cudaError_t e = launch_overlapped(view ? v->beside : v->kernel, dim3(plan.ctas), dim3(v->threads), plan.smem_bytes, s, a);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// ---- lookup tables of a small batch, built ahead of the scan ---------------------------------------
// With few queries every scan CTA would build the same handful of tables, each reading the whole codebook; here
// the tables are built once, by many CTAs per query, and stored as the exact shared-memory image the scan variant
// uses (padding included), so a scan CTA fetches a table with one linear copy.
//
// The fixed-point scale cannot wait for the largest entry (the CTAs of a query do not meet), so it comes from a
// bound: |entry(j, m)| = |s <q_m, cw_mj>| <= |s| ||q_m|| max_j ||cw_mj||.  The bound costs a bit or two of the 30
// the sum may use, which leaves the quantisation error far below the tolerance.
__global__ void codeword_norms_kernel(const float* __restrict__ cb, int dsub, float* __restrict__ cwmax) {
    __shared__ float red[KSUB / 32];
    const int m = blockIdx.x, j = threadIdx.x;  // KSUB threads: one codeword each
    float n2 = 0.f;
    for (int t = 0; t < dsub; ++t) { const float v = cb[((size_t)m * KSUB + j) * dsub + t]; n2 = fmaf(v, v, n2); }
    float n = sqrtf(n2);
    for (int o = 16; o; o >>= 1) n = fmaxf(n, __shfl_xor_sync(0xffffffffu, n, o));
    if ((j & 31) == 0) red[j >> 5] = n;
    __syncthreads();
    if (j == 0) {
        for (int w = 1; w < KSUB / 32; ++w) n = fmaxf(n, red[w]);
        cwmax[m] = n;
    }
}
cudaError_t launch_codeword_norms(const float* codebooks, int M, int dsub, float* cwmax, cudaStream_t s) {
    codeword_norms_kernel<<<M, KSUB, 0, s>>>(codebooks, dsub, cwmax);
    count_launch();
    return cudaGetLastError();
}

constexpr int BT_THREADS = 256;
__global__ void __launch_bounds__(BT_THREADS) build_tables_kernel(const TableArgs t) {
    extern __shared__ float bt_smem[];
    grid_dependency_wait();
    grid_dependents_may_launch();
    build_table_part(t, blockIdx.y, blockIdx.x, gridDim.x, bt_smem);
}
static TableArgs table_args(const IndexImpl* ix, const float* queries, uint8_t* lut_img, float* lut_inv) {
    const ScanPlan& pl = ix->plan;
    TableArgs t;
    t.queries = queries; t.cbT = ix->cbT; t.cwmax = ix->cwmax;
    t.d = ix->d; t.dsub = ix->dsub; t.M = ix->M; t.metric = ix->metric;
    t.lut_bytes = pl.lut_bytes; t.kind = pl.lut_kind;
    t.lut_img = lut_img; t.lut_inv = lut_inv;
    return t;
}
static int table_parts(const IndexImpl* ix, int nq) {
    const int parts = 2 * ix->num_sms / nq;
    return parts < 1 ? 1 : (parts > 64 ? 64 : parts);
}
// Large batches.  One CTA per (range of code values, chunk of queries): every thread keeps the codewords of its EPT
// entries in registers and walks the chunk's queries, so the codebook crosses L2 once per chunk of queries
// instead of once per query.  The scale of each query (same bound as above) comes from a kernel of
// its own, because a CTA sees only a slice of the sub-spaces.
__global__ void __launch_bounds__(128) table_scales_kernel(const float* __restrict__ queries,
                                                            const float* __restrict__ cwmax, int d, int dsub, int M,
                                                            float* __restrict__ lut_scale, float* __restrict__ lut_inv,
                                                            int32_t* __restrict__ ok) {
    __shared__ float red[4];
    grid_dependency_wait();
    grid_dependents_may_launch();
    const int q = blockIdx.x, tid = threadIdx.x;
    const float* qrow = queries + (size_t)q * d;
    float mx = 0.f;
    bool finite = true;
    for (int m = tid; m < M; m += 128) {
        float n2 = 0.f;
        for (int u = 0; u < dsub; ++u) { const float v = qrow[m * dsub + u]; n2 = fmaf(v, v, n2); }
        finite = finite && n2 < 3.0e38f;  // not so for NaN
        mx = fmaxf(mx, 2.0002f * sqrtf(n2) * cwmax[m]);
    }
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) == 0) red[tid >> 5] = mx;
    finite = __syncthreads_and(finite);
    if (tid == 0) {
        mx = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
        int ex = 0;
        if (mx > 0.f && mx < 3.0e38f) frexpf(mx * (float)M, &ex);
        if (ok != nullptr) ok[q] = finite && mx * (float)M < 1e36f ? 1 : 0;  // no sum of M entries reaches 2^30 + M / 2 (1e36 < 2^120)
        ex = ex < -90 ? -90 : (ex > 120 ? 120 : ex);
        lut_scale[q] = ldexpf(1.f, 30 - ex);
        lut_inv[q] = ldexpf(1.f, ex - 30);
    }
}

constexpr int BTB_CW_FLOATS = 96;  // codeword floats a thread keeps in registers
// blockDim.x = M * G: thread (m, g) owns sub-space m of the code values j = j0 + g + G i, i < EPT, so everything it
// needs of a query is the DSUB values of one sub-space, fetched straight into registers (the next query's while the
// current one is multiplied): no shared memory and no barrier.  Threads with consecutive m read consecutive
// codewords and write consecutive table columns.
template <int DSUB>
__global__ void __launch_bounds__(256) build_tables_batch_kernel(const TableArgs t, const float* __restrict__ lut_scale,
                                                                  int nq, int qchunk) {
    constexpr int EPT = BTB_CW_FLOATS / DSUB;  // entries per thread
    grid_dependency_wait();
    grid_dependents_may_launch();
    const int d = t.d, M = t.M, tid = threadIdx.x;
    const int G = blockDim.x / M;
    const int m = tid % M, g = tid / M;
    const int j0 = blockIdx.x * (G * EPT);
    float cw[EPT][DSUB];
    uint32_t off[EPT];  // byte offset of the entry in a table image, 0xFFFFFFFF for an unused slot
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
        const int j = j0 + g + G * i;
        off[i] = 0xFFFFFFFFu;
#pragma unroll
        for (int u = 0; u < DSUB; ++u) cw[i][u] = 0.f;
        if (j < KSUB) {
            off[i] = lut_offset(t.kind, j, m);
            const float* src = t.cbT + ((size_t)j * M + m) * DSUB;
#pragma unroll
            for (int u = 0; u < DSUB; u += 4) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(src + u));
                cw[i][u] = v.x; cw[i][u + 1] = v.y; cw[i][u + 2] = v.z; cw[i][u + 3] = v.w;
            }
        }
    }
    // second copy of a column (layouts that keep one), as a byte distance inside the image
    const uint32_t copy_delta = t.kind == LUT_DOT2 ? LUT_COPY : 0u;
    const float lut_s = t.metric == RAGO_IP ? -1.f : -2.f;
    const int q0 = blockIdx.y * qchunk;
    const int q1 = q0 + qchunk < nq ? q0 + qchunk : nq;
    // the next query's values and scale, fetched while the current one is multiplied (a scale fetched in the step that
    // uses it put a memory round trip into every step: 4 096 queries, 64 sub-spaces 239 us)
    float qn[DSUB], scale_n = 0.f;
    auto fetch = [&](int q) {
        scale_n = __ldg(lut_scale + q);
        const float* src = t.queries + (size_t)q * d + m * DSUB;
#pragma unroll
        for (int u = 0; u < DSUB; u += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(src + u));
            qn[u] = v.x; qn[u + 1] = v.y; qn[u + 2] = v.z; qn[u + 3] = v.w;
        }
    };
    if (q0 < q1) fetch(q0);
    for (int q = q0; q < q1; ++q) {
        float qv[DSUB];
#pragma unroll
        for (int u = 0; u < DSUB; ++u) qv[u] = lut_s * qn[u];
        const float scale = scale_n;
        if (q + 1 < q1) fetch(q + 1);
        uint8_t* img = t.lut_img + (size_t)q * t.lut_bytes;
#pragma unroll
        for (int i = 0; i < EPT; ++i) {
            float acc = 0.f;
#pragma unroll
            for (int u = 0; u < DSUB; ++u) acc = fmaf(qv[u], cw[i][u], acc);
            if (off[i] != 0xFFFFFFFFu) {
                const int v = __float2int_rn(acc * scale);
                *reinterpret_cast<int*>(img + off[i]) = v;
                if (copy_delta) *reinterpret_cast<int*>(img + off[i] + copy_delta) = v;
            }
        }
    }
}

cudaError_t launch_build_tables(const IndexImpl* ix, const float* queries, int nq, uint8_t* lut_img, float* lut_inv,
                                float* lut_scale, int32_t* ok, cudaStream_t s) {
    const int dsub = ix->dsub;
    const TableArgs t = table_args(ix, queries, lut_img, lut_inv);
    if (nq > 64 && lut_scale && (dsub == 4 || dsub == 8 || dsub == 12 || dsub == 16)) {
        launch_overlapped(table_scales_kernel, dim3(nq), dim3(128), 0, s, queries, ix->cwmax, ix->d, dsub, ix->M, lut_scale, lut_inv, ok);
        const int ept = BTB_CW_FLOATS / dsub;
        const int G = 256 / ix->M;  // >= 2: the scan supports M <= 128
        const int threads = ix->M * G;
        const int parts = (KSUB + G * ept - 1) / (G * ept);
        int qchunk = (int)(((long long)nq * parts + 4 * ix->num_sms - 1) / (4 * ix->num_sms));
        if (qchunk < 1) qchunk = 1;
        const dim3 grid(parts, (nq + qchunk - 1) / qchunk);
        switch (dsub) {
            case 4: launch_overlapped(build_tables_batch_kernel<4>, grid, dim3(threads), 0, s, t, lut_scale, nq, qchunk); break;
            case 8: launch_overlapped(build_tables_batch_kernel<8>, grid, dim3(threads), 0, s, t, lut_scale, nq, qchunk); break;
            case 12: launch_overlapped(build_tables_batch_kernel<12>, grid, dim3(threads), 0, s, t, lut_scale, nq, qchunk); break;
            default: launch_overlapped(build_tables_batch_kernel<16>, grid, dim3(threads), 0, s, t, lut_scale, nq, qchunk); break;
        }
        count_launch(2);
        return cudaGetLastError();
    }
    launch_overlapped(build_tables_kernel, dim3(table_parts(ix, nq), nq), dim3(BT_THREADS), (size_t)(ix->d + ix->M) * 4, s, t);
    count_launch();
    return cudaGetLastError();
}

// ---- codebook transpose: cb[m][j][t] -> cbT[j][m][t] -------------------------------------------
__global__ void transpose_codebook_kernel(const float* __restrict__ cb, int M, int dsub, float* __restrict__ cbT) {
    const int total = M * KSUB * dsub;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int t = i % dsub, jm = i / dsub, m = jm % M, j = jm / M;
        cbT[i] = cb[((size_t)m * KSUB + j) * dsub + t];
    }
}
cudaError_t launch_transpose_codebook(const float* cb, int M, int dsub, float* cbT, cudaStream_t s) {
    transpose_codebook_kernel<<<256, 256, 0, s>>>(cb, M, dsub, cbT);
    count_launch();
    return cudaGetLastError();
}

// ---- per-vector term of the squared-L2 expansion ------------------------------------------------
// ||q - (c + r)||^2 = ||q - c||^2 + (||r||^2 + 2<c, r>) - 2<q, r>,  r = decoded residual of the vector.
// The middle term depends on the stored vector only; it is computed once per index, in double, one
// warp per vector (lanes over sub-spaces), and rounded to float once.
template <bool BF16>
__global__ void vector_terms_kernel(const uint8_t* __restrict__ codes, const int64_t* __restrict__ offsets,
                                    const void* __restrict__ centroids, const float* __restrict__ cb, long long N,
                                    int nlist, int d, int M, int dsub, float* __restrict__ vterm) {
    const int lane = threadIdx.x & 31;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long pos = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; pos < N; pos += warps) {
        int lo = 0, hi = nlist;  // offsets[lo] <= pos < offsets[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (offsets[mid] <= pos) lo = mid; else hi = mid;
        }
        double acc = 0.0;
        for (int m = lane; m < M; m += 32) {
            const int code = codes[pos * M + m];
            const float* cw = cb + ((size_t)m * KSUB + code) * dsub;
            for (int t = 0; t < dsub; ++t) {
                const size_t ci = (size_t)lo * d + m * dsub + t;
                const double c = BF16 ? (double)__bfloat162float(static_cast<const __nv_bfloat16*>(centroids)[ci])
                                      : (double)static_cast<const float*>(centroids)[ci];
                const double r = (double)cw[t];
                acc += r * (r + 2.0 * c);
            }
        }
        for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) vterm[pos] = (float)acc;
    }
}

cudaError_t launch_vector_terms(const IndexImpl* ix, float* vterm, cudaStream_t s) {
    if (ix->N == 0) return cudaSuccess;
    const long long want = (ix->N * 32 + 255) / 256;
    const int blocks = (int)(want < 148LL * 64 ? want : 148LL * 64);
    if (ix->coarse_bf16)
        vector_terms_kernel<true><<<blocks, 256, 0, s>>>(ix->codes, ix->list_offsets, ix->centroids, ix->codebooks,
                                                         ix->N, ix->nlist, ix->d, ix->M, ix->dsub, vterm);
    else
        vector_terms_kernel<false><<<blocks, 256, 0, s>>>(ix->codes, ix->list_offsets, ix->centroids, ix->codebooks,
                                                          ix->N, ix->nlist, ix->d, ix->M, ix->dsub, vterm);
    count_launch();
    return cudaGetLastError();
}

// ---- work planning: tiles per pair and their exclusive prefix sum ------------------------------
// Three small launches: (1) tiles per pair with a CTA-local exclusive scan and one total per CTA,
// (2) one CTA scans the totals, (3) every CTA adds its offset; thresholds and slot counters are reset on the way.
constexpr int PT_THREADS = 256;
__global__ void __launch_bounds__(PT_THREADS) pair_tiles_kernel(const int32_t* __restrict__ probe_list,
                                                                const int64_t* __restrict__ offsets, int npairs, int nprobe,
                                                                int tile_vecs, int lead, const PairTiles pt, int64_t* __restrict__ prefix,
                                                                long long* __restrict__ block_sums) {
    __shared__ long long warp_sums[PT_THREADS / 32];
    grid_dependency_wait();
    grid_dependents_may_launch();
    const int p = blockIdx.x * PT_THREADS + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long v = 0;
    if (p < npairs) {
        const int l = probe_list[p];
        if (pt.head == nullptr) v = tiles_of(offsets[l + 1] - offsets[l], tile_vecs) + pair_lead(p, nprobe, lead);
        else v = (l < 0 ? 0 : tiles_of(offsets[l + 1] - offsets[l], entry_tile_vecs(p, nprobe, tile_vecs, pt))) + entry_lead(p, nprobe, lead, pt);
    }
    long long incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    long long before = incl - v;
    for (int w = 0; w < warp; ++w) before += warp_sums[w];
    if (p < npairs) prefix[p] = before;
    if (threadIdx.x == PT_THREADS - 1) block_sums[blockIdx.x] = before + v;
}

// In-place exclusive scan of n totals by one CTA; the grand total goes to *total_out.
__global__ void __launch_bounds__(PFX_THREADS) scan_totals_kernel(long long* __restrict__ sums, int n,
                                                                  int64_t* __restrict__ total_out) {
    __shared__ long long warp_sums[32];
    __shared__ long long carry_s;
    grid_dependency_wait();
    grid_dependents_may_launch();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) carry_s = 0;
    __syncthreads();
    for (int base = 0; base < n; base += PFX_THREADS) {
        const int i = base + tid;
        const long long v = i < n ? sums[i] : 0;
        long long incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            long long w = warp_sums[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            warp_sums[lane] = w;  // inclusive over warps
        }
        __syncthreads();
        const long long before = carry_s + (warp ? warp_sums[warp - 1] : 0) + incl - v;
        if (i < n) sums[i] = before;
        __syncthreads();
        if (tid == PFX_THREADS - 1) carry_s = before + v;
        __syncthreads();
    }
    if (tid == 0) *total_out = carry_s;
}

__global__ void __launch_bounds__(PT_THREADS) add_offsets_kernel(int64_t* __restrict__ prefix, int npairs,
                                                                 const long long* __restrict__ block_sums,
                                                                 unsigned long long* __restrict__ qthresh, int nq,
                                                                 int32_t* __restrict__ slot_cnt, int nslots) {
    grid_dependency_wait();
    grid_dependents_may_launch();
    const int p = blockIdx.x * PT_THREADS + threadIdx.x;
    if (p < npairs) prefix[p] += block_sums[blockIdx.x];
    for (int i = p; i < nq; i += gridDim.x * PT_THREADS) qthresh[i] = KEY_MAX;
    for (int i = p; i < nslots; i += gridDim.x * PT_THREADS) slot_cnt[i] = 0;
}

// Small batches: one CTA does the whole preparation of a search (tiles per pair, their prefix sum,
// threshold and slot-counter reset), which would otherwise be four launches of a few microseconds each.
// With table_parts > 0 the CTAs after the first build the batch's lookup tables meanwhile (the tables depend on the
// queries only, so nothing orders them against the planning).
__global__ void __launch_bounds__(PFX_THREADS) plan_small_kernel(const int32_t* __restrict__ probe_list,
                                                                 const int64_t* __restrict__ offsets, int npairs, int nprobe,
                                                                 int tile_vecs, int lead, const PairTiles pt, int64_t* __restrict__ prefix,
                                                                 unsigned long long* __restrict__ qthresh, int nq,
                                                                 int32_t* __restrict__ slot_cnt, int nslots,
                                                                 const TableArgs tables, int table_parts) {
    extern __shared__ float bt_smem[];
    grid_dependency_wait();
    grid_dependents_may_launch();
    if (blockIdx.x > 0) {
        const int b = blockIdx.x - 1;
        build_table_part(tables, b / table_parts, b % table_parts, table_parts, bt_smem);
        return;
    }
    __shared__ long long warp_sums[32];
    plan_pairs_cta(probe_list, offsets, npairs, nprobe, tile_vecs, lead, pt, prefix, qthresh, nq, slot_cnt, nslots, warp_sums);
}

// Small batches whose probe selection plans the scan itself (see FusedPlan): what that kernel needs, or false when
// the batch does not qualify (tables not prebuilt, too many pairs for one CTA, more than 64 queries).
bool fused_plan_args(const IndexImpl* ix, int nq, int npairs, const float* queries, uint8_t* lut_img, float* lut_inv,
                     int64_t* work_prefix, unsigned long long* qthresh, int32_t* slot_cnt, int nslots, int lead, uint32_t* ticket,
                     FusedPlan* fp) {
    fp->enabled = 0;
    if (!lut_img || npairs > PLAN_SMALL_MAX || nq > 64) return false;
    fp->enabled = 1;
    fp->nq = nq;
    fp->ticket = ticket;
    fp->offsets = ix->list_offsets;
    fp->tile_vecs = scan_tile_vecs(ix, nq, npairs / nq);
    fp->lead = lead;
    fp->prefix = work_prefix;
    fp->qthresh = qthresh;
    fp->slot_cnt = slot_cnt;
    fp->nslots = nslots;
    fp->tables = table_args(ix, queries, lut_img, lut_inv);
    fp->table_parts = table_parts(ix, nq);
    return true;
}

// view (may be null): probe_list holds the entries of a batch with pairs of queries (the tables are built by then).
cudaError_t launch_plan_work(const IndexImpl* ix, const int32_t* probe_list, int npairs, int tile_vecs, int lead, const PairView* view,
                             int32_t* pair_tiles, int64_t* work_prefix, unsigned long long* qthresh, int nq,
                             int32_t* slot_cnt, int nslots, const float* queries, uint8_t* lut_img, float* lut_inv,
                             float* lut_scale, cudaStream_t s) {
    const bool fused_tables = lut_img && npairs <= PLAN_SMALL_MAX && nq <= 64;
    if (lut_img && !fused_tables && !view) {
        const cudaError_t et = launch_build_tables(ix, queries, nq, lut_img, lut_inv, lut_scale, nullptr, s);
        if (et != cudaSuccess) return et;
    }
    PairTiles pt = {nullptr, 0, 0};
    if (view) { pt.head = view->head; pt.tile_vecs = view->tile_vecs; pt.lead = lead ? scan_pair_lead(ix, view->tile_vecs) : 0; }
    if (npairs <= PLAN_SMALL_MAX) {
        const int parts = fused_tables ? table_parts(ix, nq) : 0;
        launch_overlapped(plan_small_kernel, dim3(1 + parts * nq), dim3(PFX_THREADS),
                          parts ? (size_t)(ix->d + ix->M) * 4 : 0, s,
            probe_list, ix->list_offsets, npairs, npairs / nq, tile_vecs, lead, pt, work_prefix, qthresh, nq, slot_cnt, nslots,
            table_args(ix, queries, lut_img, lut_inv), parts);
        count_launch();
        return cudaGetLastError();
    }
    // pair_tiles (npairs int32 of scratch) holds the per-CTA totals: one 64-bit word per 256 pairs
    const int nblocks = (npairs + PT_THREADS - 1) / PT_THREADS;
    long long* block_sums = reinterpret_cast<long long*>(pair_tiles);
    launch_overlapped(pair_tiles_kernel, dim3(nblocks), dim3(PT_THREADS), 0, s, probe_list, ix->list_offsets, npairs, npairs / nq,
                      tile_vecs, lead, pt, work_prefix, block_sums);
    launch_overlapped(scan_totals_kernel, dim3(1), dim3(PFX_THREADS), 0, s, block_sums, nblocks, work_prefix + npairs);
    launch_overlapped(add_offsets_kernel, dim3(nblocks), dim3(PT_THREADS), 0, s, work_prefix, npairs, block_sums, qthresh, nq,
                      slot_cnt, nslots);
    count_launch(3);
    return cudaGetLastError();
}

}  // namespace rago
