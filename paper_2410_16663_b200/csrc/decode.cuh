// Decode-stage attention (one query row per sequence over the cached K and V), split along
// the cache: each CTA streams one chunk of one (sequence, kv head) through a TMA-fed
// shared-memory ring and keeps running (rowmax, rowsum, O) for the query heads that share
// the kv head; the CTAs of a cluster, or a second kernel, merge the per-chunk partial results.  The work is a single
// pass over the cache, so the kernel is written for HBM bandwidth: every cache byte is read
// exactly once and nothing but the partials is written.
#pragma once

#include <type_traits>

#include "prefill_simple.cuh"
#include "sm100_ptx.cuh"

namespace fa {

constexpr int kDecTile = 128;                 // keys per shared-memory tile
constexpr int kDecStages = 3;                 // ring depth (K and V tiles each)
constexpr float kDecRefDropLog2 = 6.f;        // see DecodeParams::ref_tiles
constexpr int kDecTileBytes = 32768;          // a tile of d = 128
// Head dimension D (128 or 64): a tile is 128 keys x D 16-bit elements, one or two swizzled
// boxes, in a ring of three slots per operand.  With D = 64 a CTA's rings are 96 KiB and two
// CTAs share an SM: the bytes in flight per SM are those of D = 128, and twice the consumer
// warps work on them -- a key costs the same instructions whatever D is and brings half the
// bytes (measured on 64 sequences of 1K to 32K keys: 6.99 against 6.00 TB/s with one CTA of six
// slots per SM).
template <int D>
struct DecShape {
    static_assert(D == 64 || D == 128, "head dimensions of the 16-bit decode kernel");
    static constexpr int kTileBytes = kDecTile * D * 2;
    static constexpr int kStages = kDecStages;
    static constexpr int kCtasPerSm = 128 / D;
    static constexpr int kSmem = 1024 + 2 * kStages * kTileBytes;
};

struct DecodeParams {
    const void* q;        // [B,Sq,Hq,d] 16-bit
    const int* seqlens;   // [B] device
    float* o_part;        // [B,Sq,Hq,n_chunks,d]; cut by the device (slots > 0): [slots,Sq,Hq,d], a chunk of any sequence in each
    float* lse_part;      // the same without d
    int B, Hq, Hkv, Smax;
    int chunk;            // keys per chunk (multiple of kDecTile); cut by the device: what it would be otherwise
    int n_chunks;         // ceil(Smax / chunk); cut by the device: the mean number per sequence, rounded up
    float scale_log2;
    // paged cache (block_table != nullptr): key j of sequence b is row j % page_size of page
    // block_table[b * table_stride + j / page_size]; the tensor maps then run over
    // [pages, page_size, Hkv, d]; page_size is a multiple of kDecTile, or 16, 32 or 64 (then a
    // tile is several pages and the TMA box is one page high)
    const int* block_table;
    int page_size, table_stride;
    float v_scale;        // 8-bit cache only: factor of the stored values
    int Sq;               // query rows per sequence (1; more for the append form of the fp16 kernel)
    // fp16/bf16 kernel with a single chunk per sequence (n_chunks == 1): the split kernel writes
    // the result itself and no merge kernel runs (nullptr otherwise)
    void* o_final;
    float* lse_final;
    // the chunks of a sequence are a cluster's CTAs and are merged through distributed shared
    // memory (see decode_plan); o_final and lse_final are then the result's
    int clustered = 0;
    // Tiles (a power of two) after which the reference of the probabilities, the running max, is lowered
    // by ref_drop.  The probabilities are rounded to 16 bits for the second product, all but that of the
    // key that sets the reference, which is exactly 1: the fewer keys share a reference, the smaller is
    // the rounding error.  Chunks that are longer only because a sequence is one cluster's, or because the
    // device cuts them (see decode_plan), lower it where they would end otherwise, so that the next keys set their
    // own (1 sequence, 5 heads, 8192 keys: 2.54e-4 from the result in 64 bits, 2.61e-4 without this).
    // What has been summed grows by up to 2^6 each time.  With 16-bit caches by no more than 2^42 in all, however long the
    // chunk is (see dec_lowered): the sums of probabilities stay far inside fp32, and those of the values times them do
    // for values up to 2^74.  8-bit values are below 2^9, and their chunks lower it 15 times at most, by 2^90 (see
    // DecodePlan::fill; the limit in the kernel cost two column blocks 3 %: 8 x 64/2 over 27389 keys 38.9 -> 40.3 us.  The
    // 16-bit kernels are level with it: 1 x 5 over 8192 8.4 / 8.4, 12 x 5 over up to 5861 23.9 / 23.9).
    int ref_tiles = 1 << 30;
    float ref_drop = 0.f;   // kDecRefDropLog2 / scale_log2
    // Chunks cut by the sequences' own lengths (kDecBalanced, see DecBalance): CTAs per kv head over all
    // sequences, and the tiles per chunk that are enough whatever the lengths are
    int slots = 0, most_tiles = 0;
    int bf16_io = 0;      // 8-bit cache kernel only: q and o are bf16 (fp16 otherwise)
};


// ---------------------------------------------------------------------------------------
// Split kernel.  A CTA takes one chunk of one (sequence, kv head) and up to 16 of the query
// heads that share the kv head (all of them when Hq / Hkv <= 16).  The query rows are padded
// to the 16 rows of a warp-level mma.sync (m16n8k16, fp32 accumulate): the scan is bound by
// the cache stream, and the warp-level tensor path keeps the arithmetic per cache byte far
// below what the FMA pipe would need, for one query head as well as for sixteen.  Each of the
// four consumer warps owns keys [32w, 32w+32) of every 128-key tile and keeps its own running
// (rowmax, rowsum, O) for them, so consumer warps never synchronise with each other until the
// final merge; a fifth warp issues the TMA loads into a 3-slot ring of K and V tiles.
// Cache rows past the sequence may hold NaN: their scores are masked and their V rows are
// zeroed in shared memory before the second MMA touches them.
constexpr int kDecMmaThreads = 160;

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void mma_16816_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Where a tile's bytes lie in shared memory.  A tile is loaded in boxes of `rows` keys (128, or one
// page of 16, 32 or 64), and a box holds all of d: its 64-element blocks one after the other, `rows`
// rows of 128 swizzled bytes each.  (A 16-key page of d = 128 as one box of 4 KiB instead of two of
// 2 KiB: the TMA unit's cost per box, about 100 clocks, is what bounds small pages: 48 sequences
// of 100 to 8000 keys, 8 kv heads, 164 -> 143 us; 16-key pages reach 92 to 96 % of a contiguous cache's rate.)
template <int D>
struct DecTileLayout {
    int rows_log2;
    uint32_t block;   // bytes from one 64-element block of a box to the next
    __device__ __forceinline__ explicit DecTileLayout(const DecodeParams& p) {
        const int rows = (p.block_table != nullptr && p.page_size < kDecTile) ? p.page_size : kDecTile;
        rows_log2 = 31 - __clz(rows);
        block = (uint32_t)rows * 128u;
    }
    // first byte of key `key` of the tile in its box's first block
    __device__ __forceinline__ uint32_t key(int key) const {
        const uint32_t box = (uint32_t)key >> rows_log2;
        return (D / 64 - 1) * box * block + (uint32_t)key * 128u;
    }
};

// The reference of a row (its running max, m) lowered by `drop` (see DecodeParams::ref_tiles), but no further than seven
// times that below the highest one that the chunk has had, `top`: keys whose scores do not reach up to there weigh
// less than 2^-42 of that one.
__device__ __forceinline__ float dec_lowered(float m, float& top, float drop) {
    top = fmaxf(top, m);
    return fmaxf(m - drop, fmaf(-7.f, drop, top));
}

// How a call's sequences are cut: every DecodeParams::chunk keys (kDecPlain), the chunks of a sequence the CTAs of a cluster
// (kDecCluster), or by the lengths that the device finds (kDecBalanced).
constexpr int kDecPlain = 0, kDecCluster = 1, kDecBalanced = 2;
constexpr int kDecBalancedSeqs = 32;

// Chunks of equal length for sequences of different lengths, as short as p.slots CTAs per kv head allow (no more than the
// device runs at once, and than the workspace has room for): worked out from the lengths by every warp for itself, a sequence per lane.  The sequences take the
// CTAs one after the other, each at least one (it may have no keys).  (The loops are not unrolled: this runs once per CTA, and
// fetching its instructions takes longer than executing them.)
struct DecBalance {
    int unit;                // tiles per chunk
    int len, count, first;   // of sequence `lane`
    // n / u, rounded up: exact for n below 2^15 at u up to 32 (the half keeps the quotient away from the whole numbers)
    static __device__ __forceinline__ int parts(float n, int u) { return (int)((n - 0.5f) * __frcp_rn((float)u)) + 1; }
    __device__ __forceinline__ DecBalance(const DecodeParams& p, int lane) {
        const bool mine = lane < p.B;
        len = mine ? max(0, min(p.seqlens[lane], p.Smax)) : 0;
        const int t = max(1, (len + kDecTile - 1) / kDecTile);
        int lo = max(1, (__reduce_add_sync(0xffffffffu, mine ? t : 0) + p.slots - 1) / p.slots), hi = max(lo, p.most_tiles);
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__reduce_add_sync(0xffffffffu, mine ? parts((float)t, mid) : 0) <= p.slots) hi = mid;
            else lo = mid + 1;
        }
        unit = lo;
        count = mine ? parts((float)t, unit) : 0;
        int sum = count;
#pragma unroll 1
        for (int sh = 1; sh < p.B; sh <<= 1) {
            const int low = __shfl_up_sync(0xffffffffu, sum, sh);
            if (lane >= sh) sum += low;
        }
        first = sum - count;
    }
    // The sequence of CTA `at`, its chunk and length; false past the last chunk.
    __device__ __forceinline__ bool find(int at, int& b, int& c, int& length) const {
        b = __ffs(__ballot_sync(0xffffffffu, at >= first && at < first + count)) - 1;
        if (b < 0) return false;
        c = at - __shfl_sync(0xffffffffu, first, b);
        length = __shfl_sync(0xffffffffu, len, b);
        return true;
    }
};

// Merge of the chunks of one sequence whose CTAs form a cluster (rank = chunk): part holds this
// CTA's normalised rows and their log-sum-exps.  Row r is finished by CTA r mod (chunks with
// keys); store(r, col, value, lse) writes a column of it.  Every thread of the CTA calls this.
constexpr int kDecPartOffset = 40960;   // bytes from the ring's start, past the warps' merge buffer
template <int D, typename Store>
__device__ __forceinline__ void dec_cluster_merge(const float* part, const float* part_lse, int G, int chunk_rank, int n_live,
                                                  int tid, Store store) {
    __syncwarp();
    cluster_sync_all();   // (CTAs without keys have left; their chunks are not read)
    if (tid < 128) {
        // D / 4 lanes (16 or 32) work on a row, four columns each; lane i of them also looks after chunk i's weight
        constexpr int kLanes = D / 4;
        const int sl = tid % kLanes, col = 4 * sl;
        const uint32_t po = smem_u32(part) + 4 * col, pl = smem_u32(part_lse);
        for (int r0 = chunk_rank; r0 < G; r0 += n_live * (128 / kLanes)) {
            const int r = r0 + n_live * (tid / kLanes);
            const bool live = r < G;
            float l = -INFINITY, v[8][4];
            auto load = [&](int i0) {   // rows of eight chunks
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    v[i][0] = v[i][1] = v[i][2] = v[i][3] = 0.f;
                    if (live && i0 + i < n_live) cluster_ld4(cluster_map(po + 4 * D * r, i0 + i), v[i]);
                }
            };
            if (live && sl < n_live) l = cluster_ld(cluster_map(pl + 4 * r, sl));
            load(0);   // (on their way while the weights are worked out)
            float M = l;
#pragma unroll
            for (int sh = 8; sh > 0; sh >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, sh, 16));
            M = __shfl_sync(0xffffffffu, M, 0, kLanes);
            const float w = (l == -INFINITY) ? 0.f : __expf(l - M);
            float wsum = w;
#pragma unroll
            for (int sh = 8; sh > 0; sh >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, sh, 16);
            wsum = __shfl_sync(0xffffffffu, wsum, 0, kLanes);
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            for (int i0 = 0; i0 < n_live; i0 += 8) {
                if (i0 > 0) load(i0);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float wi = __shfl_sync(0xffffffffu, w, i0 + i, kLanes);   // (zero past the live chunks)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[k] = fmaf(wi, v[i][k], acc[k]);
                }
            }
            if (live) {
                const bool any = wsum != 0.f;   // (several query tokens: one that sees no key at all)
                const float inv = any ? 1.f / wsum : 0.f;
                store(r, col, make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv), any ? M + logf(wsum) : -INFINITY);
            }
        }
    }
    __syncwarp();
    cluster_sync_all();   // nobody's shared memory goes away while others read it
}

// Merge of the four consumer warps' states of row r (mo: [4][16][D] unnormalised rows, ml: [4][16] pairs of
// max and sum): columns col .. col + 3, and the row's log-sum-exp.
template <int D>
__device__ __forceinline__ float4 dec_warp_merge(const float* mo, const float* ml, int r, int col, float scale_log2, float factor,
                                                 float& lse) {
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < 4; ++w) M = fmaxf(M, ml[(w * 16 + r) * 2]);
    float l = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const float mw = ml[(w * 16 + r) * 2];
        const float sw = (mw == -INFINITY) ? 0.f : fast_exp2((mw - M) * scale_log2);
        const float4 v = *reinterpret_cast<const float4*>(&mo[(w * 16 + r) * D + col]);
        l += sw * ml[(w * 16 + r) * 2 + 1];
        acc[0] += sw * v.x;
        acc[1] += sw * v.y;
        acc[2] += sw * v.z;
        acc[3] += sw * v.w;
    }
    // l == 0: a query token that sees none of this chunk's keys, whatever their values are.  (A NaN sum, from a
    // NaN or infinite score, makes the row and its log-sum-exp NaN here and in the merges.)
    const bool none = l == 0.f;
    lse = none ? -INFINITY : (M * scale_log2 + log2f(l)) * 0.6931471805599453f;
    const float inv = none ? 0.f : 1.f / l;
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = none ? 0.f : acc[k] * inv * factor;
    return make_float4(acc[0], acc[1], acc[2], acc[3]);
}
// Four consecutive elements of an output row.
template <typename T>
__device__ __forceinline__ void dec_store4(void* o, long long at, const float4& v) {
    *reinterpret_cast<uint2*>(static_cast<T*>(o) + at) = make_uint2(pack2<T>(v.x, v.y), pack2<T>(v.z, v.w));
}

// The consumer warps' work in the keys-as-rows form (at most 8 rows, i.e. (token, head) pairs,
// per kv head).  A warp-level MMA has 16 rows and 8 columns: with the query heads as rows, as in the
// general form below, a kv head with 1 to 8 query heads leaves half or more of every MMA to
// padding.  Here the KEYS are the rows: S^T = K q^T (A = 16 keys x 16 elements of K by plain
// ldmatrix, B = q^T, the 8 columns are the heads), and O^T += V^T P^T (A = 16 output columns x 16
// keys of V by transposing ldmatrix, B = P^T, which is the accumulator layout of S^T transposed
// 8 x 8 with movmatrix).  A tile then takes half the MMAs, a thread holds half the scores and
// half the accumulators, and the row maxima and sums run over the lanes that share a column.
// q_col: the query row that is this thread's column g of q^T (nullptr: padding).  kMulti: hide0,
// hide1 say how many of the sequence's last keys the rows in this thread's accumulator columns
// 2 t4, 2 t4 + 1 must not see (they came after the row's token).
// Leaves each warp's (max, sum, O) in mo / ml in the layout the merge expects; returns false
// after a wait that gave up.
template <bool kMulti, typename T, int D, bool kLower>
__device__ __forceinline__ bool dec_consume_key_rows(const DecodeParams& p, uint64_t* bars, volatile uint32_t* abort_flag,
                                                     uint32_t sK, uint32_t sV, float* mo, float* ml, int warp, int lane,
                                                     const T* q_col, int hide0, int hide1, int len, int k_begin, int k_end,
                                                     int n_tiles) {
    constexpr int kStages = DecShape<D>::kStages, kTileB = DecShape<D>::kTileBytes;
    constexpr bool kBf16 = std::is_same<T, __nv_bfloat16>::value;
    const int g = lane >> 2, t4 = lane & 3;
    // q^T as B fragments: column g is head g, rows 2 t4, 2 t4 + 1 (and + 8) of every 16-element step
    uint32_t qb[D / 16][2];
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        const int d0 = ks * 16 + 2 * t4;
        qb[ks][0] = q_col ? *reinterpret_cast<const uint32_t*>(q_col + d0) : 0u;
        qb[ks][1] = q_col ? *reinterpret_cast<const uint32_t*>(q_col + d0 + 8) : 0u;
    }
    // O^T: block i holds output columns 16 i + g (values 0, 1) and 16 i + 8 + g (values 2, 3) of heads 2 t4, 2 t4 + 1
    float o[D / 16][4];
#pragma unroll
    for (int i = 0; i < D / 16; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};  // heads 2 t4 and 2 t4 + 1
    float top[2] = {-INFINITY, -INFINITY};   // (kLower: see dec_lowered)
    const int key_w = warp * 32;  // this warp's keys inside a tile
    bool ok = true;
    // this lane's key of each block of 16, for the K and for the V matrices
    const DecTileLayout<D> lay(p);
    const uint32_t k_at[2] = {lay.key(key_w + ((lane >> 3) & 1) * 8 + (lane & 7)), lay.key(key_w + 16 + ((lane >> 3) & 1) * 8 + (lane & 7))};
    const uint32_t v_at[2] = {lay.key(key_w + (lane >> 4) * 8 + (lane & 7)), lay.key(key_w + 16 + (lane >> 4) * 8 + (lane & 7))};

    for (int t = 0; t < n_tiles; ++t) {
        const int st = t % kStages;
        const uint32_t parity = (t / kStages) & 1;
        const int valid = min(kDecTile, k_end - (k_begin + t * kDecTile)) - key_w;  // valid keys of this warp's 32
        const bool lower = kLower && (t & (p.ref_tiles - 1)) == 0;   // see DecodeParams
        ok = mbar_wait(smem_u32(&bars[st]), parity, abort_flag, 20);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        uint32_t pt[2][2];   // P^T as B fragments, per block of 16 keys
        if (valid > 0) {
            // ---- S^T = K q^T: two blocks of 16 keys
            float sc[2][4];  // (key 16 mb + g | heads 2 t4, 2 t4 + 1), (key 16 mb + g + 8 | the same heads)
            const uint32_t kt = sK + st * kTileB;
#pragma unroll
            for (int mb = 0; mb < 2; ++mb) {
                sc[mb][0] = sc[mb][1] = sc[mb][2] = sc[mb][3] = 0.f;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    // matrices: (keys 0-7, chunk 2 ks), (keys 8-15, chunk 2 ks), (keys 0-7, chunk 2 ks + 1), (keys 8-15, ...)
                    const int chunk = 2 * ks + (lane >> 4);
                    const uint32_t addr = kt + k_at[mb] + (chunk >> 3) * lay.block + (((chunk & 7) ^ (lane & 7)) << 4);
                    uint32_t a[4];
                    ldsm_x4(addr, a[0], a[1], a[2], a[3]);
                    if (kBf16) mma_16816_bf16(sc[mb], a, qb[ks][0], qb[ks][1]);
                    else mma_16816(sc[mb], a, qb[ks][0], qb[ks][1]);
                }
            }
            // ---- mask, running max, probabilities
            // keys of this warp's 32 that a row may see: all valid ones, minus (several query
            // rows) those among the sequence's last that came after the row's token
            const int seen0 = kMulti ? min(valid, len - hide0 - (k_begin + t * kDecTile) - key_w) : valid;
            const int seen1 = kMulti ? min(valid, len - hide1 - (k_begin + t * kDecTile) - key_w) : valid;
            float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
            for (int mb = 0; mb < 2; ++mb) {
                const int k_lo = mb * 16 + g;
                if (k_lo >= seen0) sc[mb][0] = -INFINITY;
                if (k_lo >= seen1) sc[mb][1] = -INFINITY;
                if (k_lo + 8 >= seen0) sc[mb][2] = -INFINITY;
                if (k_lo + 8 >= seen1) sc[mb][3] = -INFINITY;
                mx0 = fmaxf(mx0, fmaxf(sc[mb][0], sc[mb][2]));
                mx1 = fmaxf(mx1, fmaxf(sc[mb][1], sc[mb][3]));
            }
#pragma unroll
            for (int sh = 4; sh <= 16; sh <<= 1) {  // over the lanes that hold other keys of the same heads
                mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, sh));
                mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, sh));
            }
            // finite when key 0 of the warp is visible (always with one query token; an earlier
            // token of several may see none of the warp's keys: its state then stays empty)
            const float mn0 = fmaxf(lower ? dec_lowered(m_run[0], top[0], p.ref_drop) : m_run[0], mx0);
            const float mn1 = fmaxf(lower ? dec_lowered(m_run[1], top[1], p.ref_drop) : m_run[1], mx1);
            const float a0 = (m_run[0] == -INFINITY) ? 0.f : fast_exp2((m_run[0] - mn0) * p.scale_log2);
            const float a1 = (m_run[1] == -INFINITY) ? 0.f : fast_exp2((m_run[1] - mn1) * p.scale_log2);
            m_run[0] = mn0;
            m_run[1] = mn1;
            const float nm0 = (kMulti && mn0 == -INFINITY) ? 0.f : -mn0 * p.scale_log2;
            const float nm1 = (kMulti && mn1 == -INFINITY) ? 0.f : -mn1 * p.scale_log2;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int mb = 0; mb < 2; ++mb) {
                const int k_lo = mb * 16 + g;
                float* e = sc[mb];
                e[0] = (k_lo < seen0) ? fast_exp2(fmaf(e[0], p.scale_log2, nm0)) : 0.f;
                e[1] = (k_lo < seen1) ? fast_exp2(fmaf(e[1], p.scale_log2, nm1)) : 0.f;
                e[2] = (k_lo + 8 < seen0) ? fast_exp2(fmaf(e[2], p.scale_log2, nm0)) : 0.f;
                e[3] = (k_lo + 8 < seen1) ? fast_exp2(fmaf(e[3], p.scale_log2, nm1)) : 0.f;
                s0 += e[0] + e[2];
                s1 += e[1] + e[3];
                // (key g | heads 2 t4, 2 t4 + 1) -> transposed: (head g | keys 2 t4, 2 t4 + 1), the B fragment
                const uint32_t lo = pack2<T>(e[0], e[1]), hi = pack2<T>(e[2], e[3]);
                asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(pt[mb][0]) : "r"(lo));
                asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(pt[mb][1]) : "r"(hi));
            }
            l_run[0] = l_run[0] * a0 + s0;  // per-thread partial of the sum over keys (reduced at the end)
            l_run[1] = l_run[1] * a1 + s1;
#pragma unroll
            for (int i = 0; i < D / 16; ++i) {
                o[i][0] *= a0;
                o[i][1] *= a1;
                o[i][2] *= a0;
                o[i][3] *= a1;
            }
        }
        ok = mbar_wait(smem_u32(&bars[kStages + st]), parity, abort_flag, 21);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (valid > 0) {
            const uint32_t vt = sV + st * kTileB;
            if (valid < 32) {
                // rows past the sequence may hold NaN bits: zero them (0 * NaN would poison O)
                for (int i = lane; i < (32 - valid) * (D / 8); i += 32) {
                    const int key = key_w + valid + i / (D / 8), ch = i % (D / 8);
                    const uint32_t addr = vt + lay.key(key) + (ch >> 3) * lay.block + (((ch & 7) ^ (key & 7)) << 4);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0u) : "memory");
                }
                __syncwarp();
            }
            // ---- O^T += V^T P^T: two steps of 16 keys, D / 16 blocks of 16 output columns
#pragma unroll
            for (int mb = 0; mb < 2; ++mb) {
                // matrices: (keys 0-7, chunk 2 i), (keys 0-7, chunk 2 i + 1), (keys 8-15, chunk 2 i), (keys 8-15, chunk 2 i + 1)
#pragma unroll
                for (int i = 0; i < D / 16; ++i) {
                    const int ch = 2 * i + ((lane >> 3) & 1);
                    const uint32_t addr = vt + v_at[mb] + (ch >> 3) * lay.block + (((ch & 7) ^ (lane & 7)) << 4);
                    uint32_t a[4];
                    ldsm_x4_trans(addr, a[0], a[1], a[2], a[3]);
                    if (kBf16) mma_16816_bf16(o[i], a, pt[mb][0], pt[mb][1]);
                    else mma_16816(o[i], a, pt[mb][0], pt[mb][1]);
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars[2 * kStages + st]));
    }
#pragma unroll
    for (int sh = 4; sh <= 16; sh <<= 1) {
        l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], sh);
        l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], sh);
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");   // every warp is through with the ring: it becomes the merge buffer
    if (ok) {
        const int h0 = warp * 16 + 2 * t4;
#pragma unroll
        for (int i = 0; i < D / 16; ++i) {
            mo[h0 * D + 16 * i + g] = o[i][0];
            mo[(h0 + 1) * D + 16 * i + g] = o[i][1];
            mo[h0 * D + 16 * i + 8 + g] = o[i][2];
            mo[(h0 + 1) * D + 16 * i + 8 + g] = o[i][3];
        }
        if (g == 0) {
            ml[h0 * 2] = m_run[0];
            ml[h0 * 2 + 1] = l_run[0];
            ml[(h0 + 1) * 2] = m_run[1];
            ml[(h0 + 1) * 2 + 1] = l_run[1];
        }
    }
    return ok;
}

// kMulti: Sq > 1 query rows per sequence, the last Sq positions of its cache (decoding after
// several tokens were appended, Appendix C with more than one new token): the 16 MMA rows of a
// CTA are then (token, head) pairs of one kv head, and query token t sees the keys up to
// position len - Sq + t.  q is [B,Sq,Hq,d], the partials see DecodeParams.
// grid: (Hkv * ceil(Sq * g / 16), n_chunks, B), or (.., slots, 1) with kDecBalanced, with g = Hq / Hkv.  The kv head is the fastest
// index: CTAs that run at the same time then read the same keys' rows of neighbouring heads,
// which are contiguous in the cache (a key's Hkv * D elements), instead of key ranges whole
// chunks apart (64 sequences of 1K to 32K keys, 32 kv heads: 2.39 against 2.48 ms).
// T: the 16-bit type of q, the cache and the probabilities (__half or __nv_bfloat16).
// D: the head dimension, 128 or 64.
// kKeyRows (at most 8 (token, head) rows per kv head): the consumers work in the keys-as-rows
// form (dec_consume_key_rows).
// kMode: how the sequences are cut (kDecPlain and the others).  (The clustered form is an instantiation of its own, as lowering
// the reference costs every tile two instructions and the merge below registers: 200 sequences of up to 600 keys,
// not clustered, 10.14 us in one instantiation for both, 10.33 with the reference, 9.98 apart.)
// (The kernels here do not release the next one early: its CTAs would take the places of this one's, or those
// next to it, and wait there.  16 sequences of up to 4096 keys, d = 64, 22.3 us with an early release, 20.5
// without; one of 32768 keys, 24.9 / 23.2; 8 of up to 8000, 30.5 / 29.6; 5 heads x 8192, 7.03 / 6.85; calls
// of 6 us level.)
template <bool kMulti, typename T, int D, bool kKeyRows, int kMode>
__global__ void __launch_bounds__(kDecMmaThreads, DecShape<D>::kCtasPerSm)
fa_decode_split_mma_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                           const DecodeParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    constexpr int kStages = DecShape<D>::kStages, kTileB = DecShape<D>::kTileBytes;
    const uint32_t sK = smem_base;
    const uint32_t sV = smem_base + kStages * kTileB;
    __shared__ __align__(8) uint64_t bars[3 * kStages];  // K full, V full, slot empty
    __shared__ volatile uint32_t abort_flag;

    const int tid = threadIdx.x;
    const int warp = uniform(tid >> 5), lane = tid & 31;
    int c = blockIdx.y, b = blockIdx.z;   // (kDecBalanced: found below)
    const int g_all = p.Hq / p.Hkv;
    const int Sq = kMulti ? p.Sq : 1;
    const int rows_all = g_all * Sq;               // (token, head) rows that share a kv head
    const int n_sub = (rows_all + 15) / 16;        // CTAs per kv head when there are more than 16
    const int hk = blockIdx.x / n_sub;
    const int sub = blockIdx.x % n_sub;
    const int G = min(16, rows_all - sub * 16);    // rows of this CTA
    // row r of the CTA: token and head, and its row in q and in the partial results
    auto row_token = [&](int r) { return kMulti ? (sub * 16 + r) / g_all : 0; };
    auto row_index = [&](int r) -> long long {
        const int R = sub * 16 + r;
        const int hh = kMulti ? R % g_all : R;
        return ((long long)b * Sq + row_token(r)) * p.Hq + hk * g_all + hh;
    };

    if (tid == 0) {
        for (int i = 0; i < 2 * kStages; ++i) mbar_init(smem_u32(&bars[i]), 1);
        for (int i = 0; i < kStages; ++i) mbar_init(smem_u32(&bars[2 * kStages + i]), 4);  // one arrival per consumer warp
        abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tm_k);
        tma_prefetch_desc(&tm_v);
    }
    grid_dep_wait();
    int len, chunk = p.chunk;
    if constexpr (kMode == kDecBalanced) {
        const DecBalance bal(p, lane);
        if (!bal.find(blockIdx.y, b, c, len)) return;   // (the same for all warps)
        chunk = bal.unit * kDecTile;
    } else {
        len = max(0, min(p.seqlens[b], p.Smax));
    }
    const int k_begin = c * chunk;
    const int k_end = min(len, k_begin + chunk);
    // row r's place among the partial results
    auto part_index = [&](int r) -> long long {
        return kMode == kDecBalanced ? row_index(r) + ((long long)blockIdx.y - b) * Sq * p.Hq : row_index(r) * p.n_chunks + c;
    };
    auto lse_index = [&](int r) -> long long {   // lse is [B,Hq,Sq]
        const int R = sub * 16 + r;
        return ((long long)b * p.Hq + hk * g_all + (kMulti ? R % g_all : R)) * Sq + row_token(r);
    };
    if (k_begin >= k_end) {  // uniform for the CTA
        if (kMode == kDecBalanced) {
            if (tid < G) p.lse_part[part_index(tid)] = -INFINITY;
        } else if (p.o_final != nullptr && c == 0 && tid < D) {   // a sequence without keys, and nobody else writes its rows
            for (int r = 0; r < G; ++r) {
                static_cast<T*>(p.o_final)[row_index(r) * D + tid] = T(0.f);
                if (tid == 0 && p.lse_final) p.lse_final[lse_index(r)] = -INFINITY;
            }
        }
        return;
    }
    const int n_tiles = (k_end - k_begin + kDecTile - 1) / kDecTile;
    float* part = reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)) + kDecPartOffset);   // [16][D]
    float* part_lse = part + 16 * D;                                                                         // [16]

    __syncthreads();

    if (warp == 4) {
        // ---------------------------------------------------------------- producer
        // the cache is read once: its lines go first when L2 needs room (q and the partial results stay)
        const uint64_t stream_policy = l2_policy_evict_first();
        // paged cache: the page of a tile is looked up one tile ahead of its loads, so that
        // the table read is not on the path that refills a freed slot
        const int* table = p.block_table ? p.block_table + (long long)b * p.table_stride : nullptr;
        if (table && p.page_size < kDecTile) {
            // pages of 16, 32 or 64 keys: a tile is several pages, each its own TMA box (pages past
            // the sequence's last are not loaded: their scores are masked and their V rows zeroed
            // by the consumers).  Lane i of the warp looks up and loads page i of every tile.
            const int ps = p.page_size, n_sub = kDecTile / ps;
            auto lookup = [&](int first_key) {
                const int key = first_key + lane * ps;
                return (lane < n_sub && key < k_end) ? table[key / ps] : -1;
            };
            int pg_next = lookup(k_begin);
            for (int t = 0; t < n_tiles; ++t) {
                const int st = t % kStages;
                const uint32_t bk = smem_u32(&bars[st]), bv = smem_u32(&bars[kStages + st]);
                const int row0 = k_begin + t * kDecTile;
                const int cur = pg_next;
                if (t + 1 < n_tiles) pg_next = lookup(row0 + kDecTile);
                bool ok = true;
                if (lane == 0) ok = mbar_wait(smem_u32(&bars[2 * kStages + st]), ((t / kStages) & 1) ^ 1, &abort_flag, 22);
                if (!__shfl_sync(0xffffffffu, ok, 0)) break;
                const int live = min(n_sub, (k_end - row0 + ps - 1) / ps);   // pages of this tile that hold keys
                if (lane == 0) {
                    mbar_expect_tx(bk, (uint32_t)(live * ps) * (2u * D));
                    mbar_expect_tx(bv, (uint32_t)(live * ps) * (2u * D));
                }
                __syncwarp();
                if (lane < live) {
                    const uint32_t offs = (uint32_t)(lane * ps) * (2u * D);
                    tma_load_5d_hint(sK + st * kTileB + offs, &tm_k, bk, 0, 0, 0, hk, cur, stream_policy);
                    tma_load_5d_hint(sV + st * kTileB + offs, &tm_v, bv, 0, 0, 0, hk, cur, stream_policy);
                }
            }
        } else if (lane == 0) {
            int page_next = table ? table[k_begin / p.page_size] : 0;
            for (int t = 0; t < n_tiles; ++t) {
                const int st = t % kStages;
                const uint32_t bk = smem_u32(&bars[st]), bv = smem_u32(&bars[kStages + st]);
                int row0 = k_begin + t * kDecTile;  // first key of the tile within the sequence
                int slab = b;                        // outermost coordinate: the sequence, or the page
                if (table) {
                    slab = page_next;
                    if (t + 1 < n_tiles) page_next = table[(row0 + kDecTile) / p.page_size];
                    row0 %= p.page_size;
                }
                if (!mbar_wait(smem_u32(&bars[2 * kStages + st]), ((t / kStages) & 1) ^ 1, &abort_flag, 22)) break;
                mbar_expect_tx(bk, kTileB);
                tma_load_5d_hint(sK + st * kTileB, &tm_k, bk, 0, row0, 0, hk, slab, stream_policy);
                mbar_expect_tx(bv, kTileB);
                tma_load_5d_hint(sV + st * kTileB, &tm_v, bv, 0, row0, 0, hk, slab, stream_policy);
            }
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- consumers
        const int g = lane >> 2, t4 = lane & 3;  // fragment row (query head g and g + 8) and column pair
        float* mo = reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)));  // [4 warps][16 rows][D]
        float* ml = mo + 4 * 16 * D;                                                         // [4][16][2]: m, l
        bool ok = true;
        if constexpr (kKeyRows) {
            // column g of q^T is row g of the CTA; accumulator columns 2 t4, 2 t4 + 1 are rows 2 t4, 2 t4 + 1
            const T* q_col = (g < G) ? static_cast<const T*>(p.q) + row_index(g) * D : nullptr;
            const int hide0 = kMulti ? Sq - 1 - row_token(min(2 * t4, G - 1)) : 0;
            const int hide1 = kMulti ? Sq - 1 - row_token(min(2 * t4 + 1, G - 1)) : 0;
            ok = dec_consume_key_rows<kMulti, T, D, kMode != kDecPlain>(p, bars, &abort_flag, sK, sV, mo, ml, warp, lane, q_col, hide0, hide1,
                                                    len, k_begin, k_end, n_tiles);
        } else {
        // Q as A fragments for the D / 16 k-steps (rows >= G are zero)
        uint32_t qa[D / 16][4];
        {
            const __half* q_lo = static_cast<const __half*>(p.q) + row_index(g) * D;
            const __half* q_hi = static_cast<const __half*>(p.q) + row_index(g + 8) * D;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
                const int k0 = ks * 16 + 2 * t4;
                qa[ks][0] = (g < G) ? *reinterpret_cast<const uint32_t*>(q_lo + k0) : 0u;
                qa[ks][1] = (g + 8 < G) ? *reinterpret_cast<const uint32_t*>(q_hi + k0) : 0u;
                qa[ks][2] = (g < G) ? *reinterpret_cast<const uint32_t*>(q_lo + k0 + 8) : 0u;
                qa[ks][3] = (g + 8 < G) ? *reinterpret_cast<const uint32_t*>(q_hi + k0 + 8) : 0u;
            }
        }
        // keys an earlier query token must not see: the last Sq - 1 - t of the sequence
        const int hide_lo = kMulti ? Sq - 1 - row_token(g) : 0;
        const int hide_hi = kMulti ? Sq - 1 - row_token(min(g + 8, G - 1)) : 0;
        float o[D / 8][4];
#pragma unroll
        for (int i = 0; i < D / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
        float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;  // rows g and g + 8
        float top_lo = -INFINITY, top_hi = -INFINITY;   // (not kDecPlain: see dec_lowered)
        const int key_w = warp * 32;  // this warp's keys inside a tile
        const DecTileLayout<D> lay(p);

        for (int t = 0; t < n_tiles; ++t) {
            const int st = t % kStages;
            const uint32_t parity = (t / kStages) & 1;
            const int valid = min(kDecTile, k_end - (k_begin + t * kDecTile)) - key_w;  // valid keys of this warp's 32
            const bool lower = kMode != kDecPlain && (t & (p.ref_tiles - 1)) == 0;   // see DecodeParams
            ok = mbar_wait(smem_u32(&bars[st]), parity, &abort_flag, 20);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            float sc[4][4];
            if (valid > 0) {
                // ---- S = Q K^T for this warp's four blocks of 8 keys
                const uint32_t kt = sK + st * kTileB;
#pragma unroll
                for (int nb = 0; nb < 4; ++nb) {
                    sc[nb][0] = sc[nb][1] = sc[nb][2] = sc[nb][3] = 0.f;
                    const int key = key_w + nb * 8 + (lane & 7);
#pragma unroll
                    for (int c4 = 0; c4 < D / 32; ++c4) {  // 4 d-chunks of 8 per ldmatrix.x4 = two k-steps
                        const int chunk = c4 * 4 + (lane >> 3);
                        const uint32_t addr = kt + lay.key(key) + (chunk >> 3) * lay.block + (((chunk & 7) ^ (key & 7)) << 4);
                        uint32_t b0, b1, b2, b3;
                        ldsm_x4(addr, b0, b1, b2, b3);
                        if (std::is_same<T, __nv_bfloat16>::value) {
                            mma_16816_bf16(sc[nb], qa[2 * c4], b0, b1);
                            mma_16816_bf16(sc[nb], qa[2 * c4 + 1], b2, b3);
                        } else {
                            mma_16816(sc[nb], qa[2 * c4], b0, b1);
                            mma_16816(sc[nb], qa[2 * c4 + 1], b2, b3);
                        }
                    }
                }
                // ---- mask, running max, probabilities
                // keys of this warp's 32 that the row may see: all valid ones, minus (several query
                // rows) those among the sequence's last that came after the row's token
                const int seen_lo = kMulti ? min(valid, len - hide_lo - (k_begin + t * kDecTile) - key_w) : valid;
                const int seen_hi = kMulti ? min(valid, len - hide_hi - (k_begin + t * kDecTile) - key_w) : valid;
                float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
                for (int nb = 0; nb < 4; ++nb) {
                    const int k0 = nb * 8 + 2 * t4;
                    if (k0 >= seen_lo) sc[nb][0] = -INFINITY;
                    if (k0 + 1 >= seen_lo) sc[nb][1] = -INFINITY;
                    if (k0 >= seen_hi) sc[nb][2] = -INFINITY;
                    if (k0 + 1 >= seen_hi) sc[nb][3] = -INFINITY;
                    mx_lo = fmaxf(mx_lo, fmaxf(sc[nb][0], sc[nb][1]));
                    mx_hi = fmaxf(mx_hi, fmaxf(sc[nb][2], sc[nb][3]));
                }
                mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
                mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
                mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
                mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
                // finite when key 0 of the warp is visible (always with one query row; an earlier
                // token of several may see none of the warp's keys: its state then stays empty)
                const float mn_lo = fmaxf(lower ? dec_lowered(m_lo, top_lo, p.ref_drop) : m_lo, mx_lo);
                const float mn_hi = fmaxf(lower ? dec_lowered(m_hi, top_hi, p.ref_drop) : m_hi, mx_hi);
                const float a_lo = (m_lo == -INFINITY) ? 0.f : fast_exp2((m_lo - mn_lo) * p.scale_log2);
                const float a_hi = (m_hi == -INFINITY) ? 0.f : fast_exp2((m_hi - mn_hi) * p.scale_log2);
                m_lo = mn_lo;
                m_hi = mn_hi;
                const float nm_lo = (mn_lo == -INFINITY) ? 0.f : -mn_lo * p.scale_log2;
                const float nm_hi = (mn_hi == -INFINITY) ? 0.f : -mn_hi * p.scale_log2;
                float s_lo = 0.f, s_hi = 0.f;
#pragma unroll
                for (int nb = 0; nb < 4; ++nb) {
                    const int k0 = nb * 8 + 2 * t4;
                    sc[nb][0] = (k0 < seen_lo) ? fast_exp2(fmaf(sc[nb][0], p.scale_log2, nm_lo)) : 0.f;
                    sc[nb][1] = (k0 + 1 < seen_lo) ? fast_exp2(fmaf(sc[nb][1], p.scale_log2, nm_lo)) : 0.f;
                    sc[nb][2] = (k0 < seen_hi) ? fast_exp2(fmaf(sc[nb][2], p.scale_log2, nm_hi)) : 0.f;
                    sc[nb][3] = (k0 + 1 < seen_hi) ? fast_exp2(fmaf(sc[nb][3], p.scale_log2, nm_hi)) : 0.f;
                    s_lo += sc[nb][0] + sc[nb][1];
                    s_hi += sc[nb][2] + sc[nb][3];
                }
                l_lo = l_lo * a_lo + s_lo;  // per-thread partial of the row sum (the quad is summed at the end)
                l_hi = l_hi * a_hi + s_hi;
#pragma unroll
                for (int i = 0; i < D / 8; ++i) {
                    o[i][0] *= a_lo;
                    o[i][1] *= a_lo;
                    o[i][2] *= a_hi;
                    o[i][3] *= a_hi;
                }
            }
            ok = mbar_wait(smem_u32(&bars[kStages + st]), parity, &abort_flag, 21);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            if (valid > 0) {
                const uint32_t vt = sV + st * kTileB;
                if (valid < 32) {
                    // rows past the sequence may hold NaN bits: zero them (0 * NaN would poison O)
                    for (int i = lane; i < (32 - valid) * (D / 8); i += 32) {
                        const int key = key_w + valid + i / (D / 8), ch = i % (D / 8);
                        const uint32_t addr = vt + lay.key(key) + (ch >> 3) * lay.block + (((ch & 7) ^ (key & 7)) << 4);
                        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0u) : "memory");
                    }
                    __syncwarp();
                }
                // ---- O += P V: two k-steps of 16 keys, D / 8 blocks of 8 output columns
#pragma unroll
                for (int k2 = 0; k2 < 2; ++k2) {
                    uint32_t pa[4];
                    pa[0] = pack2<T>(sc[2 * k2][0], sc[2 * k2][1]);
                    pa[1] = pack2<T>(sc[2 * k2][2], sc[2 * k2][3]);
                    pa[2] = pack2<T>(sc[2 * k2 + 1][0], sc[2 * k2 + 1][1]);
                    pa[3] = pack2<T>(sc[2 * k2 + 1][2], sc[2 * k2 + 1][3]);
                    const int key = key_w + k2 * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
                    for (int n2 = 0; n2 < D / 16; ++n2) {  // two output blocks per ldmatrix.x4.trans
                        const int ch = n2 * 2 + (lane >> 4);
                        const uint32_t addr = vt + lay.key(key) + (ch >> 3) * lay.block + (((ch & 7) ^ (key & 7)) << 4);
                        uint32_t b0, b1, b2, b3;
                        ldsm_x4_trans(addr, b0, b1, b2, b3);
                        if (std::is_same<T, __nv_bfloat16>::value) {
                            mma_16816_bf16(o[2 * n2], pa, b0, b1);
                            mma_16816_bf16(o[2 * n2 + 1], pa, b2, b3);
                        } else {
                            mma_16816(o[2 * n2], pa, b0, b1);
                            mma_16816(o[2 * n2 + 1], pa, b2, b3);
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars[2 * kStages + st]));
        }

        // ---- merge the four warps' states and write this chunk's partial result
        // (all tiles this CTA requested have been consumed by every warp before the barrier below,
        // so the ring can be reused as the merge buffer)
        l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
        l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
        l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
        l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (ok) {
#pragma unroll
            for (int i = 0; i < D / 8; ++i) {
                const int col = i * 8 + 2 * t4;
                *reinterpret_cast<float2*>(&mo[(warp * 16 + g) * D + col]) = make_float2(o[i][0], o[i][1]);
                *reinterpret_cast<float2*>(&mo[(warp * 16 + g + 8) * D + col]) = make_float2(o[i][2], o[i][3]);
            }
            if (t4 == 0) {
                ml[(warp * 16 + g) * 2] = m_lo;
                ml[(warp * 16 + g) * 2 + 1] = l_lo;
                ml[(warp * 16 + g + 8) * 2] = m_hi;
                ml[(warp * 16 + g + 8) * 2 + 1] = l_hi;
            }
        }
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        settle_if(!ok);
        if (ok) {
            // a thread owns four output columns, so 512 / D rows go at a time
            const int col = 4 * (tid % (D / 4));
            for (int r = tid / (D / 4); r < G; r += 512 / D) {
                float lse;
                const float4 out = dec_warp_merge<D>(mo, ml, r, col, p.scale_log2, 1.f, lse);
                if (kMode == kDecCluster) {
                    *reinterpret_cast<float4*>(&part[r * D + col]) = out;
                    if (col == 0) part_lse[r] = lse;
                } else if (p.o_final != nullptr) {   // the only chunk: this is the result
                    dec_store4<T>(p.o_final, row_index(r) * D + col, out);
                    if (col == 0 && p.lse_final) p.lse_final[lse_index(r)] = lse;
                } else {
                    const long long slot = part_index(r);
                    *reinterpret_cast<float4*>(&p.o_part[slot * D + col]) = out;
                    if (col == 0) p.lse_part[slot] = lse;
                }
            }
        }
    }
    if constexpr (kMode == kDecCluster) {
        const int n_live = (len + p.chunk - 1) / p.chunk;
        dec_cluster_merge<D>(part, part_lse, G, c, n_live, tid, [&](int r, int col, const float4& out, float lse) {
            dec_store4<T>(p.o_final, row_index(r) * D + col, out);
            if (col == 0 && p.lse_final) p.lse_final[lse_index(r)] = lse;
        });
    }
}

// Merge of the per-chunk partials (rowmax/rowsum recurrence applied across chunks):
//   M = max_c LSE_c, w_c = exp(LSE_c - M), O = sum_c w_c O_c / sum_c w_c, LSE = M + ln sum_c w_c.
// grid: B * Sq * Hq blocks of D threads (row = (b, token, head)), thread t owns output dim t.
template <typename T, int D = 128, bool kBalanced = false>
__global__ void __launch_bounds__(128)
fa_decode_combine_kernel(const DecodeParams p, T* o, float* lse) {
    const int bh = blockIdx.x;
    const int b = bh / (p.Hq * p.Sq);
    // lse is [B,Hq,Sq]
    const long long lse_at = ((long long)b * p.Hq + bh % p.Hq) * p.Sq + (bh / p.Hq) % p.Sq;
    const int tid = threadIdx.x;
    // The split kernel's partial results are complete and visible from here on, and so is what came before it.  (The
    // lengths too: that every CTA of the split kernel has waited for whoever wrote them orders those CTAs, not this kernel.)
    grid_dep_wait();
    int nc;
    long long at = (long long)bh * p.n_chunks, step = 1;   // this row's first partial result, and how far the next one is
    if constexpr (kBalanced) {
        const DecBalance bal(p, tid & 31);
        const int first = __shfl_sync(0xffffffffu, bal.first, b);
        nc = __shfl_sync(0xffffffffu, bal.count, b);
        step = (long long)p.Sq * p.Hq;
        at = bh + (first - b) * step;
    } else {
        const int len = max(0, min(p.seqlens[b], p.Smax));
        nc = (len + p.chunk - 1) / p.chunk;
    }
    const float* lp = p.lse_part + at;
    const float* op = p.o_part + at * D;
    // One pass, some chunks at a time, whose loads are all on their way together; the weights are relative to the
    // largest log-sum-exp so far.  (A pass for the maximum and one for the sums, a chunk at a time, waits for L2 twice
    // per chunk: 4 sequences of up to 11139 keys, 2 tokens, 32/8 heads, 17.8 -> 17.3 us, 2 of up to 23723, 64/8 heads, 32.9 -> 32.2, 12 of up
    // to 5861, 5 heads, 27.5 -> 27.0.  Two at a time where there are no more: with eight 64 of up to 3371, 4 tokens, 89.5 -> 90.7.)
    float M = -INFINITY, wsum = 0.f, acc = 0.f;
    auto merge = [&](auto chunks) {
        constexpr int kN = decltype(chunks)::value;
        for (int c0 = 0; c0 < nc; c0 += kN) {
            float l[kN], v[kN], m = M;
#pragma unroll
            for (int i = 0; i < kN; ++i) {
                const bool live = c0 + i < nc;
                l[i] = live ? lp[(c0 + i) * step] : -INFINITY;
                v[i] = live ? op[(c0 + i) * step * D + tid] : 0.f;
            }
#pragma unroll
            for (int i = 0; i < kN; ++i) m = fmaxf(m, l[i]);
            const float ref = m == -INFINITY ? 0.f : m;
            const float keep = __expf(M - ref);
            wsum *= keep;
            acc *= keep;
            M = m;
#pragma unroll
            for (int i = 0; i < kN; ++i) {
                if (l[i] != -INFINITY) {   // (a chunk that the token sees nothing of; a NaN gets through)
                    const float w = __expf(l[i] - ref);
                    wsum += w;
                    acc = fmaf(w, v[i], acc);
                }
            }
        }
    };
    if (p.n_chunks <= 2) merge(std::integral_constant<int, 2>());
    else merge(std::integral_constant<int, 8>());
    if (wsum == 0.f) {   // no keys, or (several query rows) a token that sees none
        o[(long long)bh * D + tid] = T(0.f);
        if (lse && tid == 0) lse[lse_at] = -INFINITY;
        return;
    }
    o[(long long)bh * D + tid] = T(acc / wsum);
    if (lse && tid == 0) lse[lse_at] = M + logf(wsum);
}

}  // namespace fa
