// Prefill forward, ping-pong variant.
//
// A persistent CTA (one per SM, 384 threads) takes work items, some dealt to it and some claimed (see
// PpSource); an item is one 128-row query tile of one (batch, head).  The kv steps of the CTA are numbered g = 0, 1, 2, ...
// across items, and everything a step needs is double-buffered on the parity of g:
//   tensor memory : O [0,128)   S_0 [128,256)  S_1 [256,384)  P_0 [384,448)  P_1 [448,512)
//   warpgroup g&1 : softmax of step g, one thread per query row: reads S_{g&1}, keeps its part
//                   of the row sum, writes P (16-bit, packed) to P_{g&1}.
//   warp 8        : one thread issues S_{g&1} = Q K_g^T for every step, as soon as K_g has
//                   landed and the softmax of step g-2 has read its scores out of the buffer.
//   warp 10       : one thread issues O += P_{g&1} V_g for every step, as soon as P is written.
//   warp 9 / 11   : one thread each issues the TMA loads of Q and K / of V (separate rings, as
//                   K is consumed about two steps ahead of V); the second stores the 16-bit outputs too.
// Because P has columns of its own, Q K^T of step g+1 and g+2 run on the tensor core while the
// softmax of step g is still at work: the tensor core never waits for a softmax of the same
// tile (the Cube/Vector overlap of Section 4.1 within one query tile), and the two warpgroups
// give the exponentials two steps of time per step of tensor work.
//
// The online-softmax recurrence (Appendix A) is carried from step to step through shared
// memory: the warpgroup of step g takes the reference max left by step g-1, decides whether its
// own row max moves it (only when it outgrew it by more than 2^8, see kRescaleThreshold),
// publishes the result for step g+1 right away, and, in the rare case that it moved, rescales O
// once O += P V of step g-1 has completed.  (Waiting for that hand-over costs nothing by itself: a form that
// took the reference to be the one its own last step left, and looked only at the step's end, was 6 % slower.)  Each warpgroup keeps the row sum of its own steps;
// the one that runs an item's last step adds the other's and writes O and LSE.
// Synchronisation is by mbarriers, and every wait on one is bounded (see mbar_wait); what the bound covers is this
// kernel alone, as every role waits for the end of the kernel before it, without a bound, ahead of its first
// wait for anything that follows from that (see PpTaker).  The form whose
// CTAs share a query tile merges behind cluster barriers and a named barrier, which are not: every
// thread reaches them, those of a CTA without work and of one that gave up a wait too, because a role
// that stops only leaves its loop.
//
// The times beside a step below are of the code before and after that step, in turn on one box, whose clock
// and power state differ from box to box; steps measured apart do not multiply to the whole.  8 x 32 x 512
// from the first step of "P stored in one piece" to here, in turn: 43.9 -> 41.4 us.
#pragma once

#include <type_traits>

#include "prefill_pipelined.cuh"

namespace fa {

constexpr int kPpNK = 3;          // K ring slots
constexpr int kPpNV = 2;          // V ring slots: those of the steps' parities
constexpr int kPpQBufs = 2;
constexpr int kPpSlots = 4;       // work items the Q/K loader may be ahead of the slowest role
static_assert((kPpQBufs + kPpNK + kPpNV) * kTileBytes + 3072 <= 232448, "shared memory budget");

// What changes with FP8 e4m3 operands (kF8; Appendix D.2 evaluates the operator with 8-bit
// operands): a tile of 128 rows x 128 bytes is one swizzled TMA box of 16 KiB (a V slot keeps its
// 32 KiB, because the 16-bit output tile is staged there); one MMA covers 32 elements of the
// contraction, so a product takes four instead of eight; the probabilities are rounded to e4m3
// four to a 32-bit column of tensor memory, times kP8Scale so that they use the format's range:
// with the reference max at most 2^kP8Threshold behind the row max they stay below 2^8 < 448.
// Head dimension 64 (D; 16-bit operands only) has the same byte layout: a row of a Q, K or V tile
// is 64 elements = 128 bytes, one box; Q K^T then contracts over four MMAs of 16 elements, P V is
// eight MMAs of 16 keys with N = 64, and O takes 64 columns of tensor memory.
template <bool kF8, int D = 128>
struct PpOperands {
    static_assert(D == 128 || (D == 64 && !kF8), "head dimension 128, or 64 with 16-bit operands");
    static constexpr bool kOneBox = kF8 || D == 64;                     // a tile row is 128 bytes
    static constexpr int kKvSlotBytes = kOneBox ? 16384 : kTileBytes;   // one K ring slot, and the bytes of a K or V tile
    static constexpr int kVSlotBytes = D == 64 ? 16384 : kTileBytes;    // one V ring slot: a V tile, later an output tile
    static constexpr int kQBytes = kOneBox ? 16384 : kTileBytes;        // bytes a Q load delivers
    static constexpr int kQBufBytes = kF8 ? 16384 : kTileBytes;         // one Q buffer (d = 64 with 16 KiB: 512 x 12 x 128 66.4 -> 66.8 us)
    static constexpr int kSmem = kPpQBufs * kQBufBytes + kPpNK * kKvSlotBytes + kPpNV * kVSlotBytes;   // 224 KiB; 8-bit and d = 64 144
    static constexpr int kSteps = kOneBox ? 4 : 8;                      // MMAs of Q K^T (32 bytes of every row each)
    static constexpr int kPvSteps = kF8 ? 4 : 8;                        // MMAs of P V (32 or 16 keys each)
    static constexpr int kPCols = kF8 ? 8 : 16;                         // tensor-memory columns of 32 probabilities
};
constexpr float kP8Threshold = 4.0f;   // log2 units: how far the row max may outgrow the reference (FP8)
constexpr float kP8ScaleLog2 = 4.0f;   // log2 of the factor on the FP8 probabilities

// ---- barriers: indices into one array
namespace ppb {
constexpr int q_full = 0;                       // [2]  TMA -> S thread
constexpr int q_empty = 2;                      // [2]  S thread (commit) -> loader
constexpr int k_full = 4;                       // [NK]
constexpr int k_empty = k_full + kPpNK;         // [NK]
constexpr int v_full = k_empty + kPpNK;         // [NV]
constexpr int s_full = v_full + kPpNV;          // [2]  S thread (commit) -> softmax
constexpr int pv_done = s_full + 2;             // [2]  PV thread (commit) -> softmax, and -> V loader: V of step g is in slot g & 1
constexpr int o_final = pv_done + 2;            // [2]  PV thread (commit) -> epilogue, by item parity
constexpr int item_full = o_final + 2;          // [kPpSlots] Q/K loader -> every other role: a work item is in the slot
constexpr int item_empty = item_full + kPpSlots;   // [kPpSlots] back: three single-thread roles and eight softmax warps
constexpr int o_staged = item_empty + kPpSlots; // [2]  by item parity, 16-bit output: the four epilogue warps (count 4) -> V loader, which stores it
constexpr int claim = o_staged + 2;             // [1]  answer to a claim of work (cluster launch control) -> Q/K loader
// barriers every thread of a softmax warpgroup arrives on (count 128)
constexpr int p_full = claim + 1;               // [2]  softmax -> PV thread
constexpr int m_ready = p_full + 2;             // [2]  softmax of step g -> softmax of step g+1 (reference max
                                                //      published) and -> S thread (scores read out of S_{g&1})
constexpr int l_pub = m_ready + 2;              // [2]  softmax of an item's last-but-one step -> of its last step
constexpr int o_free = l_pub + 2;               // [1]  epilogue -> PV thread
constexpr int count = o_free + 1;
}  // namespace ppb

struct __align__(16) PpItem {
    int q0, n;      // first query row of the tile, kv tiles it visits (0: no further item)
    int b, h, hk;
    int j0;         // the first of those kv tiles (not 0 only where CTAs share a query tile)
    // packed variable-length batches only: first row of the sequence in q/o and in k/v, and
    // the sequence's own lengths
    int q_base, k_base, Sq, Skv;
    int page0;   // paged K/V: the sequence's first table entry (-1 for a sequence without keys)
};

struct PpStatic {
    uint64_t bars[ppb::count];
    uint32_t tmem_holder;
    uint32_t abort_flag;
    float m_xch[2][128];   // [warpgroup][row]: reference max after that warpgroup's latest step
    float l_xch[2][128];   // [item parity][row]: row sum of the warpgroup that does not run the last step
    PpItem items[kPpSlots];    // decoded work items, written by the Q/K loader (see PpSource)
    uint4 claim_answer;
};
constexpr int kPpStaticBytes = 3072;   // the static shared memory of the kernels: PpStatic and padding
static_assert(sizeof(PpStatic) <= kPpStaticBytes && sizeof(PpStatic) > kPpStaticBytes - 1024, "static shared state fills 3 KiB");

// Work item `idx`.  The query tiles of a head are taken in classes of C = 2^cls_log2 consecutive
// tiles, the class of the last (longest) tiles first; inside a class the items go head by head,
// a head's tiles longest first.  With the items dealt to the CTAs round by round, a round then
// works on about gridDim.x / C heads, whose K and V stay in L2 while the C tiles of each head
// read them, and the rounds still get shorter and shorter items, which keeps the deal
// balanced (the launcher picks C from the K/V bytes of a head, see launch_pingpong).
// C >= n_qtiles is the plain head-by-head order used for very long sequences.
__device__ __forceinline__ void pp_class_order(const FwdParams& p, int idx, int& bh, int& qt) {
    int c, rem;  // class, index inside the class
    p.by_class.divmod(idx, c, rem);
    const int first = c << p.cls_log2;  // tiles in the classes before this one
    int j;
    if (p.n_qtiles - first >= (1 << p.cls_log2)) {
        bh = rem >> p.cls_log2;
        j = rem & ((1 << p.cls_log2) - 1);
    } else {
        p.by_lastcls.divmod(rem, bh, j);
    }
    qt = p.n_qtiles - 1 - first - j;
}

// The work item that is query tile qt of head h of batch entry b.
// kVarlen: the sequence's lengths come from the prefix sums; n == 0 marks an item past the end
// of its sequence (nobody works on it), and a live item visits at least one kv tile (so that
// rows without any visible key are still written, as zeros).
template <bool kVarlen>
__device__ __forceinline__ PpItem pp_decode_item(const FwdParams& p, int b, int h, int qt) {
    PpItem it;
    it.b = b;
    it.h = h;
    it.hk = p.by_group.div(it.h);
    it.j0 = 0;
    it.q0 = qt * kTile;
    if (kVarlen) {
        it.q_base = p.cu_q[it.b];
        it.Sq = p.cu_q[it.b + 1] - it.q_base;
        if (p.block_table) {   // paged K/V: the keys are reached through the table
            it.k_base = 0;
            // the first table entry is fetched together with the lengths, so that a loader does
            // not start an item with two dependent global loads (the entry exists for every
            // sequence; its value is ignored when the sequence has no keys)
            const int first_page = p.block_table[(long long)it.b * p.table_stride];
            it.Skv = p.seqlens_k[it.b];
            it.page0 = it.Skv > 0 ? first_page : -1;
        } else {
            it.k_base = p.cu_k[it.b];
            it.Skv = p.cu_k[it.b + 1] - it.k_base;
        }
        it.n = (it.q0 < it.Sq) ? max(1, kv_tiles_for(it.q0, kTile, it.Sq, it.Skv, p.causal)) : 0;
    } else {
        it.n = kv_tiles_for(it.q0, kTile, p.Sq, p.Skv, p.causal);
    }
    return it;
}

// The share of this CTA where the CTAs of a cluster divide the kv tiles of one query tile: item
// blockIdx.x / p.split of the class order, kv tiles [j0, j0 + n).  Returns n (0: nothing to do).
__device__ __forceinline__ int pp_split_first(int n, int split, int rank) { return n * rank / split; }
__device__ __forceinline__ int pp_split_item(const FwdParams& p, PpItem& it) {
    const int idx = (int)blockIdx.x / p.split, rank = (int)blockIdx.x - idx * p.split;
    int bh, qt, b, h;
    pp_class_order(p, idx, bh, qt);
    p.by_hq.divmod(bh, b, h);
    it = pp_decode_item<false>(p, b, h, qt);
    it.j0 = pp_split_first(it.n, p.split, rank);
    it.n = pp_split_first(it.n, p.split, rank + 1) - it.j0;
    return it.n;
}

// The places of the item list that a CTA takes: its share.  The first deal_ctas CTAs of the grid have
// deal_rounds places each, dealt in alternating direction; every CTA after them has one place.
// A CTA walks its own share and then the share of every CTA whose launch it has cancelled.  That can be
// any CTA that has not started, one of the dealing ones included: while a kernel of another stream
// holds some SMs, CTAs that found one may be through with their deal before the others get theirs.
struct PpWalk {
    int deal_ctas, deal_rounds;
    int place = 0, step = 0;   // the next place, and how far the one after it is
    int left = 0;              // places left

    __host__ __device__ __forceinline__ bool used_up() const { return left == 0; }
    // The next place (only if the share is not used up).
    __host__ __device__ __forceinline__ int next() {
        const int at = place;
        place += step;
        step = 2 * deal_ctas - step;   // (a round that goes up is followed by one that goes down)
        --left;
        return at;
    }
    // Starts on the share of a CTA.
    __host__ __device__ __forceinline__ void take(int cta) {
        const bool dealing = cta < deal_ctas;
        place = dealing ? cta : deal_rounds * deal_ctas + cta - deal_ctas;
        step = 2 * (deal_ctas - cta) - 1;
        left = dealing ? deal_rounds : 1;
    }
};

// Where a CTA's work items come from.  One thread, the Q/K loader, decides and decodes them and
// hands them to the other roles through a ring of slots in shared memory (PpItem, item_full,
// item_empty): an item costs the others one barrier wait and one or two 16-byte reads instead of
// the divisions and, in packed batches, the dependent global loads of the decoding.
//
// The list is dealt to the first p.deal_ctas CTAs for its first p.deal_rounds rounds and claimed from
// there on (p.claim_items): the grid has one CTA for every remaining item on top of the dealing ones,
// and a running CTA takes over the share (see PpWalk) of a CTA that has not started through
// cluster launch control when it requests the last keys of the last item it has.  The launcher says
// how much of which list is dealt and why.
//
// Very long sequences (rounds_per_head > 0; one head's K and V no longer fit in L2) are all dealt,
// head by head, and every head takes a whole number of rounds of the grid: in round r
// of a head CTA b takes the head's (r * gridDim.x + b)-th longest tile -- b counted from the other
// end in every second round, and the other way around for every second head -- and nothing if the
// head has no such tile (only in a head's last round, whose items are its shortest).  The CTAs of a
// round then all walk the same head's keys from the first on, a few dozen tiles apart at most, and
// stay together from head to head, so a K or V tile is fetched from HBM once per round and
// found in L2 by everyone else.  (Without the padding a round straddles two heads, the CTAs
// that get the next head's longest tiles fall a thousand tiles behind the others, and the
// groups, each walking the head on its own, fetch everything several times.)  A cooperative
// launch (the fused projection) is all dealt as well.
//
// Packed batches: the list goes sequence by sequence and head by head, a head's tiles longest
// first.  Sequence s takes the places from floor(cu_q[s] / 128) + s on, times Hq, which leaves
// it at least its number of tiles and at most one more per head: the host can size the grid
// without knowing the lengths, and a place past a sequence's end is passed over.  Where it is not more,
// every sequence has the longest one's number of places instead (p.fixed_places): chunks of 512 new
// tokens have four tiles, for which the other count keeps five places, and a claim that finds an empty
// place is a round trip for nothing (10 chunks over up to 5300 keys, 32 heads: 365 -> 362 us; 20 of up to 666, 85.6 -> 83.7).
template <bool kVarlen>
struct PpSource {
    const FwdParams& p;
    int total_items;
    uint32_t claim_bar, answer;      // shared-memory addresses
    volatile uint32_t* abort_flag;
    PpWalk walk;
    int round = -1;                  // (rounds_per_head) rounds taken so far, less one
    int claims = 0;                  // claims answered
    bool pending = false;            // a claim is on its way
    int seq = 0;                     // packed batches: sequence of the last item

    // Asks for an item (at most once).
    __device__ __forceinline__ void request() {
        if (p.claim_items && !pending) {
            fence_proxy_async_smem();   // the last answer has been read
            mbar_expect_tx(claim_bar, 16);
            clc_request(answer, claim_bar);
            pending = true;
        }
    }
    // The same ahead of time, if the next item is a claimed one.
    __device__ __forceinline__ void request_next() {
        if (walk.used_up()) request();
    }
    __device__ __forceinline__ int place_of(int s) const { return (p.cu_q[s] >> 7) + s; }
    __device__ __forceinline__ void packed_place(int idx, int& b, int& h, int& qt) {
        int v, rem;
        if (p.fixed_places) {
            p.by_qtiles.divmod(idx, v, rem);
            p.by_hq.divmod(v, b, h);
            qt = p.n_qtiles - 1 - rem;
            return;
        }
        p.by_hq.divmod(idx, v, rem);
        // the last sequence that starts at or before place v: items nearly always come in rising order
        int lo = place_of(seq) <= v ? seq : 0, hi = p.B - 1;
        for (int k = 0; lo < hi && k < 4; ++k) {
            if (place_of(lo + 1) > v) hi = lo;
            else ++lo;
        }
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (place_of(mid) <= v) lo = mid;
            else hi = mid - 1;
        }
        seq = b = lo;
        const int first = place_of(lo);
        const int tiles = max(1, place_of(lo + 1) - first);
        rem = idx - first * p.Hq;
        h = rem < 0 ? -1 : rem / tiles;   // (a place before the first sequence, if cu_q[0] > 0)
        qt = tiles - 1 - (rem - h * tiles);
    }
    __device__ __forceinline__ bool next(PpItem& it) {
        if (!kVarlen && p.split > 1) {   // one item per cluster
            ++round;
            return round == 0 && pp_split_item(p, it) > 0;
        }
        for (;;) {
            ++round;
            int b, h, qt;
            if (!kVarlen && p.rounds_per_head > 0) {
                int bh, r;
                p.by_rph.divmod(round, bh, r);
                if (bh >= p.B * p.Hq) return false;
                const int g = gridDim.x, x = blockIdx.x;
                const int j = r * g + (((r + bh) & 1) ? (g - 1 - x) : x);
                if (j >= p.n_qtiles) continue;
                p.by_hq.divmod(bh, b, h);
                qt = p.n_qtiles - 1 - j;
            } else {
                if (walk.used_up()) {
                    if (!p.claim_items) return false;
                    request();
                    if (!mbar_wait(claim_bar, claims & 1, abort_flag, 153)) return false;
                    ++claims;
                    pending = false;
                    const int cta = clc_answer(answer);
                    if (cta < 0) return false;
                    walk.take(cta);
                }
                const int idx = walk.next();
                if (idx >= total_items) return false;   // (a list that is all dealt)
                if (kVarlen) {
                    packed_place(idx, b, h, qt);
                    if (h < 0 || h >= p.Hq || qt < 0 || qt >= p.n_qtiles) continue;
                } else {
                    int bh;
                    pp_class_order(p, idx, bh, qt);
                    p.by_hq.divmod(bh, b, h);
                }
            }
            it = pp_decode_item<kVarlen>(p, b, h, qt);
            if (!kVarlen || it.n > 0) return true;
        }
    }
};

__device__ __forceinline__ uint32_t pp_bar(uint32_t bar0, int i) { return bar0 + 8 * i; }

// The other roles' end of the ring: the ord-th item, read by a single thread, which hands the slot
// back at once.  False at the end of the list or after a wait that gave up.
// The kernel before this one in the stream may still run when the first item is taken.  A dense call's is decoded
// from the parameters alone, so the role first runs up to here, on cold instruction lines, and then waits for that
// kernel; a packed batch's needs global memory.  The wait belongs to every role, not only to the loading
// ones: what follows the item follows from the loads, and a bounded wait for that would count the time that
// kernel takes, which has no bound (a collective of another library that releases its dependents and
// waits for a peer).  (It costs next to nothing: with the loaders waiting alone 1 x 2 x 512 took 7.2 us, like this
// 7.1; few query tiles over many keys 14.6 / 14.7; 8 x 32 x 512 41.8 / 42.0.)
template <bool kVarlen>
struct PpTaker {
    const PpItem* items;
    uint32_t bar0;
    volatile uint32_t* abort_flag;
    int ord = -1;
    __device__ __forceinline__ bool next(PpItem& it, unsigned int where) {
        ++ord;
        const int slot = ord & (kPpSlots - 1);
        if (kVarlen && ord == 0) grid_dep_wait();
        if (!mbar_wait(pp_bar(bar0, ppb::item_full + slot), (ord / kPpSlots) & 1, abort_flag, where)) return false;
        it = items[slot];
        mbar_arrive(pp_bar(bar0, ppb::item_empty + slot));
        if (!kVarlen && ord == 0) grid_dep_wait();
        return it.n > 0;
    }
};

// Row max of 128 raw scores.
__device__ __forceinline__ float pp_row_max(const uint32_t (&s)[128]) {
    float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
    for (int i = 0; i < 128; i += 8) {
        m0 = max3(m0, __uint_as_float(s[i]), __uint_as_float(s[i + 1]));
        m1 = max3(m1, __uint_as_float(s[i + 2]), __uint_as_float(s[i + 3]));
        m2 = max3(m2, __uint_as_float(s[i + 4]), __uint_as_float(s[i + 5]));
        m3 = max3(m3, __uint_as_float(s[i + 6]), __uint_as_float(s[i + 7]));
    }
    return fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
}

// exp2(s * scale_log2 + neg_ms) of 32 scores -> 16 packed 16-bit pairs; adds them to (la, lb).
template <typename T, bool kF8>
__device__ __forceinline__ void pp_exp_chunk(const uint32_t (&s)[128], int c, uint64_t sc2, uint64_t nm2,
                                             uint64_t& la, uint64_t& lb, uint32_t (&pk)[PpOperands<kF8>::kPCols]) {
#pragma unroll
    for (int i = 0; i < 32; i += 8) {
        const int e = c * 32 + i;
        float pv[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint64_t x01 =
                f2_fma(f2_pack(__uint_as_float(s[e + 2 * q]), __uint_as_float(s[e + 2 * q + 1])), sc2, nm2);
            float x0, x1;
            f2_unpack(x01, x0, x1);
            pv[2 * q] = fast_exp2(x0);
            pv[2 * q + 1] = fast_exp2(x1);
        }
        la = f2_add(la, f2_pack(pv[0], pv[1]));
        lb = f2_add(lb, f2_pack(pv[2], pv[3]));
        la = f2_add(la, f2_pack(pv[4], pv[5]));
        lb = f2_add(lb, f2_pack(pv[6], pv[7]));
        if (kF8) {
            pk[i / 4] = pack4_e4m3(pv[0], pv[1], pv[2], pv[3]);
            pk[i / 4 + 1] = pack4_e4m3(pv[4], pv[5], pv[6], pv[7]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) pk[i / 2 + q] = pack2<T>(pv[2 * q], pv[2 * q + 1]);
        }
    }
}
template <bool kF8>
__device__ __forceinline__ void pp_store_p(uint32_t taddr, const uint32_t (&pk)[PpOperands<kF8>::kPCols]);
template <>
__device__ __forceinline__ void pp_store_p<false>(uint32_t taddr, const uint32_t (&pk)[16]) { tmem_st_x16(taddr, pk); }
template <>
__device__ __forceinline__ void pp_store_p<true>(uint32_t taddr, const uint32_t (&pk)[8]) { tmem_st_x8(taddr, pk); }

// Counter in global memory that one SM raises after its writes and another reads before its loads.
__device__ __forceinline__ unsigned int ld_acquire_gpu(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_gpu_add(unsigned int* p, unsigned int v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Ring cursor: slot and phase parity of the g-th entry of a ring of N slots.
template <int N>
struct PpRing {
    uint32_t slot = 0, par = 0;
    __device__ __forceinline__ void next() {
        if (++slot == N) {
            slot = 0;
            par ^= 1;
        }
    }
};

// The thread that issues S = Q K^T of every step.
template <typename T, bool kVarlen, bool kF8, int D>
__device__ __forceinline__ void pp_run_s(uint32_t bar0, uint32_t sQ, uint32_t sK, uint32_t tmem, const PpItem* slots,
                                         volatile uint32_t* abort_flag) {
    constexpr bool kBf16 = std::is_same<T, __nv_bfloat16>::value;
    constexpr uint32_t idesc = kF8 ? instr_desc_e4m3(128, 128, false, false) : instr_desc_f16(kBf16, 128, 128, false, false);
    using Op = PpOperands<kF8, D>;
    uint32_t g = 0;
    PpRing<kPpNK> ring;
    PpTaker<kVarlen> items{slots, bar0, abort_flag};
    PpItem it;
    while (items.next(it, 133)) {
        const int ord = items.ord;
        const uint32_t qb = ord & 1;
        if (!mbar_wait(pp_bar(bar0, ppb::q_full + qb), (ord >> 1) & 1, abort_flag, 130)) return;
        const uint32_t a_lo = desc_lo(sQ + qb * Op::kQBufBytes, 16);
        for (int j = 0; j < it.n; ++j, ++g, ring.next()) {
            const uint32_t buf = g & 1;
            if (!mbar_wait(pp_bar(bar0, ppb::k_full + ring.slot), ring.par, abort_flag, 131)) return;
            // the softmax of step g-2 has read its scores out of this buffer (it says so together
            // with its reference max)
            if (g >= 2 && !mbar_wait(pp_bar(bar0, ppb::m_ready + buf), ((g >> 1) - 1) & 1, abort_flag, 132)) return;
            tc_fence_after();
            const uint32_t b_lo = desc_lo(sK + ring.slot * Op::kKvSlotBytes, 16);
#pragma unroll
            for (int ks = 0; ks < Op::kSteps; ++ks) {
                // one MMA takes 32 bytes of every row: 16 16-bit elements (a row of d = 128 is two
                // 128-byte boxes, one of d = 64 a single one) or 32 8-bit ones (one box)
                const uint32_t koff = Op::kOneBox ? (uint32_t)(ks * 32) >> 4 : ((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4;
                if (kF8) mma_ss_lo_f8(tmem + 128 + 128 * buf, a_lo + koff, b_lo + koff, idesc, ks > 0 ? 1u : 0u);
                else mma_ss_lo(tmem + 128 + 128 * buf, a_lo + koff, b_lo + koff, idesc, ks > 0 ? 1u : 0u);
            }
            mma_commit(pp_bar(bar0, ppb::s_full + buf));
            mma_commit(pp_bar(bar0, ppb::k_empty + ring.slot));
            if (j == it.n - 1) mma_commit(pp_bar(bar0, ppb::q_empty + qb));
        }
    }
}

// The thread that issues O += P V of every step.
template <typename T, bool kVarlen, bool kF8, int D>
__device__ __forceinline__ void pp_run_pv(uint32_t bar0, uint32_t sV, uint32_t tmem, const PpItem* slots,
                                          volatile uint32_t* abort_flag) {
    constexpr bool kBf16 = std::is_same<T, __nv_bfloat16>::value;
    constexpr uint32_t idesc = kF8 ? instr_desc_e4m3(128, 128, false, true) : instr_desc_f16(kBf16, 128, D, false, true);
    using Op = PpOperands<kF8, D>;
    uint32_t g = 0;
    PpRing<kPpNV> ring;
    PpTaker<kVarlen> items{slots, bar0, abort_flag};
    PpItem it;
    while (items.next(it, 143)) {
        const int ord = items.ord;
        for (int j = 0; j < it.n; ++j, ++g, ring.next()) {
            const uint32_t buf = g & 1;
            if (!mbar_wait(pp_bar(bar0, ppb::v_full + ring.slot), ring.par, abort_flag, 140)) return;
            // the previous item's epilogue has read O out of tensor memory
            if (j == 0 && ord > 0 && !mbar_wait(pp_bar(bar0, ppb::o_free), (ord - 1) & 1, abort_flag, 141)) return;
            if (!mbar_wait(pp_bar(bar0, ppb::p_full + buf), (g >> 1) & 1, abort_flag, 142)) return;
            tc_fence_after();
            // V is the N-major operand: a key is a row of d elements.  16-bit, d = 128: two 128-byte
            // column blocks kHalfBytes apart, 16 keys (2048 bytes) per MMA; d = 64: one block, the
            // same 16 keys per MMA; 8-bit: one block, 32 keys (4096 bytes) per MMA.  Either way an
            // MMA reads 8 columns of P.
            const uint32_t b_lo = desc_lo(sV + ring.slot * Op::kVSlotBytes, D == 64 ? 16 : kHalfBytes);
#pragma unroll
            for (int ks = 0; ks < Op::kPvSteps; ++ks) {
                if (kF8) mma_ts_lo_f8(tmem, tmem + 384 + 64 * buf + ks * 8, b_lo + ks * (4096 >> 4), idesc,
                                      (ks > 0) ? 1u : (j > 0 ? 1u : 0u));
                else mma_ts_lo(tmem, tmem + 384 + 64 * buf + ks * 8, b_lo + ks * (2048 >> 4), idesc,
                               (ks > 0) ? 1u : (j > 0 ? 1u : 0u));
            }
            mma_commit(pp_bar(bar0, ppb::pv_done + buf));
            if (j == it.n - 1) mma_commit(pp_bar(bar0, ppb::o_final + (ord & 1)));
        }
    }
}

// Paged K/V (packed batches only): kv tile j of sequence b lies in one page; its coordinates
// become (row inside the page, page).  The page of tile j + 1 is looked up before the loader
// waits for tile j's ring slot, so that the table read is off the path that refills a slot.
template <bool kVarlen>
__device__ __forceinline__ int pp_page_of(const FwdParams& p, int b, int j, int n, int Skv) {
    // a sequence without keys still runs one (fully masked) step; it has no table entry to read:
    // page -1 is outside the tensor map, so the loads of that step deliver zeros
    if (kVarlen && p.block_table != nullptr && Skv == 0) return -1;
    if (kVarlen && p.block_table != nullptr && j < n) {
        // (volatile: issued here, ahead of the wait that follows, not where the value is used)
        int page;
        asm volatile("ld.global.s32 %0, [%1];"
                     : "=r"(page)
                     : "l"(p.block_table + (long long)b * p.table_stride + p.by_tiles_per_page.div(j))
                     : "memory");
        return page;
    }
    return 0;
}
template <bool kVarlen>
__device__ __forceinline__ void pp_paged_tile(const FwdParams& p, int page, int j, int& row, int& slab) {
    if (kVarlen && p.block_table != nullptr) {
        slab = page;
        row = (j - p.by_tiles_per_page.div(j) * (int)p.by_tiles_per_page.d) * kTile;
    }
}

// The thread that picks the work items (see PpSource) and loads Q of every item and K of every step.  (Packed batches: the tensor maps
// have one batch entry that holds every sequence back to back.)
// One tile is one box: of d = 128 and 16 bits, both 64-element blocks of the rows (see encode_map_tile), otherwise
// rows of 128 bytes.  (Two boxes of 64 columns cost the loading thread and the TMA unit twice: 8 x 32 x 512 40.6 -> 40.1
// us, 32 packed prompts of 256 to 8192 tokens 4262 -> 4164, long sequences level.)
template <bool kOneBox>
__device__ __forceinline__ void pp_load_tile(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int h, int s0, int b,
                                             uint64_t policy) {
    if (kOneBox) tma_load_4d_hint(dst, tm, bar, 0, h, s0, b, policy);
    else tma_load_5d_hint(dst, tm, bar, 0, s0, 0, h, b, policy);
}

template <bool kVarlen, bool kF8, int D>
__device__ __forceinline__ void pp_run_load_qk(uint32_t bar0, uint32_t sQ, uint32_t sK, const CUtensorMap* tm_q,
                                               const CUtensorMap* tm_k, const FwdParams& p, int total_items, PpStatic& ss,
                                               volatile uint32_t* abort_flag) {
    tma_prefetch_desc(tm_q);
    tma_prefetch_desc(tm_k);
    const uint64_t pol_q = l2_policy_evict_first(), pol_kv = l2_policy_evict_last();
    PpRing<kPpNK> ring;
    PpSource<kVarlen> source{p, total_items, pp_bar(bar0, ppb::claim), smem_u32(&ss.claim_answer), abort_flag,
                             {p.deal_ctas, p.deal_rounds}};
    source.walk.take(blockIdx.x);
    // The kernel before this one has ended: from here on global memory may be read.  A dense call's first item
    // needs none: it is decoded, and the other roles take it, while that kernel may still run (see PpTaker).
    // (1 x 2 x 512 8.1 -> 7.0 us, calls on few query tiles 17.2 -> 15.8, 14.8 -> 13.6; calls that fill the device
    // level.)
    auto after_last_kernel = [&]() {
        grid_dep_wait();
        if (p.early_next) grid_dep_launch();
    };
    if (kVarlen) after_last_kernel();
    PpItem it;
    for (int ord = 0;; ++ord) {
        if (!source.next(it)) it.n = 0;   // no further item: the others are told so
        const int slot = ord & (kPpSlots - 1);
        if (!mbar_wait(pp_bar(bar0, ppb::item_empty + slot), ((ord / kPpSlots) & 1) ^ 1, abort_flag, 154)) return;
        ss.items[slot] = it;
        mbar_arrive(pp_bar(bar0, ppb::item_full + slot));
        if (!kVarlen && ord == 0) {
            after_last_kernel();
            if (*abort_flag) return;   // (a role did not get the item in time: nothing is loaded)
        }
        if (it.n == 0) return;
        const uint32_t qb = ord & 1;
        // passes at once the first time each buffer is used
        if (!mbar_wait(pp_bar(bar0, ppb::q_empty + qb), ((ord >> 1) & 1) ^ 1, abort_flag, 150)) return;
        mbar_expect_tx(pp_bar(bar0, ppb::q_full + qb), PpOperands<kF8, D>::kQBytes);
        pp_load_tile<PpOperands<kF8, D>::kOneBox>(sQ + qb * PpOperands<kF8, D>::kQBufBytes, tm_q, pp_bar(bar0, ppb::q_full + qb), it.h,
                       kVarlen ? it.q_base + it.q0 : it.q0, kVarlen ? 0 : it.b, pol_q);
        int page = (kVarlen && p.block_table != nullptr) ? it.page0 : 0;
        for (int j = 0; j < it.n; ++j, ring.next()) {
            const int page_next = pp_page_of<kVarlen>(p, it.b, j + 1, it.n, it.Skv);
            if (j == it.n - 1) source.request_next();
            if (!mbar_wait(pp_bar(bar0, ppb::k_empty + ring.slot), ring.par ^ 1, abort_flag, 151)) return;
            mbar_expect_tx(pp_bar(bar0, ppb::k_full + ring.slot), PpOperands<kF8, D>::kKvSlotBytes);
            int row = kVarlen ? it.k_base + j * kTile : (it.j0 + j) * kTile, slab = kVarlen ? 0 : it.b;
            pp_paged_tile<kVarlen>(p, page, j, row, slab);
            page = page_next;
            pp_load_tile<PpOperands<kF8, D>::kOneBox>(sK + ring.slot * PpOperands<kF8, D>::kKvSlotBytes, tm_k, pp_bar(bar0, ppb::k_full + ring.slot), it.hk, row, slab, pol_kv);
        }
    }
}

// An item's output, staged in the V slot of its last step.
struct PpStaged {
    uint32_t end;    // that step
    int row, rows;   // first row in o and rows to store (32 at a time)
    int h, b, done_slot;
};

// The thread that loads V of every step and stores the 16-bit outputs.  An item's last P V has read its V slot when the
// epilogue gets O, and the slot is next needed by the step after next, which the same warpgroup runs once it is through
// with the epilogue: so O is staged there, and before this thread loads that step's V it sends the tile and
// waits until it has been read.  The warps that staged it neither issue nor wait for stores, and Q buffers are handed
// back by the item's last Q K^T.  (Staged in the Q buffer, by each warp for itself, as it was, a buffer came back only when the
// item after had begun, and short items began with a cold load: 8 x 32 x 512 40.4 -> 38.2 us, 4 x 32 x 2048 166.5 -> 160.3, 16 x 32 x
// 256 33.2 -> 30.7, 32 x 8192 503 -> 497; 32 packed requests of 16 to 512 tokens 87.8 -> 85.2, 10 of 100 to 3000 311 -> 305; 8-bit
// operands 8 x 32 x 512 26.5 -> 24.6, 16 x 32 x 128 10.9 -> 9.7; d = 64 level.  With a tile of its own for the output and
// two K slots, and the warps still sending: 38.9, 167.1, 31.0, but 2 to 4 % slower packed.  With 256-bit stores from
// registers instead: 44.2, 176.0, 35.1.)
template <bool kTmaOut, bool kVarlen, bool kF8, bool kProj, int D>
__device__ __forceinline__ void pp_run_v(uint32_t bar0, uint32_t sV, const CUtensorMap* tm_v, const CUtensorMap* tm_o, const FwdParams& p,
                                         const PpItem* slots, volatile uint32_t* abort_flag, unsigned int* done) {
    using Op = PpOperands<kF8, D>;
    tma_prefetch_desc(tm_v);
    const uint64_t pol_kv = l2_policy_evict_last();
    PpRing<kPpNV> ring;
    PpTaker<kVarlen> items{slots, bar0, abort_flag};
    PpItem it;
    uint32_t g = 0, sent = 0;
    PpStaged first = {}, second = {};   // outputs not yet sent, in order
    int waiting = 0;                    // how many
    int done_slot = -1;                 // kProj: row block whose stores have not been counted yet
    auto count_done = [&]() {
        if (kProj && done_slot >= 0) {
            tma_store_wait_all();       // written, not only read out of shared memory
            red_release_gpu_add(done + done_slot, 4u);
            done_slot = -1;
        }
    };
    auto send = [&]() -> bool {
        if (!mbar_wait(pp_bar(bar0, ppb::o_staged + (sent & 1)), (sent >> 1) & 1, abort_flag, 156)) return false;
        count_done();
        const uint32_t tile = sV + (first.end & 1) * Op::kVSlotBytes;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // packed batches: the rows after a sequence's last belong to the next sequence, so only 32 rows that
            // all exist go as a box (the others' threads have written them)
            if (kVarlen ? 32 * q + 32 <= first.rows : 32 * q < first.rows) {
                if (D == 128) tma_store_5d(tm_o, tile + q * 8192, 0, first.row + 32 * q, 0, first.h, first.b);
                else tma_store_4d(tm_o, tile + q * 4096, 0, first.h, first.row + 32 * q, first.b);
            }
        }
        tma_store_commit();
        if (kProj) done_slot = first.done_slot;
        ++sent;
        first = second;
        --waiting;
        return true;
    };
    while (items.next(it, 155)) {
        if (items.ord == 0 && *abort_flag) return;
        int page = (kVarlen && p.block_table != nullptr) ? it.page0 : 0;
        for (int j = 0; j < it.n; ++j, ++g, ring.next()) {
            const int page_next = pp_page_of<kVarlen>(p, it.b, j + 1, it.n, it.Skv);
            if (kTmaOut && waiting > 0 && first.end + 2 == g) {
                if (!send()) return;
                tma_store_wait_read();
            } else if (!mbar_wait(pp_bar(bar0, ppb::pv_done + ring.slot), ring.par ^ 1, abort_flag, 152)) return;
            mbar_expect_tx(pp_bar(bar0, ppb::v_full + ring.slot), Op::kKvSlotBytes);
            int row = kVarlen ? it.k_base + j * kTile : (it.j0 + j) * kTile, slab = kVarlen ? 0 : it.b;
            pp_paged_tile<kVarlen>(p, page, j, row, slab);
            page = page_next;
            pp_load_tile<Op::kOneBox>(sV + ring.slot * Op::kVSlotBytes, tm_v, pp_bar(bar0, ppb::v_full + ring.slot), it.hk, row, slab, pol_kv);
        }
        if (kTmaOut) {
            const PpStaged now = {g - 1, (kVarlen ? it.q_base : 0) + it.q0, (kVarlen ? it.Sq : p.Sq) - it.q0, it.h, kVarlen ? 0 : it.b,
                                  kProj ? it.b * p.n_qtiles + it.q0 / kTile : 0};
            if (waiting == 0) first = now;
            else second = now;
            ++waiting;
        }
    }
    if (kTmaOut) {
        while (waiting > 0)
            if (!send()) break;
        count_done();
        tma_store_wait_all();   // the stores read shared memory, which has to outlive them
    }
}

// Warp-wide wait: every lane waits, and the warp leaves together if any lane gave up (the
// tensor-memory instructions that follow need the whole warp).
__device__ __forceinline__ bool pp_warp_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                             unsigned int where) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;   // the usual case, in one branch
    const bool ok = mbar_wait(bar, parity, abort_flag, where);
    return __all_sync(0xffffffffu, ok);
}

// One thread of a softmax warpgroup: its state across the steps of an item, and the step.
template <typename T, bool kVarlen, bool kF8, int D>
struct PpSoftmax {
    static_assert(!(kF8 && kVarlen), "packed batches take 16-bit operands");
    using Op = PpOperands<kF8, D>;
    // fixed for the kernel
    uint32_t bar0;
    volatile uint32_t* abort_flag;
    float* m_mine;          // this row's slot in the reference-max exchange, written by this warpgroup
    const float* m_other;   // the same row's slot written by the other warpgroup
    int w;                  // warpgroup: runs the steps with g & 1 == w
    uint32_t tO, tS, tP;    // this warp's lane quarter of O, S_w, P_w in tensor memory
    float scale_log2;
    int causal, Skv, off;
    int kv_first;           // first key of the item's first kv tile (0 unless CTAs share a query tile)
    uint32_t sV;            // V ring in shared memory (packed batches: see the end of step())
    // per item
    int row;                // query row of this thread
    int lim0;               // packed batches: keys of the sequence that it sees
    float l_part;           // row sum over this warpgroup's steps, relative to m_loc
    float m_loc;            // reference max after this warpgroup's latest step
    float m_before;         // reference max that step received from the step before it

    // Step g of the CTA = step j of the item.  masked: the tile is crossed by the diagonal or by
    // the end of the keys.  Returns false when a wait gave up.
    __device__ __forceinline__ bool step(uint32_t (&s)[128], uint32_t g, int j, bool masked) {
        if (!pp_warp_wait(pp_bar(bar0, ppb::s_full + w), (g >> 1) & 1, abort_flag, 110 + w)) return false;
        tc_fence_after();
        tmem_ld_x32(tS, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
        tmem_ld_x32(tS + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
        tmem_ld_x32(tS + 64, *reinterpret_cast<uint32_t(*)[32]>(&s[64]));
        tmem_ld_x32(tS + 96, *reinterpret_cast<uint32_t(*)[32]>(&s[96]));
        tmem_wait_ld();
        tc_fence_before();  // for the arrival below that hands the S buffer back
        // probe and read early, look at the answer after the row max
        const bool m_there = g == 0 || mbar_test(pp_bar(bar0, ppb::m_ready + (1 - w)), ((g - 1) >> 1) & 1);
        float m_prev = *m_other;
        if (masked) {
            // hidden scores become -inf (the scale is strictly positive, so they come out as exact zeros)
            // (A packed item's lengths come from shared memory and live in registers, of which one is enough: 10 requests of 100
            // to 3000 tokens 316 -> 313 us, 2 of 250 to 8000 233 -> 229.  A dense call's are parameters, and as fast as they are.)
            int lim;
            if (kVarlen) {
                lim = lim0 - j * kTile;
            } else {
                const int kv0 = kv_first + j * kTile;
                lim = Skv - kv0;
                if (causal) lim = min(lim, row + off - kv0 + 1);
            }
            // (bits of a word instead of a comparison per score: several predicates are set at a time; 4 x 32 x 2048
            // 173.9 -> 171.2 us, 32 packed prompts of 256 to 8192 tokens 4450 -> 4399, 8 x 32 x 512 43.1 -> 42.8)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int n = lim - 32 * c;
                const uint32_t seen = n >= 32 ? 0xffffffffu : n <= 0 ? 0u : (1u << n) - 1u;
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    if (!(seen & (1u << i))) s[32 * c + i] = 0xff800000u;
            }
        }
        const float mx = pp_row_max(s);
        // reference max left by step g-1 (of the other warpgroup, read above); an item starts afresh
        if (!__all_sync(0xffffffffu, m_there)) {
            if (!pp_warp_wait(pp_bar(bar0, ppb::m_ready + (1 - w)), ((g - 1) >> 1) & 1, abort_flag, 112 + w)) return false;
            m_prev = *m_other;
        }
        if (j == 0) m_prev = -INFINITY;
        m_before = m_prev;
        // lazy reference update: the reference moves only when the row max outgrew it by more than
        // the threshold (always on the first visible score; never on -inf)
        const bool grow = (mx - m_prev) * scale_log2 > (kF8 ? kP8Threshold : kRescaleThreshold);
        const float m_new = grow ? mx : m_prev;
        *m_mine = m_new;
        // one arrival per thread: publishes its reference max and, the scores being in registers,
        // lets Q K^T of step g+2 overwrite the S buffer
        mbar_arrive(pp_bar(bar0, ppb::m_ready + w));
        // this warpgroup's row sum follows the reference (a factor of 1 rather than a branch)
        l_part *= m_loc == m_new ? 1.f : fast_exp2((m_loc - m_new) * scale_log2);
        m_loc = m_new;
        const float neg_ms = -((m_new == -INFINITY) ? 0.f : m_new) * scale_log2 + (kF8 ? kP8ScaleLog2 : 0.f);
        const uint64_t sc2 = f2_pack(scale_log2, scale_log2), nm2 = f2_pack(neg_ms, neg_ms);
        uint64_t la = f2_pack(0.f, 0.f), lb = la;
        // All of P is formed in registers (a packed pair takes the place of two scores) and goes to tensor
        // memory in one piece at the end.  Stored chunk by chunk, the first store had to wait for P V of
        // step g-2, which ends about 1400 clocks after that step's P was handed over, and a warpgroup's step
        // was that long plus the other three chunks: 32 heads x 32768 7828 -> 7615 us, 8192 keys 541 -> 527,
        // 5 heads x 4096 32.3 -> 31.3, 1001 queries over 7951 keys 472 -> 460, short sequences level.
        // From there on the steps were bound by the warpgroups' own chains, and what those lost most on were
        // branches (about 30 clocks each until they are resolved, and a scheduler has two of these warps).
        // So a step's fast path has five: one for each of three waits -- a vote on a first probe, and
        // everything rare behind it --, one for the mask and one at its end.  The same four cases: 7603 -> 7368,
        // 526 -> 509, 31.4 -> 30.1, 460 -> 442; 4 x 32 x 2048 178 -> 172, 8 x 32 x 512 44.0 -> 42.6.
        uint32_t pk[4][Op::kPCols];
#pragma unroll
        for (int c = 0; c < 3; ++c) pp_exp_chunk<T, kF8>(s, c, sc2, nm2, la, lb, pk[c]);
        const bool p_free = g < 2 || mbar_test(pp_bar(bar0, ppb::pv_done + w), ((g >> 1) - 1) & 1);
        pp_exp_chunk<T, kF8>(s, 3, sc2, nm2, la, lb, pk[3]);
        if (__builtin_expect(!__all_sync(0xffffffffu, p_free && !(j > 0 && grow)), 0)) {
            // O += P V of step g-2 has read this P buffer
            if (g >= 2 && !pp_warp_wait(pp_bar(bar0, ppb::pv_done + w), ((g >> 1) - 1) & 1, abort_flag, 116 + w)) return false;
            if (j > 0 && __any_sync(0xffffffffu, grow)) {
                // rare: the reference moved.  O holds the P V sums up to step g-1 once that step's
                // MMAs have completed (those of step g-2 have, see above, so the parity wait on the
                // other buffer's barrier is one phase at most behind).
                if (!pp_warp_wait(pp_bar(bar0, ppb::pv_done + (1 - w)), ((g - 1) >> 1) & 1, abort_flag, 114 + w)) return false;
                tc_fence_after();
                const float alpha = grow ? ((m_prev == -INFINITY) ? 0.f : fast_exp2((m_prev - mx) * scale_log2)) : 1.f;
#pragma unroll 1
                for (int c = 0; c < D / 16; ++c) {
                    uint32_t o[16];
                    tmem_ld_x16(tO + c * 16, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                    tmem_st_x16(tO + c * 16, o);
                }
            }
        }
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < 4; ++c) pp_store_p<kF8>(tP + c * Op::kPCols, pk[c]);
        {
            float a0, a1, b0, b1;
            f2_unpack(la, a0, a1);
            f2_unpack(lb, b0, b1);
            l_part += (a0 + a1) + (b0 + b1);
        }
        if (kVarlen && masked && Skv - j * kTile < kTile) {
            // Packed batches, the tile that holds a sequence's last key: the rows of V after it
            // belong to the next sequence, or to the unused rest of a page, and may hold anything.
            // Their probabilities are exact zeros, but 0 * NaN would still poison O, so those
            // rows are cleared in shared memory before P V of this step may start (a contiguous
            // tensor gets the same from the zero fill of its TMA loads).  A row's bytes are one 128-byte line in each
            // 64-element half of the tile, whatever the swizzle; eight threads clear a line.  (A thread per row hits the
            // same banks with all lanes: 32 requests of 16 to 512 tokens, GQA, 85.2 -> 82.5 us, 20 chunks of up to 666 57.1 ->
            // 55.1, 6 of up to 2000 21.9 -> 21.1, long requests level.)
            static_assert(kPpNV == 2, "the V slot of step g is taken to be g & 1");
            if (!pp_warp_wait(pp_bar(bar0, ppb::v_full + w), (g >> 1) & 1, abort_flag, 124 + w)) return false;
            const int dead = max(0, Skv - j * kTile);
            for (int r0 = dead + (int)((threadIdx.x & 127) >> 3); r0 < kTile; r0 += 16) {
                const uint32_t at = sV + (uint32_t)w * Op::kVSlotBytes + (uint32_t)r0 * 128u + (threadIdx.x & 7) * 16u;
#pragma unroll
                for (int h = 0; h < D / 64; ++h) asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(at + (uint32_t)h * kHalfBytes), "r"(0u) : "memory");
            }
            fence_proxy_async_smem();
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(pp_bar(bar0, ppb::p_full + w));
        return true;
    }
};

// Merge of the parts that a cluster's CTAs computed of one query tile: CTA `rank` of `split` finishes
// rows rank, rank + split, ..., one warp per row and four columns per lane, reading the parts through
// distributed shared memory.
constexpr uint32_t kPpPartStats = 65536;   // bytes from a part's O to its (max, sum) pairs
template <typename T>
__device__ __forceinline__ void pp_split_merge(const FwdParams& p, uint32_t part, int tid) {
    const int warp = uniform(tid >> 5), lane = tid & 31;
    const int split = p.split, idx = (int)blockIdx.x / split, rank = (int)blockIdx.x - idx * split;
    int bh, qt, b, h;
    pp_class_order(p, idx, bh, qt);
    p.by_hq.divmod(bh, b, h);
    const int q0 = qt * kTile;
    const int n = kv_tiles_for(q0, kTile, p.Sq, p.Skv, p.causal);
    // Rows `rank + split * k`, k < mine, are this CTA's.  Weights first, one thread per row and part, all at once (a
    // group of 2, 4, 8 or 16 lanes has a row): exp2 of the part's max over the largest, divided by the
    // row's sum; -1 for a part without kv tiles, which holds nothing, and one whose keys the row does
    // not see.  A sum that is NaN (a NaN or infinite score) makes every weight of the row NaN.  They go
    // where this CTA's own pairs are not.
    const uint32_t w_at = part + kPpPartStats + 2048u;   // [k][kMaxCluster]
    const int rows = min(kTile, p.Sq - q0), mine = rank < rows ? (rows - rank + split - 1) / split : 0;
    const int width_log2 = 32 - __clz(split - 1);
    {
        const int k = tid >> width_log2, i = tid & ((1 << width_log2) - 1);
        const int row = rank + split * k;
        float m = -INFINITY, l = 0.f;
        if (k < mine && i < split && pp_split_first(n, split, i + 1) > pp_split_first(n, split, i))
            cluster_ld2(cluster_map(part + kPpPartStats + (uint32_t)row * 8u, i), m, l);
        const bool nothing = l == 0.f;
        float M = nothing ? -INFINITY : m;
        for (int sh = 1 << width_log2 >> 1; sh > 0; sh >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, sh));
        const float w = nothing ? 0.f : fast_exp2((m - M) * p.scale_log2);
        float sum = w * l;
        for (int sh = 1 << width_log2 >> 1; sh > 0; sh >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, sh);
        if (k < mine) {
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(w_at + (uint32_t)(k * kMaxCluster + i) * 4u), "f"(nothing ? -1.f : w / sum) : "memory");
            if (i == 0 && p.lse != nullptr)
                p.lse[((long long)b * p.Hq + h) * p.Sq + q0 + row] = sum > 0.f ? (M * p.scale_log2 + log2f(sum)) * 0.6931471805599453f : -INFINITY;
        }
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    // Then the rows, one warp and four columns per lane, up to four rows at a time: the loads' latency is what this takes.
    // A CTA begins with the part of the CTA after it and ends with its own: from the same part on, all
    // would read one CTA's shared memory at a time.
    auto merge_rows = [&](auto rows_at_a_time) {
        constexpr int kRows = decltype(rows_at_a_time)::value;
        for (int k0 = warp; k0 < mine; k0 += 8 * kRows) {
            float acc[kRows][4];
#pragma unroll
            for (int q = 0; q < kRows; ++q) acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.f;
            int i = rank;
            auto add_part = [&](auto own) {
                i = i + 1 == split ? 0 : i + 1;
                const uint32_t from = decltype(own)::value ? part : cluster_map(part, i);
                float v[kRows][4], w[kRows];
#pragma unroll
                for (int q = 0; q < kRows; ++q) {
                    const int k = min(k0 + 8 * q, mine - 1), row = rank + split * k;
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(w[q]) : "r"(w_at + (uint32_t)(k * kMaxCluster + i) * 4u));
                    const uint32_t at = from + (uint32_t)row * 512u + (uint32_t)((lane ^ (row & 31)) << 4);
                    if (decltype(own)::value)
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[q][0]), "=f"(v[q][1]), "=f"(v[q][2]), "=f"(v[q][3]) : "r"(at));
                    else cluster_ld4(at, v[q]);
                }
#pragma unroll
                for (int q = 0; q < kRows; ++q)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[q][c] = w[q] < 0.f ? acc[q][c] : fmaf(w[q], v[q][c], acc[q][c]);
            };
#pragma unroll(kRows == 4 ? 1 : 4)
            for (int t = 0; t < split - 1; ++t) add_part(std::false_type());
            add_part(std::true_type());
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                const int k = k0 + 8 * q;
                if (k < mine) {
                    const long long at_o = (long long)b * p.o_sb + (long long)(q0 + rank + split * k) * p.o_ss + (long long)h * p.o_sh + 4 * lane;
                    if (p.o_fp32)
                        *reinterpret_cast<float4*>(static_cast<float*>(p.o) + at_o) = make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
                    else
                        *reinterpret_cast<uint2*>(static_cast<T*>(p.o) + at_o) = make_uint2(pack2<T>(acc[q][0], acc[q][1]), pack2<T>(acc[q][2], acc[q][3]));
                }
            }
        }
    };
    if (mine <= 8) merge_rows(std::integral_constant<int, 1>());
    else if (mine <= 16) merge_rows(std::integral_constant<int, 2>());
    else merge_rows(std::integral_constant<int, 4>());
}

// kTmaOut: the output has the operands' 16-bit type; an item's O goes, scaled and rounded, into
// the V slot of the item's last step (which P V has finished with by then) in the swizzled layout of a tile,
// and the thread that loads V sends it to global memory (tm_o: boxes of 32
// rows).  Rows past the end of the queries are clipped by the tensor map.  Otherwise
// (fp32 output) every thread stores its own row.
// kVarlen (needs kTmaOut): a packed batch of sequences of different lengths (see FwdParams).
// kF8: q, k, v hold FP8 e4m3 bytes (see PpOperands); T is then the type of the output only.
// kProj (needs kTmaOut): a projection phase follows in the same launch (proj_gemm.cuh): when an item's
// stores have reached global memory the thread that issued them counts
// them in done[batch * n_qtiles + query tile], 32 rows as one; four of them and Hq heads make a row
// block of O complete.
// The whole kernel but for the release of tensor memory; returns false if nothing was set up.
template <typename T, bool kTmaOut, bool kVarlen, bool kF8, bool kProj, int D = 128, bool kSplit = false>
__device__ __forceinline__ bool pp_attention(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v,
                                             const CUtensorMap& tm_o, const FwdParams& p, const int total_items,
                                             PpStatic& ss, const uint32_t smem_base, unsigned int* done) {
    static_assert(!kSplit || (!kTmaOut && !kVarlen && !kF8 && !kProj && D == 128), "one form shares query tiles");
    static_assert(!kProj || (kTmaOut && !kVarlen && D == 128), "the projection phase reads a contiguous 16-bit O of d = 128");
    const uint32_t sQ = smem_base;
    const uint32_t sK = sQ + kPpQBufs * PpOperands<kF8, D>::kQBufBytes;
    const uint32_t sV = sK + kPpNK * PpOperands<kF8, D>::kKvSlotBytes;
    const uint32_t bar0 = smem_u32(&ss.bars[0]);
    volatile uint32_t* abort_flag = &ss.abort_flag;

    const int tid = threadIdx.x;
    const int warp = uniform(tid >> 5);
    const int lane = tid & 31;
    if (smem_base & 1023u) {  // uniform for the CTA: nothing has been set up yet
        if (tid == 0) record_timeout(900);
        return false;
    }
    if (tid == 0) {
        for (int i = 0; i < ppb::count; ++i) {
            const bool staged = i == ppb::o_staged || i == ppb::o_staged + 1;
            const bool slot_back = i >= ppb::item_empty && i < ppb::item_empty + kPpSlots;
            mbar_init(pp_bar(bar0, i), i >= ppb::p_full ? 128 : (slot_back ? 11 : (staged ? 4 : 1)));
        }
        ss.abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 8) {
        tmem_alloc(smem_u32(&ss.tmem_holder), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ss.tmem_holder;
    const int off = p.Skv - p.Sq;

    if (warp < 8) {
        // ================================================================ softmax + epilogue
        setmaxnreg_inc<kPipeSoftmaxRegs>();  // a whole row of S lives in registers
        const int w = warp >> 2;             // this warpgroup runs the steps with g & 1 == w
        const int r = tid & 127;
        const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t tO = tmem_base + lane_sel;
        const uint32_t tS = tmem_base + lane_sel + 128 + 128 * w;
        const uint32_t tP = tmem_base + lane_sel + 384 + 64 * w;
        const float scale_log2 = p.scale_log2;
        PpSoftmax<T, kVarlen, kF8, D> sm;
        sm.sV = sV;
        sm.bar0 = bar0;
        sm.abort_flag = abort_flag;
        sm.m_mine = &ss.m_xch[w][r];
        sm.m_other = &ss.m_xch[1 - w][r];
        sm.w = w;
        sm.tO = tO;
        sm.tS = tS;
        sm.tP = tP;
        sm.scale_log2 = scale_log2;
        sm.causal = p.causal;
        sm.Skv = p.Skv;
        sm.off = off;
        sm.kv_first = 0;
        uint32_t g = 0;        // step counter of the CTA
        uint32_t items2 = 0;   // items with at least two steps seen so far
        bool ok = true;
        for (int ord = 0; ok; ++ord) {
            const int slot = ord & (kPpSlots - 1);
            if (kVarlen && ord == 0) grid_dep_wait();   // (see PpTaker)
            if (!pp_warp_wait(pp_bar(bar0, ppb::item_full + slot), (ord / kPpSlots) & 1, abort_flag, 122 + w)) break;
            // the epilogue reads the rest of the slot; it is handed back at the end of the item
            const PpItem& it = ss.items[slot];
            const int n = kVarlen ? uniform(it.n) : it.n, q0 = kVarlen ? uniform(it.q0) : it.q0;
            if (n == 0) break;
            if (!kVarlen && ord == 0) grid_dep_wait();
            const int row = q0 + r;   // within the sequence
            const int Sq_i = kVarlen ? it.Sq : p.Sq, Skv_i = kVarlen ? uniform(it.Skv) : p.Skv;
            const int off_i = kVarlen ? Skv_i - Sq_i : off;
            if (kVarlen) {
                sm.Skv = Skv_i;
                sm.lim0 = p.causal ? min(Skv_i, row + off_i + 1) : Skv_i;
            }
            sm.row = row;
            sm.l_part = 0.f;
            sm.m_loc = -INFINITY;
            sm.m_before = -INFINITY;
            uint32_t s[128];             // this thread's row of S, later of O
            const uint32_t xb = items2 & 1, xpar = (items2 >> 1) & 1;  // row-sum exchange buffer / phase
            // kv tiles every row of the query tile sees in full: they come first; on the few tiles
            // crossed by the diagonal or by the end of the keys, which follow, the step also masks.
            // (The step exists once and a branch skips its mask code: a second copy for the full
            // tiles was 1 % ahead from 8192 keys on while every role decoded its own items; with the
            // items handed over through shared memory the single copy is: 533 against 547 us on
            // 32 heads x 8192 causal keys.  What an item executes then stays within the 32 KB the
            // instruction cache serves at full rate.  The other operands and outputs, with all of the hand-over against the
            // state before it: FP8 4 x 32 x 2048 131 / 133 us, 8 x 32 x 512 31.7 / 35.4; d = 64 16 x 16 x 512 29.9 / 33.4,
            // 4 x 16 x 4096 level; fp32 output 8 x 32 x 512 55.1 / 60.3, 4 x 32 x 2048 209 / 207; fused projection level.)
            int n_full = Skv_i / kTile;
            if (p.causal) n_full = min(n_full, max(0, (q0 + off_i + 1) / kTile));
            if (kSplit) {
                n_full = max(0, n_full - it.j0);
                sm.kv_first = it.j0 * kTile;
            }
            n_full = min(n_full, n);
            // this warpgroup's steps of the item: those with an absolute step number of its parity
            const uint32_t g_item = g;
            int j = (int)((g_item ^ (uint32_t)w) & 1u);
            for (; j < n; j += 2) {
                ok = sm.step(s, g_item + (uint32_t)j, j, j >= n_full);
                if (!ok) break;
                if (j == n - 2) {
                    // the other warpgroup runs the last step and the epilogue: hand it this row sum
                    // (it is relative to the reference this step left, which that step receives)
                    ss.l_xch[xb][r] = sm.l_part;
                    mbar_arrive(pp_bar(bar0, ppb::l_pub + xb));
                }
            }
            const float l_part = sm.l_part, m_loc = sm.m_loc, m_before = sm.m_before;
            if (ok && ((g_item + (uint32_t)n - 1u) & 1u) == (uint32_t)w) {
                // ---- epilogue of the item, by the warpgroup that ran its last step
                float l_run = l_part;
                if (n >= 2) {
                    ok = pp_warp_wait(pp_bar(bar0, ppb::l_pub + xb), xpar, abort_flag, 118 + w);
                    if (!ok) break;
                    const float l_other = ss.l_xch[xb][r];
                    // the other warpgroup's sum is relative to the reference this one's last step received
                    // (a NaN, from a NaN or infinite score, must stay one: where CTAs share a tile the sum is all the merge looks at)
                    if (l_other != 0.f) l_run += l_other * fast_exp2((m_before - m_loc) * scale_log2);
                }
                // (before the wait for the last P V, which takes longer than this)
                // (FP8: O and the row sum carry the same factor on the probabilities; V's own factor goes on O)
                const float inv_l = (l_run > 0.f) ? (kF8 ? p.out_scale / l_run : 1.f / l_run) : 0.f;
                const long long obase = kVarlen ? (long long)(it.q_base + row) * p.o_ss + (long long)it.h * p.o_sh
                                                : (long long)it.b * p.o_sb + (long long)row * p.o_ss + (long long)it.h * p.o_sh;
                if (!kSplit && row < Sq_i && p.lse != nullptr) {
                    const float lse = (l_run > 0.f) ? (m_loc * scale_log2 + log2f(l_run) - (kF8 ? kP8ScaleLog2 : 0.f)) * 0.6931471805599453f
                                                    : -INFINITY;
                    if (kVarlen) p.lse[(long long)it.h * p.total_q + it.q_base + row] = lse;
                    else p.lse[((long long)it.b * p.Hq + it.h) * p.Sq + row] = lse;
                }
                ok = pp_warp_wait(pp_bar(bar0, ppb::o_final + (ord & 1)), (ord >> 1) & 1, abort_flag, 120 + w);
                if (!ok) break;
                tc_fence_after();
                tmem_ld_x32(tO, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
                tmem_ld_x32(tO + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
                if (D == 128) {
                    tmem_ld_x32(tO + 64, *reinterpret_cast<uint32_t(*)[32]>(&s[64]));
                    tmem_ld_x32(tO + 96, *reinterpret_cast<uint32_t(*)[32]>(&s[96]));
                }
                tmem_wait_ld();
                // O is in registers: the next item's first P V may overwrite it
                tc_fence_before();
                mbar_arrive(pp_bar(bar0, ppb::o_free));
                if (kSplit) {
                    // this CTA's part, for the merge below: the row of O as it is and its max and sum,
                    // in the K ring (read to the end by now); 16-byte chunks are swizzled by the row
                    const uint32_t part = sK + (uint32_t)r * 512u;
#pragma unroll
                    for (int c = 0; c < D / 4; ++c)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(part + (uint32_t)((c ^ (r & 31)) << 4)), "r"(s[4 * c]),
                                     "r"(s[4 * c + 1]), "r"(s[4 * c + 2]), "r"(s[4 * c + 3])
                                     : "memory");
                    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(sK + kPpPartStats + (uint32_t)r * 8u), "f"(m_loc), "f"(l_run) : "memory");
                } else if (kTmaOut) {
                    // a warp's rows, in the V slot of the item's last step (see pp_run_v): its 64-column blocks one after
                    // the other, as its store takes them
                    const uint32_t slab = sV + (uint32_t)w * PpOperands<kF8, D>::kVSlotBytes + (uint32_t)(warp & 3) * (D == 128 ? 8192u : 4096u);
                    const uint32_t row_base = slab + (uint32_t)lane * 128u;
                    // (packed multiplications: 8 x 32 x 512 42.6 -> 42.0 us, 16 x 32 x 256 34.6 -> 34.3, 10 packed requests of 100 to 3000
                    // tokens 325 -> 316, 32 of 256 to 8192 4158 -> 4072, others level)
#pragma unroll
                    for (int i = 0; i < D / 2; ++i) {
                        float x0, x1;
                        f2_unpack(f2_mul(f2_pack(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), f2_pack(inv_l, inv_l)), x0, x1);
                        s[i] = pack2<T>(x0, x1);
                    }
                    if (kVarlen && uniform(it.q0 + (warp & 3) * 32 + 32 > Sq_i)) {
                        // 32 rows that do not all exist (see pp_run_v): each thread writes its own row
                        if (row < Sq_i) {
                            uint4* dst = reinterpret_cast<uint4*>(static_cast<T*>(p.o) + obase);
#pragma unroll
                            for (int c = 0; c < D / 8; ++c) dst[c] = make_uint4(s[4 * c], s[4 * c + 1], s[4 * c + 2], s[4 * c + 3]);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < D / 8; ++c) {
                            // 16-byte chunk c & 7 of the row's half c >> 3, at its swizzled place
                            const uint32_t addr = row_base + (uint32_t)(c >> 3) * 4096u + (((uint32_t)(c & 7) ^ ((uint32_t)lane & 7u)) << 4);
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(s[4 * c]), "r"(s[4 * c + 1]), "r"(s[4 * c + 2]), "r"(s[4 * c + 3]) : "memory");
                        }
                        fence_proxy_async_smem();
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(pp_bar(bar0, ppb::o_staged + (ord & 1)));
                } else if (row < Sq_i) {
                    if (p.o_fp32) {
                        float4* dst = reinterpret_cast<float4*>(static_cast<float*>(p.o) + obase);
#pragma unroll
                        for (int i = 0; i < D / 4; ++i)
                            dst[i] = make_float4(__uint_as_float(s[4 * i]) * inv_l, __uint_as_float(s[4 * i + 1]) * inv_l,
                                                 __uint_as_float(s[4 * i + 2]) * inv_l,
                                                 __uint_as_float(s[4 * i + 3]) * inv_l);
                    } else {
                        T* dst = static_cast<T*>(p.o) + obase;
#pragma unroll
                        for (int c = 0; c < D / 8; ++c)
                            reinterpret_cast<uint4*>(dst)[c] =
                                make_uint4(pack2<T>(__uint_as_float(s[8 * c]) * inv_l, __uint_as_float(s[8 * c + 1]) * inv_l),
                                           pack2<T>(__uint_as_float(s[8 * c + 2]) * inv_l, __uint_as_float(s[8 * c + 3]) * inv_l),
                                           pack2<T>(__uint_as_float(s[8 * c + 4]) * inv_l, __uint_as_float(s[8 * c + 5]) * inv_l),
                                           pack2<T>(__uint_as_float(s[8 * c + 6]) * inv_l, __uint_as_float(s[8 * c + 7]) * inv_l));
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(pp_bar(bar0, ppb::item_empty + slot));
            g = g_item + (uint32_t)n;
            if (n >= 2) ++items2;
        }
    } else {
        setmaxnreg_dec<kPipeOtherRegs>();
        if (elect_one()) {
            if (warp == 8) pp_run_s<T, kVarlen, kF8, D>(bar0, sQ, sK, tmem_base, ss.items, abort_flag);
            else if (warp == 10) pp_run_pv<T, kVarlen, kF8, D>(bar0, sV, tmem_base, ss.items, abort_flag);
            else if (warp == 9) pp_run_load_qk<kVarlen, kF8, D>(bar0, sQ, sK, &tm_q, &tm_k, p, total_items, ss, abort_flag);
            else pp_run_v<kTmaOut, kVarlen, kF8, kProj, D>(bar0, sV, &tm_v, &tm_o, p, ss.items, abort_flag, done);
        }
        __syncwarp();
    }
    if constexpr (kSplit) {
        __syncwarp();
        cluster_sync_all();
        if (warp < 8) pp_split_merge<T>(p, sK, tid);
        __syncwarp();
        cluster_sync_all();   // nobody's shared memory goes away while others read it
    }
    return true;
}

// Few query tiles: the CTAs of a cluster share one (see pp_split_item and the launcher).
template <typename T>
__global__ void __launch_bounds__(kPipeThreads, 1)
fa_fwd_pingpong_split_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                             const __grid_constant__ CUtensorMap tm_v, const FwdParams p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(1024) uint8_t static_raw[kPpStaticBytes];
    PpStatic& ss = *reinterpret_cast<PpStatic*>(static_raw);
    if (!pp_attention<T, false, false, false, false, 128, true>(tm_q, tm_k, tm_v, tm_q, p, 0, ss, smem_u32(smem_raw), nullptr))
        return;
    tc_fence_before();
    __syncthreads();
    if ((threadIdx.x >> 5) == 8) {
        settle_if(ss.abort_flag);
        __syncwarp();
        tmem_dealloc(ss.tmem_holder, 512);
    }
}

template <typename T, bool kTmaOut, bool kVarlen, bool kF8 = false, int D = 128>
__global__ void __launch_bounds__(kPipeThreads, 1)
fa_fwd_pingpong_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o,
                       const FwdParams p, const int total_items) {
    // Shared memory is used to the last byte: 3 KiB of static state (sized so that the dynamic
    // part that follows it starts on a 1024-byte boundary, which the 128-byte swizzle needs)
    // plus seven 32 KiB tiles (d = 128, 16 bits).  The alignment is checked rather than assumed.
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(1024) uint8_t static_raw[kPpStaticBytes];
    PpStatic& ss = *reinterpret_cast<PpStatic*>(static_raw);
    if (!pp_attention<T, kTmaOut, kVarlen, kF8, false, D>(tm_q, tm_k, tm_v, tm_o, p, total_items, ss, smem_u32(smem_raw),
                                                          nullptr))
        return;
    tc_fence_before();
    __syncthreads();
    if ((threadIdx.x >> 5) == 8) {
        settle_if(ss.abort_flag);
        __syncwarp();
        tmem_dealloc(ss.tmem_holder, 512);
    }
}

// The item order of a launch on `grid` CTAs (see pp_class_order and PpSource): returns the
// parameters with the order's fields filled in.  bytes_per_key: K plus V bytes of one key and head.
inline FwdParams pp_plan_items(const FwdParams& fp, int grid, double bytes_per_key) {
    const bool varlen = fp.cu_q != nullptr;
    // Class size of the item order: large enough that the K and V of the kv heads one round of
    // CTAs works on (about grid / (C * group) of them, Skv * 512 bytes each) fit in a fraction of
    // L2, but at most half of a head's tiles and 16 (a class that is the whole head makes all
    // its tiles read the same K/V lines at the same moment, which measured slower).  Under the
    // causal mask the items of a class differ in length, which costs balance when a head has few
    // tiles: heads with fewer than 16 keep the plain longest-first order as long as all keys and
    // values together about fit in L2 (2 x 32 heads x 1900: 75 us against 81 in classes of 8; 8 x 32 x
    // 1024, 134 MB, level); past that a longest-first round finds none of its K/V there, and heads of
    // 6 tiles and more take classes of 8 (5 x 32 x 1800: 194 us against 214; 16 x 32 x 768: 146
    // against 154; 8 x 32 x 1500: 220 against 232).  When one head alone fills every CTA, a single
    // class: the plain head-by-head order.
    FwdParams fpc = fp;
    int cls_log2 = 0;
    if (fp.n_qtiles >= grid) {
        while ((1 << cls_log2) < fp.n_qtiles) ++cls_log2;
    } else {
        const double head_bytes = bytes_per_key * fp.Skv / (fp.Hq / fp.Hkv);
        const double budget = 32.0 * 1024 * 1024;
        const int half = fp.n_qtiles / 2 < 16 ? fp.n_qtiles / 2 : 16;
        if (fp.causal && fp.n_qtiles < 16) {
            if (fp.n_qtiles >= 6 && bytes_per_key * fp.Skv * fp.B * fp.Hkv > 140e6) cls_log2 = 3;
        } else {
            while ((grid >> cls_log2) * head_bytes > budget && (2 << cls_log2) <= half) ++cls_log2;
            while (cls_log2 > 0 && (1 << cls_log2) > fp.n_qtiles) --cls_log2;
        }
    }
    // From three rounds per head on (56K keys on 148 SMs) and once a head's K and V are past what
    // L2 keeps, the head-by-head order with whole rounds per head (see PpSource); the empty slots of
    // a head's last round cost little there because its items are the head's shortest.
    const double kv_bytes_per_head = bytes_per_key * fp.Skv;
    if (!varlen && fp.n_qtiles >= 3 * grid && kv_bytes_per_head > 24.0 * 1024 * 1024) {
        fpc.rounds_per_head = (fp.n_qtiles + grid - 1) / grid;
        fpc.by_rph.set(fpc.rounds_per_head);
    }
    fpc.deal_ctas = grid;
    fpc.deal_rounds = 0x7fffffff;
    fpc.cls_log2 = cls_log2;
    const long long class_items = ((long long)fp.B * fp.Hq) << cls_log2;  // > total only for a single class
    fpc.by_class.set(class_items > 0x7fffffffll ? 0x7fffffff : (int)class_items);
    const int last = fp.n_qtiles & ((1 << cls_log2) - 1);
    fpc.by_lastcls.set(last ? last : 1);
    return fpc;
}

// to: map over the output with boxes of 32 rows (see encode_map_tile); read only when the output has the
// operands' type (any valid map otherwise).
// kF8: tq, tk, tv are maps over FP8 e4m3 bytes (boxes of 128 rows x 128 bytes) and T is the output type.
// D: the head dimension, 128, or 64 with 16-bit operands (maps with boxes of 64 elements either way).
template <typename T, bool kF8 = false, int D = 128>
int launch_pingpong(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& to,
                    const FwdParams& fp, cudaStream_t st, int* cuda_err) {
    constexpr int smem = PpOperands<kF8, D>::kSmem;
    const bool varlen = fp.cu_q != nullptr;
    if (varlen && fp.o_fp32) return -3;
    if (kF8 && (varlen || fp.o_fp32)) return -3;
    auto kern = kF8 ? fa_fwd_pingpong_kernel<T, true, false, kF8, D>
                    : (varlen ? fa_fwd_pingpong_kernel<T, true, kF8 ? false : true, false, D>
                              : (fp.o_fp32 ? fa_fwd_pingpong_kernel<T, false, false, false, D>
                                           : fa_fwd_pingpong_kernel<T, true, false, false, D>));
    int sm_count = 0;
    cudaError_t e;
    if (int ce = prepare_big_smem_kernel(reinterpret_cast<const void*>(kern), smem, &sm_count)) { *cuda_err = ce; return -7; }
    // packed batches: a place for every tile of every sequence, without knowing the lengths (see PpSource)
    const long long all_tiles = (long long)fp.n_qtiles * fp.B, packed_tiles = (long long)(fp.total_q >> 7) + fp.B;
    const bool fixed_places = !varlen || all_tiles <= packed_tiles;
    const long long total = (fixed_places ? all_tiles : packed_tiles) * fp.Hq;
    if (total > 0x7fffffffll) return -3;
    // Few query tiles over many keys: the CTAs of a cluster divide the kv tiles of a query tile and
    // merge their parts through distributed shared memory, as many CTAs to a tile as the device runs
    // for all tiles at once.  A step takes 0.8 to 1 us, and the exchange of the parts (64 KiB a CTA,
    // two cluster barriers, the launch of clusters) about five more than an ordinary epilogue, so it
    // pays from about eight steps saved on the longest tile (not shared / shared): 15 tiles over 157 kv tiles
    // 113.6 / 24.5 us (124 / 33 with 15 kv heads, whose keys come from HBM), 32 over 63 51.6 / 23.5, 64 over 32
    // 28.0 / 21.7, 64 over 16 16.6 / 15.4, 24 over 16 16.1 / 13.4, 30 over 12 13.3 / 12.0.  At the line itself both
    // sides occur: eight saved 74 over 16 21.0 / 22.0, 20 over 10 11.8 / 12.3; seven saved 30 over 10 level,
    // 5 over 8 10.3 / 9.3; six saved 60 over 12 15.2 / 15.4.
    if constexpr (!kF8 && D == 128) {
        if (fp.split == 0 && !varlen) {
            const int kv_tiles = (fp.Skv + kTile - 1) / kTile;   // of the longest item
            int c = kv_tiles < kMaxCluster ? kv_tiles : kMaxCluster;
            if (c > 1 && 2 * total <= sm_count) {
                auto split_kern = fa_fwd_pingpong_split_kernel<T>;
                ClusterSlots slots;
                if (int ce = cluster_slots(reinterpret_cast<const void*>(split_kern), smem, kPipeThreads, &slots)) { *cuda_err = ce; return -7; }
                while (c > 1 && slots.n[c] < total) --c;
                if (c > 1 && kv_tiles - (kv_tiles + c - 1) / c >= 8) {
                    FwdParams fps = fp;   // the plain longest-first order
                    fps.by_class.set(fp.B * fp.Hq);
                    fps.cls_log2 = 0;
                    fps.split = c;
                    fps.early_next = total * c < sm_count;
                    e = launch_dependent_clusters(split_kern, dim3((unsigned)total * c), c, 1, kPipeThreads, smem, st, tq, tk, tv, fps);
                    if (e != cudaSuccess) { *cuda_err = (int)e; return -7; }
                    return 0;
                }
            }
        }
    }
    int grid = (int)(total < sm_count ? total : sm_count);
    FwdParams fpc = pp_plan_items(fp, grid, (kF8 || D == 64) ? 256.0 : 512.0);
    fpc.split = 1;
    fpc.fixed_places = fixed_places;
    fpc.early_next = grid < sm_count;
    if (fpc.rounds_per_head == 0) {
        // How much of the list is dealt (see PpSource).  A deal keeps neighbours of the list, which
        // read the same K and V, on neighbouring CTAs; claims balance.  Packed batches, whose places
        // differ in length without order: all claimed (32 requests of 256 to 8192 tokens: 4.58 ms
        // against 4.83 dealt).  Head by head (a head fills the grid): the last two rounds and the
        // remainder claimed (32 heads x 32768: 7.92 ms; all dealt 8.07, remainder alone 8.13).
        // Class order: the remainder claimed (8 x 32 heads x 512: 43.1 us against 45.0 all dealt,
        // 32 x 8192: 526 against 535, 4 x 32 x 2048 level; a round more claimed loses 1 %), but all
        // after the first round if there are no more than two (5 heads x 8192: 81.3 against 85.4 us).
        const int full = (int)(total / grid);
        fpc.deal_rounds = varlen ? 0 : fp.n_qtiles >= grid ? max(1, full - 2) : full > 2 ? full : 1;
        const long long rest = total - (long long)fpc.deal_rounds * grid;
        fpc.claim_items = rest > 0;
        fpc.deal_ctas = fpc.deal_rounds > 0 ? grid : 0;
        grid = fpc.deal_ctas + (int)rest;
    }
    e = launch_dependent(kern, dim3(grid), kPipeThreads, smem, st, tq, tk, tv, to, fpc, (int)total);
    if (e != cudaSuccess) { *cuda_err = (int)e; return -7; }
    return 0;
}

}  // namespace fa
