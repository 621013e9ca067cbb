// Attention forward for head dimension 64 (the short, non-causal vision workload of the
// evaluation section: DeiT-like, 197 tokens, 12 heads, large batches; causal and longer
// sequences work too).  The tcgen05 tile shapes of d = 64: Q, K and V tiles are single 128 x 64
// swizzled TMA boxes; S = Q K^T takes four k-steps of 16; O += P V is an N = 64 MMA with V as the
// N-major operand.  Three kernels:
//   fa_fwd_d64_stream_kernel (prefill_d64_stream.cuh)  128 < Skv <= 256: all keys as one tile,
//                            single-pass softmax, a persistent pipeline over (batch, head, two query tiles)
//   fa_fwd_pingpong_kernel   (prefill_pingpong.cuh, D = 64)  longer sequences, packed batches, and most
//                            calls of up to 128 keys
//   fa_fwd_d64_slim_kernel   (here) few keys where the query tiles are more than the SMs: all keys as
//                            one tile, one thread per query row
#pragma once

#include "prefill_simple.cuh"

namespace fa {

constexpr int kD64TileBytes = 16384;   // 128 rows x 64 16-bit elements: one TMA box

// ---------------------------------------------------------------------------------------
// At most 128 keys, small enough for four CTAs per SM.  One CTA per (batch, head, query tile), 128
// threads, 49 KiB of shared memory (a tile each of Q, K and V) and 128 columns of tensor memory: S
// in [0,128), P packed over [0,64), and P V in [64,128) (columns of S the thread has read by
// then).
constexpr int kD64SlimSmem = 1024 + 3 * kD64TileBytes;

template <typename T>
__global__ void __launch_bounds__(128, 4)
fa_fwd_d64_slim_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const FwdParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sQ = smem_base;
    const uint32_t sK = sQ + kD64TileBytes;
    const uint32_t sV = sK + kD64TileBytes;
    __shared__ __align__(8) uint64_t bars[6];
    __shared__ uint32_t tmem_holder;
    __shared__ volatile uint32_t abort_flag;
    const uint32_t bar_q = smem_u32(&bars[0]);
    const uint32_t bar_k = smem_u32(&bars[1]);
    const uint32_t bar_v = smem_u32(&bars[2]);
    const uint32_t bar_s = smem_u32(&bars[3]);
    const uint32_t bar_o = smem_u32(&bars[4]);

    const int tid = threadIdx.x;
    const int warp = uniform(tid >> 5);
    const int qt = p.n_qtiles - 1 - blockIdx.x;  // long (late) tiles first
    const int h = blockIdx.y;
    const int b = blockIdx.z;
    const int hk = h / (p.Hq / p.Hkv);
    const int q0 = qt * kTile;

    if (tid == 0) {
        for (int i = 0; i < 5; ++i) mbar_init(smem_u32(&bars[i]), 1);
        abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tm_q);
        tma_prefetch_desc(&tm_k);
        tma_prefetch_desc(&tm_v);
    }
    if (warp == 0) {
        __syncwarp();
        tmem_alloc(smem_u32(&tmem_holder), 128);
        tmem_relinquish();
    }
    grid_dep_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (p.early_next) grid_dep_launch();
    const uint32_t tmem_base = tmem_holder;
    const uint32_t tS = tmem_base + (static_cast<uint32_t>(warp * 32) << 16);

    constexpr bool kBf16 = std::is_same<T, __nv_bfloat16>::value;
    constexpr uint32_t idesc_qk = instr_desc_f16(kBf16, 128, 128, false, false);
    constexpr uint32_t idesc_pv = instr_desc_f16(kBf16, 128, 64, false, true);

    const int row = q0 + tid;
    bool ok = true;
    // ---- S = Q K^T
    if (tid == 0) {
        mbar_expect_tx(bar_q, kD64TileBytes);
        tma_load_4d(sQ, &tm_q, bar_q, 0, h, q0, b);
        mbar_expect_tx(bar_k, kD64TileBytes);
        tma_load_4d(sK, &tm_k, bar_k, 0, hk, 0, b);
        mbar_expect_tx(bar_v, kD64TileBytes);
        tma_load_4d(sV, &tm_v, bar_v, 0, hk, 0, b);
        ok = mbar_wait(bar_q, 0, &abort_flag, 71) && mbar_wait(bar_k, 0, &abort_flag, 72);
        if (ok) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_ss(tmem_base, smem_desc_sw128(sQ + ks * 32, 16, 1024), smem_desc_sw128(sK + ks * 32, 16, 1024),
                       idesc_qk, ks > 0);
            mma_commit(bar_s);
        }
    }
    __syncwarp();
    // (every thread passes both barriers of the CTA, whatever gave up)
    ok = __all_sync(0xffffffffu, mbar_wait(bar_s, 0, &abort_flag, 73));
    float m = -INFINITY, l = 0.f;
    if (ok) {
        tc_fence_after();
        // ---- mask limit: columns >= lim are past the keys or above the diagonal
        int lim = p.Skv;
        if (p.causal) lim = min(lim, row + p.Skv - p.Sq + 1);
        if (row >= p.Sq) lim = 0;
        const bool full = __all_sync(0xffffffffu, lim >= 128);
        // ---- pass 1: max of the scores
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t r[32];
            tmem_ld_x32(tS + c * 32, r);
            tmem_wait_ld();
            if (full) {
                float m0 = m, m1 = -INFINITY;
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    m0 = max3(m0, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
                    m1 = max3(m1, __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
                }
                m = fmaxf(m0, m1);
            } else {
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    if (c * 32 + i < lim) m = fmaxf(m, __uint_as_float(r[i]));
            }
        }
        const float m_use = (m == -INFINITY) ? 0.f : m;   // rows that see nothing stay finite
        const float neg_ms = -m_use * p.scale_log2;
        // ---- pass 2: P over S's first 64 columns, row sum
        const uint64_t sc2 = f2_pack(p.scale_log2, p.scale_log2), nm2 = f2_pack(neg_ms, neg_ms);
        uint64_t l2 = f2_pack(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t pk[16];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                uint32_t r[16];
                tmem_ld_x16(tS + c * 32 + hf * 16, r);
                tmem_wait_ld();
                const int col0 = c * 32 + hf * 16;
                if (full) {
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        float x0, x1;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), sc2, nm2), x0, x1);
                        const float e0 = fast_exp2(x0), e1 = fast_exp2(x1);
                        l2 = f2_add(l2, f2_pack(e0, e1));
                        pk[hf * 8 + (i >> 1)] = pack2<T>(e0, e1);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float e0 = (col0 + i < lim) ? fast_exp2(fmaf(__uint_as_float(r[i]), p.scale_log2, neg_ms)) : 0.f;
                        const float e1 = (col0 + i + 1 < lim) ? fast_exp2(fmaf(__uint_as_float(r[i + 1]), p.scale_log2, neg_ms)) : 0.f;
                        l += e0 + e1;
                        pk[hf * 8 + (i >> 1)] = pack2<T>(e0, e1);
                    }
                }
            }
            tmem_st_x16(tS + c * 16, pk);
        }
        float la, lb;
        f2_unpack(l2, la, lb);
        l += la + lb;
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    // ---- P V into columns [64,128)
    if (tid == 0 && ok) {
        ok = mbar_wait(bar_v, 0, &abort_flag, 74);
        if (ok) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_ts(tmem_base + 64, tmem_base + ks * 8, smem_desc_sw128(sV + ks * 2048, 16, 1024), idesc_pv, ks > 0);
            mma_commit(bar_o);
        }
    }
    __syncwarp();
    ok = __all_sync(0xffffffffu, ok && mbar_wait(bar_o, 0, &abort_flag, 75));

    if (ok) {
        tc_fence_after();
        uint32_t r0[32], r1[32];   // (all lanes of the warp)
        tmem_ld_x32(tS + 64, r0);
        tmem_ld_x32(tS + 96, r1);
        tmem_wait_ld();
        if (row < p.Sq) {
            float acc[64];
            const float inv_l = (l > 0.f) ? 1.f / l : 0.f;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                acc[i] = __uint_as_float(r0[i]) * inv_l;
                acc[32 + i] = __uint_as_float(r1[i]) * inv_l;
            }
            const long long obase = (long long)b * p.o_sb + (long long)row * p.o_ss + (long long)h * p.o_sh;
            if (p.o_fp32) {
                float4* dst = reinterpret_cast<float4*>(static_cast<float*>(p.o) + obase);
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
            } else {
                uint4* dst = reinterpret_cast<uint4*>(static_cast<T*>(p.o) + obase);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    dst[i] = make_uint4(pack2<T>(acc[8 * i], acc[8 * i + 1]), pack2<T>(acc[8 * i + 2], acc[8 * i + 3]),
                                        pack2<T>(acc[8 * i + 4], acc[8 * i + 5]), pack2<T>(acc[8 * i + 6], acc[8 * i + 7]));
            }
            if (p.lse != nullptr)
                p.lse[((long long)b * p.Hq + h) * p.Sq + row] =
                    (l > 0.f) ? (m * p.scale_log2 + log2f(l)) * 0.6931471805599453f : -INFINITY;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem_base, 128);
    }
}

}  // namespace fa
