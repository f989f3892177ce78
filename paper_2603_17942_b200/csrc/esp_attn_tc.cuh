// Device-side pieces of the tensor-core tree attention (bf16, head_dim 128) shared by the kernels that
// run it: the work of one item (one split of the cache x one KV head x one tile of 128 (row, head) pairs)
// on the tcgen05 path, and the per-(row, head) tail and merge.  The kernel that runs one attention per
// launch and the kernel that runs all layers in one launch call the same functions and give the same bits.
#pragma once

#include "esp_launch.h"
#include "esp_tc.cuh"

namespace esp {
namespace attn {

using namespace tc;

constexpr int HD = 128;
constexpr int CK = 128;                   // keys per chunk
constexpr int MP = 128;                   // (row, head) pairs per CTA
constexpr int HALF_BYTES = 128 * 128;     // one 128-row x 64-element (128-byte) swizzled tile
constexpr int Q_BYTES = 2 * HALF_BYTES, K_BYTES = 2 * HALF_BYTES, V_BYTES = 2 * HALF_BYTES;
constexpr int KV_STAGE = K_BYTES + V_BYTES;
constexpr int OFF_Q = 0, OFF_KV = Q_BYTES;
constexpr int ITEM_BYTES = OFF_KV + 2 * KV_STAGE;   // shared memory one item needs: Q, two K/V stages
constexpr int TMEM_COLS = 512;            // S0 at 0, S1 at 128, O0 at 256, O1 at 384; P of a chunk in the first 64 columns of its S

__device__ __forceinline__ int tail_start_tc(int P, int dcap) {
    int t = P - dcap;
    return t <= 0 ? 0 : (t / 16) * 16;
}

// kind::f16 instruction descriptors: D = f32, A = B = bf16, M = 128, N = 128; PV takes B (V) MN-major
constexpr uint32_t IDESC_QK = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
constexpr uint32_t IDESC_PV = IDESC_QK | (1u << 16);

// 64 consecutive columns of this lane: two loads in flight, one wait
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t (&r)[64]) {
    tmem_ld32_issue(taddr, &r[0]);
    tmem_ld32_issue(taddr + 32, &r[32]);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The producer thread waits for the kernel before this one and only then releases the kernel after it.
__device__ __forceinline__ void trigger_after_wait() {
    pdl_wait();
    pdl_launch_dependents();
}

// 2^x as one special-function instruction (results below 2^-126 flush to zero, which a softmax weight may;
// relative error about 2^-22).  Measured against exp2f(): 0.64 instead of 0.70 us for the 64 exponentials of a chunk.
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Pairs of floats as one operand of the packed instructions (each element rounded like its scalar form).
__device__ __forceinline__ uint64_t pack2(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// ---- one 128-key chunk of the online softmax, for one thread = one half (64 keys) of one pair's row.
// S (raw scores) is read from tensor memory; keys at or beyond T0row are masked; the two threads of a pair
// exchange their maxima through `xch` ([2 * MP] floats); P goes back to tensor memory as bf16 pairs, over the scores it
// came from (the A operand of P V; S of this chunk is in both threads' registers before the exchange ends), 32 columns
// per half (P through shared memory took a proxy fence and 16 KB of stores per tile and chunk: operator at 16 x 4k 203 us
// against 189 now, batch 1 38.9 against 36.6); O is rescaled in tensor memory when the running maximum moved.  Scores enter the exponent as
// fma(s, scale, -m): one rounding, spelled out so that every kernel that inlines this rounds alike.
// All 32 lanes of a warp call this together (the tensor-memory accesses are warp-wide); false = a wait ran out.
__device__ __forceinline__ bool softmax_chunk(uint32_t s_addr, uint32_t o_addr, int cbase, int T0row, float scale_log2, float& m_run,
                                              float& l_run, float* xch, uint64_t* xchg, uint32_t xchg_parity, bool wait_pv,
                                              uint64_t* pv_done, uint32_t pv_parity, bool rescale, int pair,
                                              int hf, uint64_t* p_ready, volatile int* s_abort) {
    uint32_t sv[64];
    tmem_ld64(s_addr, sv);
    if (!__all_sync(0xffffffffu, cbase + 64 <= T0row)) {     // otherwise every key of the half is visible to every row of the warp
#pragma unroll
        for (int i = 0; i < 64; ++i) sv[i] = cbase + i < T0row ? sv[i] : 0xff800000u;
    }
    float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};     // four chains: one takes 64 dependent steps
#pragma unroll
    for (int i = 0; i < 64; i += 8)
#pragma unroll
        for (int j = 0; j < 4; ++j) m4[j] = fmaxf(fmaxf(m4[j], __uint_as_float(sv[i + 2 * j])), __uint_as_float(sv[i + 2 * j + 1]));
    float cmax = __fmul_rn(fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])), scale_log2);     // in the log2 domain (scaling is monotone)
    // the chunk maximum over both halves
    // (double buffered by exchange parity: a thread can be one exchange ahead of its partner, not two)
    // (one arrival per warp, after the warp's values are in shared memory: 256 single arrivals on one barrier
    // word take several hundred cycles)
    xch[hf * MP + pair] = cmax;
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(xchg);
    if (!__all_sync(0xffffffffu, mbar_wait(xchg, xchg_parity, s_abort))) return false;
    cmax = fmaxf(xch[pair], xch[MP + pair]);
    // The running reference follows the maximum lazily: it moves only when the maximum has grown by more than
    // 2^8 over it (or there was none yet).  Until then alpha is exactly 1, O needs no rescaling, and the
    // probabilities of this chunk are at most 2^8, exact in fp32 and as precise as ever in bf16.  The decision is
    // the row's own (both threads of the pair see the same maximum), so a row's bits stay independent of its
    // neighbours; whoever merges the partial takes m_run as what it is, the reference of l and O.
    const float m_max = fmaxf(m_run, cmax);
    const float m_new = (m_run == -INFINITY || __fsub_rn(m_max, m_run) > 8.f) ? m_max : m_run;
    const float m_use = m_new == -INFINITY ? 0.f : m_new;
    const float alpha = exp2f(__fsub_rn(m_run, m_use));
    // probabilities, packed as bf16 pairs, and their sums over the even and the odd keys
    const uint64_t scale2 = pack2(scale_log2, scale_log2), neg_m2 = pack2(-m_use, -m_use);
    uint64_t csum2 = 0;
    uint32_t pk[32];
#pragma unroll
    for (int i = 0; i < 64; i += 2) {
        float p0, p1;
        unpack2(fma2(pack2(__uint_as_float(sv[i]), __uint_as_float(sv[i + 1])), scale2, neg_m2), p0, p1);
        p0 = ex2_approx(p0);
        p1 = ex2_approx(p1);
        csum2 = add2(csum2, pack2(p0, p1));
        const __nv_bfloat162 b2 = __floats2bfloat162_rn(p0, p1);
        pk[i >> 1] = *reinterpret_cast<const uint32_t*>(&b2);
    }
    float c0, c1;
    unpack2(csum2, c0, c1);
    const float csum = __fadd_rn(c0, c1);
    // (the values are pinned here: without it the compiler is free to sink the arithmetic behind the wait)
#pragma unroll
    for (int i = 0; i < 32; ++i) asm volatile("" : "+r"(pk[i]));
    // O must be final before it is rescaled (and no warp may signal this chunk's P before the previous chunk's was taken)
    if (wait_pv && !__all_sync(0xffffffffu, mbar_wait(pv_done, pv_parity, s_abort))) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tmem_st32(s_addr - hf * 32, pk);      // s_addr: column 64 * hf of S
    if (rescale) {
        // O <- alpha * O (in tensor memory), this thread's 64 of the 128 columns
        if (__any_sync(0xffffffffu, alpha != 1.0f)) {   // warp-uniform: skip when no lane's maximum moved
            tmem_ld64(o_addr, sv);
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {
#pragma unroll
                for (int i = 0; i < 32; ++i) sv[blk * 32 + i] = __float_as_uint(__fmul_rn(__uint_as_float(sv[blk * 32 + i]), alpha));
                tmem_st32(o_addr + blk * 32, *reinterpret_cast<const uint32_t(*)[32]>(&sv[blk * 32]));
            }
        }
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    l_run = __fmaf_rn(l_run, alpha, csum);     // this half's share of the row sum
    m_run = m_new;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(p_ready);      // one arrival per softmax warp
    return true;
}

// The same step for a softmax warp none of whose 32 lanes has a pair (the last row tile of a block is rarely full: 68
// rows x 4 heads leave 16 pairs in the third tile): no scores, no exponentials -- its rows of P and O are never used,
// whatever they hold --, only its arrival, behind the previous chunk's P V so that it cannot run a phase ahead.
__device__ __forceinline__ bool softmax_chunk_idle(bool wait_pv, uint64_t* pv_done, uint32_t pv_parity, uint64_t* p_ready, volatile int* s_abort) {
    if (wait_pv && !__all_sync(0xffffffffu, mbar_wait(pv_done, pv_parity, s_abort))) return false;
    if ((threadIdx.x & 31) == 0) mbar_arrive(p_ready);
    return true;
}

// ---- one item, start to finish, on freshly initialised barriers.
struct BulkMaps {
    const CUtensorMap* q;   // [rows][Hq][128], box 64 x group x rows_per_tile
    const CUtensorMap* k;   // [cache rows][128], box 64 x 128 keys
    const CUtensorMap* v;
    int group, rows_per_tile;
};
struct BulkItem {
    int split, kvh, seq, row0, n_rows, L, beg, n_chunks;
    int kv_row0;            // row of position 0 of this (sequence, KV head) in the K/V maps
};
struct BulkShared {
    unsigned char* buf;     // 1024-byte aligned, ITEM_BYTES
    uint64_t *k_full, *k_empty, *v_full, *v_empty, *s_full;   // [2] each, count 1
    uint64_t *q_full, *pv_done;              // count 1
    uint64_t* p_ready;                       // count 8: one arrival per softmax warp
    uint64_t* xchg;                          // [4], count 2: the two warps that share a tensor-memory lane quadrant
    float* s_xchg;          // [2][2 * MP]
    volatile int* s_abort;
};
__device__ __forceinline__ void bulk_init_barriers(const BulkShared& sm) {
    for (int i = 0; i < 2; ++i) {
        mbar_init(&sm.k_full[i], 1); mbar_init(&sm.k_empty[i], 1); mbar_init(&sm.v_full[i], 1); mbar_init(&sm.v_empty[i], 1);
        mbar_init(&sm.s_full[i], 1);
    }
    mbar_init(sm.q_full, 1);
    mbar_init(sm.p_ready, 8);
    mbar_init(sm.pv_done, 1);
    for (int i = 0; i < 4; ++i) mbar_init(&sm.xchg[i], 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Roles: warp 0 TMA producer, warp 1 MMA issuer, warps 2..9 softmax (two threads per pair, 64 keys each; they also
// write the item's partial output).  Other warps fall through.  PDL: the kernel is one link of a chain of
// programmatic dependent launches (the producer thread does the wait and releases the dependent kernel).
template <bool PDL>
__device__ __forceinline__ void bulk_item_roles(const BulkMaps& mp, const AttnArgs& a, const BulkItem& it, const BulkShared& sm,
                                                uint32_t tmem_base, int warp, int lane) {
    unsigned char* smem = sm.buf;
    unsigned char* sQ = smem + OFF_Q;
    volatile int* s_abort = sm.s_abort;
    if (warp == 0) {
        // ---------------- TMA producer
        if (lane == 0) {
            const int kvrow0 = it.kv_row0 + it.beg;
            bool ok = true;
            // K and V of a chunk have a stage half and a barrier pair each: a K half is free again when its Q K^T has
            // completed, about one chunk period before the V half (free when P V has), so K runs one chunk ahead of V
            // and both have two chunk periods for their trip from HBM
            auto load_k = [&](int c) -> bool {
                if (!mbar_wait(&sm.k_empty[c & 1], ((c >> 1) & 1) ^ 1, s_abort)) return false;   // a fresh barrier passes parity 1
                unsigned char* st = smem + OFF_KV + (c & 1) * KV_STAGE;
                mbar_expect_tx(&sm.k_full[c & 1], K_BYTES);
                tma_load_2d(st, mp.k, 0, kvrow0 + c * CK, &sm.k_full[c & 1]);
                tma_load_2d(st + HALF_BYTES, mp.k, 64, kvrow0 + c * CK, &sm.k_full[c & 1]);
                return true;
            };
            auto load_v = [&](int c) -> bool {
                if (!mbar_wait(&sm.v_empty[c & 1], ((c >> 1) & 1) ^ 1, s_abort)) return false;
                unsigned char* st = smem + OFF_KV + (c & 1) * KV_STAGE + K_BYTES;
                mbar_expect_tx(&sm.v_full[c & 1], V_BYTES);
                tma_load_2d(st, mp.v, 0, kvrow0 + c * CK, &sm.v_full[c & 1]);
                tma_load_2d(st + HALF_BYTES, mp.v, 64, kvrow0 + c * CK, &sm.v_full[c & 1]);
                return true;
            };
            // the cache below T0 is settled in a decode step: request it before waiting for the kernel that wrote the queries
            if (PDL && a.cache_in_flight) trigger_after_wait();
            const int n = it.n_chunks;
            ok = load_k(0) && (n < 2 || load_k(1)) && load_v(0) && (n < 2 || load_v(1));    // both stages are free
            if (PDL && !a.cache_in_flight) trigger_after_wait();
            mbar_expect_tx(sm.q_full, Q_BYTES);
            tma_load_3d(sQ, mp.q, 0, it.kvh * mp.group, it.seq * RT + it.row0, sm.q_full);
            tma_load_3d(sQ + HALF_BYTES, mp.q, 64, it.kvh * mp.group, it.seq * RT + it.row0, sm.q_full);
            if (ok && n > 2) ok = load_k(2);
            for (int c = 2; c < n && ok; ++c) ok = (c + 1 >= n || load_k(c + 1)) && load_v(c);
            if (!ok) { set_error(a.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        const bool leader = elect_lane();
        {
            bool ok = true;
            const uint32_t q_addr = smem_u32(sQ);
            auto issue_qk = [&](int c) {
                const uint32_t k_addr = smem_u32(smem + OFF_KV + (c & 1) * KV_STAGE);
                const uint32_t tmem_s = tmem_base + (c & 1) * 128;
#pragma unroll
                for (int kk = 0; kk < HD / 16; ++kk) {
                    const uint32_t off = (kk >> 2) * HALF_BYTES + (kk & 3) * 32;
                    if (leader) umma(tmem_s, smem_desc(q_addr + off, 16), smem_desc(k_addr + off, 16), IDESC_QK, kk > 0 ? 1u : 0u);
                }
                if (leader) umma_commit(&sm.s_full[c & 1]);
                if (leader) umma_commit(&sm.k_empty[c & 1]);
            };
            ok = __all_sync(0xffffffffu, mbar_wait(sm.q_full, 0, s_abort) && mbar_wait(&sm.k_full[0], 0, s_abort));
            if (ok) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                issue_qk(0);
            }
            for (int c = 0; c < it.n_chunks && ok; ++c) {
                if (c + 1 < it.n_chunks) {     // S of the next chunk while the softmax of this one runs
                    if (!__all_sync(0xffffffffu, mbar_wait(&sm.k_full[(c + 1) & 1], ((c + 1) >> 1) & 1, s_abort))) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    issue_qk(c + 1);
                }
                if (!__all_sync(0xffffffffu, mbar_wait(sm.p_ready, c & 1, s_abort) && mbar_wait(&sm.v_full[c & 1], (c >> 1) & 1, s_abort))) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t v_addr = smem_u32(smem + OFF_KV + (c & 1) * KV_STAGE + K_BYTES);
#pragma unroll
                for (int kk = 0; kk < CK / 16; ++kk) {
                    const uint32_t v_off = kk * 16 * 128;                              // V: 16 key rows of 128 bytes further
                    if (leader) umma_ta(tmem_base + 256, tmem_base + (c & 1) * 128 + kk * 8, smem_desc(v_addr + v_off, HALF_BYTES), IDESC_PV,
                            (c > 0 || kk > 0) ? 1u : 0u);
                }
                if (leader) umma_commit(sm.pv_done);
                if (leader) umma_commit(&sm.v_empty[c & 1]);
            }
            // the arrivals on the K/V stage barriers are the item's last asynchronous ones: see them land, so that
            // a kernel that runs several items may initialise the barriers again
            for (int c = it.n_chunks - 2 < 0 ? 0 : it.n_chunks - 2; c < it.n_chunks && ok; ++c)
                ok = __all_sync(0xffffffffu, mbar_wait(&sm.k_empty[c & 1], (c >> 1) & 1, s_abort) && mbar_wait(&sm.v_empty[c & 1], (c >> 1) & 1, s_abort));
            if (!ok) { set_error(a.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
        }
    } else if (warp < 10) {
        // ---------------- softmax warps 2..9: a thread owns one pair (= tensor-memory lane) and one half of the
        // chunk's 128 keys (warps 2-5 keys 0..63, warps 6-9 keys 64..127); the two threads of a pair exchange
        // their maxima (per chunk) and their sums (at the end) through shared memory
        const int q4 = warp & 3;
        const int hf = (warp - 2) >> 2;
        const int pair = q4 * 32 + lane;
        const int r = it.row0 + pair / mp.group, head = it.kvh * mp.group + pair % mp.group;
        const bool pv = pair / mp.group < mp.rows_per_tile && r < it.n_rows && r < RT;
        int T0row = 0;
        if (pv) T0row = tail_start_tc(it.L + (a.st ? a.st[it.seq].row_depth[r] : a.depth[it.seq * RT + r]), a.dcap);
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16) + hf * 64;   // this thread's 64 columns of S / O
        float m_run = -INFINITY, l_run = 0.f;
        bool ok = true;
        const bool live = __any_sync(0xffffffffu, pv);      // the same for the two warps that share the lanes' pairs
        for (int c = 0; c < it.n_chunks && ok; ++c) {
            if (!live) {
                ok = softmax_chunk_idle(c > 0, sm.pv_done, (c - 1) & 1, sm.p_ready, s_abort);
                continue;
            }
            // (a wait that fails must take the whole warp out: the tensor-memory accesses below are warp-wide)
            if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full[c & 1], (c >> 1) & 1, s_abort))) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            ok = softmax_chunk(lane_addr + (c & 1) * 128, lane_addr + 256, it.beg + c * CK + hf * 64, T0row, a.scale_log2, m_run, l_run,
                               sm.s_xchg + (c & 1) * 2 * MP, sm.xchg + q4, c & 1, c > 0, sm.pv_done, (c - 1) & 1, c > 0,
                               pair, hf, sm.p_ready, s_abort);
        }
        if (ok && !__all_sync(0xffffffffu, mbar_wait(sm.pv_done, (it.n_chunks - 1) & 1, s_abort))) ok = false;
        float* xl = sm.s_xchg + (it.n_chunks & 1) * 2 * MP;
        if (ok && live) {
            // the row sum = first half's share + second half's share
            xl[hf * MP + pair] = l_run;
            __syncwarp();
            if (lane == 0) mbar_arrive(sm.xchg + q4);
            if (!__all_sync(0xffffffffu, mbar_wait(sm.xchg + q4, it.n_chunks & 1, s_abort))) ok = false;
        }
        if (ok && live) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // O half-row -> shared memory (the K/V stages are free now) -> one 256-byte bulk copy per thread.  The
            // tensor-memory load is warp-wide: every lane takes part, lanes without a pair copy nothing.
            uint32_t ov[64];
            tmem_ld64(lane_addr + 256, ov);
            float* orow = reinterpret_cast<float*>(smem + OFF_KV) + pair * (HD + 4) + hf * 64;   // rows padded by 16 bytes: no bank conflicts
#pragma unroll
            for (int i = 0; i < 64; i += 4)
                *reinterpret_cast<uint4*>(orow + i) = make_uint4(ov[i], ov[i + 1], ov[i + 2], ov[i + 3]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (pv) {
                const size_t idx = ((size_t)(it.seq * RT + r) * a.Hq + head) * a.n_split_max + it.split;
                if (hf == 0) __stcg(a.part_ml + idx, make_float2(m_run, __fadd_rn(xl[pair], xl[MP + pair])));
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                             ::"l"(a.part_o + idx * HD + hf * 64), "r"(smem_u32(orow)), "r"(64 * 4) : "memory");
            }
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            // shared memory may be released when it has been read; the end of the kernel, where there is one, completes the copies
            if (PDL) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            else asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        } else if (!ok && lane == 0) {
            set_error(a.err, DEV_E_WAIT_TIMEOUT);
            *s_abort = 1;
        }
    }
}

// ---- tail + merge: one warp per task = up to TG query heads of one row that share a KV head
// The tail of a row: positions T0..P in position order, in chunks of 32 keys anchored at T0 (one chunk for dcap 16).  Keys
// below L are cache positions, the others block rows found through the row's ancestor mask, so every row has a key list of
// its own: a gather, for which the list has to reach registers, and then a contraction of 4 heads x 32 keys x 128 dims
// that mma.sync takes without staging anything (tcgen05 wants its operands in shared memory, 128 rows at a time).
//   S = Q K^T   m16n8k16, rows 0..3 and again 4..7 the heads, columns the keys of an 8-key tile; the 128 dims are dealt to
//               the k-steps so that a lane's 16-byte pieces of Q and K are its fragments as they come from memory;
//   softmax     a lane holds 8 keys of head (lane / 4) % 4, lanes 4 apart share a row; both copies compute the same;
//   O = P V     P in three bf16 pieces (hi + mid + lo = the 24 bits of the fp32 weight, products exact): hi in rows 0..3,
//               mid in rows 4..7, lo in rows 8..11 of ONE A operand; V's 8 x 8 blocks are transposed in registers.
// Every sum's order follows from the position in the list alone.  (The additions inside one mma.sync are not rounded one by one as a chain
// of multiply-adds is.  Error of o / l against 64 bits, 2-norm, chain / this: scores of deviation 0.3 1.19 / 0.81e-7, 1 1.66 / 1.57e-7, 3 2.48 /
// 2.29e-7, 10 3.60 / 2.82e-7; values all positive 0.98 / 0.81, 1.43 / 1.81 and 2.15 / 2.07e-7 at deviations 1, 3 and 10.)
// A KV head of a single query head leaves three of the four places empty: launches of more than 12000 (row, head) pairs then take
// 1.05 to 1.3 times as long as the kernel before this one, smaller ones and deep trees less.  What bounded the kernels before this one was their
// instruction count and a chain of dependent trips: a warp per (row, head) gathered its keys 32 cache lines per load
// (8.6 us a task), a CTA with the keys in shared memory spent about 1700 instructions per task of four heads.
constexpr int TG = 4;
__host__ __device__ constexpr int tail_heads(int group) { return group % 4 == 0 ? 4 : (group % 2 == 0 ? 2 : 1); }

struct TailTask {           // heads head0 .. head0 + gh - 1 (gh <= TG) of one row of one sequence
    int r, head0, gh, seq, L, depth;
    unsigned long long lo, hi;   // the row's ancestor-or-self mask over block rows
};
// A lane's share: head (lane / 4) % 4 of the task, dims 64 * (lane / 16) + 32 * j + 8 * (lane % 4) + 0..7, j = 0, 1
struct TailAcc {
    float m, l, o[16];
};

__device__ __forceinline__ int nth_set_bit128(unsigned long long lo, unsigned long long hi, int n) {
    int c = __popcll(lo);
    unsigned long long m = lo;
    int base = 0;
    if (n >= c) { n -= c; m = hi; base = 64; }
    for (int i = 0; i < n; ++i) m &= m - 1;
    return m ? base + __ffsll((long long)m) - 1 : -1;
}
__device__ __forceinline__ void merge_ml(float& m, float& l, float (&o)[16], float cm, float cl, const float (&co)[16]) {
    // products and sums are rounded one by one, so that every instance of the kernel rounds alike
    const float mn = fmaxf(m, cm);
    const float a = exp2f(__fsub_rn(m, mn)), b = exp2f(__fsub_rn(cm, mn));
    l = __fmaf_rn(l, a, __fmul_rn(cl, b));
#pragma unroll
    for (int i = 0; i < 16; ++i) o[i] = __fmaf_rn(o[i], a, __fmul_rn(co[i], b));
    m = mn;
}
// D += A B, 16 x 8 x 16, bf16 in, fp32 accumulators
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the warp's 8 x 8 block of 16-bit values (lane l: row l / 4, columns 2 * (l % 4), + 1), transposed
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x) {
    uint32_t y;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&b);
}

// What this step wrote shortly before, in another kernel or CTA -- the queries and the keys / values of the block's own
// rows (slots >= L) -- is read with L2 loads (ld.global.cg), never through L1; cache positions below L were written by
// earlier steps (unless a.cache_in_flight) and go through L1, where the tasks that share a KV head find them again.
__device__ __forceinline__ uint4 load_kv16(const __nv_bfloat16* p, bool settled) {
    return settled ? *reinterpret_cast<const uint4*>(p) : __ldcg(reinterpret_cast<const uint4*>(p));
}

// The slot of key t of the row's list (position T0 + t), -1 if the ancestor mask does not name it.
__device__ __forceinline__ int tail_slot(const TailTask& c, int pos) {
    if (pos < c.L) return pos;
    const int b = nth_set_bit128(c.lo, c.hi, pos - c.L);
    return b < 0 ? -1 : c.L + b;
}

// JB: 32-dim columns of the keys, and then of the values, requested at once; 4: all of both ahead of any use (160 registers).
template <int JB>
__device__ __forceinline__ void tail_task(TailAcc& t, const AttnArgs& a, const TailTask& c, int lane) {
    const int kvh = c.head0 / (a.Hq / a.Hkv);
    const int P = c.L + c.depth, T0 = tail_start_tc(P, a.dcap);
    const size_t kv0 = ((size_t)(a.kv_shared ? 0 : c.seq) * a.Hkv + kvh) * a.cap * HD;
    const int g = lane >> 2, c4 = lane & 3;
    const __nv_bfloat16* kbase = reinterpret_cast<const __nv_bfloat16*>(a.kc) + kv0 + c4 * 8;
    const __nv_bfloat16* vbase = reinterpret_cast<const __nv_bfloat16*>(a.vc) + kv0 + c4 * 8;
    const int head = c.head0 + min(g & 3, c.gh - 1);
    const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(a.q) + ((size_t)(c.seq * RT + c.r) * a.Hq + head) * HD + c4 * 8;
    uint4 qf[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) qf[j] = __ldcg(reinterpret_cast<const uint4*>(q + j * 32));
    t.m = -INFINITY; t.l = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) t.o[i] = 0.f;
    const int n_tail = P - T0 + 1;
#pragma unroll 1
    for (int t0 = 0; t0 < n_tail; t0 += 32) {
        int slot = -1;
        if (t0 + lane < n_tail) {
            slot = tail_slot(c, T0 + t0 + lane);
            if (slot < 0) set_error(a.err, DEV_E_INDEX);
        }
        // a key that is not in the chunk takes the place of one that is, with weight 0: nothing else is read
        const uint32_t in = __ballot_sync(0xffffffffu, slot >= 0);
        const int any = in ? __shfl_sync(0xffffffffu, slot, __ffs(in) - 1) : 0;
        if (slot < 0) slot = any;
        int sl[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) sl[n] = __shfl_sync(0xffffffffu, slot, n * 8 + g);
        auto load4x = [&](uint4 (&f)[4], const __nv_bfloat16* base, int j) {      // column j of this lane's four keys
#pragma unroll
            for (int n = 0; n < 4; ++n) f[n] = load_kv16(base + (size_t)sl[n] * HD + j * 32, sl[n] < c.L && !a.cache_in_flight);
        };
        uint4 kf[JB][4], vf[JB][4];
        float s[4][4];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
#pragma unroll
            for (int i = 0; i < 4; ++i) s[n][i] = 0.f;
        }
#pragma unroll
        for (int j0 = 0; j0 < 4; j0 += JB) {
#pragma unroll
            for (int j = 0; j < JB; ++j) load4x(kf[j], kbase, j0 + j);
            if (JB == 4) {
#pragma unroll
                for (int j = 0; j < JB; ++j) load4x(vf[j], vbase, j);
            }
#pragma unroll
            for (int j = 0; j < JB; ++j)
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    mma16816(s[n], qf[j0 + j].x, 0u, qf[j0 + j].y, 0u, kf[j][n].x, kf[j][n].y);
                    mma16816(s[n], qf[j0 + j].z, 0u, qf[j0 + j].w, 0u, kf[j][n].z, kf[j][n].w);
                }
        }
        // softmax over the chunk: this lane's keys are t0 + 8 n + 2 c4 + e
        float cm = -INFINITY;
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool ok = (in >> (8 * n + 2 * c4 + e)) & 1u;
                s[n][e] = ok ? __fmul_rn(s[n][e], a.scale_log2) : -INFINITY;
                cm = fmaxf(cm, s[n][e]);
            }
        cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, 1));
        cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, 2));
        float cl = 0.f;
        uint32_t pa[4][2];          // rows g and g + 8 of the A operand: hi and lo pieces (lanes 0..15), mid and nothing (16..31)
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            float hi[2], mid[2], lo[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool ok = (in >> (8 * n + 2 * c4 + e)) & 1u;
                const float p = ok ? exp2f(__fsub_rn(s[n][e], cm)) : 0.f;
                cl = __fadd_rn(cl, p);
                hi[e] = __bfloat162float(__float2bfloat16_rn(p));
                const float r1 = __fsub_rn(p, hi[e]);
                mid[e] = __bfloat162float(__float2bfloat16_rn(r1));
                lo[e] = __fsub_rn(r1, mid[e]);
            }
            pa[n][0] = lane < 16 ? pack_bf16(hi[0], hi[1]) : pack_bf16(mid[0], mid[1]);
            pa[n][1] = lane < 16 ? pack_bf16(lo[0], lo[1]) : 0u;
        }
        cl = __fadd_rn(cl, __shfl_xor_sync(0xffffffffu, cl, 1));
        cl = __fadd_rn(cl, __shfl_xor_sync(0xffffffffu, cl, 2));
        float co[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (JB < 4 && j % JB == 0) {
#pragma unroll
                for (int u = 0; u < JB; ++u) load4x(vf[u], vbase, j + u);
            }
            float d[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
#pragma unroll
                for (int i = 0; i < 4; ++i) d[r][i] = 0.f;
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {       // 16 keys per step
                const uint4 x0 = vf[j % JB][2 * k], x1 = vf[j % JB][2 * k + 1];
                const uint32_t v0[4] = {x0.x, x0.y, x0.z, x0.w}, v1[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    mma16816(d[r], pa[2 * k][0], pa[2 * k][1], pa[2 * k + 1][0], pa[2 * k + 1][1], transpose8x8(v0[r]), transpose8x8(v1[r]));
            }
            // d[r]: dims 32 j + 8 c4 + 2 r, + 1; rows g (hi, or mid) and g + 8 (lo).  Lanes 0..15 keep j = 0, 1, the others 2, 3.
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float v = __fadd_rn(d[r][e], d[r][2 + e]);
                    const float w = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 16));
                    if ((j >> 1) == 0) { if (lane < 16) co[(j & 1) * 8 + 2 * r + e] = w; }
                    else { if (lane >= 16) co[(j & 1) * 8 + 2 * r + e] = w; }
                }
        }
        // A piece of weight 0 times an infinite value is a NaN that the whole weight would not have given: sums that are not finite are
        // taken again, key by key with the whole weight (hi + mid + lo, exact), keys without weight (below 2^-133, the least of bf16)
        // left out.
        float odd = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) odd = __fmaf_rn(co[i], 0.f, odd);       // 0 x inf and 0 x NaN are NaN
        if (__any_sync(0xffffffffu, odd != 0.f)) {
#pragma unroll
            for (int i = 0; i < 16; ++i) co[i] = 0.f;
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll 1
                for (int k = 0; k < 8; ++k) {
                    const int from = (lane & 12) | (k >> 1), sh = 16 * (k & 1);      // who holds key 8 n + k of this lane's head
                    const uint32_t hi = __shfl_sync(0xffffffffu, pa[n][0], from) >> sh, mid = __shfl_sync(0xffffffffu, pa[n][0], 16 + from) >> sh,
                                   lo = __shfl_sync(0xffffffffu, pa[n][1], from) >> sh;
                    const float p = __fadd_rn(__fadd_rn(__uint_as_float(hi << 16), __uint_as_float(mid << 16)), __uint_as_float(lo << 16));
                    const __nv_bfloat16* vr = vbase + (size_t)__shfl_sync(0xffffffffu, slot, 8 * n + k) * HD + (lane >> 4) * 64;
                    if (p != 0.f) {
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const uint4 x = __ldcg(reinterpret_cast<const uint4*>(vr + j * 32));
                            const uint32_t v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                            for (int i = 0; i < 8; ++i) co[j * 8 + i] = __fmaf_rn(p, __uint_as_float(i & 1 ? v[i >> 1] & 0xffff0000u : v[i >> 1] << 16), co[j * 8 + i]);
                        }
                    }
                }
        }
        merge_ml(t.m, t.l, t.o, cm, cl, co);
    }
}

// The output of a task, o / l, as bf16 and (a.out_lo) its low-order plane.
__device__ __forceinline__ void store_task(float l, const float (&o)[16], const AttnArgs& a, const TailTask& c, int lane) {
    if (((lane >> 2) & 3) >= c.gh) return;
    const float inv = 1.0f / l;
    const size_t at = ((size_t)(c.seq * RT + c.r) * a.Hq + c.head0 + ((lane >> 2) & 3)) * HD + (lane >> 4) * 64 + (lane & 3) * 8;
    __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(a.out) + at;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        __align__(16) __nv_bfloat16 oh[8], ol[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float v = __fmul_rn(o[j * 8 + i], inv);
            oh[i] = __float2bfloat16_rn(v);
            ol[i] = __float2bfloat16_rn(__fsub_rn(v, __bfloat162float(oh[i])));
        }
        // (a caller's `out` needs no more than 8 bytes; queries and cache are under the tensor maps' 16)
        *reinterpret_cast<uint2*>(out + j * 32) = *reinterpret_cast<const uint2*>(oh);
        *reinterpret_cast<uint2*>(out + j * 32 + 4) = *reinterpret_cast<const uint2*>(oh + 4);
        if (a.out_lo)      // low-order plane for an O projection that reads the output as hi + lo
            *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.out_lo) + at + j * 32) = *reinterpret_cast<const uint4*>(ol);
    }
}

// The merge: bulk partials in split order, the tail last.  PB splits are requested before they are used.
template <int PB>
__device__ __forceinline__ void merge_task(const TailAcc& t, const AttnArgs& a, const TailTask& c, int lane) {
    const int n_sp = (tail_start_tc(c.L + c.depth, a.dcap) + a.split_len - 1) / a.split_len;
    const int head = c.head0 + min((lane >> 2) & 3, c.gh - 1);
    const size_t base = ((size_t)(c.seq * RT + c.r) * a.Hq + head) * a.n_split_max;
    const float* po = a.part_o + base * HD + (lane >> 4) * 64 + (lane & 3) * 8;
    float m = -INFINITY, l = 0.f, o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) o[i] = 0.f;
#pragma unroll 1
    for (int s0 = 0; s0 < n_sp; s0 += PB) {
        float2 ml[PB];
        float co[PB][16];
#pragma unroll
        for (int u = 0; u < PB; ++u) {
            if (s0 + u < n_sp) {
                ml[u] = __ldcg(a.part_ml + base + s0 + u);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    *reinterpret_cast<float4*>(&co[u][i * 4]) =
                        __ldcg(reinterpret_cast<const float4*>(po + (size_t)(s0 + u) * HD + (i >> 1) * 32 + (i & 1) * 4));
            }
        }
#pragma unroll
        for (int u = 0; u < PB; ++u)
            if (s0 + u < n_sp) merge_ml(m, l, o, ml[u].x, ml[u].y, co[u]);
    }
    merge_ml(m, l, o, t.m, t.l, t.o);
    store_task(l, o, a, c, lane);
}

}  // namespace attn
}  // namespace esp
