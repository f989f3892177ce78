// bf16 GEMM over several blocks of rows at once -- the full blocks of a prompt, or the blocks of several sequences in a
// decode step -- on the Blackwell tensor cores: y[row][n] = sum_k (x_hi[row][k] + x_lo[row][k]) * w[n][k], fp32
// accumulation, both planes of the activations (see esp_gemm_tc.cu) into one accumulator.
//
// With hundreds of rows per weight stream the work is a matter of the tensor cores, and what has to be kept up is
// their operand supply: shared memory delivers 128 bytes per clock, an MMA of N = 240 takes 98 of them for its
// operands, and what a tile needs from L2 passes through the same port.  A 256-feature x 240-row tile needs 32 KB of
// weights and 60 KB of activations per 64 k for 16 MMAs of N = 240 (48 bytes per clock); a 128-feature tile, as the
// small-M kernel has it, would need 79.  The tile is the whole tensor memory (two accumulators of up to 240 of 256
// columns), so there is one in flight per CTA.
//
// Work split: a row tile is BPT blocks of WB rows (one TMA box of BPT x WB rows per plane).  The (256-feature tile,
// k-block) units are cut into contiguous ranges, stream-K style; an item is a range x a row tile, the items of a range lie
// next to each other in the grid, and their CTAs walk it in step, so that a weight unit is read from HBM once and from L2
// by the other row tiles.  Every piece is stored as an fp32 partial; the kernel that consumes the result sums a tile's
// pieces in range order, as it does for the small-M kernel (StreamK with one row space for all row tiles).
// The number of ranges (WIDE_SM over row tiles of split_bpt blocks) depends on the number of blocks and not on the rows of
// a block: a row's sums have the same order in a step of 128-row trees and in a greedy step.  With BPT = split_bpt every
// CTA has one item; 128-row blocks of which two make a row tile where smaller ones would be three take two turns.
// A decode step in which some of the pass's sequences take no part: k_gemm_wide_some, below, over the blocks of those that do.
//
// Ring: seven slots of 32 KB, filled in the order [two weight units | hi rows | lo rows] per k-block.  The hi slot is
// released half a k-block before the other two.  Roles: warp 0 producer, warp 1 MMA issuer, warps 2-9 epilogue (four
// per accumulator).  Every mbarrier wait is bounded, as in esp_gemm_tc.cu.
//
// Measured, 960 rows (eight prefill blocks) of an 8B layer, on their own: QKV 71, O 52, gate/up 280, down 145 us = 1.24 to
// 1.61 PFLOP/s of two-plane products, 0.75 to 0.98 of the measured cuBLAS rate; eight passes of the small-M kernel took
// 8 x 108 us.  Four sequences of 80 rows: 229 us per layer against 2 x 129 for two passes of the small-M kernel over two
// sequences (56 KB of shared-memory fill and 74 KB of operand reads per 16 KB weight unit were its bound); eight: 424
// against 4 x 128.
#include <algorithm>
#include <new>
#include <queue>
#include <string.h>
#include <vector>

#include "esp_gemm_tc.cuh"
#include "esp_launch.h"

namespace esp {

namespace {

using namespace tc;

constexpr int SLOT_BYTES = 2 * A_BYTES;        // 32 KB: two weight units, or one plane of a row tile
constexpr int SLOTS = 7;
constexpr int WIDE_THREADS = 320;
constexpr size_t WIDE_SMEM = 1024 + (size_t)SLOTS * SLOT_BYTES + 256;
static_assert(WIDE_SMEM <= 232448, "shared memory");

struct WideParams {
    CUtensorMap map_b;          // activations [2 planes x x_blocks][RT][K], box 64 x WB x BPT
    const unsigned char* w;     // packed weight units [n_tiles][KB][A_BYTES]
    const SeqState* st;         // one state per block
    float* partials;            // [range][slot][2 halves][n_rt * WR rows][128 features]
    int* err;
    int32_t n_tiles, n_ft, KB, n_groups, n_rt, slots, plane_blocks, n_blocks;
};

// One block's WB accumulator columns of this warp's 32 features (lane = feature) -> its first n rows of the partial, CH
// columns at a time: as many 16-column loads as fit, an 8-column load for the rest, one wait.  released() is called when
// the last columns are in registers.
template <int WB, typename F>
__device__ __forceinline__ void drain_block(uint32_t taddr, float* part, int n, F released) {
    constexpr int CH = WB % 24 == 0 ? 24 : (WB % 40 == 0 ? 40 : 32);
    static_assert(WB % CH == 0 && (CH % 16 == 0 || CH % 16 == 8), "columns per wait");
#pragma unroll
    for (int c0 = 0; c0 < WB; c0 += CH) {
        uint32_t v[CH];
#pragma unroll
        for (int c = 0; c + 16 <= CH; c += 16) tmem_ld16_issue(taddr + c0 + c, *reinterpret_cast<uint32_t(*)[16]>(&v[c]));
        if constexpr (CH % 16 == 8)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(v[CH - 8]), "=r"(v[CH - 7]), "=r"(v[CH - 6]), "=r"(v[CH - 5]), "=r"(v[CH - 4]), "=r"(v[CH - 3]),
                           "=r"(v[CH - 2]), "=r"(v[CH - 1])
                         : "r"(taddr + c0 + CH - 8));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (c0 + CH >= WB) released();
#pragma unroll
        for (int i = 0; i < CH; ++i)
            if (c0 + i < n) __stcg(part + (size_t)(c0 + i) * TILE_N, __uint_as_float(v[i]));
    }
}

template <int WB, int BPT>
__global__ void __launch_bounds__(WIDE_THREADS, 1) k_gemm_wide(const __grid_constant__ WideParams p) {
    constexpr int WR = WB * BPT;               // rows of a row tile = MMA N
    constexpr int X_BYTES = WR * BK * 2;
    constexpr bool TURNS = WB == RT;           // may have more items than CTAs
    static_assert(WR % 16 == 0 && WR <= 256 && X_BYTES <= SLOT_BYTES && WB % 8 == 0 && WB <= RT, "row tile");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(ring + SLOTS * SLOT_BYTES);
    uint64_t* empty = full + SLOTS;
    uint64_t* tfull = empty + SLOTS;
    uint64_t* tempty = tfull + 1;
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(tempty + 1);
    volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long U = (long long)p.n_ft * p.KB;
    const int n_work = p.n_groups * p.n_rt;        // items: range w / n_rt, row tile w % n_rt
    int rt = blockIdx.x % p.n_rt, grp = blockIdx.x / p.n_rt;
    int u0 = (int)sk_begin(grp, U, p.n_groups), u1 = (int)sk_begin(grp + 1, U, p.n_groups);
    // the CTA's next item, if it has one
    auto next_item = [&](int& w) {
        w += gridDim.x;
        if (!TURNS || w >= n_work) return false;
        rt = w % p.n_rt; grp = w / p.n_rt;
        u0 = (int)sk_begin(grp, U, p.n_groups); u1 = (int)sk_begin(grp + 1, U, p.n_groups);
        return true;
    };

    if (threadIdx.x == 0) {
        pdl_launch_dependents();
        prefetch_tensormap(&p.map_b);
        for (int i = 0; i < SLOTS; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        mbar_init(tfull, 1);
        mbar_init(tempty, 8);           // one arrival per epilogue warp
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *s_tmem;

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t pol_w = l2_policy_evict_first(), pol_x = l2_policy_evict_last();
            auto load_w = [&](int ft, int kb, int slot) {
                unsigned char* dst = ring + slot * SLOT_BYTES;
                const int t1 = 2 * ft + 1 < p.n_tiles ? 2 * ft + 1 : 2 * ft;      // (an odd last tile fills both halves)
                mbar_expect_tx(&full[slot], SLOT_BYTES);
                bulk_load(dst, p.w + ((size_t)(2 * ft) * p.KB + kb) * A_BYTES, A_BYTES, &full[slot], pol_w);
                bulk_load(dst + A_BYTES, p.w + ((size_t)t1 * p.KB + kb) * A_BYTES, A_BYTES, &full[slot], pol_w);
            };
            auto load_x = [&](int plane, int kb, int slot) {
                mbar_expect_tx(&full[slot], X_BYTES);
                tma_load_3d_hint(ring + slot * SLOT_BYTES, &p.map_b, kb * BK, 0, plane * p.plane_blocks + rt * BPT, &full[slot], pol_x);
            };
            // load i of an item: unit u0 + i / 3; i % 3 = 0 weights, 1 hi rows, 2 lo rows
            const int n_pre = 3 * (u1 - u0) < SLOTS ? 3 * (u1 - u0) : SLOTS;
            // the weights do not depend on the kernel before this one, the activations do
            for (int i = 0; i < n_pre; i += 3) load_w((u0 + i / 3) / p.KB, (u0 + i / 3) % p.KB, i);
            pdl_wait();
            for (int i = 0; i < n_pre; ++i)
                if (i % 3) load_x(i % 3 - 1, (u0 + i / 3) % p.KB, i);
            // (no division per load: with two per load and one more for the row tile, a step of four 68-row sequences took 3600 us
            // against 3460; the 240-row tiles did not notice)
            bool ok = true;
            int slot = n_pre % SLOTS;
            uint32_t phase = n_pre == SLOTS ? 0 : 1;         // parity of the slot's release that a load waits for (a fresh barrier passes 1)
            int w = blockIdx.x, u = u0 + n_pre / 3, kind = n_pre % 3;
            do {
                for (int ft = u / p.KB, kb = u % p.KB; u < u1;) {
                    if (!mbar_wait(&empty[slot], phase, s_abort)) { ok = false; break; }
                    if (kind == 0) load_w(ft, kb, slot);
                    else load_x(kind - 1, kb, slot);
                    if (++slot == SLOTS) { slot = 0; phase ^= 1; }
                    if (++kind == 3) {
                        kind = 0; ++u;
                        if (++kb == p.KB) { kb = 0; ++ft; }
                    }
                }
                if (!ok || !next_item(w)) break;
                u = u0;
            } while (true);
            if (!ok) { set_error(p.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
        }
    } else if (warp == 1) {
        const bool leader = elect_lane();
        {
            constexpr uint32_t IDESC = idesc_of(WR);
            bool ok = true;
            int slot = 0, piece = 0;
            uint32_t phase = 0;
            auto next = [&](int& s, uint32_t& ph) { if (++s == SLOTS) { s = 0; ph ^= 1; } };
            int w = blockIdx.x;
            do {
                for (int u = u0; u < u1 && ok; ++piece) {
                    const int end = (u / p.KB + 1) * p.KB < u1 ? (u / p.KB + 1) * p.KB : u1;
                    if (!__all_sync(0xffffffffu, mbar_wait(tempty, (piece & 1) ^ 1, s_abort))) { ok = false; break; }     // (a fresh barrier passes parity 1)
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (const int beg = u; u < end; ++u) {
                        const int sw = slot;
                        const uint32_t pw = phase;
                        next(slot, phase);
                        const int sh = slot;
                        const uint32_t ph = phase;
                        next(slot, phase);
                        const int sl = slot;
                        const uint32_t pl = phase;
                        next(slot, phase);
                        if (!__all_sync(0xffffffffu, mbar_wait(&full[sw], pw, s_abort) && mbar_wait(&full[sh], ph, s_abort))) { ok = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint64_t dw = smem_desc(smem_u32(ring + sw * SLOT_BYTES), 16);
                        const uint64_t dh = smem_desc(smem_u32(ring + sh * SLOT_BYTES), 16);
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {
                            const uint32_t acc = (u > beg || k > 0) ? 1u : 0u;
                            if (leader) umma(tmem_base, dw + (uint64_t)(k * 2), dh + (uint64_t)(k * 2), IDESC, acc);
                            if (leader) umma(tmem_base + 256, dw + (uint64_t)((A_BYTES >> 4) + k * 2), dh + (uint64_t)(k * 2), IDESC, acc);
                        }
                        if (leader) umma_commit(&empty[sh]);
                        if (!__all_sync(0xffffffffu, mbar_wait(&full[sl], pl, s_abort))) { ok = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint64_t dl = smem_desc(smem_u32(ring + sl * SLOT_BYTES), 16);
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {
                            if (leader) umma(tmem_base, dw + (uint64_t)(k * 2), dl + (uint64_t)(k * 2), IDESC, 1u);
                            if (leader) umma(tmem_base + 256, dw + (uint64_t)((A_BYTES >> 4) + k * 2), dl + (uint64_t)(k * 2), IDESC, 1u);
                        }
                        if (leader) umma_commit(&empty[sw]);
                        if (leader) umma_commit(&empty[sl]);
                    }
                    if (leader && ok) umma_commit(tfull);
                }
            } while (ok && next_item(w));
            if (!ok) { set_error(p.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
        }
    } else {
        // ---------------- epilogue: tensor memory -> registers -> partial
        pdl_wait();                              // the partials' last reader has finished
        const int half = (warp - 2) >> 2, q = warp & 3, f = q * 32 + lane;
        const uint32_t taddr = tmem_base + half * 256 + ((uint32_t)(q * 32) << 16);
        const size_t rows = (size_t)p.n_rt * WR;
        bool ok = true;
        int piece = 0, w = blockIdx.x;
        do {
            int nr[BPT];
#pragma unroll
            for (int b = 0; b < BPT; ++b)
                nr[b] = rt * BPT + b < p.n_blocks && p.st[rt * BPT + b].active ? min(p.st[rt * BPT + b].n_rows, WB) : 0;
            const int ft0 = u0 / p.KB;
            for (int u = u0; u < u1 && ok; ++piece) {
                const int ft = u / p.KB;
                u = (ft + 1) * p.KB < u1 ? (ft + 1) * p.KB : u1;
                // (a wait that fails takes the whole warp out: the tensor-memory loads below are warp-wide)
                if (!__all_sync(0xffffffffu, mbar_wait(tfull, piece & 1, s_abort))) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const bool real = 2 * ft + half < p.n_tiles;
                float* part = p.partials + (((size_t)(grp * p.slots + (ft - ft0)) * 2 + half) * rows + (size_t)rt * WR) * TILE_N + f;
#pragma unroll
                for (int b = 0; b < BPT; ++b)
                    drain_block<WB>(taddr + b * WB, part + (size_t)(b * WB) * TILE_N, real ? nr[b] : 0, [&] {
                        if (b != BPT - 1) return;
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(tempty);
                    });
            }
        } while (ok && next_item(w));
        if (!ok && lane == 0) { set_error(p.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
    }
    // ---------------- teardown (every thread arrives here)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*s_abort) {
        for (int i = 0; i < 64; ++i) __nanosleep(10000);   // let copies in flight land before shared memory goes away
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

constexpr int WIDE_SM = 148;

// ---- The same GEMM over the blocks of those sequences of a pass that take part in the step.
// k_gemm_wide multiplies the rows of every block; with few of them live it does a multiple of the work (8 sequences, one
// live: 424 us per 8B layer where one block's weights stream in 67).  Its row tiles cannot simply shrink: the split of k
// is fixed by the handle (a row's bits do not depend on who else takes part), and its ranges alone would leave most SMs idle.
// So the pieces of that split -- a 128-feature tile x a range's k -- become the items here: each has an accumulator of its
// own, as there, and any CTA may take it.  Row tiles are packed from live blocks (up to 160 rows, a copy per block); the
// (piece, row tile) items are dealt to the CTAs longest first, each to the least loaded one (plan_some, when the handle is
// made).  An accumulator takes the hi and lo products of a k-block in k_gemm_wide's order: the same bits.
// Two accumulators in tensor memory, an epilogue group of four warps each; a stage of the ring is a weight unit and the
// rows' two planes.
// What bounds it: the HBM rate with one row tile, the shared-memory port (384 + 4 x rows clocks per unit) with more, and the
// longest piece where the handle's ranges are long.  Measured (8B shapes, four layers and the LM head, L 300, us per step;
// k_gemm_wide over every block -> this): 68 rows, 8 sequences of which 1 / 2 / 4 / 6 take part 2137 / 2309 / 2601 / 2815 -> 848 /
// 946 / 1670 / 2254; 4 sequences, 1 / 2 / 3 1388 / 1470 / 1627 -> 832 / 889 / 1379; 12 sequences, 1 / 4 2828 / 3251 -> 981 /
// 1565; 1 of 8 at 1, 20, 52 and 120 rows 1657, 1701, 2070 and 4482 -> 734, 816, 859 and 932 (the LM head skips idle sequences too).
struct WideItem {
    int32_t unit, kb0, len;      // weight unit (tile * KB + kb0), its k-block, units
    uint16_t idx, rt;            // piece of the partials, row tile
};
constexpr int SOME_RING = 224 * 1024, SOME_STAGES = 8, SOME_ROWS = 160;
constexpr size_t SOME_SMEM = 1024 + SOME_RING + 256;
static_assert(SOME_SMEM <= 232448, "shared memory");
__host__ __device__ constexpr int some_blocks(int wb) { return SOME_ROWS / wb > 1 ? SOME_ROWS / wb : 1; }   // blocks of a row tile

struct SomeParams {
    CUtensorMap map_b;          // activations, box of one block
    const unsigned char* w;
    const SeqState* st;         // one state per block of the pass
    float* partials;            // [piece][rows][128 features]
    int* err;
    const int32_t* first;       // [grid + 1]: the CTA's items
    const WideItem* items;
    int32_t KB, rows, plane_blocks, stages, stage_bytes, lo_off;
    uint8_t tile0[WIDE_MAX_PASS + 1], blk[WIDE_MAX_PASS];    // row tile i: blocks blk[tile0[i]] .. blk[tile0[i + 1] - 1]
};

template <int WB>
__global__ void __launch_bounds__(WIDE_THREADS, 1) k_gemm_wide_some(const __grid_constant__ SomeParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(ring + SOME_RING);
    uint64_t* empty = full + SOME_STAGES;
    uint64_t* tfull = empty + SOME_STAGES;      // [2]
    uint64_t* tempty = tfull + 2;               // [2]
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(tempty + 2);
    volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i0 = __ldg(p.first + blockIdx.x), i1 = __ldg(p.first + blockIdx.x + 1);
    auto item = [&](int i) {
        const int4 v = __ldg(reinterpret_cast<const int4*>(p.items + i));
        WideItem it;
        it.unit = v.x; it.kb0 = v.y; it.len = v.z; it.idx = (uint16_t)(v.w & 0xffff); it.rt = (uint16_t)((unsigned)v.w >> 16);
        return it;
    };

    if (threadIdx.x == 0) {
        pdl_launch_dependents();
        prefetch_tensormap(&p.map_b);
        for (int i = 0; i < SOME_STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], 4); }     // one arrival per epilogue warp
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *s_tmem;

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t pol_w = l2_policy_evict_first(), pol_x = l2_policy_evict_last();
            struct Cursor { int i, u; WideItem it; };
            auto load_w = [&](const Cursor& c, int st) {
                const int nb = p.tile0[c.it.rt + 1] - p.tile0[c.it.rt];
                mbar_expect_tx(&full[st], A_BYTES + 2 * nb * WB * BK * 2);
                bulk_load(ring + st * p.stage_bytes, p.w + (size_t)(c.it.unit + c.u) * A_BYTES, A_BYTES, &full[st], pol_w);
            };
            auto load_x = [&](const Cursor& c, int st) {
                unsigned char* dst = ring + st * p.stage_bytes + A_BYTES;
                for (int b = p.tile0[c.it.rt]; b < p.tile0[c.it.rt + 1]; ++b, dst += WB * BK * 2) {
                    tma_load_3d_hint(dst, &p.map_b, (c.it.kb0 + c.u) * BK, 0, p.blk[b], &full[st], pol_x);
                    tma_load_3d_hint(dst + p.lo_off, &p.map_b, (c.it.kb0 + c.u) * BK, 0, p.plane_blocks + p.blk[b], &full[st], pol_x);
                }
            };
            auto advance = [&](Cursor& c) {
                if (++c.u < c.it.len) return;
                c.u = 0;
                if (++c.i < i1) c.it = item(c.i);
            };
            Cursor cw = {i0, 0, {}};
            if (i0 < i1) cw.it = item(i0);
            Cursor cx = cw;
            int n_pre = 0;      // the weights do not depend on the kernel before this one, the activations do
            for (; n_pre < p.stages && cw.i < i1; ++n_pre) { load_w(cw, n_pre); advance(cw); }
            pdl_wait();
            for (int st = 0; st < n_pre; ++st) { load_x(cx, st); advance(cx); }
            bool ok = true;
            int st = 0;
            uint32_t phase = 0;
            while (cw.i < i1) {      // (every stage is taken once here)
                if (!mbar_wait(&empty[st], phase, s_abort)) { ok = false; break; }
                load_w(cw, st);
                load_x(cw, st);
                advance(cw);
                if (++st == p.stages) { st = 0; phase ^= 1; }
            }
            if (!ok) { set_error(p.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
        }
    } else if (warp == 1) {
        const bool leader = elect_lane();
        {
            bool ok = true;
            int st = 0;
            uint32_t phase = 0;
            for (int n = 0; n < i1 - i0 && ok; ++n) {
                const WideItem it = item(i0 + n);
                const uint32_t idesc = idesc_of((p.tile0[it.rt + 1] - p.tile0[it.rt]) * WB);
                const uint32_t acc = tmem_base + (n & 1) * 256;
                if (!__all_sync(0xffffffffu, mbar_wait(&tempty[n & 1], ((n >> 1) & 1) ^ 1, s_abort))) { ok = false; break; }     // (a fresh barrier passes parity 1)
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int u = 0; u < it.len; ++u) {
                    if (!__all_sync(0xffffffffu, mbar_wait(&full[st], phase, s_abort))) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t base = smem_u32(ring + st * p.stage_bytes);
                    const uint64_t dw = smem_desc(base, 16), dh = smem_desc(base + A_BYTES, 16), dl = smem_desc(base + A_BYTES + p.lo_off, 16);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) if (leader) umma(acc, dw + (uint64_t)(k * 2), dh + (uint64_t)(k * 2), idesc, (u > 0 || k > 0) ? 1u : 0u);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) if (leader) umma(acc, dw + (uint64_t)(k * 2), dl + (uint64_t)(k * 2), idesc, 1u);
                    if (leader) umma_commit(&empty[st]);
                    if (++st == p.stages) { st = 0; phase ^= 1; }
                }
                if (leader && ok) umma_commit(&tfull[n & 1]);
            }
            if (!ok) { set_error(p.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
        }
    } else {
        // ---------------- epilogue: tensor memory -> registers -> partial; group g takes every second item
        pdl_wait();                              // the partials' last reader has finished
        const int g = (warp - 2) >> 2, q = warp & 3, f = q * 32 + lane;
        const uint32_t taddr = tmem_base + g * 256 + ((uint32_t)(q * 32) << 16);
        bool ok = true;
        for (int n = g; n < i1 - i0; n += 2) {
            const WideItem it = item(i0 + n);
            // (a wait that fails takes the whole warp out: the tensor-memory loads below are warp-wide)
            if (!__all_sync(0xffffffffu, mbar_wait(&tfull[g], (n >> 1) & 1, s_abort))) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int b0 = p.tile0[it.rt], b1 = p.tile0[it.rt + 1];
            for (int b = b0; b < b1; ++b) {
                const int blk = p.blk[b], nr = p.st[blk].active ? min(p.st[blk].n_rows, WB) : 0;
                drain_block<WB>(taddr + (b - b0) * WB, p.partials + ((size_t)it.idx * p.rows + (size_t)blk * WB) * TILE_N + f, nr, [&] {
                    if (b != b1 - 1) return;
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[g]);
                });
            }
        }
        if (!ok && lane == 0) { set_error(p.err, DEV_E_WAIT_TIMEOUT); *s_abort = 1; }
    }
    // ---------------- teardown (every thread arrives here)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*s_abort) {
        for (int i = 0; i < 64; ++i) __nanosleep(10000);   // let copies in flight land before shared memory goes away
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

}  // namespace

// Ranges and partial slots of a GEMM of n_tiles 128-feature tiles and KB k-blocks, split for n_rt row tiles.
void wide_geometry(int n_tiles, int KB, int n_rt, int* n_groups, int* slots) {
    const int n_ft = (n_tiles + 1) / 2;
    const long long U = (long long)n_ft * KB;
    long long g = WIDE_SM / n_rt;
    if (g > U) g = U;
    // a consumer sums at most 15 pieces of a tile: no range smaller than a 13th of a tile
    while (g > 1 && U / g * 13 < KB) --g;
    int most = 1;
    for (int c = 0; c < g; ++c) {
        const int n = (int)((sk_begin(c + 1, U, g) - 1) / KB - sk_begin(c, U, g) / KB) + 1;
        most = n > most ? n : most;
    }
    *n_groups = (int)g;
    *slots = most;
}

size_t wide_partial_bytes(int n_tiles, int KB, int n_blocks, int wb, int bpt, int split_bpt) {
    int g, slots;
    wide_geometry(n_tiles, KB, (n_blocks + split_bpt - 1) / split_bpt, &g, &slots);
    return (size_t)g * slots * 2 * ((n_blocks + bpt - 1) / bpt * bpt) * wb * TILE_N * sizeof(float);
}

// Plans of k_gemm_wide_some for one split of k (n_rt row tiles of split_bpt blocks): the items of 1, 2, .. row tiles of
// live blocks, dealt to the CTAs, and the longest CTA's load in half units.
struct SomePlan {
    std::vector<int32_t> first;      // [row tiles][WIDE_SM + 1], offsets into items
    std::vector<WideItem> items;
    std::vector<int> load;           // [row tiles]
};
static int some_tiles(int n_blocks, int wb) { return (n_blocks + some_blocks(wb) - 1) / some_blocks(wb); }
static int count_pieces(int n_tiles, int KB, int n_rt) {
    int g, slots, n = 0;
    wide_geometry(n_tiles, KB, n_rt, &g, &slots);
    const long long U = (long long)((n_tiles + 1) / 2) * KB;
    for (int c = 0; c < g; ++c) {
        const int f0 = (int)(sk_begin(c, U, g) / KB), f1 = (int)((sk_begin(c + 1, U, g) - 1) / KB);
        for (int ft = f0; ft <= f1; ++ft) n += 2 * ft + 1 < n_tiles ? 2 : 1;
    }
    return n;
}
static void plan_some(SomePlan* o, int n_tiles, int KB, int n_rt, int row_tiles) {
    int g, slots;
    wide_geometry(n_tiles, KB, n_rt, &g, &slots);
    const long long U = (long long)((n_tiles + 1) / 2) * KB;
    std::vector<WideItem> pieces;
    for (int c = 0; c < g; ++c) {
        const int u0 = (int)sk_begin(c, U, g), u1 = (int)sk_begin(c + 1, U, g);
        for (int u = u0; u < u1;) {
            const int ft = u / KB, end = (ft + 1) * KB < u1 ? (ft + 1) * KB : u1;
            for (int half = 0; half < 2 && 2 * ft + half < n_tiles; ++half) {
                WideItem it;
                it.unit = (2 * ft + half) * KB + u % KB; it.kb0 = u % KB; it.len = end - u;
                it.idx = (uint16_t)((c * slots + (ft - u0 / KB)) * 2 + half); it.rt = 0;
                pieces.push_back(it);
            }
            u = end;
        }
    }
    std::stable_sort(pieces.begin(), pieces.end(), [](const WideItem& a, const WideItem& b) { return a.len > b.len; });
    for (int rt = 1; rt <= row_tiles; ++rt) {
        std::vector<WideItem> of[WIDE_SM];
        std::priority_queue<std::pair<int, int>, std::vector<std::pair<int, int>>, std::greater<std::pair<int, int>>> q;   // (load, CTA)
        for (int c = 0; c < WIDE_SM; ++c) q.push({0, c});
        int most = 0;
        for (const WideItem& piece : pieces)
            for (int r = 0; r < rt; ++r) {          // the row tiles of a piece side by side: its weights come from HBM once
                std::pair<int, int> e = q.top();
                q.pop();
                of[e.second].push_back(piece);
                of[e.second].back().rt = (uint16_t)r;
                e.first += 2 * piece.len + 1;       // in half units; one for the change of accumulators
                most = e.first > most ? e.first : most;
                q.push(e);
            }
        for (int c = 0; c < WIDE_SM; ++c) {
            o->first.push_back((int32_t)o->items.size());
            o->items.insert(o->items.end(), of[c].begin(), of[c].end());
        }
        o->first.push_back((int32_t)o->items.size());
        o->load.push_back(most);
    }
}
// the splits a handle's passes have: that of its full passes and that of a shorter last one
static int pass_splits(int batch, int max_blocks, int split_bpt, int n_rt[2], int blocks[2]) {
    blocks[0] = max_blocks; blocks[1] = batch % max_blocks;
    n_rt[0] = (blocks[0] + split_bpt - 1) / split_bpt; n_rt[1] = (blocks[1] + split_bpt - 1) / split_bpt;
    return blocks[1] ? 2 : 1;
}
size_t wide_some_bytes(int n_tiles, int KB, int wb, int split_bpt, int max_blocks, int batch) {
    int n_rt[2], blocks[2];
    const int n = pass_splits(batch, max_blocks, split_bpt, n_rt, blocks);
    size_t bytes = 0;
    for (int i = 0; i < n; ++i) {
        const int t = blocks[i] > 1 ? some_tiles(blocks[i] - 1, wb) : 0;      // (with every block live k_gemm_wide is the one)
        bytes += sizeof(WideItem) * (size_t)count_pieces(n_tiles, KB, n_rt[i]) * t * (t + 1) / 2 + (sizeof(int32_t) * (WIDE_SM + 1) * t + 15) / 16 * 16;
    }
    return bytes;
}

struct WideGemm {
    WideParams p;
    int max_blocks, wb, bpt, split_bpt;            // blocks at most; rows per block, blocks per row tile, blocks per row tile of the split
    int groups[WIDE_MAX_RT], slots[WIDE_MAX_RT];   // by row tiles of the split
    TileSrc* tables;            // [row tiles of the split][n_tiles]
    CUtensorMap map_one;        // activations, box of one block
    struct Some {
        int blocks = 0, tiles = 0;                 // blocks of a pass of this split; row tiles of live blocks at most
        const int32_t* first = nullptr;
        const WideItem* items = nullptr;
        std::vector<int> load;
    } some[2];
};

// Items for the passes of a decode step some of whose sequences are idle (`mem`: wide_some_bytes of device memory).
int wide_gemm_plan_some(WideGemm* g, int batch, void* mem, cudaStream_t stream) {
    int n_rt[2], blocks[2];
    const int n = pass_splits(batch, g->max_blocks, g->split_bpt, n_rt, blocks);
    char* at = reinterpret_cast<char*>(mem);
    for (int i = 0; i < n; ++i) {
        if (blocks[i] < 2) continue;
        SomePlan plan;
        plan_some(&plan, g->p.n_tiles, g->p.KB, n_rt[i], some_tiles(blocks[i] - 1, g->wb));
        const size_t nf = (sizeof(int32_t) * plan.first.size() + 15) / 16 * 16, ni = sizeof(WideItem) * plan.items.size();
        if (cudaMemcpyAsync(at, plan.first.data(), sizeof(int32_t) * plan.first.size(), cudaMemcpyHostToDevice, stream) != cudaSuccess ||
            cudaMemcpyAsync(at + nf, plan.items.data(), ni, cudaMemcpyHostToDevice, stream) != cudaSuccess || cudaStreamSynchronize(stream) != cudaSuccess)
            return -1;
        WideGemm::Some& s = g->some[i];
        s.blocks = blocks[i];
        s.tiles = (int)plan.load.size();
        s.first = reinterpret_cast<const int32_t*>(at);
        s.items = reinterpret_cast<const WideItem*>(at + nf);
        s.load = plan.load;
        at += nf + ni;
    }
    return 0;
}

// The plan of k_gemm_wide_some for n_live of n_blocks blocks of a pass, or null where k_gemm_wide is the faster: clocks of the shared-memory
// port per weight unit (fill + operands), times the units of the longest CTA; not less than the weights take from HBM (a unit
// per SM and 710 clocks).
// Measured, us per step of four 8B layers and a small LM head, k_gemm_wide / k_gemm_wide_some at 1, 2, .. sequences ready (in a row:
// the pass ends with the last one): 68 rows, 4 sequences 963 1026 1115 / 653 718 1176; 8 sequences 1534 1608 1707 1814 1878 1929 2274 /
// 767 803 1232 1357 1753 1883 2495; 12 sequences, 8 to 11 ready, 2679 2791 3059 3251 / 2453 2979 3129 3544; 52 rows, 8 sequences, 5 to 7 ready,
// 1620 1711 1867 / 1560 1725 2215; 120 rows, 8 sequences, 3 to 7 ready (k_gemm_wide needs a second turn from 7 on), 2014 2216 2498 2830
// 4238 / 1691 2344 2876 3479 4060.
static const WideGemm::Some* use_some(const WideGemm* g, int n_blocks, int pass_blocks, int n_live) {
    for (const WideGemm::Some& s : g->some) {
        if (s.blocks != pass_blocks || n_live >= pass_blocks) continue;
        const int n_rt = (n_blocks + g->bpt - 1) / g->bpt, groups = g->groups[(pass_blocks + g->split_bpt - 1) / g->split_bpt - 1];
        const double units = (double)g->p.n_ft * g->p.KB, turns = (groups * n_rt + WIDE_SM - 1) / WIDE_SM;      // (128-row blocks may take two)
        const double dense = turns * units / groups * (768 + 6 * g->wb * g->bpt);
        const int t = some_tiles(n_live, g->wb), rows = (n_live + t - 1) / t * g->wb;
        const double some = std::max(0.5 * s.load[t - 1] * (384 + 4 * rows), 2 * units * 710 / WIDE_SM);
        return some < dense ? &s : nullptr;
    }
    return nullptr;
}

int wide_gemm_create(WideGemm** out, int n_tiles, int K, const void* x, int x_blocks, int wb, int bpt, int split_bpt, int max_blocks, float* partials,
                     size_t partial_bytes, TileSrc* tables_dev, int* err, cudaStream_t stream) {
    const int n_rt_max = (max_blocks + split_bpt - 1) / split_bpt;
    if (!out || max_blocks < 1 || n_rt_max > WIDE_MAX_RT || x_blocks < bpt || K % 8 || reinterpret_cast<uintptr_t>(x) % 16) return -1;
    EncodeFn enc = get_encode();
    if (!enc) return -1;
    WideGemm* g = new (std::nothrow) WideGemm();
    if (!g) return -1;
    memset(&g->p, 0, sizeof(g->p));
    WideParams& p = g->p;
    p.n_tiles = n_tiles; p.n_ft = (n_tiles + 1) / 2; p.KB = (K + BK - 1) / BK;
    p.partials = partials; p.err = err; p.plane_blocks = x_blocks;
    g->max_blocks = max_blocks; g->wb = wb; g->bpt = bpt; g->split_bpt = split_bpt;
    g->tables = tables_dev;
    {
        cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)RT, (cuuint64_t)2 * x_blocks};
        cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)RT * K * 2};
        cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)wb, (cuuint32_t)bpt};
        cuuint32_t estr[3] = {1, 1, 1};
        if (enc(&p.map_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(x), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) { delete g; return -1; }
        box[2] = 1;
        if (enc(&g->map_one, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(x), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) { delete g; return -1; }
    }
    TileSrc* tab = new (std::nothrow) TileSrc[(size_t)n_rt_max * n_tiles];
    bool fits = tab != nullptr;
    for (int r = 1; r <= n_rt_max && fits; ++r) {
        wide_geometry(n_tiles, p.KB, r, &g->groups[r - 1], &g->slots[r - 1]);
        fits = wide_partial_bytes(n_tiles, p.KB, r * split_bpt < max_blocks ? r * split_bpt : max_blocks, wb, bpt, split_bpt) <= partial_bytes;
        const long long U = (long long)p.n_ft * p.KB, G = g->groups[r - 1];
        for (int t = 0; t < n_tiles && fits; ++t) {
            TileSrc& e = tab[(size_t)(r - 1) * n_tiles + t];
            memset(&e, 0, sizeof(e));
            const int ft = t / 2;
            const int c0 = sk_cta_of_unit((long long)ft * p.KB, U, G), c1 = sk_cta_of_unit((long long)ft * p.KB + p.KB - 1, U, G);
            if (c1 - c0 + 1 > 15 || ((long long)c1 + 1) * g->slots[r - 1] * 2 > 65535) { fits = false; break; }
            e.n = (uint16_t)(c1 - c0 + 1);
            for (int c = c0; c <= c1; ++c)
                e.idx[c - c0] = (uint16_t)((c * g->slots[r - 1] + (ft - (int)(sk_begin(c, U, G) / p.KB))) * 2 + (t & 1));
        }
    }
    if (fits && cudaMemcpyAsync(tables_dev, tab, sizeof(TileSrc) * n_rt_max * n_tiles, cudaMemcpyHostToDevice, stream) != cudaSuccess) fits = false;
    if (fits && cudaStreamSynchronize(stream) != cudaSuccess) fits = false;
    delete[] tab;
    if (!fits) { delete g; return -1; }
    *out = g;
    return 0;
}

void wide_gemm_destroy(WideGemm* g) { delete g; }

int wide_gemm_launch(const WideGemm* g, const void* packed, const SeqState* st, int n_blocks, cudaStream_t s, bool pdl, int pass_blocks, uint32_t live) {
    if (!g || n_blocks < 1) return ESP_E_ARG;
    if (n_blocks > g->max_blocks || pass_blocks > g->max_blocks) return ESP_E_ARG;
    if (pass_blocks < n_blocks) pass_blocks = n_blocks;
    const int split = (pass_blocks + g->split_bpt - 1) / g->split_bpt - 1;
    const int n_live = live ? __builtin_popcount(live) : n_blocks;
    if (const WideGemm::Some* some = use_some(g, n_blocks, pass_blocks, n_live)) {
        SomeParams p;
        memset(&p, 0, sizeof(p));
        const int tiles = some_tiles(n_live, g->wb), most = (n_live + tiles - 1) / tiles;
        p.map_b = g->map_one;
        p.w = reinterpret_cast<const unsigned char*>(packed);
        p.st = st;
        p.partials = g->p.partials; p.err = g->p.err;
        p.first = some->first + (size_t)(tiles - 1) * (WIDE_SM + 1);
        p.items = some->items;
        p.KB = g->p.KB; p.rows = n_blocks * g->wb; p.plane_blocks = g->p.plane_blocks;
        p.lo_off = most * g->wb * BK * 2;
        p.stage_bytes = A_BYTES + 2 * p.lo_off;
        p.stages = SOME_RING / p.stage_bytes < SOME_STAGES ? SOME_RING / p.stage_bytes : SOME_STAGES;
        int b = 0;
        for (int i = 0; i < n_blocks; ++i)
            if (!live || (live >> i & 1)) p.blk[b++] = (uint8_t)i;
        for (int t = 0; t <= tiles; ++t) p.tile0[t] = (uint8_t)(t * n_live / tiles);
#define ESP_SOME_CASE(WB)                                                                                               \
    if (g->wb == WB) {                                                                                                 \
        if (ensure_dynamic_smem(reinterpret_cast<const void*>(k_gemm_wide_some<WB>), (int)SOME_SMEM)) return ESP_E_CUDA; \
        return launch_k(k_gemm_wide_some<WB>, dim3(WIDE_SM), dim3(WIDE_THREADS), SOME_SMEM, s, pdl, p) == cudaSuccess ? ESP_OK : ESP_E_CUDA; \
    }
        ESP_SOME_CASE(32)
        ESP_SOME_CASE(64)
        ESP_SOME_CASE(80)
        ESP_SOME_CASE(RT)
#undef ESP_SOME_CASE
        return ESP_E_ARG;
    }
    const int n_rt = (n_blocks + g->bpt - 1) / g->bpt;
    WideParams p = g->p;
    p.w = reinterpret_cast<const unsigned char*>(packed);
    p.st = st;
    p.n_rt = n_rt; p.n_blocks = n_blocks; p.n_groups = g->groups[split]; p.slots = g->slots[split];
    const int grid = g->wb != RT || p.n_groups * n_rt < WIDE_SM ? p.n_groups * n_rt : WIDE_SM;
#define ESP_WIDE_CASE(WB, BPT)                                                                                          \
    if (g->wb == WB && g->bpt == BPT) {                                                                                \
        if (ensure_dynamic_smem(reinterpret_cast<const void*>(k_gemm_wide<WB, BPT>), (int)WIDE_SMEM)) return ESP_E_CUDA; \
        return launch_k(k_gemm_wide<WB, BPT>, dim3(grid), dim3(WIDE_THREADS), WIDE_SMEM, s, pdl, p) == cudaSuccess ? ESP_OK : ESP_E_CUDA; \
    }
    ESP_WIDE_CASE(PREFILL_CHUNK, 2)
    ESP_WIDE_CASE(32, 2)
    ESP_WIDE_CASE(32, 3)
    ESP_WIDE_CASE(64, 2)
    ESP_WIDE_CASE(64, 3)
    ESP_WIDE_CASE(80, 2)
    ESP_WIDE_CASE(80, 3)
    ESP_WIDE_CASE(RT, 2)
#undef ESP_WIDE_CASE
    return ESP_E_ARG;
}

// the row of block b, row r in the partials is b * wb + r
StreamK wide_gemm_streamk(const WideGemm* g, int n_blocks, int pass_blocks, uint32_t live) {
    if (pass_blocks < n_blocks) pass_blocks = n_blocks;
    const int split = (pass_blocks + g->split_bpt - 1) / g->split_bpt - 1;
    const bool some = use_some(g, n_blocks, pass_blocks, live ? __builtin_popcount(live) : n_blocks) != nullptr;
    StreamK k;
    k.partials = g->p.partials;
    k.table = g->tables + (size_t)split * g->p.n_tiles;
    k.n_tiles = g->p.n_tiles; k.KB = g->p.KB; k.G = g->groups[split]; k.slots = g->slots[split];
    k.rows = (some ? n_blocks : (n_blocks + g->bpt - 1) / g->bpt * g->bpt) * g->wb;
    k.seq_rows = g->wb;
    return k;
}

}  // namespace esp
