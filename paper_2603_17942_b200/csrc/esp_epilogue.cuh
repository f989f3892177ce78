// Epilogues of the small-M GEMMs that work on a whole 128-feature tile.  Both GEMM implementations (tcgen05 and
// CUDA-core) place the tile's fp32 accumulators in shared memory as s_acc[row][feature] and call run_epilogue (the
// rows of a block) or run_epilogue_rows (some of them) with exactly 128 threads (thread f owns feature f of the
// tile): rotary embedding at the tree-depth position and the KV-cache write (QKV), per-row argmax / Top-K' /
// max+sum-exp over the vocabulary tile (LM head), a plain store.
#pragma once

#include "esp_common.cuh"
#include "esp_sampling.cuh"

namespace esp {

constexpr int ACC_LD = TILE_N + 1;  // padded row stride of s_acc (floats)

// order-preserving map of a float onto an unsigned integer (larger float <=> larger key; every key > 0)
// (-0 and +0 share a key, as they compare equal)
__device__ __forceinline__ uint32_t float_order_key(float v) {
    uint32_t b = __float_as_uint(v);
    if ((b << 1) == 0u) b = 0u;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float float_from_order_key(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__device__ __forceinline__ void epi_bar(int bar_id) {
    asm volatile("bar.sync %0, 128;" ::"r"(bar_id) : "memory");
}

// s_acc: [rows][ACC_LD] fp32, rows r0 .. r1-1 of the block (r1 <= n_rows).  s_aux: >= RT*4 floats of scratch.
// tid in [0,128).  A row's result does not depend on which rows share the call.
template <typename T, int EPI>
__device__ __forceinline__ void run_epilogue_rows(float* s_acc, float* s_aux, int tile, int seq, const EpiArgs& a, int tid, int bar_id,
                                                  const SeqState* st, int n_rows, const int r0, const int r1) {
    const int f = tid;
    const int n0 = tile * TILE_N;
    const int grow0 = seq * RT;
    s_acc -= r0 * ACC_LD;       // addressed by block row below

    if constexpr (EPI == EPI_STORE_F32) {
        if (n0 + f < a.n_out)
            for (int r = r0; r < r1; ++r) a.y_f32[(size_t)(grow0 + r) * a.n_out + n0 + f] = s_acc[r * ACC_LD + f];
    } else if constexpr (EPI == EPI_QKV) {
        const int h = a.h, dq = a.Hq * h, dkv = a.Hkv * h;
        const int feat = n0 + f;  // index in the concatenated [q | k | v] feature space
        const int which = feat < dq ? 0 : (feat < dq + dkv ? 1 : 2);
        const int local = which == 0 ? feat : (which == 1 ? feat - dq : feat - dq - dkv);
        const int head = local / h, fl = local % h, half = h / 2;
        const int L = st ? st->L : 0;
        const int warp = f >> 5;
        if (which != 2) {
            if (a.qk_norm) {
                // per-head RMSNorm: sum of squares over the head's h features, per row
                for (int r = r0; r < r1; ++r) {
                    float v = s_acc[r * ACC_LD + f];
                    float ss = warp_sum(v * v);
                    if ((f & 31) == 0) s_aux[r * 4 + warp] = ss;
                }
                epi_bar(bar_id);
                const T* g = reinterpret_cast<const T*>(which == 0 ? a.q_norm : a.k_norm);
                const float gain = to_f32(g[fl]);
                const int wpw = h / 32;                    // warps per head
                const int w0 = (f / h) * wpw;              // first warp of this thread's head
                for (int r = r0; r < r1; ++r) {
                    float ss = 0.f;
                    for (int w = 0; w < wpw; ++w) ss += s_aux[r * 4 + w0 + w];
                    float rinv = 1.0f / sqrtf(ss / (float)h + a.rms_eps);
                    s_acc[r * ACC_LD + f] = s_acc[r * ACC_LD + f] * rinv * gain;
                }
            }
            epi_bar(bar_id);
            // rotary embedding at position L + depth, rotate-half pairing (i, i + h/2)
            const int partner = fl < half ? f + half : f - half;
            // (the factors of eight rows are fetched before any is used: row by row each was two dependent trips)
            for (int rb = r0; rb < r1; rb += 8) {
                float cs[8], sn[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (rb + i < r1) {
                        const int pos = L + (st ? __ldg(&st->row_depth[rb + i]) : rb + i);
                        cs[i] = __ldg(a.rope_cos + (size_t)pos * half + (fl % half));
                        sn[i] = __ldg(a.rope_sin + (size_t)pos * half + (fl % half));
                    }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = rb + i;
                    if (r >= r1) break;
                    const float me = s_acc[r * ACC_LD + f], other = s_acc[r * ACC_LD + partner];
                    const float v = fl < half ? me * cs[i] - other * sn[i] : me * cs[i] + other * sn[i];
                    if (which == 0) {
                        reinterpret_cast<T*>(a.q_out)[(size_t)(grow0 + r) * dq + head * h + fl] = from_f32<T>(v);
                    } else {
                        reinterpret_cast<T*>(a.kcache)[(((size_t)seq * a.Hkv + head) * a.cap + (L + r)) * h + fl] = from_f32<T>(v);
                    }
                }
            }
        } else {
            if (a.qk_norm) epi_bar(bar_id);
            epi_bar(bar_id);
            for (int r = r0; r < r1; ++r)
                reinterpret_cast<T*>(a.vcache)[(((size_t)seq * a.Hkv + head) * a.cap + (L + r)) * h + fl] =
                    from_f32<T>(s_acc[r * ACC_LD + f]);
        }
    } else if constexpr (EPI == EPI_LOGITS) {
        // (the row loop at the end) warp w takes every fourth row; a lane holds features lane, lane+32, lane+64, lane+96 of the row
        const int warp = f >> 5, lane = f & 31;
        const int n_nodes = st ? st->n_nodes : a.rows_fixed;
        const int Mtot = a.batch * RT;
        // Everything the row loop needs of `a` and `st`, once: behind the loop's stores the compiler has to fetch a member
        // again at every use.
        const int n_out = a.n_out, KP = a.KP;
        Cand* const cand = a.cand;
        float2* const cand_ms = a.cand_ms;
        uint32_t* const cand_floor = a.cand_floor;
        float* const logits_dump = a.logits_dump;
        const float inv_temp = st ? a.samp_inv_temp : 0.f;
        const uint32_t key0 = a.samp_key0, key1 = a.samp_key1;
        const int L = st ? st->L : 0;
        uint32_t noise_pos = 0xffffffffu;   // rows come in breadth-first order: equal depths are neighbours and
        float noise[4] = {0.f, 0.f, 0.f, 0.f};   // share their noise, which is a function of (position, token)
        // Floors.  What is already known of a probe row bounds its K'-th largest logit from below, and an entry strictly
        // below the bound cannot be in the row's final list.  The vocabulary tiles fall into K' groups (tile mod K'); the
        // largest logit of each group so far is kept as an order-preserving key (atomicMax, one per tile and row), and
        // the smallest of the K' group maxima is the bound: K' different tokens reach it.  (The K'-th best of a single
        // tile, the bound used before, is an ordinary value, the best 9 % of the tile: hardly any tile stayed below it.)
        // The bounds are fetched once per tile, all rows at a time.  Measured, 90 probe rows of 120, vocabulary 128256,
        // K' = 11: LM head 368 -> 240 us; 36 of 48 rows: 192 -> 178 us.  The second look of a CTA's first tile: 220 -> 206 us.
        const int S = n_rows <= 80 ? 80 : RT;                             // s_aux holds at least 2 * S words
        uint32_t* s_floor = reinterpret_cast<uint32_t*>(s_aux);          // [S] bounds, [S] "this probe row has entries at or above its bound"
        uint32_t* s_need = s_floor + S;
        uint32_t* group_max = cand_floor ? cand_floor + (size_t)grow0 * KP_MAX + tile % KP : nullptr;
        auto fetch_bound = [&](int r) -> uint32_t {
            const uint4* g = reinterpret_cast<const uint4*>(cand_floor + (size_t)(grow0 + r) * KP_MAX);
            uint32_t bound = 0xffffffffu;
#pragma unroll
            for (int j = 0; j < KP_MAX; j += 4) {
                if (j >= KP) break;
                const uint4 w = __ldcg(g + j / 4);
                bound = min(bound, w.x);
                if (j + 1 < KP) bound = min(bound, w.y);
                if (j + 2 < KP) bound = min(bound, w.z);
                if (j + 3 < KP) bound = min(bound, w.w);
            }
            return bound;
        };
        for (int r = r0 + f; r < r1; r += 128) s_floor[r] = r >= n_nodes && cand_floor ? fetch_bound(r) : 0u;
        epi_bar(bar_id);
        // Probe rows, one thread per row (the padded row stride keeps the threads on different banks): the tile's
        // (max, sum-exp) for the row's log-sum-exp, and whether anything of the tile can still reach the row's final
        // list.  A row whose maximum lies below its floor is done: its K' entries of this tile are empty.  With many
        // probe rows per block nearly all rows of nearly all tiles end here, without one warp-wide reduction.
        const bool many_probes = n_rows - n_nodes >= 16;     // block-uniform; a handful of probe rows is cheaper warp by warp
        if (many_probes) {
            const int r = (n_nodes > r0 ? n_nodes : r0) + f;
            if (r < r1) {
                const int n_valid = n_out - n0 < TILE_N ? n_out - n0 : TILE_N;
                const float* row = s_acc + r * ACC_LD;
                float tmax = -INFINITY;
                for (int i = 0; i < n_valid; ++i) tmax = fmaxf(tmax, row[i]);
                if (group_max) atomicMax(group_max + (size_t)r * KP_MAX, float_order_key(tmax));
                float sum = 0.f;
                for (int i = 0; i < n_valid; ++i) sum += expf(row[i] - tmax);
                cand_ms[(size_t)tile * Mtot + grow0 + r] = make_float2(tmax, sum);
                // nothing was known when the tile began (every CTA's first): by now most CTAs have reported this tile's maxima
                if (cand_floor && s_floor[r] == 0u) s_floor[r] = fetch_bound(r);
                const bool need = float_order_key(tmax) >= s_floor[r];
                s_need[r] = need ? 1u : 0u;
                if (!need) {
                    Cand* out = cand + ((size_t)tile * Mtot + grow0 + r) * KP;
                    for (int j = 0; j < KP; ++j) { out[j].val = -INFINITY; out[j].id = -1; }
                }
            }
        }
        // Tree rows under greedy matching: one thread per row too, four runs of 32 features side by side, merged in order
        // (largest value, smallest id among equals).  A warp per row spent 1750 cycles on each -- its chain of shared-memory
        // loads, comparisons and two warp-wide reductions, one row after the other --, 19 us per tile of a 64-node tree.
        // Measured, vocabulary 128256: LM head of one sequence of 68 rows 176 -> 163 us, of two 247 -> 185, 30 tree rows and
        // 90 probe rows 237 -> 220.
        const int n_arg = inv_temp > 0.f ? 0 : (n_nodes < r1 ? n_nodes : r1) - r0;     // rows r0 .. r0 + n_arg - 1
        if (f < n_arg) {
            const int r = r0 + f;
            const float* row = s_acc + r * ACC_LD;
            float bv[4];
            int bi[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) { bv[c] = -INFINITY; bi[c] = 0x7fffffff; }
#pragma unroll 8
            for (int i = 0; i < 32; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int id = n0 + 32 * c + i;
                    const float v = row[32 * c + i];
                    if (id < n_out && cand_before(v, id, bv[c], bi[c])) { bv[c] = v; bi[c] = id; }
                }
#pragma unroll
            for (int c = 1; c < 4; ++c)
                if (cand_before(bv[c], bi[c], bv[0], bi[0])) { bv[0] = bv[c]; bi[0] = bi[c]; }
            Cand* out = cand + ((size_t)tile * Mtot + grow0 + r) * KP;
            out->val = bv[0];
            out->id = bi[0] == 0x7fffffff ? -1 : bi[0];
        }
        if (logits_dump)
            for (int r = r0 + warp; r < r1; r += 4)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (n0 + lane + 32 * i < n_out) logits_dump[(size_t)(grow0 + r) * n_out + n0 + lane + 32 * i] = s_acc[r * ACC_LD + lane + 32 * i];
        epi_bar(bar_id);
        for (int r = r0 + (n_arg > 0 ? n_arg : 0) + warp; r < r1; r += 4) {
            float v[4];
            int id[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                id[i] = n0 + lane + 32 * i;
                v[i] = id[i] < n_out ? s_acc[r * ACC_LD + lane + 32 * i] : -INFINITY;
            }
            if (many_probes && r >= n_nodes && !s_need[r]) continue;       // warp-uniform
            const bool probe = r >= n_nodes;
            const int kp = probe ? KP : 1;
            Cand* out = cand + ((size_t)tile * Mtot + grow0 + r) * KP;
            if (!probe && inv_temp > 0.f) {
                // sample matching: this row's token for position L + depth + 1 is the arg-max of the noisy scores
                const uint32_t pos = (uint32_t)(L + st->row_depth[r] + 1);
                if (pos != noise_pos) {
                    noise_pos = pos;
#pragma unroll
                    for (int i = 0; i < 4; ++i) noise[i] = gumbel_noise(key0, key1, pos, (uint32_t)id[i]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (id[i] < n_out) v[i] = sample_score(v[i], inv_temp, noise[i]);
            }
            if (probe && !many_probes) {
                float tmax = warp_max(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
                float s = 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) s += id[i] < n_out ? expf(v[i] - tmax) : 0.f;
                s = warp_sum(s);
                if (lane == 0) {
                    cand_ms[(size_t)tile * Mtot + grow0 + r] = make_float2(tmax, s);
                    if (group_max) atomicMax(group_max + (size_t)r * KP_MAX, float_order_key(tmax));
                }
            }
            const uint32_t floor_key = s_floor[r];
            unsigned used = 0;
            float keep_v = -INFINITY;          // lane j keeps the j-th entry (K' <= 32); one coalesced store per row
            int keep_i = -1;
            for (int j = 0; j < kp; ++j) {
                // lane-local best among unused, then warp-wide best by (value desc, id asc)
                float bv = -INFINITY;
                int bi = 0x7fffffff, bslot = -1;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (!(used >> i & 1) && id[i] < n_out && cand_before(v[i], id[i], bv, bi)) { bv = v[i]; bi = id[i]; bslot = i; }
                // two warp-wide integer reductions: the largest value (as an order-preserving key), then the smallest
                // token id among the lanes that hold it
                const uint32_t key = bslot >= 0 ? float_order_key(bv) : 0u;
                const uint32_t wkey = __reduce_max_sync(0xffffffffu, key);
                const uint32_t wid = __reduce_min_sync(0xffffffffu, (bslot >= 0 && key == wkey) ? (uint32_t)bi : 0xffffffffu);
                const int wi = wkey == 0u ? 0x7fffffff : (int)wid;
                const float wv = wkey == 0u ? -INFINITY : float_from_order_key(wkey);
                if (wi == bi && bslot >= 0) used |= 1u << bslot;
                if (probe && wi != 0x7fffffff && wkey < floor_key) break;   // warp-uniform: this and all later entries are out
                if (lane == j) { keep_v = wv; keep_i = wi == 0x7fffffff ? -1 : wi; }
            }
            if (lane < kp) { out[lane].val = keep_v; out[lane].id = keep_i; }
        }
    }
}

// the whole block
template <typename T, int EPI>
__device__ void run_epilogue(float* s_acc, float* s_aux, int tile, int seq, const EpiArgs& a, int tid, int bar_id) {
    const SeqState* st = a.st ? a.st + seq : nullptr;
    const int n_rows = st ? st->n_rows : a.rows_fixed;
    run_epilogue_rows<T, EPI>(s_acc, s_aux, tile, seq, a, tid, bar_id, st, n_rows, 0, n_rows);
}

}  // namespace esp
