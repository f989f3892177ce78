// What follows each split GEMM in the decoder layer, as device functions: the sum of the stream-K partials
// in CTA order fused with
//   * the residual add and the next RMSNorm                      (after the O and the down projection),
//   * per-head RMSNorm (Qwen3), rotary embedding at the row's position, q to the query buffer and k, v to
//     the cache                                                   (after the QKV projection),
//   * SiLU(gate) * up                                             (after the gate/up projection).
// The kernels that run one operation per launch and the kernel that runs all layers in one launch call the
// same functions, and every product and sum whose grouping a compiler could choose is spelled out as an
// individually rounded operation: both give the same bits.
#pragma once

#include "esp_common.cuh"

namespace esp {

// An activation that feeds a two-plane GEMM is stored as hi = bf16(x) and lo = bf16(x - hi): hi + lo carries x to
// about 2^-17, and the tensor cores take the product with both.
__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
    hi = __float2bfloat16_rn(x);
    lo = __float2bfloat16_rn(__fsub_rn(x, __bfloat162float(hi)));
}

// ------------------------------------------------------------------ residual add + RMSNorm of one row
// The row is cut into groups of 128 features (= GEMM tiles).  A warp owns a group at a time, lane l the
// features 128*group + 4*l .. +3.  Sum of squares: per lane x0^2 + x1^2 + x2^2 + x3^2 (fused multiply-adds in
// that order), butterfly over the warp, groups added in ascending order.
template <typename T>
struct NormFirst {   // what a warp may fetch for its first group before the partials exist
    SkEntry en;
    T g[4];
};

template <typename T>
__device__ __forceinline__ void load4(T (&o)[4], const T* p) {
    if constexpr (sizeof(T) == 2) *reinterpret_cast<uint2*>(o) = __ldg(reinterpret_cast<const uint2*>(p));
    else *reinterpret_cast<float4*>(o) = __ldg(reinterpret_cast<const float4*>(p));
}

template <typename T>
__device__ __forceinline__ void norm_prefetch(NormFirst<T>& pf, const StreamK& sk, const T* g, int d, int warp, int lane) {
    const int j = warp * TILE_N + lane * 4;
    if (j < d) {
        if (sk.partials) pf.en = sk_entry(sk, warp);
        load4(pf.g, g + j);
    }
}

// hres[row] += partial sums (sk.partials != NULL);  y = hres[row] * rsqrt(mean(hres[row]^2) + eps) * g.
// NW warps cooperate; `red` is shared memory for (d + 127) / 128 floats; bar() synchronises those warps.
// yr_lo (bf16 only, may be NULL): the row of the low-order plane of y.
template <typename T, int NW, typename Bar>
__device__ __forceinline__ void resid_norm_row(float* xr, const StreamK& sk, int sk_row, const T* g, T* yr, T* yr_lo, int d, float eps,
                                               float* copy_row, float* red, const NormFirst<T>& pf, int warp, int lane, Bar bar) {
    const int ng = (d + TILE_N - 1) / TILE_N;
    constexpr int KEEP = 3;
    float4 keep[KEEP];
    int it = 0;
    for (int gi = warp; gi < ng; gi += NW, ++it) {
        const int j = gi * TILE_N + lane * 4;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < d) {
            x = __ldcg(reinterpret_cast<const float4*>(xr + j));
            if (sk.partials) {
                const float4 acc = it == 0 ? sk_sum4(sk, pf.en, sk_row, lane * 4) : sk_sum4(sk, gi, sk_row, lane * 4);
                x.x = __fadd_rn(x.x, acc.x); x.y = __fadd_rn(x.y, acc.y); x.z = __fadd_rn(x.z, acc.z); x.w = __fadd_rn(x.w, acc.w);
                __stcg(reinterpret_cast<float4*>(xr + j), x);
            }
        }
        if (it < KEEP) keep[it] = x;
        float ss = __fmaf_rn(x.w, x.w, __fmaf_rn(x.z, x.z, __fmaf_rn(x.y, x.y, __fmul_rn(x.x, x.x))));
        ss = warp_sum(ss);
        if (lane == 0) red[gi] = ss;
    }
    bar();
    float tot = 0.f;
#pragma unroll 8
    for (int gi = 0; gi < ng; ++gi) tot = __fadd_rn(tot, red[gi]);
    const float rinv = 1.0f / sqrtf(__fadd_rn(tot / (float)d, eps));
    it = 0;
    for (int gi = warp; gi < ng; gi += NW, ++it) {
        const int j = gi * TILE_N + lane * 4;
        if (j >= d) continue;
        const float4 x = it < KEEP ? keep[it] : __ldcg(reinterpret_cast<const float4*>(xr + j));   // beyond: this thread's own writes
        const float xv[4] = {x.x, x.y, x.z, x.w};
        T gg[4];
        if (it == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) gg[i] = pf.g[i];
        } else {
            load4(gg, g + j);
        }
        T o[4];
        if constexpr (sizeof(T) == 2) {
            T ol[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) split_bf16(__fmul_rn(__fmul_rn(xv[i], rinv), to_f32(gg[i])), o[i], ol[i]);
            *reinterpret_cast<uint2*>(yr + j) = *reinterpret_cast<const uint2*>(o);
            if (yr_lo) *reinterpret_cast<uint2*>(yr_lo + j) = *reinterpret_cast<const uint2*>(ol);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = from_f32<T>(__fmul_rn(__fmul_rn(xv[i], rinv), to_f32(gg[i])));
            *reinterpret_cast<float4*>(yr + j) = *reinterpret_cast<const float4*>(o);
        }
        if (copy_row) *reinterpret_cast<float4*>(copy_row + j) = x;
    }
}

// The same for launches of many rows (d <= 128 * NW * 4): NW warps per row, four groups per warp in registers, the pieces
// of the four groups requested together.  Sums, products and their order are resid_norm_row's, so are the bits.
// put(group, sum) hands a group's sum of squares to every warp of the row, bar() waits for all of them.
// `ahead` is what a warp has fetched before the partials exist: counts, the first seven places and the norm weights.
constexpr int NORM_MANY_WARPS = 8, NORM_MANY_D = TILE_N * NORM_MANY_WARPS * 4;
template <int NG>
struct NormAhead {
    uint32_t e[NG][4];        // first half of the group's entry: count, then places, a halfword each
    uint2 g[NG];
};

template <int NW, int NG>
__device__ __forceinline__ void norm_prefetch_many(NormAhead<NG>& ah, const StreamK& sk, const __nv_bfloat16* g, int d, int warp, int lane) {
#pragma unroll
    for (int u = 0; u < NG; ++u) {
        const int gi = warp + NW * u, j = gi * TILE_N + lane * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) ah.e[u][i] = 0;
        ah.g[u] = make_uint2(0, 0);
        if (j < d) {
            if (sk.partials) {
                const uint4 e = __ldg(reinterpret_cast<const uint4*>(sk.table + gi));
                ah.e[u][0] = e.x; ah.e[u][1] = e.y; ah.e[u][2] = e.z; ah.e[u][3] = e.w;
            }
            ah.g[u] = __ldg(reinterpret_cast<const uint2*>(g + j));
        }
    }
}

template <typename T, int NW, int NG, int PB, typename Put, typename Bar>
__device__ __forceinline__ void resid_norm_row_many(float* xr, const StreamK& sk, int sk_row, const T* g, T* yr, T* yr_lo, int d, float eps,
                                                    float* copy_row, float* red, const NormAhead<NG>* ahead, int warp, int lane, Put put, Bar bar) {
    const int ng = (d + TILE_N - 1) / TILE_N;
    float4 x[NG], acc[NG];
    int n[NG], idx0[NG];
#pragma unroll
    for (int u = 0; u < NG; ++u) {
        const int gi = warp + NW * u, j = gi * TILE_N + lane * 4;
        x[u] = acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        n[u] = 0;
        idx0[u] = gi;
        if (gi < ng && j < d) {
            x[u] = __ldcg(reinterpret_cast<const float4*>(xr + j));
            if (sk.partials) n[u] = ahead ? (int)(ahead->e[u][0] & 0xffffu) : (int)__ldg(&sk.table[gi].n);
        }
    }
    int most = 0;
#pragma unroll
    for (int u = 0; u < NG; ++u) most = max(most, n[u]);
    const float* base = sk.partials + (size_t)sk_row * TILE_N + lane * 4;
    const size_t piece = (size_t)sk.rows * TILE_N;
    int c0 = 0;
    if (ahead) {                                     // the first batch without a trip to the table
        static_assert(PB <= 7, "places of the first batch");
        float4 t[PB][NG];
#pragma unroll
        for (int c = 0; c < PB; ++c)
#pragma unroll
            for (int u = 0; u < NG; ++u) {
                t[c][u] = make_float4(0.f, 0.f, 0.f, 0.f);
                const uint32_t at = (ahead->e[u][(c + 1) >> 1] >> (((c + 1) & 1) * 16)) & 0xffffu;
                if (c < n[u]) t[c][u] = __ldcg(reinterpret_cast<const float4*>(base + (size_t)at * piece));
            }
#pragma unroll
        for (int c = 0; c < PB; ++c)
#pragma unroll
            for (int u = 0; u < NG; ++u) { acc[u].x += t[c][u].x; acc[u].y += t[c][u].y; acc[u].z += t[c][u].z; acc[u].w += t[c][u].w; }
        c0 = PB;
    }
    for (; c0 < most; c0 += PB) {          // pieces in ascending order, as sk_sum4 adds them
        float4 t[PB][NG];
#pragma unroll
        for (int c = 0; c < PB; ++c)
#pragma unroll
            for (int u = 0; u < NG; ++u) {
                t[c][u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c0 + c < n[u]) t[c][u] = __ldcg(reinterpret_cast<const float4*>(base + (size_t)__ldg(&sk.table[idx0[u]].idx[c0 + c]) * piece));
            }
#pragma unroll
        for (int c = 0; c < PB; ++c)
#pragma unroll
            for (int u = 0; u < NG; ++u) { acc[u].x += t[c][u].x; acc[u].y += t[c][u].y; acc[u].z += t[c][u].z; acc[u].w += t[c][u].w; }
    }
#pragma unroll
    for (int u = 0; u < NG; ++u) {
        const int gi = warp + NW * u, j = gi * TILE_N + lane * 4;
        if (gi >= ng) break;
        if (sk.partials && j < d) {
            x[u].x = __fadd_rn(x[u].x, acc[u].x); x[u].y = __fadd_rn(x[u].y, acc[u].y);
            x[u].z = __fadd_rn(x[u].z, acc[u].z); x[u].w = __fadd_rn(x[u].w, acc[u].w);
            __stcg(reinterpret_cast<float4*>(xr + j), x[u]);
        }
        float ss = __fmaf_rn(x[u].w, x[u].w, __fmaf_rn(x[u].z, x[u].z, __fmaf_rn(x[u].y, x[u].y, __fmul_rn(x[u].x, x[u].x))));
        ss = warp_sum(ss);
        if (lane == 0) put(gi, ss);
    }
    bar();
    float tot = 0.f;
#pragma unroll 8
    for (int gi = 0; gi < ng; ++gi) tot = __fadd_rn(tot, red[gi]);
    const float rinv = 1.0f / sqrtf(__fadd_rn(tot / (float)d, eps));
#pragma unroll
    for (int u = 0; u < NG; ++u) {
        const int j = (warp + NW * u) * TILE_N + lane * 4;
        if (j >= d) break;
        const float xv[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
        __align__(8) T gg[4];
        T o[4], ol[4];
        if (ahead) *reinterpret_cast<uint2*>(gg) = ahead->g[u];
        else load4(gg, g + j);
#pragma unroll
        for (int i = 0; i < 4; ++i) split_bf16(__fmul_rn(__fmul_rn(xv[i], rinv), to_f32(gg[i])), o[i], ol[i]);
        *reinterpret_cast<uint2*>(yr + j) = *reinterpret_cast<const uint2*>(o);
        if (yr_lo) *reinterpret_cast<uint2*>(yr_lo + j) = *reinterpret_cast<const uint2*>(ol);
        if (copy_row) *reinterpret_cast<float4*>(copy_row + j) = x[u];
    }
}

// ------------------------------------------------------------------ QKV: (row, head) tasks, one warp each
struct QkvArgs {
    void* q_out;              // [seq*RT + row][Hq*h] bf16
    void* kcache;             // this layer, first sequence of the pass: [seq][Hkv][cap][h] bf16
    void* vcache;
    const void* q_norm;       // [h] bf16 or NULL
    const void* k_norm;
    const float* rope_cos;    // [cap][h/2]
    const float* rope_sin;
    int32_t Hq, Hkv, cap, qk_norm;
    float rms_eps;
};

template <int HD>
struct QkvPre {   // fetched before the partials exist: contributor entry, rotary factors, norm weights
    SkEntry en;
    float cs[HD / 32], sn[HD / 32], gw[HD / 32];
};

// hs: head slot in the concatenated [q heads | k heads | v heads] space; pos: the row's position L + depth
template <int HD>
__device__ __forceinline__ void qkv_prefetch(QkvPre<HD>& pf, const QkvArgs& a, const StreamK& sk, int hs, int pos, int lane) {
    typedef __nv_bfloat16 T;
    constexpr int NE = HD / 32, half = HD / 2;
    const int j0 = hs * HD + lane * NE;
    pf.en = sk_entry(sk, j0 / TILE_N);
    const int which = hs < a.Hq ? 0 : (hs < a.Hq + a.Hkv ? 1 : 2);
    if (which != 2) {
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const int idx = (lane * NE + i) % half;
            pf.cs[i] = __ldg(a.rope_cos + (size_t)pos * half + idx);
            pf.sn[i] = __ldg(a.rope_sin + (size_t)pos * half + idx);
        }
        if (a.qk_norm) {
            const T* g = reinterpret_cast<const T*>(which == 0 ? a.q_norm : a.k_norm);
#pragma unroll
            for (int i = 0; i < NE; ++i) pf.gw[i] = to_f32(g[lane * NE + i]);
        }
    }
}

// sr: row in the partials; pr: row in the query buffer; slot: cache position L + row; seq: sequence within the pass
template <int HD>
__device__ __forceinline__ void qkv_finish_task(const QkvPre<HD>& pf, const QkvArgs& a, const StreamK& sk, int seq, int sr, int pr,
                                                int slot, int hs, int lane) {
    typedef __nv_bfloat16 T;
    constexpr int NE = HD / 32;
    const int j0 = hs * HD + lane * NE;
    const int f = j0 % TILE_N;
    const int which = hs < a.Hq ? 0 : (hs < a.Hq + a.Hkv ? 1 : 2);
    const int head = which == 0 ? hs : (which == 1 ? hs - a.Hq : hs - a.Hq - a.Hkv);
    float v[NE];
    if constexpr (NE == 4) {
        const float4 t = sk_sum4(sk, pf.en, sr, f);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        // narrower heads: the same sum through the four-float helper on the enclosing aligned group
        const float4 t = sk_sum4(sk, pf.en, sr, f & ~3);
        const float tv[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int i = 0; i < NE; ++i) v[i] = tv[(f & 3) + i];
    }
    if (which != 2) {
        if (a.qk_norm) {
            float ss = 0.f;
#pragma unroll
            for (int i = 0; i < NE; ++i) ss = __fmaf_rn(v[i], v[i], ss);
            ss = warp_sum(ss);
            const float rinv = 1.0f / sqrtf(__fadd_rn(ss / (float)HD, a.rms_eps));
#pragma unroll
            for (int i = 0; i < NE; ++i) v[i] = __fmul_rn(__fmul_rn(v[i], rinv), pf.gw[i]);
        }
        const bool low = lane < 16;
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const float other = __shfl_xor_sync(0xffffffffu, v[i], 16);
            const float rot = __fmul_rn(other, pf.sn[i]);
            v[i] = __fmaf_rn(v[i], pf.cs[i], low ? -rot : rot);
        }
    }
    T* dst;
    if (which == 0) dst = reinterpret_cast<T*>(a.q_out) + (size_t)pr * a.Hq * HD + head * HD + lane * NE;
    else dst = reinterpret_cast<T*>(which == 1 ? a.kcache : a.vcache) + (((size_t)seq * a.Hkv + head) * a.cap + slot) * HD + lane * NE;
    T o[NE];
#pragma unroll
    for (int i = 0; i < NE; ++i) o[i] = from_f32<T>(v[i]);
    if constexpr (NE == 4) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(o);
    else if constexpr (NE == 2) *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(o);
    else dst[0] = o[0];
}

// ------------------------------------------------------------------ gate/up: FPT features of one row per task
// A tile holds 64 gate features (columns 0..63) and the matching 64 up features (columns 64..127).
// en: the contributor entry of tile j0 / 64; act_row: the row's [F] activations; sr: row in the partials.
// act_lo_row (may be NULL): the row of the low-order plane.
// All loads of PB pieces are requested together: the sums one after the other were a round trip each, 2.8 of the kernel's 3.6
// to 6 us behind its wait.  A tile of a large matrix has one or two pieces: eight features per thread, two pieces.  Small matrices
// are cut into up to 15 pieces: four features, eight pieces (the small bf16 decoder: a 64-token request of it 5506 -> 5197 us with the rest of the change).
template <int FPT, int PB>
__device__ __forceinline__ void swiglu_task(const StreamK& sk, const SkEntry& en, int sr, __nv_bfloat16* act_row, __nv_bfloat16* act_lo_row,
                                            int j0, int F) {
    constexpr int Q = FPT / 4;
    const uint32_t w[8] = {en.e0.x, en.e0.y, en.e0.z, en.e0.w, en.e1.x, en.e1.y, en.e1.z, en.e1.w};
    const int n = (int)(w[0] & 0xffffu);
    const float* base = sk.partials + (size_t)sr * TILE_N + j0 % 64;     // (the last task's columns beyond F are padding of its tile)
    float4 g[Q], u[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) g[q] = u[q] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 15; c += PB) {
        if (c >= n) break;
        float4 t[PB][2 * Q];
#pragma unroll
        for (int e = 0; e < PB; ++e) {
            const int hw = c + e + 1;   // halfword holding idx[c + e]
#pragma unroll
            for (int i = 0; i < 2 * Q; ++i) t[e][i] = make_float4(0.f, 0.f, 0.f, 0.f);
            // (many pieces: loads without a branch, so that they do go out together; a piece that is not there reads the first)
            const bool in = hw < 16 && c + e < n;
            if (PB > 2 || in) {
                const float* p = base + (size_t)((in ? w[(hw & 15) >> 1] >> ((hw & 1) * 16) : w[0] >> 16) & 0xffffu) * ((size_t)sk.rows * TILE_N);
#pragma unroll
                for (int i = 0; i < 2 * Q; ++i) {
                    const float4 v = __ldcg(reinterpret_cast<const float4*>(p + (i / Q) * 64 + (i % Q) * 4));
                    if (in) t[e][i] = v;
                }
            }
        }
#pragma unroll
        for (int e = 0; e < PB; ++e)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                g[q].x += t[e][q].x; g[q].y += t[e][q].y; g[q].z += t[e][q].z; g[q].w += t[e][q].w;
                u[q].x += t[e][Q + q].x; u[q].y += t[e][Q + q].y; u[q].z += t[e][Q + q].z; u[q].w += t[e][Q + q].w;
            }
    }
    __align__(16) __nv_bfloat16 o[FPT], ol[FPT];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const float gv[4] = {g[q].x, g[q].y, g[q].z, g[q].w}, uv[4] = {u[q].x, u[q].y, u[q].z, u[q].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) split_bf16(__fmul_rn(gv[i] / __fadd_rn(1.0f, expf(-gv[i])), uv[i]), o[4 * q + i], ol[4 * q + i]);
    }
    if (FPT == 8 && j0 + 8 <= F) {
        *reinterpret_cast<uint4*>(act_row + j0) = *reinterpret_cast<const uint4*>(o);
        if (act_lo_row) *reinterpret_cast<uint4*>(act_lo_row + j0) = *reinterpret_cast<const uint4*>(ol);
    } else {
        *reinterpret_cast<uint2*>(act_row + j0) = *reinterpret_cast<const uint2*>(o);
        if (act_lo_row) *reinterpret_cast<uint2*>(act_lo_row + j0) = *reinterpret_cast<const uint2*>(ol);
    }
}

}  // namespace esp
