// CUDA-core kernels of the ESP step: row assembly, RMSNorm, the reference
// (CUDA-core) small-M GEMM, position-canonical tree attention (split partials,
// tail + merge), Top-K' merge, and the single-block tree kernel (verify walk,
// KV compaction, mask update, Algorithm 1 + pruner, next row table).
#include <mutex>
#include <utility>
#include <vector>

#include "esp_epilogue.cuh"
#include "esp_consumers.cuh"
#include "esp_launch.h"

namespace esp {

// ------------------------------------------------------------------ per-device caches of the launch helpers
namespace {
std::mutex g_dev_mutex;
std::vector<std::pair<const void*, int>> g_smem_done;   // (function, device) pairs whose limit has been raised
int g_sm_count[64];
}  // namespace
int ensure_dynamic_smem(const void* func, int bytes) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    for (const auto& e : g_smem_done)
        if (e.first == func && e.second == dev) return 0;
    if (cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return -1;
    g_smem_done.emplace_back(func, dev);
    return 0;
}
int current_sm_count() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (g_sm_count[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 0;
        g_sm_count[dev] = n;
    }
    return g_sm_count[dev];
}

// ------------------------------------------------------------------ small helpers
__global__ void k_rope_table(float* cs, float* sn, int n_pos, int h, float base) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int half = h / 2;
    if (i >= n_pos * half) return;
    int pos = i / half, j = i % half;
    double inv = pow((double)base, -2.0 * (double)j / (double)h);
    double ang = (double)pos * inv;
    cs[i] = (float)cos(ang);
    sn[i] = (float)sin(ang);
}

// Mask initialisation at prefill, m [slots][d].  mode 0: every slot = (1/t) sum_j E[x_j] (Eq. mask_init_mean; fp32
// running sum in prompt order).  mode 1 ("Last K"): slot i = embedding of the i-th of the last `slots` prompt tokens.
// What bounds the mean is the latency of gathering embedding rows (a thread per element, one chain: 58 ns per token, 59 us
// for 1024 tokens and 476 for 8192; now 14 and 97 us).  A block owns 32 elements; its warps gather a batch of 256 (fp32:
// 128) rows into shared memory, and the first warp sums it in prompt order while the next one is on its way.
template <typename T> constexpr int mask_threads() { return 512 / (int)sizeof(T); }      // two batches of 128 bytes per row in 32 KB
template <typename T, int MASK_BATCH>
__global__ void __launch_bounds__(MASK_BATCH) k_mask_init(const T* embed, const int32_t* prompt, int t, int d, float* m, int slots, int mode) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, j = blockIdx.x * 32 + lane;
    if (mode == 1) {
        for (int i = warp; i < slots && j < d; i += MASK_BATCH / 32) {
            int src = t - slots + i;
            if (src < 0) src = 0;
            m[(size_t)i * d + j] = to_f32(embed[(size_t)prompt[src] * d + j]);
        }
        return;
    }
    __shared__ T s_v[2][MASK_BATCH][32];
    const int jj = j < d ? j : d - 1;
    float acc = 0.f;
    const int n_batches = (t + MASK_BATCH - 1) / MASK_BATCH;
    for (int b = 0; b <= n_batches; ++b) {
        if (b < n_batches) {
            const int i0 = b * MASK_BATCH + warp * 32;
            const int tok = __ldg(prompt + (i0 + lane < t ? i0 + lane : t - 1));
            T v[32];
#pragma unroll
            for (int u = 0; u < 32; ++u) v[u] = embed[(size_t)__shfl_sync(0xffffffffu, tok, u) * d + jj];
#pragma unroll
            for (int u = 0; u < 32; ++u) s_v[b & 1][warp * 32 + u][lane] = v[u];
        }
        if (b > 0 && warp == 0) {
            const int n = t - (b - 1) * MASK_BATCH < MASK_BATCH ? t - (b - 1) * MASK_BATCH : MASK_BATCH;
#pragma unroll 8
            for (int i = 0; i < n; ++i) acc = acc + to_f32(s_v[(b - 1) & 1][i][lane]);
        }
        __syncthreads();
    }
    if (warp || j >= d) return;
    const float mean = acc / (float)t;
    for (int s = 0; s < slots; ++s) m[(size_t)s * d + j] = mean;
}

// Input rows of the block: E[token] for tree nodes; probe j of a chain gets mask vector j (rows after the
// tree nodes hold the chains back to back, k rows each).
template <typename T>
__global__ void k_assemble(const SeqState* states, const T* embed, const float* mvec, float* hres, int d, int mask_slots) {
    // let the next kernel start its own preamble (for a GEMM: the first weight tiles) while this one runs; it still
    // waits for this kernel to complete before it touches anything this kernel or its predecessors write
    if (threadIdx.x == 0) pdl_launch_dependents();
    pdl_wait();
    int seq = blockIdx.y, r = blockIdx.x;
    const SeqState* st = states + seq;
    if (!st->active || r >= st->n_rows) return;
    float* out = hres + (size_t)(seq * RT + r) * d;
    int tok = st->row_token[r];
    // four elements per thread and step (d is a multiple of 8), independent loads in flight
    if (tok >= 0) {
        const T* src = embed + (size_t)tok * d;
#pragma unroll 4
        for (int j = threadIdx.x * 4; j < d; j += blockDim.x * 4) {
            float4 v;
            if constexpr (sizeof(T) == 2) {
                const uint2 raw = *reinterpret_cast<const uint2*>(src + j);
                const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&raw.x), hi = *reinterpret_cast<const __nv_bfloat162*>(&raw.y);
                v = make_float4(__low2float(lo), __high2float(lo), __low2float(hi), __high2float(hi));
            } else {
                v = *reinterpret_cast<const float4*>(src + j);
            }
            *reinterpret_cast<float4*>(out + j) = v;
        }
    } else {
        const float* src = mvec + ((size_t)seq * mask_slots + (r - st->n_nodes) % mask_slots) * d;
#pragma unroll 4
        for (int j = threadIdx.x * 4; j < d; j += blockDim.x * 4) *reinterpret_cast<float4*>(out + j) = *reinterpret_cast<const float4*>(src + j);
    }
}

// y = x * rsqrt(mean(x^2)+eps) * g, one block per row
template <typename T>
__global__ void __launch_bounds__(256) k_rmsnorm(const SeqState* states, const float* x, const T* g, T* y, int d, float eps,
                                                float* copy_out) {
    // let the next kernel start its own preamble (for a GEMM: the first weight tiles) while this one runs; it still
    // waits for this kernel to complete before it touches anything this kernel or its predecessors write
    if (threadIdx.x == 0) pdl_launch_dependents();
    int seq = blockIdx.y, r = blockIdx.x;
    const SeqState* st = states + seq;
    const bool idle = !st->active || r >= st->n_rows;     // the row table was written by an earlier step
    pdl_wait();
    if (idle) return;
    const float* xr = x + (size_t)(seq * RT + r) * d;
    __shared__ float red[8];
    float ss = 0.f;
    for (int j = threadIdx.x; j < d; j += 256) { float v = xr[j]; ss += v * v; }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    float rinv = 1.0f / sqrtf(tot / (float)d + eps);
    T* yr = y + (size_t)(seq * RT + r) * d;
    for (int j = threadIdx.x; j < d; j += 256) yr[j] = from_f32<T>(xr[j] * rinv * to_f32(g[j]));
    if (copy_out)
        for (int j = threadIdx.x; j < d; j += 256) copy_out[(size_t)(seq * RT + r) * d + j] = xr[j];
}

// One fp32 row of up to MAX elements by a warp: y = x * rsqrt(mean(x^2) + eps) * g.  The whole row is requested at once.  The sum of
// squares: per lane over its elements in ascending order, then over the warp; the same bits wherever the norm is taken.
template <int MAX>
__device__ __forceinline__ void norm_row(float* y, const float* x, const float* g, int d, float eps, int lane, float* copy) {
    float4 v[MAX / 128];
    float ss = 0.f;
#pragma unroll
    for (int q = 0; q < MAX / 128; ++q)
        if (lane * 4 + 128 * q < d) v[q] = __ldcg(reinterpret_cast<const float4*>(x + lane * 4 + 128 * q));
#pragma unroll
    for (int q = 0; q < MAX / 128; ++q)
        if (lane * 4 + 128 * q < d) ss = fmaf(v[q].w, v[q].w, fmaf(v[q].z, v[q].z, fmaf(v[q].y, v[q].y, fmaf(v[q].x, v[q].x, ss))));
    const float rinv = 1.0f / sqrtf(warp_sum(ss) / (float)d + eps);
#pragma unroll
    for (int q = 0; q < MAX / 128; ++q) {
        const int j = lane * 4 + 128 * q;
        if (j < d) {
            if (copy) *reinterpret_cast<float4*>(copy + j) = v[q];
            *reinterpret_cast<float4*>(y + j) = make_float4(v[q].x * rinv * g[j], v[q].y * rinv * g[j + 1], v[q].z * rinv * g[j + 2], v[q].w * rinv * g[j + 3]);
        }
    }
}

// fp32 rows of up to 1024 elements, a warp per row
constexpr int NORM_ROWS_WARPS = 4, NORM_ROWS_D = 1024;
__global__ void __launch_bounds__(NORM_ROWS_WARPS * 32) k_rmsnorm_rows(const SeqState* states, const float* x, const float* g, float* y, int d,
                                                                       float eps, float* copy_out) {
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int seq = blockIdx.y, r = blockIdx.x * NORM_ROWS_WARPS + (threadIdx.x >> 5);
    const SeqState* st = states + seq;
    const bool idle = !st->active || r >= st->n_rows;     // the row table was written by an earlier step
    pdl_wait();
    if (idle) return;
    const size_t row = (size_t)(seq * RT + r) * d;
    norm_row<NORM_ROWS_D>(y + row, x + row, g, d, eps, threadIdx.x & 31, copy_out ? copy_out + row : nullptr);
}

// Consumer of a split GEMM (O or down projection) fused with the residual add and the next RMSNorm:
//   hres[r] += sum over the tile's contributors, in CTA order, of their fp32 partials;  y = rmsnorm(hres[r]) * g.
// One block per row (resid_norm_row); with sk.partials == NULL it is a plain RMSNorm of hres.  The sum order
// depends only on the GEMM's shape, never on the number of rows in the block.
template <typename T>
__global__ void __launch_bounds__(1024) k_resid_norm(const SeqState* states, float* hres, StreamK sk, const T* g, T* y, T* y_lo, int d,
                                                    float eps, float* copy_out) {
    // let the next kernel start its own preamble (for a GEMM: the first weight tiles) while this one runs; it still
    // waits for this kernel to complete before it touches anything this kernel or its predecessors write
    if (threadIdx.x == 0) pdl_launch_dependents();
    // fetched before the wait: the tile's contributor entry and the norm weights of this warp's first group
    // (neither changes after initialisation), so that only the partials are loaded behind the wait
    __shared__ float red[128];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    NormFirst<T> pf;
    norm_prefetch(pf, sk, g, d, warp, lane);
    const int seq = blockIdx.y, r = blockIdx.x;
    const SeqState* st = states + seq;
    const bool idle = !st->active || r >= st->n_rows;     // the row table was written by an earlier step
    pdl_wait();
    if (idle) return;
    const size_t row = (size_t)(seq * RT + r) * d;
    resid_norm_row<T, 32>(hres + row, sk, seq * sk.seq_rows + r, g, y + row, y_lo ? y_lo + row : nullptr, d, eps,
                          copy_out ? copy_out + row : nullptr, red, pf, warp, lane, [] { __syncthreads(); });
}

// The same, 512 threads per row: the next GEMM's block fits beside it and starts its weight stream meanwhile.  Rows of
// more than 2048 and up to 4096 elements; step of sixteen 8B layers 2158 -> 2148 us, with 120-row blocks (eight layers)
// 1554 -> 1541.
constexpr int NORM_HALF_WARPS = 16, NORM_HALF_D = TILE_N * NORM_HALF_WARPS * 2;
__global__ void __launch_bounds__(NORM_HALF_WARPS * 32, 1) k_resid_norm_half(const SeqState* states, float* hres, StreamK sk, const __nv_bfloat16* g,
                                                                          __nv_bfloat16* y, __nv_bfloat16* y_lo, int d, float eps, float* copy_out) {
    __shared__ float red[NORM_HALF_D / TILE_N];
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int seq = blockIdx.y, r = blockIdx.x;
    const SeqState* st = states + seq;
    const bool idle = !st->active || r >= st->n_rows;     // the row table was written by an earlier step
    pdl_wait();
    if (idle) return;
    const size_t row = (size_t)(seq * RT + r) * d;
    resid_norm_row_many<__nv_bfloat16, NORM_HALF_WARPS, 2, 6>(hres + row, sk, seq * sk.seq_rows + r, g, y + row, y_lo ? y_lo + row : nullptr, d, eps,
                                                              copy_out ? copy_out + row : nullptr, red, nullptr, warp, lane,
                                                              [&](int gi, float v) { red[gi] = v; }, [] { __syncthreads(); });
}

// The same with a row's two halves of 256 threads in the two blocks of a cluster, for launches of few rows, which leave half of
// the SMs idle otherwise: a row's pieces (about 96 KB out of L2) arrive through two SMs, and the table's entries and the norm
// weights are fetched before the wait.  Each block puts its groups' sums into both blocks' `red`; they are added in the same
// order.  Step of the 8B shape, 68 rows, 4020 -> 3983 us (a third of it by the fetches ahead), request with 30-row static trees
// 18.25 -> 18.08 ms.  With more blocks than SMs (120 rows) 1517 -> 1528 us: those keep the kernel above.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NORM_HALF_WARPS * 16)
k_resid_norm_pair(const SeqState* states, float* hres, StreamK sk, const __nv_bfloat16* g, __nv_bfloat16* y, __nv_bfloat16* y_lo, int d,
                  float eps, float* copy_out) {
    __shared__ float red[NORM_HALF_D / TILE_N];
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int half = blockIdx.x & 1, warp = (threadIdx.x >> 5) + half * (NORM_HALF_WARPS / 2), lane = threadIdx.x & 31;
    NormAhead<2> ahead;
    norm_prefetch_many<NORM_HALF_WARPS, 2>(ahead, sk, g, d, warp, lane);
    const int seq = blockIdx.y, r = blockIdx.x >> 1;
    const SeqState* st = states + seq;
    const bool idle = !st->active || r >= st->n_rows;     // the row table was written by an earlier step
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");      // the other block runs: its shared memory may be written
    pdl_wait();
    if (idle) return;
    uint32_t other;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(other) : "r"((uint32_t)__cvta_generic_to_shared(red)), "r"(half ^ 1));
    const size_t row = (size_t)(seq * RT + r) * d;
    resid_norm_row_many<__nv_bfloat16, NORM_HALF_WARPS, 2, 6>(hres + row, sk, seq * sk.seq_rows + r, g, y + row, y_lo ? y_lo + row : nullptr, d, eps,
        copy_out ? copy_out + row : nullptr, red, &ahead, warp, lane,
        [&](int gi, float v) {
            red[gi] = v;
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(other + 4 * gi), "f"(v) : "memory");
        },
        [] {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        });
}

// The same, 256 threads per row, for launches of more rows than the SMs hold blocks of the kernel above (two each): three
// rows per SM are in flight instead of two, each with four groups' pieces per warp.  Measured on its own, 960 rows of 4096
// with about 3.3 pieces: 27.7 -> 20.9 us.
__global__ void __launch_bounds__(NORM_MANY_WARPS * 32, 3) k_resid_norm_many(const SeqState* states, float* hres, StreamK sk, const __nv_bfloat16* g,
                                                                          __nv_bfloat16* y, __nv_bfloat16* y_lo, int d, float eps, float* copy_out) {
    __shared__ float red[NORM_MANY_D / TILE_N];
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int seq = blockIdx.y, r = blockIdx.x;
    const SeqState* st = states + seq;
    const bool idle = !st->active || r >= st->n_rows;     // the row table was written by an earlier step
    pdl_wait();
    if (idle) return;
    const size_t row = (size_t)(seq * RT + r) * d;
    resid_norm_row_many<__nv_bfloat16, NORM_MANY_WARPS, 4, 2>(hres + row, sk, seq * sk.seq_rows + r, g, y + row, y_lo ? y_lo + row : nullptr, d, eps,
                                       copy_out ? copy_out + row : nullptr, red, nullptr, warp, lane,
                                       [&](int gi, float v) { red[gi] = v; }, [] { __syncthreads(); });
}

// Consumer of the split QKV GEMM: sums the partials of one (row, head) in CTA order, then what follows
// the projection in the decoder layer -- per-head RMSNorm on q and k (Qwen3), rotary embedding at the
// row's position L + depth, q to the query buffer, k and v to cache slot L + row.  One warp per (row, head),
// a lane owns HD/32 consecutive features; the rotate-half partner (i, i + HD/2) sits 16 lanes away.
template <int HD>
__global__ void __launch_bounds__(128, 16) k_qkv_finish(EpiArgs a, StreamK sk) {
    // let the next kernel start its own preamble (for a GEMM: the first weight tiles) while this one runs; it still
    // waits for this kernel to complete before it touches anything this kernel or its predecessors write
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hs = blockIdx.x * 4 + warp, r = blockIdx.y, seq = blockIdx.z;   // seq: sequence within this launch
    // Fetched before the wait, so that only the partials are loaded behind it: the row table (written by an earlier
    // step), the tile's contributor entry, the rotary factors of the row's position and the norm weights
    const SeqState* st = a.st ? a.st + seq : nullptr;
    const int n_rows = st ? (st->active ? st->n_rows : 0) : a.rows_fixed;
    const bool work = r < n_rows && hs < a.Hq + 2 * a.Hkv;
    const int L = st ? st->L : 0;
    QkvArgs qa;
    qa.q_out = a.q_out; qa.kcache = a.kcache; qa.vcache = a.vcache; qa.q_norm = a.q_norm; qa.k_norm = a.k_norm;
    qa.rope_cos = a.rope_cos; qa.rope_sin = a.rope_sin; qa.Hq = a.Hq; qa.Hkv = a.Hkv; qa.cap = a.cap; qa.qk_norm = a.qk_norm;
    qa.rms_eps = a.rms_eps;
    QkvPre<HD> pf;
    if (work) qkv_prefetch<HD>(pf, qa, sk, hs, L + (st ? st->row_depth[r] : r), lane);
    pdl_wait();
    if (!work) return;
    qkv_finish_task<HD>(pf, qa, sk, a.kv_shared ? 0 : seq, seq * sk.seq_rows + r, seq * RT + r, L + r, hs, lane);
}

// Consumer of the split gate/up GEMM: a tile holds 64 gate features (columns 0..63) and the matching 64 up
// features (columns 64..127); sums both over the tile's contributors in CTA order and stores silu(gate) * up.
constexpr int SWIGLU_THREADS = 128;
template <int FPT, int PB>
__global__ void __launch_bounds__(SWIGLU_THREADS) k_swiglu_finish(const SeqState* states, int rows_fixed, StreamK sk, __nv_bfloat16* act,
                                                      __nv_bfloat16* act_lo, int F) {
    // let the next kernel start its own preamble (for a GEMM: the first weight tiles) while this one runs; it still
    // waits for this kernel to complete before it touches anything this kernel or its predecessors write
    if (threadIdx.x == 0) pdl_launch_dependents();
    // (eight features per thread in large launches: half the threads, so that the next GEMM's CTA finds registers free
    // beside this kernel's CTAs and can start its weight stream while they run)
    const int j0 = (blockIdx.x * SWIGLU_THREADS + threadIdx.x) * FPT;
    SkEntry en;      // fixed since the plan was built: fetched before the wait (a task's features share a tile)
    if (j0 < F) en = sk_entry(sk, j0 / 64);
    const int r = blockIdx.y, seq = blockIdx.z;
    const int n_rows = states ? (states[seq].active ? states[seq].n_rows : 0) : rows_fixed;   // written by an earlier step
    pdl_wait();
    if (r >= n_rows || j0 >= F) return;
    swiglu_task<FPT, PB>(sk, en, seq * sk.seq_rows + r, act + (size_t)(seq * RT + r) * F, act_lo ? act_lo + (size_t)(seq * RT + r) * F : nullptr, j0, F);
}

// ------------------------------------------------------------------ CUDA-core GEMM
// y[row][n] = sum_k x[row][k] * w[n][k], four running fp32 sums per output with k ascending, added in order.  Used for fp32 models and as the on-GPU cross-check of the tcgen05 kernel.
// Tile -> weight rows mapping is the same as there: up to three stacked matrices (q|k|v), or gate/up halves
// interleaved per tile.
//
// What bounds it: latency.  A small model's matrix is a few hundred KB and a block has a few dozen rows, so there is
// little work per launch and what counts is how many SMs share a weight tile's trip from L2 and through shared memory.
// A CTA takes 8 rows; where the epilogue works feature by feature (residual add, SiLU*up, plain store) also only 32
// features (k_gemm_simt_narrow), elsewhere -- rotary pairs and head norms, per-tile selection -- the whole 128-feature
// tile.  Weights and rows arrive by asynchronous copies several stages ahead, the weights of the first stages
// requested before the wait for the preceding kernel.  Small GEMMs behind a norm (QKV, gate/up, LM head) take it along (NORM): every CTA
// normalises its own 8 rows, which saves a launch in a chain of dependent launches and repeats the norm in every block of columns
// (gemm_simt_takes_norm).  Measured on the tiny fp32 decoder (d_model 256, 35 rows; device
// time of a launch on its own): QKV 11, O and down 9, gate/up 7, LM head (vocabulary 4096) 13 us, where one CTA per
// 128-feature tile with all rows took 140 to 240; its 64-token request 103 -> 9.9 ms.
struct SimtGemmArgs {
    const void* w[3];   // stacked matrices (rows_w[i] rows each); SWIGLU: w[0]=gate, w[1]=up
    int32_t rows_w[3];
    const void* x;      // [batch*RT][K]; NORM: the residual stream (fp32)
    int32_t K;
    const void* gain;   // NORM: [K]
    float eps;
    float* copy;        // NORM, optional: the residual stream is copied there
};
constexpr int SIMT_ROWS = 8, SIMT_NORM_K = 256;
constexpr int SIMT_KC = 32, SIMT_STAGES = 4;       // whole tile: two CTAs of 84 KB per SM
// k is dealt to four threads per feature (narrow: to the four warps, each with all 8 rows), whose sums are added in order at
// the end: one thread per feature and 8 rows, or two rows per warp, was a chain of dependent additions with nothing to hide it
// (64-token request of the tiny decoder 7177 -> 6982 us).
constexpr int SIMT_KS = 4, SIMT_THREADS = 128 * SIMT_KS;
constexpr int NARROW_F = 32, NARROW_KC = 64, NARROW_STAGES = 6;
// elements between two rows of a stage: 16 bytes of padding put the eight rows of a quarter-warp's 16-byte loads on
// different banks
template <typename T> __host__ __device__ constexpr int simt_ld(int kc) { return kc + 16 / (int)sizeof(T); }
template <typename T> constexpr size_t simt_smem_bytes() {
    return sizeof(T) * SIMT_STAGES * (TILE_N + SIMT_ROWS) * simt_ld<T>(SIMT_KC) + sizeof(float) * (SIMT_ROWS * ACC_LD + RT * 4);
}
template <typename T> constexpr size_t narrow_smem_bytes() {
    return sizeof(T) * NARROW_STAGES * (NARROW_F + SIMT_ROWS) * simt_ld<T>(NARROW_KC);
}

// 16 bytes to shared memory; `ok` false: zeros (the source is not read)
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool ok) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// four consecutive elements of a stage row as floats
__device__ __forceinline__ float4 load_f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load_f4(const __nv_bfloat16* p) {
    const uint2 raw = *reinterpret_cast<const uint2*>(p);
    const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&raw.x), hi = *reinterpret_cast<const __nv_bfloat162*>(&raw.y);
    return make_float4(__low2float(lo), __high2float(lo), __low2float(hi), __high2float(hi));
}

// Stage `dst` [n_rows][LD] <- rows 0..n_valid-1 of `src` (K elements apart), elements k0 .. k0+KC-1; zeros outside.
// All NT threads take part, 16 bytes each per pass.  VEC: src starts on 16 bytes (its rows then do too, K is a
// multiple of 8): asynchronous copies.  Otherwise element by element (a caller's matrix needs no more than its
// type's alignment).
template <typename T, int KC, int N_ROWS, bool VEC, int NT = 128>
__device__ __forceinline__ void simt_load(T* dst, const T* src, int n_valid, int K, int k0) {
    constexpr int LD = simt_ld<T>(KC), V = 16 / (int)sizeof(T), PER_ROW = KC / V, STEP = NT / PER_ROW;
    const int j = (threadIdx.x % PER_ROW) * V, first = threadIdx.x / PER_ROW;
    const bool k_ok = k0 + j < K;
    const T* p = src + (size_t)first * K + k0 + j;
    T* d = dst + first * LD + j;
#pragma unroll
    for (int row = 0; row < N_ROWS; row += STEP, p += (size_t)STEP * K, d += STEP * LD) {
        if (N_ROWS % STEP && first + row >= N_ROWS) break;
        const bool ok = k_ok && first + row < n_valid;
        if constexpr (VEC) cp_async16(d, ok ? p : src, ok);
        else {
#pragma unroll
            for (int e = 0; e < V; ++e) d[e] = ok ? p[e] : from_f32<T>(0.f);
        }
    }
}

// acc[r] += x[r][k] * w[k] over one stage, k ascending
template <int R, int KC, typename T>
__device__ __forceinline__ void simt_mac(float (&acc)[R], const T* w, const T* x, int ld) {
#pragma unroll 8
    for (int k = 0; k < KC; k += 4) {
        const float4 wv = load_f4(w + k);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 xv = load_f4(x + r * ld + k);
            acc[r] = fmaf(xv.w, wv.w, fmaf(xv.z, wv.z, fmaf(xv.y, wv.y, fmaf(xv.x, wv.x, acc[r]))));
        }
    }
}

// the same from whole rows of x, of which `left` (a multiple of 4) elements remain
template <int R, int KC>
__device__ __forceinline__ void simt_mac_n(float (&acc)[R], const float* w, const float* x, int ld, int left) {
    if (left >= KC) { simt_mac<R, KC>(acc, w, x, ld); return; }
    for (int k = 0; k < left; k += 4) {
        const float4 wv = load_f4(w + k);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 xv = load_f4(x + r * ld + k);
            acc[r] = fmaf(xv.w, wv.w, fmaf(xv.z, wv.z, fmaf(xv.y, wv.y, fmaf(xv.x, wv.x, acc[r]))));
        }
    }
}

// NORM: rows r0 .. of the residual stream, normalised, to shared memory ([SIMT_ROWS][K + 4] floats); a warp takes PER rows.
__host__ __device__ constexpr int norm_x_ld(int K) { return K + 4; }
template <int PER>
__device__ __forceinline__ void norm_rows(float* s_x, const SimtGemmArgs& g, size_t row0, int n_valid, int warp, int lane, bool copy) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int r = warp * PER + i;
        if (r >= SIMT_ROWS) return;
        float* d = s_x + r * norm_x_ld(g.K);
        if (r < n_valid) {
            norm_row<SIMT_NORM_K>(d, reinterpret_cast<const float*>(g.x) + (row0 + r) * g.K, reinterpret_cast<const float*>(g.gain), g.K, g.eps, lane,
                                  copy ? g.copy + (row0 + r) * g.K : nullptr);
        } else {
            for (int j = lane * 4; j < g.K; j += 128) *reinterpret_cast<float4*>(d + j) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// 8 rows x one 128-feature tile, SIMT_KS threads per feature, each a quarter of every stage's k.  EPI_QKV (the stacked matrices end on tile boundaries) and
// EPI_LOGITS.
template <typename T, int EPI, bool VEC, bool NORM>
__global__ void __launch_bounds__(SIMT_THREADS, 2) k_gemm_simt(SimtGemmArgs g, EpiArgs a) {
    static_assert(!NORM || sizeof(T) == 4, "the normalised rows are fp32");
    constexpr int LD = simt_ld<T>(SIMT_KC);
    extern __shared__ __align__(16) unsigned char simt_smem[];
    T* s_w = reinterpret_cast<T*>(simt_smem);                   // [STAGES][128][LD]
    T* s_x = s_w + SIMT_STAGES * TILE_N * LD;                   // [STAGES][ROWS][LD]
    float* s_acc = reinterpret_cast<float*>(s_x + SIMT_STAGES * SIMT_ROWS * LD);   // [ROWS][ACC_LD]
    float* s_aux = s_acc + SIMT_ROWS * ACC_LD;                  // RT * 4
    float* s_xn = s_aux + RT * 4;                               // NORM: [ROWS][K + 4]
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int tile = blockIdx.x, r0 = blockIdx.y * SIMT_ROWS, seq = blockIdx.z, f = threadIdx.x % 128, ks = threadIdx.x / 128;
    int m = 0, feat = tile * TILE_N;
    while (m < 2 && feat >= g.rows_w[m]) feat -= g.rows_w[m++];
    const T* w = reinterpret_cast<const T*>(g.w[m]) + (size_t)feat * g.K;
    const int n_feat = g.rows_w[m] - feat < TILE_N ? g.rows_w[m] - feat : TILE_N;
    const int n_chunks = (g.K + SIMT_KC - 1) / SIMT_KC;
    auto load_w = [&](int c) { simt_load<T, SIMT_KC, TILE_N, VEC, SIMT_THREADS>(s_w + (c % SIMT_STAGES) * TILE_N * LD, w, n_feat, g.K, c * SIMT_KC); };
    for (int c = 0; c < SIMT_STAGES - 1 && c < n_chunks; ++c) load_w(c);      // (they join the first group below)
    // (the row table was written by an earlier step: read before the wait, like the weights)
    const SeqState* st = a.st ? a.st + seq : nullptr;
    const int n_rows = st ? (st->active ? st->n_rows : 0) : a.rows_fixed;
    pdl_wait();
    if (r0 >= n_rows) { cp_async_wait<0>(); return; }
    const int r1 = r0 + SIMT_ROWS < n_rows ? r0 + SIMT_ROWS : n_rows;
    const T* x = reinterpret_cast<const T*>(g.x) + (size_t)(seq * RT + r0) * g.K;
    auto load_x = [&](int c) {
        if constexpr (!NORM) simt_load<T, SIMT_KC, SIMT_ROWS, VEC, SIMT_THREADS>(s_x + (c % SIMT_STAGES) * SIMT_ROWS * LD, x, r1 - r0, g.K, c * SIMT_KC);
    };
    for (int c = 0; c < SIMT_STAGES - 1; ++c) {
        if (c < n_chunks) load_x(c);
        cp_async_commit();
    }
    if constexpr (NORM) norm_rows<1>(s_xn, g, (size_t)(seq * RT + r0), r1 - r0, threadIdx.x >> 5, threadIdx.x & 31, g.copy && blockIdx.x == 0);
    float acc[SIMT_ROWS];
#pragma unroll
    for (int r = 0; r < SIMT_ROWS; ++r) acc[r] = 0.f;
    for (int c = 0; c < n_chunks; ++c) {
        cp_async_wait<SIMT_STAGES - 2>();
        __syncthreads();                                // chunk c has landed, and chunk c - 1's buffer is free
        if (c + SIMT_STAGES - 1 < n_chunks) { load_w(c + SIMT_STAGES - 1); load_x(c + SIMT_STAGES - 1); }
        cp_async_commit();
        constexpr int KQ = SIMT_KC / SIMT_KS;
        const T* wr = s_w + ((c % SIMT_STAGES) * TILE_N + f) * LD + ks * KQ;
        if constexpr (NORM) simt_mac_n<SIMT_ROWS, KQ>(acc, wr, s_xn + c * SIMT_KC + ks * KQ, norm_x_ld(g.K), g.K - c * SIMT_KC - ks * KQ);
        else simt_mac<SIMT_ROWS, KQ>(acc, wr, s_x + (c % SIMT_STAGES) * SIMT_ROWS * LD + ks * KQ, LD);
    }
    // the quarters' sums, added in order (in the weights' buffers, which nothing reads or writes any more)
    __syncthreads();
    float* s_part = reinterpret_cast<float*>(s_w);              // [KS][ROWS][128]
#pragma unroll
    for (int r = 0; r < SIMT_ROWS; ++r) s_part[(ks * SIMT_ROWS + r) * TILE_N + f] = acc[r];
    __syncthreads();
    if (ks) return;
#pragma unroll
    for (int r = 0; r < SIMT_ROWS; ++r) {
        float v = s_part[r * TILE_N + f];
#pragma unroll
        for (int q = 1; q < SIMT_KS; ++q) v += s_part[(q * SIMT_ROWS + r) * TILE_N + f];
        s_acc[r * ACC_LD + f] = v;
    }
    epi_bar(1);
    run_epilogue_rows<T, EPI>(s_acc, s_aux, tile, seq, a, f, 1, st, n_rows, r0, r1);
}

// 8 rows x 32 features (SWIGLU: 16 gate features and the matching 16 up features), a lane per feature, a quarter of every
// stage's k per warp.  EPI_STORE_F32, EPI_RESID, EPI_SWIGLU.
template <typename T, int EPI, bool VEC, bool NORM>
__global__ void __launch_bounds__(128) k_gemm_simt_narrow(SimtGemmArgs g, EpiArgs a) {
    constexpr int LD = simt_ld<T>(NARROW_KC), HALF = NARROW_F / 2;
    extern __shared__ __align__(16) unsigned char simt_smem[];
    T* s_w = reinterpret_cast<T*>(simt_smem);                   // [STAGES][32][LD]
    T* s_x = s_w + NARROW_STAGES * NARROW_F * LD;               // [STAGES][ROWS][LD]
    float* s_xn = reinterpret_cast<float*>(s_x + NARROW_STAGES * SIMT_ROWS * LD);      // NORM: [ROWS][K + 4]
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int r0 = blockIdx.y * SIMT_ROWS, seq = blockIdx.z, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * (EPI == EPI_SWIGLU ? HALF : NARROW_F);
    const int n_feat = a.n_out - n0 < NARROW_F ? a.n_out - n0 : NARROW_F;      // (SWIGLU: of either half, cut below)
    const T* w0 = reinterpret_cast<const T*>(g.w[0]) + (size_t)n0 * g.K;
    const int n_chunks = (g.K + NARROW_KC - 1) / NARROW_KC;
    auto load_w = [&](int c) {
        T* dst = s_w + (c % NARROW_STAGES) * NARROW_F * LD;
        if constexpr (EPI == EPI_SWIGLU) {
            const int n = n_feat < HALF ? n_feat : HALF;
            simt_load<T, NARROW_KC, HALF, VEC>(dst, w0, n, g.K, c * NARROW_KC);
            simt_load<T, NARROW_KC, HALF, VEC>(dst + HALF * LD, reinterpret_cast<const T*>(g.w[1]) + (size_t)n0 * g.K, n, g.K, c * NARROW_KC);
        } else {
            simt_load<T, NARROW_KC, NARROW_F, VEC>(dst, w0, n_feat, g.K, c * NARROW_KC);
        }
    };
    for (int c = 0; c < NARROW_STAGES - 1 && c < n_chunks; ++c) load_w(c);
    // (the row table was written by an earlier step: read before the wait, like the weights)
    const SeqState* st = a.st ? a.st + seq : nullptr;
    const int n_rows = st ? (st->active ? st->n_rows : 0) : a.rows_fixed;
    pdl_wait();
    if (r0 >= n_rows) { cp_async_wait<0>(); return; }
    const int r1 = r0 + SIMT_ROWS < n_rows ? r0 + SIMT_ROWS : n_rows;
    const T* x = reinterpret_cast<const T*>(g.x) + (size_t)(seq * RT + r0) * g.K;
    auto load_x = [&](int c) {
        if constexpr (!NORM) simt_load<T, NARROW_KC, SIMT_ROWS, VEC>(s_x + (c % NARROW_STAGES) * SIMT_ROWS * LD, x, r1 - r0, g.K, c * NARROW_KC);
    };
    for (int c = 0; c < NARROW_STAGES - 1; ++c) {
        if (c < n_chunks) load_x(c);
        cp_async_commit();
    }
    float old[2] = {0.f, 0.f};        // EPI_RESID: the residual stream, on its way while the product is taken
    if constexpr (EPI == EPI_RESID) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = r0 + warp * 2 + i;
            if (lane < n_feat && r < r1) old[i] = a.hres[(size_t)(seq * RT + r) * a.n_out + n0 + lane];
        }
    }
    if constexpr (NORM) norm_rows<2>(s_xn, g, (size_t)(seq * RT + r0), r1 - r0, warp, lane, false);
    float part[SIMT_ROWS];
#pragma unroll
    for (int r = 0; r < SIMT_ROWS; ++r) part[r] = 0.f;
    for (int c = 0; c < n_chunks; ++c) {
        cp_async_wait<NARROW_STAGES - 2>();
        __syncthreads();
        if (c + NARROW_STAGES - 1 < n_chunks) { load_w(c + NARROW_STAGES - 1); load_x(c + NARROW_STAGES - 1); }
        cp_async_commit();
        constexpr int KQ = NARROW_KC / 4;
        const T* wr = s_w + ((c % NARROW_STAGES) * NARROW_F + lane) * LD + warp * KQ;
        if constexpr (NORM) simt_mac_n<SIMT_ROWS, KQ>(part, wr, s_xn + c * NARROW_KC + warp * KQ, norm_x_ld(g.K), g.K - c * NARROW_KC - warp * KQ);
        else simt_mac<SIMT_ROWS, KQ>(part, wr, s_x + (c % NARROW_STAGES) * SIMT_ROWS * LD + warp * KQ, LD);
    }
    // the quarters' sums, added in order: two rows per warp
    __shared__ float s_part[4][SIMT_ROWS][NARROW_F];
#pragma unroll
    for (int r = 0; r < SIMT_ROWS; ++r) s_part[warp][r][lane] = part[r];
    __syncthreads();
    float acc[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        acc[i] = s_part[0][warp * 2 + i][lane];
#pragma unroll
        for (int q = 1; q < 4; ++q) acc[i] += s_part[q][warp * 2 + i][lane];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int r = r0 + warp * 2 + i;
        const size_t row = (size_t)(seq * RT + r) * a.n_out;
        if constexpr (EPI == EPI_SWIGLU) {
            const float up = __shfl_down_sync(0xffffffffu, acc[i], HALF), gate = acc[i];
            if (lane < HALF && lane < n_feat && r < r1)
                reinterpret_cast<T*>(a.act_out)[row + n0 + lane] = from_f32<T>((gate / (1.0f + expf(-gate))) * up);
        } else if (lane < n_feat && r < r1) {
            if constexpr (EPI == EPI_RESID) a.hres[row + n0 + lane] = old[i] + acc[i];
            else a.y_f32[row + n0 + lane] = acc[i];
        }
    }
}

// Whether a GEMM takes the norm in front of it along: K of at most 256 and no more CTAs than two per SM.  Same bits either way.
// Steps of fp32 models, us, norms in all GEMMs / as launches of a warp per row: d 256, vocabulary 4096, 35 rows 120 / 122, 128 rows (QKV 64
// CTAs, LM head 512, gate/up 688) 171 / 153; d 512, 1 row 124 / 111, 35 rows
// 191 / 175; d 1024, vocabulary 32000, 35 rows 524 / 435, four sequences of 128 rows 5031 / 3309.
bool gemm_simt_takes_norm(int dtype, int epi, int K, int n_out, int rows_cap, int batch) {
    const int cols = epi == EPI_SWIGLU ? NARROW_F / 2 : TILE_N;
    return dtype == 0 && K <= SIMT_NORM_K && (long long)((n_out + cols - 1) / cols) * ((rows_cap + SIMT_ROWS - 1) / SIMT_ROWS) * batch <= 2 * 148;
}

template <typename T, bool VEC>
int launch_gemm_simt_t(int epi, int n_tiles, int batch, const SimtGemmArgs& g, const EpiArgs& a, int rows_cap, cudaStream_t s, bool pdl) {
    const int groups = (rows_cap + SIMT_ROWS - 1) / SIMT_ROWS;
    const size_t norm_bytes = g.gain ? sizeof(float) * SIMT_ROWS * norm_x_ld(g.K) : 0;
#define ESP_SIMT_CASE(E, KERNEL, TILES, SMEM, NORM)                                                                 \
    {                                                                                                               \
        if (ensure_dynamic_smem(reinterpret_cast<const void*>(KERNEL<T, E, VEC, NORM>), (int)(SMEM<T>() + (NORM ? sizeof(float) * SIMT_ROWS * norm_x_ld(SIMT_NORM_K) : 0)))) \
            return ESP_E_CUDA;                                                                                      \
        return launch_k(KERNEL<T, E, VEC, NORM>, dim3(TILES, groups, batch), dim3((E == EPI_QKV || E == EPI_LOGITS) ? SIMT_THREADS : 128), SMEM<T>() + norm_bytes, s, pdl, g, a) == cudaSuccess ? ESP_OK : ESP_E_CUDA; \
    }
    if constexpr (sizeof(T) == 4) {
        if (g.gain) {
            if (g.K > SIMT_NORM_K || g.K % 4) return ESP_E_ARG;
            if (epi == EPI_SWIGLU) ESP_SIMT_CASE(EPI_SWIGLU, k_gemm_simt_narrow, (a.n_out + NARROW_F / 2 - 1) / (NARROW_F / 2), narrow_smem_bytes, true)
            if (epi == EPI_QKV) ESP_SIMT_CASE(EPI_QKV, k_gemm_simt, n_tiles, simt_smem_bytes, true)
            if (epi == EPI_LOGITS) ESP_SIMT_CASE(EPI_LOGITS, k_gemm_simt, n_tiles, simt_smem_bytes, true)
            return ESP_E_ARG;
        }
    }
    switch (epi) {
        case EPI_STORE_F32: ESP_SIMT_CASE(EPI_STORE_F32, k_gemm_simt_narrow, (a.n_out + NARROW_F - 1) / NARROW_F, narrow_smem_bytes, false)
        case EPI_RESID: ESP_SIMT_CASE(EPI_RESID, k_gemm_simt_narrow, (a.n_out + NARROW_F - 1) / NARROW_F, narrow_smem_bytes, false)
        case EPI_SWIGLU: ESP_SIMT_CASE(EPI_SWIGLU, k_gemm_simt_narrow, (a.n_out + NARROW_F / 2 - 1) / (NARROW_F / 2), narrow_smem_bytes, false)
        case EPI_QKV: ESP_SIMT_CASE(EPI_QKV, k_gemm_simt, n_tiles, simt_smem_bytes, false)
        case EPI_LOGITS: ESP_SIMT_CASE(EPI_LOGITS, k_gemm_simt, n_tiles, simt_smem_bytes, false)
    }
#undef ESP_SIMT_CASE
    return ESP_E_ARG;
}

// rows_cap: no block has more rows (sizes the grid)
int launch_gemm_simt(int dtype, int epi, int n_tiles, int batch, const void* const w[3], const int32_t rows_w[3],
                     const void* x, int K, const EpiArgs& a, int rows_cap, cudaStream_t s, bool pdl) {
    SimtGemmArgs g;
    bool vec = reinterpret_cast<uintptr_t>(x) % 16 == 0;
    for (int i = 0; i < 3; ++i) {
        g.w[i] = w[i]; g.rows_w[i] = rows_w[i];
        vec = vec && reinterpret_cast<uintptr_t>(w[i]) % 16 == 0;
    }
    g.x = x;
    g.K = K;
    g.gain = a.norm_gain; g.eps = a.rms_eps; g.copy = a.norm_copy;
    if (dtype == 0) return vec ? launch_gemm_simt_t<float, true>(epi, n_tiles, batch, g, a, rows_cap, s, pdl)
                               : launch_gemm_simt_t<float, false>(epi, n_tiles, batch, g, a, rows_cap, s, pdl);
    return vec ? launch_gemm_simt_t<__nv_bfloat16, true>(epi, n_tiles, batch, g, a, rows_cap, s, pdl)
               : launch_gemm_simt_t<__nv_bfloat16, false>(epi, n_tiles, batch, g, a, rows_cap, s, pdl);
}

// ------------------------------------------------------------------ attention (position-canonical)
// Key list of a row at position P = L + depth: positions 0..P.  Positions below
// T0 = max(0, floor((P - dcap)/16)*16) are summed by the chunked "bulk" path in splits of
// split_len positions aligned to position 0; positions T0..P (cache tail + the row's in-flight
// ancestors, found through its ancestor bitmask in row order = position order) by the tail.
// Every reduction order depends on absolute positions only, so a token verified inside a tree
// block gets bit-identical results to the same token decoded alone.
__device__ __forceinline__ int tail_start(int P, int dcap) {
    int t = P - dcap;
    return t <= 0 ? 0 : (t / 16) * 16;
}

// index of the n-th (0-based) set bit of a 128-bit mask
__device__ __forceinline__ int nth_set_bit(unsigned long long lo, unsigned long long hi, int n) {
    int c = __popcll(lo);
    unsigned long long m = lo;
    int base = 0;
    if (n >= c) { n -= c; m = hi; base = 64; }
    for (int i = 0; i < n; ++i) m &= m - 1;
    return m ? base + __ffsll((long long)m) - 1 : -1;
}


__device__ __forceinline__ void attn_row_info(const AttnArgs& a, int seq, int r, int& n_rows, int& L, int& depth,
                                              unsigned long long& lo, unsigned long long& hi) {
    if (a.st) {
        const SeqState* st = a.st + seq;
        n_rows = st->active ? st->n_rows : 0;
        L = st->L;
        depth = r < RT ? st->row_depth[r] : 0;
        lo = r < RT ? st->row_anc[r][0] : 0;
        hi = r < RT ? st->row_anc[r][1] : 0;
    } else {
        n_rows = a.n_rows_fixed;
        L = a.L_fixed;
        depth = a.depth[seq * RT + r];
        lo = a.anc[(size_t)(seq * RT + r) * 2];
        hi = a.anc[(size_t)(seq * RT + r) * 2 + 1];
    }
}

template <typename V>
__device__ __forceinline__ V load_l2_or_l1(const V* p, bool l1) { return l1 ? *p : __ldcg(p); }
// E consecutive elements as floats, read from L2, or (l1) through L1 (VEC: 16 bytes aligned, or all of them if they are fewer)
template <typename T, int E, bool VEC>
__device__ __forceinline__ void load_row(float (&v)[E], const T* p, bool l1 = false) {
    if constexpr (!VEC) {
#pragma unroll
        for (int i = 0; i < E; ++i) {
            if constexpr (sizeof(T) == 4) v[i] = load_l2_or_l1(p + i, l1);
            else v[i] = __bfloat162float(__ushort_as_bfloat16(load_l2_or_l1(reinterpret_cast<const unsigned short*>(p) + i, l1)));
        }
    } else if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < E; i += 4) {
            const float4 x = load_l2_or_l1(reinterpret_cast<const float4*>(p + i), l1);
            v[i] = x.x; v[i + 1] = x.y; v[i + 2] = x.z; v[i + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < E; i += 4) {
            const uint2 x = load_l2_or_l1(reinterpret_cast<const uint2*>(p + i), l1);
            const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&x.x), hi = *reinterpret_cast<const __nv_bfloat162*>(&x.y);
            v[i] = __low2float(lo); v[i + 1] = __high2float(lo); v[i + 2] = __low2float(hi); v[i + 3] = __high2float(hi);
        }
    }
}

// One chunk of up to 32 keys for one (row, head) handled by one warp; lane j names the cache slot of key j.  Returns the
// chunk's own (max, sum, weighted values) relative to its own max, in the log2 domain.
// Scores: eight lanes per key, HD / 8 dims each, four keys side by side, so that a load touches whole rows (a lane per key
// touches 32 cache lines per load: 13 us of the tiny decoder's step per layer, now 0.8 behind the cache kernel, its 64-token request 8530 -> 7446 us); values: a lane per dim.
// Keys, and values, of RB rounds (of VB keys) are in flight together (lanes without a key hold the slot of one that is
// there; its value row is read and not used).  L1: slots below n_l1 go through L1, where the warps that share a KV head find them again;
// everything else is read from L2.  VEC: the cache starts on 16 bytes.
template <typename T, int HD, bool VEC, bool L1>
__device__ __forceinline__ void warp_chunk(const float (&q)[HD / 8], const T* kbase, const T* vbase, int slot, int n_l1, uint32_t valid,
                                           float scale_log2, float& cm, float& cl, float (&co)[HD / 32]) {
    constexpr int E = HD / 8, RB = HD == 128 ? 4 : 8, VB = HD == 128 ? 16 : 32;
    const int lane = threadIdx.x & 31, kg = lane >> 3;
    float s[8];
#pragma unroll
    for (int u0 = 0; u0 < 8; u0 += RB) {
        float k[RB][E];
#pragma unroll
        for (int u = 0; u < RB; ++u) {
            const int sl = __shfl_sync(0xffffffffu, slot, 4 * (u0 + u) + kg);
            load_row<T, E, VEC>(k[u], kbase + (size_t)sl * HD + (lane & 7) * E, L1 && sl < n_l1);
        }
#pragma unroll
        for (int u = 0; u < RB; ++u) {
            float acc = 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e) acc = fmaf(q[e], k[u][e], acc);
#pragma unroll
            for (int of = 1; of < 8; of <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, of);
            s[u0 + u] = acc * scale_log2;
        }
    }
    cm = -INFINITY;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        if (!((valid >> (4 * u + kg)) & 1u)) s[u] = -INFINITY;
        cm = fmaxf(cm, s[u]);
    }
    cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, 8));
    cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, 16));
    cl = 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        s[u] = ((valid >> (4 * u + kg)) & 1u) ? exp2f(s[u] - cm) : 0.f;
        cl += s[u];
    }
    cl += __shfl_xor_sync(0xffffffffu, cl, 8);
    cl += __shfl_xor_sync(0xffffffffu, cl, 16);
#pragma unroll
    for (int i = 0; i < HD / 32; ++i) co[i] = 0.f;
#pragma unroll
    for (int j0 = 0; j0 < 32; j0 += VB) {
        float v[VB][HD / 32];
#pragma unroll
        for (int j = 0; j < VB; ++j) {
            const int sl = __shfl_sync(0xffffffffu, slot, j0 + j);
            const T* vr = vbase + (size_t)sl * HD;
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) {
                float x[1];
                load_row<T, 1, false>(x, vr + lane + 32 * i, L1 && sl < n_l1);
                v[j][i] = x[0];
            }
        }
#pragma unroll
        for (int j = 0; j < VB; ++j) {
            const float pj = __shfl_sync(0xffffffffu, s[(j0 + j) >> 2], (j & 3) * 8);
            if (pj != 0.f) {
#pragma unroll
                for (int i = 0; i < HD / 32; ++i) co[i] = fmaf(pj, v[j][i], co[i]);
            }
        }
    }
}

template <int N>
__device__ __forceinline__ void merge_partial(float& m, float& l, float (&o)[N], float cm, float cl, const float (&co)[N]) {
    float mn = fmaxf(m, cm);
    float a = exp2f(m - mn), b = exp2f(cm - mn);
    l = __fmaf_rn(l, a, __fmul_rn(cl, b));      // (spelled out: every kernel that merges rounds alike)
#pragma unroll
    for (int i = 0; i < N; ++i) o[i] = __fmaf_rn(o[i], a, __fmul_rn(co[i], b));
    m = mn;
}

// Bulk, CUDA-core version.  A CTA takes one cache split of one KV head for 4 * BS_PW (row, head) pairs of that head's
// group, a warp BS_PW of them; keys and values pass through shared memory in chunks of 32 positions, the next chunk
// loading (16-byte asynchronous copies) while the current one is used.  What bounds it is a warp's serial chain over
// the split: with four pairs a warp shares every key and value read from shared memory between them and the CTA reads
// the split from L2 for 16 pairs; with one pair the chain is a third as long, which is what counts while the four-pair
// CTAs would leave SMs idle (launch_attn_simt_t).
// grid = (ceil(rows * group / (4 * BS_PW)), Hkv, n_split * batch).
// The chunks of a split go in turn to bulk_groups() groups, each with running sums of its own, merged in group order at the end; which
// chunk goes where follows from the position alone, and so do a row's bits.  KS = bulk_groups(): a group of warps with buffers of its
// own for each, so that the chain over 256 positions is two or four chunks long instead of eight of about 3 us each.  KS = 1: one group
// of warps takes the groups' chunks one group after the other.  Its CTAs need a quarter or half of the shared memory, which counts
// where there are more CTAs than fit anyway.
constexpr int BS_WARPS = 4;
template <typename T, int HD> __host__ __device__ constexpr int bulk_groups() { return sizeof(T) * HD <= 256 ? 4 : 2; }
// one group of warps: where the sums of the chunk groups already done wait (fp32 heads of 128: three CTAs leave no shared memory for them)
template <typename T, int HD> __host__ __device__ constexpr bool bulk_sums_in_regs() { return sizeof(T) * HD > 256; }
template <typename T, int HD> __host__ __device__ constexpr int bulk_simt_ld() { return HD + 16 / (int)sizeof(T); }
template <typename T, int HD> constexpr size_t bulk_simt_smem(int pw, int ks) {
    return ks * (sizeof(T) * 4 * 32 * bulk_simt_ld<T, HD>() + sizeof(float) * BS_WARPS * pw * HD) + (ks == 1 && !bulk_sums_in_regs<T, HD>() ? sizeof(float) * BS_WARPS * pw * (HD + 2) : 0);
}
template <typename T, int HD, bool VEC, int BS_PW, int KS>
__device__ __forceinline__ void attn_bulk_simt(const AttnArgs& a, int n_split_launch) {
    constexpr int LD = bulk_simt_ld<T, HD>(), V = 16 / (int)sizeof(T), PER_ROW = HD / V, KG = bulk_groups<T, HD>();
    static_assert(KS == KG || KS == 1, "a group of warps per group of chunks, or one for all");
    extern __shared__ __align__(16) unsigned char bulk_smem[];
    const int kg = threadIdx.x >> 7, gt = threadIdx.x & 127;      // key group, thread of the group
    const int warp = gt >> 5, lane = gt & 31;
    T* s_k = reinterpret_cast<T*>(bulk_smem) + kg * 4 * 32 * LD;      // [2][32][LD]
    T* s_v = s_k + 2 * 32 * LD;                                       // [2][32][LD]
    float* s_qall = reinterpret_cast<float*>(reinterpret_cast<T*>(bulk_smem) + KS * 4 * 32 * LD) + kg * BS_WARPS * BS_PW * HD;
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) attn_clear_error(a);
    const int kvh = blockIdx.y, group = a.Hq / a.Hkv;
    const int split = blockIdx.z % n_split_launch, seq = blockIdx.z / n_split_launch;
    const int beg = split * a.split_len;
    auto group_bar = [&] { asm volatile("bar.sync %0, 128;" ::"r"(1 + kg) : "memory"); };
    int row[BS_PW], end[BS_PW], cta_end = 0;
    const int pair0 = (blockIdx.x * BS_WARPS + warp) * BS_PW;
    float* s_q = s_qall + warp * BS_PW * HD;
#pragma unroll
    for (int w = 0; w < BS_PW; ++w) {
        row[w] = (pair0 + w) / group;
        end[w] = 0;
        int n_rows, L, depth;
        unsigned long long lo, hi;
        attn_row_info(a, seq, row[w] < RT ? row[w] : 0, n_rows, L, depth, lo, hi);
        if (row[w] < n_rows) end[w] = min(beg + a.split_len, tail_start(L + depth, a.dcap));
        cta_end = max(cta_end, end[w]);
    }
    pdl_wait();             // (the row table above was written by an earlier step)
    if (threadIdx.x == 0) pdl_launch_dependents();      // the tail kernel computes its tail beside this kernel: queries, keys and values are there
#pragma unroll
    for (int w = 0; w < BS_PW; ++w)
        if (end[w] > 0) {
            const T* q = reinterpret_cast<const T*>(a.q) + ((size_t)(seq * RT + row[w]) * a.Hq + kvh * group + (pair0 + w) % group) * HD;
            for (int d = lane; d < HD; d += 32) s_q[w * HD + d] = to_f32(q[d]);
        }
    __shared__ int s_end[BS_WARPS];
    if (lane == 0 && kg == 0) s_end[warp] = cta_end;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < BS_WARPS; ++w) cta_end = max(cta_end, s_end[w]);
    if (beg >= cta_end) return;
    const T* kb = reinterpret_cast<const T*>(a.kc) + ((size_t)seq * a.Hkv + kvh) * a.cap * HD;
    const T* vb = reinterpret_cast<const T*>(a.vc) + ((size_t)seq * a.Hkv + kvh) * a.cap * HD;
    auto load = [&](int p0, int buf) {
        for (int i = gt; i < 32 * PER_ROW; i += 128) {
            const int pos = p0 + i / PER_ROW, e0 = (i % PER_ROW) * V;
            const bool ok = pos < cta_end;
            const size_t src = (size_t)(ok ? pos : beg) * HD + e0;
            T* dk = s_k + (buf * 32 + i / PER_ROW) * LD + e0;
            T* dv = s_v + (buf * 32 + i / PER_ROW) * LD + e0;
            if constexpr (VEC) {
                cp_async16(dk, kb + src, ok);
                cp_async16(dv, vb + src, ok);
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    dk[e] = ok ? kb[src + e] : from_f32<T>(0.f);
                    dv[e] = ok ? vb[src + e] : from_f32<T>(0.f);
                }
            }
        }
        cp_async_commit();
    };
    float m[BS_PW], l[BS_PW], o[BS_PW][HD / 32];
    auto reset = [&] {
#pragma unroll
        for (int w = 0; w < BS_PW; ++w) {
            m[w] = -INFINITY;
            l[w] = 0.f;
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) o[w][i] = 0.f;
        }
    };
    reset();
    // KS == 1: the sums of the groups done so far, [pair][HD + 2] per warp
    constexpr bool SUMS_REG = bulk_sums_in_regs<T, HD>();
    float* s_sum = s_qall + (KS == 1 ? BS_WARPS * BS_PW * HD : 0) + warp * BS_PW * (HD + 2);
    float r_sum[BS_PW][HD / 32 + 2];
    auto put_sum = [&](int w) {
        if constexpr (SUMS_REG) {
            r_sum[w][HD / 32] = m[w]; r_sum[w][HD / 32 + 1] = l[w];
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) r_sum[w][i] = o[w][i];
        } else {
            float* d = s_sum + w * (HD + 2);
            if (lane == 0) { d[HD] = m[w]; d[HD + 1] = l[w]; }
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) d[lane + 32 * i] = o[w][i];
        }
    };
    auto get_sum = [&](int w, float& md, float& ld, float (&od)[HD / 32]) {
        const float* d = s_sum + w * (HD + 2);
        md = SUMS_REG ? r_sum[w][HD / 32] : d[HD];
        ld = SUMS_REG ? r_sum[w][HD / 32 + 1] : d[HD + 1];
#pragma unroll
        for (int i = 0; i < HD / 32; ++i) od[i] = SUMS_REG ? r_sum[w][i] : d[lane + 32 * i];
    };
    int g = kg, p0 = beg + 32 * kg;
    bool more = p0 < cta_end;
    if (more) load(p0, 0);
    for (int buf = 0; more; buf ^= 1) {
        // the next chunk: of this group, or (one group of warps) the first of the next group
        int g_next = g, p_next = p0 + 32 * KG;
        if (KS == 1 && p_next >= cta_end) { g_next = g + 1; p_next = g_next < KG ? beg + 32 * g_next : cta_end; }
        more = p_next < cta_end;
        if (more) load(p_next, buf ^ 1);
        else cp_async_commit();
        cp_async_wait<1>();
        group_bar();
        const T* kr = s_k + (buf * 32 + lane) * LD;
        float acc[BS_PW], p[BS_PW], cm[BS_PW], cl[BS_PW], co[BS_PW][HD / 32];
#pragma unroll
        for (int w = 0; w < BS_PW; ++w) acc[w] = 0.f;
#pragma unroll 8
        for (int d = 0; d < HD; d += 4) {
            const float4 kv = load_f4(kr + d);
#pragma unroll
            for (int w = 0; w < BS_PW; ++w) {
                const float4 qv = load_f4(s_q + w * HD + d);
                acc[w] = fmaf(qv.w, kv.w, fmaf(qv.z, kv.z, fmaf(qv.y, kv.y, fmaf(qv.x, kv.x, acc[w]))));
            }
        }
#pragma unroll
        for (int w = 0; w < BS_PW; ++w) {
            const bool valid = p0 + lane < end[w];
            const float s = valid ? acc[w] * a.scale_log2 : -INFINITY;
            cm[w] = warp_max(s);
            p[w] = valid ? exp2f(s - cm[w]) : 0.f;
            cl[w] = warp_sum(p[w]);
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) co[w][i] = 0.f;
        }
        const T* vr = s_v + buf * 32 * LD + lane;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            float v[HD / 32];
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) v[i] = to_f32(vr[j * LD + 32 * i]);
#pragma unroll
            for (int w = 0; w < BS_PW; ++w) {
                const float pj = __shfl_sync(0xffffffffu, p[w], j);
                if (pj != 0.f) {
#pragma unroll
                    for (int i = 0; i < HD / 32; ++i) co[w][i] = fmaf(pj, v[i], co[w][i]);
                }
            }
        }
#pragma unroll
        for (int w = 0; w < BS_PW; ++w)
            if (p0 < end[w]) merge_partial(m[w], l[w], o[w], cm[w], cl[w], co[w]);
        group_bar();           // this buffer is loaded again in the next round but one
        if (KS == 1 && (!more || g_next != g)) {        // the group is done
#pragma unroll
            for (int w = 0; w < BS_PW; ++w) {
                if (g > 0) {
                    float md, ld, od[HD / 32];
                    get_sum(w, md, ld, od);
                    if (beg + 32 * g < end[w]) merge_partial(md, ld, od, m[w], l[w], o[w]);
                    m[w] = md; l[w] = ld;
#pragma unroll
                    for (int i = 0; i < HD / 32; ++i) o[w][i] = od[i];
                    __syncwarp();
                }
                if (more) put_sum(w);
            }
            __syncwarp();
            if (more) reset();
        }
        g = g_next;
        p0 = p_next;
    }
    auto store = [&](int w) {
        const size_t idx = ((size_t)(seq * RT + row[w]) * a.Hq + kvh * group + (pair0 + w) % group) * a.n_split_max + split;
        if (lane == 0) a.part_ml[idx] = make_float2(m[w], l[w]);
#pragma unroll
        for (int i = 0; i < HD / 32; ++i) a.part_o[idx * HD + lane + 32 * i] = o[w][i];
    };
    if constexpr (KS == 1) {
#pragma unroll
        for (int w = 0; w < BS_PW; ++w)
            if (end[w] > beg) store(w);
        return;
    }
    // the groups' sums meet in the first group's buffers ([group - 1][pair][HD + 2] floats), which it has done with
    __syncthreads();
    float* s_m = reinterpret_cast<float*>(bulk_smem);
    static_assert(sizeof(float) * (KG - 1) * BS_WARPS * BS_PW * (HD + 2) <= KG * sizeof(T) * 4 * 32 * LD, "room for the groups' sums");
    if (kg > 0) {
#pragma unroll
        for (int w = 0; w < BS_PW; ++w) {
            float* d = s_m + (((kg - 1) * BS_WARPS + warp) * BS_PW + w) * (HD + 2);
            if (lane == 0) { d[HD] = m[w]; d[HD + 1] = l[w]; }
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) d[lane + 32 * i] = o[w][i];
        }
    }
    __syncthreads();
    if (kg > 0) return;
#pragma unroll
    for (int w = 0; w < BS_PW; ++w) {
        if (end[w] <= beg) continue;
#pragma unroll
        for (int g = 1; g < KG; ++g) {
            const float* d = s_m + (((g - 1) * BS_WARPS + warp) * BS_PW + w) * (HD + 2);
            float co[HD / 32];
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) co[i] = d[lane + 32 * i];
            if (beg + 32 * g < end[w]) merge_partial(m[w], l[w], o[w], d[HD], d[HD + 1], co);
        }
        store(w);
    }
}

template <typename T, int HD, bool VEC, int BS_PW>
__global__ void __launch_bounds__(128 * bulk_groups<T, HD>()) k_attn_bulk_simt(AttnArgs a, int n_split_launch) {
    attn_bulk_simt<T, HD, VEC, BS_PW, bulk_groups<T, HD>()>(a, n_split_launch);
}
// (Blocks per SM: as many as shared memory holds with fp32 heads of 64 and 128.  Heads of 32 and 64 with 6 to 8 blocks: spills and less
// in flight, 1.2 to 1.6 times as long; with 3, 1.1 to 1.4.)
template <typename T, int HD, bool VEC>
__global__ void __launch_bounds__(128, sizeof(T) * HD > 256 ? 3 : 5) k_attn_bulk_simt_serial(AttnArgs a, int n_split_launch) {
    attn_bulk_simt<T, HD, VEC, 4, 1>(a, n_split_launch);
}

// Tail + merge: one warp per (row, head).  grid = (ceil(rows/4), Hq, batch).
// behind_bulk: launched as a dependent of the bulk kernel, whose CTAs release this one after their own wait; the tail is
// computed while they run (what the step wrote from L2 only: nothing of it comes from a stale L1 line).
template <typename T, int HD, bool VEC, bool L1>
__global__ void __launch_bounds__(128) k_attn_tail_merge(AttnArgs a, bool behind_bulk) {
    // let the next kernel start its own preamble (for a GEMM: the first weight tiles) while this one runs; it still
    // waits for this kernel to complete before it touches anything this kernel or its predecessors write
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * 4 + warp, head = blockIdx.y, seq = blockIdx.z;
    int n_rows, L, depth;
    unsigned long long lo, hi;
    attn_row_info(a, seq, r < RT ? r : 0, n_rows, L, depth, lo, hi);      // (written by an earlier step)
    if (!behind_bulk || r >= n_rows) pdl_wait();
    if (r >= n_rows) return;
    const int P = L + depth;
    const int T0 = tail_start(P, a.dcap);
    const int kvh = head / (a.Hq / a.Hkv);
    float q[HD / 8];
    load_row<T, HD / 8, false>(q, reinterpret_cast<const T*>(a.q) + ((size_t)(seq * RT + r) * a.Hq + head) * HD + (lane & 7) * (HD / 8));
    const T* kb = reinterpret_cast<const T*>(a.kc) + ((size_t)seq * a.Hkv + kvh) * a.cap * HD;
    const T* vb = reinterpret_cast<const T*>(a.vc) + ((size_t)seq * a.Hkv + kvh) * a.cap * HD;
    const int n_l1 = a.cache_in_flight ? 0 : L;      // cache positions below L were written by earlier steps
    // tail: positions T0..P in order
    const int n_tail = P - T0 + 1;
    float tm = -INFINITY, tl = 0.f, to[HD / 32];
#pragma unroll
    for (int i = 0; i < HD / 32; ++i) to[i] = 0.f;
#pragma unroll 1
    for (int t0 = 0; t0 < n_tail; t0 += 32) {
        int slot = -1;
        if (t0 + lane < n_tail) {
            const int pos = T0 + t0 + lane;
            if (pos < L) slot = pos;
            else {
                const int b = nth_set_bit(lo, hi, pos - L);
                if (b < 0) set_error(a.err, DEV_E_INDEX);
                else slot = L + b;
            }
        }
        const uint32_t valid = __ballot_sync(0xffffffffu, slot >= 0);
        const int any = valid ? __shfl_sync(0xffffffffu, slot, __ffs(valid) - 1) : 0;
        if (slot < 0) slot = any;
        float cm, cl, co[HD / 32];
        warp_chunk<T, HD, VEC, L1>(q, kb, vb, slot, n_l1, valid, a.scale_log2, cm, cl, co);
        merge_partial(tm, tl, to, cm, cl, co);
    }
    if (behind_bulk) pdl_wait();
    // bulk partials in split order, MB in flight, then the tail
    constexpr int MB = 4;
    float m = -INFINITY, l = 0.f, o[HD / 32];
#pragma unroll
    for (int i = 0; i < HD / 32; ++i) o[i] = 0.f;
    const int n_sp = (T0 + a.split_len - 1) / a.split_len;
    const size_t base = ((size_t)(seq * RT + r) * a.Hq + head) * a.n_split_max;
    for (int s0 = 0; s0 < n_sp; s0 += MB) {
        float2 ml[MB];
        float co[MB][HD / 32];
#pragma unroll
        for (int u = 0; u < MB; ++u)
            if (s0 + u < n_sp) {
                ml[u] = __ldcg(a.part_ml + base + s0 + u);
#pragma unroll
                for (int i = 0; i < HD / 32; ++i) co[u][i] = __ldcg(a.part_o + (base + s0 + u) * HD + lane + 32 * i);
            }
#pragma unroll
        for (int u = 0; u < MB; ++u)
            if (s0 + u < n_sp) merge_partial(m, l, o, ml[u].x, ml[u].y, co[u]);
    }
    merge_partial(m, l, o, tm, tl, to);
    T* out = reinterpret_cast<T*>(a.out) + ((size_t)(seq * RT + r) * a.Hq + head) * HD;
    const float inv = 1.0f / l;
#pragma unroll
    for (int i = 0; i < HD / 32; ++i) out[lane + 32 * i] = from_f32<T>(o[i] * inv);
    if constexpr (sizeof(T) == 2) {
        if (a.out_lo) {      // low-order plane for an O projection that reads the output as hi + lo
            T* out_lo = reinterpret_cast<T*>(a.out_lo) + ((size_t)(seq * RT + r) * a.Hq + head) * HD;
#pragma unroll
            for (int i = 0; i < HD / 32; ++i) {
                T hi, lo2;
                split_bf16(o[i] * inv, hi, lo2);
                out_lo[lane + 32 * i] = lo2;
            }
        }
    }
}

template <typename T, int HD, bool VEC>
static int launch_attn_simt_t(const AttnArgs& a, int batch, int n_split_launch, cudaStream_t s, bool pdl) {
    const bool behind_bulk = n_split_launch > 0;
    if (behind_bulk) {
        const int pairs = a.rows_cap * (a.Hq / a.Hkv);
        const long long ctas4 = (long long)((pairs + 15) / 16) * a.Hkv * n_split_launch * batch;
        // One pair per warp while its CTAs, four times as many, find room at once (one per SM with fp32 heads of 64 and 128, two
        // otherwise); four pairs with a group of warps per group of chunks up to one and a half CTAs per SM; then one group of warps.
        // Operator with its tail kernel, 32/8 or 4/2 heads, us, one pair / four / four with one group of warps, at CTAs of four pairs:
        // fp32, heads of 32: 20 13.7 / 16.8 / 22, 72 14.1 / 16.9 / 23, 144 20.8 / 17.9 / 23, 288 50 / 47 / 41, 544 52 / 54 / 35, 4096 1107 / 1045 /
        // 684 (656 with one chain per split); of 64: 32 14.0 / 18.7 / 25, 48 20.8 / 20.1 / 25, 72 20.9 / 18.7 / 25, 192 66 / 51.5 / 52.5, 272 50 / 31 /
        // 28, 544 112 / 62 / 49, 4096 2522 / 1229 / 990; of 128: 36 20.8 / 26.9 / 31, 48 34 / 28.8 / 32, 144 64 / 29 / 33, 288 223 / 88 / 93, 352 1051 /
        // 459 / 389, 4096 5813 / 2174 / 1716.  bf16, heads of 32: 72 12.7 / 16.7 / 21, 144 20.7 / 17.7 / 21, 544 55 / 39 / 35, 4096 1071 / 709 / 654;
        // of 64: 72 16.5 / 18.1 / 24, 144 24.9 / 18.8 / 25, 288 70 / 55.6 / 51, 4096 1637 / 1087 / 930.
#define ESP_BULK_SIMT(KERNEL, PW, KS)                                                                                  \
        {                                                                                                              \
            const auto kernel = KERNEL;                                                                                \
            if (ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), (int)bulk_simt_smem<T, HD>(PW, KS))) return -1; \
            launch_k(kernel, dim3((pairs + 4 * PW - 1) / (4 * PW), a.Hkv, n_split_launch * batch), dim3(128 * KS), bulk_simt_smem<T, HD>(PW, KS), s, pdl, a, n_split_launch); \
        }
        constexpr int KG = bulk_groups<T, HD>(), one_pair = sizeof(T) * HD >= 256 ? 37 : 74;
        if (ctas4 < one_pair) ESP_BULK_SIMT((k_attn_bulk_simt<T, HD, VEC, 1>), 1, KG)
        else if (ctas4 <= 222) ESP_BULK_SIMT((k_attn_bulk_simt<T, HD, VEC, 4>), 4, KG)
        else ESP_BULK_SIMT((k_attn_bulk_simt_serial<T, HD, VEC>), 4, 1)
#undef ESP_BULK_SIMT
    }
    const dim3 g2((a.rows_cap + 3) / 4, a.Hq, batch);
    // Through L1 from 4000 (row, head) pairs on: telling the two kinds of slots apart costs every load, which is what counts in a small
    // launch.  Tail alone, fp32, 32 heads, us, L2 / L1: heads of 128, 35 rows 16.9 / 17.2, 4 x 44 39.6 / 36.8, 4 x 128 88 / 77; of 64 12.9 / 13.8,
    // 20.8 / 20.8, 50 / 39; of 32 13.0 / 13.5, 16.6 / 14.8, 32 / 28.  A step of the tiny decoder (35 rows x 4 heads) 106 / 111.
    if ((long long)a.rows_cap * a.Hq * batch >= 4000) launch_k(k_attn_tail_merge<T, HD, VEC, true>, g2, dim3(128), 0, s, pdl || behind_bulk, a, behind_bulk);
    else launch_k(k_attn_tail_merge<T, HD, VEC, false>, g2, dim3(128), 0, s, pdl || behind_bulk, a, behind_bulk);
    return 0;
}

int launch_attn_simt(int dtype, const AttnArgs& a, int batch, int n_split_launch, cudaStream_t s, bool pdl) {
    // 16-byte loads where the caches start on 16 bytes (their rows then do too)
    const bool vec = (reinterpret_cast<uintptr_t>(a.kc) | reinterpret_cast<uintptr_t>(a.vc)) % 16 == 0;
#define ESP_ATTN_CASE(TT, H)                                                              \
    return vec ? launch_attn_simt_t<TT, H, true>(a, batch, n_split_launch, s, pdl) \
               : launch_attn_simt_t<TT, H, false>(a, batch, n_split_launch, s, pdl);
    if (dtype == 0) {
        if (a.h == 32) { ESP_ATTN_CASE(float, 32) }
        if (a.h == 64) { ESP_ATTN_CASE(float, 64) }
        if (a.h == 128) { ESP_ATTN_CASE(float, 128) }
    } else {
        if (a.h == 32) { ESP_ATTN_CASE(__nv_bfloat16, 32) }
        if (a.h == 64) { ESP_ATTN_CASE(__nv_bfloat16, 64) }
        if (a.h == 128) { ESP_ATTN_CASE(__nv_bfloat16, 128) }
    }
#undef ESP_ATTN_CASE
    return -1;
}

// ------------------------------------------------------------------ ranking by packed keys
// keys of the n given ones that are smaller
__device__ __forceinline__ int rank_among(const unsigned long long* keys, int n, unsigned long long key) {
    int rank = 0;
#pragma unroll 4
    for (int o = 0; o + 1 < n; o += 2) {
        const ulonglong2 k2 = *reinterpret_cast<const ulonglong2*>(keys + o);
        rank += (k2.x < key ? 1 : 0) + (k2.y < key ? 1 : 0);
    }
    if (n & 1) rank += keys[n - 1] < key ? 1 : 0;
    return rank;
}
// A Top-K' entry as a key: by value descending, then id ascending, smaller first (-0 and +0 are equal); none: behind all.
__device__ __forceinline__ unsigned long long cand_key(float val, int id) {
    return id < 0 ? ~0ull : ((unsigned long long)(~float_order_key(val)) << 32) | (uint32_t)id;
}
__device__ __forceinline__ Cand cand_of(unsigned long long key) {
    Cand c;
    c.id = key == ~0ull ? -1 : (int)(uint32_t)key;
    c.val = key == ~0ull ? -INFINITY : float_from_order_key(~(uint32_t)(key >> 32));
    return c;
}

// ------------------------------------------------------------------ Top-K' merge over vocabulary tiles
// One block per row: global Top-K' (value desc, id asc) of the per-tile lists, plus
// lse = max + log(sum exp) merged over tiles in a fixed order.
// What bounds it is the number of dependent trips to L2, so there are two: the heads of all tiles' lists (with the tiles'
// (max, sum) pairs), then the whole lists of the K' tiles with the best heads -- an entry of any other tile has K' heads
// before it.  A vocabulary of 1002 tiles, K' = 11, 4 probe rows of 68: 25 us with all lists of a row staged in
// shared memory and K' rounds over them, 17 with these two trips, 12.7 with the entries ranked as packed keys.
constexpr int TOPK_THREADS = 256, TOPK_WARPS = TOPK_THREADS / 32;
constexpr int TOPK_MAXT = 8;   // tiles per thread (n_tiles <= 2048)
__global__ void __launch_bounds__(TOPK_THREADS) k_topk_merge(const SeqState* states, const Cand* cand, const float2* cand_ms,
                                                             int n_tiles, int KP, int batch, Cand* topk, float* lse,
                                                             uint32_t* cand_floor) {
    __shared__ float s_v[TOPK_THREADS];
    __shared__ int s_i[TOPK_THREADS];
    __shared__ __align__(16) unsigned long long s_w[TOPK_WARPS * KP_MAX];      // the best heads of each warp's tiles
    __shared__ int s_wt[TOPK_WARPS * KP_MAX], s_tile[KP_MAX];                  // their tiles; the best of all
    __shared__ __align__(16) unsigned long long s_l[KP_MAX * (KP_MAX + 1) / 2];   // what is read of the best tiles' lists
    if (threadIdx.x == 0) pdl_launch_dependents();
    const int seq = blockIdx.y, r = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const SeqState* st = states + seq;
    const bool idle = !st->active || r >= st->n_rows, probe = r >= st->n_nodes;     // written by an earlier step
    pdl_wait();
    if (idle) return;
    const int Mtot = batch * RT, grow = seq * RT + r;
    const int kp = probe ? KP : 1;
    // tile t belongs to thread t mod 256
    unsigned long long head[TOPK_MAXT];
    float2 ms[TOPK_MAXT];
    {
        Cand c[TOPK_MAXT];
#pragma unroll
        for (int i = 0; i < TOPK_MAXT; ++i) {
            const int t = tid + TOPK_THREADS * i;
            c[i].val = -INFINITY; c[i].id = -1;
            ms[i] = make_float2(-INFINITY, 0.f);
            if (t < n_tiles) {
                c[i] = cand[((size_t)t * Mtot + grow) * KP];
                if (probe) ms[i] = cand_ms[(size_t)t * Mtot + grow];
            }
        }
#pragma unroll
        for (int i = 0; i < TOPK_MAXT; ++i) head[i] = cand_key(c[i].val, c[i].id);
    }
    if (tid < KP_MAX) s_tile[tid] = -1;
    // each warp's kp best heads, in order: a round is the lane-local best, then two warp-wide integer reductions (the high words,
    // then the low words -- ids -- of those that share the smallest); no block barrier
    for (int j = 0; j < kp; ++j) {
        unsigned long long best = head[0];
        int bt = 0;
#pragma unroll
        for (int i = 1; i < TOPK_MAXT; ++i)
            if (head[i] < best) { best = head[i]; bt = i; }
        const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(best >> 32));
        const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)(best >> 32) == hi ? (uint32_t)best : 0xffffffffu);
        const unsigned long long all = ((unsigned long long)hi << 32) | lo;
        if (all == ~0ull) {          // (no more entries)
            if (lane == 0) s_w[warp * kp + j] = ~0ull;
        } else if (best == all) {    // token ids are unique across tiles: one owner
#pragma unroll
            for (int i = 0; i < TOPK_MAXT; ++i) if (i == bt) head[i] = ~0ull;
            s_w[warp * kp + j] = best;
            s_wt[warp * kp + j] = tid + TOPK_THREADS * bt;
        }
    }
    __syncthreads();
    // the kp best of the warps' heads, by rank (ids are unique)
    if (tid < TOPK_WARPS * kp && s_w[tid] != ~0ull) {
        const int rank = rank_among(s_w, TOPK_WARPS * kp, s_w[tid]);
        if (rank < kp) {
            s_tile[rank] = s_wt[tid];
            if (!probe) topk[(size_t)grow * KP_MAX] = cand_of(s_w[tid]);
        }
    }
    __syncthreads();
    if (!probe) {
        if (tid == 0 && s_tile[0] < 0) topk[(size_t)grow * KP_MAX] = cand_of(~0ull);
        return;
    }
    // Their lists: entry q of the tile with the p-th best head has p heads and q entries of its own before it, so only
    // p + q < kp matter.  The kp best of these by rank.
    for (int i = tid; i < kp * kp; i += TOPK_THREADS) {
        const int p = i / kp, q = i % kp;
        if (p + q < kp) {
            Cand c = cand_of(~0ull);
            if (s_tile[p] >= 0) c = cand[((size_t)s_tile[p] * Mtot + grow) * KP + q];
            s_l[p * kp - p * (p - 1) / 2 + q] = cand_key(c.val, c.id);
        }
    }
    if (tid < kp) topk[(size_t)grow * KP_MAX + tid] = cand_of(~0ull);     // (if there are fewer)
    // thread-strided partial merges in tile order, then a fixed tree over threads
    float m = -INFINITY, sm = 0.f;
#pragma unroll
    for (int i = 0; i < TOPK_MAXT; ++i) {
        if (tid + TOPK_THREADS * i < n_tiles) {
            const float mn = fmaxf(m, ms[i].x);
            sm = sm * expf(m - mn) + ms[i].y * expf(ms[i].x - mn);
            m = mn;
        }
    }
    float* s_s = reinterpret_cast<float*>(s_i);
    s_v[tid] = m;
    s_s[tid] = sm;
    __syncthreads();
    const int n_l = kp * (kp + 1) / 2;
    for (int i = tid; i < n_l; i += TOPK_THREADS) {
        if (s_l[i] == ~0ull) continue;
        const int rank = rank_among(s_l, n_l, s_l[i]);
        if (rank < kp) topk[(size_t)grow * KP_MAX + rank] = cand_of(s_l[i]);
    }
    for (int o = TOPK_THREADS / 2; o > 0; o >>= 1) {
        if (tid < o) {
            const float m1 = s_v[tid], m2 = s_v[tid + o];
            const float s1 = s_s[tid], s2 = s_s[tid + o];
            const float mn = fmaxf(m1, m2);
            const float sn = (m1 == -INFINITY ? 0.f : s1 * expf(m1 - mn)) + (m2 == -INFINITY ? 0.f : s2 * expf(m2 - mn));
            s_v[tid] = mn;
            s_s[tid] = sn;
        }
        __syncthreads();
    }
    if (tid == 0) lse[grow] = s_v[0] + logf(s_s[0]);
    if (tid < KP_MAX && cand_floor) cand_floor[(size_t)grow * KP_MAX + tid] = 0;     // nothing is known about the next forward's logits
}

void launch_topk_merge(const SeqState* st, const Cand* cand, const float2* cand_ms, int n_tiles, int KP, int batch,
                       Cand* topk, float* lse, cudaStream_t s, bool pdl, int rows_cap, uint32_t* cand_floor) {
    launch_k(k_topk_merge, dim3(rows_cap, batch), dim3(TOPK_THREADS), 0, s, pdl, st, cand, cand_ms, n_tiles, KP, batch, topk, lse, cand_floor);
}

// ------------------------------------------------------------------ sampling noise, stand-alone (for checking)
__global__ void k_gumbel_noise(uint32_t key0, uint32_t key1, uint32_t position, int n, float* out) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) out[v] = gumbel_noise(key0, key1, position, (uint32_t)v);
}
void launch_gumbel_noise(uint32_t key0, uint32_t key1, uint32_t position, int n, float* out, cudaStream_t s) {
    k_gumbel_noise<<<(n + 255) / 256, 256, 0, s>>>(key0, key1, position, n, out);
}

// ------------------------------------------------------------------ row-table builders
// (depth, anc: those of the tree's rows; threads tid, tid + n_threads, .. take part)
__device__ void write_probe_rows(SeqState* st, int N, int k, int first_anchor, int n_anchor_rows, const int* depth,
                                 const unsigned long long (*anc)[2], int tid, int n_threads) {
    // probe j (1-based) of the a-th anchored node sits at row N + a*k + (j-1)
    for (int i = tid; i < n_anchor_rows * k; i += n_threads) {
        int aidx = i / k, j = i % k + 1;
        int u = first_anchor + aidx;
        int row = N + aidx * k + (j - 1);
        st->row_token[row] = -1;
        st->row_parent[row] = j == 1 ? u : row - 1;
        st->row_depth[row] = depth[u] + j;
        unsigned long long lo = anc[u][0], hi = anc[u][1];
        for (int jj = 0; jj < j; ++jj) {
            int b = N + aidx * k + jj;
            if (b < 64) lo |= 1ull << b; else hi |= 1ull << (b - 64);
        }
        st->row_anc[row][0] = lo;
        st->row_anc[row][1] = hi;
        st->row_logp[row] = 0.f;
    }
}

// rows = n consecutive prompt tokens (a chain)
__device__ void write_chain_rows(SeqState* st, const int32_t* prompt_dev, int off, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        st->row_token[i] = prompt_dev[off + i];
        st->row_parent[i] = i - 1;
        st->row_depth[i] = i;
        unsigned long long lo = i >= 63 ? ~0ull : ((1ull << (i + 1)) - 1);
        unsigned long long hi = i < 64 ? 0ull : ((1ull << (i - 63)) - 1);
        st->row_anc[i][0] = lo;
        st->row_anc[i][1] = hi;
        st->row_logp[i] = 0.f;
    }
}

// Several full prefill blocks, a state each (block b of the grid: prompt tokens off + b * PREFILL_CHUNK ..).
__global__ void k_setup_chains(SeqState* states, const int32_t* prompt_dev, int off) {
    SeqState* st = states + blockIdx.x;
    const int o = off + blockIdx.x * PREFILL_CHUNK;
    write_chain_rows(st, prompt_dev, o, PREFILL_CHUNK);
    if (threadIdx.x == 0) {
        st->L = o;
        st->n_nodes = st->n_rows = PREFILL_CHUNK;
        st->mode = 1;
        st->active = 1;
    }
}

// Prefill chunk; the last chunk appends k probes behind the last prompt token (Figure 1 middle).
__global__ void k_setup_chain(SeqState* states, int seq, const int32_t* prompt_dev, int off, int n, int last, int k) {
    SeqState* st = states + seq;
    write_chain_rows(st, prompt_dev, off, n);
    __syncthreads();
    if (last && k > 0) write_probe_rows(st, n, k, n - 1, 1, st->row_depth, st->row_anc, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) {
        st->n_nodes = n;
        st->n_rows = n + (last ? k : 0);
        st->mode = last ? 2 : 1;
        st->active = 1;
        st->L = off;
    }
}

// Caller-provided tree (test hook): tokens/parents in breadth-first order.
__global__ void k_set_tree(SeqState* states, int seq, const int32_t* tokens, const int32_t* parents, int n, int k,
                           int n_anchor, int* err) {
    SeqState* st = states + seq;
    if (threadIdx.x == 0) {
        for (int i = 0; i < n; ++i) {
            int p = parents[i];
            if (i == 0 ? p != -1 : (p < 0 || p >= i)) { set_error(err, DEV_E_INDEX); p = i == 0 ? -1 : 0; }
            st->row_token[i] = tokens[i];
            st->row_parent[i] = p;
            st->row_depth[i] = i == 0 ? 0 : st->row_depth[p] + 1;
            unsigned long long lo = i == 0 ? 0 : st->row_anc[p][0], hi = i == 0 ? 0 : st->row_anc[p][1];
            if (i < 64) lo |= 1ull << i; else hi |= 1ull << (i - 64);
            st->row_anc[i][0] = lo;
            st->row_anc[i][1] = hi;
            st->row_logp[i] = 0.f;
        }
        st->n_nodes = n;
    }
    __syncthreads();
    int nA = k > 0 ? (n_anchor == 0 ? n : min(n_anchor, n)) : 0;
    write_probe_rows(st, n, k, 0, nA, st->row_depth, st->row_anc, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) { st->n_rows = n + nA * k; st->mode = 0; st->forced = 1; }
}

// ------------------------------------------------------------------ the single-block tree kernel
// verify walk -> KV compaction -> mask update -> Algorithm 1 + pruner -> next row table.

// Total order of created nodes as one integer: (logP descending, depth ascending, creation index ascending);
// a smaller key comes first.  -0.0 and +0.0 compare equal as floats, so both map to the key of +0.0.
__device__ __forceinline__ unsigned long long node_key(float lp, int depth, int idx) {
    unsigned u = __float_as_uint(lp == 0.f ? 0.f : lp);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);   // monotone: larger float -> larger u
    return ((unsigned long long)(~u) << 32) | ((unsigned long long)depth << 16) | (unsigned long long)idx;
}

// What bounds it is one block's chain of short phases: every barrier, every dependent trip to L2 and every loop of dependent
// shared-memory loads counts.  So the first half of the block does what the next forward pass's rows hang on -- verification,
// lists, tree, row table -- and the other half compacts the cache and updates the masks meanwhile; keys are ranked from
// packed arrays, breadth-first places come from bit masks, and counters and the error word are fetched ahead of their use.
// 64 nodes, K = 10, four probes: 48 -> 32 us with the packed ranking, 26 with the halves (step of eight 8B layers
// 1278 -> 1255 us).  16 nodes, K = 5, three probes: 8.4 us (a request of 32 small steps 5209 -> 4680 us).
constexpr int TREE_THREADS = 1024, TREE_BUILD = 512;      // threads; those of them that build the tree
__device__ __forceinline__ void tree_bar() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
__device__ __forceinline__ bool tree_bar_or(bool x) {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 512, p;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"((uint32_t)x) : "memory");
    return r != 0;
}
template <typename T>
__global__ void __launch_bounds__(TREE_THREADS) k_tree_step(TreeArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long* c_sort = reinterpret_cast<unsigned long long*>(smem_raw);      // [MAX_CAND] keys that are ranked
    int* c_tok = reinterpret_cast<int*>(c_sort + MAX_CAND);
    int* c_par = c_tok + MAX_CAND;
    int* c_dep = c_par + MAX_CAND;
    float* c_lp = reinterpret_cast<float*>(c_dep + MAX_CAND);
    int* c_row = reinterpret_cast<int*>(c_lp + MAX_CAND);            // creation index -> new row
    __shared__ int s_path[PROBES_MAX + 2], s_out[PROBES_MAX + 2];
    __shared__ int s_na, s_ustar, s_delta, s_nexp, s_ncreated, s_nkeep, s_nsurv, s_err;
    __shared__ int s_exp[RT], s_sel[RT];
    __shared__ int s_rtok[RT], s_rpar[RT], s_rdep[RT], s_arg[RT];     // this step's row table and per-row argmax
    __shared__ __align__(16) unsigned long long s_keep[PROBES_MAX * RT];      // per depth, the keys of the B-1 best nodes: the only ones the final pick can take
    __shared__ unsigned long long s_anc[RT][2];                       // the next tree's ancestor masks
    __shared__ uint32_t s_dmask[PROBES_MAX + 1][RT / 32];             // by depth: which selection ranks stand there
    __shared__ Cand s_list[PROBES_MAX][KP_MAX];                       // Top-K' lists of the probes the next tree uses
    __shared__ float s_lse[PROBES_MAX];

    // Before the wait: the sequence's state and row table, which only this kernel and the set-up of a prefill block (plain
    // launches) write.
    const Dims& D = A.D;
    const int seq = blockIdx.x, tid = threadIdx.x, nt = TREE_THREADS, lane = tid & 31;
    SeqState* st = A.states + seq;
    // where this launch's record goes; every sequence, active or not, counts the handle's decode steps
    const unsigned long long rec_no = st->rec;
    int32_t* rec = A.out_ring + ((size_t)(A.is_step ? (int)(rec_no % NREC) : NREC) * D.batch + seq) * RING;
    const int active = st->active, mode = st->mode, N0 = st->n_nodes, L0 = st->L, rows0 = st->n_rows;
    for (int r = tid; r < N0 && r < RT; r += nt) {
        s_rtok[r] = st->row_token[r];
        s_rpar[r] = st->row_parent[r];
        s_rdep[r] = st->row_depth[r];
    }
    if (tid == 0) { s_err = 0; s_nsurv = 0; }
    pdl_wait();
    const int err0 = tid == 0 ? __ldcg(A.err) : 0;       // the error word before this kernel
    __syncthreads();      // every thread has read the counter
    if (A.is_step && tid == 0) st->rec = rec_no + 1;
    if (!active) {
        if (tid == 0) { rec[0] = 0; rec[RING - 1] = err0; }
        return;
    }
    const int grow0 = seq * RT;

    if (mode == 1) {  // prefill chunk: every row is a prompt token and is already in place
        if (tid == 0) st->L = L0 + N0;
        return;
    }
    auto fail = [&](int code) { set_error(A.err, code); atomicCAS(&s_err, 0, code); };
    for (int r = tid; r < N0; r += nt) {
        const int t = A.topk[(size_t)(grow0 + r) * KP_MAX].id;
        s_arg[r] = t >= 0 ? t : 0;                       // a row of NaN has no arg-max: its token would index the embeddings
        if (t < 0) fail(DEV_E_INDEX);
    }
    __syncthreads();

    // ---- verification (Section 2): follow the model's own next token through the tree.  One warp walks; its lanes look for
    // the child (one thread looking through the rows took 5000 cycles for a 32-node tree).
    if (tid < 32) {
        int a = 0, cur, n_emit = 0;
        if (mode == 2) {
            cur = N0 - 1;  // last prompt token; nothing to verify, its argmax is the first generated token
            if (tid == 0) { s_path[0] = cur; s_out[0] = s_arg[cur]; s_ustar = cur; s_delta = 0; }
            n_emit = 1;
        } else {
            cur = 0;
            if (tid == 0) s_path[0] = 0;
            for (;;) {
                const int y = s_arg[cur];
                if (tid == 0) s_out[n_emit] = y;
                ++n_emit;
                unsigned nxt = 0xffffffffu;               // the first row below cur with parent cur and token y
                for (int c = cur + 1 + tid; c < N0; c += 32)
                    if (s_rpar[c] == cur && s_rtok[c] == y) { nxt = (unsigned)c; break; }
                nxt = __reduce_min_sync(0xffffffffu, nxt);
                if (nxt == 0xffffffffu || n_emit > PROBES_MAX) break;
                cur = (int)nxt;
                ++a;
                if (tid == 0) s_path[a] = cur;
            }
        }
        __syncwarp();
        if (tid == 0) {
            if (mode != 2) {
                // deepest anchored node on the accepted path
                int nA = D.k > 0 ? (D.n_anchor == 0 ? N0 : min(D.n_anchor, N0)) : 0;
                int us = 0;
                for (int q = 0; q <= a; ++q) if (s_path[q] < nA) us = s_path[q];
                s_ustar = us;
                s_delta = a - s_rdep[us];
            }
            s_na = a;
        }
    }
    __syncthreads();
    const int a_acc = s_na;
    const int n_emit = mode == 2 ? 1 : a_acc + 1;
    const int Lnew = mode == 2 ? L0 + N0 : L0 + a_acc + 1;

    if (tid >= TREE_BUILD) {
        // ================ the other half: record, counters, KV compaction, masks
        const int ht = tid - TREE_BUILD, hn = TREE_THREADS - TREE_BUILD;
        if (ht == 0) {
            st->n_out = n_emit;
            for (int q = 0; q < n_emit; ++q) st->out_tokens[q] = s_out[q];
            rec[0] = n_emit;
            rec[1] = Lnew;
            for (int q = 0; q < n_emit; ++q) rec[2 + q] = s_out[q];
            if (mode == 0) {
                st->rows_hist[rows0 <= 16 ? 0 : (rows0 <= 32 ? 1 : (rows0 <= 64 ? 2 : 3))] += 1;
                st->steps += 1;
                st->emitted += n_emit;
                st->accept_hist[a_acc < PROBES_MAX ? a_acc : PROBES_MAX] += 1;
            }
        }
        // ---- KV compaction: cache slot L+j <- row p_j for the accepted path (row 0 is already at slot L).  A thread moves the
        // same 16 bytes of every row, all read before the first is written: sources sit at or above their destination, and
        // nothing a thread reads is written by another.
        if (mode == 0 && a_acc > 0) {
            const int vec_per_row = D.h * (int)sizeof(T) / 16;
            const size_t layer_stride = (size_t)D.batch * D.Hkv * D.cap * D.h;
            const int per_j = D.n_layers * D.Hkv * 2 * vec_per_row;
            for (int i = ht; i < per_j; i += hn) {
                const int v = i % vec_per_row;
                int rest = i / vec_per_row;
                const int kv = rest & 1;
                rest >>= 1;
                const int hh = rest % D.Hkv, l = rest / D.Hkv;
                T* basep = reinterpret_cast<T*>(kv ? A.vcache : A.kcache) + (size_t)l * layer_stride + ((size_t)seq * D.Hkv + hh) * D.cap * D.h;
                uint4 x[PROBES_MAX];
#pragma unroll
                for (int j = 1; j <= PROBES_MAX; ++j)
                    if (j <= a_acc) x[j - 1] = reinterpret_cast<const uint4*>(basep + (size_t)(L0 + s_path[j]) * D.h)[v];
#pragma unroll
                for (int j = 1; j <= PROBES_MAX; ++j)
                    if (j <= a_acc && s_path[j] != j) reinterpret_cast<uint4*>(basep + (size_t)(L0 + j) * D.h)[v] = x[j - 1];
            }
        }
        // ---- mask update, Eq. (mask_update_mean): m <- m + lambda (e - m)
        const T* E = reinterpret_cast<const T*>(A.embed);
        float* m = A.mvec + (size_t)seq * D.mask_slots * D.d;
        // four consecutive elements per thread; every load of a pass is issued before the first store
        const int e0 = D.ema_per_token ? 0 : n_emit - 1;
        for (int j = ht * 4; j < D.d; j += hn * 4) {
            float ev[PROBES_MAX + 2][4];
            float4 mv[PROBES_MAX];
            for (int e = e0; e < n_emit; ++e)
#pragma unroll
                for (int i = 0; i < 4; ++i) ev[e][i] = j + i < D.d ? to_f32(E[(size_t)s_out[e] * D.d + j + i]) : 0.f;
            const bool vec = j + 4 <= D.d;
#pragma unroll
            for (int slot = 0; slot < PROBES_MAX; ++slot) {
                if (slot < D.mask_slots) {
                    float* ms = m + (size_t)slot * D.d + j;
                    mv[slot] = vec ? *reinterpret_cast<const float4*>(ms)
                                   : make_float4(ms[0], j + 1 < D.d ? ms[1] : 0.f, j + 2 < D.d ? ms[2] : 0.f, 0.f);
                }
            }
#pragma unroll
            for (int slot = 0; slot < PROBES_MAX; ++slot) {      // every mask vector follows the same update
                if (slot < D.mask_slots) {
                    float x[4] = {mv[slot].x, mv[slot].y, mv[slot].z, mv[slot].w};
                    for (int e = e0; e < n_emit; ++e)
#pragma unroll
                        for (int i = 0; i < 4; ++i) x[i] = __fadd_rn(x[i], __fmul_rn(D.lambda, __fsub_rn(ev[e][i], x[i])));
                    float* ms = m + (size_t)slot * D.d + j;
                    if (vec) *reinterpret_cast<float4*>(ms) = make_float4(x[0], x[1], x[2], x[3]);
                    else for (int i = 0; i < 4 && j + i < D.d; ++i) ms[i] = x[i];
                }
            }
        }
        return;
    }

    // ================ the first half: next tree (Algorithm 1 with the pruner).  Depth i draws from probe delta+i of u*.
    const int root_tok = s_out[n_emit - 1];
    const int ustar = s_ustar, delta = s_delta;
    const int Dd = D.k - delta > 0 ? D.k - delta : 0;
    // the probe lists the tree draws from, staged once
    for (int w = tid; w < Dd * KP_MAX; w += TREE_BUILD) {
        const int i = w / KP_MAX + 1, q = w % KP_MAX;
        const int prow = mode == 2 ? N0 + (i - 1) : N0 + ustar * D.k + (delta + i - 1);
        s_list[i - 1][q] = A.topk[(size_t)(grow0 + prow) * KP_MAX + q];
        if (q == 0) s_lse[i - 1] = A.lse[grow0 + prow];
    }
    if (tid == 0) {
        c_tok[0] = root_tok; c_par[0] = -1; c_dep[0] = 0; c_lp[0] = 0.f; c_row[0] = 0;
        s_exp[0] = 0; s_nexp = 1; s_ncreated = 1; s_nkeep = 0;
    }
    for (int r = tid; r < RT; r += TREE_BUILD) s_sel[r] = -1;
    tree_bar();
    for (int i = 1; i <= Dd; ++i) {
        // Algorithm 1 draws min(K, B-i) candidates per expanded node; a static tree its fixed width for this depth
        const int pool = D.static_w[0] > 0 ? D.static_w[i - 1] : min(D.K, D.B - i);
        if (pool <= 0) break;
        const Cand* list = s_list[i - 1];
        const float lse_i = s_lse[i - 1];
        const int base = s_ncreated, n_exp = s_nexp, keep0 = s_nkeep;
        const int n_new = n_exp * pool;
        if (base + n_new > MAX_CAND) { if (tid == 0) fail(DEV_E_TREE_OVERFLOW); break; }
        const int width = D.W == 0 ? D.B - i : min(D.W, D.B - i);
        // Ranks of the new nodes among themselves (same depth: logP desc, creation asc) matter only below
        // R = max(width, B-1).  The expanded nodes stand in the order of their logP and all draw from one sorted list, of which
        // the pruner takes at most two entries for each: child j of the e-th node has the children up to j - 2 of every node
        // before it, and its own j earlier siblings, before it.  Where these are R it need not be ranked.  (Rounding keeps the
        // order and equal values go by creation; a NaN would break it, then every node is ranked.)  64 nodes, K = 10: 313 of
        // 620 nodes at the third depth.
        const int R = min(max(width, D.B - 1), RT);
        const int n_kept = min(min(D.B - 1, RT), n_new);
        // the keys to rank, packed (whole warps run along: the places of a warp's keys come from one addition)
        auto put = [&](bool in, unsigned long long key) {
            const uint32_t who = __ballot_sync(0xffffffffu, in);
            int at = 0;
            if (lane == 0 && who) at = atomicAdd(&s_nsurv, __popc(who));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (in) c_sort[at + __popc(who & ((1u << lane) - 1u))] = key;
        };
        bool saw_nan = false;
        for (int w0 = 0; w0 < n_new; w0 += TREE_BUILD) {
            const int w = w0 + tid;
            bool in = false;
            unsigned long long key = 0;
            if (w < n_new) {
                const int e = w / pool, j = w % pool;
                const int p = s_exp[e];
                const int ptok = c_tok[p];
                int seen = 0, q = D.KP;                  // the j-th entry that the pruner leaves
#pragma unroll 4
                for (int u = 0; u < D.KP; ++u) {
                    const int t = list[u].id;
                    const bool cut = (D.prune_parent && t == ptok) || (D.prune_root && t == root_tok);
                    if (!cut) {
                        if (seen == j) q = min(q, u);
                        ++seen;
                    }
                }
                const int c = base + w;
                float lp = -INFINITY;
                int tok = -1;      // list exhausted (logits of NaN; K' = K + pruner flags otherwise): neither it nor its children selectable
                if (ptok >= 0 && q < D.KP && list[q].id >= 0) {
                    tok = list[q].id;
                    lp = __fadd_rn(c_lp[p], __fsub_rn(list[q].val, lse_i));
                }
                c_tok[c] = tok;
                c_lp[c] = lp;
                c_par[c] = p;
                c_dep[c] = i;
                key = node_key(lp, i, c);
                saw_nan |= isnan(lp);
                in = e * (j - 1) + j < R;
            }
            put(in, key);
        }
        if (tree_bar_or(saw_nan)) {
            if (tid == 0) s_nsurv = 0;
            tree_bar();
            for (int w0 = 0; w0 < n_new; w0 += TREE_BUILD) {
                const int w = w0 + tid;
                put(w < n_new, w < n_new ? node_key(c_lp[base + w], i, base + w) : 0ull);
            }
            tree_bar();
        }
        const int n_surv = s_nsurv;
        for (int w = tid; w < n_surv; w += TREE_BUILD) {
            const unsigned long long key = c_sort[w];
            const int rank = rank_among(c_sort, n_surv, key);
            if (rank < width) s_exp[rank] = (int)(key & 0xffffu);          // (the creation index)
            // a node with B-1 or more nodes of its own depth before it cannot be among the B-1 best overall
            if (rank < n_kept) s_keep[keep0 + rank] = key;
        }
        if (tid == 0) { s_ncreated = base + n_new; s_nexp = min(width, n_new); s_nkeep = keep0 + n_kept; }
        tree_bar();
        if (tid == 0) s_nsurv = 0;      // (the next depth adds to it behind its own first barrier ...)
        tree_bar();
    }
    tree_bar();
    // final selection: root + the B-1 best created nodes by (logP desc, depth asc, creation asc)
    // (ranked among the kept nodes only: every node that precedes one of the B-1 best is itself kept)
    const int n_keep = s_nkeep;
    for (int w = tid; w < n_keep; w += TREE_BUILD) {
        const unsigned long long key = s_keep[w];
        const int c = (int)(key & 0xffffu), rank = rank_among(s_keep, n_keep, key);
        if (rank < D.B - 1 && c_tok[c] >= 0 && rank < RT) s_sel[rank] = c;
    }
    tree_bar();
    // Breadth-first row order: by depth, ties by selection rank.  (Entries with token -1 rank last because their logP is -inf:
    // what is selected ends with the first empty place.)
    int n_sel = 0, idx = 0;
    const int c_mine = tid < RT ? s_sel[tid] : -1;
    {
        const int most = min(D.B - 1, n_keep);
        bool open = true;
        for (int r0 = 0; r0 < RT && open; r0 += 32) {
            const uint32_t ok = __ballot_sync(0xffffffffu, r0 + lane < most && s_sel[r0 + lane] >= 0);
            n_sel += ok == 0xffffffffu ? 32 : __ffs(~ok) - 1;
            open = ok == 0xffffffffu;
        }
    }
    const int dp = tid < n_sel ? c_dep[c_mine] : 0;
    if (tid < RT)
        for (int d = 1; d <= Dd; ++d) {
            const uint32_t who = __ballot_sync(0xffffffffu, dp == d);
            if (lane == 0) s_dmask[d][tid >> 5] = who;
        }
    tree_bar();
    if (tid < n_sel) {
        idx = 1;
        for (int d = 1; d < dp; ++d)
#pragma unroll
            for (int w = 0; w < RT / 32; ++w) idx += __popc(s_dmask[d][w]);
#pragma unroll
        for (int w = 0; w < RT / 32; ++w)
            if (w < (tid >> 5)) idx += __popc(s_dmask[dp][w]);
        idx += __popc(s_dmask[dp][tid >> 5] & ((1u << lane) - 1u));
        c_row[c_mine] = idx;
    }
    tree_bar();
    const int N = n_sel + 1;
    if (tid < n_sel) {
        // ancestor-or-self mask by walking up the creation-time parents
        unsigned long long lo = 0, hi = 0;
        for (int x = c_mine; x >= 0; x = c_par[x]) {
            const int b = c_row[x];
            if (b < 64) lo |= 1ull << b; else hi |= 1ull << (b - 64);
        }
        st->row_token[idx] = c_tok[c_mine];
        st->row_parent[idx] = c_row[c_par[c_mine]];
        st->row_depth[idx] = dp;
        st->row_logp[idx] = c_lp[c_mine];
        st->row_anc[idx][0] = s_anc[idx][0] = lo;
        st->row_anc[idx][1] = s_anc[idx][1] = hi;
        s_rdep[idx] = dp;
    }
    if (tid == RT) {
        st->row_token[0] = root_tok; st->row_parent[0] = -1; st->row_depth[0] = 0; st->row_logp[0] = 0.f;
        st->row_anc[0][0] = s_anc[0][0] = 1ull; st->row_anc[0][1] = s_anc[0][1] = 0ull;
        s_rdep[0] = 0;
    }
    tree_bar();
    const int nA = D.k > 0 ? (D.n_anchor == 0 ? N : min(D.n_anchor, N)) : 0;
    write_probe_rows(st, N, D.k, 0, nA, s_rdep, s_anc, tid, TREE_BUILD);
    if (tid == 0) {
        st->n_nodes = N;
        st->n_rows = N + nA * D.k;
        st->L = Lnew;
        st->mode = 0;
        st->forced = 0;
        if (Lnew + RT > D.cap) fail(DEV_E_CAPACITY);
        rec[RING - 1] = err0 ? err0 : s_err;       // the error word as this step leaves it
    }
}

void launch_tree_step(int dtype, const TreeArgs& A, cudaStream_t s, bool pdl) {
    size_t smem = (size_t)MAX_CAND * 28;
    if (dtype == 0) {
        ensure_dynamic_smem(reinterpret_cast<const void*>(k_tree_step<float>), (int)smem);
        launch_k(k_tree_step<float>, dim3(A.D.batch), dim3(TREE_THREADS), smem, s, pdl, A);
    } else {
        ensure_dynamic_smem(reinterpret_cast<const void*>(k_tree_step<__nv_bfloat16>), (int)smem);
        launch_k(k_tree_step<__nv_bfloat16>, dim3(A.D.batch), dim3(TREE_THREADS), smem, s, pdl, A);
    }
}

// ------------------------------------------------------------------ thin launch wrappers
void launch_rope_table(float* cs, float* sn, int n_pos, int h, float base, cudaStream_t s) {
    int n = n_pos * (h / 2);
    k_rope_table<<<(n + 255) / 256, 256, 0, s>>>(cs, sn, n_pos, h, base);
}
void launch_mask_init(int dtype, const void* embed, const int32_t* prompt, int t, int d, float* m, int slots, int mode, cudaStream_t s) {
    if (dtype == 0) k_mask_init<float, mask_threads<float>()><<<(d + 31) / 32, mask_threads<float>(), 0, s>>>((const float*)embed, prompt, t, d, m, slots, mode);
    else k_mask_init<__nv_bfloat16, mask_threads<__nv_bfloat16>()><<<(d + 31) / 32, mask_threads<__nv_bfloat16>(), 0, s>>>((const __nv_bfloat16*)embed, prompt, t, d, m, slots, mode);
}
void launch_assemble(int dtype, const SeqState* st, const void* embed, const float* mvec, float* hres, int d, int mask_slots,
                     int batch, cudaStream_t s, bool pdl, int rows_cap) {
    dim3 grid(rows_cap, batch);
    if (dtype == 0) launch_k(k_assemble<float>, grid, dim3(128), 0, s, pdl, st, (const float*)embed, mvec, hres, d, mask_slots);
    else launch_k(k_assemble<__nv_bfloat16>, grid, dim3(128), 0, s, pdl, st, (const __nv_bfloat16*)embed, mvec, hres, d, mask_slots);
}
void launch_rmsnorm(int dtype, const SeqState* st, const float* x, const void* g, void* y, int d, float eps, int batch,
                    float* copy_out, cudaStream_t s, bool pdl, int rows_cap) {
    dim3 grid(rows_cap, batch);
    if (dtype == 0 && d <= NORM_ROWS_D)
        launch_k(k_rmsnorm_rows, dim3((rows_cap + NORM_ROWS_WARPS - 1) / NORM_ROWS_WARPS, batch), dim3(NORM_ROWS_WARPS * 32), 0, s, pdl, st, x,
                 (const float*)g, (float*)y, d, eps, copy_out);
    else if (dtype == 0) launch_k(k_rmsnorm<float>, grid, dim3(256), 0, s, pdl, st, x, (const float*)g, (float*)y, d, eps, copy_out);
    else launch_k(k_rmsnorm<__nv_bfloat16>, grid, dim3(256), 0, s, pdl, st, x, (const __nv_bfloat16*)g, (__nv_bfloat16*)y, d, eps, copy_out);
}
void launch_resid_norm(const SeqState* st, float* hres, const StreamK& sk, const void* g, void* y, void* y_lo, int d, float eps,
                       float* copy_out, int nq, cudaStream_t s, bool pdl, int rows_cap) {
    if ((long long)rows_cap * nq > 2 * 148 && d <= NORM_MANY_D) {
        launch_k(k_resid_norm_many, dim3(rows_cap, nq), dim3(NORM_MANY_WARPS * 32), 0, s, pdl, st, hres, sk, (const __nv_bfloat16*)g,
                 (__nv_bfloat16*)y, (__nv_bfloat16*)y_lo, d, eps, copy_out);
        return;
    }
    if (d > NORM_HALF_D / 2 && d <= NORM_HALF_D && 2 * rows_cap * nq <= 148) {     // a block per SM at most
        launch_k(k_resid_norm_pair, dim3(2 * rows_cap, nq), dim3(NORM_HALF_WARPS * 16), 0, s, pdl, st, hres, sk, (const __nv_bfloat16*)g,
                 (__nv_bfloat16*)y, (__nv_bfloat16*)y_lo, d, eps, copy_out);
        return;
    }
    if (d > NORM_HALF_D / 2 && d <= NORM_HALF_D) {
        launch_k(k_resid_norm_half, dim3(rows_cap, nq), dim3(NORM_HALF_WARPS * 32), 0, s, pdl, st, hres, sk, (const __nv_bfloat16*)g,
                 (__nv_bfloat16*)y, (__nv_bfloat16*)y_lo, d, eps, copy_out);
        return;
    }
    launch_k(k_resid_norm<__nv_bfloat16>, dim3(rows_cap, nq), dim3(1024), 0, s, pdl, st, hres, sk, (const __nv_bfloat16*)g,
             (__nv_bfloat16*)y, (__nv_bfloat16*)y_lo, d, eps, copy_out);
}
void launch_swiglu_finish(const SeqState* st, const StreamK& sk, void* act, void* act_lo, int F, int nq, cudaStream_t s, bool pdl, int rows_cap) {
    // (a tile of a GEMM of fewer tiles than half its CTAs has more than two pieces)
    const int fpt = sk.G > 2 * sk.n_tiles ? 4 : 8;
    const dim3 grid(((F + fpt - 1) / fpt + SWIGLU_THREADS - 1) / SWIGLU_THREADS, rows_cap, nq);
    if (fpt == 4) launch_k(k_swiglu_finish<4, 8>, grid, dim3(SWIGLU_THREADS), 0, s, pdl, st, 0, sk, (__nv_bfloat16*)act, (__nv_bfloat16*)act_lo, F);
    else launch_k(k_swiglu_finish<8, 2>, grid, dim3(SWIGLU_THREADS), 0, s, pdl, st, 0, sk, (__nv_bfloat16*)act, (__nv_bfloat16*)act_lo, F);
}
int launch_qkv_finish(const EpiArgs& a, const StreamK& sk, int nq, cudaStream_t s, bool pdl, int rows_cap) {
    const int n_heads = a.Hq + 2 * a.Hkv;
    dim3 grid((n_heads + 3) / 4, rows_cap, nq);
    if (a.h == 128) launch_k(k_qkv_finish<128>, grid, dim3(128), 0, s, pdl, a, sk);
    else if (a.h == 64) launch_k(k_qkv_finish<64>, grid, dim3(128), 0, s, pdl, a, sk);
    else if (a.h == 32) launch_k(k_qkv_finish<32>, grid, dim3(128), 0, s, pdl, a, sk);
    else return -1;
    return 0;
}
void launch_setup_chain(SeqState* st, int seq, const int32_t* prompt_dev, int off, int n, int last, int k, cudaStream_t s) {
    k_setup_chain<<<1, 128, 0, s>>>(st, seq, prompt_dev, off, n, last, k);
}
void launch_setup_chains(SeqState* st, int n, const int32_t* prompt_dev, int off, cudaStream_t s) {
    k_setup_chains<<<n, 128, 0, s>>>(st, prompt_dev, off);
}
void launch_set_tree(SeqState* st, int seq, const int32_t* tokens, const int32_t* parents, int n, int k, int n_anchor,
                     int* err, cudaStream_t s) {
    k_set_tree<<<1, 128, 0, s>>>(st, seq, tokens, parents, n, k, n_anchor, err);
}

}  // namespace esp
