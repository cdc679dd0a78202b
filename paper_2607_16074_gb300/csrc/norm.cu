// HBM-bound kernels of the backbone: the packer (gather into the canonical
// packed batch), RMSNorm, the final RMSNorm fused with the per-sample mean
// pool, and the RoPE (cos, sin) table.
#include <cooperative_groups.h>

#include <climits>
#include <cmath>

#include "jnx_dev.cuh"
#include "jnx_kernels.h"

namespace cg = cooperative_groups;

namespace jnx {

// ---------------------------------------------------------------------------
// K1 packer.  One warp per packed token; 16-byte loads of the bf16 source
// row (a vision row or the text-embedding row of the token's id), widened to
// the fp32 residual stream.  The canonical packed batch is where the samples
// of all tenants are concatenated (§4.3); gather_src comes from the plan.
// ---------------------------------------------------------------------------
// The bf16 source row of a gather index, null outside its buffer.
__device__ __forceinline__ const uint16_t* pack_source(int src, const uint16_t* vision,
                                                       int64_t n_vision, const int32_t* text_ids,
                                                       int64_t n_text, const uint16_t* table,
                                                       int vocab, int d) {
    if (src >= 0) return src < n_vision ? vision + (size_t)src * d : nullptr;
    const int64_t p = -(int64_t)src - 1;
    if (p >= n_text) return nullptr;
    const int id = text_ids[p];
    return id >= 0 && id < vocab ? table + (size_t)id * d : nullptr;
}

__global__ void __launch_bounds__(256) k_pack(const int32_t* __restrict__ gather, int n_tokens,
                                              const uint16_t* vision, int64_t n_vision,
                                              const int32_t* __restrict__ text_ids, int64_t n_text,
                                              const uint16_t* table, int vocab, int d,
                                              float* __restrict__ x, int* status) {
    pdl_entry();
    const int tok = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (tok >= n_tokens) return;
    const uint16_t* row =
        pack_source(gather[tok], vision, n_vision, text_ids, n_text, table, vocab, d);
    if (row == nullptr && lane == 0) report(status, JNX_ERR_DEVICE_BOUNDS);
    float4* out = reinterpret_cast<float4*>(x + (size_t)tok * d);
    const int nchunk = d / 8;
    for (int c0 = lane; c0 < nchunk; c0 += 128) {  // four loads ahead of their stores
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = c0 + 32 * k;
            v[k] = make_uint4(0u, 0u, 0u, 0u);
            if (row && c < nchunk) v[k] = reinterpret_cast<const uint4*>(row)[c];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = c0 + 32 * k;
            if (c >= nchunk) break;
            out[2 * c] =
                make_float4(__uint_as_float(v[k].x << 16), __uint_as_float(v[k].x & 0xFFFF0000u),
                            __uint_as_float(v[k].y << 16), __uint_as_float(v[k].y & 0xFFFF0000u));
            out[2 * c + 1] =
                make_float4(__uint_as_float(v[k].z << 16), __uint_as_float(v[k].z & 0xFFFF0000u),
                            __uint_as_float(v[k].w << 16), __uint_as_float(v[k].w & 0xFFFF0000u));
        }
    }
}

jnx_status pack_launch(const jnx_group* g, const uint16_t* vision, int64_t n_vision,
                       const int32_t* text_ids, int64_t n_text, const uint16_t* table, int vocab,
                       int d, float* x, int* status, cudaStream_t s) {
    if (d % 8) return fail(JNX_ERR_UNSUPPORTED, "pack: d %% 8 != 0");
    if (g->n_tokens == 0) return JNX_OK;
    pdl(k_pack, (g->n_tokens + 7) / 8, 256, 0, s)(g->gather_src, g->n_tokens, vision, n_vision,
                                                 text_ids, n_text, table, vocab, d, x, status);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? JNX_OK : fail(JNX_ERR_CUDA, "pack: %s", cudaGetErrorString(e));
}

// ---------------------------------------------------------------------------
// RMSNorm: one warp per row, the row held in registers (V float4 per lane) and,
// with `copy`, written out as it came,
// fp32 sum of squares reduced lane-wise then by a fixed shuffle tree, so a
// row's result does not depend on where it sits in the batch.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int V>
__global__ void __launch_bounds__(256) k_rmsnorm(const float* x,
                                                 const uint16_t* gamma, float eps,
                                                 int M, uint16_t* __restrict__ out,
                                                 float* __restrict__ copy) {
    pdl_entry();
    constexpr int D = V * 128;
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= M) return;
    const float4* xr = reinterpret_cast<const float4*>(x + (size_t)row * D);
    const uint2* g2 = reinterpret_cast<const uint2*>(gamma);
    float4 v[V];
    uint2 gg[V];  // in flight with the row: behind the first store it waited once more
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = xr[lane + 32 * i];
#pragma unroll
    for (int i = 0; i < V; ++i) gg[i] = g2[lane + 32 * i];
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < V; ++i)
        ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
    ss = warp_sum(ss);
    const float r = rsqrtf(ss / (float)D + eps);
    if (copy) {
        float4* crow = reinterpret_cast<float4*>(copy + (size_t)row * D);
#pragma unroll
        for (int i = 0; i < V; ++i) crow[lane + 32 * i] = v[i];
    }
    uint2* orow = reinterpret_cast<uint2*>(out + (size_t)row * D);
#pragma unroll
    for (int i = 0; i < V; ++i) {
        uint2 o;
        o.x = pack_bf2(v[i].x * r * bf2f(gg[i].x & 0xFFFF), v[i].y * r * bf2f(gg[i].x >> 16));
        o.y = pack_bf2(v[i].z * r * bf2f(gg[i].y & 0xFFFF), v[i].w * r * bf2f(gg[i].y >> 16));
        orow[lane + 32 * i] = o;
    }
}

// The packer with the first block's folded RMSNorm's first half (the residual
// GEMM epilogue does the same for every later norm): beside x, y = bf16(x * gamma)
// and, per row and 128-column block, the sum of x^2; the consuming GEMM scales its
// output rows by rsqrt(sum / d + eps).  One warp per row.  Bound by HBM: 2 bytes
// in, 6 out per element in one pass, where a packer and a kernel that read the
// fp32 rows back moved 12 (65,725 rows x 4,096: 340 + 400 us, now 329).
template <int V>
__global__ void __launch_bounds__(256)
    k_pack_prep(const int32_t* __restrict__ gather, int n_tokens,
                const uint16_t* vision, int64_t n_vision,
                const int32_t* __restrict__ text_ids, int64_t n_text,
                const uint16_t* table, int vocab, float* __restrict__ x, int* status,
                const uint16_t* gamma, uint16_t* __restrict__ y,
                float* __restrict__ ss) {
    pdl_entry();
    constexpr int D = V * 128;  // lane float4 i = 128-column block i
    const int tok = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (tok >= n_tokens) return;
    const uint16_t* row =
        pack_source(gather[tok], vision, n_vision, text_ids, n_text, table, vocab, D);
    if (row == nullptr && lane == 0) report(status, JNX_ERR_DEVICE_BOUNDS);
    const uint2* g2 = reinterpret_cast<const uint2*>(gamma);
    float4* xr = reinterpret_cast<float4*>(x + (size_t)tok * D);
    uint2* yr = reinterpret_cast<uint2*>(y + (size_t)tok * D);
    // G blocks at a time, the next G loaded ahead of the stores of these: a load
    // behind a store waits for its own data only then
    constexpr int G = V < 8 ? V : 8;
    uint2 w[2][G], gg[2][G];
    auto load = [&](int i0, uint2 (&wl)[G], uint2 (&gl)[G]) {
#pragma unroll
        for (int k = 0; k < G; ++k) {
            wl[k] = row ? reinterpret_cast<const uint2*>(row)[lane + 32 * (i0 + k)]
                        : make_uint2(0u, 0u);
            gl[k] = g2[lane + 32 * (i0 + k)];
        }
    };
    load(0, w[0], gg[0]);
#pragma unroll
    for (int i0 = 0; i0 < V; i0 += G) {
        const int b = i0 / G & 1;
        if (i0 + G < V) load(i0 + G, w[b ^ 1], gg[b ^ 1]);
#pragma unroll
        for (int k = 0; k < G; ++k) {
            const int i = i0 + k;
            const uint2 wk = w[b][k], gk = gg[b][k];
            const float4 v = make_float4(__uint_as_float(wk.x << 16),
                                         __uint_as_float(wk.x & 0xFFFF0000u),
                                         __uint_as_float(wk.y << 16),
                                         __uint_as_float(wk.y & 0xFFFF0000u));
            xr[lane + 32 * i] = v;
            float t = 0.f;
            t += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
            t = warp_sum(t);
            if (lane == 0) ss[(size_t)tok * V + i] = t;
            yr[lane + 32 * i] =
                make_uint2(pack_bf2(v.x * bf2f(gk.x & 0xFFFF), v.y * bf2f(gk.x >> 16)),
                           pack_bf2(v.z * bf2f(gk.y & 0xFFFF), v.w * bf2f(gk.y >> 16)));
        }
    }
}

jnx_status pack_prep_launch(const jnx_group* g, const uint16_t* vision, int64_t n_vision,
                            const int32_t* text_ids, int64_t n_text, const uint16_t* table,
                            int vocab, int d, float* x, int* status, const uint16_t* gamma,
                            uint16_t* y, float* ss, cudaStream_t s) {
    if (g->n_tokens == 0) return JNX_OK;
    auto launch = [&](auto k) {
        pdl(k, (g->n_tokens + 7) / 8, 256, 0, s)(g->gather_src, g->n_tokens, vision, n_vision,
                                                 text_ids, n_text, table, vocab, x, status, gamma,
                                                 y, ss);
    };
    switch (d) {
        case 256: launch(k_pack_prep<2>); break;
        case 512: launch(k_pack_prep<4>); break;
        case 1024: launch(k_pack_prep<8>); break;
        case 2048: launch(k_pack_prep<16>); break;
        case 4096: launch(k_pack_prep<32>); break;
        default: return fail(JNX_ERR_UNSUPPORTED, "pack: d=%d not in {256..4096}", d);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? JNX_OK : fail(JNX_ERR_CUDA, "pack: %s", cudaGetErrorString(e));
}

jnx_status rmsnorm_launch(const float* x, const uint16_t* gamma, float eps, int M, int d,
                          uint16_t* out, cudaStream_t s, float* copy) {
    if (M == 0) return JNX_OK;
    const int grid = (M + 7) / 8;
    switch (d) {
        case 256: pdl(k_rmsnorm<2>, grid, 256, 0, s)(x, gamma, eps, M, out, copy); break;
        case 512: pdl(k_rmsnorm<4>, grid, 256, 0, s)(x, gamma, eps, M, out, copy); break;
        case 1024: pdl(k_rmsnorm<8>, grid, 256, 0, s)(x, gamma, eps, M, out, copy); break;
        case 2048: pdl(k_rmsnorm<16>, grid, 256, 0, s)(x, gamma, eps, M, out, copy); break;
        case 4096: pdl(k_rmsnorm<32>, grid, 256, 0, s)(x, gamma, eps, M, out, copy); break;
        default: return fail(JNX_ERR_UNSUPPORTED, "rmsnorm: d=%d not in {256..4096}", d);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? JNX_OK : fail(JNX_ERR_CUDA, "rmsnorm: %s", cudaGetErrorString(e));
}

// ---------------------------------------------------------------------------
// Final RMSNorm + mean pool.  A cluster of kPoolCtas CTAs per sample, each
// walking its own contiguous share of the sample's rows in order (4 at a
// time); each thread owns columns tid, tid + 256, ...; a row's sum of squares
// is reduced by a fixed tree.  pooled[s] = gamma * mean_t(x_t * rstd_t): the
// CTAs' column sums meet in distributed shared memory and are added in rank
// order, so a sample's result depends on its own length only.  hidden
// (optional) = bf16(x_t * rstd_t * gamma).
//
// Bound by HBM (4 bytes in, 2 out per element).  With one CTA per sample a
// group of few samples left most SMs idle and walked each sample's rows one
// after another.  Before and after: 7 samples of 300 rows x 4096 pooled 123
// -> 21 us, 38 of 530 x 2048 hidden 333 -> 49 us (5.1 TB/s), 156 of 283 x
// 1024 both 92 -> 57 us; 222 of 296 x 4096 pooled, which filled the SMs
// already, 183 both ways (5.9 TB/s).
// ---------------------------------------------------------------------------
constexpr int kPoolCtas = 8;

// PRE: the next round's rows are loaded while this one is summed, for groups
// whose CTAs do not fill the SMs; otherwise the registers go to more CTAs.  At d
// = 4096 a round is two rows, so that three CTAs fit an SM (four rows, two CTAs:
// 222 samples 189 us, 608 489 against 467).
template <int C, bool PRE>  // C: columns per thread = d / 256
__global__ void __cluster_dims__(kPoolCtas, 1, 1) __launch_bounds__(256, C == 16 && !PRE ? 3 : 0)
    k_final_pool(const float* x, const uint16_t* gamma, float eps,
                 const int* __restrict__ cu, int parts, float* __restrict__ pooled,
                 uint16_t* __restrict__ hidden) {
    pdl_entry();
    constexpr int D = C * 256;
    constexpr int R = C == 16 ? 2 : 4;  // rows of a round
    __shared__ float red[2][R][8];
    __shared__ float sums[D];
    cg::cluster_group cluster = cg::this_cluster();
    const int s = blockIdx.x / parts, part = blockIdx.x % parts;
    const int r0 = cu[s], r1 = cu[s + 1];
    // rows of this CTA: an equal share in whole fours, the same cut in both
    // variants and for every round length, so that the sums associate alike
    static_assert(4 % R == 0, "a share is whole rounds");
    const int share = ((r1 - r0 + parts - 1) / parts + 3) / 4 * 4;
    const int t0 = min(r0 + part * share, r1), t1 = min(t0 + share, r1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float acc[C], gm[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        acc[c] = 0.f;
        gm[c] = hidden ? bf2f(gamma[tid + 256 * c]) : 0.f;
    }
    float nx[R][C];
    auto load = [&](int t) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c)
                nx[r][c] = t + r < t1 ? x[(size_t)(t + r) * D + tid + 256 * c] : 0.f;
    };
    if (PRE) load(t0);
    int buf = 0;
    for (int t = t0; t < t1; t += R, buf ^= 1) {
        float v[R][C];
        if (!PRE) load(t);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) v[r][c] = nx[r][c];
        if (PRE) load(t + R);
        float ss[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            ss[r] = 0.f;
#pragma unroll
            for (int c = 0; c < C; ++c) ss[r] += v[r][c] * v[r][c];
            ss[r] = warp_sum(ss[r]);
        }
        // the two buffers of partial sums take turns, so one barrier a round
        // is enough: a warp that writes a buffer again has passed the barrier
        // after the round that read it
        if (lane == 0) {
#pragma unroll
            for (int r = 0; r < R; ++r) red[buf][r][warp] = ss[r];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float tot = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) tot += red[buf][r][w];
            const float rs = rsqrtf(tot / (float)D + eps);
            if (t + r < t1) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    // a stated multiply-add: left to the compiler it would be one in
                    // some variants and two roundings in others
                    acc[c] = fmaf(v[r][c], rs, acc[c]);
                    if (hidden)
                        hidden[(size_t)(t + r) * D + tid + 256 * c] = f2bf(v[r][c] * rs * gm[c]);
                }
            }
        }
    }
    if (!pooled) return;
#pragma unroll
    for (int c = 0; c < C; ++c) sums[tid + 256 * c] = acc[c];
    constexpr int kCols = D / kPoolCtas;  // this CTA finishes columns [part kCols, + kCols)
    constexpr int kMine = (kCols + 255) / 256;  // of them this thread's, 256 apart
    float gl[kMine];  // their gains, loaded before the wait for the other CTAs
#pragma unroll
    for (int i = 0; i < kMine; ++i)
        gl[i] = bf2f(gamma[part * kCols + min(tid + 256 * i, kCols - 1)]);
    cluster.sync();
    const float inv = 1.0f / (float)(r1 - r0);
#pragma unroll
    for (int i = 0; i < kMine; ++i) {
        const int c = part * kCols + tid + 256 * i;
        if (tid + 256 * i >= kCols) break;
        float tot = 0.f;
#pragma unroll
        for (int k = 0; k < kPoolCtas; ++k) tot += *cluster.map_shared_rank(&sums[c], k);
        pooled[(size_t)s * D + c] = tot * inv * gl[i];
    }
    cluster.sync();  // no CTA's shared memory goes away while another reads it
}

jnx_status final_pool_launch(const float* x, const uint16_t* gamma, float eps, const int* cu,
                             int S, int d, float* pooled, uint16_t* hidden, cudaStream_t s) {
    if (S == 0 || (!pooled && !hidden)) return JNX_OK;
    // hidden rows alone need no cluster's sum: finer shares fill the SMs
    const int parts = pooled ? kPoolCtas : 4 * kPoolCtas;
    if (S > INT_MAX / parts) return fail(JNX_ERR_UNSUPPORTED, "final_pool: too many samples");
    const int grid = S * parts;
    // under four CTAs an SM the deep variant's loads hide the latency (7 x 4096:
    // 21 us against 26), above it the flat one is faster (222 x 4096: 183 us
    // against 195; 222 of 530 x 2048: 153 against 173)
    const bool pre = grid < 4 * num_sms();
    auto launch = [&](auto deep, auto flat) {
        if (pre)
            pdl(deep, grid, 256, 0, s)(x, gamma, eps, cu, parts, pooled, hidden);
        else
            pdl(flat, grid, 256, 0, s)(x, gamma, eps, cu, parts, pooled, hidden);
    };
    switch (d) {
        case 256: launch(k_final_pool<1, true>, k_final_pool<1, false>); break;
        case 512: launch(k_final_pool<2, true>, k_final_pool<2, false>); break;
        case 1024: launch(k_final_pool<4, true>, k_final_pool<4, false>); break;
        case 2048: launch(k_final_pool<8, true>, k_final_pool<8, false>); break;
        case 4096: launch(k_final_pool<16, true>, k_final_pool<16, false>); break;
        default: return fail(JNX_ERR_UNSUPPORTED, "final_pool: d=%d not in {256..4096}", d);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? JNX_OK : fail(JNX_ERR_CUDA, "final_pool: %s", cudaGetErrorString(e));
}

// ---------------------------------------------------------------------------
// RoPE table: (cos, sin) of pos * theta^(-2i/hd), evaluated in double and
// rounded to fp32 once, stored frequency-major (tab[i * max_pos + p]) so that
// rows of consecutive positions read consecutive entries.
//
// One CTA per (frequency, kRopeSpan positions).  Position p = kRopeFine a + b:
// the CTA evaluates sincos for the fine angles b and the coarse ones a only,
// and every entry by the angle-addition formulas in double (the error stays
// at a few 2^-53, invisible in the fp32 entry).  FP64 is what bounds this
// kernel (a few operations per clock and SM): with a pow and a sincos per
// entry 88 positions x 32 frequencies took 11.8 us and 830 x 128 36.7 us, this
// way 3.3 and 8.4 us.
// ---------------------------------------------------------------------------
constexpr int kRopeFine = 32, kRopeCoarse = 64, kRopeSpan = kRopeFine * kRopeCoarse;

struct RopeFreqs {
    double inv[128];  // theta^(-2i/hd), i < hd / 2
};

__global__ void __launch_bounds__(256) k_rope_table(float2* tab, int max_pos,
                                                    const __grid_constant__ RopeFreqs fr) {
    pdl_entry();
    __shared__ double2 fine[kRopeFine], coarse[kRopeCoarse];
    const int i = blockIdx.x, p0 = blockIdx.y * kRopeSpan;
    const int t = threadIdx.x;
    if (t < kRopeFine + kRopeCoarse) {
        const int p = t < kRopeFine ? t : p0 + (t - kRopeFine) * kRopeFine;
        if (p < max_pos) {
            double sn, cs;
            sincos((double)p * fr.inv[i], &sn, &cs);
            (t < kRopeFine ? fine[t] : coarse[t - kRopeFine]) = make_double2(cs, sn);
        }
    }
    __syncthreads();
    const int p1 = min(p0 + kRopeSpan, max_pos);
    for (int p = p0 + t; p < p1; p += 256) {
        const double2 a = coarse[(p - p0) / kRopeFine], b = fine[(p - p0) % kRopeFine];
        tab[(size_t)i * max_pos + p] =
            make_float2((float)(a.x * b.x - a.y * b.y), (float)(a.y * b.x + a.x * b.y));
    }
}

jnx_status rope_table_launch(float2* tab, int max_pos, int hd, float theta, cudaStream_t s) {
    const int half = hd / 2;
    if (max_pos <= 0 || half <= 0) return JNX_OK;
    if (half > 128) return fail(JNX_ERR_UNSUPPORTED, "rope table: head dim %d", hd);
    RopeFreqs fr;
    for (int i = 0; i < half; ++i) fr.inv[i] = pow((double)theta, -2.0 * i / (2.0 * half));
    pdl(k_rope_table, dim3(half, (max_pos + kRopeSpan - 1) / kRopeSpan), 256, 0, s)(tab, max_pos,
                                                                                  fr);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? JNX_OK : fail(JNX_ERR_CUDA, "rope table: %s", cudaGetErrorString(e));
}

}  // namespace jnx
