// Dense bf16 GEMM on the 5th-generation tensor cores (tcgen05, sm_103a).
//
//   C[M, N] = A[M, K] . B[N, K]^T      (A = activations, B = weights [out, in])
//
// Four kernels, of which the first three share the epilogues and the order of every
// K reduction:
//   k_gemm        persistent CTAs over output tiles of 128 x 256, 128 or 64
//                 (narrower for the fewer rows), with the per-tenant forms (LoRA
//                 up-projections, segmented weights)
//   k_gemm_pair   plain launches on CTA pairs (cta_group::2), tiles of 256 x 256
//                 or 128
//   k_gemm_batch  a table of products in one launch, either operand as it lies
//   k_gemm_split  K over a cluster of four CTAs (the samplers' long contractions):
//                 partial sums, added in rank order and stored by itself
// pick_bn has the rule among the first two.  Warp roles:
//   warp 0     TMA producer: A and B boxes of 64 K columns (128-byte swizzle)
//              into a shared-memory ring (4 stages of 128 x 256), completion on
//              mbarriers; all lanes wait, an elected one issues;
//   warp 1     MMA issuer: tcgen05.mma (K=16) into a TMEM accumulator,
//              double-buffered so the epilogue of tile i overlaps the
//              mainloop of tile i+1; tcgen05.commit frees smem stages /
//              signals the epilogue;
//   warps 2-5  epilogue: tcgen05.ld of their 32-lane TMEM quarter (one row
//              per thread), fused op, global store (2-9 where it is the bound).
// Fused epilogues used by the backbone block:
//   EPI_BF16   C -> bf16
//   EPI_F32    C -> fp32
//   EPI_RESID  x[M, N] (fp32 residual stream) += C
//   EPI_GLU    weights interleaved in 128-row gate/up blocks: out[M, N/2] =
//              act(C_gate) * C_up -> bf16   (SwiGLU / tanh-GeGLU)
//   EPI_ROPE   the fused Q|K|V projection: rotate-half RoPE at each row's
//              position on columns < rope_cols, then bf16
// and by the training paths (the GLU's backward, with the gate/up GEMM
// recomputed): EPI_GLU_SAVE (the multipliers u act'(g) | act(g)),
// EPI_GLU_BWD (dm times those multipliers), EPI_GLU_DM (the gate/up
// product times a dm already stored in the up columns).
// Every output element's K reduction runs in the same order whatever M is
// or where the row sits, so packed (grouped) and per-tenant runs agree
// bit for bit.  The split's order is another one, taken whatever the rows: an
// expert's last bits may differ between sampling and training, not by its group.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "jnx_dev.cuh"
#include "jnx_kernels.h"

namespace jnx {

namespace gemm {
constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;
constexpr int B_BYTES = BN * BK * 2;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int TMEM_COLS = 512;  // two 256-column fp32 accumulators
constexpr int STG_BYTES = 4 * 2048;  // epilogue staging, 2 KB per epilogue warp (4 warps)
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/ + STG_BYTES;
// with eight epilogue warps (two per TMEM lane quarter, each taking half of
// a tile's columns) for the epilogues whose column halves are independent;
// their staging slots are 4 KB (32 rows x 32 fp32 columns)
constexpr int STG_SLOT_EW8 = 4096;
constexpr int SMEM_BYTES_EW8 = SMEM_BYTES - STG_BYTES + 8 * STG_SLOT_EW8;
static_assert(SMEM_BYTES_EW8 <= 227 * 1024, "shared memory per CTA");
constexpr int RING_MAX = 24;  // stages of a narrow tile's ring, at most
// LoRA operands of one tile (K = 16, 32-byte rows): t rows and B rows, a
// 2-deep ring after the main stages.
constexpr int LT_BYTES = BM * 16 * 2;
constexpr int LB_BYTES = BN * 16 * 2;
constexpr int LSTAGE = LT_BYTES + LB_BYTES;
constexpr int SMEM_BYTES_LORA = SMEM_BYTES + 2 * LSTAGE;

// Narrow tiles (128 x BN, BN = 128 or 64) for launches whose 256-wide tiles
// leave SMs idle.  A tile's BN columns are two groups of BN / 2, so that one
// tile still holds what an epilogue combines: a gate group and its up group,
// or the two halves of a head that RoPE rotates.  Everything else is the wide
// kernel: the same K order, the same MMA depth, the same epilogues, so a
// result has the same bits whatever tile width the launch chose.
// Shared memory: a ring of p.stages stages of a_rows (16 .. 128) A rows and BN
// B rows, then the barriers and the staging slots.  The MMA always reads 128 A
// rows; those past a_rows are whatever follows in shared memory and land in
// accumulator rows that no epilogue stores.
// K steps of its tile's weights that a CTA asks into L2 while the grid ahead drains,
// where a launch is one round of tiles: a chain of such launches waits on HBM in each
// (300 launches of a sampling call 2,056 -> 1,932 us).  In longer launches the first
// tile's weights are little of the whole (65,725 rows 16.9 ms with and without).
constexpr int PREFETCH = 32;
constexpr int NARROW_BAR = 512;  // barrier block of a narrow ring
constexpr int narrow_smem(int bn, int stages, int a_rows, bool lora) {
    return stages * (a_rows + bn) * BK * 2 + A_BYTES - a_rows * BK * 2 +
           (lora ? 2 * (LT_BYTES + bn * 32) : 0) + 1024 + NARROW_BAR + STG_BYTES;
}
}  // namespace gemm

// Descriptor of a K-major bf16 tile with 32-byte rows (K = 16) stored with
// the 32-byte swizzle: 8-row atoms of 256 bytes.
__device__ __forceinline__ uint64_t sw32_desc(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;              // leading byte offset (unused: K fits one row)
    d |= (uint64_t)(256 >> 4) << 32;     // stride byte offset: next 8-row atom
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)6 << 61;              // layout: 32-byte swizzle
    return d;
}

struct NoLora {};

// Rows [row0, row_end) and column block nb of one output tile.  Without
// LoRA, tiles are plain 128-row blocks of M; with LoRA they are laid out per
// tenant segment so every tile belongs to one tenant (`seg`).
// Its columns: the two groups start at weight rows c0 and c1 (a 256-wide
// tile is one contiguous block, c1 = c0 + 128).
struct TileGeo {
    int row0, row_end, nb, seg;
    int c0, c1;
};

// Tile order: groups of `group_m` row-blocks, N fastest inside a group, so
// the CTAs resident at one time share a few A row-blocks and a band of B.
__device__ __forceinline__ void tile_coords(int tile, int num_m, int num_n, int group_m, int& mb,
                                            int& nb) {
    const int per_group = group_m * num_n;
    const int grp = tile / per_group;
    const int first_m = grp * group_m;
    const int gm = min(group_m, num_m - first_m);
    const int in = tile - grp * per_group;
    mb = first_m + in % gm;
    nb = in / gm;
}

// Both activations are g sigmoid(z): SiLU with z = g, and the tanh-form
// GELU 0.5 g (1 + tanh(u)) with z = 2 u, u = sqrt(2/pi) (g + 0.044715 g^3),
// since 0.5 (1 + tanh(u)) = sigmoid(2 u).  The sigmoid takes the fast
// exponential and an approximate reciprocal (a few ulp, far below the bf16
// rounding of every product that reads it); its limits are exact (an
// overflowing exponential gives 0).
__device__ __forceinline__ float sigmoid_fast(float z) {
    return __fdividef(1.0f, 1.0f + __expf(-z));
}
__device__ __forceinline__ float gelu_arg(float g) {
    return 1.5957691216057308f * (g + 0.044715f * g * g * g);  // 2 sqrt(2/pi) (g + a g^3)
}

__device__ __forceinline__ float act_fn(float g, int act) {
    return g * sigmoid_fast(act == JNX_GLU_SWIGLU ? g : gelu_arg(g));
}

// act(g) and its derivative, s = sigmoid(z): SiLU' = s (1 + g (1 - s)); for
// the GELU, with tanh(u) = 2 s - 1 and 1 - tanh(u)^2 = 4 s (1 - s),
// d/dg [0.5 g (1 + tanh(u))] = s + 2 g s (1 - s) sqrt(2/pi) (1 + 3 a g^2).
__device__ __forceinline__ void act_grad(float g, int act, float& a, float& da) {
    if (act == JNX_GLU_SWIGLU) {
        const float s = sigmoid_fast(g);
        a = g * s;
        da = s * (1.0f + g * (1.0f - s));
    } else {
        const float s = sigmoid_fast(gelu_arg(g));
        a = g * s;
        da = s + 2.0f * g * s * (1.0f - s) * 0.7978845608028654f *
                     (1.0f + 3.0f * 0.044715f * g * g);
    }
}

// Epilogue staging: each epilogue warp turns its 32 rows x 64 bytes from
// one-row-per-thread (the TMEM layout) into row-contiguous global accesses
// through a 2 KB shared-memory slot.  Writer: thread `lane` puts row `lane`.
// Reader: in step i (0..3) thread `lane` takes row 8 i + lane / 4, 16-byte
// unit lane % 4, so one instruction touches 8 rows x 64 contiguous bytes
// instead of 32 rows x 16 bytes.  Units are XOR-swizzled by (row / 2) % 4,
// which keeps both sides free of bank conflicts.
__device__ __forceinline__ void stg_put(uint8_t* stg, int lane, const uint4 (&v)[4]) {
    uint8_t* rowp = stg + lane * 64;
    const int sw = (lane >> 1) & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(rowp + ((j ^ sw) << 4)) = v[j];
}

__device__ __forceinline__ uint4 stg_get(const uint8_t* stg, int lane, int i) {
    const int r = 8 * i + (lane >> 2), j = lane & 3;
    return *reinterpret_cast<const uint4*>(stg + r * 64 + ((j ^ ((r >> 1) & 3)) << 4));
}

__device__ __forceinline__ uint4 pack8_bf16(const float* f) {
    uint4 w;
    w.x = pack_bf2(f[0], f[1]);
    w.y = pack_bf2(f[2], f[3]);
    w.z = pack_bf2(f[4], f[5]);
    w.w = pack_bf2(f[6], f[7]);
    return w;
}

// 32 bf16 per row (64 bytes) from this thread's row to rows row_base + 0..31
// at column `col` of a bf16 [*, ldo] matrix.
__device__ __forceinline__ void stg_store_bf16(uint8_t* stg, int lane, const uint4 (&v)[4],
                                               bf16_t* out, int ldo, int row_base, int row_end,
                                               int col, uint64_t pol) {
    stg_put(stg, lane, v);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 w = stg_get(stg, lane, i);
        const int row = row_base + 8 * i + (lane >> 2);
        if (row < row_end) st_global_u4_hint(out + (size_t)row * ldo + col + (lane & 3) * 8, w, pol);
    }
    __syncwarp();
}

// RMSNorm factor of a row whose A row is y = bf16(x * gamma) (folded norm):
// rsqrt(mean(x^2) + eps) from the row's partial sums of squares, added in a
// fixed order; 1 without a folded norm.
__device__ __forceinline__ float row_norm_scale(const GemmParams& p, int row, bool valid) {
    if (p.ss_in == nullptr || !valid) return 1.f;
    // d / 128 of them, an even number
    const float2* sp = reinterpret_cast<const float2*>(p.ss_in + (size_t)row * p.ss_parts);
    float t = 0.f;
    for (int i = 0; i < p.ss_parts / 2; ++i) {
        const float2 v = sp[i];
        t += v.x;
        t += v.y;
    }
    return rsqrtf(t / (float)p.ss_cols + p.ss_eps);
}

// The accumulator tile at tbase (this warp's 32 TMEM lanes = rows
// row_base..row_base+31, BN fp32 columns) -> the epilogue's output.
// NC, cb: the 32-column chunks [cb, cb + NC) of the tile this warp handles
// (all of them, or one half of a 256-wide tile with eight epilogue warps:
// EPI_GLU_BWD and EPI_GLU_DM).  Ring slots are indexed by the pass within
// this warp's range, so they stay compile-time.
template <int EPI, int NC, int BN>
__device__ __forceinline__ void epilogue_tile(uint32_t tbase, uint8_t* stg, int lane,
                                              int row_base, int row_end, const TileGeo& geo,
                                              const GemmParams& p, int cb) {
    constexpr int HC = BN / 64;  // chunks of one column group
    constexpr bool WIDE = BN == 256;
    const int n0 = geo.c0;
    const int my_row = row_base + lane;
    const bool valid = my_row < row_end;
    const uint64_t pol = l2_evict_first_policy();  // outputs and residual are streamed
    if constexpr (EPI == EPI_BF16) {
#pragma unroll 1
        for (int c = cb; c < cb + NC; ++c) {
            uint32_t r[32];
            tmem_ld32(tbase + c * 32, r);
            tmem_ld_wait();
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = pack8_bf16(reinterpret_cast<const float*>(r) + 8 * u);
            // a 32-column chunk never straddles a 128-column block
            const int n = n0 + c * 32;
            const int col = p.pack_up ? 256 * (n / 128) + 128 + n % 128 : n;
            stg_store_bf16(stg, lane, v, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           col, pol);
        }
    } else if constexpr (EPI == EPI_F32 || EPI == EPI_RESID) {
        // 16 fp32 columns (64 bytes) per staging pass; the residual is
        // loaded RD - 1 passes ahead of its use, so several passes' loads
        // are in flight while the accumulator is staged (a shallower ring for
        // half-tile warps, which run with fewer registers per thread)
        constexpr int RD = WIDE && NC == 4 ? 3 : 4;
        float* dst = EPI == EPI_RESID ? p.resid : static_cast<float*>(p.out);
        const int ld = EPI == EPI_RESID ? p.ldr : p.ldo;
        float4 xr[RD][4];
        uint2 gr[RD];  // folded norm: this lane's four gamma values of each pass
        const bool norm = EPI == EPI_RESID && p.norm_gamma != nullptr;
        auto load_resid = [&](int pass, float4 (&x)[4], uint2& gq) {
            const int col = n0 + pass * 16 + (lane & 3) * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = row_base + 8 * i + (lane >> 2);
                uint4 u = make_uint4(0u, 0u, 0u, 0u);
                if (row < row_end) u = ld_global_u4_hint(dst + (size_t)row * ld + col, pol);
                x[i] = make_float4(__uint_as_float(u.x), __uint_as_float(u.y),
                                   __uint_as_float(u.z), __uint_as_float(u.w));
            }
            if (norm) gq = *reinterpret_cast<const uint2*>(p.norm_gamma + col);
        };
        constexpr int NP = 2 * NC;  // staging passes of this warp
        const int pb = 2 * cb;
        if constexpr (EPI == EPI_RESID) {
#pragma unroll
            for (int q = 0; q < RD - 1; ++q) load_resid(pb + q, xr[q], gr[q]);
        }
        // folded RMSNorm (EPI_RESID with norm_gamma): y = bf16(x * gamma) and
        // the sums of x^2 of each of this lane's four rows over its columns,
        // one per 128-column half of the tile (8 staging passes each)
        float ssq[NC < 4 ? 1 : NC / 4][4] = {};
#pragma unroll
        for (int lc = 0; lc < NC; ++lc) {
            const int c = cb + lc;
            uint32_t r[32];
            tmem_ld32(tbase + c * 32, r);
            tmem_ld_wait();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int lp = 2 * lc + h;  // pass within this warp's range
                const int pass = pb + lp;
                if constexpr (EPI == EPI_RESID)
                    if (lp + RD - 1 < NP)
                        load_resid(pass + RD - 1, xr[(lp + RD - 1) % RD], gr[(lp + RD - 1) % RD]);
                uint4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[u] = make_uint4(r[16 * h + 4 * u], r[16 * h + 4 * u + 1],
                                      r[16 * h + 4 * u + 2], r[16 * h + 4 * u + 3]);
                stg_put(stg, lane, v);
                __syncwarp();
                const int col = n0 + pass * 16 + (lane & 3) * 4;
                float gf[4] = {0.f, 0.f, 0.f, 0.f};
                if (EPI == EPI_RESID && norm) {
                    const uint2 g = gr[lp % RD];
                    gf[0] = bf2f(g.x & 0xFFFF);
                    gf[1] = bf2f(g.x >> 16);
                    gf[2] = bf2f(g.y & 0xFFFF);
                    gf[3] = bf2f(g.y >> 16);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 w = stg_get(stg, lane, i);
                    const int row = row_base + 8 * i + (lane >> 2);
                    float4 o = make_float4(__uint_as_float(w.x), __uint_as_float(w.y),
                                           __uint_as_float(w.z), __uint_as_float(w.w));
                    if constexpr (EPI == EPI_RESID) {
                        const float4 x = xr[lp % RD][i];
                        o.x += x.x;
                        o.y += x.y;
                        o.z += x.z;
                        o.w += x.w;
                    }
                    if (row < row_end)
                        st_global_u4_hint(dst + (size_t)row * ld + col,
                                          make_uint4(__float_as_uint(o.x), __float_as_uint(o.y),
                                                     __float_as_uint(o.z), __float_as_uint(o.w)),
                                          pol);
                    if (EPI == EPI_RESID && norm) {
                        ssq[lp / 8][i] += o.x * o.x + o.y * o.y + o.z * o.z + o.w * o.w;
                        if (row < row_end)
                            *reinterpret_cast<uint2*>(p.norm_out + (size_t)row * p.N + col) =
                                make_uint2(pack_bf2(o.x * gf[0], o.y * gf[1]),
                                           pack_bf2(o.z * gf[2], o.w * gf[3]));
                    }
                }
                __syncwarp();
            }
        }
        if (norm) {
            // the four lanes of a row hold each half's columns between them
            const int parts = p.N / 128;
#pragma unroll
            for (int hb = 0; hb < NC / 4; ++hb)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float t = ssq[hb][i];
                    t += __shfl_xor_sync(0xffffffffu, t, 1);
                    t += __shfl_xor_sync(0xffffffffu, t, 2);
                    const int row = row_base + 8 * i + (lane >> 2);
                    if ((lane & 3) == 0 && row < row_end)
                        p.ss_out[(size_t)row * parts + (n0 + 32 * cb) / 128 + hb] = t;
                }
        }
    } else if constexpr (EPI == EPI_GLU) {
        const float rs = row_norm_scale(p, my_row, valid);
#pragma unroll 1
        for (int c = 0; c < HC; ++c) {
            uint32_t g[32], u[32];
            tmem_ld32(tbase + c * 32, g);
            tmem_ld32(tbase + (c + HC) * 32, u);
            tmem_ld_wait();
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float o[8];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    o[e] = act_fn(rs * __uint_as_float(g[8 * q + e]), p.act) *
                           (rs * __uint_as_float(u[8 * q + e]));
                v[q] = pack8_bf16(o);
            }
            stg_store_bf16(stg, lane, v, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           geo.nb * (BN / 2) + c * 32, pol);
        }
    } else if constexpr (EPI == EPI_GLU_SAVE) {
        const float rs = row_norm_scale(p, my_row, valid);
#pragma unroll 1
        for (int c = 0; c < HC; ++c) {
            uint32_t g[32], u[32];
            tmem_ld32(tbase + c * 32, g);
            tmem_ld32(tbase + (c + HC) * 32, u);
            tmem_ld_wait();
            uint4 vg[4], vu[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float og[8], ou[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    float a, da;
                    act_grad(rs * __uint_as_float(g[8 * q + e]), p.act, a, da);
                    og[e] = rs * __uint_as_float(u[8 * q + e]) * da;
                    ou[e] = a;
                }
                vg[q] = pack8_bf16(og);
                vu[q] = pack8_bf16(ou);
            }
            stg_store_bf16(stg, lane, vg, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           n0 + c * 32, pol);
            stg_store_bf16(stg, lane, vu, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           geo.c1 + c * 32, pol);
        }
    } else if constexpr (EPI == EPI_GLU_DM) {
        // as EPI_GLU_SAVE over the chunk pairs (gate c, up c + 4) of this
        // warp's range (all four, or two of them with eight epilogue warps),
        // with dm (this thread's row, the chunk's 32 F columns: 64
        // contiguous bytes of the up slot, through L1 so each 32-byte sector
        // is fetched once) loaded one chunk ahead; every lane of the warp has
        // its chunk's dm in registers before any lane's stores reach that
        // chunk's columns, so out may be aux
        const int c0 = cb / 2, nc = NC / 2;
        const float rs = row_norm_scale(p, my_row, valid);
        const bf16_t* dmrow = p.aux + (size_t)my_row * p.ldaux + n0 + 128;
        uint4 dmv[2][4];
        auto load_dm = [&](int c, uint4 (&v)[4]) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q] = valid ? *reinterpret_cast<const uint4*>(dmrow + c * 32 + 8 * q)
                             : make_uint4(0u, 0u, 0u, 0u);
        };
        load_dm(c0, dmv[0]);
#pragma unroll
        for (int lc = 0; lc < nc; ++lc) {
            const int c = c0 + lc;
            uint32_t g[32], u[32];
            tmem_ld32(tbase + c * 32, g);
            tmem_ld32(tbase + (c + 4) * 32, u);
            if (lc + 1 < nc) load_dm(c + 1, dmv[(lc + 1) & 1]);
            tmem_ld_wait();
            uint4 vg[4], vu[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 m4 = dmv[lc & 1][q];
                const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w};
                float og[8], ou[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    float a, da;
                    act_grad(rs * __uint_as_float(g[8 * q + e]), p.act, a, da);
                    const float dm = bf2f((mw[e / 2] >> (16 * (e & 1))) & 0xFFFF);
                    og[e] = dm * (rs * __uint_as_float(u[8 * q + e]) * da);
                    ou[e] = dm * a;
                }
                vg[q] = pack8_bf16(og);
                vu[q] = pack8_bf16(ou);
            }
            stg_store_bf16(stg, lane, vg, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           n0 + c * 32, pol);
            stg_store_bf16(stg, lane, vu, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           n0 + 128 + c * 32, pol);
        }
    } else if constexpr (EPI == EPI_GLU_BWD && WIDE && NC == 4) {
        // half-tile warps (4 KB staging slot): one staging round per 32-column
        // chunk, so each lane takes 8 contiguous columns of rows 8 i + lane / 4
        // and its multiplier loads and result stores are 16 bytes; the next
        // chunk's multipliers are in flight while one is finished.  F column f
        // has its gate slot at packed column 256 (f / 128) + f % 128, its up
        // slot 128 later; a lane reads each element before it writes it, so
        // out may be aux.
        auto pcol = [&](int c) {
            const int f = n0 + c * 32 + (lane & 3) * 8;
            return (f / 128) * 256 + (f % 128);
        };
        uint4 mg[2][4], mu[2][4];
        auto load_m = [&](int c, uint4 (&g)[4], uint4 (&u)[4]) {
            const int pc = pcol(c);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = row_base + 8 * i + (lane >> 2);
                g[i] = u[i] = make_uint4(0u, 0u, 0u, 0u);
                if (row < row_end) {
                    const bf16_t* src = p.aux + (size_t)row * p.ldaux + pc;
                    g[i] = ld_global_u4_hint(src, pol);
                    u[i] = ld_global_u4_hint(src + 128, pol);
                }
            }
        };
        load_m(cb, mg[0], mu[0]);
#pragma unroll
        for (int lc = 0; lc < NC; ++lc) {
            const int c = cb + lc;
            if (lc + 1 < NC) load_m(c + 1, mg[(lc + 1) & 1], mu[(lc + 1) & 1]);
            uint32_t r[32];
            tmem_ld32(tbase + c * 32, r);
            tmem_ld_wait();
            // row `lane` puts its 32 fp32 (8 units of 16 bytes, XOR-swizzled
            // by row % 8)
            uint8_t* rowp = stg + lane * 128;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                *reinterpret_cast<uint4*>(rowp + ((j ^ (lane & 7)) << 4)) =
                    make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
            __syncwarp();
            const int pc = pcol(c);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int rr = 8 * i + (lane >> 2), u0 = (lane & 3) * 2;
                const uint8_t* rp = stg + rr * 128;
                const uint4 a = *reinterpret_cast<const uint4*>(rp + ((u0 ^ (rr & 7)) << 4));
                const uint4 b = *reinterpret_cast<const uint4*>(rp + (((u0 + 1) ^ (rr & 7)) << 4));
                const float dm[8] = {__uint_as_float(a.x), __uint_as_float(a.y),
                                     __uint_as_float(a.z), __uint_as_float(a.w),
                                     __uint_as_float(b.x), __uint_as_float(b.y),
                                     __uint_as_float(b.z), __uint_as_float(b.w)};
                const uint4 gm = mg[lc & 1][i], um = mu[lc & 1][i];
                const uint32_t gw[4] = {gm.x, gm.y, gm.z, gm.w};
                const uint32_t uw[4] = {um.x, um.y, um.z, um.w};
                float og[8], ou[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    og[e] = dm[e] * bf2f((gw[e / 2] >> (16 * (e & 1))) & 0xFFFF);
                    ou[e] = dm[e] * bf2f((uw[e / 2] >> (16 * (e & 1))) & 0xFFFF);
                }
                const int row = row_base + rr;
                if (row < row_end) {
                    bf16_t* dst = static_cast<bf16_t*>(p.out) + (size_t)row * p.ldo + pc;
                    st_global_u4_hint(dst, pack8_bf16(og), pol);
                    st_global_u4_hint(dst + 128, pack8_bf16(ou), pol);
                }
            }
            __syncwarp();
        }
    } else if constexpr (EPI == EPI_GLU_BWD) {
        // accumulator: dm for F columns [n0, n0 + 256); F column f has its
        // gate slot at packed column 256 (f / 128) + f % 128 and its up slot
        // 128 later.  As EPI_RESID: 16 columns per pass, dm staged through
        // shared memory so lane handles 4 columns of rows 8 i + lane / 4 (its
        // loads and stores cover 8 rows x 32 contiguous bytes per
        // instruction), the multipliers of pass + RD - 1 in flight.  Each
        // element is read before the same lane writes it, so out may be aux.
        constexpr int RD = 4;
        auto pcol = [&](int pass) {
            const int f = n0 + pass * 16 + (lane & 3) * 4;
            return (f / 128) * 256 + (f % 128);
        };
        uint2 mg[RD][4], mu[RD][4];
        auto load_m = [&](int pass, uint2 (&g)[4], uint2 (&u)[4]) {
            const int pc = pcol(pass);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = row_base + 8 * i + (lane >> 2);
                g[i] = u[i] = make_uint2(0u, 0u);
                if (row < row_end) {
                    const bf16_t* src = p.aux + (size_t)row * p.ldaux + pc;
                    g[i] = ld_global_u2_hint(src, pol);
                    u[i] = ld_global_u2_hint(src + 128, pol);
                }
            }
        };
        constexpr int NP = 2 * NC;  // staging passes of this warp
        const int pb = 2 * cb;
#pragma unroll
        for (int q = 0; q < RD - 1; ++q) load_m(pb + q, mg[q], mu[q]);
#pragma unroll
        for (int lc = 0; lc < NC; ++lc) {
            const int c = cb + lc;
            uint32_t r[32];
            tmem_ld32(tbase + c * 32, r);
            tmem_ld_wait();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int lp = 2 * lc + h;  // pass within this warp's range
                const int pass = pb + lp;
                if (lp + RD - 1 < NP) load_m(pass + RD - 1, mg[(lp + RD - 1) % RD],
                                             mu[(lp + RD - 1) % RD]);
                uint4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[u] = make_uint4(r[16 * h + 4 * u], r[16 * h + 4 * u + 1],
                                      r[16 * h + 4 * u + 2], r[16 * h + 4 * u + 3]);
                stg_put(stg, lane, v);
                __syncwarp();
                const int pc = pcol(pass);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 wv = stg_get(stg, lane, i);
                    const int row = row_base + 8 * i + (lane >> 2);
                    const float dm[4] = {__uint_as_float(wv.x), __uint_as_float(wv.y),
                                         __uint_as_float(wv.z), __uint_as_float(wv.w)};
                    const uint2 gm = mg[lp % RD][i], um = mu[lp % RD][i];
                    const uint2 og = make_uint2(
                        pack_bf2(dm[0] * bf2f(gm.x & 0xFFFF), dm[1] * bf2f(gm.x >> 16)),
                        pack_bf2(dm[2] * bf2f(gm.y & 0xFFFF), dm[3] * bf2f(gm.y >> 16)));
                    const uint2 ou = make_uint2(
                        pack_bf2(dm[0] * bf2f(um.x & 0xFFFF), dm[1] * bf2f(um.x >> 16)),
                        pack_bf2(dm[2] * bf2f(um.y & 0xFFFF), dm[3] * bf2f(um.y >> 16)));
                    if (row < row_end) {
                        bf16_t* dst = static_cast<bf16_t*>(p.out) + (size_t)row * p.ldo + pc;
                        st_global_u2_hint(dst, og, pol);
                        st_global_u2_hint(dst + 128, ou, pol);
                    }
                }
                __syncwarp();
            }
        }
    } else if constexpr (EPI == EPI_ROPE) {
        const int hc = p.hd / 64;  // 32-column chunks in half a head
        const int half = p.hd / 2;
        // a position outside the (cos, sin) table is reported and its row
        // is left unrotated (the table load is skipped)
        int pos = valid ? p.pos[my_row] : 0;
        const bool pos_ok = pos >= 0 && pos < p.rope_ld;
        if (valid && !pos_ok) report(p.status, JNX_ERR_DEVICE_BOUNDS);
        if (!pos_ok) pos = 0;
        const float rs = row_norm_scale(p, my_row, valid);
        // a chunk pair's columns and its frequencies: a wide tile holds whole
        // heads (partner chunk hc further), a narrow one the groups' chunks
        const int pair = WIDE ? hc : HC;
        const int fr0 = WIDE ? 0 : (n0 % p.hd) / 32;
#pragma unroll 1
        for (int c = 0; c < (WIDE ? 8 : HC); ++c) {
            const int hchunk = WIDE ? c % (2 * hc) : fr0 + c;
            if (hchunk >= hc) continue;  // handled with its lower partner
            const int col = n0 + c * 32;
            const bool rot = valid && pos_ok && col < p.rope_cols;
            // (cos, sin) of this row's position for the chunk's 32
            // frequencies, loaded before the TMEM read so their latency
            // overlaps it; the table is frequency-major, so the warp's rows
            // (mostly consecutive positions) read consecutive entries
            float2 cs[32];
            if (rot) {
                const float2* src = p.rope + (size_t)(hchunk * 32) * p.rope_ld + pos;
#pragma unroll
                for (int e = 0; e < 32; ++e) cs[e] = src[(size_t)e * p.rope_ld];
            }
            uint32_t lo[32], hi[32];
            tmem_ld32(tbase + c * 32, lo);
            tmem_ld32(tbase + (c + pair) * 32, hi);
            tmem_ld_wait();
            float a[32], b[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                a[e] = rs * __uint_as_float(lo[e]);
                b[e] = rs * __uint_as_float(hi[e]);
            }
            if (rot) {
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const float cr = cs[e].x, sr = cs[e].y;
                    const float x0 = a[e], x1 = b[e];
                    a[e] = x0 * cr - x1 * sr;
                    b[e] = x1 * cr + x0 * sr;
                }
            }
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = pack8_bf16(a + 8 * q);
            stg_store_bf16(stg, lane, v, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           col, pol);
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = pack8_bf16(b + 8 * q);
            stg_store_bf16(stg, lane, v, static_cast<bf16_t*>(p.out), p.ldo, row_base, row_end,
                           col + half, pol);
        }
    }
}

// The two column groups of tile column nb.
template <int EPI, int BN>
__device__ __forceinline__ void tile_columns(int nb, const GemmParams& p, TileGeo& g) {
    g.nb = nb;
    constexpr int HB = BN / 2;
    if (BN < 256 && EPI == EPI_ROPE) {  // BN <= hd: a slice of one head and its rotation partner
        const int per_head = p.hd / BN;
        g.c0 = nb / per_head * p.hd + nb % per_head * HB;
        g.c1 = g.c0 + p.hd / 2;
    } else if (BN < 256 && (EPI == EPI_GLU || EPI == EPI_GLU_SAVE)) {
        const int f = nb * HB;  // F columns f .. f + HB - 1: gate and up blocks of 128 in turn
        g.c0 = 256 * (f / 128) + f % 128;
        g.c1 = g.c0 + 128;
    } else {
        g.c0 = nb * BN;
        g.c1 = g.c0 + HB;
    }
}

template <int EPI, bool LORA, int BN, class LG>
__device__ __forceinline__ TileGeo tile_geo(int tile, int num_m, int num_n, const GemmParams& p,
                                            const LG& lg) {
    int mb, nb;
    tile_coords(tile, num_m, num_n, p.group_m, mb, nb);
    TileGeo g;
    tile_columns<EPI, BN>(nb, p, g);
    if constexpr (LORA) {
        int sg = 0;
        while (sg + 1 < lg.n_seg && lg.seg_tile0[sg + 1] <= mb) ++sg;
        g.seg = sg;
        g.row0 = lg.seg_r0[sg] + (mb - lg.seg_tile0[sg]) * gemm::BM;
        g.row_end = min(g.row0 + gemm::BM, lg.seg_r1[sg]);
    } else {
        g.seg = 0;
        g.row0 = mb * gemm::BM;
        g.row_end = min(g.row0 + gemm::BM, p.M);
    }
    return g;
}

// One CTA's rows of a pair's 256-row tile, and the tile's columns.
template <int EPI, int BN>
__device__ __forceinline__ TileGeo pair_geo(int tile, int num_m, int num_n, const GemmParams& p,
                                            uint32_t rank) {
    int mb, nb;
    tile_coords(tile, num_m, num_n, p.group_m, mb, nb);
    TileGeo g;
    tile_columns<EPI, BN>(nb, p, g);
    g.seg = 0;
    g.row0 = mb * 256 + (int)rank * 128;
    g.row_end = min(g.row0 + 128, p.M);
    return g;
}

// The LoRA part holding weight row c (of a tile's columns), and its place there.
__device__ __forceinline__ void lora_part(const LoraGemm& lg, int c, int& part, int& c0) {
    part = 0;
    while (part + 1 < lg.n_parts && c >= lg.part_cols[part]) {
        c -= lg.part_cols[part];
        ++part;
    }
    c0 = c;
}

// BMN: B is MN-major, [K rows, N] as it lies (segmented launches: a tenant's K
// rows), for the gradient through a projection.
template <int EPI, bool LORA, int EW, int BN, bool BMN>
__global__ void __launch_bounds__(64 + 32 * EW, BN == 256 ? 1 : 2)
    k_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
           const __grid_constant__ typename std::conditional<LORA, LoraGemm, NoLora>::type lg,
           GemmParams p) {
    using gemm::A_BYTES;
    using gemm::BK;
    using gemm::BM;
    constexpr bool WIDE = BN == 256;
    constexpr uint32_t IDESC = idesc_bf16_f32(BM, BN) | (BMN ? 1u << 16 : 0u);
    static_assert(!BMN || EPI == EPI_F32 || EPI == EPI_GLU_BWD, "contiguous tile columns");
    constexpr int LT_BYTES = gemm::LT_BYTES, LSTAGE = LT_BYTES + BN * 32;
    constexpr int RING = WIDE ? gemm::STAGES : gemm::RING_MAX;  // barriers per direction
    constexpr uint32_t TMEM_COLS = 2 * BN;
    const int stages = WIDE ? gemm::STAGES : p.stages;
    const int a_bytes = WIDE ? A_BYTES : p.a_rows * BK * 2;
    const int stage_bytes = a_bytes + BN * BK * 2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* lsm = smem + stages * stage_bytes + A_BYTES - a_bytes;  // LoRA ring (LORA only)
    uint64_t* full = reinterpret_cast<uint64_t*>(lsm + (LORA ? 2 * LSTAGE : 0));
    uint64_t* empty = full + RING;
    uint64_t* tfull = empty + RING;
    uint64_t* tempty = tfull + 2;
    uint64_t* drain = tempty + 2;
    uint64_t* lfull = drain + 1;   // [2]
    uint64_t* lempty = lfull + 2;  // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(lempty + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* consumed = abort_flag + 1;
    volatile int* lconsumed = abort_flag + 2;

    const int warp = warp_uniform(threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < RING; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 32 * EW);
            mbar_init(&lfull[a], 1);
            mbar_init(&lempty[a], 1);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        *consumed = 0;
        *lconsumed = 0;
        fence_barrier_init();
        fence_proxy_async();
    }
    int num_m;
    if constexpr (LORA)
        num_m = lg.seg_tile0[lg.n_seg];
    else
        num_m = (p.M + BM - 1) / BM;
    const int num_n = p.N / BN;
    const int num_k = p.K / BK;
    const int num_tiles = num_m * num_n;
    if (warp == 0 && num_tiles <= gridDim.x && elect_one()) {
        // this tile's weights into L2, shared out over the row blocks that read them
        const TileGeo g = tile_geo<EPI, LORA, BN>(blockIdx.x, num_m, num_n, p, lg);
        int at = g.row0 / BM, of = num_m, brow = 0;
        if constexpr (LORA) {
            at = (g.row0 - lg.seg_r0[g.seg]) / BM;
            of = lg.seg_tile0[g.seg + 1] - lg.seg_tile0[g.seg];
            if (lg.seg_b) brow = lg.seg_tenant[g.seg] * (BMN ? p.K : p.N);
        }
        for (int kb = at; kb < min(num_k, gemm::PREFETCH); kb += of) {
            if constexpr (BMN) {
#pragma unroll
                for (int i = 0; i < BN / 64; ++i)
                    tma_prefetch_2d(&tb, g.c0 + 64 * i, brow + kb * BK);
            } else {
                tma_prefetch_2d(&tb, kb * BK, brow + g.c0);
                if constexpr (!WIDE) tma_prefetch_2d(&tb, kb * BK, brow + g.c1);
            }
        }
    }
    __syncwarp();
    pdl_entry();  // TMEM is taken once the grid ahead has given its own back
    if (warp == 1) {
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&ta);
        tma_prefetch_desc(&tb);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);

    int issued = 0, l_issued = 0;

    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        int lj = 0;
        uint32_t lphase = 0;
        bool ok = true;
        for (int tile = blockIdx.x; ok && tile < num_tiles && !__any_sync(0xffffffffu, *abort_flag);
             tile += gridDim.x) {
            const TileGeo g = tile_geo<EPI, LORA, BN>(tile, num_m, num_n, p, lg);
            int brow = 0;
            if constexpr (LORA)
                if (lg.seg_b) brow = lg.seg_tenant[g.seg] * (BMN ? p.K : p.N);
            for (int kb = 0; kb < num_k; ++kb) {
                if (!mbar_wait_warp(&empty[stage], phase ^ 1)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    uint8_t* sa = smem + stage * stage_bytes;
                    mbar_arrive_expect_tx(&full[stage], stage_bytes);
                    tma_load_2d(sa, &ta, kb * BK, g.row0, &full[stage]);
                    if constexpr (BMN) {
#pragma unroll
                        for (int i = 0; i < BN / 64; ++i)
                            tma_load_2d(sa + a_bytes + i * 64 * BK * 2, &tb, g.c0 + 64 * i,
                                        brow + kb * BK, &full[stage]);
                    } else {
                        tma_load_2d(sa + a_bytes, &tb, kb * BK, brow + g.c0, &full[stage]);
                        if constexpr (!WIDE)
                            tma_load_2d(sa + a_bytes + BN / 2 * BK * 2, &tb, kb * BK, brow + g.c1,
                                        &full[stage]);
                    }
                }
                __syncwarp();
                ++issued;
                if (++stage == stages) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            if constexpr (LORA) {
                if (!ok) break;
                if (lg.n_parts == 0) continue;  // segmented weights only
                // this tile's t rows (its part) and its tenant's B rows
                if (!mbar_wait_warp(&lempty[lj], lphase ^ 1)) {
                    ok = false;
                    break;
                }
                int part, c0;
                lora_part(lg, g.c0, part, c0);
                const int lrow = lg.seg_tenant[g.seg] * lg.part_cols[part] + c0;
                if (elect_one()) {
                    uint8_t* lt = lsm + lj * LSTAGE;
                    mbar_arrive_expect_tx(&lfull[lj], LSTAGE);
                    tma_load_2d(lt, &lg.tt, part * 16, g.row0, &lfull[lj]);
                    tma_load_2d(lt + LT_BYTES, &lg.tb[part], 0, lrow, &lfull[lj]);
                    if constexpr (!WIDE)  // both groups lie in one part
                        tma_load_2d(lt + LT_BYTES + BN / 2 * 32, &lg.tb[part], 0,
                                    lrow + g.c1 - g.c0, &lfull[lj]);
                }
                __syncwarp();
                ++l_issued;
                if (++lj == 2) {
                    lj = 0;
                    lphase ^= 1;
                }
            }
        }
        if (!ok) {
            *abort_flag = 1;
            report(p.status, JNX_ERR_TIMEOUT);
        }
    } else if (warp == 1) {
        int stage = 0, local = 0, lj = 0, n_used = 0, l_used = 0;
        uint32_t phase = 0, lphase = 0;
        bool ok = true;
        const uint32_t a_lo = sw128_desc_lo(smem_u32(smem));
        const uint32_t b_lo = sw128_desc_lo(smem_u32(smem) + a_bytes);
        for (int tile = blockIdx.x; ok && tile < num_tiles && !__any_sync(0xffffffffu, *abort_flag);
             tile += gridDim.x, ++local) {
            const int acc = local & 1;
            const uint32_t acc_phase = (local >> 1) & 1;
            if (!mbar_wait_warp(&tempty[acc], acc_phase ^ 1)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem_base + acc * BN;
            for (int kb = 0; kb < num_k; ++kb) {
                if (!mbar_wait_warp(&full[stage], phase)) {
                    ok = false;
                    break;
                }
                ++n_used;
                tc_fence_after();
                const uint32_t off = (uint32_t)(stage * stage_bytes) >> 4;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {
                        uint64_t db = desc_of(b_lo + off + 2 * kk, kSw128DescHi);
                        if constexpr (BMN)  // 16 K rows are two 8-row atoms
                            db = sw128_desc_mn(
                                smem_u32(smem) + stage * stage_bytes + a_bytes + kk * 2048,
                                64 * BK * 2, 1024);
                        tc_mma_f16(d, desc_of(a_lo + off + 2 * kk, kSw128DescHi), db, IDESC,
                                   (kb | kk) != 0);
                    }
                    tc_commit(&empty[stage]);
                }
                __syncwarp();
                if (++stage == stages) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            if constexpr (LORA) {
                // D += t[rows, part] . B_part[tenant][cols]^T (one K = 16 step);
                // none with segmented weights only (n_parts == 0)
                if (ok && lg.n_parts > 0) {
                    if (!mbar_wait_warp(&lfull[lj], lphase)) {
                        ok = false;
                    } else {
                        ++l_used;
                        tc_fence_after();
                        const uint32_t la = smem_u32(lsm + lj * LSTAGE);
                        if (elect_one()) {
                            tc_mma_f16(d, sw32_desc(la), sw32_desc(la + LT_BYTES), IDESC, 1);
                            tc_commit(&lempty[lj]);
                        }
                        __syncwarp();
                        if (++lj == 2) {
                            lj = 0;
                            lphase ^= 1;
                        }
                    }
                }
            }
            if (!ok) break;
            if (elect_one()) tc_commit(&tfull[acc]);
            __syncwarp();
        }
        if (!ok) {
            *abort_flag = 1;
            report(p.status, JNX_ERR_TIMEOUT);
        }
        *consumed = n_used;
        *lconsumed = l_used;
        // make sure no MMA is still writing TMEM before teardown
        if (elect_one()) tc_commit(drain);
        __syncwarp();
        mbar_wait(drain, 0);
    } else {
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        // with eight epilogue warps, warps 2-5 take chunks 0-3 of a tile and
        // warps 6-9 chunks 4-7 (the same lane quarters)
        const int cb = EW == 8 ? ((warp - 2) >> 2) * 4 : 0;
        // this warp's staging slot, after the barrier block
        uint8_t* stg = reinterpret_cast<uint8_t*>(full) + (WIDE ? 256 : gemm::NARROW_BAR) +
                       (warp - 2) * (EW == 8 ? gemm::STG_SLOT_EW8 : 2048);
        int local = 0;
        for (int tile = blockIdx.x; tile < num_tiles; tile += gridDim.x, ++local) {
            const int acc = local & 1;
            const uint32_t acc_phase = (local >> 1) & 1;
            const TileGeo g = tile_geo<EPI, LORA, BN>(tile, num_m, num_n, p, lg);
            const int row_base = g.row0 + q * 32;
            if constexpr (EPI == EPI_GLU_DM) {
                // this thread's dm for the tile (its row, its chunks of the
                // up slot) into L2 while the tile's K loop runs
                const int row = row_base + lane;
                const int nbytes = (EW == 8 ? 2 : 4) * 64;
                if (row < g.row_end)
                    for (int b = 0; b < nbytes; b += 128)
                        prefetch_l2(reinterpret_cast<const uint8_t*>(
                                        p.aux + (size_t)row * p.ldaux + g.nb * BN + 128 + cb * 16) +
                                    b);
            }
            if (!mbar_wait(&tfull[acc], acc_phase) || *abort_flag) {
                *abort_flag = 1;
                report(p.status, JNX_ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            epilogue_tile<EPI, EW == 8 ? BN / 64 : BN / 32, BN>(
                tmem_base + acc * BN + ((uint32_t)(q * 32) << 16), stg, lane, row_base, g.row_end,
                g, p, cb);
            tc_fence_before();
            mbar_arrive(&tempty[acc]);
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*abort_flag && warp == 0 && lane == 0) {
        // wait (bounded) for TMA copies this CTA issued but nobody consumed
        for (int i = *consumed; i < issued; ++i)
            mbar_wait(&full[i % stages], (i / stages) & 1, 100000000LL);
        for (int i = *lconsumed; i < l_issued; ++i)
            mbar_wait(&lfull[i & 1], (i >> 1) & 1, 100000000LL);
    }
    __syncwarp();
    if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
}

// ---------------------------------------------------------------------------
// The same GEMM on CTA pairs: tiles of 256 x BN shared by the two SMs of a
// cluster.  Each CTA stages its 128 A rows and its half of the tile's B rows;
// the leader's MMA warp issues M = 256 instructions over both CTAs' operands,
// and each CTA's epilogue warps take its own 128 accumulator rows.
//
// Why: a lone CTA's 128 x 256 tile takes in 48 KB per 64-deep K step, and an SM
// takes in about 70 bytes a clock, so the step lasts 690 clocks while its MMAs
// need 512 (clock64 in both warps of an instrumented build; more ring stages
// changed nothing).  With B split between the pair it is 32 KB, in six stages
// instead of four, and the MMAs bound it.  Single-CTA tiles against
// pairs: 8,192 x 4,096 x K 4,096 with the residual 187 -> 162 us (1,696 TFLOP/s),
// GeGLU gate/up of 4,800 rows x N 32,768 x K 2,048 364 -> 323 us (1,994).
// Tiles of 256 x 128 (24 KB a step and CTA, eight stages) are for the few rows that
// a chain of K steps bounds: 607 x 2,048 x K 16,384 with the residual 56.4 us in lone
// 128 x 128 tiles, 47.2 here.
//
// Barriers: `full` (leader only) counts both CTAs' bytes; `empty` and `tfull`
// are signalled in both CTAs by the leader's commits; `tempty` (leader only)
// counts the epilogue warps of both.  A CTA leaves only after a cluster barrier,
// so no barrier, operand or accumulator goes away under its peer.
// ---------------------------------------------------------------------------
namespace pair {
constexpr int BM = 256, BK = 64;
constexpr int A_BYTES = 128 * BK * 2;  // one CTA's rows of a stage
constexpr int stages(int bn) { return bn == 256 ? 6 : 8; }
constexpr int stage_bytes(int bn) { return A_BYTES + bn / 2 * BK * 2; }
constexpr int smem_bytes(int bn, int ew) {
    return stages(bn) * stage_bytes(bn) + 1024 + 256 +
           (ew == 8 ? 8 * gemm::STG_SLOT_EW8 : gemm::STG_BYTES);
}
static_assert(smem_bytes(256, 8) <= 227 * 1024 && smem_bytes(128, 4) <= 227 * 1024,
              "shared memory per CTA");
}  // namespace pair

template <int EPI, int EW, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(64 + 32 * EW, 1)
    k_gemm_pair(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                GemmParams p) {
    using pair::A_BYTES;
    using pair::BK;
    constexpr int STAGES = pair::stages(BN), STAGE_BYTES = pair::stage_bytes(BN);
    constexpr uint32_t IDESC = idesc_bf16_f32(pair::BM, BN);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* drain = tempty + 2;
    uint64_t* never = drain + 1;  // nothing arrives on it: a bounded pause when giving up
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = warp_uniform(threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 2 * EW);
        }
        mbar_init(drain, 1);
        mbar_init(never, 1);
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async();
    }
    const int num_m = (p.M + pair::BM - 1) / pair::BM;
    const int num_n = p.N / BN;
    const int num_k = p.K / BK;
    const int num_tiles = num_m * num_n;
    const int first = blockIdx.x >> 1, step = gridDim.x >> 1;
    if (warp == 0 && num_tiles <= step && elect_one()) {
        const TileGeo g = pair_geo<EPI, BN>(first, num_m, num_n, p, rank);
        for (int kb = g.row0 / pair::BM; kb < min(num_k, gemm::PREFETCH); kb += num_m)
            tma_prefetch_2d(&tb, kb * BK, rank ? g.c1 : g.c0);
    }
    __syncwarp();
    pdl_entry();  // TMEM is taken once the grid ahead has given its own back
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, 2 * BN);
        tmem_relinquish_pair();
    }
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&ta);
        tma_prefetch_desc(&tb);
    }
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);

    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = first; ok && tile < num_tiles && !__any_sync(0xffffffffu, *abort_flag);
             tile += step) {
            const TileGeo g = pair_geo<EPI, BN>(tile, num_m, num_n, p, rank);
            const int brow = rank ? g.c1 : g.c0;
            for (int kb = 0; kb < num_k; ++kb) {
                if (!mbar_wait_warp(&empty[stage], phase ^ 1)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    uint8_t* sa = smem + stage * STAGE_BYTES;
                    const uint32_t bar = map_rank(&full[stage], 0);
                    if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * STAGE_BYTES);
                    tma_load_2d_pair(sa, &ta, kb * BK, g.row0, bar);
                    tma_load_2d_pair(sa + A_BYTES, &tb, kb * BK, brow, bar);
                }
                __syncwarp();
                if (++stage == STAGES) {
                    stage = 0;
                    phase ^= 1;
                }
            }
        }
        if (!ok) {
            *abort_flag = 1;
            report(p.status, JNX_ERR_TIMEOUT);
        }
    } else if (warp == 1 && rank == 0) {
        int stage = 0, local = 0;
        uint32_t phase = 0;
        bool ok = true;
        const uint32_t a_lo = sw128_desc_lo(smem_u32(smem));
        const uint32_t b_lo = sw128_desc_lo(smem_u32(smem) + A_BYTES);
        for (int tile = first; ok && tile < num_tiles && !__any_sync(0xffffffffu, *abort_flag);
             tile += step, ++local) {
            const int acc = local & 1;
            if (!mbar_wait_cluster_warp(&tempty[acc], ((local >> 1) & 1) ^ 1)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem_base + acc * BN;
            for (int kb = 0; kb < num_k; ++kb) {
                if (!mbar_wait_cluster_warp(&full[stage], phase)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t off = (uint32_t)(stage * STAGE_BYTES) >> 4;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        tc_mma_f16_pair(d, desc_of(a_lo + off + 2 * kk, kSw128DescHi),
                                        desc_of(b_lo + off + 2 * kk, kSw128DescHi), IDESC,
                                        (kb | kk) != 0);
                    tc_commit_pair(&empty[stage]);
                }
                __syncwarp();
                if (++stage == STAGES) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            if (!ok) break;
            if (elect_one()) tc_commit_pair(&tfull[acc]);
            __syncwarp();
        }
        if (!ok) {
            *abort_flag = 1;
            report(p.status, JNX_ERR_TIMEOUT);
        }
        // no MMA still reads or writes either CTA after this
        if (elect_one()) tc_commit_pair(drain);
        __syncwarp();
        mbar_wait(drain, 0);
    } else if (warp == 1) {
        mbar_wait(drain, 0);  // the leader's last commit has reached this CTA
    } else {
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        const int cb = EW == 8 ? ((warp - 2) >> 2) * 4 : 0;
        uint8_t* stg = reinterpret_cast<uint8_t*>(full) + 256 +
                       (warp - 2) * (EW == 8 ? gemm::STG_SLOT_EW8 : 2048);
        int local = 0;
        for (int tile = first; tile < num_tiles; tile += step, ++local) {
            const int acc = local & 1;
            const TileGeo g = pair_geo<EPI, BN>(tile, num_m, num_n, p, rank);
            const int row_base = g.row0 + q * 32;
            if constexpr (EPI == EPI_GLU_DM) {
                // this thread's dm for the tile into L2 while its K loop runs
                const int row = row_base + lane;
                if (row < g.row_end)
                    prefetch_l2(p.aux + (size_t)row * p.ldaux + g.c0 + 128 + cb * 16);
            }
            if (!mbar_wait(&tfull[acc], (local >> 1) & 1) || *abort_flag) {
                *abort_flag = 1;
                report(p.status, JNX_ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            epilogue_tile<EPI, EW == 8 ? BN / 64 : BN / 32, BN>(
                tmem_base + acc * BN + ((uint32_t)(q * 32) << 16), stg, lane, row_base, g.row_end,
                g, p, cb);
            tc_fence_before();
            __syncwarp();
            if (elect_one()) mbar_arrive_cluster(map_rank(&tempty[acc], 0));
            __syncwarp();
        }
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    // giving up: time for copies in flight to land before any CTA leaves
    if (*abort_flag && warp == 0) mbar_wait(never, 0, 100000000LL);
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, 2 * BN);
}

// ---------------------------------------------------------------------------
// Segmented residual GEMM with K split over a cluster: x += A . B_t^T in tiles
// of 128 x 64, one per cluster of kSplit CTAs, each over its share of the K
// steps; the partial tiles meet in distributed shared memory and are added in
// rank order, then to x.  For the experts' long contractions over a tenant's few
// rows: a chain of 64 K steps of 0.18 us is all a narrow tile does (K = 4,096, 16
// rows: 17 us, 10.0 split).  Taken by the sampler for K >= 2,048, whatever the
// rows, so that a tenant's bits do not depend on its group; a training step's
// rows fill the SMs without it (5,300 us against 5,322 for eight tenants of 64).
// ---------------------------------------------------------------------------
constexpr int kSplit = 4;
constexpr int kSplitPad = 68;  // row stride of a partial tile (floats)
constexpr int split_smem(int stages, int a_rows) {
    return gemm::narrow_smem(64, stages, a_rows, false) - gemm::STG_BYTES +
           gemm::BM * kSplitPad * 4;
}

__global__ void __cluster_dims__(kSplit, 1, 1) __launch_bounds__(192)
    k_gemm_split(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                 const __grid_constant__ LoraGemm lg, GemmParams p) {
    using gemm::A_BYTES;
    using gemm::BK;
    using gemm::BM;
    constexpr int BN = 64, RING = gemm::RING_MAX;
    constexpr uint32_t IDESC = idesc_bf16_f32(BM, BN);
    const int stages = p.stages, a_bytes = p.a_rows * BK * 2, stage_bytes = a_bytes + BN * BK * 2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + stages * stage_bytes + A_BYTES - a_bytes);
    uint64_t* empty = full + RING;
    uint64_t* tfull = empty + RING;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* consumed = abort_flag + 1;
    float* part = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(full) + gemm::NARROW_BAR);
    const int warp = warp_uniform(threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank();

    if (threadIdx.x == 0) {
        for (int s = 0; s < RING; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(tfull, 1);
        *abort_flag = 0;
        *consumed = 0;
        fence_barrier_init();
        fence_proxy_async();
    }
    const TileGeo g = tile_geo<EPI_RESID, true, BN>(blockIdx.x / kSplit, lg.seg_tile0[lg.n_seg],
                                                    p.N / BN, p, lg);
    const int num_k = p.K / BK;
    const int k0 = rank * num_k / kSplit, k1 = (rank + 1) * num_k / kSplit;
    const int brow = lg.seg_tenant[g.seg] * p.N + g.c0;
    if (warp == 0 && elect_one())
        for (int kb = k0; kb < min(k1, k0 + gemm::PREFETCH); ++kb)
            tma_prefetch_2d(&tb, kb * BK, brow);
    __syncwarp();
    pdl_entry();  // TMEM is taken once the grid ahead has given its own back
    if (warp == 1) {
        tmem_alloc(tmem_slot, BN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);

    int issued = 0;
    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int kb = k0; kb < k1; ++kb) {
            if (!mbar_wait_warp(&empty[stage], phase ^ 1)) {
                ok = false;
                break;
            }
            if (elect_one()) {
                uint8_t* sa = smem + stage * stage_bytes;
                mbar_arrive_expect_tx(&full[stage], stage_bytes);
                tma_load_2d(sa, &ta, kb * BK, g.row0, &full[stage]);
                tma_load_2d(sa + a_bytes, &tb, kb * BK, brow, &full[stage]);
            }
            __syncwarp();
            ++issued;
            if (++stage == stages) {
                stage = 0;
                phase ^= 1;
            }
        }
        if (!ok) {
            *abort_flag = 1;
            report(p.status, JNX_ERR_TIMEOUT);
        }
    } else if (warp == 1) {
        int stage = 0, n_used = 0;
        uint32_t phase = 0;
        bool ok = true;
        const uint32_t a_lo = sw128_desc_lo(smem_u32(smem));
        const uint32_t b_lo = sw128_desc_lo(smem_u32(smem) + a_bytes);
        for (int kb = k0; kb < k1; ++kb) {
            if (!mbar_wait_warp(&full[stage], phase)) {
                ok = false;
                break;
            }
            ++n_used;
            tc_fence_after();
            const uint32_t off = (uint32_t)(stage * stage_bytes) >> 4;
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk)
                    tc_mma_f16(tmem_base, desc_of(a_lo + off + 2 * kk, kSw128DescHi),
                               desc_of(b_lo + off + 2 * kk, kSw128DescHi), IDESC,
                               kb > k0 || kk > 0);
                tc_commit(&empty[stage]);
            }
            __syncwarp();
            if (++stage == stages) {
                stage = 0;
                phase ^= 1;
            }
        }
        if (!ok) {
            *abort_flag = 1;
            report(p.status, JNX_ERR_TIMEOUT);
        }
        *consumed = n_used;
        if (elect_one()) tc_commit(tfull);  // all MMAs of this CTA
        __syncwarp();
        mbar_wait_warp(tfull, 0);
    } else {
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        if (!mbar_wait_warp(tfull, 0)) {
            *abort_flag = 1;
            report(p.status, JNX_ERR_TIMEOUT);
        } else if (g.row0 + q * 32 < g.row_end) {
            tc_fence_after();
            float* row = part + (q * 32 + lane) * kSplitPad;
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + c * 32, r);
                tmem_ld_wait();
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    *reinterpret_cast<uint4*>(row + c * 32 + 4 * u) =
                        make_uint4(r[4 * u], r[4 * u + 1], r[4 * u + 2], r[4 * u + 3]);
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem_base, BN);
    __syncwarp();
    cluster_sync_all();
    if (warp >= 2 && !*abort_flag) {
        // this rank's quarter of the columns: four threads a row, 32 rows a pass
        const int i = threadIdx.x - 64, c = rank * (BN / kSplit) + 4 * (i & 3);
        for (int r = i >> 2; g.row0 + r < g.row_end; r += 32) {
            float4* xp = reinterpret_cast<float4*>(p.resid + (size_t)(g.row0 + r) * p.ldr + g.c0 + c);
            const float4 x = *xp;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < kSplit; ++k) {
                float4 t;
                asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                             : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w)
                             : "r"(map_rank(part + r * kSplitPad + c, k))
                             : "memory");
                v.x += t.x;
                v.y += t.y;
                v.z += t.z;
                v.w += t.w;
            }
            *xp = make_float4(x.x + v.x, x.y + v.y, x.z + v.z, x.w + v.w);
        }
    }
    if (*abort_flag && warp == 0 && lane == 0)
        // wait (bounded) for TMA copies this CTA issued but nobody consumed
        for (int i = *consumed; i < issued; ++i)
            mbar_wait(&full[i % stages], (i / stages) & 1, 100000000LL);
    __syncwarp();
    cluster_sync_all();  // no CTA's partial tile goes away while another reads it
}

// ---------------------------------------------------------------------------
// A batch of GEMMs in one launch (GemmBatch): the wide single-CTA kernel over
// the tiles of all problems in turn, each with its own tensor maps and output.
// An operand may be MN-major (its rows are K): 64 x 64 boxes of it, 128-byte
// swizzled, are the tensor core's transposed operand as they are, which saves
// a transposed copy in memory.  What it replaces and the times stand at its
// callers.
// ---------------------------------------------------------------------------
template <int EPI, bool AMN, bool BMN>
__global__ void __launch_bounds__(192, 1) k_gemm_batch(const __grid_constant__ GemmBatch gb) {
    using namespace gemm;
    constexpr uint32_t IDESC =
        idesc_bf16_f32(BM, BN) | (AMN ? 1u << 15 : 0u) | (BMN ? 1u << 16 : 0u);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* drain = tempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* consumed = abort_flag + 1;
    const int warp = warp_uniform(threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 128);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        *consumed = 0;
        fence_barrier_init();
        fence_proxy_async();
    }
    pdl_entry();  // TMEM is taken once the grid ahead has given its own back
    if (warp == 1) {
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);
    int issued = 0;

    // the problem of a tile, and the tile's place in it (row blocks fastest)
    int pi = 0;
    auto find = [&](int tile, int& mb, int& nb) -> const GemmBatch::Problem& {
        while (pi + 1 < gb.n && gb.p[pi + 1].tile0 <= tile) ++pi;
        const GemmBatch::Problem& q = gb.p[pi];
        const int mt = (q.m + BM - 1) / BM, in = tile - q.tile0;
        mb = in % mt;
        nb = in / mt;
        return q;
    };

    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = blockIdx.x; ok && tile < gb.tiles && !__any_sync(0xffffffffu, *abort_flag);
             tile += gridDim.x) {
            int mb, nb;
            const GemmBatch::Problem& q = find(tile, mb, nb);
            for (int kb = 0; kb < q.k; ++kb) {
                if (!mbar_wait_warp(&empty[stage], phase ^ 1)) {
                    ok = false;
                    break;
                }
                const bool second = kb >= q.k1;
                const int ka = second ? kb - q.k1 : kb;
                const int bk = (ka >> q.b_twice) * BK;
                const CUtensorMap* ma = &gb.map[q.a];
                const CUtensorMap* mbp = &gb.map[second ? q.b2 : q.b];
                if (elect_one()) {
                    uint8_t* sa = smem + stage * STAGE_BYTES;
                    mbar_arrive_expect_tx(&full[stage], STAGE_BYTES);
                    if constexpr (AMN) {
#pragma unroll
                        for (int i = 0; i < BM / 64; ++i)
                            tma_load_2d(sa + i * 64 * BK * 2, ma, mb * BM + 64 * i, kb * BK,
                                        &full[stage]);
                    } else {
                        tma_load_2d(sa, ma, (second ? q.ax2 : q.ax) + ka * BK, q.arow + mb * BM,
                                    &full[stage]);
                    }
                    if constexpr (BMN) {
#pragma unroll
                        for (int i = 0; i < BN / 64; ++i)
                            tma_load_2d(sa + A_BYTES + i * 64 * BK * 2, mbp, nb * BN + 64 * i, bk,
                                        &full[stage]);
                    } else {
                        tma_load_2d(sa + A_BYTES, mbp, bk, nb * BN, &full[stage]);
                    }
                }
                __syncwarp();
                ++issued;
                if (++stage == STAGES) {
                    stage = 0;
                    phase ^= 1;
                }
            }
        }
        if (!ok) {
            *abort_flag = 1;
            report(gb.status, JNX_ERR_TIMEOUT);
        }
    } else if (warp == 1) {
        int stage = 0, local = 0, n_used = 0;
        uint32_t phase = 0;
        bool ok = true;
        const uint32_t a0 = smem_u32(smem), b0 = a0 + A_BYTES;
        for (int tile = blockIdx.x; ok && tile < gb.tiles && !__any_sync(0xffffffffu, *abort_flag);
             tile += gridDim.x, ++local) {
            int mb, nb;
            const GemmBatch::Problem& q = find(tile, mb, nb);
            const int acc = local & 1;
            if (!mbar_wait_warp(&tempty[acc], ((local >> 1) & 1) ^ 1)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem_base + acc * BN;
            for (int kb = 0; kb < q.k; ++kb) {
                if (!mbar_wait_warp(&full[stage], phase)) {
                    ok = false;
                    break;
                }
                ++n_used;
                tc_fence_after();
                const uint32_t off = stage * STAGE_BYTES;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {
                        // 16 K rows of an MN-major operand are two 8-row atoms
                        const uint64_t da =
                            AMN ? sw128_desc_mn(a0 + off + kk * 2048, 64 * BK * 2, 1024)
                                : sw128_desc(a0 + off + kk * 32);
                        const uint64_t db =
                            BMN ? sw128_desc_mn(b0 + off + kk * 2048, 64 * BK * 2, 1024)
                                : sw128_desc(b0 + off + kk * 32);
                        tc_mma_f16(d, da, db, IDESC, (kb | kk) != 0);
                    }
                    tc_commit(&empty[stage]);
                }
                __syncwarp();
                if (++stage == STAGES) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            if (!ok) break;
            if (elect_one()) tc_commit(&tfull[acc]);
            __syncwarp();
        }
        if (!ok) {
            *abort_flag = 1;
            report(gb.status, JNX_ERR_TIMEOUT);
        }
        *consumed = n_used;
        if (elect_one()) tc_commit(drain);
        __syncwarp();
        mbar_wait(drain, 0);
    } else {
        const int q4 = warp & 3;  // TMEM lane quarter this warp may access
        uint8_t* stg = reinterpret_cast<uint8_t*>(full) + 256 + (warp - 2) * 2048;
        int local = 0;
        for (int tile = blockIdx.x; tile < gb.tiles; tile += gridDim.x, ++local) {
            int mb, nb;
            const GemmBatch::Problem& q = find(tile, mb, nb);
            const int acc = local & 1;
            if (!mbar_wait(&tfull[acc], (local >> 1) & 1) || *abort_flag) {
                *abort_flag = 1;
                report(gb.status, JNX_ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            TileGeo g;
            g.nb = nb;
            g.seg = 0;
            g.c0 = nb * BN;
            g.c1 = g.c0 + 128;
            g.row0 = mb * BM;
            g.row_end = min(g.row0 + BM, q.m);
            GemmParams p{};
            p.out = p.resid = q.out;
            p.ldo = p.ldr = gb.ldo;
            epilogue_tile<EPI, 8, 256>(tmem_base + acc * BN + ((uint32_t)(q4 * 32) << 16), stg,
                                       lane, g.row0 + q4 * 32, g.row_end, g, p, 0);
            tc_fence_before();
            mbar_arrive(&tempty[acc]);
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*abort_flag && warp == 0 && lane == 0) {
        // wait (bounded) for TMA copies this CTA issued but nobody consumed
        for (int i = *consumed; i < issued; ++i)
            mbar_wait(&full[i % STAGES], (i / STAGES) & 1, 100000000LL);
    }
    __syncwarp();
    if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

typedef CUresult (*PFN_tmapEncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                        const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                        const cuuint32_t*, CUtensorMapInterleave,
                                        CUtensorMapSwizzle, CUtensorMapL2promotion,
                                        CUtensorMapFloatOOBfill);

static PFN_tmapEncodeTiled encode_fn() {
    static PFN_tmapEncodeTiled fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void* f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_tmapEncodeTiled>(f);
    });
    return fn;
}

bool make_tmap_bf16(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols,
                    uint64_t row_stride_elems, uint32_t box_rows, uint32_t box_cols,
                    int swizzle_bytes) {
    PFN_tmapEncodeTiled fn = encode_fn();
    if (!fn) return false;
    if ((reinterpret_cast<uintptr_t>(ptr) & 15) || ((row_stride_elems * 2) & 15)) return false;
    if (box_cols * 2 > (uint32_t)swizzle_bytes) return false;  // a box row within one swizzle span
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {row_stride_elems * 2};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t estr[2] = {1, 1};
    const CUtensorMapSwizzle sw = swizzle_bytes == 128  ? CU_TENSOR_MAP_SWIZZLE_128B
                                  : swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                        : CU_TENSOR_MAP_SWIZZLE_32B;
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int num_sms() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

cudaError_t set_smem_limit(const void* fn, int bytes, std::atomic<uint64_t>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

// Whether tiles of bn columns hold what the launch's epilogue combines: RoPE needs a
// tile within one head, a folded norm's sums of squares one of 128 columns; the GLU
// backward with dm has wide tiles only.
static bool tile_holds(int bn, const GemmParams& p) {
    if (bn >= 256) return true;
    const bool wide_only = p.epi == EPI_GLU_DM || (p.epi == EPI_GLU_BWD && !p.seg_bn);
    return !(wide_only || (p.epi == EPI_ROPE && bn > p.hd) || (p.norm_gamma && bn < 128));
}

// A launch's output tiles: the form with the least estimated time, `fixed` (the
// launch, the first loads, the last tile's epilogue) + (rounds of tiles an SM works
// through) x (K / 64 steps) x the step.  GB300's times in microseconds, fitted over
// 42 launches of 8 to 10,000 tiles (K = 1,024 to 16,384; the picks lose 1 % to the
// best form): `alone` where every tile has its own SM (or pair), `busy` otherwise,
// which for a narrow tile is a round of two CTAs an SM.  Wide tiles are faster per
// column, so narrower ones win only where wide ones leave SMs idle, and pairs wherever
// they divide as well over the SMs.  N 2,048 x K 16,384, in the order of the table:
// 300 rows 92, 79, 46, 55 and 45 us; 607 rows 93, 80, 47, 56 and 73; 2,400 rows 97,
// 169, 142, 112 and 167; and 1,000 rows x N 32,768 x K 2,048 86, 75, 86, 93 and 131.
// Adapters, segments and MN-major operands have no pairs.
constexpr int kPairTile = 512, kPairNarrow = 384;  // a pair's tiles of 256 and of 128 columns

static int pick_bn(int m_tiles, const GemmParams& p, bool pairs) {
    static const struct { int form, bn, rows, per_sm; double fixed, alone, busy; } kForms[] = {
        {256, 256, 1, 1, 6.1, 0.34, 0.345},
        {kPairTile, 256, 2, 1, 9.4, 0.273, 0.295},
        {kPairNarrow, 128, 2, 1, 6.9, 0.157, 0.17},
        {128, 128, 1, 2, 5.3, 0.197, 0.395},
        {64, 64, 1, 2, 4.8, 0.156, 0.32}};
    const int sms = num_sms();
    int best = 256;
    double least = 1e30;
    for (const auto& f : kForms) {
        if (f.rows == 2 && !pairs) continue;
        if (!tile_holds(f.bn, p)) continue;
        const long long tiles = (long long)((m_tiles + f.rows - 1) / f.rows) * (p.N / f.bn);
        const int slots = sms / f.rows * f.per_sm;
        const double step = tiles <= sms / f.rows ? f.alone : (tiles + slots - 1) / slots * f.busy;
        const double t = f.fixed + step * (p.K / gemm::BK);
        if (t < least) {
            best = f.form;
            least = t;
        }
    }
    return best;
}

// The ring of a narrow launch: as many stages as fit one CTA's shared memory,
// or half of it where the tiles are more than the SMs and two CTAs share one.
static void narrow_ring(GemmParams& p, int bn, long long tiles, bool lora) {
    const int budget = (tiles > num_sms() ? 112 : 224) * 1024;
    p.stages = gemm::RING_MAX;
    while (p.stages > 2 && gemm::narrow_smem(bn, p.stages, p.a_rows, lora) > budget) --p.stages;
}

template <int EPI, bool LORA, class LG, int EW, int BN, bool BMN>
static cudaError_t launch_bn(const CUtensorMap& ta, const CUtensorMap& tb, const LG& lg,
                             GemmParams p, long long tiles, cudaStream_t s) {
    static_assert(EW == 4 || (EW == 8 && !LORA && BN == 256 &&
                              (EPI == EPI_GLU_BWD || EPI == EPI_GLU_DM)),
                  "eight epilogue warps: the epilogue-bound GLU backward only");
    constexpr bool wide = BN == 256;
    constexpr int limit = wide ? (LORA ? gemm::SMEM_BYTES_LORA
                                       : (EW == 8 ? gemm::SMEM_BYTES_EW8 : gemm::SMEM_BYTES))
                               : 224 * 1024;
    if (!wide) narrow_ring(p, BN, tiles, LORA);
    const int smem = wide ? limit : gemm::narrow_smem(BN, p.stages, p.a_rows, LORA);
    const int per_sm = wide || smem > 112 * 1024 ? 1 : 2;
    const int grid = (int)std::min<long long>(tiles, (long long)num_sms() * per_sm);
    static std::atomic<uint64_t> attr{0};  // per instantiation, one bit per device
    cudaError_t e =
        set_smem_limit(reinterpret_cast<const void*>(k_gemm<EPI, LORA, EW, BN, BMN>), limit, attr);
    if (e != cudaSuccess) return e;
    pdl(k_gemm<EPI, LORA, EW, BN, BMN>, grid, 64 + 32 * EW, smem, s)(ta, tb, lg, p);
    return cudaGetLastError();
}

template <int EPI, int EW, int BN>
static cudaError_t launch_pair(const CUtensorMap& ta, const CUtensorMap& tb, GemmParams p,
                               cudaStream_t s) {
    constexpr int smem = pair::smem_bytes(BN, EW);
    p.group_m = std::max(1, p.group_m / 2);  // row blocks of 256
    const long long tiles = (long long)((p.M + pair::BM - 1) / pair::BM) * (p.N / BN);
    const int grid = 2 * (int)std::min<long long>(tiles, num_sms() / 2);
    static std::atomic<uint64_t> attr{0};
    cudaError_t e =
        set_smem_limit(reinterpret_cast<const void*>(k_gemm_pair<EPI, EW, BN>), smem, attr);
    if (e != cudaSuccess) return e;
    pdl(k_gemm_pair<EPI, EW, BN>, grid, 64 + 32 * EW, smem, s)(ta, tb, p);
    return cudaGetLastError();
}

// The launch of one epilogue at the tile width bn (kPairTile: a CTA pair's).
template <int EPI, bool LORA, class LG, int EW = 4, bool BMN = false>
static cudaError_t launch_epi(const CUtensorMap& ta, const CUtensorMap& tb, const LG& lg,
                              const GemmParams& p, int bn, long long tiles, cudaStream_t s) {
    // whoever picked bn: a RoPE tile wider than a head would divide by zero heads
    if (!tile_holds(bn == kPairNarrow ? 128 : bn, p)) return cudaErrorInvalidValue;
    if constexpr (!LORA)
        if (bn == kPairTile) return launch_pair<EPI, EW, 256>(ta, tb, p, s);
    if constexpr (EW == 4) {
        if constexpr (!LORA)
            if (bn == kPairNarrow) return launch_pair<EPI, EW, 128>(ta, tb, p, s);
        if (bn == 64) return launch_bn<EPI, LORA, LG, EW, 64, BMN>(ta, tb, lg, p, tiles, s);
        if (bn == 128) return launch_bn<EPI, LORA, LG, EW, 128, BMN>(ta, tb, lg, p, tiles, s);
    }
    return launch_bn<EPI, LORA, LG, EW, 256, BMN>(ta, tb, lg, p, tiles, s);
}

// Box rows of the two operands' tensor maps at tile width bn.
static int b_box(int bn) {
    if (bn == kPairTile || bn == kPairNarrow) return bn == kPairTile ? 128 : 64;
    return bn == 256 ? 256 : bn / 2;
}

// Rows of A a narrow stage holds: the tallest tile's rows, in powers of two.
static int a_box(int bn, int most_rows) {
    int r = gemm::BM;
    while (bn < 256 && r > 16 && r / 2 >= most_rows) r /= 2;
    return r;
}

// Tile-order group height: enough 128-row blocks of A to hold ~40 MB in L2
// while the group sweeps all column blocks, so each weight band is re-read
// once per group rather than once per few row blocks.  Measured on GB300 at
// 65,536 tokens: gate/up (K=4096) 1810 -> ~1870 TFLOP/s going from 16 to 40,
// QKV best at 32-48, down (K=11008) best at 14-16.
static int default_group_m(int K) {
    const double a_block = (double)gemm::BM * K * 2.0;
    int g = (int)(40.0 * 1024 * 1024 / a_block + 0.5);
    return g < 8 ? 8 : (g > 48 ? 48 : g);
}

jnx_status gemm_check(int M, int N, int K) {
    if (M < 0 || N <= 0 || K <= 0 || N % gemm::BN || K % gemm::BK)
        return fail(JNX_ERR_UNSUPPORTED, "gemm: need N %% 256 == 0 and K %% 64 == 0 (M=%d N=%d K=%d)",
                    M, N, K);
    return JNX_OK;
}

jnx_status gemm_launch(const uint16_t* A, int lda, const uint16_t* B, int ldb, GemmParams p,
                       cudaStream_t s) {
    jnx_status st = gemm_check(p.M, p.N, p.K);
    if (st != JNX_OK) return st;
    if (p.M == 0) return JNX_OK;
    const int m_tiles = (p.M + gemm::BM - 1) / gemm::BM;
    const int bn = pick_bn(m_tiles, p, true);
    p.a_rows = a_box(bn, std::min(p.M, gemm::BM));
    CUtensorMap ta, tb;
    if (!make_tmap_bf16(&ta, A, p.M, p.K, lda, p.a_rows, gemm::BK) ||
        !make_tmap_bf16(&tb, B, p.N, p.K, ldb, b_box(bn), gemm::BK))
        return fail(JNX_ERR_CUDA, "gemm: tensor map encode failed (alignment or driver)");
    const long long tiles = (long long)m_tiles * (p.N / std::min(bn, 256));
    if (p.group_m <= 0) p.group_m = default_group_m(p.K);
    cudaError_t e;
    const NoLora none{};
    switch (p.epi) {
        case EPI_BF16: e = launch_epi<EPI_BF16, false>(ta, tb, none, p, bn, tiles, s); break;
        // eight epilogue warps only where the epilogue is the bottleneck: with
        // the fp32 and residual epilogues they slowed the GEMMs on GB300 (the
        // 7B-class O / down projections 1,314 / 1,460 -> 1,246 / 1,419 TFLOP/s)
        case EPI_F32: e = launch_epi<EPI_F32, false>(ta, tb, none, p, bn, tiles, s); break;
        case EPI_RESID: e = launch_epi<EPI_RESID, false>(ta, tb, none, p, bn, tiles, s); break;
        case EPI_GLU: e = launch_epi<EPI_GLU, false>(ta, tb, none, p, bn, tiles, s); break;
        case EPI_ROPE: e = launch_epi<EPI_ROPE, false>(ta, tb, none, p, bn, tiles, s); break;
        case EPI_GLU_BWD:
            e = launch_epi<EPI_GLU_BWD, false, NoLora, 8>(ta, tb, none, p, bn, tiles, s);
            break;
        case EPI_GLU_SAVE: e = launch_epi<EPI_GLU_SAVE, false>(ta, tb, none, p, bn, tiles, s); break;
        case EPI_GLU_DM:
            e = launch_epi<EPI_GLU_DM, false, NoLora, 8>(ta, tb, none, p, bn, tiles, s);
            break;
        default: return fail(JNX_ERR_INVALID_ARG, "gemm: unknown epilogue %d", p.epi);
    }
    if (e != cudaSuccess) return fail(JNX_ERR_CUDA, "gemm launch: %s", cudaGetErrorString(e));
    return JNX_OK;
}

jnx_status gemm_launch_seg(const uint16_t* A, int lda, const uint16_t* B, int ldb, int n_tenants,
                           GemmParams p, int n_seg, const int* seg_r0, const int* seg_r1,
                           const int* seg_tenant, cudaStream_t s, bool b_mn, bool split_k) {
    jnx_status st = gemm_check(p.M, p.N, p.K);
    if (st != JNX_OK) return st;
    if (n_seg < 0 || n_seg > kLoraMaxSlots || n_tenants <= 0)
        return fail(JNX_ERR_UNSUPPORTED, "gemm: bad segment description");
    if (p.M == 0 || n_seg == 0) return JNX_OK;
    static thread_local LoraGemm lg;  // staging of the kernel argument (copied at launch)
    lg = LoraGemm{};
    lg.n_parts = 0;
    lg.seg_b = 1;
    lg.n_seg = n_seg;
    int tiles = 0, most = 0;
    for (int i = 0; i < n_seg; ++i) {
        if (seg_r0[i] < 0 || seg_r1[i] < seg_r0[i] || seg_r1[i] > p.M || seg_tenant[i] < 0 ||
            seg_tenant[i] >= n_tenants)
            return fail(JNX_ERR_INVALID_ARG, "gemm: bad segment %d", i);
        lg.seg_r0[i] = seg_r0[i];
        lg.seg_r1[i] = seg_r1[i];
        lg.seg_tenant[i] = seg_tenant[i];
        lg.seg_tile0[i] = tiles;
        tiles += (seg_r1[i] - seg_r0[i] + gemm::BM - 1) / gemm::BM;
        most = std::max(most, std::min(seg_r1[i] - seg_r0[i], gemm::BM));
    }
    lg.seg_tile0[n_seg] = tiles;
    if (tiles == 0) return JNX_OK;
    p.seg_bn = 1;
    const bool split = split_k && p.epi == EPI_RESID && !b_mn && !p.norm_gamma && p.K >= 2048;
    const int bn = split ? 64 : pick_bn(tiles, p, false);
    p.a_rows = a_box(bn, most);
    CUtensorMap ta, tb;
    if (!make_tmap_bf16(&ta, A, p.M, p.K, lda, p.a_rows, gemm::BK) ||
        !(b_mn ? make_tmap_bf16(&tb, B, (uint64_t)n_tenants * p.K, p.N, ldb, gemm::BK, 64)
               : make_tmap_bf16(&tb, B, (uint64_t)n_tenants * p.N, p.K, ldb,
                                split ? 64 : b_box(bn), gemm::BK)))
        return fail(JNX_ERR_CUDA, "gemm: tensor map encode failed (alignment or driver)");
    const long long total = (long long)tiles * (p.N / bn);
    if (p.group_m <= 0) p.group_m = default_group_m(p.K);
    cudaError_t e;
    if (split) {
        const long long ctas = total * kSplit;
        if (ctas > 0x7FFFFFFFLL) return fail(JNX_ERR_UNSUPPORTED, "gemm: too many tiles");
        const int budget = (ctas > num_sms() ? 112 : 224) * 1024;
        p.stages = std::min(gemm::RING_MAX, std::max(2, p.K / gemm::BK / kSplit));
        while (p.stages > 2 && split_smem(p.stages, p.a_rows) > budget) --p.stages;
        static std::atomic<uint64_t> attr{0};
        e = set_smem_limit(reinterpret_cast<const void*>(k_gemm_split), 224 * 1024, attr);
        if (e == cudaSuccess)
            e = pdl(k_gemm_split, (unsigned)ctas, 192, split_smem(p.stages, p.a_rows), s)(ta, tb,
                                                                                        lg, p);
        if (e != cudaSuccess) return fail(JNX_ERR_CUDA, "gemm launch: %s", cudaGetErrorString(e));
        return JNX_OK;
    }
    if (b_mn) {
        if (p.epi == EPI_F32)
            e = launch_epi<EPI_F32, true, LoraGemm, 4, true>(ta, tb, lg, p, bn, total, s);
        else if (p.epi == EPI_GLU_BWD)
            e = launch_epi<EPI_GLU_BWD, true, LoraGemm, 4, true>(ta, tb, lg, p, bn, total, s);
        else
            return fail(JNX_ERR_INVALID_ARG, "gemm: epilogue %d unsupported here", p.epi);
        if (e != cudaSuccess) return fail(JNX_ERR_CUDA, "gemm launch: %s", cudaGetErrorString(e));
        return JNX_OK;
    }
    switch (p.epi) {
        case EPI_BF16: e = launch_epi<EPI_BF16, true>(ta, tb, lg, p, bn, total, s); break;
        case EPI_F32: e = launch_epi<EPI_F32, true>(ta, tb, lg, p, bn, total, s); break;
        case EPI_RESID: e = launch_epi<EPI_RESID, true>(ta, tb, lg, p, bn, total, s); break;
        case EPI_GLU: e = launch_epi<EPI_GLU, true>(ta, tb, lg, p, bn, total, s); break;
        case EPI_GLU_SAVE: e = launch_epi<EPI_GLU_SAVE, true>(ta, tb, lg, p, bn, total, s); break;
        default: return fail(JNX_ERR_INVALID_ARG, "gemm: epilogue %d unsupported here", p.epi);
    }
    if (e != cudaSuccess) return fail(JNX_ERR_CUDA, "gemm launch: %s", cudaGetErrorString(e));
    return JNX_OK;
}

int batch_map(GemmBatch& gb, const uint16_t* ptr, uint64_t rows, uint64_t cols, uint64_t ld,
              bool mn, int box) {
    if (gb.n_maps >= kBatchMaps) return -1;
    if (!make_tmap_bf16(&gb.map[gb.n_maps], ptr, rows, cols, ld, mn ? gemm::BK : box, 64)) return -1;
    return gb.n_maps++;
}

bool batch_add(GemmBatch& gb, GemmBatch::Problem p) {
    if (gb.n >= kBatchMax) return false;
    p.tile0 = gb.tiles;
    gb.tiles += (p.m + gemm::BM - 1) / gemm::BM * p.nb;
    gb.p[gb.n++] = p;
    return true;
}

template <int EPI, bool AMN, bool BMN>
static cudaError_t launch_batch(const GemmBatch& gb, cudaStream_t s) {
    static std::atomic<uint64_t> attr{0};
    cudaError_t e = set_smem_limit(reinterpret_cast<const void*>(k_gemm_batch<EPI, AMN, BMN>),
                                   gemm::SMEM_BYTES, attr);
    if (e != cudaSuccess) return e;
    pdl(k_gemm_batch<EPI, AMN, BMN>, std::min(gb.tiles, num_sms()), 192, gemm::SMEM_BYTES, s)(gb);
    return cudaGetLastError();
}

jnx_status gemm_batch_launch(const GemmBatch& gb, int epi, bool a_mn, bool b_mn, cudaStream_t s) {
    if (gb.tiles == 0) return JNX_OK;
    cudaError_t e = cudaErrorInvalidValue;
    if (epi == EPI_F32 && !a_mn && !b_mn) e = launch_batch<EPI_F32, false, false>(gb, s);
    if (epi == EPI_F32 && !a_mn && b_mn) e = launch_batch<EPI_F32, false, true>(gb, s);
    if (epi == EPI_F32 && a_mn && b_mn) e = launch_batch<EPI_F32, true, true>(gb, s);
    if (epi == EPI_RESID && a_mn && b_mn) e = launch_batch<EPI_RESID, true, true>(gb, s);
    if (e != cudaSuccess) return fail(JNX_ERR_CUDA, "gemm batch launch: %s", cudaGetErrorString(e));
    return JNX_OK;
}

jnx_status gemm_launch_lora(const uint16_t* A, int lda, const uint16_t* B, int ldb, GemmParams p,
                            const LoraSpec& ls, cudaStream_t s) {
    jnx_status st = gemm_check(p.M, p.N, p.K);
    if (st != JNX_OK) return st;
    if (p.epi != EPI_ROPE && p.epi != EPI_RESID)
        return fail(JNX_ERR_UNSUPPORTED, "gemm: LoRA only with the RoPE or residual epilogue");
    if (ls.n_seg < 0 || ls.n_seg > kLoraMaxSlots || ls.n_parts < 1 || ls.n_parts > 3 ||
        (ls.ldt * 2) % 16 || ls.ldt < 16 * ls.n_parts)
        return fail(JNX_ERR_UNSUPPORTED, "gemm: bad LoRA description");
    int cols = 0;
    for (int i = 0; i < ls.n_parts; ++i) {
        if (ls.cols[i] <= 0 || ls.cols[i] % gemm::BN)
            return fail(JNX_ERR_UNSUPPORTED, "gemm: LoRA part widths must be multiples of 256");
        cols += ls.cols[i];
    }
    if (cols != p.N) return fail(JNX_ERR_INVALID_ARG, "gemm: LoRA parts do not cover N");
    if (p.M == 0 || ls.n_seg == 0) return JNX_OK;
    static thread_local LoraGemm lg;  // staging of the kernel argument (copied at launch)
    lg = LoraGemm{};
    lg.n_parts = ls.n_parts;
    lg.n_seg = ls.n_seg;
    int tiles = 0;
    for (int i = 0; i < ls.n_seg; ++i) {
        if (ls.seg_r0[i] < 0 || ls.seg_r1[i] < ls.seg_r0[i] || ls.seg_r1[i] > p.M ||
            ls.seg_tenant[i] < 0 || ls.seg_tenant[i] >= ls.n_tenants)
            return fail(JNX_ERR_INVALID_ARG, "gemm: bad LoRA segment %d", i);
        lg.seg_r0[i] = ls.seg_r0[i];
        lg.seg_r1[i] = ls.seg_r1[i];
        lg.seg_tenant[i] = ls.seg_tenant[i];
        lg.seg_tile0[i] = tiles;
        tiles += (ls.seg_r1[i] - ls.seg_r0[i] + gemm::BM - 1) / gemm::BM;
    }
    lg.seg_tile0[ls.n_seg] = tiles;
    if (tiles == 0) return JNX_OK;
    const int bn = pick_bn(tiles, p, false);
    p.a_rows = gemm::BM;  // the adapters' t rows come in whole tiles too
    CUtensorMap ta, tb;
    bool ok = make_tmap_bf16(&ta, A, p.M, p.K, lda, p.a_rows, gemm::BK) &&
              make_tmap_bf16(&tb, B, p.N, p.K, ldb, b_box(bn), gemm::BK) &&
              make_tmap_bf16(&lg.tt, ls.t, p.M, ls.ldt, ls.ldt, gemm::BM, 16, 32);
    for (int i = 0; i < ls.n_parts && ok; ++i) {
        lg.part_cols[i] = ls.cols[i];
        ok = make_tmap_bf16(&lg.tb[i], ls.b[i], (uint64_t)ls.n_tenants * ls.cols[i], kLoraRank,
                            kLoraRank, b_box(bn), 16, 32);
    }
    if (!ok) return fail(JNX_ERR_CUDA, "gemm: LoRA tensor map encode failed");
    const long long total = (long long)tiles * (p.N / bn);
    if (p.group_m <= 0) p.group_m = default_group_m(p.K);
    cudaError_t e = p.epi == EPI_ROPE ? launch_epi<EPI_ROPE, true>(ta, tb, lg, p, bn, total, s)
                                      : launch_epi<EPI_RESID, true>(ta, tb, lg, p, bn, total, s);
    if (e != cudaSuccess) return fail(JNX_ERR_CUDA, "gemm launch: %s", cudaGetErrorString(e));
    return JNX_OK;
}

}  // namespace jnx
