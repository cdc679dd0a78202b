// Attention backward on the 5th-generation tensor cores (tcgen05, sm_103a):
// the gradients of the per-sample bidirectional attention (one sample's
// tokens attend to each other only), for the per-tenant LoRA backward.
//
// With S = q k^T / sqrt(hd), P = softmax(S) (rows), O = P v and the
// incoming dO:  dv = P^T dO,  dP = dO v^T,  dS = P * (dP - D) with
// D = rowsum(dO * O),  dq = dS k / sqrt(hd),  dk = dS^T q / sqrt(hd).
// P is recomputed from the forward's saved log2-sum-exp of each row, so no
// row max or normalisation is needed here.
//
// One kernel k_attn_bwd<HD> runs the passes of its head dim (bwd_pass<HD, MODE>):
//   DQ   outer tile = 128 queries of head h, inner loop over the sample's
//        64-key tiles:       S = Q K^T, dP = dO V^T, dS, dQ += dS K
//   DKV  outer tile = 128 keys of K/V head g, inner loop over (query head
//        of the group, 64-query tile):  S^T = K Q^T, dP^T = V dO^T, P^T,
//        dS^T, dK += dS^T Q, dV += P^T dO       (head dims 64 / 128)
//   DK   as DKV without dV; DV as DKV without dP and dK (head dim 256,
//        whose two 256-column accumulators do not fit TMEM together)
// A CTA claims items from one queue of all passes, those of the keys before those of
// the queries, so the long ones start first and the short ones fill the end.  A launch
// a pass, its items dealt out in turn, left SMs idle at the end of each, and every
// warp looked each item up for itself (24,000 tokens with the forward: 995 -> 826 us
// at head dim 256, 1,344 -> 1,332 at 128, 571 -> 563 at 64).
// Each pass accumulates in TMEM and writes its rows once, so no atomics and
// a fixed summation order: a sample's gradients do not depend on where it
// sits in the packed batch.
//
// Warp roles (320 threads, one CTA per SM, persistent over work items):
//   warp 0     claims the items and hands them to the other warps; TMA producer:
//              the item's outer operands (A1, and A2 when the pass has a dP
//              product) into one buffer, inner operands B1 / B2 through rings that
//              run on from item to item
//   warp 1     MMA issuer: the two score-shaped products of inner tile j
//              into score buffer j % 2 (S at column 64 b, dP at 128 + 64 b),
//              issued two tiles ahead of the accumulating products, which
//              read P / dS (bf16, written by the elementwise warps over the
//              first 32 columns of the buffer they came from) as the TMEM A
//              operand and the inner tile from shared memory as the MN-major
//              B operand, into the accumulator(s) at column 256
//   warps 2-9  elementwise (a thread takes half of an outer row's 64 columns:
//              warps 2-5 the first, 6-9 the second): P = 2^(S c - lse),
//              dS = P (dP - D); then the epilogue: scale, inverse RoPE for
//              dq / dk, bf16, store, column chunks in turn between the halves
//              (four warps with a whole row a thread: layer forward + backward of
//              24,000 tokens 616 -> 571 us at head dim 64, 1,425 -> 1,343 at 128,
//              1,108 -> 1,095 at 256, whose 128 x 64 x 16 score MMAs bound it)
// Operands by pass:          A1   A2   B1   B2   accumulating products
//   DQ                       Q    dO   K_j  V_j  dQ += dS B1
//   DKV / DK / DV            K    V    Q_j  dO_j dK += dS^T B1, dV += P^T B2
// Rows of a tile past the sample's end hold other rows' data (or the
// tensor's zero fill): their scores are finite, their probabilities are set
// to zero through lse = +inf (inner columns) or an explicit mask (DQ keys),
// and their gradient rows are never stored.
#include <algorithm>

#include "jnx_bwd.h"
#include "jnx_dev.cuh"
#include "jnx_kernels.h"

namespace jnx {

namespace abwd {
constexpr int BM = 128;  // outer rows per item
constexpr int BN = 64;   // inner rows per tile
enum { DQ = 0, DKV = 1, DK = 2, DV = 3 };
constexpr int kBars = 27;  // of one pass; each pass of a launch has its own
constexpr int EW = 8;    // elementwise warps: two per TMEM lane quarter, one column half each
}  // namespace abwd

template <int HD, int MODE>
struct AttnBwdCfg {
    static_assert(HD == 64 || HD == 128 || HD == 256, "head dim 64, 128 or 256");
    static constexpr bool NEED_DP = MODE != abwd::DV;
    static constexpr int NACC = MODE == abwd::DKV ? 2 : 1;
    static constexpr int BM = abwd::BM, BN = abwd::BN;
    static constexpr int OB = BM * HD * 2;  // one outer operand tile
    static constexpr int IB = BN * HD * 2;  // one inner operand tile
    static constexpr int NB1 = HD == 256 ? 2 : 3;
    static constexpr int NB2 = (HD == 256 && NEED_DP) ? 1 : 2;
    // The accumulating product of tile j holds B1's tile until it is done, so with
    // two B1 slots the scores of tile j + 2 would wait for their whole load right
    // after it, and the product of tile j + 1 behind them.  There tiles go in
    // pairs instead: both accumulating products, then both tiles' scores, whose
    // loads have been under way since.  (MMA warp of head dim 256: 1,080 clocks a
    // tile waiting for B1 in the dQ pass and 1,940 in the dK pass of 4,350 and
    // 4,100; 24,000 tokens, dQ 283 -> 250 us and dK 380 -> 319.)
    static constexpr bool PAIRED = NB1 == 2 && NEED_DP;
    static constexpr int OFF_A2 = OB;
    static constexpr int OFF_B1 = NEED_DP ? 2 * OB : OB;
    static constexpr int OFF_B2 = OFF_B1 + NB1 * IB;
    static constexpr int END = OFF_B2 + NB2 * IB;
    static constexpr uint32_t S_COL = 0;        // score buffer b at b * BN
    static constexpr uint32_t DP_COL = 2 * BN;  // dP buffer b at 2 BN + b * BN
    static constexpr uint32_t ACC_COL = 256;
    static_assert(ACC_COL + NACC * HD <= 512, "TMEM columns");
    static_assert(MODE != abwd::DKV || HD <= 128, "dK and dV together need head dim <= 128");
};

// The passes of a head dim, in the queue's order, and a launch's shared memory.
template <int HD>
struct AttnBwdPasses {
    static constexpr int N = HD == 256 ? 3 : 2;
    static constexpr int KEY = HD == 256 ? abwd::DK : abwd::DKV;  // the first
    static constexpr int K_END = AttnBwdCfg<HD, KEY>::END, Q_END = AttnBwdCfg<HD, abwd::DQ>::END;
    static constexpr int OFF_BAR = K_END > Q_END ? K_END : Q_END;  // DV stages less than DK
    static constexpr int SMEM = OFF_BAR + N * abwd::kBars * 8 + 48 + 1024;
    static_assert(SMEM <= 227 * 1024, "shared memory per CTA");
};

struct BwdItems {
    const int2* list;  // (sample, 128-row tile), most expensive first
    int n;
    int* claimed;      // items taken beyond the grid's first, 0 at launch
};

// A launch's arguments beyond the tensor maps.
struct BwdArgs {
    const int* cu;
    BwdItems items;
    int H, Hkv;
    float scale_log2, scale;
    const float *lse, *Dsum;
    const int* pos;
    const float2* rope;
    int rope_ld;
    uint16_t* dqkv;
    int ldq;
    int* status;
};

// Item w of a pass: list entry w / HP, head (query head for DQ, K/V head otherwise)
// w % HP.  L < 0: past the pass's last.
struct BwdWork {
    int tile, hp, start, L;
};

// The items of one pass, [q0, q0 + items) of the queue.  Warp 0 passes its claim and
// gets back the first one past the pass.
template <int HD, int MODE>
__device__ __forceinline__ int bwd_pass(const CUtensorMap& t_qkv_o, const CUtensorMap& t_qkv_i,
                                        const CUtensorMap& t_do_o, const CUtensorMap& t_do_i,
                                        const BwdArgs& p, uint8_t* sm, uint64_t* bars,
                                        volatile int* fail_flag, uint32_t tbase, int q0,
                                        int claim) {
    using C = AttnBwdCfg<HD, MODE>;
    constexpr int BM = C::BM, BN = C::BN;
    constexpr int NCH = HD / 64;  // 64-column (128-byte) chunks of an operand row
    constexpr bool IS_DQ = MODE == abwd::DQ;
    const int H = p.H, Hkv = p.Hkv, rope_ld = p.rope_ld, ldq = p.ldq;
    const int* __restrict__ cu = p.cu;
    const float* lse = p.lse;
    const float* Dsum = p.Dsum;
    const int* __restrict__ pos = p.pos;
    const float2* rope = p.rope;
    uint16_t* __restrict__ dqkv = p.dqkv;
    const float scale_log2 = p.scale_log2, scale = p.scale;
    uint8_t* sA1 = sm;
    uint8_t* sA2 = sm + C::OFF_A2;
    auto sB1 = [&](int b) { return sm + C::OFF_B1 + b * C::IB; };
    auto sB2 = [&](int b) { return sm + C::OFF_B2 + b * C::IB; };
    uint64_t* o_full = bars + 0;
    uint64_t* o_empty = bars + 1;
    uint64_t* b1_full = bars + 2;   // [3]
    uint64_t* b1_empty = bars + 5;  // [3]
    uint64_t* b2_full = bars + 8;   // [2]
    uint64_t* b2_empty = bars + 10; // [2]
    uint64_t* s_full = bars + 12;   // [2]
    uint64_t* p_full = bars + 14;   // [2]
    uint64_t* acc_full = bars + 16;
    uint64_t* acc_free = bars + 17;
    uint64_t* drain = bars + 18;
    uint64_t* xbar = bars + 19;  // [4] the two warps of a lane quarter have read a score tile
    uint64_t* w_full = bars + 23;   // [2] an item is in its slot; at 25 [2]: its readers have it
    uint64_t* w_empty = bars + 25;
    volatile int* slot = fail_flag + 1;  // [2] items
    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int group = H / Hkv;
    const int HP = IS_DQ ? H : Hkv;
    const int n_work = p.items.n * HP;
    // the next item as warp 0 hands it to the others
    int seen = 0;
    auto next_item = [&](bool& ok) -> BwdWork {
        const int b = seen & 1;
        if (!(ok = mbar_wait_warp(&w_full[b], (seen >> 1) & 1))) return BwdWork{0, 0, 0, -1};
        const BwdWork a{warp_uniform(slot[4 * b]), warp_uniform(slot[4 * b + 1]),
                        warp_uniform(slot[4 * b + 2]), warp_uniform(slot[4 * b + 3])};
        if (elect_one()) mbar_arrive(&w_empty[b]);
        __syncwarp();
        ++seen;
        return a;
    };
    // inner tiles of an item
    auto n_inner = [&](int L) { return IS_DQ ? (L + BN - 1) / BN : group * ((L + BN - 1) / BN); };

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        // all lanes run the loop, an elected one issues (see elect_one)
        {
            if (elect_one()) {
                tma_prefetch_desc(&t_qkv_o);
                tma_prefetch_desc(&t_qkv_i);
                tma_prefetch_desc(&t_do_o);
                tma_prefetch_desc(&t_do_i);
            }
            bool ok = true;
            int told = 0;            // items handed out
            auto tell = [&](const BwdWork& a) {
                const int b = told & 1;
                if (!mbar_wait_warp(&w_empty[b], ((told >> 1) & 1) ^ 1)) return false;
                if (elect_one()) {
                    slot[4 * b] = a.tile;
                    slot[4 * b + 1] = a.hp;
                    slot[4 * b + 2] = a.start;
                    slot[4 * b + 3] = a.L;
                    mbar_arrive(&w_full[b]);
                }
                __syncwarp();
                ++told;
                return true;
            };
            int no = 0;              // outer tiles loaded
            uint32_t g1 = 0, g2 = 0;  // inner tiles loaded into each ring
            auto load_inner = [&](const CUtensorMap* map, uint8_t* dst, int col, int row,
                                  uint64_t* full) {
                if (elect_one()) {
                    mbar_arrive_expect_tx(full, C::IB);
#pragma unroll
                    for (int c = 0; c < NCH; ++c)
                        tma_load_2d(dst + c * BN * 128, map, col + c * 64, row, full);
                }
                __syncwarp();
            };
            // The next item is claimed at an item's start, its list entry fetched with the
            // second tile's loads and its rows with the third's, each a step later than
            // what it needs was asked for: none of the three is waited for.
            int2 entry = make_int2(0, 0);
            int r0 = 0, r1 = 0;
            auto fetch_entry = [&]() {
                claim = __shfl_sync(0xffffffffu, claim, 0);
                if (claim - q0 < n_work) entry = p.items.list[(claim - q0) / HP];
            };
            auto fetch_rows = [&]() {
                if (claim - q0 < n_work) {
                    r0 = cu[entry.x];
                    r1 = cu[entry.x + 1];
                }
            };
            fetch_entry();
            fetch_rows();
            while (claim - q0 < n_work) {
                if (__any_sync(0xffffffffu, *fail_flag)) {
                    ok = false;
                    break;
                }
                const BwdWork a{warp_uniform(entry.y), warp_uniform((claim - q0) % HP),
                                warp_uniform(r0), warp_uniform(r1 - r0)};
                if (lane == 0) claim = (int)gridDim.x + atomicAdd(p.items.claimed, 1);
                __syncwarp();
                if (a.tile * BM >= a.L) {  // no rows
                    fetch_entry();
                    fetch_rows();
                    continue;
                }
                if (!(ok = tell(a))) break;
                const int row0 = a.start + a.tile * BM;
                if (no > 0 && !(ok = mbar_wait_warp(o_empty, (no - 1) & 1))) break;
                if (elect_one()) {
                    mbar_arrive_expect_tx(o_full, C::NEED_DP ? 2 * C::OB : C::OB);
                    const int k1 = (IS_DQ ? a.hp : H + a.hp) * HD;
                    const int k2 = (IS_DQ ? a.hp : H + Hkv + a.hp) * HD;
#pragma unroll
                    for (int c = 0; c < NCH; ++c) {
                        tma_load_2d(sA1 + c * BM * 128, &t_qkv_o, k1 + c * 64, row0, o_full);
                        if (C::NEED_DP)
                            tma_load_2d(sA2 + c * BM * 128, IS_DQ ? &t_do_o : &t_qkv_o, k2 + c * 64,
                                        row0, o_full);
                    }
                }
                __syncwarp();
                ++no;
                const int n = n_inner(a.L);
                const int nq = (a.L + BN - 1) / BN;
                for (int j = 0; j < n && ok; ++j) {
                    if (j == 1) fetch_entry();
                    if (j == 2) fetch_rows();
                    int row, c1, c2;
                    const CUtensorMap* m2;
                    if (IS_DQ) {
                        const int g = a.hp / group;
                        row = a.start + j * BN;
                        c1 = (H + g) * HD;
                        c2 = (H + Hkv + g) * HD;
                        m2 = &t_qkv_i;
                    } else {
                        const int hq = a.hp * group + j / nq;
                        row = a.start + (j % nq) * BN;
                        c1 = hq * HD;
                        c2 = hq * HD;
                        m2 = &t_do_i;
                    }
                    const int s1 = g1 % C::NB1;
                    if (!(ok = mbar_wait_warp(&b1_empty[s1], ((g1 / C::NB1) & 1) ^ 1))) break;
                    load_inner(&t_qkv_i, sB1(s1), c1, row, &b1_full[s1]);
                    ++g1;
                    const int s2 = g2 % C::NB2;
                    if (!(ok = mbar_wait_warp(&b2_empty[s2], ((g2 / C::NB2) & 1) ^ 1))) break;
                    load_inner(m2, sB2(s2), c2, row, &b2_full[s2]);
                    ++g2;
                }
                if (!ok) break;
                if (n < 2) fetch_entry();
                if (n < 3) fetch_rows();
            }
            ok = ok && tell(BwdWork{0, 0, 0, -1});
            if (!ok) *fail_flag = 1;
            // teardown: every copy issued has landed before the CTA exits
            if (no > 0) mbar_wait_warp(o_full, (no - 1) & 1, 100000000LL);
            for (uint32_t k = 0; k < (uint32_t)C::NB1 && k < g1; ++k) {
                const uint32_t i = g1 - 1 - k;
                mbar_wait_warp(&b1_full[i % C::NB1], (i / C::NB1) & 1, 100000000LL);
            }
            for (uint32_t k = 0; k < (uint32_t)C::NB2 && k < g2; ++k) {
                const uint32_t i = g2 - 1 - k;
                mbar_wait_warp(&b2_full[i % C::NB2], (i / C::NB2) & 1, 100000000LL);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        {
            constexpr uint32_t IDESC_S = idesc_bf16_f32(BM, BN);
            constexpr uint32_t IDESC_ACC = idesc_bf16_f32(BM, HD) | (1u << 16);  // B MN-major
            bool ok = true, issued = false;
            int no = 0;
            uint32_t c1s = 0, c2s = 0;  // B1 / B2 tiles taken by the score products
            uint32_t c1a = 0, c2a = 0;  // B1 / B2 tiles taken by the accumulating products
            uint32_t gs = 0, gp = 0;    // score tiles issued / P tiles consumed
            int items_done = 0;
            const uint32_t a1 = sw128_desc_lo(smem_u32(sA1)), a2 = sw128_desc_lo(smem_u32(sA2));
            auto issue_scores = [&]() -> bool {
                const int s1 = c1s % C::NB1;
                if (!mbar_wait_warp(&b1_full[s1], (c1s / C::NB1) & 1)) return false;
                tc_fence_after();
                const uint32_t b1 = sw128_desc_lo(smem_u32(sB1(s1)));
                const uint32_t d = tbase + C::S_COL + (gs & 1) * BN;
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < HD / 16; ++ks)
                        tc_mma_f16(d,
                                   desc_of(a1 + (ks >> 2) * BM * 8 + (ks & 3) * 2, kSw128DescHi),
                                   desc_of(b1 + (ks >> 2) * BN * 8 + (ks & 3) * 2, kSw128DescHi),
                                   IDESC_S, ks > 0);
                    if (MODE == abwd::DV) tc_commit(&b1_empty[s1]);
                }
                __syncwarp();
                ++c1s;
                if (C::NEED_DP) {
                    const int s2 = c2s % C::NB2;
                    if (!mbar_wait_warp(&b2_full[s2], (c2s / C::NB2) & 1)) return false;
                    tc_fence_after();
                    const uint32_t b2 = sw128_desc_lo(smem_u32(sB2(s2)));
                    const uint32_t d2 = tbase + C::DP_COL + (gs & 1) * BN;
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < HD / 16; ++ks)
                            tc_mma_f16(
                                d2, desc_of(a2 + (ks >> 2) * BM * 8 + (ks & 3) * 2, kSw128DescHi),
                                desc_of(b2 + (ks >> 2) * BN * 8 + (ks & 3) * 2, kSw128DescHi),
                                IDESC_S, ks > 0);
                        if (MODE == abwd::DQ || MODE == abwd::DK) tc_commit(&b2_empty[s2]);
                    }
                    __syncwarp();
                    ++c2s;
                }
                if (elect_one()) tc_commit(&s_full[gs & 1]);
                __syncwarp();
                ++gs;
                issued = true;
                return true;
            };
            // acc += X(tmem, 128 x 64 bf16) . B(smem inner tile, MN-major)
            auto acc_mma = [&](uint32_t acc_col, uint32_t xa, uint8_t* b, bool accumulate) {
                const uint32_t ba = smem_u32(b);
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < BN / 16; ++ks)  // 16 inner rows = 8 TMEM columns of X
                        tc_mma_f16_ts(tbase + acc_col, xa + ks * 8,
                                      sw128_desc_mn(ba + ks * 16 * 128, BN * 128, 1024), IDESC_ACC,
                                      accumulate || ks > 0);
                }
                __syncwarp();
            };
            auto commit = [&](uint64_t* bar) {
                if (elect_one()) tc_commit(bar);
                __syncwarp();
            };
            while (ok) {
                const BwdWork a = next_item(ok);
                if (a.L < 0 || __any_sync(0xffffffffu, *fail_flag)) break;
                const int n = n_inner(a.L);
                if (!(ok = mbar_wait_warp(o_full, no & 1))) break;
                ++no;
                tc_fence_after();
                ok = issue_scores() && (n < 2 || issue_scores());
                int ns = min(n, 2);  // score tiles issued
                if (ok && ns == n) commit(o_empty);
                for (int kt = 0; kt < n && ok; ++kt) {
                    const uint32_t pb = gp & 1;
                    if (!(ok = mbar_wait_warp(&p_full[pb], (gp >> 1) & 1))) break;
                    ++gp;
                    // the first accumulating product of an item overwrites the
                    // accumulator: the previous item's epilogue must have read it
                    if (kt == 0 && items_done > 0 &&
                        !(ok = mbar_wait_warp(acc_free, (items_done - 1) & 1)))
                        break;
                    tc_fence_after();
                    const uint32_t sb = tbase + C::S_COL + pb * BN;
                    const uint32_t db = tbase + C::DP_COL + pb * BN;
                    if (MODE == abwd::DQ || MODE == abwd::DK) {
                        const int s1 = c1a % C::NB1;
                        acc_mma(C::ACC_COL, sb, sB1(s1), kt > 0);  // dS (over S) . B1
                        commit(&b1_empty[s1]);
                        ++c1a;
                    } else if (MODE == abwd::DV) {
                        const int s2 = c2a % C::NB2;
                        if (!(ok = mbar_wait_warp(&b2_full[s2], (c2a / C::NB2) & 1))) break;
                        tc_fence_after();
                        acc_mma(C::ACC_COL, sb, sB2(s2), kt > 0);  // P^T (over S) . dO
                        commit(&b2_empty[s2]);
                        ++c2a;
                    } else {  // DKV
                        const int s1 = c1a % C::NB1, s2 = c2a % C::NB2;
                        acc_mma(C::ACC_COL, db, sB1(s1), kt > 0);       // dS^T (over dP) . Q
                        acc_mma(C::ACC_COL + HD, sb, sB2(s2), kt > 0);  // P^T (over S) . dO
                        commit(&b1_empty[s1]);
                        commit(&b2_empty[s2]);
                        ++c1a;
                        ++c2a;
                    }
                    // the score products of tile kt + 2 reuse buffer pb: the
                    // tensor core runs this thread's MMAs in issue order, so
                    // the products above have read it before they land
                    const int upto = !C::PAIRED ? kt + 3 : kt & 1 ? kt + 3 : 0;
                    for (; ok && ns < min(upto, n); ++ns) {
                        ok = issue_scores();
                        if (ok && ns + 1 == n) commit(o_empty);
                    }
                }
                if (!ok) break;
                commit(acc_full);
                ++items_done;
            }
            if (!ok) *fail_flag = 1;
            if (issued) {
                commit(drain);
                mbar_wait_warp(drain, 0, 100000000LL);
            }
        }
    } else {
        // ---------------- elementwise + epilogue ----------------
        const int quarter = warp & 3;
        const int half = (warp - 2) >> 2;  // this warp's 32 columns of a 64-column tile
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        uint32_t gs = 0;
        int items_done = 0;
        bool ok = true;
        while (ok) {
            const BwdWork a = next_item(ok);
            if (a.L < 0 || __any_sync(0xffffffffu, *fail_flag != 0)) break;
            const int L = a.L, n = n_inner(L);
            const int nq = (L + BN - 1) / BN;
            const int r = a.tile * BM + quarter * 32 + lane;  // this thread's outer row
            const bool rv = r < L;
            float lse_r = INFINITY, d_r = 0.f;
            if (IS_DQ && rv) {
                lse_r = lse[(size_t)(a.start + r) * H + a.hp];
                d_r = Dsum[(size_t)(a.start + r) * H + a.hp];
            }
            for (int j = 0; j < n; ++j) {
                // DKV / DK / DV: this half's 32 query columns' lse and D, one per
                // lane, broadcast with shuffles below
                float lq = INFINITY, dq = 0.f;
                if (!IS_DQ) {
                    const int hq = a.hp * group + j / nq;
                    const int q0 = (j % nq) * BN + half * 32;
                    if (q0 + lane < L) {
                        lq = lse[(size_t)(a.start + q0 + lane) * H + hq];
                        if (C::NEED_DP) dq = Dsum[(size_t)(a.start + q0 + lane) * H + hq];
                    }
                }
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(&s_full[gs & 1], (gs >> 1) & 1))))
                    break;
                tc_fence_after();
                const uint32_t tS = tbase + lane_base + C::S_COL + (gs & 1) * BN;
                const uint32_t tP = tbase + lane_base + C::DP_COL + (gs & 1) * BN;
                const int kvalid = L - j * BN - half * 32;  // DQ: this half's keys in the sample
                uint32_t pk[16], dk[16];
                {
                    uint32_t sv[32], dv[32];
                    tmem_ld32(tS + half * 32, sv);
                    if (C::NEED_DP) tmem_ld32(tP + half * 32, dv);
                    tmem_ld_wait();
                    // P and dS go over the first 32 columns of the buffers they
                    // come from: both warps of a lane quarter have read theirs
                    tc_fence_before();
                    __syncwarp();
                    if (elect_one()) mbar_arrive(&xbar[quarter]);
                    __syncwarp();
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(&xbar[quarter], gs & 1)))) break;
                    tc_fence_after();
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        float p[2], ds[2];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const float sc_s = __uint_as_float(sv[e + u]);
                            float l, dd = 0.f;
                            if (IS_DQ) {
                                l = lse_r;
                                dd = d_r;
                            } else {
                                l = __shfl_sync(0xffffffffu, lq, e + u);
                                if (C::NEED_DP) dd = __shfl_sync(0xffffffffu, dq, e + u);
                            }
                            p[u] = ex2_approx(sc_s * scale_log2 - l);
                            if (IS_DQ && e + u >= kvalid) p[u] = 0.f;
                            ds[u] = C::NEED_DP ? p[u] * (__uint_as_float(dv[e + u]) - dd) : 0.f;
                        }
                        pk[e / 2] = pack_bf2(p[0], p[1]);
                        dk[e / 2] = pack_bf2(ds[0], ds[1]);
                    }
                }
                if (MODE == abwd::DQ || MODE == abwd::DK) {
                    tmem_st16(tS + half * 16, dk);
                } else if (MODE == abwd::DV) {
                    tmem_st16(tS + half * 16, pk);
                } else {
                    tmem_st16(tS + half * 16, pk);
                    tmem_st16(tP + half * 16, dk);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (elect_one()) mbar_arrive(&p_full[gs & 1]);
                __syncwarp();
                ++gs;
            }
            if (!ok) break;
            // ---- epilogue: the accumulator rows -> dqkv (bf16) ----
            if (!(ok = __all_sync(0xffffffffu, mbar_wait(acc_full, items_done & 1)))) break;
            tc_fence_after();
            const int grow = a.start + r;
            const uint32_t tacc = tbase + lane_base + C::ACC_COL;
            for (int acc = 0; acc < C::NACC; ++acc) {
                // which gradient: dq (DQ), dk (DK, DKV first), dv (DV, DKV second)
                const bool is_v = MODE == abwd::DV || acc == 1;
                const int colo = IS_DQ ? a.hp * HD : (is_v ? (H + Hkv + a.hp) * HD : (H + a.hp) * HD);
                const float sc = is_v ? 1.f : scale;
                const uint32_t ta = tacc + acc * HD;
                if (!is_v) {
                    // a position outside the (cos, sin) table is reported
                    // and read as position 0 (no rotation)
                    int pr = rv ? pos[grow] : 0;
                    if (pr < 0 || pr >= rope_ld) {
                        if (rv) report(p.status, JNX_ERR_DEVICE_BOUNDS);
                        pr = 0;
                    }
#pragma unroll 1
                    for (int c = half; c < HD / 64; c += 2) {  // the two warps' chunks in turn
                        float2 cs[32];
                        if (rv) {
                            const float2* src = rope + (size_t)(c * 32) * rope_ld + pr;
#pragma unroll
                            for (int e = 0; e < 32; ++e) cs[e] = src[(size_t)e * rope_ld];
                        }
                        uint32_t lo[32], hi[32];
                        tmem_ld32(ta + c * 32, lo);
                        tmem_ld32(ta + HD / 2 + c * 32, hi);
                        tmem_ld_wait();
                        if (rv) {
                            uint32_t plo[16], phi[16];
#pragma unroll
                            for (int e = 0; e < 32; e += 2) {
                                float x[2], y[2];
#pragma unroll
                                for (int u = 0; u < 2; ++u) {
                                    const float a0 = sc * __uint_as_float(lo[e + u]);
                                    const float b0 = sc * __uint_as_float(hi[e + u]);
                                    x[u] = a0 * cs[e + u].x + b0 * cs[e + u].y;
                                    y[u] = b0 * cs[e + u].x - a0 * cs[e + u].y;
                                }
                                plo[e / 2] = pack_bf2(x[0], x[1]);
                                phi[e / 2] = pack_bf2(y[0], y[1]);
                            }
                            uint4* olo = reinterpret_cast<uint4*>(dqkv + (size_t)grow * ldq + colo + c * 32);
                            uint4* ohi = reinterpret_cast<uint4*>(dqkv + (size_t)grow * ldq + colo +
                                                                  HD / 2 + c * 32);
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                olo[u] = make_uint4(plo[4 * u], plo[4 * u + 1], plo[4 * u + 2], plo[4 * u + 3]);
                                ohi[u] = make_uint4(phi[4 * u], phi[4 * u + 1], phi[4 * u + 2], phi[4 * u + 3]);
                            }
                        }
                    }
                } else {
#pragma unroll 1
                    for (int c = half; c < HD / 32; c += 2) {
                        uint32_t v[32];
                        tmem_ld32(ta + c * 32, v);
                        tmem_ld_wait();
                        if (rv) {
                            uint4* o = reinterpret_cast<uint4*>(dqkv + (size_t)grow * ldq + colo + c * 32);
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                o[u] = make_uint4(pack_bf2(__uint_as_float(v[8 * u]), __uint_as_float(v[8 * u + 1])),
                                                  pack_bf2(__uint_as_float(v[8 * u + 2]), __uint_as_float(v[8 * u + 3])),
                                                  pack_bf2(__uint_as_float(v[8 * u + 4]), __uint_as_float(v[8 * u + 5])),
                                                  pack_bf2(__uint_as_float(v[8 * u + 6]), __uint_as_float(v[8 * u + 7])));
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (elect_one()) mbar_arrive(acc_free);
            __syncwarp();
            ++items_done;
        }
        if (!ok) *fail_flag = 1;
    }
    return claim;
}

template <int HD>
__global__ void __launch_bounds__(64 + 32 * abwd::EW, 1)
    k_attn_bwd(const __grid_constant__ CUtensorMap t_qkv_o, const __grid_constant__ CUtensorMap t_qkv_i,
               const __grid_constant__ CUtensorMap t_do_o, const __grid_constant__ CUtensorMap t_do_i,
               const __grid_constant__ BwdArgs p) {
    using P = AttnBwdPasses<HD>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + P::OFF_BAR);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + P::N * abwd::kBars);
    volatile int* fail_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);  // then the slots

    const int warp = warp_uniform(threadIdx.x >> 5);
    if (threadIdx.x == 0) {
        for (int k = 0; k < P::N * abwd::kBars; ++k) {
            const int i = k % abwd::kBars;
            mbar_init(&bars[k], i == 14 || i == 15 || i == 17 ? abwd::EW
                                : i >= 25                     ? abwd::EW + 1
                                : i >= 19 && i < 23           ? 2
                                                              : 1);
        }
        *fail_flag = 0;
        fence_barrier_init();
        fence_proxy_async();
    }
    pdl_entry();  // TMEM is taken once the grid ahead has given its own back
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = warp_uniform(*tmem_slot);

    // A pass leaves no copy, MMA or TMEM read of its own behind, so the next may
    // reuse the buffers; its barriers are its own.
    const int nk = p.items.n * p.Hkv;
    bool failed;
    auto end_pass = [&]() {
        __syncwarp();
        tc_fence_before();
        failed = __syncthreads_or(*fail_flag);
        tc_fence_after();
    };
    int claim = blockIdx.x, q0 = 0;
    claim = bwd_pass<HD, P::KEY>(t_qkv_o, t_qkv_i, t_do_o, t_do_i, p, sm, bars, fail_flag, tbase,
                                 q0, claim);
    q0 += nk;
    bars += abwd::kBars;
    end_pass();
    if constexpr (HD == 256) {
        if (!failed) {
            claim = bwd_pass<HD, abwd::DV>(t_qkv_o, t_qkv_i, t_do_o, t_do_i, p, sm, bars, fail_flag,
                                           tbase, q0, claim);
            q0 += nk;
            bars += abwd::kBars;
            end_pass();
        }
    }
    if (!failed) {
        bwd_pass<HD, abwd::DQ>(t_qkv_o, t_qkv_i, t_do_o, t_do_i, p, sm, bars, fail_flag, tbase, q0,
                               claim);
        end_pass();
    }
    if (failed && threadIdx.x == 0) report(p.status, JNX_ERR_TIMEOUT);
    if (warp == 1) tmem_dealloc(tbase, 512);
}

template <int HD>
static jnx_status launch_bwd(const CUtensorMap (&maps)[4], BwdArgs p, cudaStream_t s) {
    constexpr int smem = AttnBwdPasses<HD>::SMEM;
    static std::atomic<uint64_t> attr{0};
    if (set_smem_limit(reinterpret_cast<const void*>(k_attn_bwd<HD>), smem, attr) != cudaSuccess)
        return fail(JNX_ERR_CUDA, "attention backward: smem attribute");
    const int key_passes = AttnBwdPasses<HD>::N - 1;
    const long long n_work = (long long)p.items.n * (key_passes * p.Hkv + p.H);
    // (claims run past the last item by one for each CTA)
    if (n_work > 0x7FFFFFFFLL - 2 * num_sms())
        return fail(JNX_ERR_UNSUPPORTED, "attention backward: too many items");
    const int grid = (int)std::min<long long>(n_work, num_sms());
    p.scale_log2 = (float)(1.4426950408889634 / sqrt((double)HD));
    p.scale = (float)(1.0 / sqrt((double)HD));
    if (cudaMemsetAsync(p.items.claimed, 0, sizeof(int), s) != cudaSuccess)
        return fail(JNX_ERR_CUDA, "attention backward: %s", cudaGetErrorString(cudaGetLastError()));
    pdl(k_attn_bwd<HD>, grid, 64 + 32 * abwd::EW, smem, s)(maps[0], maps[1], maps[2], maps[3], p);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? JNX_OK
                            : fail(JNX_ERR_CUDA, "attention backward: %s", cudaGetErrorString(e));
}

jnx_status attention_bwd_launch(const uint16_t* qkv, int ldq, const uint16_t* dO, const float* lse,
                                const float* D, int n_tokens, int H, int Hkv, int hd,
                                const int* cu, const int* pos, const float2* rope, int rope_ld,
                                const int2* items, int n_items, int* claimed, uint16_t* dqkv,
                                int* status, cudaStream_t s) {
    if (n_tokens == 0 || n_items == 0) return JNX_OK;
    if (!items || !claimed) return fail(JNX_ERR_INVALID_ARG, "attention backward: null work items");
    if (Hkv <= 0 || H % Hkv) return fail(JNX_ERR_UNSUPPORTED, "attention backward: H %% Hkv != 0");
    if (ldq != (H + 2 * Hkv) * hd)
        return fail(JNX_ERR_INVALID_ARG, "attention backward: q|k|v row stride");
    CUtensorMap maps[4];
    if (!make_tmap_bf16(&maps[0], qkv, n_tokens, ldq, ldq, abwd::BM, 64) ||
        !make_tmap_bf16(&maps[1], qkv, n_tokens, ldq, ldq, abwd::BN, 64) ||
        !make_tmap_bf16(&maps[2], dO, n_tokens, (uint64_t)H * hd, (uint64_t)H * hd, abwd::BM, 64) ||
        !make_tmap_bf16(&maps[3], dO, n_tokens, (uint64_t)H * hd, (uint64_t)H * hd, abwd::BN, 64))
        return fail(JNX_ERR_CUDA, "attention backward: tensor map encode failed");
    const BwdArgs p{cu, {items, n_items, claimed}, H, Hkv, 0.f, 0.f, lse, D, pos, rope, rope_ld,
                    dqkv, ldq, status};
    switch (hd) {
        case 64: return launch_bwd<64>(maps, p, s);
        case 128: return launch_bwd<128>(maps, p, s);
        case 256: return launch_bwd<256>(maps, p, s);
        default:
            return fail(JNX_ERR_UNSUPPORTED, "attention backward: head_dim %d", hd);
    }
}

}  // namespace jnx
