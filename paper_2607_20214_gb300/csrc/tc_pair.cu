// Block attention for key blocks of 256 (b = 256, d_h = 128, gamma = 4) on
// CTA pairs: the sortLSH block step (Algorithm "sortLSH Sparse Exact
// Attention Branch"), the RACE readout (Algorithm "RACE Low-Rank Attention
// Branch" steps 9-10) and the fusion of Eq. (5)-(6), the same arithmetic as
// the one-CTA kernel of tc_ws.cu.
//
// The two 128-query tiles of one sorted block attend the same 256 keys, so
// a cluster of two CTAs on neighbouring SMs takes one block at a time: the
// even CTA the block's first 128 queries, the odd CTA the other 128. Every
// product is one cta_group::2 MMA (M = 256: each CTA's 128 query rows in its
// own tensor memory) whose B operand is split by columns between the CTAs:
//   scores   S = Q [K; W]^T: each CTA gathers 64 of the pass's 128 keys and
//            holds 32 of the 64 RACE plane rows (its row half's tables);
//   P V:     each CTA gathers its 64 of the 128 value columns;
//   Phi' B:  each CTA holds its 64 columns of the bf16 B summary.
// So each SM gathers half a block's keys and values instead of all of them,
// and the freed shared memory double-buffers the query tile and holds one
// key and one value buffer per pass.
//
// Roles (768 threads per CTA, as in the one-CTA kernel): warps 0-15 compute
// (two TMEM slots of 256 columns, slot g takes the CTA's blocks of local
// index = g mod 2; within a slot warps w and w + 4 split each row's keys,
// tables and output columns in halves and meet at a barrier of their 64
// threads), warp 16 issues every MMA in the even CTA and relays the odd
// CTA's readiness to it, warp 17 loads the per-head planes and summaries
// with TMA, warps 18-19 gather values, warps 20-23 queries and keys.
//
// What bounds it: the slots' own chain of hand-offs (the two slots' work is
// about a third of the issue slots and the products about a quarter of the
// tensor pipe's), so everything that another slot or pass can cover is off
// that chain: gathers have warps of their own, the two slots' products are
// issued as they become ready (block by block at each stage: pair_order.h),
// P is handed over before the features and the fusion scalars are computed,
// and all features go to one product: c4
// (B1 H32 N65536 d128 L16) 697 -> 646 us; products issued by a converged warp
// from descriptors made once, and a lane per relayed barrier: 587 us (0.54 of
// the measured HBM bandwidth).
//
// TMEM columns of a slot (same layout in both CTAs): pass 0 scores keys
// [0, 64) at [0, 64), the projections of row half 0's tables at [64, 96),
// keys [64, 128) at [96, 160), row half 1's projections at [160, 192);
// pass 1 scores keys [0, 64) at [0, 64), keys [64, 128) at [64, 128); P of
// row half h in quarter 2h ([64h, 64h + 32)); the output accumulator at
// [128, 256); the pre-scaled features of buckets [0, 128) at [32, 64) and
// [96, 128), those of buckets [128, 256) over P once P V is complete.
//
// Every hand-off is an mbarrier with a bounded wait; the odd CTA's
// arrivals reach the even CTA's barriers through the relay (one remote
// arrival per phase), the MMA completions reach both CTAs by multicast.
#include "device_common.cuh"
#include "pair_order.h"
#include "tc_common.cuh"
#include "tc_race.cuh"

namespace elsaa {

namespace {

using namespace tc;

constexpr int kPrThreads = 768;
constexpr int kPrMmaWarp = 16;
constexpr int kPrVWarp = 18;   // 2 warps
constexpr int kPrQkWarp = 20;  // 4 warps
constexpr int kPrVThreads = 64, kPrQkThreads = 128;
// registers: 16 compute warps and 8 others share the launch's 80 a thread
constexpr int kPrRegsCompute = 96, kPrRegsOther = 48;
static_assert(512 * kPrRegsCompute + 256 * kPrRegsOther <= kPrThreads * 80,
              "register shares exceed what the block is launched with");
constexpr int kPrNK = 128;   // keys per pass, query rows per CTA
constexpr int kPrNP = 2;     // passes per block (b = 256)
constexpr int kPrD = 128;    // head dimension
constexpr int kPrKRows0 = 96;  // pass-0 key buffer: 64 keys + 32 plane rows
constexpr int kPrKRows1 = 64;  // pass-1 key buffer: 64 keys

struct PrBars {
    // copies, relayed: the even CTA's copy also counts the odd CTA's phase
    uint64_t q_full[2], k_full[kPrNP], v_full[kPrNP], wb_full;
    // compute hand-offs: one arrival per warp of the slot in both CTAs
    uint64_t tmem_empty[2], p_full[2], phi_full[2];
    // MMA completions, committed to both CTAs
    uint64_t q_empty[2], k_empty[kPrNP], v_empty[kPrNP];
    uint64_t s_full[2], pv0_done[2], pv_done[2], o_full[2], head_done;
};
constexpr int kPrRelayed = 2 + kPrNP + kPrNP + 1;  // copy barriers

template <bool O32>
__global__ void __launch_bounds__(kPrThreads, 1)
    k_block_attn_pair(const uint16_t *__restrict__ qx,
                      const uint16_t *__restrict__ kx,
                      const uint16_t *__restrict__ vx,
                      const __grid_constant__ CUtensorMap tmW,
                      const __grid_constant__ CUtensorMap tmB,
                      const int32_t *__restrict__ perm_q,
                      const int32_t *__restrict__ perm_k,
                      const float *__restrict__ Ag,
                      const float *__restrict__ lambda_tok,
                      const float *__restrict__ gates,
                      uint16_t *__restrict__ ox, float *__restrict__ o32,
                      float *__restrict__ log_ds_out,
                      float *__restrict__ dlr_out, float *__restrict__ m_out,
                      int N, int H, int L, int Lg_pad, float beta, float eps,
                      float scale, float lambda, int mode, int blocks_per_head,
                      long total_blocks, DeviceStatus *status) {
    constexpr int G = 4, R = 16, nk = kPrNK, d = kPrD, NP = kPrNP;
    extern __shared__ unsigned char smem_raw[];
    __shared__ PrBars bars;
    __shared__ uint32_t tbase;
    __shared__ int abort_flag;
    __shared__ float xmax[kPrNP][2][2][128];  // by pass
    __shared__ float2 xsum[2][2][128];        // partial sums, Den
    volatile int *abort = &abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane_id = tid & 31;
    const uint32_t crank = cluster_rank();  // 0: issues the MMAs
    const bool leader = crank == 0;
    const int r = L * R;
    const long pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const long b_begin = total_blocks * pair / npairs;
    const long b_end = total_blocks * (pair + 1) / npairs;
    const int nblk = (int)(b_end - b_begin);
    const int bb = (int)b_begin;  // block indices fit in int (host check)
    auto blk_head = [=](int j) { return (bb + j) / blocks_per_head; };
    // sorted position of this CTA's first query of block j
    auto blk_pos = [=](int j) {
        return (bb + j) % blocks_per_head * 256;
    };
    auto new_head = [=](int j) {
        return j == 0 || (bb + j) % blocks_per_head == 0;
    };
    auto last_of_head = [=](int j) {
        return j == nblk - 1 || (bb + j + 1) % blocks_per_head == 0;
    };

    // shared memory: two query tiles, the pass-0 key buffer (64 keys and
    // this CTA's 32 plane rows), the pass-1 key buffer, one value buffer per
    // pass (128 keys x this CTA's 64 columns), this CTA's 64 columns of the
    // B summary, the A summary, 2 KB per compute warp for output rows
    const uint32_t tileQ = (uint32_t)nk * d * 2u;
    const uint32_t base = align1k(smem_u32(smem_raw));
    const uint32_t sQ = base;
    const uint32_t sK0 = sQ + 2 * tileQ;
    const uint32_t sK1 = sK0 + kPrKRows0 * d * 2;
    const uint32_t sV = sK1 + kPrKRows1 * d * 2;
    const uint32_t sB = sV + NP * 16384u;
    const uint32_t sA = sB + align1k((uint32_t)r * 128u);
    const uint32_t sO = sA + align1k((uint32_t)r * 4u);
    const float *Asm = reinterpret_cast<const float *>(
        smem_raw + (sA - smem_u32(smem_raw)));
    auto kbuf = [=](int p) { return p == 0 ? sK0 : sK1; };
    auto krows = [=](int p) { return p == 0 ? kPrKRows0 : kPrKRows1; };

    if (warp == kPrMmaWarp) tmem_alloc_pair(&tbase, 512);
    if (tid == 0) {
        const uint32_t x = leader ? 1u : 0u;  // the relayed odd-CTA phase
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars.q_full[s], kPrQkThreads + x);
            mbar_init(&bars.q_empty[s], 1);
            mbar_init(&bars.tmem_empty[s], 16);
            mbar_init(&bars.p_full[s], 16);
            mbar_init(&bars.phi_full[s], 16);
            mbar_init(&bars.s_full[s], 1);
            mbar_init(&bars.pv0_done[s], 1);
            mbar_init(&bars.pv_done[s], 1);
            mbar_init(&bars.o_full[s], 1);
        }
        for (int p = 0; p < NP; ++p) {
            mbar_init(&bars.k_full[p], kPrQkThreads + x);
            mbar_init(&bars.k_empty[p], 1);
            mbar_init(&bars.v_full[p], kPrVThreads + x);
            mbar_init(&bars.v_empty[p], 1);
        }
        mbar_init(&bars.wb_full, 1 + x);
        mbar_init(&bars.head_done, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers exist before any remote arrival
    tc_fence_after();
    const uint32_t tm = tbase;

    // global row number of sorted position pos of one head (rowbase = its
    // first row); an entry outside [0, N) is read as row 0 (the orders come
    // from the sort); the checked build records it
    auto global_row = [=](const int32_t *pm, int bh, int pos) {
        int v = pm[(size_t)bh * N + pos];  // pos < N: N is a multiple of 256
        if (v < 0 || v >= N) {
#ifdef ELSAA_CHECKED
            report(status, kDevPermRange, 14, bh, v);
#endif
            v = 0;
        }
        return bh * N + v;
    };

    if (warp >= kPrMmaWarp)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(
            kPrRegsOther));
    if (warp > kPrMmaWarp) {
        // ------------------------------------------------------------ loaders
        const int lt = lane_id;
        auto lwait = [=](uint64_t *bar, uint32_t par, int site) {
            return __all_sync(0xffffffffu,
                              mbar_wait_or_abort(bar, par, abort, status,
                                                 site));
        };
        if (warp >= kPrQkWarp) {
            // queries and keys: per block this warp's 32 of the CTA's 128
            // queries and, per pass, 16 of the CTA's 64 keys, two rows an
            // instruction; lane l holds the number of query row l and of
            // key l & 15 of pass l >> 4
            const int w = warp - kPrQkWarp;
            const int sub = lt >> 4, ch = lt & 15;
            int qn = 0, kn = 0;  // of the next block
            auto ahead = [&](int j) {
                const int bh = blk_head(j), pos = blk_pos(j);
                qn = global_row(perm_q, bh, pos + 128 * (int)crank + 32 * w +
                                                lt);
                kn = global_row(perm_k, bh,
                                pos + 128 * (lt >> 4) + 64 * (int)crank +
                                    16 * w + (lt & 15));
            };
            auto gather_k = [&](int p, int rows) {
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    const int rn =
                        __shfl_sync(0xffffffffu, rows, 16 * p + i + sub);
                    cp_async16(kbuf(p) + panel_offset(16 * w + i + sub, ch,
                                                      krows(p)),
                               kx + (size_t)rn * d + ch * 8);
                }
                cp_async_mbar_arrive(&bars.k_full[p]);
            };
            if (nblk > 0) ahead(0);
            for (int j = 0; j < nblk; ++j) {
                const int qr = qn, kr = kn, s = j & 1;
                if (j + 1 < nblk) ahead(j + 1);
                if (j >= 1 && !lwait(&bars.k_empty[0], (j - 1) & 1, 70)) break;
                gather_k(0, kr);
                if (j >= 2 &&
                    !lwait(&bars.q_empty[s], ((j >> 1) - 1) & 1, 75))
                    break;
#pragma unroll 4
                for (int i = 0; i < 32; i += 2) {
                    const int rn = __shfl_sync(0xffffffffu, qr, i + sub);
                    cp_async16(sQ + s * tileQ +
                                   panel_offset(32 * w + i + sub, ch, nk),
                               qx + (size_t)rn * d + ch * 8);
                }
                cp_async_mbar_arrive(&bars.q_full[s]);
                if (j >= 1 && !lwait(&bars.k_empty[1], (j - 1) & 1, 76)) break;
                gather_k(1, kr);
            }
            cp_async_wait<0>();
        } else if (warp == kPrMmaWarp + 1) {
            // per head, TMA: this CTA's 32 plane rows (its row half's tables:
            // rows [16 c, 16 c + 16) and [32 + 16 c, 48 + 16 c) of the head's
            // planes) under the pass-0 keys, its 64 columns of the B summary,
            // the A summary
            int hc = 0;
            for (int j = 0; j < nblk; ++j) {
                if (!new_head(j)) continue;
                const int bh = blk_head(j);
                if (j > 0 && !lwait(&bars.head_done, (hc - 1) & 1, 71)) break;
                if (lt == 0) {
                    mbar_expect_tx(&bars.wb_full,
                                   32u * d * 2u + (uint32_t)r * 128u +
                                       (uint32_t)r * 4u);
                    const int w0 = (bh % H) * Lg_pad + 16 * (int)crank;
                    for (int pn = 0; pn < d / 64; ++pn) {
                        const uint32_t dst = sK0 + pn * kPrKRows0 * 128;
                        tma_load_2d(dst + 64 * 128, &tmW, 64 * pn, w0,
                                    &bars.wb_full);
                        tma_load_2d(dst + 80 * 128, &tmW, 64 * pn, w0 + 32,
                                    &bars.wb_full);
                    }
                    tma_load_2d(sB, &tmB, 64 * (int)crank, bh * r,
                                &bars.wb_full);
                    bulk_load(sA, Ag + (size_t)bh * r, (uint32_t)r * 4u,
                              &bars.wb_full);
                }
                __syncwarp();
                ++hc;
            }
        } else {
            // values: for each pass, this warp's 64 of the pass's 128 keys,
            // this CTA's 64 columns (128 bytes of each row, four rows an
            // instruction) into the pass's buffer once the previous block's
            // P V product of that pass is done
            const int r0 = 64 * (warp - kPrVWarp);
            const int sub = lt >> 3, ch = lt & 7;
            int n0 = 0, n1 = 0;  // of the next unit
            auto ahead = [&](int u) {
                const int j = u / NP;
                const int bh = blk_head(j);
                const int pos = blk_pos(j) + 128 * (u - j * NP) + r0 + lt;
                n0 = global_row(perm_k, bh, pos);
                n1 = global_row(perm_k, bh, pos + 32);
            };
            if (nblk > 0) ahead(0);
            for (int u = 0; u < nblk * NP; ++u) {
                const int a0 = n0, a1 = n1, j = u / NP, p = u - j * NP;
                if (u + 1 < nblk * NP) ahead(u + 1);
                if (j >= 1 && !lwait(&bars.v_empty[p], (j - 1) & 1, 72)) break;
                const uint32_t dst = sV + p * 16384u;
#pragma unroll 4
                for (int i = 0; i < 64; i += 4) {
                    const int rn = __shfl_sync(0xffffffffu, i < 32 ? a0 : a1,
                                               (i + sub) & 31);
                    cp_async16(dst + panel_offset(r0 + i + sub, ch, nk),
                               vx + (size_t)rn * d + 64 * (int)crank +
                                   ch * 8);
                }
                cp_async_mbar_arrive(&bars.v_full[p]);
            }
            cp_async_wait<0>();
        }
    } else if (warp == kPrMmaWarp) {
        if (!leader) {
            // ------------------------------------------------------ relay
            // Each phase of this CTA's copy barriers (cp.async and TMA
            // completions, which can only arrive locally) completes here
            // first, then counts once more on the even CTA's copy. A phase
            // cannot complete twice before it is relayed: the next one needs
            // MMAs that wait for this relay.
            // One lane per barrier.
            static_assert(kPrRelayed == 2 + 2 * kPrNP + 1, "lane order below");
            uint64_t *bar = &bars.wb_full;
            int want = 0, done = 0;
            if (lane_id < 2) {
                bar = &bars.q_full[lane_id];
                want = (nblk + 1 - lane_id) / 2;
            } else if (lane_id < 2 + NP) {
                bar = &bars.k_full[lane_id - 2];
                want = nblk;
            } else if (lane_id < 2 + 2 * NP) {
                bar = &bars.v_full[lane_id - 2 - NP];
                want = nblk;
            } else if (lane_id == 2 + 2 * NP) {
                for (int j = 0; j < nblk; ++j) want += new_head(j) ? 1 : 0;
            }
            unsigned long long t_last = global_ns();
            uint32_t idle = 0;  // the clock is read every 256 idle rounds
            while (__any_sync(0xffffffffu, done < want)) {
                const bool hit =
                    done < want && mbar_test(bar, (uint32_t)done & 1u);
                if (hit) {
                    // this CTA's cp.async data -> the pair's MMAs
                    fence_proxy_async_smem();
                    mbar_arrive_remote(bar, 0);
                    ++done;
                }
                if (__any_sync(0xffffffffu, hit)) {
                    idle = 0;
                } else if ((++idle & 255u) == 0) {
                    if (idle == 256) t_last = global_ns();
                    const bool late = global_ns() - t_last > kWaitLimitNs;
                    if (late) {
                        *abort = 1;
                        record_timeout(status, 73);
                    }
                    if (__any_sync(0xffffffffu, late || *abort)) break;
                }
            }
        } else if (nblk > 0) {
            // ------------------------------------------------- MMA issue
            // Event driven, each slot at a stage of its own: the order is
            // PairOrder's (pair_order.h). A new head's planes and summaries
            // replace the old ones only after head_done: its first scores
            // wait until every product of the blocks before is issued.
            const uint32_t id_sp = idesc_bf16(256, nk + 64, false, false);
            const uint32_t id_s = idesc_bf16(256, nk, false, false);
            const uint32_t id_o = idesc_bf16(256, d, false, true);
            // The whole warp runs the loop, so that its state and the
            // operands' descriptors are warp-uniform; one lane issues.
            const bool el = elect_one();
            auto test = [&](PairBar bar, int i, uint32_t par) -> bool {
                uint64_t *b = bar == PairBar::k_full       ? &bars.k_full[i]
                              : bar == PairBar::q_full     ? &bars.q_full[i]
                              : bar == PairBar::v_full     ? &bars.v_full[i]
                              : bar == PairBar::pv0_done   ? &bars.pv0_done[i]
                              : bar == PairBar::tmem_empty ? &bars.tmem_empty[i]
                              : bar == PairBar::p_full     ? &bars.p_full[i]
                              : bar == PairBar::phi_full   ? &bars.phi_full[i]
                                                           : &bars.wb_full;
                return __all_sync(0xffffffffu, mbar_test(b, par));
            };
            const uint64_t dQ = smem_desc(sQ, 16, 1024),
                           dK0 = smem_desc(sK0, 16, 1024),
                           dK1 = smem_desc(sK1, 16, 1024),
                           dV = smem_desc(sV, (uint32_t)nk * 128, 1024),
                           dB = smem_desc(sB, (uint32_t)r * 128, 1024);
            auto scores = [&](int s, int p) {
                fence_proxy_async_smem();  // cp.async data -> MMA
                tc_fence_after();
                const uint32_t so = tm + 256u * s;
                const uint64_t a = desc_at(dQ, s * tileQ);
                if (el) {
                    // pass 0: scores and projections (N = 192); pass 1:
                    // scores only
                    if (p == 0) {
#pragma unroll
                        for (int kk = 0; kk < d / 16; ++kk)
                            mma_pair_ss(
                                so,
                                desc_at(a, (kk >> 2) * 16384 + (kk & 3) * 32),
                                desc_at(dK0, (kk >> 2) * kPrKRows0 * 128 +
                                                 (kk & 3) * 32),
                                id_sp, kk > 0);
                    } else {
#pragma unroll
                        for (int kk = 0; kk < d / 16; ++kk)
                            mma_pair_ss(
                                so,
                                desc_at(a, (kk >> 2) * 16384 + (kk & 3) * 32),
                                desc_at(dK1, (kk >> 2) * kPrKRows1 * 128 +
                                                 (kk & 3) * 32),
                                id_s, kk > 0);
                    }
                    mma_commit_pair(&bars.s_full[s]);
                    mma_commit_pair(&bars.k_empty[p]);
                    if (p == NP - 1) mma_commit_pair(&bars.q_empty[s]);
                }
            };
            auto values = [&](int s, int p) {  // O (+)= P V
                fence_proxy_async_smem();
                tc_fence_after();
                const uint32_t so = tm + 256u * s;
                const uint64_t b = desc_at(dV, p * 16384u);
                if (el) {
#pragma unroll
                    for (int kk = 0; kk < nk / 16; ++kk)
                        mma_pair_ts(so + nk, so + quarter_col(kk, 0),
                                    desc_at(b, kk * 2048), id_o,
                                    p > 0 || kk > 0);
                    mma_commit_pair(&bars.v_empty[p]);
                    mma_commit_pair(p == 0 ? &bars.pv0_done[s]
                                           : &bars.pv_done[s]);
                }
            };
            auto features = [&](int s, int n) {  // O += Phi' B
                tc_fence_after();
                const uint32_t so = tm + 256u * s;
                if (el) {
#pragma unroll
                    for (int kk = 0; kk < 16; ++kk)
                        if (16 * kk < r)
                            mma_pair_ts(so + nk,
                                        so + (kk < 8 ? quarter_col(kk, 32)
                                                     : quarter_col(kk - 8, 0)),
                                        desc_at(dB, kk * 2048), id_o, 1);
                    mma_commit_pair(&bars.o_full[s]);
                    if (last_of_head(n)) mma_commit_pair(&bars.head_done);
                }
            };
            PairOrder order;
            unsigned long long t_last = global_ns();
            uint32_t idle = 0;  // the clock is read every 256 idle rounds
            while (order.done < nblk) {
                const bool did = order.round(nblk, new_head, test, scores,
                                             values, features);
                if (did) {
                    idle = 0;
                } else if ((++idle & 255u) == 0) {
                    if (idle == 256) t_last = global_ns();
                    const bool late = global_ns() - t_last > kWaitLimitNs;
                    if (late) {
                        *abort = 1;
                        record_timeout(status, 74);
                    }
                    if (__any_sync(0xffffffffu, late || *abort)) break;
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------ compute groups
        // warps 0-7: slot 0, warps 8-15: slot 1; within a slot, warps
        // (w, w + 4) share TMEM lanes and split each row in two halves: half
        // h takes keys [64 h, 64 h + 64) of each pass (the keys this CTA's
        // half of the pair gathered when h equals its rank), the tables of
        // the 64-bucket chunks h and h + 2 and output columns [64 h, 64 h +
        // 64).
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(
            kPrRegsCompute));
        const int g = warp >> 3;
        const int half = (warp >> 2) & 1;
        const int row = (warp & 3) * 32 + lane_id;  // query row = TMEM lane
        const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
        constexpr int T = 64 / R;  // tables per 64-bucket chunk
        const int ta0 = min(half * T, L), nt0 = min(ta0 + T, L) - ta0;
        const int ta1 = min((half + 2) * T, L), nt1 = min(ta1 + T, L) - ta1;
        const uint32_t cb0 = half ? 96u : 32u, cb1 = half ? 64u : 0u;
        const float sl2e = scale * kLog2e;
        // barrier of the row's two warps; a pair's 64 threads leave a wait
        // with one verdict (an abort seen by one warp only would strand the
        // other there)
        const int pid = 1 + g * 4 + (warp & 3);
        auto pwait = [=](uint64_t *bar, uint32_t par, int site) {
            const bool ok = mbar_wait_or_abort(bar, par, abort, status, site);
            return named_sync_and(pid, 64, ok);
        };
        // a hand-off to the MMA issuer: once per warp, on the even CTA's
        // barrier
        auto signal = [&](uint64_t *bar) {
            tc_fence_before();
            __syncwarp();
            if (lane_id == 0) {
                if (leader)
                    mbar_arrive(bar);
                else
                    mbar_arrive_remote(bar, 0);
            }
        };
        for (int j = g; j < nblk; j += 2) {
            const int k = j >> 1;
            const uint32_t so = tm + 256u * g + lane;
            const int bh = blk_head(j);
            const int qpos = blk_pos(j) + 128 * (int)crank + row;
            int qi = perm_q[(size_t)bh * N + qpos];  // prefetch
            if (!pwait(&bars.s_full[g], 0, 77)) break;
            // the A summary came by TMA: acquire its head's stage (complete
            // already: this block's scores waited for it)
            if ((j < 2 || blk_head(j) != blk_head(j - 2)) &&
                !pwait(&bars.wb_full, (bh - blk_head(0)) & 1, 78))
                break;
            tc_fence_after();
            // row maximum of both halves (an array per pass: pass 1 writes
            // its own while the other half may still read pass 0's)
            auto row_max = [&](int ps, const float (&m)[4]) {
                xmax[ps][g][half][row] =
                    fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
                named_sync(pid, 64);
                return fmaxf(xmax[ps][g][0][row], xmax[ps][g][1][row]);
            };
            // maximum over this half's 64 scores at column c0
            auto max64 = [&](uint32_t c0, float (&m)[4]) {
#pragma unroll
                for (int c = 0; c < 64; c += 16) {
                    uint32_t v[16];
                    tmem_ld16(so + c0 + c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 16; q += 2)
                        m[(q >> 1) & 3] =
                            max3(m[(q >> 1) & 3], __uint_as_float(v[q]),
                                 __uint_as_float(v[q + 1]));
                }
            };
            // P of this half's 64 scores at column c0, into quarter 2 half
            // (behind scores already read); returns its row sum
            const uint32_t pc = 64u * half;
            auto exp64 = [&](uint32_t c0, float M) -> float {
                const float2 sl2 = make_float2(sl2e, sl2e),
                             mn = make_float2(-M, -M);
                float2 ls[2] = {make_float2(0.0f, 0.0f),
                                make_float2(0.0f, 0.0f)};
#pragma unroll
                for (int c = 0; c < 64; c += 32) {
                    uint32_t v[32], pw[16];
                    tmem_ld32(so + c0 + c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 32; q += 2) {
                        const float2 z =
                            fma2(make_float2(__uint_as_float(v[q]),
                                             __uint_as_float(v[q + 1])),
                                 sl2, mn);
                        const float2 e =
                            make_float2(ex2_approx(z.x), ex2_approx(z.y));
                        ls[(q >> 1) & 1] = add2(ls[(q >> 1) & 1], e);
                        pw[q >> 1] = pack_bf16x2(e.x, e.y);
                    }
                    tmem_st16(so + pc + (c >> 1), pw);
                }
                return (ls[0].x + ls[1].x) + (ls[0].y + ls[1].y);
            };
            // pass 0. This half's raw projections are read first (P and the
            // output accumulator go over them), its 64 scores start at 96 h
            uint32_t pr[32];
            const uint32_t pcol = 64u + 96u * half;
            tmem_ld16(so + pcol, *reinterpret_cast<uint32_t(*)[16]>(pr));
            tmem_ld16(so + pcol + 16,
                      *reinterpret_cast<uint32_t(*)[16]>(pr + 16));
            const uint32_t kc0 = 96u * half;
            float mxa[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            max64(kc0, mxa);
            float M2 = row_max(0, mxa) * sl2e;
            float lsum = exp64(kc0, M2);  // this half's
            tmem_wait_st();
            signal(&bars.p_full[g]);
            // per-bit factors of this half's tables (sp[0, 16): chunk half,
            // sp[16, 32): chunk half + 2) and its part of Den, while pass
            // 0's P V product and pass 1's scores run. The second chunk's
            // factors wait for the last P V product: kept as fp16 pairs
            // (factors lie in (0.11, 0.89); relative rounding 2^-11, below
            // the bf16 rounding of the features they make)
            qi = (qi < 0 || qi >= N) ? 0 : qi;
            const size_t tok = (size_t)bh * N + qi;
            const float lam = lambda_tok ? lambda_tok[tok] : lambda;
            const float gs = gates ? gates[2 * tok] : 1.0f;
            const float gl = gates ? gates[2 * tok + 1] : 1.0f;
            float sp[16];
            uint32_t sp1[8];
            float den;
            {
                float dacc[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // independent chains
                if (nt1 > 0) {
                    float s1[16];
                    race_factors<16>(pr + 16, beta, s1);
                    chunk_den<G, T>(s1, nt1, Asm + ta1 * R, dacc);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        sp1[q] = pack_f16x2(s1[2 * q], s1[2 * q + 1]);
                }
                race_factors<16>(pr, beta, sp);
                chunk_den<G, T>(sp, nt0, Asm + ta0 * R, dacc);
                den = (dacc[0] + dacc[1]) + (dacc[2] + dacc[3]);
            }
            // pass 1
            if (!pwait(&bars.s_full[g], 1, 79)) break;
            tc_fence_after();
            {
                float mxb[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                max64(pc, mxb);
                const float M2b = row_max(1, mxb) * sl2e;
                // online softmax: keep the running reference unless the
                // row's max grew by more than 2^8; then rescale the
                // accumulator (the previous P V product is complete: these
                // scores waited for it) and the running sum
                const bool need = M2b > M2 + 8.0f;
                const float f = need ? ex2_approx(M2 - M2b) : 1.0f;
                if (__any_sync(0xffffffffu, need)) {
#pragma unroll
                    for (int c = 0; c < 64; c += 16) {
                        uint32_t v[16];
                        tmem_ld16(so + nk + half * 64 + c, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            v[q] = __float_as_uint(__uint_as_float(v[q]) * f);
                        tmem_st16(so + nk + half * 64 + c, v);
                    }
                }
                if (need) {
                    lsum *= f;
                    M2 = M2b;
                }
                lsum += exp64(pc, M2);
            }
            tmem_wait_st();
            signal(&bars.p_full[g]);
            // fusion scalars (Eq. (5) in log-sum-exp form, Eq. (6))
            xsum[g][half][row] = make_float2(lsum, den);
            named_sync(pid, 64);
            {
                const float2 o = xsum[g][half ^ 1][row];
                lsum += o.x;
                den += o.y;
            }
            const float denf = den * (1.0f / (float)L);
            const float log_ds = M2 * kLn2 + __logf(lsum);
            const float msp =
                fusion_multiplier_fast(log_ds, lam, denf, eps, mode);
            const float c1 =
                __fdividef(gs * msp, lsum + eps * ex2_approx(-M2));
            const float c1e = fmaxf(c1, 1e-30f);
            const float ratio =
                __fdividef(gl, (float)L * (denf + eps) * c1e);
            if (nt0 > 0) write_phi_chunk<G, T>(sp, nt0, ratio, so + cb0);
            if (r > nk) {
                // over P: its product is complete
                if (!pwait(&bars.pv_done[g], k & 1, 110)) break;
                tc_fence_after();
                if (nt1 > 0) {
                    float f1[16];
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        unpack_f16x2(sp1[q], f1[2 * q], f1[2 * q + 1]);
                    write_phi_chunk<G, T>(f1, nt1, ratio, so + cb1);
                }
            }
            tmem_wait_st();
            signal(&bars.phi_full[g]);
            if (!pwait(&bars.o_full[g], k & 1, 111)) break;
            tc_fence_after();
            // O = c1 acc, this half's 64 columns: bf16 through this warp's
            // 2 KB, 16 rows at a time, out in 128-byte rows; fp32 from the
            // registers
            if constexpr (O32) {
#pragma unroll
                for (int c = 0; c < 64; c += 16) {
                    uint32_t v[16];
                    tmem_ld16(so + nk + half * 64 + c, v);
                    tmem_wait_ld();
                    float4 *dst = reinterpret_cast<float4 *>(
                        o32 + tok * (size_t)d + half * 64 + c);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        dst[q] = make_float4(c1e * __uint_as_float(v[4 * q]),
                                             c1e * __uint_as_float(v[4 * q + 1]),
                                             c1e * __uint_as_float(v[4 * q + 2]),
                                             c1e * __uint_as_float(v[4 * q + 3]));
                }
                signal(&bars.tmem_empty[g]);
            } else {
                uint32_t ob[32];
#pragma unroll
                for (int c = 0; c < 64; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(so + nk + half * 64 + c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const float2 x = mul2(
                            make_float2(c1e, c1e),
                            make_float2(__uint_as_float(v[2 * q]),
                                        __uint_as_float(v[2 * q + 1])));
                        ob[c / 2 + q] = pack_bf16x2(x.x, x.y);
                    }
                }
                signal(&bars.tmem_empty[g]);
                const uint32_t ow = sO + 2048u * warp;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    if ((lane_id >> 4) == hh) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            st_shared_v4(ow + (lane_id & 15) * 128 +
                                             ((q ^ (lane_id & 7)) << 4),
                                         ob[4 * q], ob[4 * q + 1],
                                         ob[4 * q + 2], ob[4 * q + 3]);
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int rl = 4 * i + (lane_id >> 3);
                        const int to = __shfl_sync(0xffffffffu, (int)tok,
                                                   16 * hh + rl);
                        const uint4 val = ld_shared_v4(
                            ow + rl * 128 +
                            (((lane_id & 7) ^ (rl & 7)) << 4));
                        *reinterpret_cast<uint4 *>(ox + (size_t)to * d +
                                                   half * 64 +
                                                   (lane_id & 7) * 8) = val;
                    }
                    __syncwarp();
                }
            }
            if (half == 0) {
                if (log_ds_out) log_ds_out[tok] = log_ds;
                if (dlr_out) dlr_out[tok] = denf;
                if (m_out) m_out[tok] = msp;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // no CTA leaves while the pair's MMAs may read it
    if (warp == kPrMmaWarp) tmem_dealloc_pair(tm, 512);
}

}  // namespace

bool pair_supported(const Plan &P) {
    const long rows = (long)P.N * P.BH;
    return tc_supported(P) && P.d == 128 && P.b == 256 && P.nb == 0 &&
           !P.sel && P.gamma == 4 && P.L <= 16 && P.N % 256 == 0 &&
           rows < (1L << 31);
}

size_t pair_smem(const Plan &P) {
    const size_t r = (size_t)P.r;
    return 1024 + 2 * (size_t)kPrNK * kPrD * 2 +
           (size_t)(kPrKRows0 + kPrKRows1) * kPrD * 2 + kPrNP * 16384 +
           (r * 128 + 1023) / 1024 * 1024 + (r * 4 + 1023) / 1024 * 1024 +
           16 * 2048;
}

cudaError_t launch_block_attn_pair(
    const Plan &P, const void *q, const void *k, const void *v,
    const uint16_t *w_bf16, const int32_t *perm_q, const int32_t *perm_k,
    const float *A, const uint16_t *Bh, const float *lambda_tok,
    const float *gates, void *o, float *log_d_sparse, float *d_lr,
    float *m_sparse, DeviceStatus *status, cudaStream_t st) {
    const size_t smem = pair_smem(P);
    const int bph = P.N / 256;
    const long total = (long)bph * P.BH;
    CUtensorMap tmW, tmB;
    cudaError_t e = make_tma_map_bf16(&tmW, w_bf16, (uint64_t)P.H * P.Lg_pad,
                                      P.d, 16u);
    if (e == cudaSuccess)
        e = make_tma_map_bf16(&tmB, Bh, (uint64_t)P.BH * P.r, P.d,
                              (uint32_t)P.r);
    if (e != cudaSuccess) return e;
    auto launch = [&](auto kern) {
        cudaError_t err = cudaFuncSetAttribute(
            kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (err != cudaSuccess) return taken(err);
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.blockDim = dim3(kPrThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        // one pair per two SMs that can hold it at once, at most one per
        // block
        int clusters = 0;
        cfg.gridDim = dim3(2 * 76);
        err = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
        if (err != cudaSuccess) return taken(err);
        if (clusters < 1) return cudaErrorInvalidConfiguration;
        const long ncl = total < clusters ? total : clusters;
        cfg.gridDim = dim3((unsigned)(2 * ncl));
        return taken(cudaLaunchKernelEx(
            &cfg, kern, (const uint16_t *)q, (const uint16_t *)k,
            (const uint16_t *)v, tmW, tmB, perm_q, perm_k, A, lambda_tok,
            gates, P.o32 ? nullptr : (uint16_t *)o,
            P.o32 ? (float *)o : nullptr, log_d_sparse, d_lr, m_sparse, P.N,
            P.H, P.L, P.Lg_pad, P.beta, P.eps, P.scale, P.lambda,
            P.fusion_mode, bph, total, status));
    };
    return P.o32 ? launch(k_block_attn_pair<true>)
                 : launch(k_block_attn_pair<false>);
}

}  // namespace elsaa
