// Persistent, warp-specialised sortLSH block attention + RACE readout +
// fusion (Algorithm "sortLSH Sparse Exact Attention Branch" block step,
// Algorithm "RACE Low-Rank Attention Branch" steps 9-10, Eq. (5)-(6)) for
// bf16 inputs: key blocks of up to 256, neighbour windows and the top-k
// selector's candidate blocks, 128 keys per pass.
//
// One CTA per SM walks a contiguous range of 128-query tiles (ordered by
// head, then sorted position, so the per-head B summary, A summary and RACE
// planes are loaded once per head). Roles:
//   warps 0-7,  compute for TMEM slot 0 / slot 1 (256 columns each: scores,
//   8-15        P and pre-scaled features, then the output accumulator);
//               slot g takes the tiles of local index = g (mod 2), so one
//               slot's softmax overlaps the other slot's MMAs and loads.
//               Within a slot, warps w and w + 4 share TMEM lanes (lane
//               group w mod 4) and split each row's key columns and output
//               columns in halves; half h owns the RACE buckets of the
//               64-bucket chunks h and h + 2. The two warps exchange row
//               maxima and sums over a barrier of their 64 threads; nothing
//               else synchronises the slot.
//   warp 16     allocates tensor memory and issues every MMA (one lane of it).
//   warp 17     per head, TMA loads of the bf16 RACE planes (under the key
//               rows), the bf16 B summary and the fp32 A summary.
//   warps 18-19 V rows; warps 20-23 Q and K rows: cp.async gathers, whole
//               rows per instruction, row numbers read a unit ahead.
//
// Per tile: S and projections MMA -> (slot) softmax, P into TMEM -> P V MMA,
// meanwhile (slot) features, Den, fusion scalars -> pre-scaled features into
// TMEM -> Phi'B MMA into the same accumulator -> (slot) epilogue
// O = c1 * acc, stored from registers. Every hand-off is an mbarrier; every
// wait is bounded and a stalled pipeline drains through a shared abort flag.
//
// What bounds it: a slot's own chain of these steps, about 17 K clocks per
// tile at d = 128 (clock traces: the next tile's scores are there when the
// slot asks for them; two slots gave a tile per 8.5 K clocks, where the
// copies need 6 K). Every step taken off the chain shows in the time: copies
// by warps of their own, features under the P V product, barriers of 64
// threads only (c3: 163 -> 143 us; c2: 45 -> 42; c5: 138 -> 129; c3 top-k, two
// passes: 313 -> 263), products issued by a converged warp from descriptors
// made once (c3: 137 -> 133; c2: 41 -> 37; c5: 126 -> 106; top-k: 263 -> 229),
// Den folded bit by bit (c3: 133 -> 127). When c3 took 143 us, Den made up 22
// of it, the features 15, the stores 7, the bit factors 5.
#include "device_common.cuh"
#include "tc_common.cuh"
#include "tc_race.cuh"

#include <type_traits>

namespace elsaa {

namespace {

using namespace tc;

constexpr int kWsThreads = 768;   // 16 compute warps and 8 others
constexpr int kWsMmaWarp = 16;
constexpr int kWsVWarp = 18, kWsVWarps = 2;
constexpr int kWsQkWarp = 20, kWsQkWarps = 4;
constexpr int kWsNK = 128;        // keys per query tile
// Registers: 768 x 80 at launch = 512 x 96 (compute) + 256 x 48 (others).
constexpr int kWsRegsCompute = 96, kWsRegsOther = 48;
static_assert(512 * kWsRegsCompute + 256 * kWsRegsOther <= kWsThreads * 80,
              "register shares within the launch's total");
// TMEM slot layout (256 columns): S/P/features region [0, 128) in four
// 32-column quarters, output accumulator [128, 128 + d). P of keys
// [64h, 64h + 64) (row half h) lives in quarter 2h, packed in place over
// the scores already read; the pre-scaled RACE features of buckets
// [0, 128) go to quarters 1 and 3, buckets [128, 256) to quarters 0 and 2
// once the P V product is done. The projections come out in columns
// [128, 128 + Lg_pad), read before the first P V product overwrites them.

template <int QS, int VS>
struct WsBars {
    uint64_t qk_full[QS], qk_empty[QS], v_full[VS], v_empty[VS];
    uint64_t wb_full, head_done;
    uint64_t s_full[2], p_full[2], pv_done[2], phi_full[2], o_full[2];
    uint64_t tmem_empty[2];
};

// NPASS 128-key passes per query tile, online softmax across them: 1 for
// b <= 128; b / 128 for larger blocks; with nb neighbouring sorted key
// blocks per side (b >= 128), (2 nb + 1) b / 128 passes over the window.
// KM: which keys the passes walk. 0: the query block's own key block.
// 1 (WIN): a neighbour window (nb > 0), whose passes past either end of
// the sequence are masked. 2 (SEL): the top-k selector's candidate blocks
// (cand, tk_c per query block), each key masked unless the row's bit in
// selmask is set. The checks of the other modes are compiled out. O32: O
// is written as fp32 (out_fp32).
// QS: buffers of the Q and key tiles (one pass per tile when > 1), so that
// the rows of tile t + QS are copied while tiles t + 1 .. t + QS - 1 wait
// for their scores, with as many value buffers.
// KB: b when it is 32 or 64 (0: any b). The 32 rows of a warp then share one
// key block of KB scores, half for each of the row's two threads; the
// general path takes all 128 columns with a mask.
template <int G, int NPASS, int KM, bool O32 = false, int QS = 1, int KB = 0>
__global__ void __launch_bounds__(kWsThreads, 1)
    k_block_attn_ws(const uint16_t *__restrict__ qx,
                    const uint16_t *__restrict__ kx,
                    const uint16_t *__restrict__ vx,
                    const __grid_constant__ CUtensorMap tmW,
                    const __grid_constant__ CUtensorMap tmB,
                    const int32_t *__restrict__ perm_q,
                    const int32_t *__restrict__ perm_k,
                    const float *__restrict__ Ag,
                    const float *__restrict__ lambda_tok,
                    const float *__restrict__ gates, uint16_t *__restrict__ ox,
                    float *__restrict__ o32,
                    float *__restrict__ log_ds_out, float *__restrict__ dlr_out,
                    float *__restrict__ m_out, int N, int d, int H, int b,
                    int nb, int L, int Lg_pad, float beta, float eps,
                    float scale,
                    float lambda, int mode, int tiles_per_head,
                    long total_tiles, DeviceStatus *status,
                    const int32_t *__restrict__ cand,
                    const uint32_t *__restrict__ selmask, int tk_c) {
    constexpr bool WIN = KM == 1, SEL = KM == 2;
    constexpr int VS = QS > 2 ? QS : 2;  // value buffers
    static_assert((QS == 1 && KB == 0) || (NPASS == 1 && KM == 0),
                  "one pass per tile");
    constexpr int R = 1 << G;
    constexpr int nk = kWsNK;
    extern __shared__ unsigned char smem_raw[];
    __shared__ WsBars<QS, VS> bars;
    __shared__ uint32_t tbase;
    __shared__ int abort_flag;
    __shared__ float xmax[2][2][128];
    __shared__ float2 xsum[2][2][128];  // row sum, Den
    volatile int *abort = &abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane_id = tid & 31;
    const int r = L * R;
    const long t_begin = total_tiles * blockIdx.x / gridDim.x;
    const long t_end = total_tiles * (blockIdx.x + 1) / gridDim.x;
    const int ntiles = (int)(t_end - t_begin);
    const int nunits = ntiles * NPASS;

    const uint32_t tileB = (uint32_t)nk * d * 2u;  // one [128 x d] tile
    const uint32_t base = align1k(smem_u32(smem_raw));
    // key tile and RACE planes stacked as one B operand of NR rows: the
    // scores and the query projections come out of one MMA (N = NR) into
    // TMEM columns [0, 128) and [128, 128 + Lg_pad)
    const int NR = nk + Lg_pad;
    const uint32_t sQ = base;
    const uint32_t sKW = sQ + QS * tileB;
    const uint32_t tileKW = align1k((uint32_t)NR * d * 2u);
    const uint32_t sV0 = sKW + QS * tileKW;
    const uint32_t sB = sV0 + VS * tileB;
    const uint32_t sA = sB + align1k(r * d * 2);  // fp32 [r]
    const float *Asm = reinterpret_cast<const float *>(smem_raw + (sA - smem_u32(smem_raw)));

    if (warp == kWsMmaWarp) tmem_alloc(&tbase, 512);
    if (tid == 0) {
        for (int s = 0; s < QS; ++s) {
            mbar_init(&bars.qk_full[s], 32 * kWsQkWarps);
            mbar_init(&bars.qk_empty[s], 1);
        }
        for (int s = 0; s < VS; ++s) {
            mbar_init(&bars.v_full[s], 32 * kWsVWarps);
            // one pass: the slot's warps, after their stores (freeing the
            // buffer earlier brings its copies into busier phases: 42 -> 43
            // us at c2); several: the P V product's commit
            mbar_init(&bars.v_empty[s], NPASS == 1 ? 8 : 1);
        }
        mbar_init(&bars.wb_full, 1);
        mbar_init(&bars.head_done, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars.s_full[s], 1);
            mbar_init(&bars.p_full[s], 256);
            mbar_init(&bars.pv_done[s], 1);
            mbar_init(&bars.phi_full[s], 256);
            mbar_init(&bars.o_full[s], 1);
            mbar_init(&bars.tmem_empty[s], 256);
        }
        abort_flag = 0;
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tbase;

    // tile indices fit in int (checked on the host)
    const int tb = (int)t_begin;
    auto tile_head = [=](int i) { return (tb + i) / tiles_per_head; };
    auto tile_p0 = [=](int i) { return (tb + i) % tiles_per_head * 128; };
    auto new_head = [=](int i) {
        return i == 0 || (tb + i) % tiles_per_head == 0;
    };
    // sorted position of key column 0 of pass p of the tile starting at
    // query position p0: the passes walk the key window of the tile's
    // query block (the block and nb neighbouring blocks per side) in
    // 128-key steps. A pass past either end of the sequence holds no keys:
    // its rows are read from a valid position and its scores are masked.
    // SEL: pass p holds candidate keys [128 p, 128 p + 128) of the query
    // block, i.e. keys of candidate block 128 p / b (b >= 128)
    auto key_pos_raw = [=](int bh, int p0, int p) {
        if (SEL) {
            const int T = N / b, t = p0 / b;
            int u = cand[((size_t)bh * T + t) * tk_c + (128 * p) / b];
            u = (u < 0 || u >= T) ? t : u;
            return u * b + (128 * p) % b;
        }
        return NPASS == 1 ? p0 : (p0 / b - (WIN ? nb : 0)) * b + 128 * p;
    };
    auto pass_valid = [=](int p0, int p) {
        if (!WIN) return true;
        const int k0 = key_pos_raw(0, p0, p);
        return k0 >= 0 && k0 < N;
    };
    auto key_pos = [=](int bh, int p0, int p) {
        const int k0 = key_pos_raw(bh, p0, p);
        if (NPASS == 1) return k0;  // the tile's own keys (ragged end kept)
        return k0 < 0 ? 0 : (k0 > N - 128 ? N - 128 : k0);
    };
    // global row number of sorted position pos (the ragged end repeats the
    // last row; those rows are never stored). An entry outside [0, N) is
    // read as row 0 (the orders come from the sort, in range by
    // construction); the checked build (ELSAA_CHECKED) also records it.
    auto global_row = [=](const int32_t *pm, int bh, int pos) {
        int v = pm[(size_t)bh * N + min(pos, N - 1)];
        if (v < 0 || v >= N) {
#ifdef ELSAA_CHECKED
            report(status, kDevPermRange, 4, bh, v);
#endif
            v = 0;
        }
        return bh * N + v;
    };

    if (warp >= kWsMmaWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(
            kWsRegsOther));
        auto lwait = [=](uint64_t *bar, uint32_t par, int site) {
            return __all_sync(0xffffffffu,
                              mbar_wait_or_abort(bar, par, abort, status,
                                                 site));
        };
        const int cpr = d >> 3;    // 16-byte chunks per row
        const int rpi = 32 / cpr;  // rows per instruction
        const int sub = lane_id / cpr, ch = lane_id - sub * cpr;
        // copies rows [r0, r0 + 32) of a tile of `rows` rows; lane l holds
        // the global number of row r0 + l
        auto copy32 = [=](uint32_t dst, int rows, int r0,
                          const uint16_t *src, int rowno) {
#pragma unroll 4
            for (int i = sub; i < 32; i += rpi) {
                const int row = __shfl_sync(0xffffffffu, rowno, i);
                cp_async16(dst + panel_offset(r0 + i, ch, rows),
                           src + (size_t)row * d + ch * 8);
            }
        };
        if (warp >= kWsQkWarp) {
            // ------------------------------------------------ Q and K rows
            const int r0 = (warp - kWsQkWarp) * 32;
            int qn = 0, kn = 0;  // of the next unit
            auto ahead = [&](int u) {
                const int t = u / NPASS, ps = u - t * NPASS;
                const int bh = tile_head(t), p0 = tile_p0(t);
                if (ps == 0) qn = global_row(perm_q, bh, p0 + r0 + lane_id);
                kn = global_row(perm_k, bh,
                                key_pos(bh, p0, ps) + r0 + lane_id);
            };
            if (nunits > 0) ahead(0);
            for (int u = 0; u < nunits; ++u) {
                const int qr = qn, kr = kn, st = u % QS;
                if (u + 1 < nunits) ahead(u + 1);
                if (u >= QS &&
                    !lwait(&bars.qk_empty[st], (u / QS - 1) & 1, 30))
                    break;
                if (NPASS == 1 || u % NPASS == 0)
                    copy32(sQ + st * tileB, nk, r0, qx, qr);
                copy32(sKW + st * tileKW, NR, r0, kx, kr);
                cp_async_mbar_arrive(&bars.qk_full[st]);
            }
            cp_async_wait<0>();
        } else if (warp >= kWsVWarp) {
            // ------------------------------------------------------ V rows
            const int r0 = (warp - kWsVWarp) * 64;
            int n0 = 0, n1 = 0;  // of the next unit
            auto ahead = [&](int u) {
                const int t = u / NPASS, ps = u - t * NPASS;
                const int bh = tile_head(t);
                const int p = key_pos(bh, tile_p0(t), ps) + r0 + lane_id;
                n0 = global_row(perm_k, bh, p);
                n1 = global_row(perm_k, bh, p + 32);
            };
            if (nunits > 0) ahead(0);
            for (int u = 0; u < nunits; ++u) {
                const int a0 = n0, a1 = n1, st = u % VS;
                if (u + 1 < nunits) ahead(u + 1);
                if (u >= VS &&
                    !lwait(&bars.v_empty[st], (u / VS - 1) & 1, 33))
                    break;
                copy32(sV0 + st * tileB, nk, r0, vx, a0);
                copy32(sV0 + st * tileB, nk, r0 + 32, vx, a1);
                cp_async_mbar_arrive(&bars.v_full[st]);
            }
            cp_async_wait<0>();
        } else if (warp == kWsMmaWarp + 1) {
            // -------------------------------------- planes, B and A summary
            int hc = 0;
            for (int i = 0; i < ntiles; ++i) {
                if (!new_head(i)) continue;
                const int bh = tile_head(i);
                if (i > 0 && !lwait(&bars.head_done, (hc - 1) & 1, 31)) break;
                if (lane_id == 0) {
                    mbar_expect_tx(&bars.wb_full,
                                   (uint32_t)(QS * Lg_pad + r) * d * 2u +
                                       r * 4u);
                    for (int p = 0; p < (d >> 6); ++p) {
                        for (int q = 0; q < QS; ++q)
                            tma_load_2d(
                                sKW + q * tileKW + p * NR * 128 + nk * 128,
                                &tmW, 64 * p, (bh % H) * Lg_pad,
                                &bars.wb_full);
                        tma_load_2d(sB + p * r * 128, &tmB, 64 * p, bh * r,
                                    &bars.wb_full);
                    }
                    bulk_load(sA, Ag + (size_t)bh * r, (uint32_t)r * 4u,
                              &bars.wb_full);
                }
                __syncwarp();
                ++hc;
            }
        } else if (ntiles > 0) {
            // ------------------------------------------------------ MMA issue
            // Event driven: each round issues whichever MMA group is ready,
            // the oldest tile's first (Phi'B, then P V, then the next
            // scores), so one slot's epilogue never holds back the other
            // slot's products. Units: (tile, pass); a tile's later scores
            // wait for its previous P V product, which reads P from the S
            // columns. (Sent out right behind it they took 226 us against 233
            // at c3 with two passes (top-k), but products of different
            // accumulators are not documented to run in the order of their
            // issue; two tiles' passes in turn, with a second query buffer,
            // took 259.)
            const uint32_t id_sp = idesc_bf16(128, NR, false, false);
            const uint32_t id_s = idesc_bf16(128, nk, false, false);
            const uint32_t id_o = idesc_bf16(128, d, false, true);
            // The whole warp runs the loop, so that its state and the
            // operands' descriptors are warp-uniform; one lane issues. (One
            // thread alone took about 2 K clocks to issue a group.)
            const bool el = elect_one();
            auto test = [&](uint64_t *bar, uint32_t par) -> bool {
                return __all_sync(0xffffffffu, mbar_test(bar, par));
            };
            const uint64_t dQ = smem_desc(sQ, 16, 1024),
                           dKW = smem_desc(sKW, 16, 1024),
                           dV = smem_desc(sV0, (uint32_t)nk * 128, 1024),
                           dB = smem_desc(sB, (uint32_t)r * 128, 1024);
            int us = 0, up = 0, i2 = 0;  // next unit for S, unit for P V, tile
                                         // for Phi'B
            int tiles_pv = 0;            // tiles whose last P V is issued
            // position of the S and Phi'B cursors' tiles within their heads
            // (advanced incrementally: no divisions in the issue loop)
            const int tph = tiles_per_head;
            int ps = (int)(t_begin % tph), p2 = ps;
            auto adv = [tph](int q) { return q + 1 == tph ? 0 : q + 1; };
            int hc = 0;                  // heads whose planes were consumed
            unsigned long long t_last = global_ns();
            uint32_t idle = 0;  // the clock is read every 256 idle rounds
            while (i2 < ntiles) {
                bool did = false;
                if (i2 < tiles_pv) {
                    const int s = i2 & 1;
                    const uint32_t so = tm + 256u * s;
                    if (test(&bars.phi_full[s], (i2 >> 1) & 1)) {
                        tc_fence_after();
                        if (el) {
#pragma unroll
                            for (int kk = 0; kk < 16; ++kk)
                                if (16 * kk < r)  // O += Phi' B
                                    mma_ts(so + nk,
                                           so + (kk < 8
                                                     ? quarter_col(kk, 32)
                                                     : quarter_col(kk - 8, 0)),
                                           desc_at(dB, kk * 2048), id_o, 1);
                            mma_commit(&bars.o_full[s]);
                            if (i2 == ntiles - 1 || p2 == tph - 1)
                                mma_commit(&bars.head_done);
                        }
                        ++i2;
                        p2 = adv(p2);
                        did = true;
                    }
                }
                if (up < us) {
                    const int t = up / NPASS, pass = up - t * NPASS;
                    const int s = t & 1;
                    const int su = (t >> 1) * NPASS + pass;  // unit in slot
                    const int vb = up % VS;
                    const uint32_t so = tm + 256u * s;
                    if (test(&bars.p_full[s], su & 1) &&
                        test(&bars.v_full[vb], up / VS & 1)) {
                        fence_proxy_async_smem();  // cp.async data -> MMA
                        tc_fence_after();
                        const uint64_t bv = desc_at(dV, vb * tileB);
                        if (el) {
#pragma unroll
                            for (int kk = 0; kk < nk / 16; ++kk)  // O (+)= P V
                                mma_ts(so + nk, so + quarter_col(kk, 0),
                                       desc_at(bv, kk * 2048), id_o,
                                       pass > 0 || kk > 0);
                            if (pass == NPASS - 1)
                                mma_commit(&bars.pv_done[s]);
                            if (NPASS > 1) mma_commit(&bars.v_empty[vb]);
                        }
                        if (pass == NPASS - 1) ++tiles_pv;
                        ++up;
                        did = true;
                    }
                }
                // a new head's planes and B summary replace the old ones
                // only after head_done: its first S waits for every MMA of
                // the previous head to be issued
                const int ts = us / NPASS, spass = us - ts * NPASS;
                const bool nh = spass == 0 && (ts == 0 || ps == 0);
                if (us < nunits && !(nh && ts > 0 && i2 < ts)) {
                    const int s = ts & 1, qb = us % QS;
                    const uint32_t so = tm + 256u * s;
                    bool ready = test(&bars.qk_full[qb], us / QS & 1);
                    if (ready && spass == 0)
                        ready = (ts < 2 || test(&bars.tmem_empty[s],
                                                     ((ts >> 1) - 1) & 1)) &&
                                (!nh || test(&bars.wb_full, hc & 1));
                    // the S columns hold P of the pass before: its product
                    // must be complete. (That stage's barrier cannot run on:
                    // its next phase is a later unit's product.)
                    if (spass > 0)
                        ready = ready && up == us &&
                                test(&bars.v_empty[(us - 1) % VS],
                                     (us - 1) / VS & 1);
                    if (ready) {
                        if (nh) ++hc;
                        fence_proxy_async_smem();  // cp.async data -> MMA
                        tc_fence_after();
                        const uint64_t qd = desc_at(dQ, qb * tileB),
                                       kd = desc_at(dKW, qb * tileKW);
                        // pass 0: scores and projections (N = NR); later
                        // passes: scores only
                        const uint32_t id = spass == 0 ? id_sp : id_s;
                        if (el) {
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk)
                                if (16 * kk < d)
                                    mma_ss(so,
                                           desc_at(qd, (kk >> 2) * 16384 +
                                                           (kk & 3) * 32),
                                           desc_at(kd, (uint32_t)(kk >> 2) *
                                                               NR * 128 +
                                                           (kk & 3) * 32),
                                           id, kk > 0);
                            mma_commit(&bars.s_full[s]);
                            mma_commit(&bars.qk_empty[qb]);
                        }
                        ++us;
                        if (spass == NPASS - 1) ps = adv(ps);
                        did = true;
                    }
                }
                if (did) {
                    idle = 0;
                } else if ((++idle & 255u) == 0) {
                    if (idle == 256u) t_last = global_ns();
                    const bool late = global_ns() - t_last > kWaitLimitNs;
                    if (late) {
                        *abort = 1;
                        record_timeout(status, 41);
                    }
                    if (__any_sync(0xffffffffu, late || *abort)) break;
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------ compute groups
        // warps 0-7: slot 0, warps 8-15: slot 1; within a slot, warps
        // (w, w + 4) share TMEM lanes and split the row in two halves.
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(
            kWsRegsCompute));
        const int g = warp >> 3;                     // TMEM slot / tile parity
        const int half = (warp >> 2) & 1;
        const int row = (warp & 3) * 32 + lane_id;   // query row = TMEM lane
        const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
        // RACE buckets of this half: the 64-bucket chunks c = half and
        // c = half + 2 (buckets past 128); chunk c holds tables
        // [c T, c T + T)
        constexpr int T = R >= 64 ? 1 : 64 / R;
        const int ta0 = min(half * T, L), nt0 = min(ta0 + T, L) - ta0;
        const int ta1 = min((half + 2) * T, L), nt1 = min(ta1 + T, L) - ta1;
        const uint32_t cb0 = half ? 96u : 32u, cb1 = half ? 64u : 0u;
        const float sl2e = scale * kLog2e;
        const int kbeg = half * (nk / 2);
        // barrier of the row's two warps; a pair's 64 threads leave a wait
        // with one verdict (an abort seen by one warp only would strand the
        // other there)
        const int pid = 1 + g * 4 + (warp & 3);
        auto pwait = [=](uint64_t *bar, uint32_t par, int site) {
            const bool ok = mbar_wait_or_abort(bar, par, abort, status, site);
            return named_sync_and(pid, 64, ok);
        };
        const int bh0 = tile_head(0);
        int bh = tile_head(g), tih = tile_p0(g) / 128, last_bh = -1;
        for (int j = g; j < ntiles; j += 2, tih += 2) {
            const int k = j >> 1;
            const uint32_t so = tm + 256u * g + lane;
            while (tih >= tiles_per_head) {
                tih -= tiles_per_head;
                ++bh;
            }
            const int p0 = tih * 128;
            const int qpos = p0 + row;
            const bool qvalid = qpos < N;
            int qi = perm_q[(size_t)bh * N + min(qpos, N - 1)];  // prefetch
            if (!pwait(&bars.s_full[g], (k * NPASS) & 1, 51)) break;
            tc_fence_after();
            // the A summary (read below) came by TMA: acquire its head's
            // stage (complete already: S of this tile waited for it)
            if (bh != last_bh && !pwait(&bars.wb_full, (bh - bh0) & 1, 55))
                break;
            last_bh = bh;
            // SEL: this row's selected candidates among this half's 64 keys
            // of pass ps (bit k of the 64-bit word: key kbeg + k)
            const size_t selrow = (size_t)bh * N + (size_t)min(qpos, N - 1);
            auto selbits = [&](int ps) -> unsigned long long {
                if (!SEL) return ~0ull;
                const uint32_t *w = selmask + selrow * (tk_c * b / 32) +
                                    4 * ps + 2 * half;
                return (unsigned long long)w[0] |
                       ((unsigned long long)w[1] << 32);
            };
            // row maximum of both halves
            auto row_max = [&](const float (&m)[4]) {
                xmax[g][half][row] =
                    fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
                named_sync(pid, 64);
                return fmaxf(xmax[g][0][row], xmax[g][1][row]);
            };
            float M2, lsum;  // reference (log2 units), this half's row sum
            float lam = lambda, gs = 1.0f, gl = 1.0f;
            size_t tok = 0;
            auto token = [&] {
                qi = (qi < 0 || qi >= N) ? 0 : qi;
                tok = (size_t)bh * N + qi;
                if (lambda_tok && qvalid) lam = lambda_tok[tok];
                if (gates && qvalid) {
                    const float2 gg =
                        *reinterpret_cast<const float2 *>(gates + 2 * tok);
                    gs = gg.x;
                    gl = gg.y;
                }
            };
            // per-bit factors of this half's tables: sp[0, 16) chunk half,
            // sp[16, 32) chunk half + 2; up to 32 of chunk half when it has
            // more projection columns (no second chunk exists then)
            uint32_t pr[32];
            auto load_projections = [&] {
                if (T * G <= 16) {
                    uint32_t a[16], c[16];
                    tmem_ld16(so + nk + ta0 * G, a);
                    tmem_ld16(so + nk + ta1 * G, c);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        pr[q] = a[q];
                        pr[16 + q] = c[q];
                    }
                } else {
                    tmem_ld32(so + nk + ta0 * G, pr);
                    tmem_wait_ld();
                }
            };
            // Den stays a sum over broadcast A values: through tensor memory
            // into the 16x256b layout (every value of A read serves four
            // rows) it took as long.
            float den = 0.0f;
            float sp[32];
            auto features = [&] {
                constexpr int n1 = T * G <= 16 ? 16 : 32;
                race_factors<n1>(pr, beta, sp);
                float dacc[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // independent chains
                constexpr bool fold = QS == 1 && !WIN;  // see table_den4
                chunk_den<G, T, fold>(sp, nt0, Asm + ta0 * R, dacc);
                if constexpr (T * G <= 16) {
                    if (nt1 > 0) {
                        race_factors<16>(pr + 16, beta, sp + 16);
                        chunk_den<G, T, fold>(sp + 16, nt1, Asm + ta1 * R,
                                              dacc);
                    }
                }
                den = (dacc[0] + dacc[1]) + (dacc[2] + dacc[3]);
            };
            auto hand_over = [&](uint64_t *bar) {
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(bar);
            };
            bool fail = false;
            if constexpr (NPASS == 1) {
                // this half's scores, up to 32 at a time: kept in registers
                // from the maximum to P when that is all of them
                constexpr int KN = KB > 0 ? KB / 2 : nk / 2;
                constexpr int KC = KN < 32 ? KN : 32;
                const int kl = KB > 0 ? (warp & 3) * 32 / KN / 2 * KB : 0;
                const uint32_t own = so + kl + half * KN;
                uint32_t sv[KC];
                uint32_t sb[2] = {~0u, ~0u};
                if constexpr (SEL) {
                    const unsigned long long x = selbits(0);
                    sb[0] = (uint32_t)x;
                    sb[1] = (uint32_t)(x >> 32);
                }
                const int klo = (row / b) * b - kbeg;  // within the half
                auto load = [&](int c) {  // scores [c, c + KC), masked
                    if constexpr (KC == 32)
                        tmem_ld32(own + c, sv);
                    else
                        tmem_ld16(own + c, sv);
                    tmem_wait_ld();
                    if (KB == 0 && b < 128) {
#pragma unroll
                        for (int q = 0; q < KC; ++q)
                            if (c + q < klo || c + q >= klo + b)
                                sv[q] = 0xff800000u;
                    }
                    if constexpr (SEL) {
#pragma unroll
                        for (int q = 0; q < KC; ++q)
                            if (!(sb[c / 32] >> q & 1u)) sv[q] = 0xff800000u;
                    }
                };
                float mxa[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int c = 0; c < KN; c += KC) {
                    load(c);
#pragma unroll
                    for (int q = 0; q < KC; q += 2)
                        mxa[(q >> 1) & 3] =
                            max3(mxa[(q >> 1) & 3], __uint_as_float(sv[q]),
                                 __uint_as_float(sv[q + 1]));
                }
                M2 = row_max(mxa) * sl2e;
                token();
                float2 ls[2] = {make_float2(0.0f, 0.0f),
                                make_float2(0.0f, 0.0f)};
                const float2 sl2 = make_float2(sl2e, sl2e),
                             m2n = make_float2(-M2, -M2);
#pragma unroll
                for (int c = 0; c < KN; c += KC) {
                    if constexpr (KC < KN) load(c);
                    uint32_t pw[KC / 2];
#pragma unroll
                    for (int q = 0; q < KC; q += 2) {
                        const float2 z =
                            fma2(make_float2(__uint_as_float(sv[q]),
                                             __uint_as_float(sv[q + 1])),
                                 sl2, m2n);
                        const float2 e =
                            make_float2(ex2_approx(z.x), ex2_approx(z.y));
                        ls[(q >> 1) & 1] = add2(ls[(q >> 1) & 1], e);
                        pw[q >> 1] = pack_bf16x2(e.x, e.y);
                    }
                    if constexpr (KB == 0)  // over scores already read
                        tmem_st16(so + kbeg + (c >> 1), pw);
                    // KB: over the first columns of the block's quarter
                    // (both threads have read the scores there: row_max)
                    if constexpr (KB == 64)
                        tmem_st16(so + kl + half * 16, pw);
                    if constexpr (KB == 32)
                        tmem_st8(so + (kl & 64) + (kl & 32) / 2 + half * 8,
                                 pw);
                }
                lsum = (ls[0].x + ls[1].x) + (ls[0].y + ls[1].y);
                if constexpr (KB > 0) {  // zeros for the tile's other keys
                    uint32_t zero[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) zero[x] = 0u;
                    tmem_st16(so + (kl & 64 ^ 64) + half * 16, zero);
                    if constexpr (KB == 32) {
                        uint32_t z8[8];
#pragma unroll
                        for (int x = 0; x < 8; ++x) z8[x] = 0u;
                        tmem_st8(so + (kl & 64) + ((kl & 32) / 2 ^ 16) +
                                     half * 8,
                                 z8);
                    }
                }
                load_projections();
                hand_over(&bars.p_full[g]);
                features();
            } else {
                M2 = -INFINITY;
                lsum = 0.0f;
#pragma unroll
                for (int ps = 0; ps < NPASS; ++ps) {
                    if (ps > 0) {
                        if (!pwait(&bars.s_full[g], (k * NPASS + ps) & 1,
                                   56)) {
                            fail = true;
                            break;
                        }
                        tc_fence_after();
                    }
                    const bool pvalid = !WIN || pass_valid(p0, ps);
                    const unsigned long long sb = selbits(ps);
                    const uint32_t s0 = (uint32_t)sb, s1 = (uint32_t)(sb >> 32);
                    auto keep = [=](int q) {  // key q of this half is attended
                        return (!WIN || pvalid) &&
                               (!SEL ||
                                ((q < 32 ? s0 : s1) >> (q & 31) & 1u));
                    };
                    float mxa[4] = {-INFINITY, -INFINITY, -INFINITY,
                                    -INFINITY};
#pragma unroll
                    for (int c = 0; c < nk / 2; c += 16) {
                        uint32_t v[16];
                        tmem_ld16(so + kbeg + c, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            if (keep(c + q))
                                mxa[q & 3] =
                                    fmaxf(mxa[q & 3], __uint_as_float(v[q]));
                    }
                    const float M2b = row_max(mxa) * sl2e;
                    if (ps == 0) {
                        token();
                        M2 = M2b;
                    } else {
                        // online softmax: keep the running reference unless
                        // the row's max grew by more than 2^8; then rescale
                        // the accumulator (the previous P V product is
                        // complete: these scores waited for it) and
                        // the running sum. From an empty start (M2 = -inf) the
                        // factor is 0.
                        const bool need = M2b > M2 + 8.0f;
                        const float f = need ? ex2_approx(M2 - M2b) : 1.0f;
                        if (__any_sync(0xffffffffu, need)) {
#pragma unroll
                            for (int c = 0; c < 64; c += 16) {
                                if (c < (d >> 1)) {
                                    uint32_t v[16];
                                    const uint32_t at =
                                        so + nk + half * (d >> 1) + c;
                                    tmem_ld16(at, v);
                                    tmem_wait_ld();
#pragma unroll
                                    for (int q = 0; q < 16; ++q)
                                        v[q] = __float_as_uint(
                                            __uint_as_float(v[q]) * f);
                                    tmem_st16(at, v);
                                }
                            }
                        }
                        if (need) {
                            lsum *= f;
                            M2 = M2b;
                        }
                    }
                    float ls[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int c = 0; c < nk / 2; c += 32) {
                        uint32_t pw[16];
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh) {
                            uint32_t v[16];
                            tmem_ld16(so + kbeg + c + 16 * hh, v);
                            tmem_wait_ld();
#pragma unroll
                            for (int q = 0; q < 16; q += 2) {
                                const int kq = c + 16 * hh + q;
                                float a0 = ex2_approx(
                                    fmaf(__uint_as_float(v[q]), sl2e, -M2));
                                float a1 = ex2_approx(fmaf(
                                    __uint_as_float(v[q + 1]), sl2e, -M2));
                                a0 = keep(kq) ? a0 : 0.0f;
                                a1 = keep(kq + 1) ? a1 : 0.0f;
                                ls[(q >> 1) & 3] += a0 + a1;
                                pw[8 * hh + (q >> 1)] = pack_bf16x2(a0, a1);
                            }
                        }
                        // quarter 2h, over scores of this half already read
                        tmem_st16(so + kbeg + (c >> 1), pw);
                    }
                    lsum += (ls[0] + ls[1]) + (ls[2] + ls[3]);
                    if (ps == 0) load_projections();
                    hand_over(&bars.p_full[g]);
                    if (ps == 0) features();
                }
            }
            if (fail) break;
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
                if (!pwait(&bars.pv_done[g], k & 1, 52))
                    break;
                tc_fence_after();
                if constexpr (T * G <= 16) {
                    if (nt1 > 0)
                        write_phi_chunk<G, T>(sp + 16, nt1, ratio, so + cb1);
                }
            }
            hand_over(&bars.phi_full[g]);
            if (!pwait(&bars.o_full[g], k & 1, 53)) break;
            tc_fence_after();
            // O = c1 acc, this half's d / 2 columns. d = 128: staged as bf16
            // in the tile's value buffer (its products are complete) in the
            // swizzled panel layout, 32 rows per warp, and stored in 128-byte
            // rows; from registers, 32 bytes per lane and row, the kernel
            // took 166 us at c3 where staging took 149. d = 64 (half of the
            // bytes): from registers, 42 against 45 us at c2. An fp32 output
            // is stored from registers.
            // With several passes the value buffers are wanted sooner:
            // staging took 284 us against 263 (two passes, c3 top-k).
            const bool staged = !O32 && NPASS == 1 && d == 128;
            const uint32_t sVg = sV0 + (uint32_t)(j % VS) * tileB;
            constexpr int OW = O32 ? 32 : 16;  // words of 32 columns
            uint32_t ov[2][OW];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (c == 0 || d == 128) {
                    uint32_t v[32];
                    tmem_ld32(so + nk + half * (d >> 1) + 32 * c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < OW; ++q) {
                        if constexpr (O32) {
                            ov[c][q] =
                                __float_as_uint(c1e * __uint_as_float(v[q]));
                        } else {
                            const float2 x = mul2(
                                make_float2(c1e, c1e),
                                make_float2(__uint_as_float(v[2 * q]),
                                            __uint_as_float(v[2 * q + 1])));
                            ov[c][q] = pack_bf16x2(x.x, x.y);
                        }
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&bars.tmem_empty[g]);
            if (!staged) {
                if (qvalid) {
                    uint32_t *dst =
                        (O32 ? reinterpret_cast<uint32_t *>(o32)
                             : reinterpret_cast<uint32_t *>(ox)) +
                        (tok * (size_t)d + half * (d >> 1)) * OW / 32;
                    const bool a32 = ((uintptr_t)dst & 31u) == 0;
#pragma unroll
                    for (int c = 0; c < 2; ++c)
#pragma unroll
                        for (int q = 0; q < OW; q += 8)
                            if (c == 0 || d == 128) {
                                const uint32_t w[8] = {
                                    ov[c][q],     ov[c][q + 1], ov[c][q + 2],
                                    ov[c][q + 3], ov[c][q + 4], ov[c][q + 5],
                                    ov[c][q + 6], ov[c][q + 7]};
                                uint32_t *p = dst + c * OW + q;
                                if (a32) {
                                    st_global_v8(p, w);
                                } else {
                                    uint4 *p4 = reinterpret_cast<uint4 *>(p);
                                    p4[0] =
                                        make_uint4(w[0], w[1], w[2], w[3]);
                                    p4[1] =
                                        make_uint4(w[4], w[5], w[6], w[7]);
                                }
                            }
                }
            } else {
                const int orow = qvalid ? (int)tok : -1;
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int q = 0; q < OW; q += 4)
                        st_shared_v4(
                            sVg + panel_offset(row, 8 * half + 4 * c + q / 4,
                                               nk),
                            ov[c][q], ov[c][q + 1], ov[c][q + 2],
                            ov[c][q + 3]);
                __syncwarp();
                const int c16 = 8 * half + (lane_id & 7);
#pragma unroll 4
                for (int i = 0; i < 8; ++i) {
                    const int rl = 4 * i + (lane_id >> 3);
                    const int to = __shfl_sync(0xffffffffu, orow, rl);
                    const uint4 val = ld_shared_v4(
                        sVg + panel_offset((warp & 3) * 32 + rl, c16, nk));
                    if (to >= 0)
                        *reinterpret_cast<uint4 *>(ox + (size_t)to * d +
                                                   c16 * 8) = val;
                }
                __syncwarp();  // the value buffer is read
            }
            if (NPASS == 1 && lane_id == 0) mbar_arrive(&bars.v_empty[j % VS]);
            if (qvalid) {
                if (half == 0) {
                    if (log_ds_out) log_ds_out[tok] = log_ds;
                    if (dlr_out) dlr_out[tok] = denf;
                    if (m_out) m_out[tok] = msp;
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWsMmaWarp) tmem_dealloc(tm, 512);
}

}  // namespace

// 128-key passes per query tile, or 0 when no instantiation covers it:
// b <= 128 without neighbours: 1; b = 256: 2; neighbouring blocks (b of
// 128 or 256, gamma = 4): the (2 nb + 1) b / 128 passes of the window, 3 or
// 6 for nb = 1.
static int ws_passes(const Plan &P) {
    if (P.sel) {  // the candidate blocks, 128 keys per pass (b >= 128)
        if (P.gamma != 4 || (P.b != 128 && P.b != 256)) return 0;
        const int n = P.tk_c * P.b / 128;
        return n <= 4 ? n : 0;
    }
    if (P.nb == 0) return P.b <= 128 ? 1 : (P.b == 256 ? 2 : 0);
    if (P.nb != 1 || P.gamma != 4 || (P.b != 128 && P.b != 256)) return 0;
    return 3 * (P.b / 128);
}

bool ws_supported(const Plan &P) {
    // a half's chunks: the first may use up to 32 projection columns, the
    // second (buckets past 128) at most 16, i.e. gamma >= 4 when r > 128;
    // row numbers in int
    const long rows = (long)P.N * P.BH;  // row numbers are int
    // fp32 output is instantiated for gamma = 4; other gamma with out_fp32
    // run the CUDA-core block kernel
    if (P.o32 && P.gamma != 4) return false;
    return tc_supported(P) && ws_passes(P) > 0 &&
           (P.gamma >= 4 || P.r <= 128) && rows < (1L << 31);
}

cudaError_t launch_block_attn_ws(
    const Plan &P, const void *q, const void *k, const void *v,
    const uint16_t *w_bf16, const int32_t *perm_q, const int32_t *perm_k,
    const float *A, const uint16_t *Bh, const float *lambda_tok,
    const float *gates, void *o, float *log_d_sparse, float *d_lr,
    float *m_sparse, DeviceStatus *status, cudaStream_t st,
    const int32_t *cand, const uint32_t *selmask) {
    const int lg_pad = (P.L * P.gamma + 15) / 16 * 16;
    const size_t tileB = (size_t)kWsNK * P.d * 2;
    auto smem_for = [&](int qs) {
        const int vs = qs > 2 ? qs : 2;
        return 1024 + (2 * qs + vs) * tileB +
               qs * (((size_t)lg_pad * P.d * 2 + 1023) / 1024 * 1024) +
               ((size_t)P.r * P.d * 2 + 1023) / 1024 * 1024 +
               (size_t)P.r * 4;
    };
    const int tiles_per_head = (P.N + 127) / 128;
    const long total = (long)tiles_per_head * P.BH;
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = (int)(total < sms ? total : sms);
    const int lg = lg_pad;
    CUtensorMap tmW, tmB;
    cudaError_t e = make_tma_map_bf16(&tmW, w_bf16, (uint64_t)P.H * P.Lg_pad,
                                      P.d, (uint32_t)P.Lg_pad);
    if (e == cudaSuccess)
        e = make_tma_map_bf16(&tmB, Bh, (uint64_t)P.BH * P.r, P.d,
                              (uint32_t)P.r);
    if (e != cudaSuccess) return e;
    auto launch = [&](auto kern, int qs = 1) {
        const size_t smem = smem_for(qs);
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
        kern<<<grid, kWsThreads, smem, st>>>(
            (const uint16_t *)q, (const uint16_t *)k, (const uint16_t *)v,
            tmW, tmB, perm_q, perm_k, A, lambda_tok, gates,
            P.o32 ? nullptr : (uint16_t *)o, P.o32 ? (float *)o : nullptr,
            log_d_sparse, d_lr, m_sparse, P.N, P.d, P.H, P.b, P.nb, P.L, lg,
            P.beta, P.eps, P.scale, P.lambda, P.fusion_mode, tiles_per_head,
            total, status, cand, selmask, P.tk_c);
        return cudaGetLastError();
    };
    const int passes = ws_passes(P);
    // d = 64 leaves shared memory for three Q/K and value buffers (172 KB at
    // r = 128); at d = 128 one fits. Key blocks of 32 and 64 take half and a
    // quarter of the softmax work of the masked path. Both together, B4 H12
    // N4096 d64 b64 r128: 63 -> 45 us; B8 H12 N8192: 215 -> 138 us; B3 H5
    // N4800 d128 b64 (KB alone): 35 -> 27 us. (37, 106 and 23 us since the
    // copies and the products' issue do not bound them.)
    if (P.gamma == 4 && P.sel == 0 && passes == 1) {
        auto pick = [&](auto o32) {
            constexpr bool F = decltype(o32)::value;
            if (P.d == 64 && smem_for(3) <= 216 * 1024) {
                if (P.b == 32)
                    return launch(k_block_attn_ws<4, 1, 0, F, 3, 32>, 3);
                if (P.b == 64)
                    return launch(k_block_attn_ws<4, 1, 0, F, 3, 64>, 3);
                return launch(k_block_attn_ws<4, 1, 0, F, 3>, 3);
            }
            if (P.b == 32) return launch(k_block_attn_ws<4, 1, 0, F, 1, 32>);
            if (P.b == 64) return launch(k_block_attn_ws<4, 1, 0, F, 1, 64>);
            return launch(k_block_attn_ws<4, 1, 0, F>);
        };
        return P.o32 ? pick(std::true_type{}) : pick(std::false_type{});
    }
    if (P.o32) {  // fp32 output: gamma = 4 (ws_supported)
        if (P.sel) {
            switch (passes) {
                case 1: return launch(k_block_attn_ws<4, 1, 2, true>);
                case 2: return launch(k_block_attn_ws<4, 2, 2, true>);
                case 3: return launch(k_block_attn_ws<4, 3, 2, true>);
                case 4: return launch(k_block_attn_ws<4, 4, 2, true>);
                default: return cudaErrorInvalidValue;
            }
        }
        if (passes == 3) return launch(k_block_attn_ws<4, 3, 1, true>);
        if (passes == 6) return launch(k_block_attn_ws<4, 6, 1, true>);
        if (P.gamma != 4) return cudaErrorInvalidValue;
        return launch(k_block_attn_ws<4, 2, 0, true>);
    }
    if (P.sel) {
        switch (passes) {
            case 1: return launch(k_block_attn_ws<4, 1, 2>);
            case 2: return launch(k_block_attn_ws<4, 2, 2>);
            case 3: return launch(k_block_attn_ws<4, 3, 2>);
            case 4: return launch(k_block_attn_ws<4, 4, 2>);
            default: return cudaErrorInvalidValue;
        }
    }
    if (passes == 3) return launch(k_block_attn_ws<4, 3, 1>);
    if (passes == 6) return launch(k_block_attn_ws<4, 6, 1>);
    switch (P.gamma) {
        case 1: return P.b > 128 ? launch(k_block_attn_ws<1, 2, 0>) : launch(k_block_attn_ws<1, 1, 0>);
        case 2: return P.b > 128 ? launch(k_block_attn_ws<2, 2, 0>) : launch(k_block_attn_ws<2, 1, 0>);
        case 3: return P.b > 128 ? launch(k_block_attn_ws<3, 2, 0>) : launch(k_block_attn_ws<3, 1, 0>);
        case 4: return launch(k_block_attn_ws<4, 2, 0>);
        case 5: return P.b > 128 ? launch(k_block_attn_ws<5, 2, 0>) : launch(k_block_attn_ws<5, 1, 0>);
        case 6: return P.b > 128 ? launch(k_block_attn_ws<6, 2, 0>) : launch(k_block_attn_ws<6, 1, 0>);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace elsaa
