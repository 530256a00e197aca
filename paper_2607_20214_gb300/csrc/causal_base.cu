// Exact causal attention of the base segments (the leaves of Algorithm
// "Causal sortLSH Sparse Exact Attention Branch"): rows of a segment of
// n_leaf rows attend to keys j <= i of the same segment; writes the running
// sparse result O (fp32) and log d.
//
// One persistent CTA per SM takes pairs of 128-query tiles of a segment,
// longest pairs first, from a work counter. The two tiles (slots) share
// every key and value tile. Roles:
//   warps 0-3, 4-7  softmax of slot 0 / 1: one thread per query row holds all
//                   128 scores of a key tile in registers, so neither the row
//                   maximum nor the sum needs another thread
//   warp 8          issues every MMA: S = Q K^T, O += P V (P from TMEM)
//   warp 9          takes the items, TMA loads of Q, K (two buffers), V (two)
// TMEM: S_s at 128 s, O_s at 256 + 128 s, P_s behind O_s at D = 64, over S_s at
// D = 128. O stays in tensor memory; a softmax warp rescales it when the maximum of one of its
// rows grows. (Only beyond 2^8 it was no faster, and off by up to 2.5 times as
// much in peaked heads: the weight of the largest key is exactly 1 only
// against its own maximum; otherwise bf16 rounds it.)
//
// What bounds it: per slot and key tile the chain S MMA -> softmax -> P V MMA;
// the other slot's chain runs beside it. Two CTAs per SM with two threads per
// row, which met at six CTA barriers per key tile and kept O in registers,
// took 730 us at B2 H16 N16384 d128 with 4096-row segments (550 GFLOP); this
// kernel 467 us (0.62 of the measured bf16 peak).
// Softmax takes 1.1 K clocks of a slot's 3.6 K per key tile; the products'
// issue, one slot behind the other, most of the rest.
#include "device_common.cuh"
#include "tc_common.cuh"
#include "tc_race.cuh"

#include <type_traits>

namespace elsaa {

namespace {

using namespace tc;

// 384 x 168 registers at launch = 256 x 208 (softmax) + 128 x 88
constexpr int kCbThreads = 384;
constexpr int kCbRegsSoft = 208, kCbRegsOther = 88;
static_assert(256 * kCbRegsSoft + 128 * kCbRegsOther <= kCbThreads * 168,
              "register shares within the launch's total");

struct CbBars {
    uint64_t item_full[2], item_empty[2], q_full, q_empty;
    uint64_t k_full[2], k_empty[2], v_full[2], v_empty[2];
    uint64_t s_full[2], p_full[2], o_done[2], o_empty[2];
};

// Item -> first row and the key tiles of its two query tiles. Items are
// numbered longest first: the last pair of every segment, then the one
// before it, ... Both slots walk the key tiles up from the first. (Down from
// the diagonal, slot 1 beginning a tile earlier, both ended together, but the
// slots then held different tiles of the two-deep rings: 537 us.)
struct CbItem {
    size_t row0;  // first row of the segment (over all heads)
    int q0, n[2];
    __device__ CbItem(int item, int N, int n_leaf, int segs) {
        const int nq = n_leaf / 128, np = (nq + 1) / 2;
        const int p = np - 1 - item / segs, seg = item % segs;
        row0 = (size_t)seg * n_leaf;  // segments tile [BH][N] in order
        q0 = 2 * p;
        n[0] = q0 + 1;
        n[1] = q0 + 1 < nq ? q0 + 2 : 0;
    }
};

template <int D>
__global__ void __launch_bounds__(kCbThreads, 1)
    k_causal_base(const __grid_constant__ CUtensorMap tmQ,
                  const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV, int N, int n_leaf,
                  int segs, int items, int *__restrict__ next_item,
                  float scale, float eps, float *__restrict__ RO,
                  float *__restrict__ RL, DeviceStatus *status) {
    wait_for_stream();
    extern __shared__ unsigned char smem_raw[];
    __shared__ CbBars bars;
    __shared__ uint32_t tbase;
    __shared__ int abort_flag, item_s[2];
    volatile int *abort = &abort_flag;
    constexpr uint32_t kTileB = 128 * D * 2;
    const int tid = threadIdx.x, warp = tid >> 5, lane_id = tid & 31;
    const uint32_t sQ = align1k(smem_u32(smem_raw));
    const uint32_t sK = sQ + 2 * kTileB, sV = sK + 2 * kTileB;

    if (warp == 8) tmem_alloc(&tbase, 512);
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars.item_full[s], 1);
            mbar_init(&bars.item_empty[s], 9);  // eight softmax warps, MMA
            mbar_init(&bars.k_full[s], 1);
            mbar_init(&bars.k_empty[s], 1);
            mbar_init(&bars.v_full[s], 1);
            mbar_init(&bars.v_empty[s], 1);
            mbar_init(&bars.s_full[s], 1);
            mbar_init(&bars.p_full[s], 128);
            mbar_init(&bars.o_done[s], 1);
            mbar_init(&bars.o_empty[s], 128);
        }
        mbar_init(&bars.q_full, 1);
        mbar_init(&bars.q_empty, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tbase;

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(
            kCbRegsOther));
        if (warp == 9 && lane_id == 0) {
            // ---------------------------------------------- items and loads
            int c = 0;  // key tiles loaded so far
            bool ok = true;
            auto load = [&](uint64_t *full, uint64_t *empty, uint32_t dst,
                            const CUtensorMap *map, int row, int site) {
                const int st = c & 1;
                if (c >= 2 && !mbar_wait_or_abort(&empty[st],
                                                  ((c >> 1) - 1) & 1, abort,
                                                  status, site))
                    return false;
                mbar_expect_tx(&full[st], kTileB);
                for (int p = 0; p < D / 64; ++p)
                    tma_load_2d(dst + st * kTileB + p * 16384, map, 64 * p,
                                row, &full[st]);
                return true;
            };
            for (int it = 0; ok; ++it) {
                int item = atomicAdd(next_item, 1);
                if (item >= items) item = -1;
                if (it >= 2 && !mbar_wait_or_abort(&bars.item_empty[it & 1],
                                                   ((it >> 1) - 1) & 1, abort,
                                                   status, 150))
                    break;
                item_s[it & 1] = item;
                mbar_arrive(&bars.item_full[it & 1]);
                if (item < 0) break;
                const CbItem w(item, N, n_leaf, segs);
                if (it >= 1 && !mbar_wait_or_abort(&bars.q_empty, (it - 1) & 1,
                                                   abort, status, 151))
                    break;
                const int nt = w.n[1] ? 2 : 1;
                mbar_expect_tx(&bars.q_full, nt * kTileB);
                for (int s = 0; s < nt; ++s)
                    for (int p = 0; p < D / 64; ++p)
                        tma_load_2d(sQ + s * kTileB + p * 16384, &tmQ, 64 * p,
                                    (int)w.row0 + 128 * (w.q0 + s),
                                    &bars.q_full);
                const int nk = max(w.n[0], w.n[1]);
                for (int kt = 0; kt < nk && ok; ++kt, ++c) {
                    const int row = (int)w.row0 + 128 * kt;
                    ok = load(bars.k_full, bars.k_empty, sK, &tmK, row, 152) &&
                         load(bars.v_full, bars.v_empty, sV, &tmV, row, 153);
                }
            }
        } else if (warp == 8) {
            // ---------------------------------------------------- MMA issue
            // Whenever a slot's P is ready: its P V product, and right behind
            // it the scores of its next key tile; the softmax sees these only
            // when both are complete (a commit covers all that was issued
            // before it). At D = 128 the scores go over P. That relies on the
            // two products running in the order of their issue, as products
            // of one thread do on this chip, though it is documented for
            // products of one accumulator only; a wait for the P V product
            // takes 539 us instead of 465 (B2 H16 N16384, 4096-row segments)
            // and there are no other columns. At D = 64 P has columns of its
            // own.
            // The whole warp runs the loop, so that its state and the
            // operands' descriptors are warp-uniform; one lane issues.
            const bool el = elect_one();
            auto test = [&](uint64_t *bar, uint32_t par) -> bool {
                return __all_sync(0xffffffffu, mbar_test(bar, par));
            };
            auto wait = [&](uint64_t *bar, uint32_t par, int site) -> bool {
                return __all_sync(0xffffffffu,
                                  mbar_wait_or_abort(bar, par, abort, status,
                                                     site));
            };
            const uint32_t id_s = idesc_bf16(128, 128, false, false);
            const uint32_t id_o = idesc_bf16(128, D, false, true);
            const uint64_t dQ = smem_desc(sQ, 16, 1024);
            const uint64_t dK = smem_desc(sK, 16, 1024);
            const uint64_t dV = smem_desc(sV, 16384, 1024);
            constexpr uint32_t kTile = kTileB >> 4;  // in descriptor units
            int c0 = 0;                // key tiles of earlier items
            int gp0 = 0, gp1 = 0;      // P V products issued per slot
            int go0 = 0, go1 = 0;      // items finished per slot
            bool ok = true;
            for (int it = 0; ok; ++it) {
                ok = wait(&bars.item_full[it & 1], (it >> 1) & 1, 154);
                if (!ok) break;
                const int item = item_s[it & 1];
                __syncwarp();
                if (el) mbar_arrive(&bars.item_empty[it & 1]);
                if (item < 0) break;
                const CbItem w(item, N, n_leaf, segs);
                const int n0 = w.n[0], n1 = w.n[1];
                ok = wait(&bars.q_full, it & 1, 155);
                if (!ok) break;
                int us0 = 0, us1 = 0, up0 = 0, up1 = 0;
                // the scores of slot s's next key tile
                auto scores = [&](auto slot, int &us, int n, int us_o,
                                  int n_o) {
                    constexpr int s = decltype(slot)::value;
                    const int st = (c0 + us) & 1;
                    if (!wait(&bars.k_full[st], ((c0 + us) >> 1) & 1, 160))
                        return false;
                    tc_fence_after();
                    const uint64_t q = dQ + s * kTile, k = dK + st * kTile;
                    if (el) {
#pragma unroll
                        for (int x = 0; x < D / 16; ++x) {
                            const uint32_t o = (x >> 2) * 1024 + (x & 3) * 2;
                            mma_ss(tm + 128u * s, q + o, k + o, id_s, x > 0);
                        }
                        mma_commit(&bars.s_full[s]);
                        // both slots have used the tile
                        if (us >= n_o || us_o > us)
                            mma_commit(&bars.k_empty[st]);
                        if (us + 1 == n && us_o == n_o)
                            mma_commit(&bars.q_empty);
                    }
                    ++us;
                    return true;
                };
                auto step = [&](auto slot, int &us, int &up, int &gp, int go,
                                int n, int us_o, int up_o, int n_o) {
                    constexpr int s = decltype(slot)::value;
                    constexpr uint32_t cO = 128u * s + 256u;
                    constexpr uint32_t cP = D == 64 ? cO + 64 : 128u * s;
                    const int st = (c0 + up) & 1;
                    if (up == us || !test(&bars.p_full[s], gp & 1) ||
                        !test(&bars.v_full[st], ((c0 + up) >> 1) & 1) ||
                        (up == 0 && go > 0 &&
                         !test(&bars.o_empty[s], (go - 1) & 1)))
                        return false;
                    tc_fence_after();
                    const uint64_t v = dV + st * kTile;
                    const uint32_t more = up > 0;
                    if (el) {
#pragma unroll
                        for (int x = 0; x < 8; ++x)
                            mma_ts(tm + cO, tm + cP + 8 * x, v + 128 * x, id_o,
                                   x > 0 ? 1u : more);
                        mma_commit(&bars.o_done[s]);
                        if (up >= n_o || up_o > up)
                            mma_commit(&bars.v_empty[st]);
                    }
                    ++up;
                    ++gp;
                    if (us < n) ok = scores(slot, us, n, us_o, n_o);
                    return true;
                };
                using S0 = std::integral_constant<int, 0>;
                using S1 = std::integral_constant<int, 1>;
                ok = scores(S0{}, us0, n0, us1, n1);
                if (ok && n1 > 0) ok = scores(S1{}, us1, n1, us0, n0);
                unsigned long long t_last = 0;
                uint32_t idle = 0;
                while (ok && (up0 < n0 || up1 < n1)) {
                    const bool a = step(S0{}, us0, up0, gp0, go0, n0, us1,
                                        up1, n1);
                    const bool b = step(S1{}, us1, up1, gp1, go1, n1, us0,
                                        up0, n0);
                    if (a || b) {
                        idle = 0;
                    } else if ((++idle & 255u) == 0) {
                        if (idle == 256u) t_last = global_ns();
                        const bool late = global_ns() - t_last > kWaitLimitNs;
                        if (late) {
                            *abort = 1;
                            record_timeout(status, 156);
                        }
                        ok = !__any_sync(0xffffffffu, late || *abort);
                    }
                }
                c0 += max(n0, n1);
                ++go0;
                go1 += n1 > 0;
            }
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------- softmax
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kCbRegsSoft));
        const int s = warp >> 2, row = (warp & 3) * 32 + lane_id;
        const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tm + lane + 128u * s, tO = tS + 256u;
        const uint32_t tP = D == 64 ? tO + 64 : tS;
        const float sl2 = scale * kLog2e;
        const float2 sl22 = make_float2(sl2, sl2);
        auto wwait = [=](uint64_t *bar, uint32_t par, int site) {
            return __all_sync(0xffffffffu,
                              mbar_wait_or_abort(bar, par, abort, status,
                                                 site));
        };
        int g = 0;  // key tiles of this slot so far
        bool ok = true;
        for (int it = 0; ok; ++it) {
            ok = wwait(&bars.item_full[it & 1], (it >> 1) & 1, 157);
            if (!ok) break;
            const int item = item_s[it & 1];
            __syncwarp();
            if (lane_id == 0) mbar_arrive(&bars.item_empty[it & 1]);
            if (item < 0) break;
            const CbItem w(item, N, n_leaf, segs);
            const int n = w.n[s];
            if (n == 0) continue;
            float mref = 0.0f, lsum = 0.0f;
            for (int kt = 0; kt < n; ++kt, ++g) {
                ok = wwait(&bars.s_full[s], g & 1, 158);
                if (!ok) break;
                tc_fence_after();
                float v[128];
                {
                    uint32_t a[32], b[32], c[32], e[32];
                    tmem_ld32(tS, a);
                    tmem_ld32(tS + 32, b);
                    tmem_ld32(tS + 64, c);
                    tmem_ld32(tS + 96, e);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 32; ++q) {
                        v[q] = __uint_as_float(a[q]);
                        v[32 + q] = __uint_as_float(b[q]);
                        v[64 + q] = __uint_as_float(c[q]);
                        v[96 + q] = __uint_as_float(e[q]);
                    }
                }
                if (kt == w.q0 + s) {  // the diagonal tile
#pragma unroll
                    for (int q = 0; q < 128; ++q)
                        if (q > row) v[q] = -INFINITY;
                }
                float mx[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                for (int q = 4; q < 124; q += 8)
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        mx[x] = max3(mx[x], v[q + 2 * x], v[q + 2 * x + 1]);
                mx[0] = max3(mx[0], v[124], v[125]);
                mx[1] = max3(mx[1], v[126], v[127]);
                const float z =
                    fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]) * sl2;
                if (kt == 0) {
                    mref = z;
                } else {
                    // these scores were issued behind the last tile's P V
                    // product: it is complete when they are
                    const bool need = z > mref;
                    if (__any_sync(0xffffffffu, need)) {
                        const float f = need ? ex2_approx(mref - z) : 1.0f;
                        const float2 f2 = make_float2(f, f);
#pragma unroll 1
                        for (int c = 0; c < D; c += 16) {
                            uint32_t o[16];
                            tmem_ld16(tO + c, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int q = 0; q < 16; q += 2) {
                                const float2 y =
                                    mul2(make_float2(__uint_as_float(o[q]),
                                                     __uint_as_float(
                                                         o[q + 1])),
                                         f2);
                                o[q] = __float_as_uint(y.x);
                                o[q + 1] = __float_as_uint(y.y);
                            }
                            tmem_st16(tO + c, o);
                        }
                        lsum *= f;
                        if (need) mref = z;
                    }
                }
                const float2 nm = make_float2(-mref, -mref);
                float2 ls[2] = {make_float2(0.0f, 0.0f),
                                make_float2(0.0f, 0.0f)};
#pragma unroll
                for (int c = 0; c < 128; c += 32) {
                    uint32_t pw[16];
#pragma unroll
                    for (int q = 0; q < 32; q += 2) {
                        const float2 x = fma2(
                            make_float2(v[c + q], v[c + q + 1]), sl22, nm);
                        const float2 p =
                            make_float2(ex2_approx(x.x), ex2_approx(x.y));
                        ls[(q >> 1) & 1] = add2(ls[(q >> 1) & 1], p);
                        pw[q >> 1] = pack_bf16x2(p.x, p.y);
                    }
                    tmem_st16(tP + c / 2, pw);
                }
                lsum += (ls[0].x + ls[1].x) + (ls[0].y + ls[1].y);
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(&bars.p_full[s]);
            }
            if (!ok) break;
            // O = sum e^z V / (sum e^z + eps), log d (natural log)
            ok = wwait(&bars.o_done[s], (g - 1) & 1, 159);
            if (!ok) break;
            tc_fence_after();
            const size_t tok = w.row0 + 128 * (size_t)(w.q0 + s) + row;
            const float inv = 1.0f / (lsum + eps * ex2_approx(-mref));
            float *o = RO + tok * D;
#pragma unroll
            for (int c = 0; c < D; c += 32) {
                uint32_t a[32];
                tmem_ld32(tO + c, a);
                tmem_wait_ld();
                if (c + 32 == D) {
                    tc_fence_before();
                    mbar_arrive(&bars.o_empty[s]);
                }
#pragma unroll
                for (int q = 0; q < 32; q += 8) {
                    uint32_t y[8];
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        y[x] = __float_as_uint(__uint_as_float(a[q + x]) *
                                               inv);
                    st_global_v8(o + c + q, y);
                }
            }
            RL[tok] = (mref + log2f(lsum)) * kLn2;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tm, 512);
}

}  // namespace

cudaError_t launch_causal_base(const Plan &P, int n_leaf, const void *q,
                               const void *k, const void *v, int *next_item,
                               float *RO, float *RL, DeviceStatus *status,
                               cudaStream_t st) {
    const int segs = P.BH * (P.N / n_leaf);
    const int items = segs * ((n_leaf / 128 + 1) / 2);
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = 1024 + (size_t)6 * 128 * P.d * 2;
    CUtensorMap tmQ, tmK, tmV;
    const uint64_t rows = (uint64_t)P.BH * P.N;
    cudaError_t e = make_tma_map_bf16(&tmQ, q, rows, P.d, 128);
    if (e == cudaSuccess) e = make_tma_map_bf16(&tmK, k, rows, P.d, 128);
    if (e == cudaSuccess) e = make_tma_map_bf16(&tmV, v, rows, P.d, 128);
    if (e != cudaSuccess) return e;
    auto launch = [&](auto kern) {
        return launch_after(kern, dim3(items < sms ? items : sms), kCbThreads,
                            smem, st, tmQ, tmK, tmV, P.N, n_leaf, segs, items,
                            next_item, P.scale, P.eps, RO, RL, status);
    };
    return P.d == 128 ? launch(k_causal_base<128>) : launch(k_causal_base<64>);
}

}  // namespace elsaa
