// Warp-specialised RACE key side (Algorithm "RACE Low-Rank Attention
// Branch", steps 3-7) for bf16 inputs: one CTA accumulates the partial
// bucket summaries B += Phi_K^T V and A += Phi_K^T 1 of one chunk of keys of
// one head in tensor memory. A comes out of the same MMAs as B: the value
// tile is followed in shared memory by a panel of ones, so each MMA has
// N = d + 16 and its last 16 columns accumulate Phi^T 1.
//
// Roles (320 threads):
//   warp 0      loader (lane 0): TMA loads of key tiles and value tiles
//               (two buffers, one tile behind the keys); completion is
//               counted in bytes on the buffers' mbarriers.
//   warp 1      allocates tensor memory and issues the MMAs (lane 0): the
//               projections W^(l) K of tile i+1 (double-buffered in TMEM)
//               are issued before the summary MMAs of tile i.
//   warps 2-9   features: thread pairs (warps w, w + 4) share a key row and
//               split its tables (half h writes buckets of its tables into
//               the one shared feature tile). The tile is handed over per
//               half: a half may write tile i+1 as soon as the MMAs that
//               read its buckets of tile i are done.
// Every hand-off is an mbarrier with a bounded wait.
#include "device_common.cuh"
#include "tc_common.cuh"
#include "tc_race.cuh"

namespace elsaa {

namespace {

using namespace tc;

constexpr int kKwThreads = 320;

struct KwBars {
    uint64_t k_full[2], k_empty[2], v_full[2], v_empty[2], w_full, done;
    uint64_t proj_full[2];
    uint64_t phi_full[2], phi_empty[2];  // per row half
};

template <int G>
__global__ void __launch_bounds__(kKwThreads, 2)
    k_race_keys_ws(const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV,
                   const __grid_constant__ CUtensorMap tmW, int N, int d,
                   int H,
                   int L, int r_pad, int Lg_pad, int chunk, float beta,
                   uint32_t tmem_cols, float *__restrict__ part,
                   DeviceStatus *status) {
    constexpr int R = 1 << G;
    extern __shared__ unsigned char smem_raw[];
    __shared__ KwBars bars;
    __shared__ uint32_t tbase;
    __shared__ int abort_flag;
    volatile int *abort = &abort_flag;
    const int s = blockIdx.x, bh = blockIdx.y, S = gridDim.x;
    const int h = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5, lane_id = tid & 31;
    const int Lg = L * G, r = L * R;
    const int nM = r_pad >> 7;

    const uint32_t base = align1k(smem_u32(smem_raw));
    const uint32_t tileB = 128u * d * 2u;
    // One feature tile, two value tiles and one panel of ones that serves
    // both: the panels of a B operand are a fixed stride apart, so value tile
    // 0 lies 16 KB panel by panel before the ones and value tile 1 at a
    // wider stride, around a key tile. d = 128: key tiles 0 and 1, d = 64:
    // one (two CTAs then still fit an SM).
    //   d = 128  W | K1 | V1.0 | K0 | V1.1 | V0.0 | V0.1 | ones | features
    //   d = 64   W | K0 | V1 | V0 | ones | features
    const int nkb = d == 128 ? 2 : 1;
    const uint32_t sW = base;
    const uint32_t s1 = sW + align1k(Lg_pad * d * 2);
    const uint32_t sK0 = d == 128 ? s1 + tileB + 16384u : s1;
    const uint32_t sK1 = s1;
    const uint32_t sV1 = s1 + tileB;
    const uint32_t vs1 = d == 128 ? 49152u : 32768u;  // panel stride of V1
    const uint32_t sOnes = sV1 + vs1 * (d / 64);
    const uint32_t sV0 = sOnes - tileB;
    const uint32_t sPhi = sOnes + 16384u;

    // TMEM columns: per M-tile an accumulator of d + 16 columns (B, then A
    // repeated 16 times), then two projection buffers of 64 columns.
    const uint32_t accN = (uint32_t)d + 16u;
    const uint32_t colP = nM * accN;

    if (warp == 1) tmem_alloc(&tbase, tmem_cols);
    if (tid == 0) {
        mbar_init(&bars.done, 1);
        mbar_init(&bars.w_full, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars.k_full[b], 1);
            mbar_init(&bars.k_empty[b], 1);
            mbar_init(&bars.v_full[b], 1);
            mbar_init(&bars.v_empty[b], 1);
            mbar_init(&bars.proj_full[b], 1);
            mbar_init(&bars.phi_full[b], 128);
            mbar_init(&bars.phi_empty[b], 1);
        }
        abort_flag = 0;
        fence_mbar_init();
    }
    for (int i = tid; i < 16384 / 16; i += kKwThreads)  // bf16 ones
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                         sOnes + i * 16),
                     "r"(0x3F803F80u)
                     : "memory");
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t t = tbase;
    // this head's bf16 planes (one TMA box of Lg_pad rows per 64 columns)
    if (tid == 0) {
        mbar_expect_tx(&bars.w_full, (uint32_t)Lg_pad * d * 2u);
        for (int pnl = 0; pnl < d / 64; ++pnl)
            tma_load_2d(sW + pnl * Lg_pad * 128, &tmW, 64 * pnl, h * Lg_pad,
                        &bars.w_full);
    }

    const int c0 = s * chunk;
    const int c1 = min(N, c0 + chunk);
    const int ntiles = c1 > c0 ? (c1 - c0 + 127) / 128 : 0;
    // buckets [0, sb) come from row half 0, [sb, r_pad) from half 1 (the
    // tail owner also zero-fills [r, r_pad)); M-tile m covers
    // [128 m, 128 m + 128)
    const int sb = table_split(L, G) * R;
    const bool h1_has = table_split(L, G) < L;
    auto tile_needs = [=](int m, int hf) {
        const int lo = 128 * m, hi = 128 * m + 128;
        if (hf == 0) return sb > lo || !h1_has;
        return h1_has && hi > sb;
    };
    auto last_mtile = [=](int hf) {  // last M-tile that reads half hf
        int last = -1;
        for (int m = 0; m < nM; ++m)
            if (tile_needs(m, hf)) last = m;
        return last;
    };

    if (warp == 0) {
        // ------------------------------------------------------------- loader
        if (lane_id == 0) {
            // K(i) needs the projection of tile i - nkb done, V(i) the
            // summary MMAs of tile i - 2; V runs one tile behind K
            auto load_v = [&](int i) {
                if (i >= 2 && !mbar_wait_or_abort(&bars.v_empty[i & 1],
                                                  ((i >> 1) - 1) & 1, abort,
                                                  status, 62))
                    return false;
                mbar_expect_tx(&bars.v_full[i & 1], tileB);
                for (int pnl = 0; pnl < d / 64; ++pnl)
                    tma_load_2d((i & 1) ? sV1 + pnl * vs1
                                        : sV0 + pnl * 16384,
                                &tmV, 64 * pnl, bh * N + c0 + i * 128,
                                &bars.v_full[i & 1]);
                return true;
            };
            for (int i = 0; i <= ntiles; ++i) {
                if (i < ntiles) {
                    const int b = i % nkb;
                    if (i >= nkb && !mbar_wait_or_abort(&bars.k_empty[b],
                                                        (i / nkb - 1) & 1,
                                                        abort, status, 61))
                        break;
                    // rows past the chunk are loaded too (next head, or
                    // zeros past the tensor) and get zero features
                    mbar_expect_tx(&bars.k_full[b], tileB);
                    for (int pnl = 0; pnl < d / 64; ++pnl)
                        tma_load_2d((b ? sK1 : sK0) + pnl * 16384, &tmK,
                                    64 * pnl, bh * N + c0 + i * 128,
                                    &bars.k_full[b]);
                }
                if (i > 0 && !load_v(i - 1)) break;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ----------------------------------------------------------- MMA issue
        if (ntiles > 0) {
            // the whole warp runs the loop (its state and the operands'
            // descriptors are warp-uniform); one lane issues
            const bool el = elect_one();
            auto wait = [&](uint64_t *bar, uint32_t par, int site) -> bool {
                return __all_sync(0xffffffffu,
                                  mbar_wait_or_abort(bar, par, abort, status,
                                                     site));
            };
            const uint32_t id_proj = idesc_bf16(128, Lg_pad, false, false);
            const uint32_t id_b = idesc_bf16(128, d + 16, true, true);
            const int last0 = last_mtile(0), last1 = last_mtile(1);
            auto proj = [=](int it) {
                const int kb = it % nkb;
                const uint32_t sK = kb ? sK1 : sK0;
                const uint32_t dst = t + colP + 64u * (it & 1);
                const uint64_t a = smem_desc(sK, 16, 1024),
                               b = smem_desc(sW, 16, 1024);
                if (!el) return;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (16 * k < d)
                        mma_ss(dst,
                               desc_at(a, (k >> 2) * 16384 + (k & 3) * 32),
                               desc_at(b, (uint32_t)(k >> 2) * Lg_pad * 128 +
                                              (k & 3) * 32),
                               id_proj, k > 0);
                mma_commit(&bars.proj_full[it & 1]);
                mma_commit(&bars.k_empty[kb]);
            };
            // projections run two tiles ahead (both TMEM buffers); each
            // iteration issues the summary MMAs of tile i, then the
            // projection of tile i + 2
            bool ok = wait(&bars.w_full, 0, 60);
            for (int it = 0; it < 2 && it < ntiles && ok; ++it) {
                ok = wait(&bars.k_full[it % nkb], (it / nkb) & 1, 63);
                if (ok) {
                    tc_fence_after();
                    proj(it);
                }
            }
            for (int i = 0; i < ntiles && ok; ++i) {
                const int b = i & 1;
                ok = wait(&bars.v_full[b], (i >> 1) & 1, 66);
                const uint32_t sV = b ? sV1 : sV0;
                const uint32_t vst = b ? vs1 : 16384u;
                bool got0 = false, got1 = false;
                for (int m = 0; m < nM && ok; ++m) {
                    if (tile_needs(m, 0) && !got0)
                        got0 = ok = wait(&bars.phi_full[0], i & 1, 65);
                    if (ok && tile_needs(m, 1) && !got1)
                        got1 = ok = wait(&bars.phi_full[1], i & 1, 65);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t da = smem_desc(sPhi + 2 * m * 16384, 16384,
                                                  1024),
                                   db = smem_desc(sV, vst, 1024);
                    const uint32_t more = i > 0;
                    if (el) {
#pragma unroll
                        for (int k = 0; k < 8; ++k)  // 128 keys, 16 per step
                            mma_ss(t + m * accN, desc_at(da, k * 2048),
                                   desc_at(db, k * 2048), id_b,
                                   k > 0 ? 1u : more);
                        if (m == last0) mma_commit(&bars.phi_empty[0]);
                        if (m == last1) mma_commit(&bars.phi_empty[1]);
                    }
                }
                if (!ok) break;
                if (el) mma_commit(&bars.v_empty[b]);
                if (i + 2 < ntiles) {
                    // the features of tile i have read projection buffer b
                    ok = wait(&bars.k_full[(i + 2) % nkb], ((i + 2) / nkb) & 1, 64);
                    if (!ok) break;
                    tc_fence_after();
                    proj(i + 2);
                }
            }
            if (ok && el) mma_commit(&bars.done);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ features
        const int cw = warp - 2;
        const int half = cw >> 2;
        const int row = (warp & 3) * 32 + lane_id;  // key row = TMEM lane
        const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
        const int split = table_split(L, G);
        const int l0 = half ? split : 0, l1 = half ? L : split;
        const bool tail_owner = (l1 == L) && (l1 > l0 || half == 0);
        auto wwait = [=](uint64_t *bar, uint32_t par, int site) {
            return __all_sync(0xffffffffu,
                              mbar_wait_or_abort(bar, par, abort, status,
                                                 site));
        };
        bool ok = true;
        const bool writes = l1 > l0 || tail_owner;  // this half has buckets
        const int hb = (l1 > l0 || half == 0) ? half : 0;  // barrier to use
        for (int i = 0; i < ntiles; ++i) {
            const int b = i & 1;
            ok = wwait(&bars.proj_full[b], (i >> 1) & 1, 67);
            if (!ok) break;
            tc_fence_after();
            // the bit factors need only the projections: they are computed
            // while the summary MMAs still read the last features
            float sp[32];
            race_bits32(t + lane + colP + 64u * b + l0 * G, (l1 - l0) * G,
                        beta, sp);
            if (i >= 1 && writes)
                ok = wwait(&bars.phi_empty[hb], (i - 1) & 1, 68);
            if (!ok) break;
            const bool valid = c0 + i * 128 + row < c1;
            float buf[8];
#pragma unroll
            for (int lt = 0; lt < 32 / G; ++lt) {
                if (G == 4 && l0 + lt < l1) {
                    float u[4], w[4];
                    table_uw4(&sp[lt * G], valid ? 1.0f : 0.0f, u, w);
                    uint32_t pk[8];
                    table_pack4(u, w, pk);
                    const int cc = (l0 * R + lt * R) >> 3;
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh)
                        asm volatile(
                            "st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                                sPhi + panel_offset(row, cc + hh, 128)),
                            "r"(pk[4 * hh]), "r"(pk[4 * hh + 1]),
                            "r"(pk[4 * hh + 2]), "r"(pk[4 * hh + 3])
                            : "memory");
                } else if (l0 + lt < l1) {
                    float phi[R];
                    table_phi<G>(&sp[lt * G], phi);
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        const int prel = lt * R + q;  // l0 * R is 32-aligned
                        buf[prel & 7] = valid ? phi[q] : 0.0f;
                        if ((prel & 7) == 7)
                            st_shared_bf16x8(
                                sPhi + panel_offset(row, (l0 * R + prel) >> 3,
                                                    128),
                                buf);
                    }
                }
            }
            if (tail_owner) {
                if ((r & 7) != 0) {  // partial last chunk (< 8 buckets)
                    for (int q = r & 7; q < 8; ++q) buf[q] = 0.0f;
                    st_shared_bf16x8(sPhi + panel_offset(row, r >> 3, 128),
                                     buf);
                }
                for (int c = (r + 7) >> 3; c < (r_pad >> 3); ++c)
                    st_shared_zero16(sPhi + panel_offset(row, c, 128));
            }
            fence_proxy_async_smem();
            tc_fence_before();
            mbar_arrive(&bars.phi_full[half]);
        }
        // partial summaries of this chunk (each half: half the columns)
        float *out = part + ((size_t)bh * S + s) * ((size_t)r * d + r);
        if (ok && ntiles > 0) ok = wwait(&bars.done, 0, 69);
        if (ok && ntiles > 0) {
            tc_fence_after();
            for (int m = 0; m < nM; ++m) {
                const int rrow = m * 128 + row;
                for (int c = half * (d >> 1); c < (half + 1) * (d >> 1);
                     c += 32) {
                    uint32_t v[32];
                    tmem_ld32(t + lane + m * accN + c, v);
                    tmem_wait_ld();
                    if (rrow < r) {
                        float4 *dst = reinterpret_cast<float4 *>(
                            out + (size_t)rrow * d + c);
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            dst[j] = make_float4(
                                __uint_as_float(v[4 * j]),
                                __uint_as_float(v[4 * j + 1]),
                                __uint_as_float(v[4 * j + 2]),
                                __uint_as_float(v[4 * j + 3]));
                    }
                }
                if (half == 0) {
                    uint32_t a16[16];
                    tmem_ld16(t + lane + m * accN + d, a16);
                    tmem_wait_ld();
                    if (rrow < r)
                        out[(size_t)r * d + rrow] = __uint_as_float(a16[0]);
                }
            }
        } else if (ntiles == 0) {
            for (int i = tid - 64; i < r * d + r; i += 256) out[i] = 0.0f;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(t, tmem_cols);
}

// The same summaries for d = 128 and gamma = 4, with the product turned
// round: D = V^T Phi, lanes = value dimensions, N = r buckets, so that a tile
// takes 8 MMAs of N = r where Phi^T [V | 1] takes 16 of N = 144 (which ran at
// 80 ns each beside the copies and feature stores: shared-memory bandwidth),
// and the feature tile is handed over per 64 keys. A = Phi^T 1 comes from MMAs
// of N = 16 against ones in the same key steps, so that A and B are sums of the
// same unit and its truncations cancel in Num / Den. (Summed from the same
// features by four warps, with rounding to nearest, A is 2.4e-5 larger at
// N = 64K and d_lr off by 1.36e-4 there instead of 1.13e-4; c3 took 82 us and c4
// 340 so.) k_race_keys_ws took 103 and 412 us, this kernel takes 84 and 345, all
// live beside the sort hash. Roles and copies as above.
struct KtBars {
    uint64_t k_full[2], k_empty[2], v_full[2], v_empty[2], w_full, done;
    uint64_t proj_full[2];
    uint64_t phi_full[2], phi_empty[2];  // per 64 keys
};

template <int NT>  // tables per row half, 4 or 8 (L <= 2 NT)
__global__ void __launch_bounds__(kKwThreads, 1)
    k_race_keys_t(const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV,
                  const __grid_constant__ CUtensorMap tmW, int N, int H, int L,
                  int Lg_pad, int chunk, float beta, float *__restrict__ part,
                  DeviceStatus *status) {
    constexpr int d = 128;
    constexpr uint32_t tileB = 128u * d * 2u, colP = 256, colA = 384;
    extern __shared__ unsigned char smem_raw[];
    __shared__ KtBars bars;
    __shared__ uint32_t tbase;
    __shared__ int abort_flag;
    volatile int *abort = &abort_flag;
    const int s = blockIdx.x, bh = blockIdx.y, S = gridDim.x;
    const int h = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5, lane_id = tid & 31;
    const int r = 16 * L;
    const uint32_t sW = align1k(smem_u32(smem_raw));
    const uint32_t sK0 = sW + align1k(Lg_pad * d * 2);
    const uint32_t sV0 = sK0 + 2 * tileB;
    const uint32_t sOnes = sV0 + 2 * tileB;  // [16 x 64], B operand of A
    const uint32_t sPhi = sOnes + 2048;
    const int nM = (r + 127) >> 7;

    if (warp == 1) tmem_alloc(&tbase, 512);
    if (tid == 0) {
        mbar_init(&bars.done, 1);
        mbar_init(&bars.w_full, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars.k_full[b], 1);
            mbar_init(&bars.k_empty[b], 1);
            mbar_init(&bars.v_full[b], 1);
            mbar_init(&bars.v_empty[b], 1);
            mbar_init(&bars.proj_full[b], 1);
            mbar_init(&bars.phi_full[b], 128);
            mbar_init(&bars.phi_empty[b], 1);
        }
        abort_flag = 0;
        fence_mbar_init();
    }
    for (int i = tid; i < 2048 / 16; i += kKwThreads)  // bf16 ones
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                         sOnes + i * 16),
                     "r"(0x3F803F80u)
                     : "memory");
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t t = tbase;
    const int c0 = s * chunk;
    const int c1 = min(N, c0 + chunk);
    const int ntiles = c1 > c0 ? (c1 - c0 + 127) / 128 : 0;

    if (warp == 0) {
        // ------------------------------------------------------------- loader
        if (lane_id == 0 && ntiles > 0) {
            mbar_expect_tx(&bars.w_full, (uint32_t)Lg_pad * d * 2u);
            for (int pnl = 0; pnl < 2; ++pnl)
                tma_load_2d(sW + pnl * Lg_pad * 128, &tmW, 64 * pnl,
                            h * Lg_pad, &bars.w_full);
            // K(i) needs the projection of tile i - 2 done, V(i) the summary
            // MMAs of tile i - 2; V runs one tile behind K. Rows past the
            // chunk are loaded too (next head, or zeros past the tensor)
            // and get zero features.
            auto load = [&](int i, uint64_t *full, uint64_t *empty,
                            uint32_t dst, const CUtensorMap *map, int site) {
                const int b = i & 1;
                if (i >= 2 && !mbar_wait_or_abort(&empty[b],
                                                  ((i >> 1) - 1) & 1, abort,
                                                  status, site))
                    return false;
                mbar_expect_tx(&full[b], tileB);
                for (int pnl = 0; pnl < 2; ++pnl)
                    tma_load_2d(dst + b * tileB + pnl * 16384, map, 64 * pnl,
                                bh * N + c0 + i * 128, &full[b]);
                return true;
            };
            for (int i = 0; i <= ntiles; ++i) {
                if (i < ntiles &&
                    !load(i, bars.k_full, bars.k_empty, sK0, &tmK, 101))
                    break;
                if (i > 0 &&
                    !load(i - 1, bars.v_full, bars.v_empty, sV0, &tmV, 102))
                    break;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ----------------------------------------------------------- MMA issue
        if (ntiles > 0) {
            // the whole warp runs the loop (its state and the operands'
            // descriptors are warp-uniform); one lane issues
            const bool el = elect_one();
            auto wait = [&](uint64_t *bar, uint32_t par, int site) -> bool {
                return __all_sync(0xffffffffu,
                                  mbar_wait_or_abort(bar, par, abort, status,
                                                     site));
            };
            const uint32_t id_proj = idesc_bf16(128, Lg_pad, false, false);
            const uint32_t id_b = idesc_bf16(128, r, true, true);
            const uint32_t id_a = idesc_bf16(128, 16, true, false);
            const uint64_t d1 = smem_desc(sOnes, 16, 1024);
            auto proj = [=](int it) {
                const uint32_t sK = sK0 + (it & 1) * tileB;
                const uint32_t dst = t + colP + 64u * (it & 1);
                const uint64_t a = smem_desc(sK, 16, 1024),
                               b = smem_desc(sW, 16, 1024);
                if (!el) return;
#pragma unroll
                for (int k = 0; k < d / 16; ++k)
                    mma_ss(dst, desc_at(a, (k >> 2) * 16384 + (k & 3) * 32),
                           desc_at(b, (uint32_t)(k >> 2) * Lg_pad * 128 +
                                          (k & 3) * 32),
                           id_proj, k > 0);
                mma_commit(&bars.proj_full[it & 1]);
                mma_commit(&bars.k_empty[it & 1]);
            };
            // projections run two tiles ahead (both TMEM buffers)
            bool ok = wait(&bars.w_full, 0, 100);
            for (int it = 0; it < 2 && it < ntiles && ok; ++it) {
                ok = wait(&bars.k_full[it], 0, 103);
                if (ok) {
                    tc_fence_after();
                    proj(it);
                }
            }
            for (int i = 0; i < ntiles && ok; ++i) {
                const int b = i & 1;
                ok = wait(&bars.v_full[b], (i >> 1) & 1, 106);
                for (int kh = 0; kh < 2 && ok; ++kh) {
                    ok = wait(&bars.phi_full[kh], i & 1, 105);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t da = smem_desc(sV0 + b * tileB + kh * 8192,
                                                  16384, 1024),
                                   db = smem_desc(sPhi + kh * 8192, 16384,
                                                  1024);
                    const uint32_t more = i > 0 || kh > 0;
                    if (el) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)  // 16 keys each
                            mma_ss(t, desc_at(da, k * 2048),
                                   desc_at(db, k * 2048), id_b,
                                   k > 0 ? 1u : more);
#pragma unroll
                        for (int m = 0; m < 2; ++m)
                            if (m < nM)
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    mma_ss(t + colA + 16 * m,
                                           desc_at(db, m * 32768 + k * 2048),
                                           d1, id_a, k > 0 ? 1u : more);
                        mma_commit(&bars.phi_empty[kh]);
                    }
                }
                if (!ok) break;
                if (el) mma_commit(&bars.v_empty[b]);
                if (i + 2 < ntiles) {
                    // the features of tile i have read projection buffer b
                    ok = wait(&bars.k_full[b], ((i + 2) >> 1) & 1, 104);
                    if (!ok) break;
                    tc_fence_after();
                    proj(i + 2);
                }
            }
            if (ok && el) mma_commit(&bars.done);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ features
        const int half = (warp - 2) >> 2;
        const int row = (warp & 3) * 32 + lane_id;  // key row = TMEM lane
        const int kh = row >> 6;
        const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
        const int l0 = min(half * NT, L), nt = min(l0 + NT, L) - l0;
        auto wwait = [=](uint64_t *bar, uint32_t par, int site) {
            return __all_sync(0xffffffffu,
                              mbar_wait_or_abort(bar, par, abort, status,
                                                 site));
        };
        bool ok = true;
        for (int i = 0; i < ntiles; ++i) {
            const int b = i & 1;
            ok = wwait(&bars.proj_full[b], (i >> 1) & 1, 107);
            if (!ok) break;
            tc_fence_after();
            float sp[NT * 4];
            if constexpr (NT == 8) {
                uint32_t pr[32];
                tmem_ld32(t + lane + colP + 64u * b + l0 * 4, pr);
                tmem_wait_ld();
                race_factors<32>(pr, beta, sp);
            } else {
                uint32_t pr[16];
                tmem_ld16(t + lane + colP + 64u * b + l0 * 4, pr);
                tmem_wait_ld();
                race_factors<16>(pr, beta, sp);
            }
            if (i >= 1) ok = wwait(&bars.phi_empty[kh], (i - 1) & 1, 108);
            if (!ok) break;
            const float one = c0 + i * 128 + row < c1 ? 1.0f : 0.0f;
#pragma unroll
            for (int lt = 0; lt < NT; ++lt) {
                if (lt < nt) {
                    float u[4], w[4];
                    table_uw4(&sp[lt * 4], one, u, w);
                    uint32_t pk[8];
                    table_pack4(u, w, pk);
                    const uint32_t cc = (uint32_t)(l0 + lt) * 2;
                    st_shared_v4(sPhi + panel_offset(row, cc, 128), pk[0],
                                 pk[1], pk[2], pk[3]);
                    st_shared_v4(sPhi + panel_offset(row, cc + 1, 128), pk[4],
                                 pk[5], pk[6], pk[7]);
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            mbar_arrive(&bars.phi_full[kh]);
        }
        // partial summaries of this chunk: lane = value dimension; the
        // halves take every other 16 buckets
        float *out = part + ((size_t)bh * S + s) * ((size_t)r * d + r);
        if (ok && ntiles > 0) ok = wwait(&bars.done, 0, 109);
        if (ok && ntiles > 0) {
            tc_fence_after();
            for (int c = half; c < L; c += 2) {
                uint32_t v[16];
                tmem_ld16(t + lane + 16 * c, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    out[(size_t)(16 * c + j) * d + row] =
                        __uint_as_float(v[j]);
            }
            if (half < nM) {  // lane = bucket of tile `half`
                uint32_t v[16];
                tmem_ld16(t + lane + colA + 16 * half, v);
                tmem_wait_ld();
                const int bucket = 128 * half + row;
                if (bucket < r)
                    out[(size_t)r * d + bucket] = __uint_as_float(v[0]);
            }
        } else if (ntiles == 0) {
            for (int i = tid - 64; i < r * d + r; i += 256) out[i] = 0.0f;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(t, 512);
}

uint32_t pow2_cols_kw(uint32_t n) {
    uint32_t c = 32;
    while (c < n) c <<= 1;
    return c;
}

}  // namespace

size_t race_keys_ws_smem(const Plan &P) {
    const size_t r_pad = (P.r + 127) / 128 * 128;
    const size_t lg_pad = (P.L * P.gamma + 15) / 16 * 16;
    return 1024 + (lg_pad * P.d * 2 + 1023) / 1024 * 1024 +
           (P.d == 128 ? 4 : 3) * (size_t)128 * P.d * 2 + 16384 +
           128 * r_pad * 2;
}

uint32_t race_keys_ws_cols(const Plan &P) {
    const int r_pad = (P.r + 127) / 128 * 128;
    return pow2_cols_kw((r_pad / 128) * (P.d + 16) + 128);
}

namespace {
__global__ void k_prep_planes(const float *__restrict__ w, int H, int Lg,
                              int Lg_pad, int d, uint16_t *__restrict__ out,
                              DeviceStatus *status) {
    const long n = (long)H * Lg_pad * d;
    if (status && blockIdx.x == 0 && threadIdx.x < 4)
        reinterpret_cast<int *>(status)[threadIdx.x] = 0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n;
         i += (long)gridDim.x * blockDim.x) {
        const int c = (int)(i % d);
        const long hr = i / d;
        const int row = (int)(hr % Lg_pad), h = (int)(hr / Lg_pad);
        const float x = row < Lg ? w[((long)h * Lg + row) * d + c] : 0.0f;
        const __nv_bfloat16 b = __float2bfloat16_rn(x);
        out[i] = *reinterpret_cast<const uint16_t *>(&b);
    }
}
}  // namespace

cudaError_t launch_prep_planes(const Plan &P, const float *w_race,
                               uint16_t *w_bf16, cudaStream_t st) {
    return launch_begin(P, w_race, w_bf16, nullptr, st);
}

cudaError_t launch_begin(const Plan &P, const float *w_race, uint16_t *w_bf16,
                         DeviceStatus *status, cudaStream_t st) {
    static_assert(sizeof(DeviceStatus) == 16, "four ints");
    const long n = (long)P.H * P.Lg_pad * P.d;
    const int blocks = (int)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
    k_prep_planes<<<blocks, 256, 0, st>>>(w_race, P.H, P.L * P.gamma,
                                          P.Lg_pad, P.d, w_bf16, status);
    return cudaGetLastError();
}

namespace {
__global__ void k_clear(int *status, int *zero, int n) {
    if (threadIdx.x < 4) status[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) zero[i] = 0;
}
}  // namespace

cudaError_t launch_clear(DeviceStatus *status, int *zero, int n,
                         cudaStream_t st) {
    k_clear<<<1, 32, 0, st>>>(reinterpret_cast<int *>(status), zero, n);
    return cudaGetLastError();
}

cudaError_t launch_race_keys_ws(const Plan &P, const void *k, const void *v,
                                const uint16_t *w_bf16, float *part,
                                DeviceStatus *status, cudaStream_t st) {
    const int r_pad = (P.r + 127) / 128 * 128;
    const int lg_pad = (P.L * P.gamma + 15) / 16 * 16;
    const uint32_t cols = race_keys_ws_cols(P);
    const size_t need = race_keys_ws_smem(P);
    // cap residency at what TMEM allows
    const int fit = 512 / (int)cols;
    const size_t cap = (size_t)233472 / (fit + 1) + 1;
    const size_t smem = need > cap ? need : cap;
    dim3 grid(P.S, P.BH);
    CUtensorMap tmK, tmV, tmW;
    const uint64_t rows = (uint64_t)P.BH * P.N;
    cudaError_t e = make_tma_map_bf16(&tmK, k, rows, P.d, 128);
    if (e == cudaSuccess) e = make_tma_map_bf16(&tmV, v, rows, P.d, 128);
    if (e == cudaSuccess)
        e = make_tma_map_bf16(&tmW, w_bf16, (uint64_t)P.H * P.Lg_pad, P.d,
                              (uint32_t)P.Lg_pad);
    if (e != cudaSuccess) return e;
    auto launch = [&](auto kern) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
        kern<<<grid, kKwThreads, smem, st>>>(
            tmK, tmV, tmW, P.N, P.d, P.H, P.L, r_pad, lg_pad, P.chunk,
            P.beta, cols, part, status);
        return cudaGetLastError();
    };
    if (P.d == 128 && P.gamma == 4) {
        const size_t sm = 1024 + (size_t)lg_pad * P.d * 2 +
                          4 * (size_t)128 * P.d * 2 + 2048 +
                          (size_t)((P.r + 127) / 128) * 32768;
        auto launch_t = [&](auto kern) {
            cudaFuncSetAttribute(
                kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
            kern<<<grid, kKwThreads, sm, st>>>(tmK, tmV, tmW, P.N, P.H, P.L,
                                               lg_pad, P.chunk, P.beta, part,
                                               status);
            return cudaGetLastError();
        };
        return P.L > 8 ? launch_t(k_race_keys_t<8>)
                       : launch_t(k_race_keys_t<4>);
    }
    switch (P.gamma) {
        case 1: return launch(k_race_keys_ws<1>);
        case 2: return launch(k_race_keys_ws<2>);
        case 3: return launch(k_race_keys_ws<3>);
        case 4: return launch(k_race_keys_ws<4>);
        case 5: return launch(k_race_keys_ws<5>);
        case 6: return launch(k_race_keys_ws<6>);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace elsaa
