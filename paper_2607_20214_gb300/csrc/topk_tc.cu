// Per-query top-k selection on the tensor cores (selector = 1, bf16, key
// blocks of a multiple of 128): the same key sets as k_topk_select.
//
// The decision is defined in the canonical fp32 chain e_ij = <q_i, k_j>.
// One CTA per 128 sorted queries computes every score s_ij of its c b
// candidates with tcgen05 MMAs (bf16 products are exact in fp32; only the
// order and rounding of the sum differ from the chain), and a thread per
// query row searches a threshold T with exactly k scores >= T. With
// |s - e| <= E for every candidate of a row,
//   s > T + 2E  =>  e is among the k largest (at most k scores exceed s - 2E)
//   s < T - 2E  =>  it is not (k scores lie above T, whose e exceed this e)
// so only candidates within 2E of T are scored again with the canonical
// chain, and only if they do not all fit (or all fall). The search may stop
// anywhere with a bracket lo <= T < hi (count(>= lo) >= k > count(>= hi));
// the window is then [lo - 2E, hi + 2E].
//
// E = 2^-15 |q| max|k| = 3.05e-5 of it. The chain's own error is at most
// d 2^-24 sum|q k| <= 2^-17 |q| |k| at d = 128 (7.6e-6). For the MMA it is
// assumed, as its additions are not documented, that each of the 8 steps
// aligns 16 products and the accumulator to the largest of them, truncates
// every term at 2^-23 of it or finer and the sum once more: at most 8 * 18 *
// 2^-23 |q| |k| (1.72e-5). Together 2.48e-5, so E has a margin of 1.2 over what
// is assumed; samples are well inside (the largest |s - e| / (|q| |k|) of 2^26
// scores per distribution: 2^-22.3 Gaussian, 2^-20.5 with exponents spread
// over 2^24, 2^-19.6 with two elements holding the norm). Rows whose norms
// are not finite, overflow in their squares or are below 1e-15 (where squares
// and products underflow) are selected by the chain alone.
//
// What bounds it: the issue slots of the search (about five passes over the
// scores at 1.5 FP32 instructions each, one more that makes the masks). Two
// persistent CTAs per SM; the next tile's rows are copied while the current
// tile is searched (the panels are free once its MMAs are done), in strided
// tile order, so that the CTAs work on two or three heads at a time, whose
// keys stay in L2. The CUDA-core kernel is bound by the 2 d FMAs of every
// score instead. Measured at B2 H16 N16384 d128 b128 c2 k128: 206 us against
// 1434 us (227 us when the search stops at 48 open scores, 245 us when it goes
// on to none; 246 us without the copy-ahead).
#include "device_common.cuh"
#include "tc_common.cuh"

namespace elsaa {

namespace {

using namespace tc;

constexpr int kTselThreads = 256;
constexpr int kTselList = 64;    // open candidates of 32 rows, one lane each
// The search ends with at most so many open candidates: 10, 20 and 40 take
// 209, 210 and 223 us at 256 candidates a row, 145, 143 and 151 at 128, 400,
// 390 and 414 at 384, 487, 492 and 530 at 512 (B2 H16 N16384 d128).
constexpr int kTselLeft = 20;
constexpr int kTselRowMax = 8;   // of one row; more: the row's own pass
constexpr int kTselSteps = 48;   // search steps before the bracket is taken

__device__ __forceinline__ uint32_t score_key(float f) {
    if (f == 0.0f) f = 0.0f;  // -0 is taken as +0
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// tcgen05.wait::ld that also carries the loaded registers, so that nothing
// reads them before it.
__device__ __forceinline__ void wait_ld_regs(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]),
                   "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                   "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
                   "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]),
                   "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]),
                   "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

// Calls f(chunk, scores) for the row's NC scores, 32 at a time, the next
// 32 on their way from tensor memory meanwhile. Whole warps.
template <int NC, typename F>
__device__ __forceinline__ void for_scores(uint32_t taddr, F f) {
    uint32_t a[32], b[32];
    tmem_ld32(taddr, a);
    wait_ld_regs(a);
#pragma unroll 1
    for (int c = 0; c < NC / 32; c += 2) {
        tmem_ld32(taddr + (c + 1) * 32, b);
        f(c, a);
        wait_ld_regs(b);
        if (c + 2 < NC / 32) tmem_ld32(taddr + (c + 2) * 32, a);
        f(c + 1, b);
        wait_ld_regs(a);
    }
}

// The canonical chain of two rows of d bf16 values, 64 values in flight.
__device__ __forceinline__ float row_chain(const uint16_t *__restrict__ a,
                                           const uint16_t *__restrict__ b,
                                           int d) {
    float acc = 0.0f;
    for (int e = 0; e < d; e += 64) {
        uint4 x[8], y[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            x[i] = *reinterpret_cast<const uint4 *>(a + e + 8 * i);
            y[i] = *reinterpret_cast<const uint4 *>(b + e + 8 * i);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t xw[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
            const uint32_t yw[4] = {y[i].x, y[i].y, y[i].z, y[i].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc = fmaf(__uint_as_float(xw[j] << 16),
                           __uint_as_float(yw[j] << 16), acc);
                acc = fmaf(__uint_as_float(xw[j] & 0xffff0000u),
                           __uint_as_float(yw[j] & 0xffff0000u), acc);
            }
        }
    }
    return acc;
}

// Persistent CTAs over the B H N / 128 tiles of 128 sorted queries. norms
// [2][BH][N]: squared norms of the queries and keys by sorted position
// (k_topk_sums).
template <int NC>
__global__ void __launch_bounds__(kTselThreads, NC <= 256 ? 2 : 1)
    k_topk_select_tc(const uint16_t *__restrict__ qx,
                     const uint16_t *__restrict__ kx,
                     const int32_t *__restrict__ perm_q,
                     const int32_t *__restrict__ perm_k,
                     const int32_t *__restrict__ cand,
                     const float *__restrict__ norms, int BH, int N, int d,
                     int b, int c, int k, uint32_t *__restrict__ selmask,
                     DeviceStatus *status) {
    constexpr int M = NC / 32;
    constexpr uint32_t kCols = NC <= 128 ? 128 : NC <= 256 ? 256 : 512;
    extern __shared__ unsigned char tsel_raw[];
    __shared__ int kidx[2][NC], qidx[2][128];  // by tile parity
    // per pair of warps: the halves' score sums, then the open candidates
    __shared__ __align__(16) uint32_t scratch[4][2 * kTselList];
    __shared__ uint32_t keepw[4][2];
    __shared__ int nneed[4][32];
    __shared__ float part[2][2][128];  // counts of each half, per row
    __shared__ uint32_t words[4][2][M];
    __shared__ uint32_t tmem_base, kmax_bits[2];
    __shared__ __align__(8) uint64_t bar;
    const int T = N / b, per = N / 128, tiles = BH * per;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t sq = (smem_u32(tsel_raw) + 1023u) & ~1023u;
    const uint32_t sk = sq + 128 * d * 2;
    const int cpr = d / 8;  // 16-byte chunks per row
    if (tid == 0) {
        kmax_bits[0] = kmax_bits[1] = 0;
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, kCols);
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tmem_base;
    // A warp resolves 32 rows at a time (4 groups of queries, then M of
    // candidates) and copies them, whole rows per instruction. The row
    // numbers are read a tile ahead.
    constexpr int kGroups = (M + 4 + 7) / 8;  // per warp
    int rowno[kGroups];
    uint32_t kmax = 0;
    auto read_rows = [&](int tile) {
        const int bh = tile / per, p0 = (tile - bh * per) * 128, t = p0 / b;
        const int32_t *cb = cand + ((size_t)bh * T + t) * c;
        kmax = 0;
#pragma unroll
        for (int x = 0; x < kGroups; ++x) {
            const int grp = warp + 8 * x;
            if (grp >= M + 4) break;
            const int r = (grp < 4 ? grp : grp - 4) * 32 + lane;
            if (grp < 4) {
                rowno[x] = perm_q[(size_t)bh * N + p0 + r];
            } else {
                int u = cb[r / b];
                if (u < 0 || u >= T) u = t;
                const int p = u * b + r % b;
                rowno[x] = perm_k[(size_t)bh * N + p];
                kmax = max(kmax, __float_as_uint(
                                     norms[(size_t)(BH + bh) * N + p]));
            }
        }
    };
    auto gather = [&](int tile, int par) {
        const int bh = tile / per;
        const int ch = lane & (cpr - 1), rpi = 32 / cpr, sub = lane / cpr;
#pragma unroll
        for (int x = 0; x < kGroups; ++x) {
            const int grp = warp + 8 * x;
            if (grp >= M + 4) break;
            const bool isq = grp < 4;
            const int r0 = (isq ? grp : grp - 4) * 32;
            int j = rowno[x];
            if (j < 0 || j >= N) {
                report(status, kDevPermRange, isq ? 22 : 21, bh, j);
                j = 0;
            }
            (isq ? qidx[par] : kidx[par])[r0 + lane] = j;
            const uint16_t *src =
                (isq ? qx : kx) + (size_t)bh * N * d + 8 * ch;
            const uint32_t to = isq ? sq : sk;
            const int rows = isq ? 128 : NC;
#pragma unroll 4
            for (int i = sub; i < 32; i += rpi) {
                const int jr = __shfl_sync(0xffffffffu, j, i);
                cp_async16(to + panel_offset(r0 + i, ch, rows),
                           src + (size_t)jr * d);
            }
        }
        // the largest key norm (as bits: NaN and infinity sort above every
        // finite norm)
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        if (lane == 0) atomicMax(&kmax_bits[par], kmax);
        cp_async_commit();
    };
    const int g = warp & 3, half = warp >> 2, row = g * 32 + lane;
    const uint32_t taddr = tm + ((uint32_t)(g * 32) << 16) + half * (NC / 2);
    auto pair_sync = [&] { named_sync(1 + g, 64); };
    int par = 0, phase = 0;
    if ((int)blockIdx.x < tiles) {
        read_rows(blockIdx.x);
        gather(blockIdx.x, 0);
    }
    for (int tile = blockIdx.x; tile < tiles;
         tile += gridDim.x, par ^= 1, phase ^= 1) {
        const int bh = tile / per, p0 = (tile - bh * per) * 128;
        const uint16_t *qh = qx + (size_t)bh * N * d;
        const uint16_t *kh = kx + (size_t)bh * N * d;
        const int *cidx = kidx[par];
        const int next = tile + (int)gridDim.x;
        if (next < tiles) read_rows(next);
        cp_async_wait<0>();
        fence_proxy_async_smem();
        tc_fence_before();  // the last tile's scores have been read
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
            kmax_bits[par ^ 1] = 0;  // the next gather's
            for (int n0 = 0; n0 < NC; n0 += 256) {
                const int n = NC - n0 < 256 ? NC - n0 : 256;
                const uint32_t idesc = idesc_bf16(128, n, false, false);
                for (int ks = 0; ks < d / 16; ++ks) {
                    const uint32_t in = (uint32_t)(ks & 3) * 32;
                    mma_ss(
                        tm + n0,
                        smem_desc(sq + (ks >> 2) * 128 * 128 + in, 16, 1024),
                        smem_desc(sk + (ks >> 2) * NC * 128 + n0 * 128 + in,
                                  16, 1024),
                        idesc, ks > 0);
                }
            }
            mma_commit(&bar);
        }
        const float qn = norms[(size_t)bh * N + p0 + row];
        const float kn = __uint_as_float(kmax_bits[par]);
        bool ok = mbar_wait(&bar, phase, status, 170);
        if (!__syncthreads_and(ok)) break;
        tc_fence_after();
        if (next < tiles) gather(next, par ^ 1);
        // Warps g and g + 4 share rows 32 g ..: half h of the columns each.
        // Both take every decision from the same combined counts.
        // win = 2E and the counting's own blur; the row is decided by the
        // chain alone unless its norms are ordinary numbers
        const float reach = sqrtf(qn) * sqrtf(kn);  // |s| <= reach
        const float win = reach * 6.104e-5f * 1.02f + 1e-30f;
        const bool chain_only =
            !(qn >= 1e-30f && kn >= 1e-30f && win <= 1e30f);
        float lo = -1.01f * reach, hi = 1.01f * reach;
        float clo = NC, chi = 0;  // counts above lo and hi
        int sides = 0;            // 1: lo is a counted tt, 2: hi is
        float tt, slope;
        {
            float2 s1 = make_float2(0.f, 0.f), s2 = s1;
            for_scores<NC / 2>(taddr, [&](int, const uint32_t(&s)[32]) {
#pragma unroll
                for (int i = 0; i < 32; i += 2) {
                    const float2 v = make_float2(__uint_as_float(s[i]),
                                                 __uint_as_float(s[i + 1]));
                    s1 = add2(s1, v);
                    s2 = fma2(v, v, s2);
                }
            });
            float2 *stat = reinterpret_cast<float2 *>(scratch[g]);
            const float2 mine = make_float2(s1.x + s1.y, s2.x + s2.y);
            pair_sync();  // the last tile's lists have been read
            stat[half * 32 + lane] = mine;
            pair_sync();
            const float2 o = stat[(half ^ 1) * 32 + lane];
            const float mean = (mine.x + o.x) * (1.0f / NC);
            const float sd = sqrtf(fmaxf(
                fmaf(mine.y + o.y, 1.0f / NC, -mean * mean), 0.0f));
            // a normal quantile to begin with, and the spacing there
            const float z = normcdfinvf(1.0f - (k - 0.5f) / NC);
            tt = fmaf(z, sd, mean);
            slope = sd * 2.5066283f * __expf(0.5f * z * z) * (1.0f / NC);
        }
        // The bracket is narrowed until the rows of the warp together have
        // few enough scores inside for the chain pass below (a row with
        // exactly k scores above tt has none): about four steps, where
        // going on to an exact split of every row takes nine.
        bool done = chain_only || k == NC;
        for (int step = 0; step < kTselSteps; ++step) {
            if (!(tt > lo && tt < hi)) tt = 0.5f * lo + 0.5f * hi;
            if (!(tt > lo && tt < hi) || hi - lo <= 0.25f * win) done = true;
            const int left = done ? 0 : (int)ceilf(clo - chi);
            if (__reduce_add_sync(0xffffffffu, left) <= kTselLeft &&
                __all_sync(0xffffffffu, left <= kTselRowMax))
                break;
            // scores above tt: (s - tt) 512 / win clamped to [0, 1], so a
            // score within win / 512 of tt may count in part
            const float big = 512.0f / win, off0 = -tt * big;
            float2 n0 = make_float2(0.f, 0.f), n1 = n0;
            for_scores<NC / 2>(taddr, [&](int, const uint32_t(&s)[32]) {
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    float f[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        f[x] = __saturatef(
                            fmaf(__uint_as_float(s[i + x]), big, off0));
                    n0 = add2(n0, make_float2(f[0], f[1]));
                    n1 = add2(n1, make_float2(f[2], f[3]));
                }
            });
            const float own = (n0.x + n0.y) + (n1.x + n1.y);
            part[step & 1][half][row] = own;
            pair_sync();
            if (!done) {
                const float cnt = own + part[step & 1][half ^ 1][row];
                const float off = cnt - k;
                if (off == 0.0f) {
                    lo = hi = tt;
                    done = true;
                } else {
                    if (off > 0.0f) {
                        lo = tt;
                        clo = cnt;
                        sides |= 1;
                    } else {
                        hi = tt;
                        chi = cnt;
                        sides |= 2;
                    }
                    if (step < 2 || sides != 3) {
                        // past the target by the count's own spread, so
                        // that the other side of the bracket closes too
                        float more;
                        asm("sqrt.approx.f32 %0, %1;"
                            : "=f"(more)
                            : "f"(fabsf(off)));
                        tt = fmaf(off + copysignf(0.7f * more, off), slope,
                                  tt);
                        if (step > 2) slope *= 2.0f;
                    } else if ((step & 3) == 3) {
                        tt = 0.5f * lo + 0.5f * hi;
                    } else {
                        tt = lo + (hi - lo) * __fdividef(clo - k, clo - chi);
                    }
                }
            }
        }
        // certain candidates and those within the window
        constexpr int MH = M / 2;  // mask words of this half
        uint32_t out[MH], amb[MH];
        const float above = hi + win, below = lo - win;
        int n_in = 0, n_amb = 0;
        for_scores<NC / 2>(taddr, [&](int ch, const uint32_t(&s)[32]) {
            uint32_t w0 = 0, w1 = 0;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const float v = __uint_as_float(s[i]);
                w0 = __funnelshift_l(__float_as_uint(above - v), w0, 1);
                w1 = __funnelshift_l(__float_as_uint(v - below), w1, 1);
            }
            w0 = __brev(w0);
            w1 = __brev(~w1) & ~w0;
            if (chain_only) {
                w0 = 0u;
                w1 = 0xffffffffu;
            }
            if (k == NC) {
                w0 = 0xffffffffu;
                w1 = 0u;
            }
#pragma unroll
            for (int m = 0; m < MH; ++m)
                if (m == ch) {
                    out[m] = w0;
                    amb[m] = w1;
                }
            n_in += __popc(w0);
            n_amb += __popc(w1);
        });
        pair_sync();  // the last step's counts have been read
        part[0][half][row] = __int_as_float(n_in | n_amb << 16);
        pair_sync();
        const int other = __float_as_int(part[0][half ^ 1][row]);
        const int amb0 = half ? other >> 16 : n_amb;  // of the lower half
        const int all_amb = n_amb + (other >> 16);
        const int need = k - n_in - (other & 0xffff);
        const bool all_fit = all_amb <= need;
        if (all_fit) {
#pragma unroll
            for (int m = 0; m < MH; ++m) out[m] |= amb[m];
        }
        const bool open = !all_fit && need > 0;
        // rows with a few open candidates: one lane per candidate
        int mine = open && all_amb <= kTselRowMax ? all_amb : 0;
        int at = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += x;
        }
        at -= mine;
        if (at + mine > kTselList) mine = 0;
        const int total =
            __reduce_max_sync(0xffffffffu, mine ? at + mine : 0);
        uint32_t *list = scratch[g], *lkey = scratch[g] + kTselList;
        if (mine) {
            // entry: row start and length in the list, row, candidate
            int e = at + (half ? amb0 : 0);
#pragma unroll
            for (int m = 0; m < MH; ++m)
                for (uint32_t w = amb[m]; w; w &= w - 1)
                    list[e++] = (uint32_t)at << 24 | (uint32_t)mine << 16 |
                                (uint32_t)lane << 10 |
                                (uint32_t)(half * (NC / 2) + 32 * m +
                                           __ffs(w) - 1);
            if (!half) nneed[g][lane] = need;
        }
        pair_sync();
        const int mye = half * 32 + lane;
        uint32_t key0 = 0, ent = 0;
        if (mye < total) {
            ent = list[mye];
            key0 = score_key(row_chain(
                qh + (size_t)qidx[par][g * 32 + (ent >> 10 & 31)] * d,
                kh + (size_t)cidx[ent & 1023] * d, d));
            lkey[mye] = key0;
        }
        pair_sync();
        bool keep = false;
        if (mye < total) {
            const int from = ent >> 24, n = ent >> 16 & 255;
            int better = 0;
            for (int x = from; x < from + n; ++x) {
                const uint32_t kx2 = lkey[x];
                better += kx2 > key0 ||
                          (kx2 == key0 &&
                           cidx[list[x] & 1023] < cidx[ent & 1023]);
            }
            keep = better < nneed[g][ent >> 10 & 31];
        }
        const uint32_t kept = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) keepw[g][half] = kept;
        pair_sync();
        if (mine) {
            int e = at + (half ? amb0 : 0);
#pragma unroll
            for (int m = 0; m < MH; ++m)
                for (uint32_t w = amb[m]; w; w &= w - 1, ++e)
                    if (keepw[g][e >> 5] >> (e & 31) & 1u)
                        out[m] |= w & (0u - w);
        }
        // rows with many: a warp scores all of a row's open candidates and
        // searches the need-th largest key, then (ties) the index limit;
        // the two warps of the pair take a row each
        uint32_t rest = __ballot_sync(0xffffffffu, open && !mine);
        while (rest) {
            const int r0 = __ffs(rest) - 1;
            rest &= rest - 1;
            const int r1 = rest ? __ffs(rest) - 1 : -1;
            if (rest) rest &= rest - 1;
            uint32_t *slot = words[g][lane == r1];
            if (lane == r0 || lane == r1) {
#pragma unroll
                for (int m = 0; m < MH; ++m) slot[half * MH + m] = amb[m];
            }
            pair_sync();
            const int src = half ? r1 : r0;
            if (src >= 0) {
                uint32_t *mw = words[g][half];
                const int nd = __shfl_sync(0xffffffffu, need, src);
                uint32_t key[M];
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    key[m] = 0u;
                    if ((mw[m] >> lane) & 1u)
                        key[m] = score_key(row_chain(
                            qh + (size_t)qidx[par][g * 32 + src] * d,
                            kh + (size_t)cidx[32 * m + lane] * d, d));
                }
                uint32_t pre = 0;
                for (int bit = 31; bit >= 0; --bit) {
                    const uint32_t want = pre | 1u << bit;
                    int n = 0;
#pragma unroll
                    for (int m = 0; m < M; ++m) n += key[m] >= want;
                    if (__reduce_add_sync(0xffffffffu, n) >= nd) pre = want;
                }
                int gt = 0, eq = 0;
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    gt += key[m] > pre;
                    eq += key[m] == pre;
                }
                gt = __reduce_add_sync(0xffffffffu, gt);
                eq = __reduce_add_sync(0xffffffffu, eq);
                int jmax = 0x7fffffff;
                if (eq > nd - gt) {
                    uint32_t jp = 0, jm = 0;
                    int under = 0;
                    for (int bit = 30; bit >= 0; --bit) {
                        const uint32_t bm = 1u << bit, mk = jm | bm;
                        int n = 0;  // ties whose index has this bit clear
#pragma unroll
                        for (int m = 0; m < M; ++m)
                            n += key[m] == pre &&
                                 ((uint32_t)cidx[32 * m + lane] & mk) == jp;
                        n = __reduce_add_sync(0xffffffffu, n);
                        if (under + n < nd - gt) {
                            under += n;
                            jp |= bm;
                        }
                        jm = mk;
                    }
                    jmax = (int)jp;
                }
                __syncwarp();
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const bool sel = key[m] > pre ||
                                     (key[m] == pre && pre != 0u &&
                                      cidx[32 * m + lane] <= jmax);
                    const uint32_t w = __ballot_sync(0xffffffffu, sel);
                    if (lane == 0) mw[m] = w;
                }
            }
            pair_sync();
            if (lane == r0 || lane == r1) {
#pragma unroll
                for (int m = 0; m < MH; ++m) out[m] |= slot[half * MH + m];
            }
            // the next rows' lanes write the words that these have read
            __syncwarp();
        }
        uint32_t *dst =
            selmask + ((size_t)bh * N + p0 + row) * M + half * MH;
#pragma unroll
        for (int m = 0; m < MH; m += 2)
            *reinterpret_cast<uint2 *>(dst + m) =
                make_uint2(out[m], out[m + 1]);
    }
    cp_async_wait<0>();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tm, kCols);
}

template <int NC>
cudaError_t run_select_tc(const Plan &P, const void *q, const void *k,
                          const int32_t *perm_q, const int32_t *perm_k,
                          const int32_t *cand, const float *norms,
                          uint32_t *selmask, DeviceStatus *status,
                          cudaStream_t st) {
    const int smem = 1024 + (NC + 128) * P.d * 2;
    auto kern = k_topk_select_tc<NC>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         smem);
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long tiles = (long)P.BH * (P.N / 128);
    const long slots = (NC <= 256 ? 2 : 1) * (long)sms;
    kern<<<(int)(tiles < slots ? tiles : slots), kTselThreads, smem, st>>>(
        (const uint16_t *)q, (const uint16_t *)k, perm_q, perm_k, cand, norms,
        P.BH, P.N, P.d, P.b, P.tk_c, P.tk_k, selmask, status);
    return cudaGetLastError();
}

}  // namespace

// bf16 with d_h of 64 or 128 (whole swizzled panels) and blocks of whole
// 128-query tiles; c b <= 512 fp32 scores per row fill at most the 512
// columns of tensor memory. Smaller blocks have fewer than 128 queries per
// candidate set and stay on the CUDA cores.
bool topk_tc_supported(const Plan &P) {
    return P.impl == 2 && P.dtype == ELSAA_BF16 &&
           (P.d == 64 || P.d == 128) && P.b % 128 == 0 &&
           P.tk_c * P.b <= 512;
}

cudaError_t launch_topk_select_tc(const Plan &P, const void *q, const void *k,
                                  const int32_t *perm_q,
                                  const int32_t *perm_k, const int32_t *cand,
                                  const float *norms, uint32_t *selmask,
                                  DeviceStatus *status, cudaStream_t st) {
    switch (P.tk_c * P.b) {
        case 128:
            return run_select_tc<128>(P, q, k, perm_q, perm_k, cand, norms,
                                      selmask, status, st);
        case 256:
            return run_select_tc<256>(P, q, k, perm_q, perm_k, cand, norms,
                                      selmask, status, st);
        case 384:
            return run_select_tc<384>(P, q, k, perm_q, perm_k, cand, norms,
                                      selmask, status, st);
        case 512:
            return run_select_tc<512>(P, q, k, perm_q, perm_k, cand, norms,
                                      selmask, status, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace elsaa
