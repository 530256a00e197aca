// Runs PairOrder, the issue order of the CTA-pair block kernel, against
// modelled mbarriers, buffers and copies: every copy, softmax step and epilogue
// may take any time, some far longer than a block. A product must find exactly
// its own block's rows in every buffer it reads, and all blocks must finish.
// argv: seeds, then "class late" is drawn per seed inside. Exit 0: every run
// was right; otherwise the first fault is printed.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <random>
#include <vector>

#include "pair_order.h"

using elsaa::PairBar;
using elsaa::PairOrder;

namespace {

// an mbarrier by its completed phases: a parity test holds for the phase
// just completed, and so also one phase too early
struct Bar {
    int phases = 0;
    bool test(int parity) const { return (phases & 1) != parity; }
    // what a blocking wait for phase n means
    bool complete(int n) const { return phases > n; }
};

struct Event {
    long at;
    std::function<void()> run;
};

struct Run {
    int nblk, per_head;
    std::mt19937 rng;
    std::vector<int> late;  // percent of late steps per kind
    long now = 0;
    std::vector<Event> events;
    Bar k_full[2], q_full[2], v_full[2], wb_full, tmem_empty[2], p_full[2],
        phi_full[2], q_empty[2], k_empty[2], v_empty[2], s_full[2],
        pv0_done[2], pv_done[2], o_full[2], head_done;
    int k[2] = {-1, -1}, q[2] = {-1, -1}, v[2] = {-1, -1}, wb = -1;
    const char *fault = nullptr;
    long mma_free = 0;  // products end in the order of their issue

    bool new_head(int j) const { return j == 0 || j % per_head == 0; }
    long delay(int kind, int usual) {
        const bool is_late = (int)(rng() % 100) < late[kind];
        return 1 + rng() % usual + (is_late ? rng() % (usual * 40) : 0);
    }
    void after(long d, std::function<void()> f) {
        events.push_back({now + d, std::move(f)});
    }
    void product(std::function<void()> end) {
        mma_free = std::max(mma_free, now) + 1 + rng() % 4;
        events.push_back({mma_free, std::move(end)});
    }
    void expect(bool ok, const char *what) {
        if (!ok && !fault) fault = what;
    }
    // a copy for block j into `buf`: not to be read until it lands
    void copy(int &buf, int j, Bar &full, int kind) {
        buf = -1;
        after(delay(kind, 12), [&buf, j, &full] {
            buf = j;
            ++full.phases;
        });
    }

    // copy warps: keys and queries, values, planes
    int kq_j = 0, kq_step = 0, v_u = 0, wb_j = 0, wb_n = 0;
    void copies() {
        if (kq_j < nblk) {
            const int j = kq_j, s = j & 1;
            if (kq_step == 0) {
                if (j < 1 || k_empty[0].complete(j - 1)) {
                    copy(k[0], j, k_full[0], 0);
                    kq_step = 1;
                }
            } else if (kq_step == 1) {
                if (j < 2 || q_empty[s].complete((j >> 1) - 1)) {
                    copy(q[s], j, q_full[s], 1);
                    kq_step = 2;
                }
            } else if (j < 1 || k_empty[1].complete(j - 1)) {
                copy(k[1], j, k_full[1], 2);
                kq_step = 0;
                ++kq_j;
            }
        }
        if (v_u < 2 * nblk) {
            const int j = v_u >> 1, p = v_u & 1;
            if (j < 1 || v_empty[p].complete(j - 1)) {
                copy(v[p], j, v_full[p], 3 + p);
                ++v_u;
            }
        }
        while (wb_j < nblk && !new_head(wb_j)) ++wb_j;
        if (wb_j < nblk && (wb_n == 0 || head_done.complete(wb_n - 1))) {
            copy(wb, wb_j / per_head, wb_full, 5);
            ++wb_j;
            ++wb_n;
        }
    }

    // a slot's compute warps: P, P, features, output, one step after another
    int c_step[2] = {0, 0}, c_k[2] = {0, 0};
    bool c_busy[2] = {false, false};
    void compute(int g) {
        const int kk = c_k[g];
        if (c_busy[g] || 2 * kk + g >= nblk) return;
        Bar *out = nullptr;
        if (c_step[g] == 0 && s_full[g].complete(2 * kk)) out = &p_full[g];
        if (c_step[g] == 1 && s_full[g].complete(2 * kk + 1))
            out = &p_full[g];
        if (c_step[g] == 2 && pv_done[g].complete(kk)) out = &phi_full[g];
        if (c_step[g] == 3 && o_full[g].complete(kk)) out = &tmem_empty[g];
        if (!out) return;
        c_busy[g] = true;
        after(delay(6 + c_step[g], 20), [this, g, out] {
            ++out->phases;
            c_busy[g] = false;
            if (++c_step[g] == 4) {
                c_step[g] = 0;
                ++c_k[g];
            }
        });
    }

    bool run() {
        PairOrder order;
        int s0 = 0, s1 = 0;          // blocks whose scores went out, by pass
        int blk[2] = {0, 1};         // block of each slot
        auto nh = [&](int j) { return new_head(j); };
        auto test = [&](PairBar b, int i, int par) {
            switch (b) {
                case PairBar::k_full: return k_full[i].test(par);
                case PairBar::q_full: return q_full[i].test(par);
                case PairBar::v_full: return v_full[i].test(par);
                case PairBar::pv0_done: return pv0_done[i].test(par);
                case PairBar::tmem_empty: return tmem_empty[i].test(par);
                case PairBar::p_full: return p_full[i].test(par);
                case PairBar::phi_full: return phi_full[i].test(par);
                default: return wb_full.test(par);
            }
        };
        auto scores = [&](int s, int p) {
            const int j = blk[s];
            expect((p ? s1 : s0)++ == j, "scores out of order");
            expect(k[p] == j, "scores of keys that are not there");
            expect(q[s] == j, "scores of queries that are not there");
            if (p == 0) {
                expect(wb == j / per_head, "planes that are not there");
                expect(tmem_empty[s].phases >= j >> 1,
                       "scores over an output that is not read");
            } else {
                expect(pv0_done[s].phases == (j >> 1) + 1,
                       "scores over a P that is still read");
            }
            product([this, s, p, j] {
                expect(k[p] == j && q[s] == j, "operands overwritten");
                ++s_full[s].phases;
                ++k_empty[p].phases;
                if (p == 1) ++q_empty[s].phases;
            });
        };
        auto values = [&](int s, int p) {
            const int j = blk[s];
            expect(v[p] == j, "P V of values that are not there");
            expect(p_full[s].phases == 2 * (j >> 1) + p + 1,
                   "P V of a P that is not there");
            product([this, s, p, j] {
                expect(v[p] == j, "values overwritten");
                ++v_empty[p].phases;
                ++(p ? pv_done : pv0_done)[s].phases;
            });
        };
        auto features = [&](int s, int n) {
            const int j = blk[s];
            expect(wb == j / per_head, "summary that is not there");
            expect(phi_full[s].phases == (j >> 1) + 1,
                   "features that are not there");
            const bool last = n == nblk - 1 || (n + 1) % per_head == 0;
            product([this, s, last] {
                ++o_full[s].phases;
                if (last) ++head_done.phases;
            });
            blk[s] += 2;
        };
        for (; order.done < nblk && !fault; ++now) {
            if (now > 40000L * (nblk + 1)) fault = "stalled";
            for (size_t i = 0; i < events.size();) {
                if (events[i].at <= now) {
                    auto f = std::move(events[i].run);
                    events.erase(events.begin() + (long)i);
                    f();
                    i = 0;  // in any case the earliest issued first
                } else {
                    ++i;
                }
            }
            copies();
            compute(0);
            compute(1);
            order.round(nblk, nh, test, scores, values, features);
        }
        return !fault;
    }
};

}  // namespace

int main(int argc, char **argv) {
    const int seeds = argc > 1 ? atoi(argv[1]) : 100;
    const int heads[] = {1, 2, 3, 5, 64};
    for (int seed = 0; seed < seeds; ++seed)
        for (int per_head : heads)
            for (int nblk : {1, 2, 3, 9}) {
                Run r;
                r.nblk = nblk;
                r.per_head = per_head;
                r.rng.seed(1000u * (unsigned)seed + 10u * (unsigned)per_head +
                           (unsigned)nblk);
                r.late.assign(10, 0);
                // none late, one kind of step late, or all
                if (seed % 12 < 10) r.late[(size_t)(seed % 12)] = 50;
                if (seed % 12 == 10) r.late.assign(10, 25);
                if (!r.run()) {
                    printf("seed %d, %d blocks, %d a head: %s\n", seed, nblk,
                           per_head, r.fault);
                    return 1;
                }
            }
    printf("ok\n");
    return 0;
}
