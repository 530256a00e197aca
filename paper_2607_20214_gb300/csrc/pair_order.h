// Which product of the CTA-pair block kernel (tc_pair.cu) is issued next.
// Apart from the kernel, and without CUDA, so that tests/test_pair_order.py
// can run it on the host against modelled barriers and late copies.
//
// Two slots, block j in slot j & 1, each at a stage of its own:
//   0 scores and projections of pass 0   1 P V of pass 0
//   2 scores of pass 1                   3 P V of pass 1
//   4 the features' product, which ends the block
// A stage goes when everything it reads is there.
//
// A barrier's parity test tells two neighbouring phases apart and no more: a
// test for phase n also holds while phase n - 1 is still open. So phase n may
// be tested only once phase n - 1 is known to be complete. The barriers of a
// slot are tested by that slot's blocks alone, one phase after the other. The
// key and value buffers have one phase per block and both slots read them, so
// each of their stages goes through the blocks in order: block j's test comes
// only when block j - 1's product of the same stage, which waited for the
// phase before, has been issued. Block j - 1 waits for nothing of block j, so
// the order cannot stall; the slots are half a block apart, so it hardly costs
// anything (B1 H32 N65536 d128 r256: 585 us, 584 without it).
//
// The scores of pass 1 go over P of pass 0, so they wait until the product
// that reads it is complete (pv0_done, of the slot: the value buffer's own
// barrier may be two phases on by then). Products of different accumulators are
// not documented to run in the order of their issue; relying on it would gain
// 2 us of the 587.
#pragma once

#ifdef __CUDACC__
#define ELSAA_DEV __device__ __forceinline__
#else
#define ELSAA_DEV inline
#endif

namespace elsaa {

// barriers that the issuer tests: per pass (k_full, v_full), per slot, or one
enum class PairBar { k_full, q_full, v_full, pv0_done, tmem_empty, p_full,
                     phi_full, wb_full };

struct PairOrder {
    int j = 0, stage = 0;    // the slot at hand (j & 1)
    int jo = 1, stageo = 0;  // the other slot
    int done = 0;            // blocks finished
    int heads = 0;           // heads begun
    int issued0 = 0, issued1 = 0;  // blocks whose scores of pass 0, 1 are
    int values0 = 0, values1 = 0;  // issued; whose P V of pass 0, 1 are

    // Issues the next product of the slot at hand if it is ready, then turns
    // to the other slot. new_head(j): block j is its head's first here.
    // test(bar, index, parity): that barrier's parity test. scores(slot,
    // pass), values(slot, pass), features(slot, n) issue a product; n: blocks
    // finished before this one. Blocks of one head may finish out of order,
    // but the first block of a head begins when all before it are finished,
    // so the finish that makes up the count of a head's last block is the
    // head's last finish.
    template <class NewHead, class Test, class Scores, class Values,
              class Features>
    ELSAA_DEV bool round(int nblk, NewHead new_head, Test test, Scores scores,
                         Values values, Features features) {
        bool go = false;
        if (j < nblk) {
            const int s = j & 1, k = j >> 1;  // k: the slot's own count
            if (stage == 0) {
                const bool nh = new_head(j);
                go = issued0 == j && !(nh && done < j) &&
                     test(PairBar::k_full, 0, j & 1) &&
                     test(PairBar::q_full, s, k & 1) &&
                     (j < 2 || test(PairBar::tmem_empty, s, (k - 1) & 1)) &&
                     (!nh || test(PairBar::wb_full, 0, heads & 1));
                if (go) {
                    if (nh) ++heads;
                    scores(s, 0);
                    ++issued0;
                }
            } else if (stage == 1) {
                go = values0 == j && test(PairBar::p_full, s, 0) &&
                     test(PairBar::v_full, 0, j & 1);
                if (go) {
                    values(s, 0);
                    ++values0;
                }
            } else if (stage == 2) {
                go = issued1 == j && test(PairBar::k_full, 1, j & 1) &&
                     test(PairBar::pv0_done, s, k & 1);
                if (go) {
                    scores(s, 1);
                    ++issued1;
                }
            } else if (stage == 3) {
                go = values1 == j && test(PairBar::p_full, s, 1) &&
                     test(PairBar::v_full, 1, j & 1);
                if (go) {
                    values(s, 1);
                    ++values1;
                }
            } else {
                go = test(PairBar::phi_full, s, k & 1);
                if (go) {
                    features(s, done);
                    ++done;
                    j += 2;
                }
            }
            if (go) stage = stage == 4 ? 0 : stage + 1;
        }
        int x = j;  // the slots take turns
        j = jo;
        jo = x;
        x = stage;
        stage = stageo;
        stageo = x;
        return go;
    }
};

}  // namespace elsaa
