// batch_plan.h -- how a batched launch whose width is left to the library splits its items
// over CTAs (host only; no CUDA).
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <numeric>

namespace rh {

constexpr int kMaxBatch = 32;   // items of one batched launch

struct BatchItem {
    double levels, flops;       // levels of a direction's four sweeps, its flops
    int N, cap;                 // directions; the most a CTA can hold
    int n_x;
    bool line;                  // k_dir1_batch takes it (line schedules for 512 threads)
};
struct BatchPlan {
    int G[kMaxBatch];           // CTAs (0: no directions, or one per CTA in k_dir1_batch)
    bool alone[kMaxBatch];      // one direction per CTA in k_dir1_batch
};

// A CTA of the batched direction kernel with D directions of a grid takes about
//   t(D) = kLevelUs x levels + (kRowUs + kFlopUs x D) x flops,
// with the SM's CTA slots occupied: a level's chain, the rows' loads, which the directions
// share, and their arithmetic (fitted on GB300, D = 1 / 2 / 3: 2196 / 2526 / 3013 us on the
// 9241-bus grid, 744 / 795 / 1001 on 2869 buses, 360 / 401 / 476 on 1354 buses, 119 / 122 /
// 130 on 118 buses).  The items run side by side, so the launch ends with its slowest CTA:
// the least T is taken for which every item, at the most directions per CTA that end by T,
// gets all its CTAs into the slots at once.  One CTA a direction instead, whatever the
// batch, puts a batch of many directions through the slots in several waves of the
// latency-bound sweeps: a round of 15 requests (118 to 9241 buses, 1912 directions) took
// 5.6 ms, 8 x 64 directions on the 1354-bus grid 0.92 ms.
//
// With half of its slots occupied an SM runs each CTA in kHalf x t(D) (one direction for
// two: 281 us for 360 at 1354 buses, 571 for 744 at 2869), so fewer CTAs of more directions
// can end sooner: 8 x 64 directions at 1354 buses 488 us in 256 CTAs of 2, 479 in 128 of 4.
// Half, not one CTA: in CTAs of 128 threads, six to an SM, a batch of 461 directions (30 to
// 1354 buses) takes 534 us in one each, 704 in one an SM, 532 in at most three.
//
// The slots that are left go to the items in proportion: what ends by T in fewer CTAs by the
// model does not always on the device, where a CTA of many directions of a small grid also
// pays for loads, tail and products that the model has no term for.  166 directions, 130 of
// them on 30 buses: 273 us with those in one CTA, 264 spread; in CTAs of 128 threads 392 and
// 288.  A batch of no more directions than the SMs is one direction per CTA.
//
// The items on the largest grids may run one direction per CTA with x in shared memory
// instead (k_dir1_batch, an SM each, t(1) x kAlone), the others filling the SMs it leaves
// and, once its last CTA has started, those that are done.  Their few directions are the
// longest chains of a mixed batch: next to CTAs of many directions, which keep an SM's FP64
// pipes busy, they end it.  Of the sets "the items on grids of at least n rows" the one with
// the least predicted time is taken: the round of 15 requests takes 3.2 ms with none, 1.9
// ms with the 9241-bus grid (184 directions), 2.3 with 2869 buses and more, 2.2 with 1354
// buses and more; 8 x 64 directions on the 1354-bus grid take 488 us with none, 509 with all.
//
// A plan is host time in front of the launch: T is found to 0.2 %, and sets that cannot win
// are left out before their items are spread (32 grids of different sizes, 100 directions
// each, on a CPU: 277 us to the last bit, 20 so).
class BatchPlanner {
public:
    BatchPlanner(const BatchItem* items, int n, int n_sm, int per_sm, bool may_alone)
        : it_(items), n_(n), n_sm_(n_sm), per_sm_(per_sm), may_alone_(may_alone) {}

    void plan(BatchPlan& P) const {
        const int slots = n_sm_ * per_sm_;
        std::fill(P.alone, P.alone + n_, false);
        Spread best = spread(P.alone, slots);
        double least = best.t;
        if (may_alone_) {
            int order[kMaxBatch], m = 0;
            for (int k = 0; k < n_; k++)
                if (it_[k].N > 0) order[m++] = k;
            std::stable_sort(order, order + m, [&](int p, int q) { return it_[p].n_x > it_[q].n_x; });
            bool alone[kMaxBatch] = {};
            double sm_us = 0.0, longest = 0.0;
            int64_t dirs = 0;
            for (int i = 0; i < m && it_[order[i]].line; i++) {
                const BatchItem& b = it_[order[i]];
                alone[order[i]] = true;
                const double t1 = kAlone * time(b, 1, 1.0);
                longest = std::max(longest, t1);
                sm_us += t1 * b.N;
                dirs += b.N;
                if (i + 1 < m && it_[order[i + 1]].n_x == b.n_x) continue;
                // SMs that the last wave leaves, and when it starts
                const int last = (int)((dirs - 1) % n_sm_) + 1;
                const double wave = sm_us / (double)dirs, start = wave * (double)((dirs - 1) / n_sm_);
                const int room = per_sm_ * (n_sm_ - last);
                double t = std::max(start + wave, longest);
                if (t >= least) continue;
                Spread s;
                if (i + 1 < m) {
                    s = spread(alone, room > 0 ? room : slots);
                    t = room > 0 ? std::max(t, start + s.t) : t + s.t;
                }
                if (t < least) {
                    least = t;
                    best = s;
                    std::copy(alone, alone + n_, P.alone);
                }
            }
        }
        thin(P.alone, best, P.G);
    }

private:
    static constexpr double kLevelUs = 1.1, kRowUs = 0.78e-3, kFlopUs = 0.3e-3, kAlone = 0.36, kHalf = 0.77;
    struct Spread {
        double t = 0.0;          // predicted time
        int D[kMaxBatch] = {};   // the most directions per CTA (0: none)
        int room = 0;            // slots the items have
    };
    // c: 1, or kHalf
    static double time(const BatchItem& b, double D, double c) {
        return c * (kLevelUs * b.levels + (kRowUs + kFlopUs * D) * b.flops);
    }
    static int ctas(const BatchItem& b, int D) { return (b.N + D - 1) / D; }
    bool in(const bool* alone, int k) const { return !alone[k] && it_[k].N > 0; }

    // the items outside `alone` on `room` slots at rate c
    Spread fill(const bool* alone, int room, double c) const {
        Spread s;
        s.room = room;
        double lo = 0.0, hi = 0.0, base[kMaxBatch], per[kMaxBatch];
        for (int k = 0; k < n_; k++) {
            if (!in(alone, k)) continue;
            base[k] = time(it_[k], 0, c);
            per[k] = 1.0 / (c * kFlopUs * std::max(it_[k].flops, 1.0));
            lo = std::max(lo, time(it_[k], 1, c));
            hi = std::max(hi, time(it_[k], it_[k].cap, c));
        }
        auto total = [&](double t) {
            int64_t sum = 0;
            for (int k = 0; k < n_; k++) {
                if (!in(alone, k)) continue;
                s.D[k] = std::max(1, (int)std::min((double)it_[k].cap, (t - base[k]) * per[k]));
                sum += ctas(it_[k], s.D[k]);
            }
            return sum;
        };
        s.t = lo;
        if (total(lo) <= room) return s;
        while (hi - lo > 2e-3 * hi) {
            const double mid = 0.5 * (lo + hi);
            (total(mid) <= room ? hi : lo) = mid;
        }
        // more CTAs than slots even at the caps: further waves
        const int64_t all = total(hi);
        s.t = hi * (double)((all + room - 1) / room);
        return s;
    }
    // the same, or half the slots where that ends sooner
    Spread spread(const bool* alone, int room) const {
        Spread all = fill(alone, room, 1.0);
        const int few = room * std::max(1, per_sm_ / 2) / per_sm_;
        if (few < 1 || few == room) return all;
        Spread half = fill(alone, few, kHalf);
        return half.t < all.t ? half : all;
    }
    // the CTAs of each item: its share of the slots that are left taken too
    void thin(const bool* alone, const Spread& s, int* G) const {
        auto total = [&](double f) {
            int64_t sum = 0;
            for (int k = 0; k < n_; k++) {
                G[k] = 0;
                if (!in(alone, k)) continue;
                const int D = std::max(1, (int)std::ceil(f * s.D[k]));
                G[k] = ctas(it_[k], std::min(D, s.D[k]));
                sum += G[k];
            }
            return sum;
        };
        double lo = 0.0, hi = 1.0;       // at hi the CTAs fit, or do not at all
        if (total(lo) <= s.room) return;
        for (int i = 0; i < 10; i++) {
            const double mid = 0.5 * (lo + hi);
            (total(mid) <= s.room ? hi : lo) = mid;
        }
        total(hi);
    }

    const BatchItem* it_;
    int n_, n_sm_, per_sm_;
    bool may_alone_;
};

}  // namespace rh
