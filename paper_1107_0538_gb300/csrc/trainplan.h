// Which lane of a net's training workspace takes which pair of a mini-batch.
//
// The gradient is the sum, in order, of up to kTrainSlots partial gradients:
// pair k of the mini-batch belongs to slot k mod kTrainSlots.  A lane adds the
// pairs of one slot at a time, so every lane holds one partial gradient.  With a
// lane for every slot all of them run at once; with fewer (no memory for more)
// the slots take the lanes in rounds, and the sums, and so the gradient's bits,
// stay the same.
#pragma once

#include <algorithm>
#include <vector>

namespace gbcg {

constexpr int kTrainSlots = 4;

struct TrainPair {
    int pair, lane;
    bool first;   // the slot's first pair: its gradient is stored, the others' are added
};
struct TrainRound {
    int lanes = 0;   // lanes 0 .. lanes - 1 hold one slot each, in slot order
    std::vector<TrainPair> pairs;
};

inline std::vector<TrainRound> plan_training(int count, int lanes) {
    std::vector<TrainRound> rounds;
    const int slots = std::min(kTrainSlots, count);
    for (int s0 = 0; s0 < slots; s0 += lanes) {
        TrainRound r;
        r.lanes = std::min(lanes, slots - s0);
        for (int k = 0; k < count; ++k) {
            const int lane = k % kTrainSlots - s0;
            if (lane >= 0 && lane < r.lanes) r.pairs.push_back({k, lane, k < kTrainSlots});
        }
        rounds.push_back(std::move(r));
    }
    return rounds;
}

}  // namespace gbcg
