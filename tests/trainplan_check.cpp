// CPU check of csrc/trainplan.h: for every number of lanes the slots hold the
// same pairs in the same order and are added in the same order, and no lane
// holds two slots in one round.
#include <cstdio>

#include "trainplan.h"

using namespace gbcg;

int main() {
    int bad = 0;
    for (int count = 0; count <= 13; ++count)
        for (int lanes = 1; lanes <= kTrainSlots; ++lanes) {
            std::vector<std::vector<int>> slots;   // in the order they are added to the gradient
            for (const TrainRound &r : plan_training(count, lanes)) {
                if (r.lanes < 1 || r.lanes > lanes) ++bad;
                std::vector<std::vector<int>> part((size_t)r.lanes);
                for (const TrainPair &t : r.pairs) {
                    if (t.lane < 0 || t.lane >= r.lanes) return 1;
                    if (t.first != part[(size_t)t.lane].empty()) ++bad;
                    part[(size_t)t.lane].push_back(t.pair);
                }
                for (auto &p : part) slots.push_back(p);
            }
            if ((int)slots.size() != (count < kTrainSlots ? count : kTrainSlots)) ++bad;
            for (size_t s = 0; s < slots.size(); ++s) {
                std::vector<int> want;
                for (int k = (int)s; k < count; k += kTrainSlots) want.push_back(k);
                if (slots[s] != want) ++bad;
            }
        }
    std::printf("%d\n", bad);
    return bad != 0;
}
