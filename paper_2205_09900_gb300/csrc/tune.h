// tune.h -- timing of the variants that the autotuner chooses from.
#pragma once
#include <vector>

namespace fpk {

constexpr float kNoTime = 1e30f;   // a variant that does not run here

// The time of each of n variants, kNoTime for one that cannot run: run(i, counted, ms) runs variant i
// once, sets ms to its time and returns 0, 1 where it cannot run, or a negative status, which ends the
// timing and is returned.  The first run of a variant is not counted (and may be of a part of the
// work): it loads the variant's code, which takes longer than a small batch itself, so it says
// nothing about which is faster.
template <typename F>
int time_variants(int n, std::vector<float> &ms, F run) {
    ms.assign((size_t)n, kNoTime);
    for (int i = 0; i < n; ++i)
        for (int rep = 0; rep < 2; ++rep) {
            float t = 0;
            const int s = run(i, rep == 1, t);
            if (s < 0) return s;
            if (s > 0) break;
            if (rep == 1) ms[(size_t)i] = t;
        }
    return 0;
}

}  // namespace fpk
