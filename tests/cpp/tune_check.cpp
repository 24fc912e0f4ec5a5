// time_variants (tune.h) on a fake clock: the first run of a variant costs its code's load.
#include <cstdio>

#include "tune.h"

using namespace fpk;

#define EXPECT(c)                                   \
    do {                                            \
        if (!(c)) {                                 \
            std::printf("failed: %s\n", #c);        \
            return 1;                               \
        }                                           \
    } while (0)

int main() {
    const float warm[4] = {0.05f, 0.03f, 0.02f, 0.04f};
    const float load[4] = {2.0f, 0.0f, 5.0f, 1.0f};   // variant 1's code is loaded already
    int runs[4] = {0, 0, 0, 0};
    std::vector<float> ms;
    auto clock = [&](int i, bool counted, float &t) {
        if (counted != (runs[i] == 1)) return -1;
        t = warm[i] + (runs[i]++ ? 0.0f : load[i]);
        return 0;
    };
    EXPECT(time_variants(4, ms, clock) == 0);
    for (int i = 0; i < 4; ++i) EXPECT(ms[i] == warm[i]);   // variant 2 is the fastest, whatever its load

    // one that cannot run here, and one that fails on its second run only
    int n = 0;
    EXPECT(time_variants(3, ms, [&](int i, bool, float &t) {
               t = 1.0f;
               return i == 0 ? 1 : i == 1 ? n++ : 0;
           }) == 0);
    EXPECT(ms[0] == kNoTime && ms[1] == kNoTime && ms[2] == 1.0f);

    // an error ends it
    int calls = 0;
    EXPECT(time_variants(3, ms, [&](int i, bool, float &t) {
               ++calls;
               t = 1.0f;
               return i == 1 ? -4 : 0;
           }) == -4);
    EXPECT(calls == 3 && ms[2] == kNoTime);
    std::puts("ok");
    return 0;
}
