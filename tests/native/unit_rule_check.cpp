// Checks of the counting work-unit rule (host code only): the size that the autotuner times for an
// instance is the size that the batch then runs, whatever the instance's size, and a single call's
// units are small enough for every SM to have some.
// Built and run by tests/test_unit_rule_host.py; prints one line per failed check and exits 1 if any.
#include <cstdio>

#include "unit_rule.h"

static int failures = 0;
#define CHECK(cond)                                                                                     \
    do {                                                                                                \
        if (!(cond)) {                                                                                  \
            std::printf("FAILED line %d: %s (users %lld, items %lld)\n", __LINE__, #cond, users, items); \
            ++failures;                                                                                 \
        }                                                                                               \
    } while (0)

int main() {
    for (long long users = 1; users <= 16000; users = users * 3 + 1)
        for (long long items = 0; items <= 2000; items = items * 4 + 1) {
            for (int g : {8, 16, 32}) {
                CHECK(rkm::batch_units(g, true).tiles(users, items, 152) == g);
                // FP32 batches launch each instance by itself, under the single call's rule.
                CHECK(rkm::batch_units(g, false).tiles(users, items, 152) == (rkm::UnitRule{g, false}).tiles(users, items, 152));
            }
            // A stored choice is read from a text file: no value makes an empty unit.
            for (int g : {0, -5}) CHECK(rkm::batch_units(g, true).tiles(users, items, 152) == 1);
            const int t = rkm::UnitRule{}.tiles(users, items, 152);
            CHECK(t >= 1 && t <= 32);
            CHECK(t == 1 || (long long)t * 152 * 8 <= users * items);
        }
    if (failures == 0) std::printf("ok\n");
    return failures != 0;
}
