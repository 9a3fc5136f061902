// Host check of the steps at which a column pass publishes its row groups: in order, no more than
// lane 31 has finished, no more than 32 groups late, and never the last one.
#include <cstdio>

#include "cm_internal.h"

int main()
{
    for (int32_t groups = 1; groups <= 400; ++groups) {
        int32_t done = 0;
        for (int32_t t = 0; t < groups + 31; ++t) {
            const int32_t g = cm::groups_after_step(t, groups);
            if (g != 0) {
                if (g <= done || g > t - 30 || g >= groups) return 1;
                done = g;
            }
            if (t < groups + 30 && t - 30 - done >= 32) return 2;
        }
        if (done >= groups) return 3;
    }
    return 0;
}
