// Host check of the counting sort of csrc/plan.h: the order of std::stable_sort for keys from few
// to many buckets, and cost buckets that never put a larger cost behind one 1/64 smaller.
#include <algorithm>
#include <cstdio>
#include <numeric>
#include <random>
#include <vector>

#include "plan.h"

int main()
{
    std::mt19937_64 rng(5);
    for (int64_t n : {0, 1, 2, 1000})
        for (int64_t buckets : {1, 7, 5000}) {
            std::vector<int64_t> key((size_t)n);
            for (auto& k : key) k = (int64_t)(rng() % (uint64_t)buckets);
            std::vector<int64_t> want((size_t)n);
            std::iota(want.begin(), want.end(), 0);
            std::stable_sort(want.begin(), want.end(), [&](int64_t x, int64_t y) { return key[x] < key[y]; });
            if (cm::counting_order(n, buckets, [&](int64_t i) { return key[i]; }) != want) return 1;
        }
    int64_t prev = cm::cost_bucket(0);
    if (prev != cm::kCostBuckets - 1) return 2;
    for (int64_t c = 1; c < ((int64_t)1 << 62); c += 1 + (c >> 9)) {
        const int64_t b = cm::cost_bucket(c);
        if (b < 0 || b > prev || (c >= 64 && cm::cost_bucket(c + c / 63 + 1) >= b)) return 3;
        prev = b;
    }
    return cm::cost_bucket(INT64_MAX) >= 0 ? 0 : 4;
}
