// Checks of csrc/spread3_items.cuh (compiled and run by test_spread3_items.py).
#include <cstdio>
#include <cstdlib>
#include <random>

#include "spread3_items.cuh"

#define NEED(c)                                    \
    do {                                           \
        if (!(c)) {                                \
            printf("line %d: %s\n", __LINE__, #c); \
            exit(1);                               \
        }                                          \
    } while (0)

// every tile's entries exactly once, in order, in pieces of at most `item`
static void check(const std::vector<int>& n, const Spread3Items& s, int64_t item) {
    int64_t at = 0;
    size_t i = 0;
    int slot = 0;
    for (size_t t = 0; t < n.size(); ++t) {
        NEED(s.first[t] == at);
        const int k = s.tinfo[t].x;
        NEED(k >= 1 && (k > 1) == (n[t] > item));
        NEED(s.tinfo[t].y == (k > 1 ? slot : -1));
        int e = 0;
        for (int j = 0; j < k; ++j, ++i) {
            NEED(i < s.items.size());
            const int4 it = s.items[i];
            NEED(it.x == (int)t && it.y == e && it.z >= e && it.z - it.y <= item);
            NEED(it.w == (k > 1 ? slot + j : -1));
            e = it.z;
        }
        NEED(e == n[t]);
        if (k > 1) slot += k;
        at += n[t];
    }
    NEED(i == s.items.size() && at == s.entries && slot == s.slots);
}

int main() {
    std::mt19937 r(1);
    for (int c = 0; c < 200; ++c) {
        std::vector<int> n(1 + r() % 300);
        for (int& v : n) v = r() % 4 ? (int)(r() % 300) : (int)(r() % 20000);
        const int item = 1 << (r() % 12);
        check(n, spread3_items(n, item), item);
        // within a number of partial tiles: the first size that fits, whole tiles if none does
        const int64_t room = r() % 3 ? r() % 200 : 0;
        int64_t fit = item;
        while (spread3_items(n, fit).slots > room) fit *= 2;
        const Spread3Items w = spread3_items_within(n, item, room);
        NEED(w.slots <= room);
        check(n, w, fit);
    }
    for (int v : {0, 1, 255, 256, 257, 512, 513}) check({v, 0, v}, spread3_items({v, 0, v}, 256), 256);
    // more entries in all than 31 bits hold, and a tile of nearly as many
    std::vector<int> big(64, 100000000);
    check(big, spread3_items(big, 1 << 20), 1 << 20);
    NEED(spread3_items(big, 1 << 20).entries == 6400000000ll);
    check({2147483647}, spread3_items({2147483647}, 1 << 20), 1 << 20);
    check({2147483647, 5}, spread3_items_within({2147483647, 5}, 256, 0), 1ll << 31);
    printf("ok\n");
}
