// The long rows' packed counter (csrc/join_rows.cuh): the reservations of a step, played on the host beside exact sums.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "join_rows.cuh"

using namespace gsi;
using u128 = unsigned __int128;

#define CHECK(c)                                             \
    do {                                                     \
        if (!(c)) {                                          \
            std::printf("line %d: %s\n", __LINE__, #c);      \
            std::exit(1);                                    \
        }                                                    \
    } while (0)

int main() {
    std::mt19937_64 rng(7);
    const uint64_t sizes[] = {0, 1, 2, 3, 255, 256, 1000, (1u << 20) - 1, 1u << 20, 119000000, 1ull << 30, (1ull << 40) - 1};
    for (uint64_t R : sizes)
        for (uint64_t cap : sizes) {
            const uint64_t most = R < cap ? R : cap;
            const int rb = long_row_bits(R, cap);
            CHECK(rb >= 1 && rb <= 40 && most >> rb == 0 && (rb == 1 || most >> (rb - 1)));
            // from the beginning, and from counts near the room's end or the slots' limit
            for (int from = 0; from < 3; ++from)
                for (int rep = 0; rep < 50; ++rep) {
                    uint64_t rows = from == 1 && most > 600 ? most - 600 : 0;
                    u128 slots = from == 2 ? ((u128)1 << (64 - rb)) - 3000000 : 0;
                    if (slots >> (64 - rb)) slots = 0;
                    unsigned long long ctr = ((unsigned long long)slots << rb) | rows;
                    unsigned fail = 0;
                    for (int i = 0; i < 40 && rows < R; ++i) {
                        const uint64_t n = 1 + rng() % 512, add = n < R - rows ? n : R - rows;
                        const uint64_t len = add * (17 + rng() % 2000);
                        const unsigned long long old = ctr;
                        ctr += (len << rb) | add;
                        if (!fail) {                  // a reservation that nothing has spoilt: its places are exact
                            CHECK((old & ((1ull << rb) - 1)) == rows && old >> rb == (uint64_t)slots);
                            CHECK(rows <= cap);
                        }
                        const unsigned f = long_fails(old, add, len, rb, cap);
                        rows += add;
                        slots += len;
                        if (!fail) {
                            CHECK(((f & LONG_FULL) != 0) == (rows > cap));
                            CHECK(((f & LONG_NEVER) != 0) == (slots >> (64 - rb) != 0));
                        }
                        fail |= f;
                        CHECK(fail || (rows <= cap && slots >> (64 - rb) == 0));
                    }
                }
        }
    // a step of 2^30 rows that meets the table of a first arena has as many slots as one of the table's rows
    CHECK(long_row_bits(1ull << 30, 119000000) == 27);
    std::printf("ok\n");
    return 0;
}
