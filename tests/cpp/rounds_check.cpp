// Host check of the allocation-free sweep's staged rounds (jac_rounds.h): every
// entry of a block is staged once, in order, within [p0, p1), and every row finds
// its entries in the rounds, for blocks anywhere up to the last int32 position.
// Signed overflow aborts under the UndefinedBehaviorSanitizer; a bound on the
// rounds ends the check where a wrapped position would let them run on.
#include <climits>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "jac_rounds.h"

constexpr int CAP = 7 * 256, ROWS = 256;

static void require(bool ok, const char* what, int p0, int p1)
{
    if (ok) return;
    std::printf("FAIL: %s (block [%d, %d))\n", what, p0, p1);
    std::exit(1);
}

static void check(int p0, int p1, int row_len)
{
    // the block's rows: row_len entries each, the last row takes what is left
    std::vector<int> ptr(ROWS + 1, p1);
    for (int r = 0; r < ROWS; ++r) {
        const long long at = (long long)p0 + (long long)r * row_len;
        ptr[r] = at < p1 ? (int)at : p1;
    }
    std::vector<int> summed(ROWS, 0);
    long long next = p0, rounds = 0;
    jac::for_each_round<CAP>(p0, p1, [&](int first, int count) {
        require(++rounds <= ((long long)p1 - p0) / CAP + 1, "too many rounds", p0, p1);
        require(first == next && count >= 0 && count <= CAP, "a round does not follow the one before", p0, p1);
        for (int at = 0; at < CAP; ++at)
            if (at < count) {
                const long long e = (long long)first + at;
                require(e >= p0 && e < p1, "an entry outside the block is staged", p0, p1);
            }
        for (int r = 0; r < ROWS; ++r) {
            int from = 0;
            const int len = jac::row_part(ptr[r], ptr[r + 1], first, count, from);
            require(len == 0 || (from >= 0 && from + len <= count), "a row reads past its round", p0, p1);
            require(len == 0 || first + from == ptr[r] + summed[r], "a row skips an entry", p0, p1);
            summed[r] += len;
        }
        next += count;
    });
    require(next == p1, "entries are left", p0, p1);
    for (int r = 0; r < ROWS; ++r) require(summed[r] == ptr[r + 1] - ptr[r], "a row is short", p0, p1);
}

int main()
{
    const int sizes[] = {0, 1, 255, CAP - 1, CAP, CAP + 1, 2 * CAP - 1, 2 * CAP, 2 * CAP + 1, 20 * CAP + 17};
    for (int size : sizes)
        for (int row_len : {1, 7, 512, 100000}) {
            for (int p0 : {0, 3, 1 << 20}) check(p0, p0 + size, row_len);
            for (int back : {0, 1, 255, 256, CAP - 1, CAP, CAP + 1}) check(INT_MAX - back - size, INT_MAX - back, row_len);
        }
    std::printf("ok\n");
    return 0;
}
