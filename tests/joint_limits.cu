// Drives the choice of the limits that the joint recurrence tests (test_joint_limits.py; no GPU is needed) with lists of stage costs:
// prints, per list, most tests of a search, searches whose limits left [lo, hi) or that did not end, and wrong answers.
#include "../paper_2609_39350_b200/csrc/hap_tree.cuh"
#include "../paper_2609_39350_b200/csrc/hap_joint.cuh"

#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>

using namespace hap;

static int most, lost, wrong;

// costs in order; the smallest limit that can do is `answer` (kInf: none)
static void search(const std::vector<i64> &costs, i64 answer, i64 low, i64 floor_b, i64 guess, bool doubtful)
{
    LimitSearch s;
    s.begin(low, floor_b, guess, doubtful);
    for (int n = 1; ; ++n) {
        const i64 lo = s.lo, hi = s.hi;
        if (n > 128 || s.B < lo || s.B >= hi) { ++lost; return; }
        // what a test leaves: costs further than 2^32 from the limit are not looked at
        const auto above = std::upper_bound(costs.begin(), costs.end(), s.B);
        i64 dn = above == costs.begin() ? 0 : above[-1], up = above == costs.end() ? kInf : std::min(*above, kInf);
        if (s.B + 1 - 4294967296ll > dn) dn = s.B + 1 - 4294967296ll;
        if (s.B + 4294967296ll < up) up = s.B + 4294967296ll;
        const bool more = s.next(s.B >= answer, dn, up);
        most = std::max(most, n);
        if (more && (s.lo < lo || s.hi > hi || (s.lo == lo && s.hi == hi))) { ++lost; return; }
        if (!more) break;
    }
    wrong += s.lo != answer;
}

static void report(const char *name, std::vector<i64> costs)
{
    std::sort(costs.begin(), costs.end());
    costs.erase(std::unique(costs.begin(), costs.end()), costs.end());
    most = lost = wrong = 0;
    const i64 any[] = {0, 1, 12345, 1ll << 40, kInf - 1, kInf, -1, -(1ll << 60)};
    const size_t n = costs.size(), every = n / 24 + 1;
    for (size_t a = 0; a <= n; a += a + 1 < n && a + every >= n ? n - a - 1 : every) {
        const i64 answer = a < n ? costs[a] : kInf;
        std::vector<i64> guesses(any, any + 8), lows = {0, costs[0], a ? costs[(a - 1) / 2] : 0, a ? costs[a - 1] : 0};
        for (size_t g = 0; g < n; g += every) guesses.push_back(costs[g]);
        guesses.push_back(costs[n - 1]);
        if (a < n) lows.push_back(answer);
        for (i64 low : lows)
            for (i64 guess : guesses)
                for (i64 floor_b : {(i64)0, low, a ? costs[a / 2 ? a / 2 : 0] : 0, answer < kInf ? answer : 0})
                    for (bool doubtful : {false, true})
                        if (floor_b <= answer) search(costs, answer, low, floor_b, guess, doubtful);
        if (a == n) break;
    }
    printf("%s %d %d %d\n", name, most, lost, wrong);
}

int main()
{
    std::mt19937_64 rng(7);
    for (int top = 20; top <= 61; ++top) {
        std::vector<i64> up, down, both, even, odd;
        const i64 end = 1ll << top;
        for (int i = 0; i <= top; ++i) {                        // crowded towards one end or the middle
            up.push_back((1ll << i)); down.push_back(end - (1ll << i) + 1);
            both.push_back(end / 2 + (1ll << i) / 2); both.push_back(end / 2 - (1ll << i) / 2 + 1);
        }
        for (int i = 1; i <= 300; ++i) { even.push_back(end / 300 * i); odd.push_back(1 + (i64)(rng() % (u64)end)); }
        report("above", up); report("below", down); report("middle", both); report("even", even); report("random", odd);
        report("one", {end}); report("two", {1, end}); report("last", {end - 1, end});
    }
    // layer times that grow by a steady factor
    for (double f : {1.05, 1.1, 1.3, 1.7, 2.0, 3.0}) {
        std::vector<i64> c;
        for (double v = 1; v < 2.0e18; v *= f) c.push_back((i64)v);
        report("growing", c);
    }
    return 0;
}
