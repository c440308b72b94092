// The key switch's launches for runs of samples of several keys, against every
// way to cut them into launches.  ks_plan SMS (n N log2_Bks l_ks count)...:
// prints each launch as first:count:cpt; exits 1 when one is cheaper.
#include <cstdio>
#include <cstdlib>

#include "ks_plan.cuh"

using namespace ksp;

static u64 cost(const std::vector<Run> &r, size_t a, size_t b, bool tiled, u32 sms) {
    u64 c = 0;
    if (tiled) return b - a == 1 && tile(r[a].key, r[a].count, sms, c) ? c + kLaunch : ~0ull >> 1;
    Blocks s;
    for (size_t i = a; i < b; i++) s.add(r[i].key, r[i].count);
    return s.cost(sms) + kLaunch;
}

// (neighbouring runs that no tile can take are one part)
static bool together(const std::vector<Run> &r, size_t i, u32 sms) {
    u64 c;
    return i > 0 && i < r.size() && !tile(r[i - 1].key, r[i - 1].count, sms, c) && !tile(r[i].key, r[i].count, sms, c);
}

static u64 search(const std::vector<Run> &r, size_t a, u32 sms) {
    u64 best = a == r.size() ? 0 : ~0ull;
    for (size_t b = a + 1; b <= r.size(); b++) {
        if (together(r, b, sms)) continue;
        const u64 rest = search(r, b, sms);
        best = std::min(best, std::min(cost(r, a, b, false, sms), cost(r, a, b, true, sms)) + rest);
    }
    return best;
}

int main(int argc, char **argv) {
    const u32 sms = (u32)atoi(argv[1]);
    std::vector<Run> r;
    for (int i = 2; i + 4 < argc; i += 5)
        r.push_back({(uint32_t)atoi(argv[i + 4]),
                     {(u32)atoi(argv[i + 1]), (u32)atoi(argv[i]), (u32)atoi(argv[i + 3]), (u32)atoi(argv[i + 2])}});
    u64 total = 0;
    size_t at = 0;      // run
    uint32_t first = 0;
    for (const Launch &l : plan(r, sms)) {
        size_t b = at;
        uint32_t c = 0;
        while (b < r.size() && c < l.count) c += r[b++].count;
        if (l.first != first || c != l.count) return 2;
        total += cost(r, at, b, l.cpt != 0, sms);
        printf("%u:%u:%u\n", l.first, l.count, l.cpt);
        at = b;
        first += c;
    }
    if (at != r.size()) return 3;
    if (r.size() == 1 && plan(r, sms)[0].cpt != tile_cpt(r[0].key, r[0].count, sms)) return 4;
    return r.size() <= 12 && total > search(r, 0, sms) ? 1 : 0;
}
