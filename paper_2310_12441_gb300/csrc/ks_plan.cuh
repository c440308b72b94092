// Which kernel switches which samples: tiles of samples (ks_tile.cuh) or one
// block, or cluster of blocks, per sample.  Host code.
#pragma once
#include <algorithm>
#include <vector>

#include "ks_tile.cuh"

namespace ksp {

// What the rule needs of a key.
struct Key {
    u32 N, n, lks, log2_Bks;
};
// Consecutive samples of one key.
struct Run {
    uint32_t count;
    Key key;
};
// One launch over samples [first, first + count): cpt samples per thread of a
// tile, all of key `key`; cpt 0: a block or cluster per sample, any keys.
struct Launch {
    uint32_t first, count;
    u32 cpt;
    Key key;
};

inline u32 slices(const Key &k) { return (k.n + kKskCols) / kKskCols; }

// Blocks per sample without tiles: the largest S in {1, 2, 4, 8} with count S <=
// SMs (one block per sample once they fill the GPU).
inline u32 split(u64 count, u32 sms) {
    u32 S = 1;
    while (S < 8 && count * (2 * S) <= sms) S *= 2;
    return S;
}

// Costs in cycles, measured for l_ks = 3..16, B_ks = 2..128, n = 64..1030, 80..2049
// samples of one key.  Per coefficient of the ring, a tile: 700 per stage, 50 and
// 36 per sample of a thread for every digit, at least its key rows at 64 B per
// cycle.  A block per sample: per digit 230 (n < 256) or 340, 370 with more
// blocks than SMs, 900 with more than the three an SM holds (latency, shared by
// the blocks of a cluster), or for every
// sample 1/8 per column slice, at least 9/8 (throughput).  (n = 630, N = 1024: 64
// samples 0.68 ms against 1.08 in tiles; 96: 1.32 against 1.08; 2000: 9.6 against
// 3.2; B_ks = 128, n = 830, N = 256: 300 samples 0.24 against 0.52, 2049: 1.44
// against 0.81.)
struct Blocks {        // one launch of a block or cluster per sample
    u64 count = 0, thr = 0, few = 0, many = 0, waves = 0;      // latency up to SMs, 3 SMs samples, above
    void add(const Key &k, u64 samples) {
        const u64 digits = (u64)k.N * k.lks;
        add(Blocks{samples, k.N * (k.lks * (samples * std::max(slices(k), 9u) / 8)), digits * (k.n < 256 ? 230 : 340),
             digits * 370, digits * 900});
    }
    void add(const Blocks &b) {
        count += b.count;
        thr += b.thr;
        few = std::max(few, b.few);
        many = std::max(many, b.many);
        waves = std::max(waves, b.waves);
    }
    u64 cost(u32 sms) const {
        return std::max(thr, (count > 3ull * sms ? waves : count > sms ? many : few) / split(count, sms));
    }
};

constexpr u64 kLaunch = 5000;     // a launch more on the stream

// The cheapest tile of `count` samples of one key: samples per thread, 0 when
// its rows do not fit a stage or a cluster per sample is to be had (faster).
inline u32 tile(const Key &k, uint32_t count, u32 sms, u64 &cost) {
    const u32 jn = kst::digits_per_stage(k.lks, k.log2_Bks);
    u32 best = 0;
    if (jn == 0 || 2ull * count <= sms) return best;
    const u32 parts = (k.lks + jn - 1) / jn;
    const u64 fill = (u64)k.lks * ((1u << k.log2_Bks) - 1) * kKskCols * 8 / 64;
    for (u32 cpt = 4; cpt <= kst::kMaxCpt; cpt += 4) {
        if (kst::smem_bytes(k.lks, k.log2_Bks, cpt * kst::kWarpsPer, 2) > kst::kMaxSmem) break;
        const u64 tiles = (count + cpt * kst::kWarpsPer - 1) / (cpt * kst::kWarpsPer);
        const u64 waves = (tiles * slices(k) + sms - 1) / sms;
        const u64 c = k.N * (waves * std::max<u64>(700 * parts + k.lks * (50 + 36 * cpt), fill));
        if (!best || c < cost) {
            cost = c;
            best = cpt;
        }
    }
    return best;
}

// Samples per thread for `count` samples of one key, 0: a block or cluster per sample.
inline u32 tile_cpt(const Key &k, uint32_t count, u32 sms) {
    u64 cost = 0;
    const u32 cpt = tile(k, count, sms, cost);
    Blocks b;
    b.add(k, count);
    return cpt && cost < b.cost(sms) ? cpt : 0;
}

// Launches for runs of several keys, which follow each other on one stream: a
// tile launch holds one run, a launch of blocks any number of neighbouring
// ones, so many runs of less than a GPU's worth are better off in blocks
// together (30 runs of 80 samples at n = 630, N = 1024: 11.6 ms, 39.7 as 30 tile
// launches) and long ones in tiles of their own (2 x 1200: 4.3 ms against
// 11.1).  The cheapest sequence by the costs above.
inline std::vector<Launch> plan(const std::vector<Run> &runs, u32 sms) {
    // parts: a run that tiles can take, or neighbouring ones that they cannot
    struct Part {
        uint32_t first;
        Blocks blocks;
        u32 cpt;
        u64 tile_cost;
        Key key;
    };
    std::vector<Part> p;
    uint32_t at = 0;
    for (const Run &r : runs) {
        Part x{at, {}, 0, 0, r.key};
        x.blocks.add(r.key, r.count);
        x.cpt = tile(r.key, r.count, sms, x.tile_cost);
        if (!x.cpt && !p.empty() && !p.back().cpt) p.back().blocks.add(x.blocks);
        else p.push_back(x);
        at += r.count;
    }
    // best[i]: parts 0 .. i - 1; from[i]: first part of the last launch, blocks unless tiled
    const size_t n = p.size();
    std::vector<u64> best(n + 1, 0);
    std::vector<uint32_t> from(n + 1, 0);
    std::vector<char> tiled(n + 1, 0);
    for (size_t i = 1; i <= n; i++) {
        const Part &l = p[i - 1];
        if ((tiled[i] = l.cpt != 0)) {
            best[i] = best[i - 1] + l.tile_cost + kLaunch;
            from[i] = (uint32_t)(i - 1);
        }
        Blocks sum;
        for (size_t j = i; j-- > 0;) {
            sum.add(p[j].blocks);
            const u64 c = best[j] + sum.cost(sms) + kLaunch;
            if ((!tiled[i] && j + 1 == i) || c < best[i]) {
                best[i] = c;
                from[i] = (uint32_t)j;
                tiled[i] = 0;
            }
            if (sum.thr >= best[i]) break;     // more parts only cost more
        }
    }
    std::vector<Launch> out;
    for (size_t i = n; i > 0; i = from[i]) {
        const Part &a = p[from[i]], &b = p[i - 1];
        out.push_back({a.first, b.first + (uint32_t)b.blocks.count - a.first, tiled[i] ? b.cpt : 0, b.key});
    }
    std::reverse(out.begin(), out.end());
    return out;
}

}  // namespace ksp
