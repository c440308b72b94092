// Exact check of the tensor-core stages' recombination for one key: the limb
// sums of worst-case digits, every class, through the library's own tables and
// recombine_sums.  Prints the variant, the largest |limb sum| and the smallest
// and largest E and O in units of Q / 1000 (rounded outwards); exits 1 when a
// value is not congruent to the exact sum.
//   tc_bounds N Q log2_B
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "tc_tables.cuh"

typedef unsigned __int128 u128;
typedef __int128 i128;

static u64 mulmod(u64 a, u64 b, u64 Q) { return (u64)((u128)a * b % Q); }
static u64 powmod(u64 a, u64 e, u64 Q) {
    u64 r = 1;
    for (; e; e >>= 1, a = mulmod(a, a, Q))
        if (e & 1) r = mulmod(r, a, Q);
    return r;
}

template <int TC, bool LAZY>
static int check(const bm_key_params &p, const std::vector<u64> &tab) {
    constexpr int NL = brt::Limbs<TC>::NL, R = brt::Limbs<TC>::R;
    const u64 Q = p.Q;
    KeyDev K = {};
    while ((1u << K.logN) < p.N) K.logN++;
    const std::vector<unsigned char> t = brt::tc_tables(p, choose_variant(p), tab, K);
    const int half = 1 << (p.log2_B - 1);
    long top = 0;
    i128 lo[2] = {(i128)1 << 100, (i128)1 << 100}, hi[2] = {-((i128)1 << 100), -((i128)1 << 100)};
    u64 rng = 88172645463325252ull;
    for (int c = 0; c < 64; c++)
        for (int e = 0; e < 2; e++) {
            int w[64][NL];
            for (int i = 0; i < 64; i++)
                for (int l = 0; l < NL; l++) {
                    __half h;
                    memcpy(&h, &t[(e * NL + l) * 8192 + (c / 8) * 1024 + (i / 8) * 128 + (c % 8) * 16 + (i % 8) * 2], 2);
                    w[i][l] = (int)__half2float(h);
                }
            u64 cst;
            memcpy(&cst, &t[NL * 16384 + e * 512 + c * 8], 8);
            // digits that drive limb l (l = NL: the whole value, above: none) up
            // or down, the others by chance
            for (int pat = 0; pat < 2 * (NL + 1) + 40; pat++) {
                int32_t o[NL] = {};
                u64 exact = 0;
                for (int i = 0; i < 64; i++) {
                    const int l = pat / 2;
                    i128 v = 0;
                    for (int q = 0; q < NL; q++) v += (i128)w[i][q] << (R * q);
                    rng ^= rng << 13, rng ^= rng >> 7, rng ^= rng << 17;
                    const bool up = (l < NL ? w[i][l] > 0 : v > 0) == !(pat & 1);
                    const int d = l <= NL ? (up ? half - 1 : -half) : (int)((rng >> 20) % (u32)(2 * half)) - half;
                    for (int q = 0; q < NL; q++) o[q] += d * w[i][q];
                    // the digit itself is d + half, its weight psi's power (centred in the table)
                    const u64 f = v < 0 ? (u64)(v + Q) : (u64)v;
                    exact = (exact + mulmod(f, d + half, Q)) % Q;
                }
                for (int q = 0; q < NL; q++) top = labs(o[q]) > top ? labs(o[q]) : top;
                const u64 got = brt::recombine_sums<TC, LAZY>(o, cst, K.tc_t0, K.tc_m, (u32)(Q >> 32));
                // as a signed value: E never comes near 2^64, O is small
                const i128 x = e ? (i128)(int64_t)got : (i128)got;
                i128 r = (x - (i128)exact) % (i128)Q;
                if (r) {
                    printf("class %d %c pattern %d is not congruent\n", c, e ? 'O' : 'E', pat);
                    return 1;
                }
                lo[e] = x < lo[e] ? x : lo[e];
                hi[e] = x > hi[e] ? x : hi[e];
            }
        }
    auto floor1000 = [&](i128 x) { i128 v = x * 1000; return (long)(v >= 0 ? v / Q : -((-v + Q - 1) / Q)); };
    printf("%u %ld %ld %ld %ld %ld\n", choose_variant(p), top, floor1000(lo[0]), floor1000(hi[0]) + 1, floor1000(lo[1]),
           floor1000(hi[1]) + 1);
    return 0;
}

int main(int argc, char **argv) {
    if (argc != 4) return 2;
    bm_key_params p = {};
    p.n = 4;
    p.N = (u32)atoi(argv[1]);
    p.Q = strtoull(argv[2], nullptr, 10);
    p.log2_B = (u32)atoi(argv[3]);
    p.l_B = 6;
    u64 psi = 0;      // a primitive 2N-th root of unity
    for (u64 g = 2; !psi; g++) {
        const u64 x = powmod(g, (p.Q - 1) / (2 * p.N), p.Q);
        if (powmod(x, p.N, p.Q) == p.Q - 1) psi = x;
    }
    u32 logN = 0;
    while ((1u << logN) < p.N) logN++;
    std::vector<u64> tab(8 * (size_t)p.N);
    for (u32 k = 0; k < p.N; k++) {
        u32 br = 0;
        for (u32 b = 0; b < logN; b++) br |= ((k >> b) & 1) << (logN - 1 - b);
        tab[k] = powmod(psi, br, p.Q);
    }
    const u32 v = choose_variant(p);
    if (v & BR_V_TC1) return check<1, true>(p, tab);
    if (v & BR_V_TC2) return (v & BR_V_LAZY) ? check<2, true>(p, tab) : check<2, false>(p, tab);
    printf("%u 0 0 0 0 0\n", v);
    return 0;
}
