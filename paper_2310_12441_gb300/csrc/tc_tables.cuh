// Weights of the tensor-core transform stages (br_tc.cuh) and the way back from
// their limb sums to values modulo Q: what the host prepares for a key and what
// the transform warps compute, side by side because one's constants carry the
// other's bounds.  The recombination also compiles for the host, where a test
// checks those bounds with exact integers.
#pragma once
#include <cstring>
#include <vector>

#include <cuda_fp16.h>

#include "common.cuh"

namespace brt {

// Tensor-core configurations (signed limbs of the weights): TC1 for Q < 2^54
// and log2 B <= 9, TC2 for Q < 2^60 and log2 B <= 10.
template <int TC>
struct Limbs {
    static constexpr int NL = TC == 1 ? 5 : 6;
    static constexpr int R = TC == 1 ? 11 : 10;
};

// Units of 2^((NL - 1) R - 4) taken off the quotient estimate of recombine, so
// that it never exceeds the quotient: the limb sums that it leaves out and the
// part it cuts off those it reads.  TC1 leaves out limbs 0..2, below 65 units;
// TC2 limbs 0..3, below 257; lazy TC2 limbs 0..2, below 1.
template <int TC, bool LAZY>
struct Bias {
    static constexpr u32 value = TC == 2 && LAZY ? 4 : 600;
};

// Limb sums of one value -> E or O modulo Q: sum_l o_l 2^(R l) + cst - q Q with
// the quotient q of the value's top bits, the sum modulo 2^64.  cst carries the
// centring constant, a multiple of Q above every negative value (which the
// quotient takes off again) and the multiple that the later stages start from.
//
// Without the last, the result lies in [0, 2.34 Q): below Q of centring
// constant, below Q of the quotient's fraction, 0.13 Q of its factor m (v below
// 2^29.1, m one below 2^(32 + unit) / Q), and bias and cut-off parts.  These are
// units of 2^40 (TC1) or 2^46 (TC2), at most 666 and 859 of them: 0.11 Q at
// TC1's smallest Q of 2^52.6, 0.21 Q at 2^58, the smallest Q of TC2 without
// LAZY.  Lazy TC2 goes down to 2^52.5, where 859 units are 9 Q, so it reads a
// third limb and is left with 8 units, 0.08 Q.
template <int TC, bool LAZY>
__host__ __device__ __forceinline__ u64 recombine_sums(const int32_t (&o)[Limbs<TC>::NL], u64 cst, u32 t0, u32 mq,
                                                       u32 c) {
    constexpr int R = Limbs<TC>::R, NL = Limbs<TC>::NL;
    // (on the device written out so that the additions stay off the multiplier)
#ifdef __CUDA_ARCH__
    auto add = [](u64 a, u64 b) { return add64c(a, b); };
    auto sub = [](u64 a, u64 b) { return sub64c(a, b); };
    auto mulhi = [](u32 a, u32 b) { return __umulhi(a, b); };
    auto plus = [](u64 t, int32_t v, int32_t k) {
        u64 r;
        asm("{\n\t.reg .u64 p;\n\tmul.wide.s32 p, %2, %3;\n\tadd.u64 %0, %1, p;\n\t}" : "=l"(r) : "l"(t), "r"(v), "r"(k));
        return r;
    };
#else
    auto add = [](u64 a, u64 b) { return a + b; };
    auto sub = [](u64 a, u64 b) { return a - b; };
    auto mulhi = [](u32 a, u32 b) { return (u32)(((u64)a * b) >> 32); };
    auto plus = [](u64 t, int32_t v, int32_t k) { return t + (u64)((int64_t)v * k); };
#endif
    // value modulo 2^64
    u64 t = plus(plus(cst, o[1], 1 << R), o[2], 1 << (2 * R));
    if constexpr (NL == 6) t = plus(t, o[3], 1 << (3 * R));
    t = add(t, (u64)(int64_t)o[0]);
    u32 hi = (u32)(t >> 32) + ((u32)o[NL - 1] << ((NL - 1) * R - 32));
    hi += (u32)o[NL - 2] << ((NL - 2) * R - 32);
    if constexpr (NL == 5) static_assert((NL - 2) * R >= 32, "high limbs");
    // quotient from the top limbs, in units of 2^((NL - 1) R - 4)
    u32 v = ((u32)o[NL - 1] << 4) + (u32)(o[NL - 2] >> (R - 4)) + t0;
    if constexpr (TC == 2 && LAZY) v += (u32)(o[NL - 3] >> (2 * R - 4));
    const u32 q = mulhi(v, mq);
    hi -= q * c;
    return sub(((u64)hi << 32) | (u32)t, q);
}
#ifdef __CUDACC__
template <int TC, bool LAZY>
__device__ __forceinline__ u64 recombine(const u32 (&f)[Limbs<TC>::NL], u64 cst, u32 t0, u32 mq, u32 c) {
    int32_t o[Limbs<TC>::NL];
#pragma unroll
    for (int l = 0; l < Limbs<TC>::NL; l++) o[l] = __float2int_rn(__uint_as_float(f[l]));
    return recombine_sums<TC, LAZY>(o, cst, t0, mq, c);
}
#endif

// Tables of the tensor-core transform stages (br_tc.cuh) for a key with a
// BR_V_TC* flag: fp16 limbs of the weights w_p^(2i), w_p^(2i + 1) (centred
// modulo Q, signed limbs of R bits, K-major 8x16-byte core matrices), the
// additive constants of the E and O sums, the twiddle pairs of stages 7 and
// up, [stage position][class parity][class / 2], and the inverse pairs in the
// order of ntr::inv_twiddle_slot for radix 8.
inline std::vector<unsigned char> tc_tables(const bm_key_params &p, u32 variant, const std::vector<u64> &tab,
                                            KeyDev &K) {
    typedef unsigned __int128 u128;
    auto mulmod = [&](u64 a, u64 b) { return (u64)((u128)a * b % p.Q); };
    auto shoup = [&](u64 w) { return (u64)(((u128)w << 64) / p.Q); };
    const u32 NL = (variant & BR_V_TC1) ? 5 : 6, R = (variant & BR_V_TC1) ? 11 : 10, N = p.N;
    const u64 Q = p.Q;
    const u32 nt = N / 128 - 1;
    std::vector<unsigned char> out(NL * 16384 + 1024 + (size_t)nt * 2048 + (size_t)N * 16);
    // a multiple of Q above every |sum|: sums stay within 64 2^(log2 B - 1) 2^(R - 1) per limb
    const u32 sbits = 6 + p.log2_B - 1 + R - 1 + (NL - 1) * R;
    const u128 off = ((((u128)1 << sbits) + ((u128)1 << (sbits - 4))) / Q + 1) * Q;
    const u32 unit = (NL - 1) * R - 4;
    const u32 bias = (variant & BR_V_TC1) ? Bias<1, true>::value
                     : (variant & BR_V_LAZY) ? Bias<2, true>::value : Bias<2, false>::value;
    K.tc_t0 = (u32)(off >> unit) - bias;
    K.tc_m = (u32)(((u128)1 << (unit + 32)) / Q);
    // limb radices of the multiply-accumulate with their Shoup companions
    const u32 lb = br_qlow1_limb(variant);
    K.tc_b1 = (1ull << lb) % Q;
    K.tc_b1s = shoup(K.tc_b1);
    K.tc_b2 = (1ull << (2 * lb)) % Q;
    K.tc_b2s = shoup(K.tc_b2);
    // (v >> 32) / (c + 1) with c = Q >> 32, 2^tc_fsh <= c < 2^(tc_fsh + 1)
    const u64 c1 = (Q >> 32) + 1;
    K.tc_fsh = 0;
    while ((2ull << K.tc_fsh) < c1) K.tc_fsh++;
    K.tc_fs = (u32)(((u128)1 << (32 + K.tc_fsh)) / c1);
    // (8192 powers and 40960 or more limbs: Shoup products and looked-up halves
    // instead of 128-bit divisions and conversions)
    uint16_t half[2049];       // -1024 .. 1024 in fp16
    for (int v = -1024; v <= 1024; v++) {
        const __half h = __float2half((float)v);
        memcpy(&half[v + 1024], &h, 2);
    }
    for (u32 c = 0; c < 64; c++) {
        const u64 w = tab[64 + c], w2 = mulmod(w, w), w2s = shoup(w2);
        u64 f[2] = {1 % Q, w};
        u128 sum[2] = {0, 0};
        for (u32 i = 0; i < 64; i++) {
            for (u32 e = 0; e < 2; e++) {
                sum[e] += f[e];
                int64_t v = f[e] > Q / 2 ? (int64_t)f[e] - (int64_t)Q : (int64_t)f[e];
                for (u32 l = 0; l < NL; l++) {
                    int64_t r = v;
                    if (l + 1 < NL) {
                        r = ((v + (1 << (R - 1))) & ((1 << R) - 1)) - (1 << (R - 1));
                        v = (v - r) >> R;
                    }
                    memcpy(&out[(e * NL + l) * 8192 + (c / 8) * 1024 + (i / 8) * 128 + (c % 8) * 16 + (i % 8) * 2],
                           &half[r + 1024], 2);
                }
                const u64 x = f[e] * w2 - (u64)(((u128)f[e] * w2s) >> 64) * Q;
                f[e] = x >= Q ? x - Q : x;
            }
        }
        for (u32 e = 0; e < 2; e++) {
            u64 cst = mulmod((u64)(sum[e] % Q), (1ull << (p.log2_B - 1)) % Q);
            // E in [2Q, 4.34Q), O in [-2Q, 0.34Q) (recombine_sums); lazy keys
            // start 4Q higher per remaining stage but the last
            const u64 up = (variant & BR_V_LAZY) ? 4 * (u64)(K.logN - 8) : 0;
            cst += (u64)off + (e == 0 ? (2 + up) * Q : 0 - 2 * Q);
            memcpy(&out[NL * 16384 + e * 512 + c * 8], &cst, 8);
        }
    }
    u32 pos = 0;
    for (u32 s = 7; (1u << s) < N; s++)
        for (u32 g = 0; g < (1u << (s - 7)); g++, pos++)
            for (u32 k = 0; k < 128; k++)
                memcpy(&out[NL * 16384 + 1024 + pos * 2048 + ((k & 1) * 64 + k / 2) * 16],
                       &tab[4 * (size_t)N + 2 * ((1u << s) + (k << (s - 7)) + g)], 16);
    for (u32 i = 1; i < N; i++) {
        u32 s = 0;
        while ((2u << s) <= i) s++;
        const u32 q = (K.logN - 1 - s) / 3, F = q < (K.logN + 2) / 3 - 1 ? 3 * q : K.logN - 3, sh = K.logN - 3 - F;
        const u32 r = i - (1u << s), j = r >> sh, high = r & ((1u << sh) - 1);
        memcpy(&out[NL * 16384 + 1024 + (size_t)nt * 2048 + (size_t)i * 16],
               &tab[6 * (size_t)N + 2 * ((1u << s) + ((high << (s - sh)) | j))], 16);
    }
    return out;
}

}  // namespace brt
