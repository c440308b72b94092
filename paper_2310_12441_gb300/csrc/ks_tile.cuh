// Key switching of many samples under one key: a thread block works on a tile
// of samples and kKskCols columns of the key.
//
// One block per sample (key_switch_block) reads N l_ks (n + 1) selected words
// of the key for every sample, 34 MB at n = 630, N = 1024: at 2000 samples that
// kernel takes 9.6 ms, bound by the L2 (7.1 TB/s).  Here the rows of a
// coefficient, all digits j and all digit values, come to shared memory once per
// tile of samples by one bulk copy of a contiguous slice of the key (copies by
// the threads took as long as the adds: 4.4 ms), and every sample adds the row
// its digit selects, so the L2 traffic falls by the samples of a tile and the
// bound is the shared-memory port: one 64-bit load per added word.  2000 samples
// 3.2 ms (2.0 ms for those loads at 128 B per cycle), 1000: 5.0 -> 2.1 ms, 300:
// 1.45 -> 1.10 ms.  Columns are split, not coefficients, so that few blocks
// share few samples with long sums and no partial results meet.
#pragma once
#include "common.cuh"
#include "modarith.cuh"

// a~ = floor((a P + floor(Q/2)) / Q) mod P, exact: the Shoup-style quotient
// estimate floor(a P' / 2^64), P' = floor(P 2^64 / Q), is at most 2 below the
// true quotient; the remainder fits in 64 bits and fixes it.
__device__ __forceinline__ u64 ks_round(u64 a, const KeyDev &K) {
    const u32 sh = K.log2_Bks * K.l_ks;
    const u64 Q = K.mq.Q;
    u64 q = __umul64hi(a, K.ks_pq);
    u64 r = (a << sh) + Q / 2 - q * Q;
    for (int it = 0; it < 3 && r >= Q; it++) { r -= Q; q++; }
    return q & ((1ull << sh) - 1);
}

namespace kst {

constexpr u32 kWarpsPer = 8;              // groups of samples per block, two warps (64 columns) each
constexpr u32 kThreads = kWarpsPer * kKskCols;
constexpr u32 kGroup = 4;                 // coefficients whose digits are made together
constexpr u32 kStageRows = 128;           // rows of a stage, the zero row included
constexpr u32 kMaxStages = 3;
constexpr u32 kMaxCpt = 24;               // samples per thread
constexpr u32 kMaxSmem = 227 * 1024;

// Digits j per stage: as many as have their rows and the zero row in it.
inline __host__ __device__ u32 digits_per_stage(u32 lks, u32 log2_Bks) {
    const u32 per = (kStageRows - 1) / ((1u << log2_Bks) - 1);
    return per < lks ? per : lks;
}
inline __host__ __device__ u32 stage_bytes(u32 lks, u32 log2_Bks) {
    return (1 + digits_per_stage(lks, log2_Bks) * ((1u << log2_Bks) - 1)) * kKskCols * 8;
}
// Shared memory: the stages, row offsets [2][kGroup][l_ks][samples], barriers.
inline __host__ __device__ u32 smem_bytes(u32 lks, u32 log2_Bks, u32 samples, u32 stages) {
    return stages * stage_bytes(lks, log2_Bks) + 2 * kGroup * lks * samples * 4 + 8 * kMaxStages;
}
// Two stages hide the copies of long tiles, three those of short ones.
inline __host__ __device__ u32 stages_of(u32 lks, u32 log2_Bks, u32 samples) {
    return smem_bytes(lks, log2_Bks, samples, 3) <= kMaxSmem ? 3 : 2;
}

__device__ __forceinline__ u32 smem_addr(const void *p) { return (u32)__cvta_generic_to_shared(p); }
// Bulk copy to shared memory, counted by the barrier `bar` (addresses and bytes
// multiples of 16).
__device__ __forceinline__ void bulk_load(void *dst, const void *src, u32 bytes, u64 *bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
// Bounded wait (2^20 polls, each of which may suspend the thread): false when
// it gave up.
__device__ __forceinline__ bool wait(u64 *bar, u32 parity) {
    for (u32 it = 0; it < (1u << 20); it++) {
        u32 ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(smem_addr(bar)), "r"(parity)
                     : "memory");
        if (ok) return true;
    }
    return false;
}

// CPT samples per thread.  load(s, i, v): kGroup coefficients i .. of sample s
// (the LWE mask words a_i .. a_i+kGroup-1); store(s, c, sum): sum of the
// selected rows, reduced.  A copy that never arrives (no correct launch has one)
// leaves ~0, no residue, in the outputs and BM_ETIMEDOUT in status, if given.
template <int CPT, class Load, class Store>
__device__ __forceinline__ void tile(const KeyDev &K, u32 first, u32 count, u32 col0, unsigned char *sm, Load load,
                                     Store store, u32 *status) {
    constexpr u32 SAMPLES = CPT * kWarpsPer;
    const u32 N = K.N, n = K.n, lks = K.l_ks, lb = K.log2_Bks, B1 = (1u << lb) - 1;
    const u32 tid = threadIdx.x, col = tid % kKskCols, grp = tid / kKskCols;
    const u32 jn = digits_per_stage(lks, lb);
    const u32 parts = (lks + jn - 1) / jn;                // stages per coefficient
    const u32 sbytes = stage_bytes(lks, lb), stages = stages_of(lks, lb, SAMPLES);
    const u32 width = ksk_slice_width(n, col0);
    u32 *offs = (u32 *)(sm + stages * sbytes);
    u64 *full = (u64 *)(offs + 2 * kGroup * lks * SAMPLES);
    // the zero row, which digit 0 selects, leads every stage
    for (u32 i = tid; i < stages * kKskCols; i += kThreads) ((u64 *)(sm + i / kKskCols * sbytes))[i % kKskCols] = 0;
    if (tid < stages)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full[tid])) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    const u32 total = N * parts;
    const u64 *slice = K.ksk + (size_t)col0 * lks * B1;
    const size_t coef = (size_t)lks * B1 * ksk_pitch(n);
    u32 fi = 0, fp = 0, fs = 0;               // the next fetch: coefficient, part, stage
    auto fetch = [&]() {                      // (one thread)
        const u32 j0 = fp * jn, j1 = j0 + jn < lks ? j0 + jn : lks;
        bulk_load(sm + fs * sbytes + kKskCols * 8, slice + fi * coef + (size_t)j0 * B1 * width, (j1 - j0) * B1 * width * 8,
                  &full[fs]);
        if (++fp == parts) fp = 0, fi++;
        if (++fs == stages) fs = 0;
    };
    if (tid == 0)
        for (u32 t = 0; t + 1 < stages && t < total; t++) fetch();
    // byte offsets in a stage of the rows that kGroup coefficients from i
    // select, one sample per thread
    const u32 s_own = first + tid;
    const bool own = tid < SAMPLES && s_own < count;
    u64 av[kGroup];
    auto digits = [&](u32 i) {
        if (tid >= SAMPLES) return;
        u32 *o = offs + ((i / kGroup) & 1) * kGroup * lks * SAMPLES + tid;
#pragma unroll
        for (u32 g = 0; g < kGroup; g++) {
            const u64 at = own ? ks_round(av[g], K) : 0;
            for (u32 j = 0, r = 0; j < lks; j++, r = r + 1 == jn ? 0 : r + 1) {
                const u32 d = (u32)(at >> (lb * j)) & B1;
                o[(g * lks + j) * SAMPLES] = d ? kKskCols * 8 + (r * B1 + d - 1) * width * 8 : 0;
            }
        }
    };
    u64 lo[CPT];
    u32 hi[CPT];
#pragma unroll
    for (int q = 0; q < CPT; q++) lo[q] = hi[q] = 0;
    if (own) load(s_own, 0, av);
    digits(0);
    if (own && kGroup < N) load(s_own, kGroup, av);
    bool dead = false;
    u32 st = 0, parity = 0, i = 0, p = 0;
    for (u32 t = 0; t < total; t++) {
        dead = !wait(&full[st], parity);
        // stage t and its offsets are there; stage t - 1 has been read
        if (__syncthreads_or(dead)) break;
        if (tid == 0 && t + stages - 1 < total) fetch();
        if (p == 0 && i % kGroup == kGroup - 1 && i + 1 < N) {
            digits(i + 1);            // (the next group's, read after the next barrier)
            if (own && i + 1 + kGroup < N) load(s_own, i + 1 + kGroup, av);
        }
        const u32 j0 = p * jn, j1 = j0 + jn < lks ? j0 + jn : lks;
        const unsigned char *sc = sm + st * sbytes + col * 8;
        const u32 *o = offs + (((i / kGroup) & 1) * kGroup + i % kGroup) * lks * SAMPLES + grp * CPT;
        for (u32 j = j0; j < j1; j++) {
#pragma unroll
            for (int q = 0; q < CPT; q += 4) {
                const uint4 r = *reinterpret_cast<const uint4 *>(o + j * SAMPLES + q);
                const u32 rr[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const u64 v = *reinterpret_cast<const u64 *>(sc + rr[k]);
                    asm("add.cc.u64 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+l"(lo[q + k]), "+r"(hi[q + k]) : "l"(v));
                }
            }
        }
        if (++st == stages) st = 0, parity ^= 1;
        if (++p == parts) p = 0, i++;
    }
    if (i < N) {      // gave up: no copy may be in flight when the block ends
        for (u32 k = 0; k < stages; k++) wait(&full[k], k < st ? parity ^ 1 : parity);
        if (tid == 0 && status) atomicCAS(status, 0u, (u32)(-BM_ETIMEDOUT));
    }
    if (col0 + col <= n) {
#pragma unroll
        for (int q = 0; q < CPT; q++) {
            const u32 s = first + grp * CPT + q;
            if (s < count) store(s, col0 + col, reduce128(lo[q], hi[q], K.mq), i < N);
        }
    }
}

}  // namespace kst
