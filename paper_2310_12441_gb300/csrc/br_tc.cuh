// Blind rotation with the first seven forward-transform stages on the tensor
// cores (ring degrees 1024 and 2048, moduli Q = c 2^32 + 1).
//
// The digit polynomials are small (log2 B <= 10 bits), so the leading stages
// of their transforms are a contraction of small integers with fixed 64-bit
// weights.  With N = 64 S, coefficient S i + j' (i < 64, j' < S) and r_p the
// root of node p after six Cooley-Tukey stages (x^S - r_p, r_p = w_p^2,
// w_p = psi^bitrev(64 + p)), stage 6 gives, for j < S/2,
//   Y_2p[j]   = E + O,   E = sum_i d[S i + j]       w_p^(2i),
//   Y_2p+1[j] = E - O,   O = sum_i d[S i + S/2 + j] w_p^(2i+1):
// two matrix products with K = 64 and no twiddle multiplication.  The weights
// are centred, split into NL signed limbs of R bits (fp16, exact), the digits
// are centred (d - 2^(log2 B - 1), fp16, exact; the missing constant times
// sum_i w is one additive constant per class), and every limb product sum
// stays within +-2^24, so the fp32 accumulators hold it
// exactly.  The transform warps recombine the limbs modulo Q and run the
// remaining log N - 7 stages in registers.
//
// Tensor-core layout: A = weights [64 classes p][64 i] per limb and E / O
// (K-major, 8x16-byte core matrices), B = digits [32 columns][64 i].  An
// M = 64 product occupies lanes 0-15 of every 32-lane TMEM quadrant, so two
// products (column halves) interleave: half 0 in lanes 0-15, half 1 in lanes
// 16-31.  At N = 1024 the halves are two digit polynomials, at N = 2048 the
// two halves of j of one polynomial (lanes L and L ^ 16 then swap one class
// each).  Either way a transform thread holds 16 values of one or two classes.
//
// Roles of the 20 warps (the phases would otherwise leave each other's units
// idle: with every warp doing all of them in turn the same work took 2x as
// long, waiting for L2, TMEM and barriers):
//   - transform warps 0-7: accumulators -> transformed polynomials, in
//     shared-memory stages of 64 KB / 2;
//   - product warps 8-15: multiply-accumulate with the key rows, inverse
//     transforms, accumulator update, order of the work;
//   - warp 16 issues the tensor-core instructions;
//   - digit warps 17-19: the digits of the next row.
// A block works on two jobs in turn, one CMux step of each at a time, so the
// inverse transforms and digits at a job's step boundary overlap the other
// job's transforms; blocks take further jobs from a counter.
//
// What bounds it: at N = 1024 the 32-bit multiplier pipe (recombination, three
// remaining stages, multiply-accumulate, inverse transforms), 67% busy with two
// jobs in every block (63% with one) against 54% (51%) of the issue slots and 11%
// of the tensor pipe.  At N = 2048 no unit: multiplier and issue slots read 52%
// with one job or two, and long scoreboard (key rows and accumulators from the
// L2, TMEM) leads the stalls, so the roles wait for one another.
// Per row of one CMux step and SM, blocks full: N = 1024, Q < 2^54: 24.9 us with
// all stages in the CUDA cores (br_job), 16.7 us here; N = 2048, Q < 2^60: 64.2
// and 56.3 us.  1000 bootstraps at N = 1024 with m = 4: 444 and 312 ms; 200 at
// N = 2048 with m = 8: 579 and 512 ms.
#pragma once
#include "blind_rotate.cuh"
#include "tc_tables.cuh"

namespace brt {

constexpr u32 kT = 256, kM = 256;            // transform and product threads
constexpr u32 kD = 96;                       // digit threads
constexpr u32 kThreads = kT + kM + 32 + kD;  // + the issuing warp
constexpr u32 kTile = 16384;                 // B bytes of one batch (8 half-column tiles of 2 KB)

template <int LOGN, int TC>
struct Cfg {
    static constexpr int N = 1 << LOGN;
    static constexpr int S = N / 64;                 // coefficients per node after six stages
    static constexpr int NL = Limbs<TC>::NL;
    static constexpr int CB = 8192 / N;              // digit polynomials per batch
    static constexpr int RC = CB / 2;                // per round (two rounds per batch)
    static constexpr int PH = N / 512;               // pairs of adjacent positions per product thread
    static constexpr int PAIRS = LOGN == 10 ? 4 : 1;  // (sign, component) pairs whose digits are made at once
    static constexpr int NT = N / 128 - 1;           // twiddles per class (stages 7 .. log N - 1)
    static constexpr u32 A_BYTES = NL * 2 * 8192;
    static constexpr u32 TW_TAB = A_BYTES + 1024;    // offsets in the key's table: twiddles,
    static constexpr u32 ITW_TAB = TW_TAB + NT * 2048;   // inverse twiddles
    static constexpr u32 B_OFF = A_BYTES;
    static constexpr u32 TILES = LOGN == 10 ? 3 : 2; // batches whose digits are resident
    static constexpr u32 X_OFF = B_OFF + TILES * kTile;
    static constexpr u32 XS = 32768;                 // bytes of one of the two stages
    static constexpr u32 I_OFF = X_OFF + 2 * XS;     // inverse transforms
    static constexpr int NTS = 7;                    // twiddles per class in shared memory
    static constexpr u32 TW_OFF = I_OFF + 16384;
    static constexpr u32 SMEM = TW_OFF + NTS * 2048;
    static constexpr u32 SUM_COL = NL * 64;          // TMEM columns of the row sums
    static_assert(SUM_COL + 2 * PH * 16 <= 512, "TMEM columns");
    static_assert(SMEM <= 227 * 1024 - 1024, "shared memory per block");
};

// ---- tcgen05 ------------------------------------------------------------
__device__ __forceinline__ u64 smem_desc(u32 addr, u32 lbo, u32 sbo) {
    return (u64)((addr >> 4) & 0x3fff) | ((u64)(lbo >> 4) << 16) | ((u64)(sbo >> 4) << 32) | (1ull << 46);
}
__device__ __forceinline__ u32 elect_one() {
    u32 p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p;
}
template <bool ACC>
__device__ __forceinline__ void mma_f16(u32 d, u64 a, u64 b, u32 idesc) {
    if constexpr (ACC)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, 0, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b),
                     "r"(idesc)
                     : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, 0, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b),
                     "r"(idesc)
                     : "memory");
}
__device__ __forceinline__ void mma_commit(u64 *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld2(u32 addr, u32 (&r)[2]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 16 words of this thread's lane: the row sums of one pair of positions.
__device__ __forceinline__ void tmem_ld16(u32 addr, u32 (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_st16(u32 addr, const u32 (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15, %16};" ::"r"(addr),
                 "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
                 "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Barrier of the product warps.
__device__ __forceinline__ void bar_m() { asm volatile("bar.sync 5, 256;" ::: "memory"); }

// Waits of a whole warp for the phase of `bar` with this parity (acquire, CLUSTER:
// from the blocks of the cluster).  Bounded: a warp that polled `polls` times
// (each poll may suspend it for a while) sets BM_ETIMEDOUT in the status word
// and `dead` for the block, which every wait that goes on polling looks at.
// False, for the whole warp alike: the block has given up.  (No correct launch
// has such a wait.)  Transform, digit and issuing warps then leave at once;
// product warps share barriers, so they go on without waiting, on words that
// need not be what they should be, to the step's end and leave there together
// (bar_or), before another job's state can take the slot's place.
constexpr u32 kPolls = 1u << 24;
template <bool CLUSTER = false>
__device__ __forceinline__ bool poll(u64 *bar, u32 parity) {
    u32 ok;
    if constexpr (CLUSTER)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(smem_u32(bar)), "r"(parity)
                     : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(smem_u32(bar)), "r"(parity)
                     : "memory");
    return __all_sync(0xffffffffu, ok);
}
template <bool CLUSTER = false>
[[nodiscard]] __device__ __forceinline__ bool wait(u64 *bar, u32 parity, u32 *dead, u32 *status, u32 polls = kPolls) {
    for (u32 it = 0; !poll<CLUSTER>(bar, parity); it++) {
        if (it == polls) {
            set_status(status, BM_ETIMEDOUT);
            *(volatile u32 *)dead = 1;
            return false;
        }
        if (it % 32 == 31 && __any_sync(0xffffffffu, *(volatile u32 *)dead)) return false;
    }
    return true;
}

// Register split of the 640 threads launched with 96 each: per thread of four
// warps 2 x 88 + 2 x 112 + 80 = 480 = 5 x 96, exactly what the block holds.
__device__ __forceinline__ void regs_transform() { asm volatile("setmaxnreg.dec.sync.aligned.u32 88;"); }
__device__ __forceinline__ void regs_product() { asm volatile("setmaxnreg.inc.sync.aligned.u32 112;"); }
__device__ __forceinline__ void regs_other() { asm volatile("setmaxnreg.dec.sync.aligned.u32 80;"); }

// A job's state in its block slot.
struct Slot {
    u64 *cur, *nxt;
    const u64 *ct;
    const u32 *gpre;
    u32 m, mr, k, steps, gS;
    u32 on;
};

// A unit of work: the digits of PAIRS pairs of one row.
struct Unit {
    u32 slot, row, part;
    u32 ncomb;              // its digit polynomials (0: leave)
    u32 newkey;
};

// Shared control block.
struct Shared {
    Slot slot[2];           // written by one product thread between barriers
    Unit unit[4];           // unit u at u & 3
    const KeyDev *key;      // key of the units
    u64 post[2];            // unit u posted (u & 1; one product thread)
    u64 bfull[3], bempty[3];    // digit tiles: stored (digit warps) / consumed (products complete)
    u64 tfull, tempty;      // a batch's accumulators complete / read (transform warps)
    u64 xfull[2], xempty[2];    // a stage's polynomials stored / multiplied
    u64 cbar;               // cluster barrier of the product warps
    u64 drain;              // every product complete
    u32 dead;               // a wait of this block has given up: every role leaves
    u32 tmem;
    u32 next;               // a job index taken from the counter
    u32 taken;              // jobs this block has started
    int bad;
};

// bar_m that says, to all product warps alike, whether the block has given up.
__device__ __forceinline__ bool bar_or(Shared &sh) {
    u32 r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 5, 256, p;\n\t"
                 "selp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(r)
                 : "r"(*(volatile u32 *)&sh.dead)
                 : "memory");
    return r != 0;
}

__device__ __forceinline__ void open(Shared &sh, u32 csize) {
    if (threadIdx.x == 0) {
        for (int i = 0; i < 3; i++) {
            mbar_init(&sh.bfull[i], kD / 32);
            mbar_init(&sh.bempty[i], 1);
        }
        mbar_init(&sh.tfull, 1);
        mbar_init(&sh.tempty, kT / 32);
        for (int i = 0; i < 2; i++) {
            mbar_init(&sh.post[i], 1);
            mbar_init(&sh.xfull[i], kT / 32);
            mbar_init(&sh.xempty[i], kM / 32);
        }
        mbar_init(&sh.cbar, csize * (kM / 32));
        mbar_init(&sh.drain, 1);
        sh.dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x / 32 == (kT + kM) / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sh.tmem))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    if (csize > 1) cluster_sync();     // peers arrive on this block's cbar
    fence_after();
}
__device__ __forceinline__ void close(Shared &sh, u32 csize) {
    fence_before();
    __syncthreads();
    if (csize > 1) cluster_sync();
    fence_after();
    if (threadIdx.x / 32 == (kT + kM) / 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(sh.tmem));
}

// One step's barrier over the product warps of every block of a cluster
// (global writes before it are visible after it); false as wait().
[[nodiscard]] __device__ __forceinline__ bool cluster_bar_m(Shared &sh, u32 csize, u32 &parity, u32 *status) {
    __threadfence();
    __syncwarp();
    if (threadIdx.x % 32 == 0) {
        const u32 local = smem_u32(&sh.cbar);
        for (u32 r = 0; r < csize; r++) {
            u32 remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(r));
            asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
        }
    }
    const bool ok = wait<true>(&sh.cbar, parity, &sh.dead, status);
    parity ^= 1;
    __threadfence();
    return ok;
}

// The issuing warp: per unit its batches; per batch A E / O x limbs x two
// column halves, K = 64 in four steps.
template <class C>
__device__ __forceinline__ void issuer(Shared &sh, unsigned char *sm, u32 *status) {
    const u32 sa = smem_u32(sm), sb = sa + C::B_OFF, tmem = sh.tmem;
    constexpr u32 idesc = (1u << 4) | ((32u >> 3) << 17) | ((64u >> 4) << 24);
    const u64 da = smem_desc(sa, 128, 1024);
    u32 pb = 0, pe = 1;      // (tempty: the first wait passes, as if a batch had been read)
    for (u32 u = 0;; u++) {
        bool ok = wait(&sh.post[u & 1], (u >> 1) & 1, &sh.dead, status);
        const u32 ncomb = *(volatile u32 *)&sh.unit[u & 3].ncomb;
        for (u32 b = 0; ok && b * C::CB < ncomb; b++) {
            // (tempty: the previous batch's accumulators have been read)
            ok = wait(&sh.bfull[b], (pb >> b) & 1, &sh.dead, status) && wait(&sh.tempty, pe, &sh.dead, status);
            if (!ok) break;
            pb ^= 1u << b;
            pe ^= 1;
            fence_after();
            if (elect_one()) {
                const u64 db = smem_desc(sb + b * kTile, 128, 4096);
#pragma unroll 1
                for (u32 el = 0; el < 2 * C::NL; el++) {
                    const u64 a = da + el * (8192 >> 4), bb = db + (el >= C::NL ? 1024 >> 4 : 0);
                    const u32 d = tmem + el * 32;
#pragma unroll
                    for (u32 hf = 0; hf < 2; hf++) {
                        const u64 bh = bb + hf * (2048 >> 4);
                        const u32 dh = d + (hf << 20);
                        mma_f16<false>(dh, a, bh, idesc);
                        mma_f16<true>(dh, a + 16, bh + 16, idesc);
                        mma_f16<true>(dh, a + 32, bh + 32, idesc);
                        mma_f16<true>(dh, a + 48, bh + 48, idesc);
                    }
                }
                mma_commit(&sh.tfull);
                mma_commit(&sh.bempty[b]);
            }
            __syncwarp();
        }
        if (!ok) break;
        if (ncomb == 0) {      // wakes the transform warps, which leave too
            if (elect_one()) mbar_arrive(&sh.tfull);
            break;
        }
    }
    // no product may be outstanding when the block ends (none is, unless it gave up)
    if (elect_one()) mma_commit(&sh.drain);
    __syncwarp();
    for (u32 it = 0; it < kPolls && !poll(&sh.drain, 0); it++) {}
}

// Digit warps: for every unit and pair the differences D = P(c) ACC - ACC of
// the row, four coefficients S (8 ig + 4 f + i) + j' per item, and their
// digits, centred, as 8 bytes of each digit's B tile.
template <int LOGN, int TC>
__device__ __forceinline__ void digit_warps(Shared &sh, unsigned char *sm, u32 crank, u32 csize, u32 *status) {
    using C = Cfg<LOGN, TC>;
    constexpr u32 N = C::N, S = C::S;
    const u32 dt = threadIdx.x - (kT + kM + 32), lane = dt % 32;
    u32 pe = 7;              // bempty parities (first waits pass)
    for (u32 u = 0;; u++) {
        if (!wait(&sh.post[u & 1], (u >> 1) & 1, &sh.dead, status)) return;
        const Unit un = *(const Unit *)&sh.unit[u & 3];
        if (un.ncomb == 0) break;
        const KeyDev *K = sh.key;
        const Slot &s = sh.slot[un.slot];
        const u32 lB = K->l_B, log2B = K->log2_B, m = s.m, r = crank + csize * un.row, qp = 2u * N * m;
        const u64 Q = K->mq.Q;
        const u64 *cur = s.cur;
        const u64 ctk = s.ct[s.k];
        const u32 ak = (qp & (qp - 1)) == 0 ? (u32)ctk & (qp - 1) : (u32)(ctk % qp);
        if constexpr (LOGN == 10) {
            // A few clusters walk the key, larger than the L2, one step's rows at
            // a time and at HBM latency: the launch's blocks bring the next
            // step's rows to the L2, 1 KB each in turn (30 jobs of 630 steps 16.4
            // -> 15.7 ms; one job 15.7, without it 15.4 to 17.1 by where the key
            // lies; at N = 2048 the loads are spread over twice the work and it
            // costs 1%).
            if (csize > 1 && un.row == 0 && un.part == 0 && s.k + 1 < s.steps) {
                const u32 chunks = 4 * lB * 2 * N * 8 / 1024;
                const unsigned char *next = (const unsigned char *)(K->bsk + (size_t)(s.k + 1) * 4 * lB * 2 * N);
                for (u32 ch = blockIdx.x + dt * gridDim.x; ch < chunks; ch += kD * gridDim.x)
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(next + (size_t)ch * 1024), "r"(1024u)
                                 : "memory");
            }
        }
        const u32 dmask = ((1u << log2B) - 1) * 0x10001u;
        const u32 dcen = (0x6400u | (1u << (log2B - 1))) * 0x10001u;     // fp16 1024 + 2^(log2 B - 1), twice
        u32 got = 0, c = 0;  // tiles taken, digit polynomials done
#pragma unroll 1
        for (u32 pr = 0; pr < (u32)C::PAIRS; pr++) {
            for (u32 b = c / C::CB; b <= (c + lB - 1) / C::CB; b++)
                if (!((got >> b) & 1)) {
                    if (!wait(&sh.bempty[b], (pe >> b) & 1, &sh.dead, status)) return;
                    pe ^= 1u << b;
                    got |= 1u << b;
                }
            const u32 pair = C::PAIRS * un.part + pr, sgn = pair >> 1, comp = pair & 1;
            const u32 cv = sgn == 0 ? (ak ? qp - ak : 0u) : ak;
            u32 src, e;
            mmpm_row(cv, r, m, 2 * N, s.gS, s.gpre, src, e);
            const bool flip = e >= N;
            const u32 es = flip ? e - N : e;
            const u64 *srow = cur + (size_t)(src * 2 + comp) * N;
            const u64 *orow = cur + (size_t)(r * 2 + comp) * N;
            u64 vn[4], on[4];
            auto fetch = [&](u32 item) {
                const u32 i0 = S * (8 * (item / (2 * S)) + 4 * ((item / S) & 1)) + item % S;
#pragma unroll
                for (u32 i = 0; i < 4; i++) {
                    vn[i] = __ldcg(srow + ((i0 + S * i - es) & (N - 1)));
                    on[i] = __ldcg(orow + i0 + S * i);
                }
            };
            fetch(dt);
#pragma unroll 1
            for (u32 item = dt; item < 16 * S; item += kD) {
                // (the accumulator words of the next item are requested first)
                u64 D[4], o[4];
#pragma unroll
                for (u32 i = 0; i < 4; i++) {
                    D[i] = vn[i];
                    o[i] = on[i];
                }
                if (item + kD < 16 * S) fetch(item + kD);
                const u32 jp = item % S, f = (item / S) & 1, ig = item / (2 * S);
                const u32 i0 = S * (8 * ig + 4 * f) + jp;
                // digit polynomial c at c kTile / CB; its tile of (half, e): N = 1024
                // e = j' / 8 (half from the polynomial), N = 2048 half and e from j'
                u32 at = smem_u32(sm) + C::B_OFF + c * (kTile / C::CB) + ig * 128 + (jp & 7) * 16 + f * 8;
                if constexpr (LOGN == 10) at += (jp >> 3) * 1024;
                else at += ((jp >> 3) & 1) * 2048 + (jp >> 4) * 1024;
                u32 lo[4], hi[4];
#pragma unroll
                for (u32 i = 0; i < 4; i++) {
                    const u64 sv = ((i0 + S * i < es) != flip) ? sub_mod(0, D[i], Q) : D[i];
                    const u64 v = sub_mod(sv, o[i], Q);
                    lo[i] = (u32)v;
                    hi[i] = (u32)(v >> 32);
                }
#pragma unroll 6
                for (u32 d = 0; d < lB; d++) {
                    u32 w[2];
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        const u32 v = (__byte_perm(lo[2 * i], lo[2 * i + 1], 0x5410) & dmask) | 0x64006400u;
                        const __half2 hh = __hsub2(*reinterpret_cast<const __half2 *>(&v),
                                                   *reinterpret_cast<const __half2 *>(&dcen));
                        w[i] = *reinterpret_cast<const u32 *>(&hh);
                    }
                    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(w[0]), "r"(w[1]) : "memory");
                    at += kTile / C::CB;
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        lo[i] = __funnelshift_r(lo[i], hi[i], log2B);
                        hi[i] >>= log2B;
                    }
                }
            }
            // tiles that are complete
            const u32 c1 = c + lB;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                for (u32 b = c / C::CB; b * C::CB < c1; b++)
                    if (c1 >= (b + 1) * C::CB || c1 == un.ncomb) mbar_arrive(&sh.bfull[b]);
            }
            c = c1;
        }
    }
}

// v minus 8Q when v >= 2^63 (Q < 2^60: the result is below 2^63).
__device__ __forceinline__ u64 csub8q(u64 v, u64 eightQ) {
    const u64 mask = (u64)((int64_t)v >> 63);
    return v - (eightQ & mask);
}

// Last stages of one class in registers: V values, twiddles tw(t) (t = 0 ..
// V - 2 in stage order).  LAZY: no corrections, every stage but the last widens
// the range by 4Q to both sides (the last by 4Q upwards); else (Q < 2^60,
// values start below 6.34Q) two stages without correction (14.34Q), one
// subtraction of 8Q from values above 2^63, two more stages: below 2^63 + 8Q.
template <int V, bool LAZY, class Tw>
__device__ __forceinline__ void class_stages(u64 (&x)[V], Tw tw, u32 c, u64 fourQ) {
    static_assert(V == 8 || V == 16, "three or four stages");
#pragma unroll
    for (int h = V / 2, g0 = 0; h >= 1; g0 = 2 * g0 + 1, h /= 2) {
        if (!LAZY && g0 == 3) {
#pragma unroll
            for (int i = 0; i < V; i++) x[i] = csub8q(x[i], 2 * fourQ);
        }
#pragma unroll
        for (int g = 0; g < V / (2 * h); g++) {
            const ulonglong2 w = tw(g0 + g);
#pragma unroll
            for (int j = 0; j < h; j++) {
                u64 &X = x[g * 2 * h + j], &Y = x[g * 2 * h + j + h];
                if (!LAZY || h == 1) {
                    bfly_lazy_qlow1(X, Y, w.x, w.y, c, fourQ);
                } else {
                    // X + T, X - T: the values start 4Q higher per such stage
                    const u64 T = shoup3_qlow1_lazy(Y, w.x, w.y, c), x0 = X;
                    X = add64c(x0, T);
                    Y = sub64c(x0, T);
                }
            }
        }
    }
}

// 32 bytes of key words: two adjacent positions of one combo.
struct Key2 { u64 a0, a1, b0, b1; };
__device__ __forceinline__ Key2 key_load4(const u64 *p) {
    Key2 k;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(k.a0), "=l"(k.a1), "=l"(k.b0), "=l"(k.b1) : "l"(p));
    return k;
}

// Karatsuba limb products of x with the key words of both columns (LB-bit
// limbs, products and additions split as in brk::br_job's kara2).
template <u32 LB>
__device__ __forceinline__ void kara2(u64 xv, u64 w0, u64 w1, u64 (&kh)[2], u64 (&kl)[2], u64 (&km)[2]) {
    asm("{\n\t.reg .u32 v0, v1, x0, x1, xs, a0, a1, as, c0, c1, cs;\n\t.reg .u64 s, t;\n\t"
        "mov.b64 {v0, v1}, %6;\n\t"
        "shf.r.clamp.b32 x1, v0, v1, %9;\n\t"
        "and.b32 x0, v0, %10;\n\t"
        "add.u32 xs, x0, x1;\n\t"
        "mov.b64 {a0, c0}, %7;\n\t"
        "mov.b64 {a1, c1}, %8;\n\t"
        "add.u64 s, %7, %8;\n\t"
        "mov.b64 {as, cs}, s;\n\t"
        "mul.wide.u32 t, x1, a1;\n\tadd.u64 %0, %0, t;\n\t"
        "mad.wide.u32 %1, x0, a0, %1;\n\t"
        "mul.wide.u32 t, xs, as;\n\tadd.u64 %2, %2, t;\n\t"
        "mul.wide.u32 t, x1, c1;\n\tadd.u64 %3, %3, t;\n\t"
        "mad.wide.u32 %4, x0, c0, %4;\n\t"
        "mul.wide.u32 t, xs, cs;\n\tadd.u64 %5, %5, t;\n\t}"
        : "+l"(kh[0]), "+l"(kl[0]), "+l"(km[0]), "+l"(kh[1]), "+l"(kl[1]), "+l"(km[1])
        : "l"(xv), "l"(w0), "l"(w1), "n"(LB), "n"((1u << LB) - 1));
}

// Read-only 16 bytes that shall not displace the forward twiddles in the small
// L1 left beside the shared memory.
__device__ __forceinline__ ulonglong2 ld_stream(const ulonglong2 *p) {
    ulonglong2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    return v;
}

// The inverse transform's phase of NST stages on bits SB .. of field [F, F + 3)
// (ntr::inv_phase with its twiddles fetched beforehand): twiddle pairs in the
// order they are used.
template <int LOGN, int F, int SB, int NST>
__device__ __forceinline__ void inv_twiddles(ulonglong2 (&w)[7], u32 l, const u64 *itw) {
    const ulonglong2 *tp = reinterpret_cast<const ulonglong2 *>(itw);
    int n = 0;
#pragma unroll
    for (int st = 0; st < NST; st++) {
        const int lb = SB + st - F;
#pragma unroll
        for (int j = 0; j < (4 >> lb); j++)
            w[n++] = ld_stream(tp + (1u << (LOGN - 1 - SB - st)) + ((u32)j << (LOGN - 3 - F)) + (l >> F));
    }
}
template <int NST, bool LAZY>
__device__ __forceinline__ void inv_run(u64 (&x)[8], const ulonglong2 (&w)[7], u64 Q) {
    int n = 0;
#pragma unroll
    for (int lb = 3 - NST; lb < 3; lb++) {
#pragma unroll
        for (int j = 0; j < (4 >> lb); j++, n++)
#pragma unroll
            for (int i = 0; i < (1 << lb); i++) {
                u64 &U = x[(j << (lb + 1)) + i], &V = x[(j << (lb + 1)) + i + (1 << lb)];
                if constexpr (LAZY) bfly_gs_lazy_qlow1(U, V, w[n].x, w[n].y, (u32)(Q >> 32), Q << 6);
                else bfly_gs_qlow1(U, V, w[n].x, w[n].y, (u32)(Q >> 32), 4 * Q);
            }
    }
}

// Transform warps: for every unit the rounds of its batches.  Round r of a
// batch: warpgroup w takes TMEM column group 2 r + w (N = 1024: two digit
// polynomials, N = 2048: one) and stores into stage r.
template <int LOGN, int TC, bool LAZY>
__device__ __forceinline__ void transform_warps(Shared &sh, unsigned char *sm, u32 *status) {
    using C = Cfg<LOGN, TC>;
    constexpr int N = C::N, NL = C::NL;
    const u32 tid = threadIdx.x, lane = tid % 32, quad = (tid / 32) & 3, w = tid / 128;
    const u32 p = quad * 16 + (lane & 15), half = lane >> 4;
    const u32 taddr = sh.tmem + ((quad * 32) << 16) + w * 8;
    u64 cE = 0, cO = 0, Q = 0;
    u32 t0 = 0, tcm = 0, fs = 0, fsh = 0;
    const ulonglong2 *tw = nullptr;
    const ulonglong2 *tws = (const ulonglong2 *)(sm + C::TW_OFF);
    u32 pf = 0, px = 3;      // parities; px: one bit per stage (first waits pass)
    for (u32 u = 0;; u++) {
        if (!wait(&sh.tfull, pf, &sh.dead, status)) return;     // the unit's first batch (or the end)
        const u32 ncu = *(volatile u32 *)&sh.unit[u & 3].ncomb;
        if (ncu == 0) break;
        if (*(volatile u32 *)&sh.unit[u & 3].newkey) {
            const KeyDev *K = sh.key;
            const unsigned char *tab = (const unsigned char *)K->tc;
            cE = __ldg((const u64 *)(tab + C::A_BYTES) + p);
            cO = __ldg((const u64 *)(tab + C::A_BYTES) + 64 + p);
            t0 = K->tc_t0;
            tcm = K->tc_m;
            fs = K->tc_fs;
            fsh = K->tc_fsh;
            Q = K->mq.Q;
            tw = (const ulonglong2 *)(tab + C::TW_TAB);
        }
        const u32 cq = (u32)(Q >> 32);
        const u64 fourQ = 4 * Q;
        for (u32 c0 = 0; c0 < ncu; c0 += C::CB) {
            const u32 nc = ncu - c0 < (u32)C::CB ? ncu - c0 : (u32)C::CB;
            const u32 rounds = (nc + C::RC - 1) / C::RC;
            if (c0 && !wait(&sh.tfull, pf, &sh.dead, status)) return;
            pf ^= 1;
            fence_after();
#pragma unroll 1
            for (u32 r = 0; r < rounds; r++) {
                u64 y0[8], y1[8];
                {
                    // two columns of every limb at a time, the next ones in flight
                    // while these are recombined
                    const u32 ta = taddr + r * 16;
                    u32 f[2][2 * NL][2];
#pragma unroll
                    for (int l = 0; l < 2 * NL; l++) tmem_ld2(ta + l * 32, f[0][l]);
#pragma unroll
                    for (int jj = 0; jj < 4; jj++) {
                        tmem_wait();
                        if (jj < 3) {
#pragma unroll
                            for (int l = 0; l < 2 * NL; l++) tmem_ld2(ta + l * 32 + 2 * jj + 2, f[(jj + 1) & 1][l]);
                        }
#pragma unroll
                        for (int j = 0; j < 2; j++) {
                            u32 a[NL], o[NL];
#pragma unroll
                            for (int l = 0; l < NL; l++) {
                                a[l] = f[jj & 1][l][j];
                                o[l] = f[jj & 1][NL + l][j];
                            }
                            const u64 E = recombine<TC, LAZY>(a, cE, t0, tcm, cq);
                            const u64 O = recombine<TC, LAZY>(o, cO, t0, tcm, cq);
                            y0[jj * 2 + j] = add64c(E, O);      // class 2p
                            y1[jj * 2 + j] = sub64c(E, O);      // class 2p + 1
                        }
                    }
                }
                if (r + 1 == rounds) {
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh.tempty);
                }
                auto fin = [&](u64 v) {
                    if constexpr (LAZY) return v;
                    else {
                        // v - (quotient estimate) Q in [0, 2Q)
                        const u32 qe = __umulhi((u32)(v >> 32), fs) >> fsh;
                        return sub64c(((u64)((u32)(v >> 32) - qe * cq) << 32) | (u32)v, qe);
                    }
                };
                u64 *xs = (u64 *)(sm + C::X_OFF + r * C::XS);
                if constexpr (LOGN == 10) {
                    class_stages<8, LAZY>(y0, [&](int i) { return tws[i * 128 + p]; }, cq, fourQ);
                    class_stages<8, LAZY>(y1, [&](int i) { return tws[i * 128 + 64 + p]; }, cq, fourQ);
                    if (!wait(&sh.xempty[r], (px >> r) & 1, &sh.dead, status)) return;
                    u64 *xo = xs + (size_t)(2 * w + half) * N + p * 16;
#pragma unroll
                    for (u32 i = 0; i < 4; i++) {
                        *reinterpret_cast<ulonglong2 *>(xo + 2 * (i ^ (p & 7))) =
                            make_ulonglong2(fin(y0[2 * i]), fin(y0[2 * i + 1]));
                        *reinterpret_cast<ulonglong2 *>(xo + 2 * ((4 + i) ^ (p & 7))) =
                            make_ulonglong2(fin(y1[2 * i]), fin(y1[2 * i + 1]));
                    }
                } else {
                    // lanes L (j < 8) and L ^ 16 (j >= 8): the first takes class
                    // 2p, the second class 2p + 1
                    u64 x[16];
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const u64 keep = half ? y1[j] : y0[j], send = half ? y0[j] : y1[j];
                        const u64 recv = __shfl_xor_sync(0xffffffffu, send, 16);
                        x[j] = half ? recv : keep;
                        x[8 + j] = half ? keep : recv;
                    }
                    class_stages<16, LAZY>(x, [&](int i) {
                        return i < C::NTS ? tws[i * 128 + half * 64 + p] : __ldg(tw + i * 128 + half * 64 + p);
                    }, cq, fourQ);
                    if (!wait(&sh.xempty[r], (px >> r) & 1, &sh.dead, status)) return;
                    u64 *xo = xs + (size_t)w * N + (2 * p + half) * 16;
#pragma unroll
                    for (u32 i = 0; i < 8; i++)
                        *reinterpret_cast<ulonglong2 *>(xo + 2 * (i ^ (p & 7))) =
                            make_ulonglong2(fin(x[2 * i]), fin(x[2 * i + 1]));
                }
                px ^= 1u << r;
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.xfull[r]);
            }
        }
    }
}

// Product warps: the jobs of the block, two slots in turn.
template <int LOGN, int TC, bool LAZY>
struct Product {
    using C = Cfg<LOGN, TC>;
    static constexpr int N = C::N;
    static constexpr u32 LB = br_qlow1_limb(LAZY ? BR_V_LAZY : 0);
    // N = 1024 (lazy keys, Q < 2^54, values below 26.3 Q): the 64-bit sums of
    // limb products hold a whole row, 24 ((26.3 Q >> 28) + 2^28) (2^26 + 2^28) <
    // 2^64, so they stay in registers and are reduced once per row; N = 2048
    // folds them per round into 128-bit row sums in TMEM.
    static constexpr bool KEEP = C::PH == 2;
    static_assert(!KEEP || LAZY, "limb sums of a whole row");
    Shared &sh;
    unsigned char *sm;
    u32 *status;
    u64 *ws;
    const DevJob *jobs;
    const u64 *ct_in;
    const u32 *luts;
    u32 steps_limit, crank, csize;
    const KeyDev *K;
    u32 lB;
    u32 mtid, lane, pcl, ucount, px;
    bool newkey;

    // Hands out the next unit (word u & 3, barrier u & 1: unit u - 2 is done
    // when this is called).  Every product thread has passed a barrier since
    // the accumulators the unit reads were written.
    __device__ __forceinline__ void post(u32 slot, u32 row, u32 part, bool leave = false) {
        if (mtid == 0) {
            Unit &un = sh.unit[ucount & 3];
            un.slot = slot;
            un.row = row;
            un.part = part;
            un.ncomb = leave ? 0 : lB * C::PAIRS;
            un.newkey = newkey;
            mbar_arrive(&sh.post[ucount & 1]);
        }
        ucount++;
        newkey = false;
    }

    // Makes `key` the one the block works with: its weights to shared memory
    // (no product of the previous key is outstanding).
    __device__ __forceinline__ void load_key(const KeyDev *key) {
        K = key;
        lB = key->l_B;
        newkey = true;
        const uint4 *src = (const uint4 *)key->tc;
        uint4 *dst = (uint4 *)sm;
        for (u32 i = mtid; i < C::A_BYTES / 16; i += kM) dst[i] = __ldg(src + i);
        for (u32 i = mtid; i < C::NTS * 128; i += kM)
            ((uint4 *)(sm + C::TW_OFF))[i] = __ldg((const uint4 *)((const unsigned char *)key->tc + C::TW_TAB) + i);
        if (mtid == 0) sh.key = key;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }

    // Job `idx` into slot s: table check and ACC initialisation (this block's
    // rows).  The slot stays off when the table is not negacyclic.
    __device__ __forceinline__ void start(int si, u32 idx) {
        Slot &s = sh.slot[si];
        const DevJob &J = jobs[idx];
        const u32 m = J.m, t = J.t, n = J.n;
        const size_t vec = (size_t)m * 2 * N;
        u64 *cur = ws + J.acc_off;
        const u64 *ct = ct_in + J.in_off;
        const u32 *gpre = J.gS ? status + J.gpre : nullptr;
        const u32 *lut = luts + J.lut_off;
        if (mtid == 0) sh.bad = 0;
        bar_m();
        for (u32 k = mtid; k < t / 2; k += kM) {
            const u32 a = lut[k], b = lut[k + t / 2];
            if (a >= t || b >= t || b != (t - a) % t) *(volatile int *)&sh.bad = 1;
        }
        bar_m();
        const bool ok = *(volatile int *)&sh.bad == 0;
        if (!ok) {
            if (mtid == 0 && crank == 0) set_status(status, BM_ENONNEGACYCLIC);
            for (size_t i = mtid; i < 2 * vec; i += kM)
                if ((i / (2 * N)) % m % csize == crank) cur[i] = 0;
        } else {
            acc_init(cur, lut, ct[n] % (2ull * N * m), m, t, N, J.key->mq.Q, J.gS, J.gSinv, gpre, crank, csize, mtid,
                     kM);
        }
        if (mtid == 0) {
            const u32 steps = steps_limit < n ? steps_limit : n;
            s.cur = cur;
            s.nxt = cur + vec;
            s.ct = ct;
            s.gS = J.gS;
            s.gpre = gpre;
            s.m = m;
            s.mr = crank < m ? (m - 1 - crank) / csize + 1 : 0;
            s.k = 0;
            s.steps = steps;
            s.on = ok && steps;
            sh.taken++;
        }
        bar_m();
    }

    // Row sums of pair h of positions: (column, position) low and high words.
    __device__ __forceinline__ u32 sum_col(u32 h) const {
        return sh.tmem + (((mtid / 32) & 3) << 21) + C::SUM_COL + (mtid / 128) * (C::PH * 16) + h * 16;
    }

    // Limb sums of a pair of positions into its row sums r (two positions x two
    // columns x 128 bits).
    __device__ __forceinline__ static void fold(u32 (&r)[16], const u64 (&kh)[2][2], const u64 (&kl)[2][2],
                                                const u64 (&km)[2][2]) {
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int c = 0; c < 2; c++) {
                u32 *q = r + 8 * i + 4 * c;
                u64 l = q[0] | (u64)q[1] << 32, hh = q[2] | (u64)q[3] << 32;
                add128(l, hh, kl[i][c]);
                add128_shl(l, hh, km[i][c] - kh[i][c] - kl[i][c], LB);
                add128_shl(l, hh, kh[i][c], 2 * LB);
                q[0] = (u32)l;
                q[1] = (u32)(l >> 32);
                q[2] = (u32)hh;
                q[3] = (u32)(hh >> 32);
            }
    }

    // Multiply-accumulate of one unit (row part `part`) of a slot.  The row
    // sums sit in TMEM: those of a pair of positions are requested before its
    // products and stored after them.
    __device__ __forceinline__ void products(const Slot &s, u32 part) {
        const u32 ncu = lB * C::PAIRS;
        const u64 *kp = K->bsk + ((size_t)s.k * 4 * lB + part * ncu) * 2 * N + 4 * (size_t)mtid;
        // key words of the eight (h, combo) of a round, KD loads ahead
        constexpr int KD = 2;
        static_assert(C::PH * C::RC == 8, "eight loads per round");
        Key2 kv[KD];
        auto key_at = [&](const u64 *base, int i) {
            return key_load4(base + (size_t)(i % C::RC) * 2 * N + (i / C::RC) * (4 * kM));
        };
#pragma unroll
        for (int i = 0; i < KD; i++) kv[i] = key_at(kp, i);
        constexpr int KS = KEEP ? C::PH : 1;
        u64 kh[KS][2][2], kl[KS][2][2], km[KS][2][2];
        auto clear = [&](int a) {
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int c = 0; c < 2; c++) kh[a][i][c] = kl[a][i][c] = km[a][i][c] = 0;
        };
#pragma unroll
        for (int a = 0; a < KS; a++) clear(a);
        for (u32 c0 = 0; c0 < ncu; c0 += C::CB) {
            const u32 nc = ncu - c0 < (u32)C::CB ? ncu - c0 : (u32)C::CB;
            const u32 rounds = (nc + C::RC - 1) / C::RC;
#pragma unroll 1
            for (u32 r = 0; r < rounds; r++) {
                const u64 *xs = (const u64 *)(sm + C::X_OFF + r * C::XS);
                const u64 *kr = kp + (size_t)(c0 + r * C::RC) * 2 * N;
                const bool last = c0 + (r + 1) * C::RC >= ncu;
                const bool first = part == 0 && c0 == 0 && r == 0;
                // (given up: on to the step's end)
                (void)wait(&sh.xfull[r], (px >> r) & 1, &sh.dead, status);
                px ^= 1u << r;
#pragma unroll
                for (int h = 0; h < C::PH; h++) {
                    const u32 un = h * kM + mtid;                       // pair of positions
                    const u32 blk = un >> 3;                            // block of 16 positions
                    const u32 sw = blk * 16 + 2 * ((un & 7) ^ ((LOGN == 10 ? blk : blk >> 1) & 7));
                    constexpr bool sums = !KEEP;
                    const int a = KEEP ? h : 0;
                    u32 w[16];
                    if constexpr (sums) tmem_ld16(sum_col(h), w);
#pragma unroll
                    for (int q = 0; q < C::RC; q++) {
                        const ulonglong2 xv = *reinterpret_cast<const ulonglong2 *>(xs + (size_t)q * N + sw);
                        const int i = h * C::RC + q;
                        const Key2 kw = kv[i % KD];
                        if (i + KD < 8) kv[i % KD] = key_at(kr, i + KD);
                        else if (!last) kv[i % KD] = key_at(kr + (size_t)C::RC * 2 * N, i + KD - 8);
                        kara2<LB>(xv.x, kw.a0, kw.a1, kh[a][0], kl[a][0], km[a][0]);
                        kara2<LB>(xv.y, kw.b0, kw.b1, kh[a][1], kl[a][1], km[a][1]);
                    }
                    if constexpr (sums) {
                        tmem_wait();
                        tmem_wait_st();      // the previous pair's store, long done
                        if (first) {
#pragma unroll
                            for (int i = 0; i < 16; i++) w[i] = 0;
                        }
                        fold(w, kh[a], kl[a], km[a]);
                        clear(a);
                        tmem_st16(sum_col(h), w);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.xempty[r]);
            }
        }
        if constexpr (KEEP) {
            // kl + (km - kh - kl) 2^LB + kh 2^(2 LB) mod Q in [0, 11Q) to the
            // inverse transforms' region (which take values below 16Q, Q < 2^54)
            u64 *reg = (u64 *)(sm + C::I_OFF);
            const u64 Q = K->mq.Q, b1 = K->tc_b1, b1s = K->tc_b1s, b2 = K->tc_b2, b2s = K->tc_b2s;
            const u32 c = (u32)(Q >> 32), one = (u32)K->mq.one_sh;
#pragma unroll
            for (int h = 0; h < C::PH; h++)
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int cc = 0; cc < 2; cc++) {
                        const u64 hi = kh[h % KS][i][cc], lo = kl[h % KS][i][cc];
                        const u64 mid = sub64c(sub64c(km[h % KS][i][cc], hi), lo);
                        const u64 v = add64c(add64c(shoup3_qlow1_lazy(mid, b1, b1s, c), shoup3_qlow1_lazy(hi, b2, b2s, c)),
                                             reduce_est_qlow1(lo, one, c));
                        reg[(size_t)cc * N + ntr::swz<3>(2 * (h * kM + mtid) + i)] = v;
                    }
        }
    }

    // Reduced sums of pair h of positions to the inverse transforms' region:
    // both columns (N = 1024) or column cp.
    __device__ __forceinline__ void put_sums(const u32 (&w)[16], u32 h, u32 cp) {
        constexpr int PP = 2048 / N;
        u64 *reg = (u64 *)(sm + C::I_OFF);
        const u32 q = 2 * (h * kM + mtid);
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int c = 0; c < PP; c++) {
                const u32 *v = w + 8 * i + 4 * c;
                u64 l = v[0] | (u64)v[1] << 32, hh = v[2] | (u64)v[3] << 32;
                if (PP == 1 && cp) {
                    l = v[4] | (u64)v[5] << 32;
                    hh = v[6] | (u64)v[7] << 32;
                }
                reg[(size_t)c * N + ntr::swz<3>(q + i)] = reduce128q<true>(l, hh, K->mq);
            }
    }

    // Row sums -> inverse transforms -> accumulator update of row `row`; false
    // when the block has given up.
    __device__ __forceinline__ bool finish_row(const Slot &s, u32 row) {
        constexpr int RB = 3, T = N / 8, PP = 2048 / N;         // polynomials at a time
        constexpr int NPH = (LOGN + RB - 1) / RB;
        const ModQ mq = K->mq;
        const u64 Q = mq.Q, twoQ = 2 * Q;
        const u64 *itw = (const u64 *)((const unsigned char *)K->tc + C::ITW_TAB);
        const u32 r = crank + csize * row;
        u64 *reg = (u64 *)(sm + C::I_OFF);
        const u32 ip = mtid / T, il = mtid % T;
        if constexpr (!KEEP) tmem_wait_st();
#pragma unroll 1
        for (u32 cp = 0; cp < 2; cp += PP) {
            if constexpr (!KEEP) {
#pragma unroll 1
                for (u32 h = 0; h < (u32)C::PH; h++) {
                    u32 w[16];
                    tmem_ld16(sum_col(h), w);
                    tmem_wait();
                    put_sums(w, h, cp);
                }
            }
            ulonglong2 t0[7];
            inv_twiddles<LOGN, 0, 0, 3>(t0, il, itw);
            bar_m();
            {
            u64 x[8];
            u64 *rg = reg + (size_t)ip * N;
            auto between = [&]() {
                if constexpr (LAZY) {
#pragma unroll
                    for (int i = 0; i < 8; i++) x[i] = reduce_est_qlow1(x[i], (u32)mq.one_sh, (u32)(Q >> 32));
                }
            };
            auto gsync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(6 + ip), "n"(T) : "memory"); };
            // every phase's twiddles and the accumulator words are requested
            // before the barrier that precedes their use
            static_assert(NPH == 4, "four phases");
            const size_t base = (size_t)(r * 2 + cp + ip) * N;
            ulonglong2 w0[7], w1[7];
            u64 o[8];
            inv_twiddles<LOGN, 3, 3, 3>(w1, il, itw);
            ntr::load_field<RB, 0>(x, rg, il);
            inv_run<3, LAZY>(x, t0, Q);
            between();
            ntr::store_field<RB, 0>(x, rg, il);
            gsync();
            inv_twiddles<LOGN, 6, 6, 3>(w0, il, itw);
            ntr::load_field<RB, 3>(x, rg, il);
            inv_run<3, LAZY>(x, w1, Q);
            between();
            ntr::store_field<RB, 3>(x, rg, il);
            gsync();
            inv_twiddles<LOGN, LOGN - RB, 9, LOGN - 9>(w1, il, itw);
            ntr::load_field<RB, 6>(x, rg, il);
            inv_run<3, LAZY>(x, w0, Q);
            between();
            ntr::store_field<RB, 6>(x, rg, il);
#pragma unroll
            for (int i = 0; i < 8; i++) o[i] = __ldcg(s.cur + base + il + T * i);
            gsync();
            ntr::load_field<RB, LOGN - RB>(x, rg, il);
            inv_run<LOGN - 9, LAZY>(x, w1, Q);
            between();
#pragma unroll
            for (int i = 0; i < 8; i++) {
                s.nxt[base + il + T * i] = add_mod(o[i], csub63(csub63(x[i], twoQ), Q), Q);
            }
            }
            bar_m();     // the region is read: the next sums may be written
        }
        return true;
    }
};

// One block: in a cluster its share of the rows of job blockIdx.x / csize,
// else jobs blockIdx.x and blockIdx.x + gridDim.x side by side, then further
// ones from the counter (null: none).
template <int LOGN, int TC, bool LAZY>
__device__ __forceinline__ void product_warps(Shared &sh, unsigned char *sm, const DevJob *__restrict__ jobs, u32 count,
                                              u32 steps, const u64 *__restrict__ ct_in, const u32 *__restrict__ luts,
                                              u64 *ws, u32 *status, u32 *counter) {
    using P = Product<LOGN, TC, LAZY>;
    using C = Cfg<LOGN, TC>;
    const u32 csize = cluster_size();
    P pr{sh, sm, status, ws, jobs, ct_in, luts, steps, cluster_rank(), csize, nullptr, 0,
         threadIdx.x - kT, threadIdx.x % 32, 0, 0, 0, false};
    constexpr u32 units = 4 / C::PAIRS;
    Slot *const sl = sh.slot;
    if (pr.mtid < 2) sl[pr.mtid].on = sh.taken = 0;
    bar_m();
    // a job waiting for its slot (its key is not the one loaded), or none
    u32 wait0 = blockIdx.x / csize, wait1 = csize > 1 ? count : blockIdx.x + gridDim.x;
    bool dead = false;     // the block has given up
    // Fills an idle slot: the waiting job, or the next of the counter.
    auto fill = [&](int s) {
        u32 &w = s ? wait1 : wait0;
        while (!sl[s].on) {
            if (w == 0xffffffffu) {
                if (!counter) break;
                // Side by side two jobs gain little over one (throughput 1.08 to
                // 1), so a block whose other slot is at work takes no more than
                // its even share of the jobs.
                if (sl[s ^ 1].on && sh.taken * gridDim.x + blockIdx.x >= count) break;
                bar_m();
                if (pr.mtid == 0) *(volatile u32 *)&sh.next = atomicAdd(counter, 1u) + 2 * gridDim.x;
                bar_m();
                w = *(volatile u32 *)&sh.next;
            }
            if (w >= count) {
                w = count;
                break;
            }
            const KeyDev *key = jobs[w].key;
            if (key != pr.K) {
                if (sl[s ^ 1].on) break;      // the other slot's job keeps its key until it ends
                bar_m();
                pr.load_key(key);
            }
            pr.start(s, w);
            if (csize > 1) {
                (void)cluster_bar_m(sh, csize, pr.pcl, status);
                dead = bar_or(sh);
            }
            w = csize > 1 ? count : 0xffffffffu;
        }
    };
    fill(0);
    fill(1);
    u32 cs = sl[0].on ? 0 : 1;
    if (dead) {
    } else if (sl[cs].on && sl[cs].mr == 0) {
        // a cluster block without rows: only the barriers
        for (u32 k = 0; k < sl[cs].steps && cluster_bar_m(sh, csize, pr.pcl, status); k++) {}
    } else if (sl[cs].on) {
        u32 row = 0, h = 0;
        pr.post(cs, 0, 0);
        for (;;) {
            // the unit after this one
            u32 ns = cs, nrow = row, nh = h + 1;
            bool same = true;      // of this slot's step
            if (nh == units) {
                nh = 0;
                if (++nrow == sl[cs].mr) {
                    nrow = 0;
                    same = false;
                    if (sl[cs ^ 1].on) ns = cs ^ 1;
                }
            }
            const bool ahead = same || ns != cs;
            if (ahead) pr.post(ns, nrow, nh);
            pr.products(sl[cs], h);
            if (h + 1 == units) {
                if (!pr.finish_row(sl[cs], row)) break;
                if (!same) {
                    if (csize > 1) (void)cluster_bar_m(sh, csize, pr.pcl, status);
                    if (pr.mtid == 0) {
                        Slot &s = sl[cs];
                        u64 *tmp = s.cur;
                        s.cur = s.nxt;
                        s.nxt = tmp;
                        if (++s.k == s.steps) s.on = 0;
                    }
                    if (bar_or(sh)) break;
                    if (!sl[cs].on) {
                        // (a job that has waited for its key comes before new
                        // ones: they are in order of cost)
                        fill(cs ^ 1);
                        fill(cs);
                    }
                    if (!ahead) {
                        if (!sl[ns].on) ns = cs ^ 1;
                        if (!sl[ns].on) break;
                        pr.post(ns, nrow, nh);
                    }
                }
            }
            cs = ns;
            row = nrow;
            h = nh;
        }
    }
    pr.post(0, 0, 0, true);
}

}  // namespace brt
