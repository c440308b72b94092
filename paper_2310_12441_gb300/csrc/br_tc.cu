// Launches of the tensor-core form of the blind rotation (br_tc.cuh): one job
// per block or per cluster of blocks, and persistent blocks pulling jobs.
#include "br_launch.cuh"
#include "br_tc.cuh"

namespace {

template <int LOGN, int TC, bool LAZY>
__global__ void __launch_bounds__(brt::kThreads, 1)
    k_blind_rotate_tc(const DevJob *__restrict__ jobs, u32 count, u32 steps, const u64 *__restrict__ ct_in,
                      const u32 *__restrict__ luts, u64 *ws, u32 *status, u32 *counter) {
    extern __shared__ __align__(1024) unsigned char smb[];
    __shared__ __align__(16) brt::Shared sh;
    const u32 csize = cluster_size();
    brt::open(sh, csize);
    if (threadIdx.x < brt::kT) {
        brt::regs_transform();
        brt::transform_warps<LOGN, TC, LAZY>(sh, smb, status);
    } else if (threadIdx.x < brt::kT + brt::kM) {
        brt::regs_product();
        brt::product_warps<LOGN, TC, LAZY>(sh, smb, jobs, count, steps, ct_in, luts, ws, status, counter);
    } else {
        brt::regs_other();
        if (threadIdx.x < brt::kT + brt::kM + 32) brt::issuer<brt::Cfg<LOGN, TC>>(sh, smb, status);
        else brt::digit_warps<LOGN, TC>(sh, smb, cluster_rank(), csize, status);
    }
    brt::close(sh, csize);
}

// Grouped launch (max_cluster > 1 lets a small batch take a cluster of blocks
// per job) or persistent class: one block per SM, jobs from the counter.
//
// At N = 2048 the lazy keys (Q < 2^54.4) gain from the tensor cores only while a
// block has two jobs to alternate between, or many rows of one: grouped launches
// of clusters, or of single blocks without a second job for any of them and
// fewer than eight rows, keep the CUDA-core kernel.  (24 steps, Q < 2^54, 9-bit
// digits, CUDA cores against tensor cores: 1 job, m = 4 1.40 / 1.45 ms; 8, m = 8
// 1.43 / 1.51; 76, m = 3 2.67 / 2.76; 130, m = 1 1.39 / 1.44; 152, m = 6, 10-bit
// digits 7.78 / 7.90; but 152, m = 8 10.58 / 10.37; 304, m = 1 2.75 / 2.62; 304,
// m = 3 7.94 / 7.72.)
template <int LOGN, int TC, bool LAZY>
bm_status launch_tc(const DevJob *jobs, uint32_t cnt, u32 mmax, u32 max_cluster, u32 steps, const uint64_t *ct_in,
                    const uint32_t *lut, u64 *ws_acc, u32 *status, u32 *counter, int sms, bool persistent,
                    cudaStream_t st, bool dry) {
    constexpr u32 smem = brt::Cfg<LOGN, TC>::SMEM;
    static std::atomic<uint64_t> attr_done{0};
    auto kern = k_blind_rotate_tc<LOGN, TC, LAZY>;
    bm_status s = ensure_smem(kern, smem, attr_done);
    if (s != BM_OK) return s;
    const u32 S = max_cluster > 1 ? pick_cluster(kern, brt::kThreads, smem, cnt, mmax, max_cluster) : 1;
    if constexpr (LOGN == 11 && LAZY)
        if (!persistent && (dry || S > 1 || (cnt <= (u32)sms && mmax < 8)))
            return bm_launch_br_n2048(BR_V_LAZY | BR_V_QLOW1, 1, jobs, cnt, mmax, max_cluster, steps, ct_in, lut, ws_acc,
                                      status, st, dry);
    if (dry) return BM_OK;
    if (S == 1) {
        BM_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(u32), st));
        kern<<<cnt < (u32)sms ? cnt : (u32)sms, brt::kThreads, smem, st>>>(jobs, cnt, steps, ct_in, lut, ws_acc, status,
                                                                          counter);
    } else {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cnt * S);
        cfg.blockDim = dim3(brt::kThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = S;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        BM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, jobs, cnt, steps, ct_in, lut, ws_acc, status, (u32 *)nullptr));
    }
    BM_CUDA_TRY(cudaGetLastError());
    return BM_OK;
}

}  // namespace

// The (ring degree, limbs, arithmetic) combinations of choose_variant.
#define BM_TC_DISPATCH(FN, ...)                                                                        \
    const bool lazy = (variant & BR_V_LAZY) != 0, tc1 = (variant & BR_V_TC1) != 0;                      \
    if (N == 1024 && lazy && tc1) return FN<10, 1, true>(__VA_ARGS__);                                 \
    if (N == 2048 && lazy) return tc1 ? FN<11, 1, true>(__VA_ARGS__) : FN<11, 2, true>(__VA_ARGS__);    \
    if (N == 2048 && !tc1) return FN<11, 2, false>(__VA_ARGS__);                                        \
    return BM_EINVAL

bm_status bm_launch_br_tc(u32 N, u32 variant, const DevJob *jobs, uint32_t cnt, u32 mmax, u32 max_cluster, u32 steps,
                          const uint64_t *ct_in, const uint32_t *lut, u64 *ws_acc, u32 *status, u32 *counter, int sms,
                          cudaStream_t st, bool dry) {
    const bool persistent = sms != 0;
    if (!persistent) {
        int dev = 0;
        BM_CUDA_TRY(cudaGetDevice(&dev));
        BM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    }
    BM_TC_DISPATCH(launch_tc, jobs, cnt, mmax, max_cluster, steps, ct_in, lut, ws_acc, status, counter, sms, persistent, st,
                   dry);
}
