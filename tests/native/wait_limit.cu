// One block: warp 0 waits for a barrier that has been arrived at, then with a
// short limit for one that nothing arrives at; warp 1 waits for another such
// barrier with the kernels' own limit.  out: [0] the first wait's answer,
// [1] the second's, [2] warp 1's, [3] the status word (returned as its code).
#include "br_tc.cuh"

static __global__ void k_waits(u32 *out) {
    __shared__ u64 bar[3];
    __shared__ u32 dead;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 3; i++) mbar_init(&bar[i], 1);
        dead = 0;
        mbar_arrive(&bar[0]);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const bool a = brt::wait(&bar[0], 0, &dead, out + 3);
        const bool b = brt::wait(&bar[1], 0, &dead, out + 3, 100);
        if (threadIdx.x == 0) out[0] = a, out[1] = b;
    } else {
        const bool c = brt::wait(&bar[2], 0, &dead, out + 3);
        if (threadIdx.x == 32) out[2] = c;
    }
}

extern "C" int wait_limit(int *got) {
    u32 *out = nullptr;
    if (cudaMalloc(&out, 16) != cudaSuccess) return 1;
    cudaMemset(out, 0xff, 12);
    cudaMemset(out + 3, 0, 4);
    k_waits<<<1, 64>>>(out);
    const cudaError_t e = cudaMemcpy(got, out, 16, cudaMemcpyDeviceToHost);
    cudaFree(out);
    got[3] = -got[3];
    return e == cudaSuccess ? 0 : 2;
}
