// One warp waits on an mbarrier (csrc/async.cuh) three times; prints, per time, how many lanes were told that
// the phase completed and whether the wait was given up. Driven by test_gpu_waits.py.
#include <cstdio>

#include "async.cuh"

using namespace cbct;

enum Mode { COMPLETES, SPLIT, RUNS_OUT };

// COMPLETES: the second warp arrives. SPLIT: it arrives after the first 16 lanes, which are told to give
// up, have left the loop. RUNS_OUT: nothing arrives, the wait ends at its limit.
__global__ void wait_once(Mode mode, int *verdict, int *given_up)
{
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int flag[2];
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1u);
        flag[0] = 0;
        flag[1] = mode == SPLIT;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        verdict[threadIdx.x] = mbar_wait(&bar, 0u, threadIdx.x < 16 ? &flag[1] : &flag[0]);
        if (threadIdx.x == 0) *given_up = flag[0] || flag[1];
    } else if (threadIdx.x == 32 && mode != RUNS_OUT) {
        const long long t0 = clock64();
        while (clock64() - t0 < 20000000ll) { // about 10 ms, some tries of the waiting lanes
        }
        mbar_arrive(&bar);
    }
}

int main()
{
    int *d = nullptr, h[33];
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return 2;
    for (int mode = COMPLETES; mode <= RUNS_OUT; ++mode) {
        wait_once<<<1, 64>>>((Mode)mode, d, d + 32);
        const cudaError_t e = cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) {
            std::printf("%s\n", cudaGetErrorString(e));
            return 1;
        }
        int n = 0;
        for (int i = 0; i < 32; ++i) n += h[i] != 0;
        std::printf("%d %d\n", n, h[32]);
    }
    return 0;
}
