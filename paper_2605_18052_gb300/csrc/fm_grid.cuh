// Persistent kernels that keep a whole optimiser loop on the device: a cooperative launch whose
// blocks meet at a grid-wide barrier between the phases of an iteration. A barrier costs 1.2 us on
// 125 to 152 blocks (1.4 us on 304), a dependent kernel launch 3 us and more (launch, prologue, the
// tail of the kernel before).
#pragma once

#include <cuda_runtime.h>

#include <stdint.h>

namespace fm {

constexpr unsigned ERR_GRID = 128u;                    // a grid barrier ran into its limit
constexpr long long GRID_WAIT_CYCLES = 4000000000LL;   // about two seconds

__device__ __forceinline__ void red_release_add(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// state[0] counts the arrivals of all blocks, state[1] is its value when a launch starts: block 0
// writes it after its last barrier, when every block has read the old one, so a launch needs no
// reset. The counts may wrap. One state serves the launches of one stream; after a timeout the host
// clears it. (One counter: a flag per block, polled by a warp with acquire loads, took 2.1 us on
// 125 blocks and 4.4 us on 304.)
constexpr int GRID_STATE_WORDS = 2;

struct GridBarrier {
    unsigned *state;
    unsigned *err;
    unsigned target;
    __device__ GridBarrier(unsigned *st, unsigned *e)
        : state(st), err(e), target(*reinterpret_cast<volatile unsigned *>(st + 1)) {}

    // Warp 0 only: publish the block's arrival (what its lanes wrote, and what the block wrote before
    // a __syncthreads, is visible to every block behind the barrier).
    __device__ __forceinline__ void arrive() {
        target += gridDim.x;
        __syncwarp();
        if ((threadIdx.x & 31) == 0) red_release_add(state, 1u);
    }
    // Warp 0 only: wait for every block; false after the limit (then the whole grid gives up: a
    // block that leaves arrives nowhere, so the others run into their limit as well). All lanes poll the
    // one word, so the warp stays converged: with one lane polling, the block that came last ran the
    // serial FP64 code behind the barrier with its lanes apart, three to four times as long, and so came last
    // again (conjugate gradients on 1,000 cameras 12.4 -> 9.7 us an iteration).
    __device__ __forceinline__ bool wait() {
        bool ok = true;
        const long long t0 = clock64();
        while ((int)(ld_acquire(state) - target) < 0) {
            if (clock64() - t0 > GRID_WAIT_CYCLES) {
                ok = false;
                if ((threadIdx.x & 31) == 0) atomicOr(err, ERR_GRID);
                break;
            }
        }
        return __all_sync(0xffffffffu, ok);
    }
    // whole block: everything written before is visible to every block after
    __device__ __forceinline__ bool sync() {
        __syncthreads();
        bool ok = true;
        if (threadIdx.x < 32) {
            arrive();
            ok = wait();
        }
        return __syncthreads_and(ok);
    }
    // thread 0 of block 0, after the last barrier
    __device__ __forceinline__ void finish() {
        if (blockIdx.x == 0 && threadIdx.x == 0) state[1] = target;
    }
};

// cooperative launch (all blocks resident at once, or an error)
template <typename... KArgs, typename... Args>
static cudaError_t launch_coop(void (*kernel)(KArgs...), int grid, int block, int smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// most blocks of a cooperative launch on the current device
template <typename K>
static cudaError_t coop_blocks(K kernel, int block, int *out, int smem = 0) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, block, smem);
    *out = sms * per;
    if (e == cudaSuccess && *out < 1) e = cudaErrorLaunchOutOfResources;
    return e;
}

}  // namespace fm
