// lbve_gridbar.cuh -- barrier over the blocks of one cooperative launch, with a bounded wait,
// and the host side of such launches.  For kernels that take several time steps of a grid
// small enough to be resident on the device as a whole: between steps the blocks meet here
// instead of at a kernel boundary.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

namespace lbve {

// Limits of a barrier's wait.  At the launch's first barrier some blocks may not have started
// yet, held up by another stream's kernel on their SMs; from then on all of them are resident
// and a step takes microseconds.
constexpr unsigned long long GB_FIRST_NS = 20000000000ull;  // 20 s
constexpr unsigned long long GB_WAIT_NS = 1000000000ull;    // 1 s
constexpr unsigned GB_LEFT = 1u << 31;  // set in the word by a block that gave up

// Steps that the next launch of a call takes when `steps` are left on a grid of `blocks`
// blocks.  The barrier's word counts steps x blocks in 32 bits and must not wrap (a call of
// 12.6 M steps on 343 blocks would), and a launch should end within tens of milliseconds;
// 4096 steps of a few microseconds make the launch itself a few parts in ten thousand.
constexpr int GB_LAUNCH_STEPS = 4096;
inline int launch_steps(int steps, long long blocks) {
    const long long most = std::min<long long>(GB_LAUNCH_STEPS, (1LL << 30) / std::max(1LL, blocks));
    return (int)std::min<long long>(steps, std::max(1LL, most));
}

// Barrier number k (0, 1, ...) of `blocks` blocks on word[0], which was 0 at the launch's start:
// they count up to (k + 1) blocks, at most 2^30 (launch_steps).  False (in every thread of
// the block) when the wait gave up, after writing 2 to *status, 1 to word[1] and marking
// word[0], or when another block did: the caller returns then, and so do the others, at this
// barrier or the next.  While word[1] stays set the first barrier of a launch returns false
// at once, so that the launches of a long call do not each wait in turn.  The block barriers around the release add and the acquire load make every thread's
// earlier writes visible to every thread's later reads (PTX causality order); fences of their
// own would only add to it.
__device__ __forceinline__ bool grid_barrier(unsigned *word, unsigned k, unsigned blocks, unsigned *status,
                                             unsigned long long first_ns = GB_FIRST_NS,
                                             unsigned long long wait_ns = GB_WAIT_NS) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        const unsigned target = (k + 1u) * blocks;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(word) : "memory");
        const unsigned long long limit = k == 0 ? first_ns : wait_ns;
        unsigned long long t0 = 0;
        const unsigned given_up = k == 0 ? *(volatile const unsigned *)(word + 1) : 0u;
        ok = given_up == 0u;
        for (unsigned n = 0; given_up == 0u; ++n) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
            if (v >= target) {
                ok = v < GB_LEFT;
                break;
            }
            if ((n & 255u) == 255u) {
                unsigned long long t;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t0 == 0)
                    t0 = t;
                else if (t - t0 > limit) {
                    atomicOr(word, GB_LEFT);
                    *(volatile unsigned *)(word + 1) = 1u;
                    if (status) *(volatile unsigned *)status = 2u;
                    ok = 0;
                    break;
                }
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

// Blocks of `kernel` that the current device holds at once (0: no cooperative launches).
template <class K>
inline int resident_blocks(K kernel, int threads, size_t smem) {
    int dev = 0, sms = 0, per = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return sms * per;
}

inline int device_sms() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        cudaGetLastError();
    return sms;
}

// True when the stream is being captured (or its state cannot be asked for): the plain
// launches are recorded then.
inline bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return st != cudaStreamCaptureStatusNone;
}

} // namespace lbve
