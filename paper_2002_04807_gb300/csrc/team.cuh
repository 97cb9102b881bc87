// Barrier of a team of CTAs inside a cooperative launch, with a time limit.
#pragma once

namespace feast {

// The nc CTAs of a team meet: each adds one arrival to a counter that only
// grows (team_arrive, after which work that no other CTA waits for may follow),
// then waits for its generation to be complete (team_wait).  False (in every
// thread) once any CTA of the launch has waited longer than `limit` cycles.
__device__ __forceinline__ void team_arrive(unsigned* count, unsigned& target, int nc)
{
    __syncthreads();
    target += (unsigned)nc;
    if (nc > 1 && threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
}

__device__ __forceinline__ bool team_wait(unsigned* count, unsigned target, int nc, int* err, long long limit)
{
    int good = 1;
    if (nc > 1 && threadIdx.x == 0) {
        const long long t0 = clock64();
        for (;;) {
            unsigned cur;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(count) : "memory");
            if ((int)(cur - target) >= 0) break;
            if (*(volatile int*)err) {
                good = 0;
                break;
            }
            if (clock64() - t0 > limit) {
                atomicExch(err, 1);
                good = 0;
                break;
            }
        }
    }
    return __syncthreads_and(good) != 0;
}

__device__ __forceinline__ bool team_sync(unsigned* count, unsigned& target, int nc, int* err, long long limit)
{
    if (nc == 1) {
        __syncthreads();
        return true;
    }
    team_arrive(count, target, nc);
    return team_wait(count, target, nc, err, limit);
}

}  // namespace feast
