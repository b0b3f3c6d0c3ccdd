// Test helper, not part of the library.
#include "../../paper_2601_07891_b200/csrc/ptx.cuh"

// One thread counts `rounds` times n arrivals in on one counter, as the slices of a tile do launch after launch, and records which
// of them were told to be the last and what the counter was after each.
__global__ void arrivals_kernel(uint32_t *counter, uint32_t n, int rounds, int *last, uint32_t *after)
{
    for (int i = 0; i < rounds * static_cast<int>(n); ++i) {
        last[i] = kvzap::arrive_last(counter, n) ? 1 : 0;
        after[i] = *static_cast<volatile uint32_t *>(counter);
    }
}

// last, after: rounds * n entries each.  Returns the CUDA error code of the launch.
extern "C" int launch_arrivals(void *counter, unsigned n, int rounds, void *last, void *after, void *stream)
{
    arrivals_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<uint32_t *>(counter), n, rounds,
                                                                    static_cast<int *>(last), static_cast<uint32_t *>(after));
    return static_cast<int>(cudaGetLastError());
}

// n CTAs of one warp each (none waits for another): every lane stores a value, the warp counts itself in, and the last one's lanes
// each add up what another lane of every warp has stored.
__global__ void warp_arrivals_kernel(uint32_t *counter, int *parts, int value, int *sums, int *lasts)
{
    const int lane = threadIdx.x, n = gridDim.x;
    __stcg(parts + blockIdx.x * 32 + lane, value + static_cast<int>(blockIdx.x) * 32 + lane);
    if (!kvzap::arrive_last_warp(counter, static_cast<uint32_t>(n))) return;
    int sum = 0;
    for (int i = 0; i < n; ++i) sum += __ldcg(parts + i * 32 + (lane * 5 + 7) % 32);
    sums[lane] = sum;
    atomicAdd(lasts, 1);
}

// parts: n * 32 entries, sums: 32, lasts: 1.
extern "C" int launch_warp_arrivals(void *counter, unsigned n, void *parts, int value, void *sums, void *lasts, void *stream)
{
    warp_arrivals_kernel<<<n, 32, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<uint32_t *>(counter), static_cast<int *>(parts), value,
                                                                          static_cast<int *>(sums), static_cast<int *>(lasts));
    return static_cast<int>(cudaGetLastError());
}
