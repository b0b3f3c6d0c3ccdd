// Test helper, not part of the library: one thread counts `rounds` times n arrivals in on one counter, as the slices of a
// tile do launch after launch, and records which of them were told to be the last and what the counter was after each.
#include "../../paper_2601_07891_b200/csrc/ptx.cuh"

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
