// muca_batch.cu - the batched persistent kernel: one launch advances many instances of
// uneven L and walker count (work list and counter in library memory).
#include "muca_device.cuh"

namespace muca {
namespace {

// ---------------------------------------------------------------------------------
// Batched persistent kernel: one launch advances many instances (uneven L, walker
// counts, tables and histograms).  The work list holds (instance, first walker, walker
// count) items; each block takes the next item from a global counter, runs it with the
// body of the sweep kernel for that instance's L, and takes another until the list is
// exhausted.  The counter must be zero at launch.
// ---------------------------------------------------------------------------------
__global__ void __launch_bounds__(kBatchThreads, 1) batch_kernel(const SweepArgs *__restrict__ insts,
                                                                  const BatchItem *__restrict__ items, int32_t n_items,
                                                                  uint32_t *counter, const bool record)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int32_t s_item;
    for (;;) {
        if (threadIdx.x == 0)
            s_item = (int32_t)atomicAdd(counter, 1u);
        __syncthreads();
        const int32_t k = s_item;
        __syncthreads();
        if (k >= n_items)
            break;
        const BatchItem it = items[k];
        const SweepArgs a = insts[it.inst];
        switch (a.L) {
        case 8: batch_item<8>(a, it, smem, record); break;
        case 16: batch_item<16>(a, it, smem, record); break;
        case 24: batch_item<24>(a, it, smem, record); break;
        case 32: batch_item<32>(a, it, smem, record); break;
        case 48: batch_item<48>(a, it, smem, record); break;
        case 64: batch_item<64, false, batch_table_stride(64)>(a, it, smem, record); break;
        default: break;
        }
    }
}

}  // namespace

cudaError_t configure_batch(size_t smem)
{
    return cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

int batch_resident_blocks(size_t smem)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_kernel, kBatchThreads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_batch(const SweepArgs *insts, const BatchItem *items, int32_t n_items, uint32_t *counter,
                         int grid, size_t smem, bool record, cudaStream_t s)
{
    if (n_items <= 0)
        return cudaSuccess;
    batch_kernel<<<grid, kBatchThreads, smem, s>>>(insts, items, n_items, counter, record);
    return cudaGetLastError();
}

}  // namespace muca
