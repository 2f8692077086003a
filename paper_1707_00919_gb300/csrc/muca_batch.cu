// muca_batch.cu - the batched persistent kernel: one launch advances many instances of
// uneven L and walker count (work list and counter in library memory).
#include <mutex>

#include "muca_device.cuh"

namespace muca {
namespace {

// Whether the item that SM k would start with has a neighbour (SMs 2i and 2i + 1 share an
// instruction cache) of another L, together too long for the cache.  How long a row's code is
// goes by L; measured, L = 64 beside 48 is too long and 64 beside 32 is not, so that of the
// sizes that are batched the rule names that one pair (to be measured again when the rows'
// code changes).  Of the pair the one with the shorter chain, which is the odd one, then stays
// out; a few blocks of the grid at most do, so that the others are there to take its items.
constexpr uint32_t kMostIdle = 4;
__device__ __forceinline__ bool crowded(const SweepArgs *insts, const BatchItem *items, int32_t n_items, uint32_t k)
{
    if (k % 2 == 0 || k >= (uint32_t)n_items || gridDim.x < 4 * kMostIdle)
        return false;
    const int32_t a = insts[items[k - 1].inst].L, b = insts[items[k].inst].L;
    return a != b && a + b > 96;
}

// ---------------------------------------------------------------------------------
// Batched persistent kernel: one launch advances many instances (uneven L, walker
// counts, tables and histograms).  The work list holds (instance, first walker, walker
// count) items; each block takes an item, runs it with the body of the sweep kernel for that
// instance's L, and takes another until the list is exhausted.  Its first item goes by the
// SM it runs on, so that neighbouring SMs start with items of one L: where two that share
// an instruction cache ran the unrolled rows of L = 64 and of L = 48, an item took 6.5 ms
// instead of 4.5 (twelve instances of L = 16 to 64: iterations of 6.1 to
// 6.9 ms, by chance, now 5.8).  The others
// come from a counter.  work: the counter, the number of blocks that stay out, then a word
// per item, set by whoever takes it first; all zero at launch.
// ---------------------------------------------------------------------------------
__global__ void __launch_bounds__(kBatchThreads, 1) batch_kernel(const SweepArgs *__restrict__ insts,
                                                                  const BatchItem *__restrict__ items, int32_t n_items,
                                                                  uint32_t *work, const bool record)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int32_t s_item;
    bool first = true;
    for (;;) {
        if (threadIdx.x == 0) {
            uint32_t k = 0;
            if (first)
                asm volatile("mov.u32 %0, %%smid;" : "=r"(k));
            if (first && crowded(insts, items, n_items, k) && atomicAdd(&work[1], 1u) < kMostIdle) {
                k = (uint32_t)n_items;
            } else if (!first || k >= (uint32_t)n_items || atomicExch(&work[2 + k], 1u) != 0u) {
                do
                    k = atomicAdd(&work[0], 1u);
                while (k < (uint32_t)n_items && atomicExch(&work[2 + k], 1u) != 0u);
            }
            s_item = (int32_t)k;
        }
        first = false;
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
    // the bound is the kernel's, for all batches alive: one that needs less leaves it
    static std::mutex mutex;
    static size_t bound[64] = {};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess)
        return err;
    const std::lock_guard<std::mutex> lock(mutex);
    if (dev < 64 && smem <= bound[dev])
        return cudaSuccess;
    err = cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err == cudaSuccess && dev < 64)
        bound[dev] = smem;
    return err;
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

cudaError_t launch_batch(const SweepArgs *insts, const BatchItem *items, int32_t n_items, uint32_t *work,
                         int grid, size_t smem, bool record, cudaStream_t s)
{
    if (n_items <= 0)
        return cudaSuccess;
    const cudaError_t err = cudaMemsetAsync(work, 0, sizeof(uint32_t) * (2 + (size_t)n_items), s);
    if (err != cudaSuccess)
        return err;
    batch_kernel<<<grid, kBatchThreads, smem, s>>>(insts, items, n_items, work, record);
    return cudaGetLastError();
}

}  // namespace muca
