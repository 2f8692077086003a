// muca_full.cuh - the sweep kernel for one lattice size; included by muca_full_L.cu with
// MUCA_L defined, so that the sizes compile in parallel.
#pragma once

#include "muca_device.cuh"
#include "muca_pair.cuh"

#ifndef MUCA_L
#error "define MUCA_L before including muca_full.cuh"
#endif

namespace muca {
namespace {

template <int L, class Stream>
__global__ void __launch_bounds__(256, 1) sweep_full_kernel(const SweepArgs a, const __grid_constant__ LaunchPlan plan,
                                                            const bool record)
{
    extern __shared__ __align__(16) unsigned char smem[];
    sweep_block<L, false, kTableStride, Stream>(a, HostPlans{plan}, (int64_t)blockIdx.x * blockDim.x, blockDim.x, smem,
                                                record);
}

template <int L, class Stream>
cudaError_t allow_full()
{
    static std::atomic<uint64_t> allowed{0};
    return allow_smem(sweep_full_kernel<L, Stream>, allowed);
}

// Warps of the kernel that an SM holds at once in blocks of wpb walkers, as the runtime counts
// them (0 if it does not answer), asked once per block size and device.
template <int L, class Stream>
int resident_warps(int wpb)
{
    static std::atomic<int16_t> known[64][8];   // plus one
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || allow_full<L, Stream>() != cudaSuccess)
        return 0;
    std::atomic<int16_t> *const slot = dev < 64 ? &known[dev][wpb / 32 - 1] : nullptr;
    int n = slot ? slot->load(std::memory_order_relaxed) - 1 : -1;
    if (n < 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sweep_full_kernel<L, Stream>, wpb,
                                                          launch_smem_bytes(L, wpb)) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        n *= wpb / 32;
        if (slot)
            slot->store((int16_t)(n + 1), std::memory_order_relaxed);
    }
    return n;
}

template <int L, class Stream>
cudaError_t launch_full_t(const SweepArgs &a, int wpb, bool record, cudaStream_t s)
{
    const size_t smem = launch_smem_bytes(L, wpb);
    auto kern = sweep_full_kernel<L, Stream>;
    const cudaError_t err = allow_full<L, Stream>();
    if (err != cudaSuccess)
        return err;
    const int64_t blocks = (a.W + wpb - 1) / wpb;
    LaunchPlan plan;
    plan.phase[0] = row_plan(L, a.t0, a.n_therm);
    plan.phase[1] = row_plan(L, a.t0 + a.n_therm, a.n);
    kern<<<(unsigned)blocks, wpb, smem, s>>>(a, plan, record);
    return cudaGetLastError();
}

}  // namespace

#define MUCA_CAT2(a, b) a##b
#define MUCA_CAT(a, b) MUCA_CAT2(a, b)

cudaError_t MUCA_CAT(launch_full_L, MUCA_L)(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s)
{
    using Ahead = AttemptStream<MUCA_L, kTableStride, (MUCA_L <= 32 ? 1 : 0)>;
    using Direct = DirectStream<MUCA_L, kTableStride>;
    if constexpr (MUCA_L == 8 || MUCA_L == 32)   // for tests
        if (form.chains > 0 && form.no_waits)
            return launch_pair_t<MUCA_L, 0>(a, form.chains, record, s);
    if (form.chains > 0)
        return launch_pair_t<MUCA_L>(a, form.chains, record, s);
    // the walkers are many, but an SM may hold two warps per sub-partition at a time all the
    // same (L = 44 in blocks of 192: 6 warps)
    form.ahead = form.ahead || resident_warps<MUCA_L, Direct>(wpb) <= 8;
    return form.ahead ? launch_full_t<MUCA_L, Ahead>(a, wpb, record, s) : launch_full_t<MUCA_L, Direct>(a, wpb, record, s);
}

}  // namespace muca
