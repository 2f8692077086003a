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
cudaError_t launch_full_t(const SweepArgs &a, int wpb, bool record, cudaStream_t s)
{
    const size_t smem = launch_smem_bytes(L, wpb);
    auto kern = sweep_full_kernel<L, Stream>;
    static std::atomic<uint64_t> allowed{0};
    const cudaError_t err = allow_smem(kern, allowed);
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

cudaError_t MUCA_CAT(launch_full_L, MUCA_L)(const SweepArgs &a, int wpb, SweepForm form, bool record, cudaStream_t s)
{
    if (form.chains > 0)
        return launch_pair_t<MUCA_L>(a, form.chains, record, s);
    return form.ahead ? launch_full_t<MUCA_L, AttemptStream<MUCA_L, kTableStride, (MUCA_L <= 32 ? 1 : 0)>>(a, wpb, record, s)
                      : launch_full_t<MUCA_L, DirectStream<MUCA_L, kTableStride>>(a, wpb, record, s);
}

}  // namespace muca
