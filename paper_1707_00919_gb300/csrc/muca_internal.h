// muca_internal.h - launch interface between the host library (muca_api*.cu) and the
// device kernels (muca_kernels.cu and the other kernel files).  Not part of the public ABI.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace muca {

// Shared-memory table of the sweep kernels: one row of kTableStride words per
// energy, thresholds in words 0..4, the block's histogram count in word kHistSlot.
constexpr int kTableStride = 7;
constexpr int kHistSlot = 5;
// Zero rows below energy 0 and above N for the allocation-free entry point, whose
// energies come from the caller: the threshold candidates loaded ahead of a decision lie
// within two rows of the current energy, so they stay inside the table even for
// energies that do not match the lattices.
constexpr int kTableGuard = 2;
// Table row stride of the batched kernel: 6 words at L = 64, so that 256 walkers fit next to the 4097-row table.
__host__ __device__ constexpr int batch_table_stride(int L) { return L == 64 ? 6 : kTableStride; }

// Device error word bits.
constexpr uint32_t kErrEnergyRange = 1u;   // a walker's energy index was off the grid
constexpr uint32_t kErrSyncTimeout = 2u;   // a bounded wait inside a kernel gave up

struct SweepArgs {
    int32_t L;                  // lattice side (multiple of 4, <= 64)
    int32_t layout;             // MUCA_LAYOUT_*
    int64_t W;                  // walkers
    uint64_t seed;              // Philox key
    uint64_t t0;                // attempt counter of the first attempt
    uint64_t n;                 // attempts per walker in this launch
    void *lattice;              // layout-dependent, see muca.h
    int32_t *energy;            // [W]
    const uint32_t *table;      // [(N+1)*5]
    unsigned long long *hist;   // [N+1], accumulated when recording
    uint32_t *err;              // device error word
    const uint32_t *skip = nullptr;   // when set and nonzero at launch: the launch does nothing
    uint32_t walker0 = 0;             // global index of walker 0 (the Philox walker word is walker0 + w)
    // Thermalization attempts run before the launch's n recorded ones, from t0 (the
    // recorded attempts then start at t0 + n_therm).  Only a recording launch in typewriter
    // order sets it.
    uint64_t n_therm = 0;
};

// A range of attempts row by row: part of a first row, whole rows, part of a last row, all
// with the same Philox counter word 1.
struct RowPlan {
    int32_t y0, x0, x0_end;        // first row, attempts [x0, x0_end) of it (none if equal)
    int32_t y1;                    // first whole row
    int32_t y2, tail;              // last row, attempts [0, tail) of it
    uint32_t blk0, blk1, blk2;     // Philox blocks of column 0 of rows y0, y1 and y2
    uint32_t c1;                   // counter word 1
    uint64_t rows;                 // whole rows
};

struct LaunchPlan {
    RowPlan phase[2];   // thermalization, the launch's own attempts
};

// The attempts from t0 on, at most n, that share t0's counter word 1 (t >> 34).
__host__ __device__ inline uint64_t same_word1(uint64_t t0, uint64_t n)
{
    const uint64_t room = (((t0 >> 34) + 1) << 34) - t0;
    return n < room ? n : room;
}

__host__ __device__ inline RowPlan row_plan(int L, uint64_t t0, uint64_t n)
{
    RowPlan p;
    const int32_t i = (int32_t)(t0 % (uint64_t)(L * L));
    p.y0 = p.y1 = i / L;
    p.x0 = p.x0_end = i % L;
    p.blk0 = p.blk1 = (uint32_t)((t0 - (uint64_t)p.x0) >> 2);
    p.c1 = (uint32_t)(t0 >> 34);
    if (p.x0 != 0) {
        const uint64_t m = n < (uint64_t)(L - p.x0) ? n : (uint64_t)(L - p.x0);
        p.x0_end = p.x0 + (int32_t)m;
        n -= m;
        p.y1 = p.y0 + 1 == L ? 0 : p.y0 + 1;
        p.blk1 = p.blk0 + (uint32_t)(L / 4);
    }
    p.rows = n / (uint64_t)L;
    p.tail = (int32_t)(n % (uint64_t)L);
    p.y2 = (int32_t)(((uint64_t)p.y1 + p.rows) % (uint64_t)L);
    p.blk2 = p.blk1 + (uint32_t)p.rows * (uint32_t)(L / 4);
    return p;
}

// Largest dynamic shared memory a block may use on this device (bytes; 0 if the device does
// not answer).
size_t sweep_smem_limit();

// Allows a kernel the device's whole shared memory, once per kernel and device: `done` has
// a bit per device (the attribute is a bound only, and setting it takes microseconds).
template <class Kernel>
cudaError_t allow_smem(Kernel kern, std::atomic<uint64_t> &done)
{
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess)
        return err;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
    if (done.load(std::memory_order_acquire) & bit)
        return cudaSuccess;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sweep_smem_limit());
    if (err == cudaSuccess)
        done.fetch_or(bit, std::memory_order_release);
    return err;
}

// Form of a sweep launch: `chains` > 0: paired kernel with that many chain warps per block
// (muca_pair.cuh); else one thread per walker, the thresholds loaded two attempts ahead or
// directly (muca_device.cuh).
struct SweepForm {
    int32_t chains;
    bool ahead;
    bool no_waits = false;   // for tests, L = 8 and 32: every wait of the paired kernel runs out at once
};

// Waits between the warps of the paired kernel: tries of at most 20 us each before a wait
// gives up (a slot of the ring turns over in a few microseconds).
constexpr uint32_t kPairWaitTries = 1u << 16;
constexpr int kPairMaxThreads = 128;

// Device state of an iteration whose recursion runs on the device (muca_iterate_device).
struct IterState {
    uint32_t done;       // 0: running; 1: the last histogram was flat; 2: iteration limit
    uint32_t update;     // the last metric asked for the recursion and the next table
    int32_t iterations;  // iterations whose histogram was tested
    int32_t prev_lo;     // energy range visited in the previous iteration (-1: none)
    int32_t prev_hi;
    int32_t pad;
    double metric;       // stop metric of the last tested histogram
};

// The steps of one device-side iteration after its recorded sweeps (muca_iterate.cu):
// zeroing the histogram (skipped once done), the stop metric (one block; skipped once
// done), the Eq. (4) recursion and the table of the next iteration (both only when the
// metric kernel set `update`).
cudaError_t launch_iter_reset_hist(unsigned long long *hist, int32_t nb, const IterState *st, cudaStream_t s);
cudaError_t configure_iter_metric(int32_t N);
cudaError_t launch_iter_metric(IterState *st, int32_t N, const unsigned long long *hist, int32_t stop_rule,
                               double flat_threshold, int32_t max_iterations, cudaStream_t s);
cudaError_t launch_iter_recursion(const IterState *st, int32_t N, double *lnW, const unsigned long long *hist,
                                  cudaStream_t s);
cudaError_t launch_iter_table(const IterState *st, int32_t N, const double *lnW, uint32_t *table, cudaStream_t s);

// New weights of an instance: src[N + 1] (pinned host memory) to lnW, thresholds T[e][k]
// (the host's build_table arithmetic, bit for bit), the histogram zeroed unless hist is null.
struct TableJob {
    const double *src;
    double *lnW;
    uint32_t *table;
    unsigned long long *hist;
    int32_t N;
};
cudaError_t launch_table(const TableJob &job, cudaStream_t s);

// The same for all members of a batch (jobs in device memory, bins: the most of any).
struct BatchJob {
    TableJob table;
    const uint32_t *err;            // to h_err and, with the histogram, h_hist (pinned)
    uint32_t *h_err;
    unsigned long long *h_hist;
};
cudaError_t launch_batch_tables(const BatchJob *jobs, int32_t n, int32_t bins, cudaStream_t s);
cudaError_t launch_batch_read(const BatchJob *jobs, int32_t n, int32_t bins, cudaStream_t s);

// One work item of the batched kernel: walkers wbase .. wbase + wpb - 1 of instance inst.
struct BatchItem {
    int32_t inst;
    int32_t wpb;
    int64_t wbase;
};

constexpr int kBatchThreads = 256;   // threads per block of the batched kernel

// Shared memory bytes that the sizing rule counts for an L without a register count of its
// own (bit rows, thresholds and counts; not what the kernel takes, launch_smem_bytes).
size_t sizing_smem_bytes(int L, int walkers_per_block);

// Shared memory bytes of the sweep kernel's table and rows, by which block sizes are
// chosen, and those of a launch (with the row of zeros).
size_t full_smem_bytes(int L, int walkers_per_block, bool record, bool guard = false, int stride = kTableStride);
size_t launch_smem_bytes(int L, int walkers_per_block, bool guard = false, int stride = kTableStride);

// Runs a.n_therm thermalization attempts from a.t0 (recording launches only; may be 0),
// then a.n attempts of every walker: one launch unless the range crosses a step of counter
// word 1 (every 2^34 attempts).  alone: no other sweep that the library knows of is in flight
// on the device, so that the launch may take more SMs than its walkers fill.  *form receives
// the form taken.
cudaError_t launch_sweep(const SweepArgs &a, int walkers_per_block, bool alone, bool record, cudaStream_t s,
                         SweepForm *form);

// Runs attempts [t0, t0 + n) of every walker in random shared site order (muca_random.cu;
// any L, any attempt range; the given block size, or a smaller one that fits shared
// memory).
cudaError_t launch_random_sweep(const SweepArgs &a, int walkers_per_block, bool record, cudaStream_t s);

// Draws the initial spins (tag 1 stream) and their energy indices.
cudaError_t launch_init(int32_t L, int32_t layout, int64_t W, uint64_t seed, uint32_t walker0, void *lattice,
                        int32_t *energy, cudaStream_t s);

// Packs lattices given as int8 in[walker][site] (+1/-1) and recomputes their energies.
cudaError_t launch_pack(int32_t L, int32_t layout, int64_t W, const int8_t *in, void *lattice, int32_t *energy,
                        cudaStream_t s);

// Unpacks lattices into int8 out[walker][site] (+1/-1).
cudaError_t launch_unpack(int32_t L, int32_t layout, int64_t W, const void *lattice, int8_t *out,
                          cudaStream_t s);

// Evaluates the device Philox4x32-10 on n counters.
cudaError_t launch_philox(const uint32_t *ctr, uint32_t k0, uint32_t k1, size_t n, uint32_t *out,
                          cudaStream_t s);

// Kernels of one L each (muca_full_L.cu): launch over any attempt range in the given form;
// direct loads (not ahead) only if an SM holds more than eight warps at once, else form.ahead
// is set.
cudaError_t launch_full_L4(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L8(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L12(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L16(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L20(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L24(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L28(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L32(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L36(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L40(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L44(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L48(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L52(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L56(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L60(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);
cudaError_t launch_full_L64(const SweepArgs &a, int wpb, SweepForm &form, bool record, cudaStream_t s);

// Blocks for this L, layout and block size that one SM holds at once by the sizing rule of the
// default walker count and block size (0 if the configuration does not fit).
int resident_blocks(int L, int layout, int walkers_per_block);

// Batched persistent kernel: allows `smem` bytes of dynamic shared memory, reports how
// many blocks of it an SM holds, and launches it over a work list (work: 2 + n_items words,
// zeroed on the stream in front of it; L must be one of 8, 16, 24, 32, 48, 64).
cudaError_t configure_batch(size_t smem);
int batch_resident_blocks(size_t smem);
cudaError_t launch_batch(const SweepArgs *insts, const BatchItem *items, int32_t n_items, uint32_t *work,
                         int grid, size_t smem, bool record, cudaStream_t s);
// Allocation-free batched sweep (see muca_batch_sweep_noalloc in muca.h): descriptors,
// walkers per item and the prefix sums of the work items per instance (prefix[0] = 0,
// prefix[n] = all items, below 2^31) come from the host and travel in the launch
// parameters; the kernel's only scratch, its work counter, is a file-scope device array
// of kNoAllocScratchBytes, looked up on the first call per device.
constexpr int kNoAllocMaxInstances = 64;
constexpr int kNoAllocMaxDevices = 64;
constexpr size_t kNoAllocScratchBytes = 256;
cudaError_t launch_batch_noalloc(const SweepArgs *descs, const int32_t *wpbs, const int32_t *prefix, int32_t n,
                                 size_t smem, bool record, cudaStream_t s);

// Issue rate of one instruction class (muca_probe.cu, see muca_measure_issue_rate).
cudaError_t measure_issue_rate(int kind, double *per_second);

// Bytes of the lattice storage of W walkers.
size_t lattice_bytes(int32_t L, int32_t layout, int64_t W);

}  // namespace muca
