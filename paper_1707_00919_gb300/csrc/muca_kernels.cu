// muca_kernels.cu - the launch choice of the sweep kernels (muca_full.cuh) and the kernels
// around them (initial spins, lattice packing and unpacking, the Philox test kernel) of the
// parallel multicanonical 2D Ising update (Gross, Zierenberg, Weigel, Janke,
// arXiv:1707.00919, Sec. 2.3).
#include <algorithm>
#include <cstdint>

#include "muca_device.cuh"

namespace muca {
namespace {

// ---------------------------------------------------------------------------------
// Initial spins: +1 iff the top bit of the tag-1 word for attempt number t = site is
// clear; the energy index is the number of unsatisfied bonds over two.
// ---------------------------------------------------------------------------------
// Blocks of 32 walkers, one lane each, and a warp per strip of kStrip rows.  One thread per
// walker and all its rows left most of the device idle and the strips' latency in series:
// a lattice of L = 64 and 8106 walkers (33 MB) took 148 us to make and 360 us to take over from
// the host's format, in strips 53 and 52.
constexpr int kStrip = 4;
constexpr int kMaxStrips = 64 / kStrip;

// Writes a walker's lattice, given row by row (bit x = spin at x is down), in the
// instance's layout, and its energy index: the number of unsatisfied bonds over two.
// Every thread of the block calls it.
template <typename RowT, int LAYOUT, class RowSource>
__device__ __forceinline__ void write_lattice(int32_t L, int64_t W, int64_t w, const RowSource &rows, void *lattice,
                                              int32_t *energy)
{
    __shared__ RowT first[kMaxStrips][32];   // first row of each strip
    __shared__ int32_t bonds[kMaxStrips][32];
    const int lane = threadIdx.x & 31, strip = threadIdx.x >> 5, strips = L / kStrip;
    const RowT mask = (L == (int)(8 * sizeof(RowT))) ? ~(RowT)0 : (((RowT)1 << L) - 1);
    RowT prev = 0;
    int unsat = 0;
    if (w < W) {
        for (int i = 0; i < kStrip; ++i) {
            const int y = strip * kStrip + i;
            const RowT r = rows(y);
            const RowT rot = (r >> 1) | ((r & 1) << (L - 1));   // bit x = spin at x+1 (mod L)
            unsat += __popcll((unsigned long long)((r ^ rot) & mask));
            if (i == 0)
                first[strip][lane] = r;
            else
                unsat += __popcll((unsigned long long)((r ^ prev) & mask));
            prev = r;
            if (LAYOUT == MUCA_LAYOUT_PACKED) {
                reinterpret_cast<RowT *>(lattice)[(size_t)y * W + w] = r;
            } else {
                int8_t *g = reinterpret_cast<int8_t *>(lattice);
                for (int x = 0; x < L; ++x)
                    g[(size_t)(y * L + x) * W + w] = bit_at(r, x) ? (int8_t)-1 : (int8_t)1;
            }
        }
    }
    __syncthreads();
    if (w < W) {   // the strip's last row to the next strip's first (row L-1 to row 0)
        const RowT next = first[strip + 1 < strips ? strip + 1 : 0][lane];
        bonds[strip][lane] = unsat + __popcll((unsigned long long)((prev ^ next) & mask));
    }
    __syncthreads();
    if (w < W && strip == 0) {
        unsat = 0;
        for (int i = 0; i < strips; ++i)
            unsat += bonds[i][lane];
        energy[w] = unsat / 2;
    }
}

template <typename RowT>
struct InitRows {
    int32_t L;
    uint32_t k0, k1, w;
    __device__ RowT operator()(int y) const
    {
        RowT r = 0;
        for (int x = 0; x < L; x += 4) {
            const uint32_t site = (uint32_t)(y * L + x);
            const uint4 q = philox4x32_10(make_uint4(site >> 2, 0u, w, kTagInit), k0, k1);
            const uint32_t words[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                r |= (RowT)(words[u] >> 31) << (x + u);
        }
        return r;
    }
};

template <typename RowT>
struct GivenRows {
    int32_t L;
    const int8_t *spins;   // this walker's N spins, +1 / -1
    bool words;            // whether they can be read as 4-byte words
    __device__ RowT operator()(int y) const
    {
        RowT r = 0;
        for (int x = 0; x < L; x += 4) {
            const int8_t *p = spins + y * L + x;
            if (words)
                r |= (RowT)gather_signs(*reinterpret_cast<const uint32_t *>(p)) << x;
            else
                for (int u = 0; u < 4; ++u)
                    r |= (RowT)(p[u] < 0) << (x + u);
        }
        return r;
    }
};

template <typename RowT, int LAYOUT>
__global__ void __launch_bounds__(32 * kMaxStrips) init_kernel(int32_t L, int64_t W, uint64_t seed, uint32_t walker0,
                                                               void *lattice, int32_t *energy)
{
    const int64_t w = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
    const InitRows<RowT> rows{L, (uint32_t)seed, (uint32_t)(seed >> 32), walker0 + (uint32_t)w};
    write_lattice<RowT, LAYOUT>(L, W, w, rows, lattice, energy);
}

// Lattices given as int8 in[walker][site] (+1 / -1) into the layout, energies recomputed.
template <typename RowT, int LAYOUT>
__global__ void __launch_bounds__(32 * kMaxStrips) pack_kernel(int32_t L, int64_t W, const int8_t *in, void *lattice,
                                                               int32_t *energy)
{
    const int64_t w = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
    const GivenRows<RowT> rows{L, in + (size_t)w * (size_t)(L * L), reinterpret_cast<uintptr_t>(in) % 4 == 0};
    write_lattice<RowT, LAYOUT>(L, W, w, rows, lattice, energy);
}

// The layout to int8 out[walker][site]: bound by memory, a transposition for int8.  A thread
// writes 16 consecutive sites of its walker (L is a multiple of four, N of 16), which it
// reads coalesced over the lanes, all at once.  One thread per walker and a byte at a time
// took 539 us for L = 32 and 16384 walkers of bytes (16.8 MB each way), this 13 (2.6 TB/s).
constexpr int kUnpackWarps = 8;

template <typename RowT, int LAYOUT>
__global__ void __launch_bounds__(32 * kUnpackWarps) unpack_kernel(int32_t L, int64_t W, const void *lattice, int8_t *out)
{
    const int64_t w = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
    const int N = L * L, i0 = 16 * (int)(blockIdx.y * kUnpackWarps + (threadIdx.x >> 5));
    if (w >= W || i0 >= N)
        return;
    uint32_t v[4];
    if (LAYOUT == MUCA_LAYOUT_PACKED) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {   // four sites lie in one row
            const int y = (i0 + 4 * j) / L, x = i0 + 4 * j - y * L;
            v[j] = spread_signs((uint32_t)(reinterpret_cast<const RowT *>(lattice)[(size_t)y * W + w] >> x) & 15u);
        }
    } else {
        const uint8_t *g = reinterpret_cast<const uint8_t *>(lattice) + (size_t)i0 * W + w;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j] = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                v[j] |= (uint32_t)g[(size_t)(4 * j + u) * W] << (8 * u);
        }
    }
    int8_t *o = out + (size_t)w * N + i0;
    if (reinterpret_cast<uintptr_t>(out) % 16 == 0) {
        *reinterpret_cast<uint4 *>(o) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            o[j] = (int8_t)(v[j / 4] >> (8 * (j % 4)));
    }
}

__global__ void philox_kernel(const uint32_t *ctr, uint32_t k0, uint32_t k1, size_t n, uint32_t *out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 r = philox4x32_10(c, k0, k1);
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
}

// The form of a launch by the warps of walkers per SM.  Up to two, and with the device to
// itself: the paired kernel, its generator warps on the sub-partitions that would idle
// (when sweeps of other instances run, it would take SMs from them for less throughput:
// eight instances of L = 32 with 4096 walkers, all queued, 1724 us per 20 sweeps with it
// against 890).  Up to eight, two per sub-partition: the two-ahead loads.  More than that
// resident at once: direct loads, whose latency the other warps cover (how many the kernel's
// blocks leave resident is looked at where it is launched, muca_full.cuh).
SweepForm sweep_form(const SweepArgs &a, bool alone)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return {0, true};
    const int64_t warps = (a.W + 31) / 32;
    if (alone && warps <= 2 * (int64_t)sms) {
        // one chain warp per block spreads them over the SMs; from L = 52 on the table leaves
        // room for one block per SM only, and two chains share it, so that a sweep queued
        // after this one finds SMs
        const bool two = warps > sms || (a.L >= 52 && warps > 1);
        return {two ? 2 : 1, true};
    }
    return {0, warps <= 8 * (int64_t)sms};
}

// Dispatches a launch to the kernel for L.
cudaError_t launch_full(const SweepArgs &a, int wpb, bool alone, bool record, cudaStream_t s, SweepForm &form)
{
    const bool no_waits = form.no_waits;
    form = sweep_form(a, alone);
    form.no_waits = no_waits;
    switch (a.L) {
    case 4: return launch_full_L4(a, wpb, form, record, s);
    case 8: return launch_full_L8(a, wpb, form, record, s);
    case 12: return launch_full_L12(a, wpb, form, record, s);
    case 16: return launch_full_L16(a, wpb, form, record, s);
    case 20: return launch_full_L20(a, wpb, form, record, s);
    case 24: return launch_full_L24(a, wpb, form, record, s);
    case 28: return launch_full_L28(a, wpb, form, record, s);
    case 32: return launch_full_L32(a, wpb, form, record, s);
    case 36: return launch_full_L36(a, wpb, form, record, s);
    case 40: return launch_full_L40(a, wpb, form, record, s);
    case 44: return launch_full_L44(a, wpb, form, record, s);
    case 48: return launch_full_L48(a, wpb, form, record, s);
    case 52: return launch_full_L52(a, wpb, form, record, s);
    case 56: return launch_full_L56(a, wpb, form, record, s);
    case 60: return launch_full_L60(a, wpb, form, record, s);
    case 64: return launch_full_L64(a, wpb, form, record, s);
    default: return cudaErrorNotSupported;
    }
}

}  // namespace

size_t full_smem_bytes(int L, int wpb, bool record, bool guard, int stride)
{
    (void)record;
    const size_t rows = (size_t)L * L + 1 + (guard ? 2 * kTableGuard : 0);
    const size_t per_walker = L <= 32 ? (size_t)L * row_words(L) * 4 : (size_t)L * 8;
    return align_up(rows * (size_t)stride * 4, 16) + per_walker * (size_t)wpb;
}

size_t launch_smem_bytes(int L, int wpb, bool guard, int stride)
{
    const size_t rows = (size_t)L * L + 2 + (guard ? 2 * kTableGuard : 0);
    const size_t per_walker = L <= 32 ? (size_t)L * row_words(L) * 4 : (size_t)L * 8;
    return align_up(rows * (size_t)stride * 4, 16) + per_walker * (size_t)wpb;
}

size_t sizing_smem_bytes(int L, int wpb)
{
    const size_t nb = (size_t)L * L + 1;
    const size_t row = L <= 32 ? 4 : 8;
    return align_up(nb * 6 * 4, 16) + (size_t)L * wpb * row;
}

size_t sweep_smem_limit()
{
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;   // nothing fits: callers report it
    return (size_t)v;
}

cudaError_t launch_sweep(const SweepArgs &a, int wpb, bool alone, bool record, cudaStream_t s, SweepForm *form)
{
    if (a.W == 0 || (a.n == 0 && a.n_therm == 0))
        return cudaSuccess;
    SweepArgs part = a;
    if (a.n_therm > 0 && (a.t0 >> 34) != ((a.t0 + a.n_therm + a.n - 1) >> 34)) {
        // not one launch: the thermalization by itself
        part.n_therm = 0;
        part.n = a.n_therm;
        const cudaError_t err = launch_sweep(part, wpb, alone, false, s, form);
        if (err != cudaSuccess)
            return err;
        part.t0 = a.t0 + a.n_therm;
        part.n = a.n;
        return launch_sweep(part, wpb, alone, record, s, form);
    }
    for (uint64_t left = a.n; left > 0; left -= part.n, part.t0 += part.n) {
        part.n = a.n_therm > 0 ? left : same_word1(part.t0, left);
        const cudaError_t err = launch_full(part, wpb, alone, record, s, *form);
        if (err != cudaSuccess)
            return err;
    }
    return cudaSuccess;
}

cudaError_t launch_init(int32_t L, int32_t layout, int64_t W, uint64_t seed, uint32_t walker0, void *lattice,
                        int32_t *energy,
                        cudaStream_t s)
{
    const int threads = 32 * (L / kStrip);
    const unsigned blocks = (unsigned)((W + 31) / 32);
    if (L <= 32) {
        if (layout == MUCA_LAYOUT_PACKED)
            init_kernel<uint32_t, MUCA_LAYOUT_PACKED><<<blocks, threads, 0, s>>>(L, W, seed, walker0, lattice, energy);
        else
            init_kernel<uint32_t, MUCA_LAYOUT_INT8><<<blocks, threads, 0, s>>>(L, W, seed, walker0, lattice, energy);
    } else {
        if (layout == MUCA_LAYOUT_PACKED)
            init_kernel<unsigned long long, MUCA_LAYOUT_PACKED><<<blocks, threads, 0, s>>>(L, W, seed, walker0, lattice, energy);
        else
            init_kernel<unsigned long long, MUCA_LAYOUT_INT8><<<blocks, threads, 0, s>>>(L, W, seed, walker0, lattice, energy);
    }
    return cudaGetLastError();
}

cudaError_t launch_pack(int32_t L, int32_t layout, int64_t W, const int8_t *in, void *lattice, int32_t *energy,
                        cudaStream_t s)
{
    const int threads = 32 * (L / kStrip);
    const unsigned blocks = (unsigned)((W + 31) / 32);
    if (L <= 32) {
        if (layout == MUCA_LAYOUT_PACKED)
            pack_kernel<uint32_t, MUCA_LAYOUT_PACKED><<<blocks, threads, 0, s>>>(L, W, in, lattice, energy);
        else
            pack_kernel<uint32_t, MUCA_LAYOUT_INT8><<<blocks, threads, 0, s>>>(L, W, in, lattice, energy);
    } else {
        if (layout == MUCA_LAYOUT_PACKED)
            pack_kernel<unsigned long long, MUCA_LAYOUT_PACKED><<<blocks, threads, 0, s>>>(L, W, in, lattice, energy);
        else
            pack_kernel<unsigned long long, MUCA_LAYOUT_INT8><<<blocks, threads, 0, s>>>(L, W, in, lattice, energy);
    }
    return cudaGetLastError();
}

cudaError_t launch_unpack(int32_t L, int32_t layout, int64_t W, const void *lattice, int8_t *out, cudaStream_t s)
{
    const int threads = 32 * kUnpackWarps;
    const dim3 blocks((unsigned)((W + 31) / 32), (unsigned)((L * L + 16 * kUnpackWarps - 1) / (16 * kUnpackWarps)));
    if (L <= 32) {
        if (layout == MUCA_LAYOUT_PACKED)
            unpack_kernel<uint32_t, MUCA_LAYOUT_PACKED><<<blocks, threads, 0, s>>>(L, W, lattice, out);
        else
            unpack_kernel<uint32_t, MUCA_LAYOUT_INT8><<<blocks, threads, 0, s>>>(L, W, lattice, out);
    } else {
        if (layout == MUCA_LAYOUT_PACKED)
            unpack_kernel<unsigned long long, MUCA_LAYOUT_PACKED><<<blocks, threads, 0, s>>>(L, W, lattice, out);
        else
            unpack_kernel<unsigned long long, MUCA_LAYOUT_INT8><<<blocks, threads, 0, s>>>(L, W, lattice, out);
    }
    return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t *ctr, uint32_t k0, uint32_t k1, size_t n, uint32_t *out, cudaStream_t s)
{
    if (n == 0)
        return cudaSuccess;
    const int threads = 128;
    philox_kernel<<<(unsigned)((n + threads - 1) / threads), threads, 0, s>>>(ctr, k0, k1, n, out);
    return cudaGetLastError();
}

// Registers per thread that the sizing rule counts with, by L and layout; 0 where it counts
// bit rows, six words per table row and threads alone.  The walker count of full occupancy
// and with it the chains of an instance created without an explicit count, and the default
// block size, follow from this rule, so it is fixed and does not move with the sweep kernels.
// It is theirs at L = 16, 24, 32, 36, 48, 52, 56, 60 and 64; at the other sizes they need more
// (100 registers at L = 8, 106 at L = 4) and fewer walkers fit an SM than it says (muca.h).
// What a launch takes for granted is asked of its kernel (muca_full.cuh).
static int sizing_registers(int L, int layout)
{
    const bool packed = layout == MUCA_LAYOUT_PACKED;
    switch (L) {
    case 8: return packed ? 104 : 80;
    case 16: return 88;
    case 24: return 104;
    case 32: return packed ? 112 : 120;
    case 48: return packed ? 248 : 168;
    case 64: return packed ? 168 : 200;
    default: return 0;
    }
}

int resident_blocks(int L, int layout, int wpb)
{
    int dev = 0, smem_sm = 0, smem_block = 0, regs_sm = 0, thr_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&thr_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev) != cudaSuccess)
        return 0;   // no resident block: callers skip this block size
    const int regs = sizing_registers(L, layout);
    const size_t smem = regs ? full_smem_bytes(L, wpb, true) : sizing_smem_bytes(L, wpb);
    if (regs && smem > (size_t)smem_block)
        return 0;
    // a block takes its shared memory rounded up (128 bytes) and 1 KB of its own
    const size_t need = regs ? align_up(smem, 128) + 1024 : smem + 1024;
    int n = (int)std::min((size_t)smem_sm / need, (size_t)(thr_sm / wpb));
    if (regs)   // a quarter of the registers per sub-partition, whole warps
        n = std::min(n, (regs_sm / 4 / (regs * 32)) * 4 / (wpb / 32));
    return n;
}

size_t lattice_bytes(int32_t L, int32_t layout, int64_t W)
{
    if (layout == MUCA_LAYOUT_PACKED)
        return (size_t)L * (size_t)W * (L <= 32 ? 4 : 8);
    return (size_t)L * L * (size_t)W;
}

}  // namespace muca
