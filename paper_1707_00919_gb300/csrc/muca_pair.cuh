// muca_pair.cuh - the sweep kernel for launches of few walkers: the warps that run the
// chains get their random words from other warps of the block.  Included by muca_full.cuh.
//
// With at most two warps of walkers per SM, sub-partitions are idle and a chain warp is
// bound by its own instruction issue (one half-rate instruction per two cycles, a wide
// multiply twice that): Philox is half of it.  Generator warps on the idle sub-partitions
// draw the words into a ring in shared memory, a chunk of about 128 attempts at a time, and
// the chain warp reads four words per 16-byte load.  What bounds it now is the chain warp's
// issue again, 18 instructions per attempt.  Measured, us per sweep without and with the
// generators: L = 8, 128 walkers 1.58 -> 1.19; L = 16, 4096 walkers 6.30 -> 4.41; L = 24,
// 5003 walkers 14.2 -> 10.4; L = 32, 4096 walkers 24.4 -> 17.7; L = 48, 1024 walkers 56.5 ->
// 42.0; L = 64, 4096 or 9728 walkers 99.4 -> 73.4.
#pragma once

#include "muca_device.cuh"

namespace muca {
namespace {

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Waits for the phase of the given parity, TRIES times at most 20 us; false on expiry.  (A
// number of tries that comes with the launch made the kernel 2 % slower.)
template <uint32_t TRIES>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
#pragma unroll 1
    for (uint32_t i = 0; i < TRIES; ++i) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(bar), "r"(parity), "r"(20000u)
                     : "memory");
        if (done)
            return true;
    }
    return false;
}

// One chain warp's ring: two slots of a chunk of rows each, 16 bytes per lane and Philox
// block, with a full and an empty barrier per slot.  Chunks are counted over the launch
// (c), so that both sides agree on slot and phase.
template <int L, uint32_t TRIES>
struct PairRing {
    static constexpr int kRows = 128 / L;                           // rows per chunk
    static constexpr int kTogether = 4;                             // blocks drawn together
    static constexpr int kBlocks = (kRows * (L / 4) + kTogether - 1) / kTogether * kTogether;
    static constexpr uint32_t kSlotBytes = kBlocks * 512;
    // barriers, slots, and room for the load ahead of a chunk's last group
    __host__ __device__ static constexpr size_t bytes() { return 32 + 2 * (size_t)kSlotBytes + 512; }

    uint32_t bars;         // shared address of the four barriers
    uint32_t base;         // of this lane's part of slot 0
    uint32_t c = 0;        // current chunk
    bool ok = true;        // no wait has expired; after one that has, nothing is waited for

    __device__ __forceinline__ uint32_t slot() const { return base + (c & 1u) * kSlotBytes; }
    __device__ __forceinline__ uint32_t full() const { return bars + (c & 1u) * 8u; }
    __device__ __forceinline__ uint32_t empty() const { return bars + 16u + (c & 1u) * 8u; }

    // Generator j of `gens`: the words of its chunks of `nrows` whole rows from block b.
    __device__ __forceinline__ void generate(uint32_t b, uint64_t nrows, const PhiloxKeys &pk, int j, int gens, int lane)
    {
#pragma unroll 1
        for (uint64_t left = nrows; left > 0;) {
            const int rows = left < (uint64_t)kRows ? (int)left : kRows;
            if ((int)(c & (uint32_t)(gens - 1)) == j) {
                ok = ok && mbar_wait<TRIES>(empty(), ((c >> 1) & 1u) ^ 1u);
                uint32_t at = slot();
                const int nb = rows * (L / 4);
#pragma unroll 1
                for (int k = 0; k < nb; k += kTogether) {
                    uint4 w[kTogether];
                    words_together(b + (uint32_t)k, pk, w);
#pragma unroll
                    for (int i = 0; i < kTogether; ++i) {
                        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(w[i].x), "r"(w[i].y), "r"(w[i].z),
                                     "r"(w[i].w)
                                     : "memory");
                        at += 512u;
                    }
                }
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(full());
            }
            b += (uint32_t)(rows * (L / 4));
            left -= (uint64_t)rows;
            ++c;
        }
    }

    // Clamped words of kTogether consecutive blocks, round by round: their chains of ten
    // dependent products overlap.
    static __device__ __forceinline__ void words_together(uint32_t b, const PhiloxKeys &p, uint4 (&w)[kTogether])
    {
#pragma unroll
        for (int i = 0; i < kTogether; ++i) {
            const uint3 h = block_head(b + (uint32_t)i, p);
            w[i] = make_uint4(h.x ^ p.lo_w, h.y, h.z ^ p.r1_hi, p.r1_lo);
        }
#pragma unroll
        for (int r = 2; r < 10; ++r)
#pragma unroll
            for (int i = 0; i < kTogether; ++i) {
                const unsigned long long p0 = (unsigned long long)0xD2511F53u * w[i].x;
                const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * w[i].z;
                w[i] = make_uint4((uint32_t)(p1 >> 32) ^ w[i].y ^ p.k0[r], (uint32_t)p1, (uint32_t)(p0 >> 32) ^ w[i].w ^ p.k1[r],
                                  (uint32_t)p0);
            }
#pragma unroll
        for (int i = 0; i < kTogether; ++i)
            w[i] = make_uint4(min(w[i].x, 0xFFFFFFFEu), min(w[i].y, 0xFFFFFFFEu), min(w[i].z, 0xFFFFFFFEu),
                              min(w[i].w, 0xFFFFFFFEu));
    }
};

// The chain side's words of a row, loaded one group ahead of their use (past the chunk's
// last group into the next bytes of the ring, unused).
struct RingSource {
    uint32_t at;      // shared address of the group after the next
    uint4 ahead;      // words of the next group

    __device__ __forceinline__ void load()
    {
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(ahead.x), "=r"(ahead.y), "=r"(ahead.z), "=r"(ahead.w)
                     : "r"(at));
        at += 512u;
    }
    __device__ __forceinline__ uint4 get(int)
    {
        const uint4 w = ahead;
        load();
        return w;
    }
    __device__ __forceinline__ void advance() const {}
};

// Whole rows of a chain warp (see stream_rows) with the words of its ring.
template <int L, int STRIDE, uint32_t TRIES>
__device__ __forceinline__ uint32_t ring_rows(const SmemRows<L> &rows, uint32_t E, int y, uint64_t nrows,
                                              PairRing<L, TRIES> &ring, int lane)
{
    constexpr int NW = row_words(L);
    uint32_t U[NW], C[NW], D[NW];
    rows.load(y == 0 ? L - 1 : y - 1, U);
    rows.load(y, C);
    rows.load(y + 1 == L ? 0 : y + 1, D);
    AttemptStream<L, STRIDE, (L > 8 ? 2 : 1)> st;
    st.start(U, C, D, E);
#pragma unroll 1
    for (uint64_t left = nrows; left > 0;) {
        const int n = left < (uint64_t)ring.kRows ? (int)left : ring.kRows;
        ring.ok = ring.ok && mbar_wait<TRIES>(ring.full(), (ring.c >> 1) & 1u);
        RingSource src;
        src.at = ring.slot();
        src.load();
#pragma unroll 1
        for (int r = 0; r < n; ++r) {
            const int y2 = (y + 2 < L) ? y + 2 : y + 2 - L;
            uint32_t D2[NW];
            rows.load(y2, D2);
            st.row(U, C, D, D2, src);
            rows.store(y, C);
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                U[i] = C[i];
                C[i] = D[i];
                D[i] = D2[i];
            }
            y = (y + 1 == L) ? 0 : y + 1;
        }
        __syncwarp();   // every lane has read the chunk's words
        if (lane == 0)
            mbar_arrive(ring.empty());
        ++ring.c;
        left -= (uint64_t)n;
    }
    return st.E;
}

// Blocks of `chains` chain warps (32 walkers each), then `gens` (1 or 2) generator warps
// per chain warp.
template <int L, uint32_t TRIES>
__global__ void __launch_bounds__(kPairMaxThreads, 1) pair_kernel(const SweepArgs a, const __grid_constant__ LaunchPlan plan,
                                                                  const int chains, const int gens, const bool record)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if (a.skip && *a.skip)   // an iteration run on the device has finished
        return;
    constexpr int N = L * L;
    constexpr int NB = N + 1;
    constexpr int STRIDE = kTableStride;
    const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool chain = warp < chains;
    const int pair = chain ? warp : (warp - chains) % chains;
    uint32_t *sTab = reinterpret_cast<uint32_t *>(smem);
    unsigned char *sRows = smem + align_up((size_t)(NB + 1) * STRIDE * 4, 16);
    unsigned char *sRing = sRows + (size_t)(32 * chains) * SmemRows<L>::bytes_per_walker() + (size_t)pair * PairRing<L, TRIES>::bytes();
    const SmemRows<L> rows{sRows, 32 * chains, 32 * pair + lane};
    PairRing<L, TRIES> ring;
    ring.bars = (uint32_t)__cvta_generic_to_shared(sRing);
    ring.base = ring.bars + 32u + 16u * (uint32_t)lane;
    const int64_t w = ((int64_t)blockIdx.x * chains + pair) * 32 + lane;
    const bool pair_on = w - lane < a.W;   // uniform over the pair's warps
    bool active = chain && w < a.W;
    const bool warp_full = w - lane + 32 <= a.W && a.W % 16 == 0;
    if (chain && lane < 4)
        mbar_init(ring.bars + 8u * (uint32_t)lane, 1u);

    load_table<NB, NB + 1, 0, STRIDE>(sTab, a.table, tid, nthr);
    int32_t e = 0;
    if (chain && pair_on) {
        // Eight rows in flight: one warp per SM has only its own loads to hide their latency
        // behind, and in this kernel the registers are free (L = 48, 1024 walkers, spins as
        // bytes: 45 us of a launch that are not sweeps with four, 32 with eight).
        load_lattice<L, (L % 8 == 0 ? 8 : 4)>(a, rows, w, active, warp_full, lane);
        if (active) {
            e = a.energy[w];
            if (e < 0 || e > N) {
                atomicOr(a.err, kErrEnergyRange);
                active = false;
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    const uint32_t tbase = (uint32_t)__cvta_generic_to_shared(sTab);
    uint32_t E = tbase + (active ? (uint32_t)e : (uint32_t)NB) * (4u * STRIDE);
    const bool fused = record && a.n_therm > 0;   // uniform over the launch
#pragma unroll 1
    for (int phase = fused ? 0 : 1; phase < 2; ++phase) {
        const RowPlan &p = plan.phase[phase];
        if (pair_on) {
            const PhiloxKeys pk = make_keys(a.seed, a.walker0 + (uint32_t)w, p.c1);
            if (!chain) {
                ring.generate(p.blk1, p.rows, pk, (warp - chains) / chains, gens, lane);
            } else {
#pragma unroll 1
                for (int part = 0; part < 3; ++part) {
                    if (part == 1) {
                        if (p.rows > 0)
                            E = ring_rows<L, STRIDE, TRIES>(rows, E, p.y1, p.rows, ring, lane);
                    } else {
                        const int x0 = part == 0 ? p.x0 : 0, x1 = part == 0 ? p.x0_end : p.tail;
                        if (x0 < x1)
                            E = cut_row<L, STRIDE>(rows, E, part == 0 ? p.y0 : p.y2, x0, x1, part == 0 ? p.blk0 : p.blk2, pk);
                    }
                }
            }
        }
        if (phase == 0) {
            __syncthreads();
            for (int i = tid; i < NB; i += nthr)
                sTab[i * STRIDE + kHistSlot] = 0u;
            __syncthreads();
        }
    }
    if (active) {
        e = (int32_t)((E - tbase) / (4u * STRIDE));
        if (E < tbase || e > N || (E - tbase) % (4u * STRIDE) != 0u)   // corrupted energy address
            atomicOr(a.err, kErrEnergyRange);
    }
    if (!ring.ok)
        atomicOr(a.err, kErrSyncTimeout);
    __syncthreads();
    if (record)
        for (int i = tid; i < NB; i += nthr) {
            const uint32_t v = sTab[i * STRIDE + kHistSlot];
            if (v)
                atomicAdd(&a.hist[i], (unsigned long long)v);
        }
    if (chain && pair_on)
        store_lattice<L>(a, rows, w, active, warp_full, lane);
    if (active)
        a.energy[w] = e;
}

template <int L, uint32_t TRIES = kPairWaitTries>
cudaError_t launch_pair_t(const SweepArgs &a, int chains, bool record, cudaStream_t s)
{
    const size_t smem = align_up((size_t)(L * L + 2) * kTableStride * 4, 16) +
                        (size_t)chains * (32 * SmemRows<L>::bytes_per_walker() + PairRing<L, TRIES>::bytes());
    static std::atomic<uint64_t> allowed{0};
    const cudaError_t err = allow_smem(pair_kernel<L, TRIES>, allowed);
    if (err != cudaSuccess)
        return err;
    LaunchPlan plan;
    plan.phase[0] = row_plan(L, a.t0, a.n_therm);
    plan.phase[1] = row_plan(L, a.t0 + a.n_therm, a.n);
    const int gens = chains == 1 ? 2 : 1;
    const int64_t blocks = (a.W + 32 * chains - 1) / (32 * chains);
    pair_kernel<L, TRIES><<<(unsigned)blocks, 32 * chains * (1 + gens), smem, s>>>(a, plan, chains, gens, record);
    return cudaGetLastError();
}

}  // namespace
}  // namespace muca
