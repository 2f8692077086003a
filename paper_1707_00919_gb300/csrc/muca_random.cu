// muca_random.cu - updates in random shared site order, the paper's scheme of Sec. 2.3:
// one random site sequence drives all walkers and each walker draws its acceptance from
// its own stream.  The site of attempt t is floor(u N / 2^32) with u the Philox word t & 3
// of counter (t >> 2, 0xFFFFFFFF, tag 2); the acceptance word is the one of typewriter
// order (tag 0, the walker's counter).
//
// One thread runs one walker.  All walkers of a warp visit the same site, so a warp keeps
// its 32 lattices as one word per site (bit = lane), and the neighbour counts of up to 32
// attempts, a window, are formed together: one attempt per lane, the 32 walkers as the bits
// of its words, so that a count costs a fraction of an instruction instead of three row
// loads, a rotation and three population counts (quarter-rate) per walker.  A window ends
// before the first group of four (one Philox block) with a site that coincides with or
// neighbours an earlier site of the window: until then its counts stand.  A group with such
// a pair inside runs attempt by attempt.
//
// What bounds it at one warp per SM sub-partition: 39 instructions per attempt (18 ALU, 14
// multiply pipe, of them 4.6 wide) on one warp's issue, and the latency of a window's
// preparation (about 17 attempts at L = 32, 30 at L = 64, 7 at L = 16).  Measured, us per
// sweep, before and after: L = 32, 16384 walkers 74.6 -> 54.8 (48 640 walkers 120 -> 105);
// L = 64, 32 768 walkers 678 -> 257; L = 16, 4096 walkers 22.4 -> 19.4; L = 8 7.4 -> 6.75.
#include <cstdint>

#include "muca_device.cuh"

namespace muca {
namespace {

constexpr int kChunk = 512;        // attempts whose sites are drawn at once by the block
constexpr int kWindow = 32;        // attempts of a window at most
constexpr int kRandStride = 6;     // words per table row: thresholds of k = 0..4, histogram count
constexpr int kRandGuard = 2;      // zero rows below energy 0 and above N (speculative loads)
// Rows of the table: guards, energies 0..N, guards, the row of zeros for lanes without a
// walker, guards.
__host__ __device__ constexpr int random_rows(int N) { return N + 1 + 3 * kRandGuard + 1; }
// Per warp: the count records of a window (one byte per walker, and four records read ahead).
constexpr int kRecBytes = (kWindow + 4) * 32;

__host__ __device__ constexpr size_t random_table_bytes(int N) { return align_up((size_t)random_rows(N) * kRandStride * 4, 16); }

size_t random_smem_bytes(int L, int wpb)
{
    const int N = L * L;
    return random_table_bytes(N) + (size_t)kChunk * 16 + kChunk + (size_t)(kChunk + kWindow) * 2 + (size_t)(wpb / 32) * (kRecBytes + (size_t)N * 4);
}

// A site of the sequence: the byte offsets of its word and of its neighbours' words, left
// and right, above and below.
__device__ __forceinline__ uint4 site_record(uint32_t i, int L)
{
    const uint32_t y = i / (uint32_t)L, x = i - y * (uint32_t)L, n = (uint32_t)L;
    const uint32_t l = x == 0 ? i + n - 1 : i - 1, r = x == n - 1 ? i + 1 - n : i + 1;
    const uint32_t u = y == 0 ? i + n * (n - 1) : i - n, d = y == n - 1 ? i - n * (n - 1) : i + n;
    return make_uint4(4u * i, 4u * l | (4u * r << 16), 4u * u | (4u * d << 16), 0u);
}

// 32 x 32 bit transpose across a warp: lane i bit j <-> lane j bit i.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t m, int lane)
{
    const uint32_t part = __shfl_xor_sync(0xFFFFFFFFu, m, 16);
    m = (lane & 16) ? ((m & 0xFFFF0000u) | (part >> 16)) : ((m & 0x0000FFFFu) | (part << 16));
    return warp_swap_low4(m, lane);
}

__device__ __forceinline__ uint32_t lds_u8(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

__global__ void __launch_bounds__(256, 1) random_sweep_kernel(const SweepArgs a, const bool record)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if (a.skip && *a.skip)   // an iteration run on the device has finished
        return;
    const int L = a.L;
    const int N = L * L;
    const int wpb = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t *sT = reinterpret_cast<uint32_t *>(smem);
    uint4 *sSite = reinterpret_cast<uint4 *>(smem + random_table_bytes(N));
    uint16_t *sIdx = reinterpret_cast<uint16_t *>(sSite + kChunk) + kWindow;   // site indices, after a window of none
    uint8_t *sDist = reinterpret_cast<uint8_t *>(sIdx + kChunk);   // to the latest conflicting attempt, 0: none in reach
    unsigned char *sRec = sDist + kChunk + (size_t)warp * kRecBytes;
    uint32_t *lat = reinterpret_cast<uint32_t *>(sDist + kChunk + (size_t)(wpb / 32) * kRecBytes) + (size_t)warp * N;
    const int64_t w = (int64_t)blockIdx.x * wpb + tid;
    const int64_t w0 = w - lane;
    const bool warp_on = w0 < a.W;   // uniform over the warp
    bool active = w < a.W;

    for (int i = tid; i < random_rows(N) * kRandStride; i += wpb) {
        const int r = i / kRandStride, k = i - r * kRandStride;
        const int e = r - kRandGuard;
        sT[i] = (k < 5 && e >= 0 && e <= N) ? a.table[e * 5 + k] : 0u;
    }
    for (int i = lane; i < kRecBytes / 4; i += 32)
        reinterpret_cast<uint32_t *>(sRec)[i] = 0u;
    if (tid < kWindow)
        sIdx[tid - kWindow] = 0xFFFFu;
    int32_t e = 0;
    // the warp's 32 bytes per site are whole and 16-byte aligned: uniform
    const bool whole = a.layout == MUCA_LAYOUT_INT8 && w0 + 32 <= a.W && a.W % 16 == 0;
    if (warp_on) {
        if (a.layout == MUCA_LAYOUT_PACKED) {
            // a walker's row word (its bits are sites) transposed into the sites' words
            for (int y = 0; y < L; ++y)
                for (int half = 0; half * 32 < L; ++half) {
                    uint32_t m = 0;
                    if (active) {
                        if (L <= 32)
                            m = reinterpret_cast<const uint32_t *>(a.lattice)[(size_t)y * a.W + w];
                        else
                            m = (uint32_t)(reinterpret_cast<const unsigned long long *>(a.lattice)[(size_t)y * a.W + w] >> (32 * half));
                    }
                    m = warp_transpose(m, lane);
                    if (half * 32 + lane < L)
                        lat[y * L + half * 32 + lane] = m;
                }
        } else if (whole) {
            // one site per lane: its 32 walkers' signs
            const int8_t *g = reinterpret_cast<const int8_t *>(a.lattice) + w0;
#pragma unroll 4
            for (int i = lane; i < N; i += 32) {
                const uint4 *p = reinterpret_cast<const uint4 *>(g + (size_t)i * a.W);
                lat[i] = gather16(p[0]) | (gather16(p[1]) << 16);
            }
        } else {
            const int8_t *g = reinterpret_cast<const int8_t *>(a.lattice) + w;
            for (int i0 = 0; i0 < N; i0 += 16) {   // N is a multiple of 16
                int8_t v[16];
#pragma unroll
                for (int u = 0; u < 16; ++u)
                    v[u] = active ? g[(size_t)(i0 + u) * a.W] : (int8_t)1;
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const uint32_t m = __ballot_sync(0xFFFFFFFFu, v[u] < 0);
                    if (lane == u)
                        lat[i0 + u] = m;
                }
            }
        }
        if (active) {
            e = a.energy[w];
            if (e < 0 || e > N) {
                atomicOr(a.err, kErrEnergyRange);
                active = false;
            }
        }
    }
    constexpr uint32_t kRowBytes = 4u * kRandStride;
    const uint32_t tbase = (uint32_t)__cvta_generic_to_shared(sT) + kRandGuard * kRowBytes;
    // byte address of the current energy's row; lanes without a walker, or whose energy is
    // off the grid, sit on a row of zeros, where nothing is accepted
    uint32_t E = tbase + (active ? (uint32_t)e : (uint32_t)(N + 1 + kRandGuard)) * kRowBytes;
    const PhiloxKeys pk = make_keys(a.seed, a.walker0 + (uint32_t)w, (uint32_t)(a.t0 >> 34));
    // the lane's byte of record 0 (see the records below), the sites' words
    const uint32_t rec0 = (uint32_t)__cvta_generic_to_shared(sRec);
    const uint32_t rec_of_lane = rec0 + 8u * (uint32_t)(lane & 3) + ((uint32_t)lane & 4u) + (uint32_t)(lane >> 3);
    unsigned char *const latb = reinterpret_cast<unsigned char *>(lat);
    auto word = [&](uint32_t off) -> uint32_t & { return *reinterpret_cast<uint32_t *>(latb + off); };
    const uint64_t tend = a.t0 + a.n;
    for (uint64_t tc = a.t0; tc < tend;) {
        // attempts j0 .. m - 1 of the chunk that starts at the Philox block of tc
        const uint64_t tb = tc & ~3ull;
        const int j0 = (int)(tc - tb);
        const int m = tend - tb < (uint64_t)kChunk ? (int)(tend - tb) : kChunk;
        __syncthreads();   // the previous chunk's sites are consumed (and the setup done)
        for (int q = tid; 4 * q < m; q += wpb) {
            const uint64_t blk = (tb >> 2) + (uint64_t)q;
            const uint4 r = philox4x32_10(make_uint4((uint32_t)blk, (uint32_t)(blk >> 32), kSharedStream, kTagSite),
                                          (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
            const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const uint32_t i = __umulhi(u[v], (uint32_t)N);
                sSite[4 * q + v] = site_record(i, L);
                sIdx[4 * q + v] = 4 * q + v >= j0 ? (uint16_t)(4u * i) : (uint16_t)0xFFFFu;
            }
        }
        __syncthreads();
        // the distance to the latest earlier attempt (within a window's reach) whose site is
        // this attempt's or a neighbour of it
        for (int j = tid; j < m; j += wpb) {
            const uint4 n = sSite[j];
            const uint32_t nl = n.y & 0xFFFFu, nr = n.y >> 16, nu = n.z & 0xFFFFu, nd = n.z >> 16;
            int dist = 0;
#pragma unroll
            for (int d = kWindow - 1; d > 0; --d) {
                const uint32_t s = sIdx[j - d];
                dist = (s == n.x || s == nl || s == nr || s == nu || s == nd) ? d : dist;
            }
            sDist[j] = (uint8_t)dist;
        }
        __syncthreads();
        if (warp_on) {
            // one attempt on the current words
            auto single = [&](int j, uint32_t r) {
                const uint4 n = sSite[j];
                const uint32_t c = word(n.x);
                const uint32_t k = (((c ^ word(n.y & 0xFFFFu)) >> lane) & 1u) + (((c ^ word(n.y >> 16)) >> lane) & 1u) +
                                   (((c ^ word(n.z & 0xFFFFu)) >> lane) & 1u) + (((c ^ word(n.z >> 16)) >> lane) & 1u);
                const bool acc = r < lds_u32(E + 4u * k);
                E = acc ? E + (2u - k) * kRowBytes : E;
                const uint32_t flips = __ballot_sync(0xFFFFFFFFu, acc);
                if (lane == 0)
                    word(n.x) = c ^ flips;
                hist_add_one(E);
                __syncwarp();
            };
            // the window from attempt j, one attempt per lane: its sites and its groups of four
            struct Window {
                uint4 n;
                int groups;
            };
            auto window = [&](int j) {
                Window v;
                const int most = m - j < kWindow ? (m - j) & ~3 : kWindow;
                const bool in = lane < most;
                v.n = in ? sSite[j + lane] : make_uint4(0u, 0u, 0u, 0u);
                const int dist = in ? (int)sDist[j + lane] : 0;
                const uint32_t stop = __ballot_sync(0xFFFFFFFFu, dist != 0 && dist <= lane);
                v.groups = (stop ? __ffs((int)stop) - 1 : most) >> 2;
                return v;
            };
            uint32_t b = (uint32_t)(tb >> 2);   // Philox block of attempt j
            uint4 next = block_words(block_head(b, pk), pk);
            int j = 0;
            if (j0 > 0) {   // the head of a launch that starts inside a Philox block
                const uint32_t q[4] = {next.x, next.y, next.z, next.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (u >= j0 && u < m)
                        single(u, q[u]);
                next = block_words(block_head(++b, pk), pk);
                j = 4;
            }
            Window win = window(j);
            while (m - j >= 4) {
                const int groups = win.groups;
                if (groups == 0) {
                    const uint4 q = next;
                    next = block_words(block_head(++b, pk), pk);
                    single(j, q.x);
                    single(j + 1, q.y);
                    single(j + 2, q.z);
                    single(j + 3, q.w);
                    j += 4;
                    win = window(j);
                    continue;
                }
                // counts of the lane's attempt, bit-sliced over the warp's walkers
                const uint4 n = win.n;
                const uint32_t c = word(n.x);
                const uint32_t x0 = c ^ word(n.y & 0xFFFFu), x1 = c ^ word(n.y >> 16), x2 = c ^ word(n.z & 0xFFFFu),
                               x3 = c ^ word(n.z >> 16);
                const uint32_t p = x0 ^ x1 ^ x2, q3 = (x0 & x1) | (x2 & (x0 | x1)), both = p & x3;
                const uint32_t k0 = p ^ x3, k1 = q3 ^ both, k2 = q3 & both;
                // its record: four times the count of walker 8 h + 4 v + r in byte h of word 2 r + v
                uint32_t rec[8];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t nib = ((k0 >> r) & 0x11111111u) | (((k1 >> r) & 0x11111111u) << 1) | (((k2 >> r) & 0x11111111u) << 2);
                    rec[2 * r] = (nib << 2) & 0x3C3C3C3Cu;
                    rec[2 * r + 1] = (nib >> 2) & 0x3C3C3C3Cu;
                }
                uint4 *out = reinterpret_cast<uint4 *>(sRec + 32 * lane);
                out[0] = make_uint4(rec[0], rec[1], rec[2], rec[3]);
                out[1] = make_uint4(rec[4], rec[5], rec[6], rec[7]);
                __syncwarp();
                // decisions, the two threshold candidates of each attempt loaded two ahead
                uint32_t kk[6];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    kk[u] = lds_u8(rec_of_lane + 32u * (uint32_t)u);
                uint32_t Eacc = E + 2u * kRowBytes - kRandStride * kk[0];
                uint32_t T0n = lds_u32(E + kk[0]), T1n = T0n;
                uint32_t T0nn = lds_u32(E + kk[1]), T1nn = lds_u32(Eacc + kk[1]);
                bool prev = false;
                uint32_t flips = 0u;
                uint32_t at = rec_of_lane + 128u;
#pragma unroll 1
                for (int g = 0; g < groups; ++g) {
                    const uint4 qg = next;
                    next = block_words(block_head(++b, pk), pk);
                    // the next group's counts (past the window: unused)
                    kk[4] = lds_u8(at);
                    kk[5] = lds_u8(at + 32u);
                    const uint32_t k6 = lds_u8(at + 64u), k7 = lds_u8(at + 96u);
                    at += 128u;
                    const uint32_t words[4] = {qg.x, qg.y, qg.z, qg.w};
                    uint32_t nib = 0u;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t T = prev ? T1n : T0n;
                        const bool acc = words[u] < T;
                        E = acc ? Eacc : E;
                        nib |= acc ? 1u << u : 0u;
                        hist_add_one(E);
                        Eacc = E + 2u * kRowBytes - kRandStride * kk[u + 1];
                        T0n = T0nn;
                        T1n = T1nn;
                        T0nn = lds_u32(E + kk[u + 2]);
                        T1nn = lds_u32(Eacc + kk[u + 2]);
                        prev = acc;
                    }
                    flips |= nib << (4 * g);
                    kk[0] = kk[4];
                    kk[1] = kk[5];
                    kk[2] = k6;
                    kk[3] = k7;
                }
                // the flips back to one attempt per lane, into its site's word
                flips = warp_transpose(flips, lane);
                if (lane < 4 * groups)
                    word(n.x) = c ^ flips;
                __syncwarp();
                j += 4 * groups;
                win = window(j);
            }
            if (j < m) {   // the tail of a launch that ends inside a Philox block
                const uint32_t q[4] = {next.x, next.y, next.z, next.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (j + u < m)
                        single(j + u, q[u]);
            }
        }
        tc = tb + (uint64_t)m;
    }
    if (active) {
        e = (int32_t)((E - tbase) / kRowBytes);
        if (E < tbase || e > N || (E - tbase) % kRowBytes != 0u)   // corrupted energy address
            atomicOr(a.err, kErrEnergyRange);
    }
    __syncthreads();
    if (record)
        for (int i = tid; i <= N; i += wpb) {
            const uint32_t v = sT[(i + kRandGuard) * kRandStride + 5];
            if (v)
                atomicAdd(&a.hist[i], (unsigned long long)v);
        }
    // a walker whose energy is off the grid kept its lattice unchanged
    if (warp_on) {
        if (a.layout == MUCA_LAYOUT_PACKED) {
            for (int y = 0; y < L; ++y) {
                const uint32_t lo = warp_transpose(lane < L ? lat[y * L + lane] : 0u, lane);
                if (L <= 32) {
                    if (w < a.W)
                        reinterpret_cast<uint32_t *>(a.lattice)[(size_t)y * a.W + w] = lo;
                } else {
                    const uint32_t hi = warp_transpose(32 + lane < L ? lat[y * L + 32 + lane] : 0u, lane);
                    if (w < a.W)
                        reinterpret_cast<unsigned long long *>(a.lattice)[(size_t)y * a.W + w] =
                            ((unsigned long long)hi << 32) | lo;
                }
            }
        } else if (whole) {
            int8_t *g = reinterpret_cast<int8_t *>(a.lattice) + w0;
            for (int i = lane; i < N; i += 32) {
                uint4 *p = reinterpret_cast<uint4 *>(g + (size_t)i * a.W);
                const uint32_t v = lat[i];
                p[0] = scatter16(v & 0xFFFFu);
                p[1] = scatter16(v >> 16);
            }
        } else if (w < a.W) {
            int8_t *g = reinterpret_cast<int8_t *>(a.lattice) + w;
            for (int i = 0; i < N; ++i)
                g[(size_t)i * a.W] = ((lat[i] >> lane) & 1u) ? (int8_t)-1 : (int8_t)1;
        }
    }
    if (active)
        a.energy[w] = e;
}

cudaError_t launch_random_t(const SweepArgs &a, int wpb, bool record, cudaStream_t s)
{
    static std::atomic<uint64_t> allowed{0};
    const cudaError_t err = allow_smem(random_sweep_kernel, allowed);
    if (err != cudaSuccess)
        return err;
    const int64_t blocks = (a.W + wpb - 1) / wpb;
    random_sweep_kernel<<<(unsigned)blocks, wpb, random_smem_bytes(a.L, wpb), s>>>(a, record);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_random_sweep(const SweepArgs &a, int walkers_per_block, bool record, cudaStream_t s)
{
    if (a.n == 0 || a.W == 0)
        return cudaSuccess;
    // the instance's block size (one warp per SM sub-partition where the walker count
    // allows), else the largest block of whole warps whose words fit next to the table and
    // the sites (the walker-to-thread mapping does not affect the result)
    const size_t limit = sweep_smem_limit();
    int wpb = walkers_per_block >= 32 && walkers_per_block <= 256 ? walkers_per_block : 256;
    while (wpb > 32 && random_smem_bytes(a.L, wpb) > limit)
        wpb -= 32;
    if (random_smem_bytes(a.L, wpb) > limit)
        return cudaErrorInvalidConfiguration;
    // the kernel keeps Philox counter word 1 (t >> 34) fixed within a launch: a range that
    // crosses a multiple of 2^34 runs in parts
    SweepArgs part = a;
    for (uint64_t left = a.n; left > 0; left -= part.n, part.t0 += part.n) {
        part.n = same_word1(part.t0, left);
        const cudaError_t err = launch_random_t(part, wpb, record, s);
        if (err != cudaSuccess)
            return err;
    }
    return cudaSuccess;
}

}  // namespace muca
