// muca_device.cuh - device code of the sweep kernels, shared by the per-L translation units
// (muca_full_L.cu), the batched kernels (muca_batch.cu, muca_noalloc.cu), the kernel of the
// random site order (muca_random.cu) and those around the sweeps (muca_kernels.cu).  Parallel multicanonical 2D Ising update of Gross,
// Zierenberg, Weigel, Janke (arXiv:1707.00919), Sec. 2.3.
#pragma once

#include <cstddef>
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "../../include/muca.h"
#include "muca_internal.h"

namespace muca {
namespace {

__host__ __device__ constexpr size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

template <typename RowT>
__device__ __forceinline__ uint32_t bit_at(RowT w, int x)
{
    return (uint32_t)(w >> x) & 1u;
}

// ---------------------------------------------------------------------------------
// Sweep kernels in typewriter order, specialised on L (every multiple of 4 up to 64).  A
// launch covers any attempt range; its whole rows run unrolled, so bit positions and neighbour columns are
// compile-time constants; the Philox round keys are computed once per thread.
//
// Row representation: the rows above (U), at (C) and below (D) the current row are held
// as nibble words, eight spins per 32-bit register, one spin in bit 0 of each 4-bit
// field (1 = spin down).  Field-parallel arithmetic gives for all sites of a row at once
//   kb = [s != s_up] + [s != s_down] + [s != s_right]    h0 = [s != s_left]
// with the original spins, so the antiparallel count of site x is k0 = kb + h0 if the
// previous attempt (at x - 1) did not flip, else k1 = kb + 1 - h0.  Site 0's left
// neighbour is site L-1 of the same row, not yet visited, so k1 = k0 there; site L-1's
// right neighbour is site 0, so its counts move by one if site 0 flipped.
//
// Shared-memory table: one 28-byte row per energy index e, words 0..4 the acceptance
// thresholds T[e][k], word 5 the block's histogram count of e, word 6 padding (a stride
// of 7 words spreads the rows over all 32 banks).  The energy is carried as the byte
// address E of its row, so a threshold is at E + 4k, the histogram word at E + 20, and
// an accepted flip moves E by 28 (2 - k).  The batched kernel's L = 64 items use 6-word
// rows instead (24 bytes), which lets 256 walkers share an SM with the 4097-row table.
//
// Latency: the threshold an attempt needs depends on whether the previous attempt
// flipped (through E and through k).  Both candidates are loaded two attempts ahead and
// the right one is picked once the previous decision is known, which takes the shared-
// memory latency off the attempt-to-attempt dependency chain (a select and a compare).
// ---------------------------------------------------------------------------------
template <int L>
struct RowOf {
    using type = typename std::conditional<(L <= 32), uint32_t, unsigned long long>::type;
};

// Nibble words of a row.  With L = 4 mod 8 the last word holds four spins, its upper
// fields zero.
__host__ __device__ constexpr int row_words(int L) { return (L + 7) / 8; }


// Philox4x32-10 of Salmon et al. (SC'11), the generator of Sec. 2.3, on counter c with
// key (k0, k1).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        if (round > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t lo0 = 0xD2511F53u * c.x;
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// Counter tags of the Philox streams: updates, initial spins, random site order.
constexpr uint32_t kTagMetropolis = 0u;
constexpr uint32_t kTagInit = 1u;
constexpr uint32_t kTagSite = 2u;
constexpr uint32_t kSharedStream = 0xFFFFFFFFu;   // walker word of the site stream

// Round keys of the seed, and what depends only on the walker and on counter word 1 = c1:
// with tag word 0, round 0 turns (c0, c1, walker, 0) into
// (hi_w ^ c1 ^ k0, lo_w, hi(M0 c0) ^ k1, lo(M0 c0)), so round 1's product of its first word
// is fixed for as long as c1 is (2^34 attempts).
struct PhiloxKeys {
    uint32_t k0[10], k1[10];   // round keys
    uint32_t lo_w;             // low half of round 0's product of the walker word
    uint32_t r1_hi, r1_lo;     // round 1's product of the first word, (hi_w ^ c1 ^ k0) * M0
};

__device__ __forceinline__ PhiloxKeys make_keys(uint64_t seed, uint32_t walker, uint32_t c1)
{
    PhiloxKeys p;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        p.k0[r] = (uint32_t)seed + (uint32_t)r * 0x9E3779B9u;
        p.k1[r] = (uint32_t)(seed >> 32) + (uint32_t)r * 0xBB67AE85u;
    }
    const unsigned long long pw = (unsigned long long)0xCD9E8D57u * walker;
    p.lo_w = (uint32_t)pw;
    const unsigned long long p1 = (unsigned long long)0xD2511F53u * ((uint32_t)(pw >> 32) ^ c1 ^ p.k0[0]);
    p.r1_hi = (uint32_t)(p1 >> 32);
    p.r1_lo = (uint32_t)p1;
    return p;
}

// Rounds 0 and 1 of block c0 as far as they are the same for every walker: two of the wide
// multiplies.  The walkers' own part of round 1 is two exclusive-ors (block_words).
__device__ __forceinline__ uint3 block_head(uint32_t c0, const PhiloxKeys &p)
{
    const unsigned long long q = (unsigned long long)0xD2511F53u * c0;
    const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * ((uint32_t)(q >> 32) ^ p.k1[0]);
    return make_uint3((uint32_t)(p1 >> 32) ^ p.k0[1], (uint32_t)p1, (uint32_t)q ^ p.k1[1]);
}

// Philox4x32-10 on counter (c0, c1, walker, tag 0) from the block's head: 16 wide
// multiplies, each giving both halves of a product.
__device__ __forceinline__ uint4 philox_walker_c1(uint3 head, const PhiloxKeys &p)
{
    uint32_t x0 = head.x ^ p.lo_w, x1 = head.y, x2 = head.z ^ p.r1_hi, x3 = p.r1_lo;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * x0;
        const unsigned long long pp = (unsigned long long)0xCD9E8D57u * x2;
        const uint32_t n0 = (uint32_t)(pp >> 32) ^ x1 ^ p.k0[r];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ x3 ^ p.k1[r];
        x0 = n0;
        x1 = (uint32_t)pp;
        x2 = n2;
        x3 = (uint32_t)p0;
    }
    return make_uint4(x0, x1, x2, x3);
}

// The same, clamped to 0xFFFFFFFE so that "r < T" also accepts every attempt when
// T = 0xFFFFFFFF.
__device__ __forceinline__ uint4 block_words(uint3 head, const PhiloxKeys &k)
{
    const uint4 rw = philox_walker_c1(head, k);
    return make_uint4(min(rw.x, 0xFFFFFFFEu), min(rw.y, 0xFFFFFFFEu), min(rw.z, 0xFFFFFFFEu), min(rw.w, 0xFFFFFFFEu));
}

// Sign bits of four int8 spins (-1 = 0xFF, +1 = 0x01) as a nibble.
__device__ __forceinline__ uint32_t gather_signs(uint32_t v) { return ((v & 0x80808080u) * 0x00204081u) >> 28; }

// Nibble of down-spin bits to four int8 spins.
__device__ __forceinline__ uint32_t spread_signs(uint32_t n)
{
    return 0x01010101u | (((n * 0x00204081u) & 0x01010101u) * 0xFEu);
}

// Butterfly stages 8, 4, 2, 1 of a 32x32 bit transpose across a warp: swaps bits 0-3 of
// the lane index with bits 0-3 of the bit position (bit 4 of each stays in place).
__device__ __forceinline__ uint32_t warp_swap_low4(uint32_t m, int lane)
{
    const uint32_t masks[4] = {0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int s = 8 >> i;
        const uint32_t part = __shfl_xor_sync(0xFFFFFFFFu, m, s);
        m = (lane & s) ? ((m & ~masks[i]) | ((part >> s) & masks[i])) : ((m & masks[i]) | ((part & masks[i]) << s));
    }
    return m;
}

// Sign bits of 16 int8 spins as a 16-bit mask (bit i = byte i).
__device__ __forceinline__ uint32_t gather16(uint4 u)
{
    return gather_signs(u.x) | (gather_signs(u.y) << 4) | (gather_signs(u.z) << 8) | (gather_signs(u.w) << 12);
}

// Bit rows of the warp's 32 walkers from the int8 [site][walker] layout, R rows at a
// time so that their loads are in flight together; lane j receives walker w0 + j.
// Lanes 2p and 2p + 1 read the two halves of one site's 32 walker bytes (sites 32h + p and
// 32h + 16 + p of row half h), so each load instruction covers 16 whole 32-byte sectors.
// Lane 2p + q then holds bit 16r + s = spin of walker 16q + s at site 32h + 16r + p; a
// lane shuffle to lane 16q + p and four butterfly stages (lane bits 0-3 against bit
// positions 0-3) leave in lane 16q + s the spins of walker 16q + s, bit x at site 32h + x.
// All 32 walkers must exist and W % 16 == 0.
template <int L, int R, typename RowT>
__device__ __forceinline__ void warp_load_rows_int8(const int8_t *g, int64_t W, int64_t w0, int y0, int lane,
                                                    RowT (&out)[R])
{
    constexpr int HALVES = (L + 31) / 32;
    const int p = lane >> 1, q = lane & 1;
    uint4 a[R][HALVES], b[R][HALVES];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int half = 0; half < HALVES; ++half) {
            const int xa = half * 32 + p, xb = xa + 16;
            const int8_t *row = g + (size_t)((y0 + r) * L) * (size_t)W + (size_t)w0 + 16 * q;
            a[r][half] = xa < L ? *reinterpret_cast<const uint4 *>(row + (size_t)xa * (size_t)W) : make_uint4(0, 0, 0, 0);
            b[r][half] = xb < L ? *reinterpret_cast<const uint4 *>(row + (size_t)xb * (size_t)W) : make_uint4(0, 0, 0, 0);
        }
    const int src = 2 * (lane & 15) + (lane >> 4);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        RowT row = 0;
#pragma unroll
        for (int half = 0; half < HALVES; ++half) {
            uint32_t m = gather16(a[r][half]) | (gather16(b[r][half]) << 16);
            m = __shfl_sync(0xFFFFFFFFu, m, src);
            m = warp_swap_low4(m, lane);
            row |= (RowT)m << (32 * half);
        }
        out[r] = row;
    }
}

// 16 spins of a 16-bit mask (bit i = byte i, set = -1) as int8.
__device__ __forceinline__ uint4 scatter16(uint32_t h)
{
    return make_uint4(spread_signs(h & 15u), spread_signs((h >> 4) & 15u), spread_signs((h >> 8) & 15u),
                      spread_signs((h >> 12) & 15u));
}

// The inverse of warp_load_rows_int8 for one row: lane j holds walker w0 + j's bits.
template <int L, typename RowT>
__device__ __forceinline__ void warp_store_row_int8(int8_t *g, int64_t W, int64_t w0, int y, int lane, RowT r)
{
    const int p = lane >> 1, q = lane & 1;
    const int src = 16 * q + p;
#pragma unroll
    for (int half = 0; half < (L + 31) / 32; ++half) {
        uint32_t m = warp_swap_low4((uint32_t)(r >> (32 * half)), lane);
        m = __shfl_sync(0xFFFFFFFFu, m, src);
        const int xa = half * 32 + p, xb = xa + 16;
        int8_t *row = g + (size_t)(y * L) * (size_t)W + (size_t)w0 + 16 * q;
        if (xa < L)
            *reinterpret_cast<uint4 *>(row + (size_t)xa * (size_t)W) = scatter16(m & 0xFFFFu);
        if (xb < L)
            *reinterpret_cast<uint4 *>(row + (size_t)xb * (size_t)W) = scatter16(m >> 16);
    }
}

// Eight bits -> eight nibbles (bit i to bit 4i), and back.
__device__ __forceinline__ uint32_t spread8(uint32_t b)
{
    uint32_t x = b & 0xFFu;
    x = (x | (x << 12)) & 0x000F000Fu;
    x = (x | (x << 6)) & 0x03030303u;
    x = (x | (x << 3)) & 0x11111111u;
    return x;
}

__device__ __forceinline__ uint32_t pack8(uint32_t x)
{
    x &= 0x11111111u;
    x = (x | (x >> 3)) & 0x03030303u;
    x = (x | (x >> 6)) & 0x000F000Fu;
    x = (x | (x >> 12)) & 0xFFu;
    return x;
}

template <int L>
__device__ __forceinline__ void to_nibbles(typename RowOf<L>::type r, uint32_t (&n)[row_words(L)])
{
#pragma unroll
    for (int i = 0; i < row_words(L); ++i)
        n[i] = spread8((uint32_t)(r >> (8 * i)));
}

template <int L>
__device__ __forceinline__ typename RowOf<L>::type from_nibbles(const uint32_t (&n)[row_words(L)])
{
    using RowT = typename RowOf<L>::type;
    RowT r = 0;
#pragma unroll
    for (int i = 0; i < row_words(L); ++i)
        r |= (RowT)pack8(n[i]) << (8 * i);
    return r;
}

// Row storage in shared memory during a launch.  L <= 32: nibble words,
// [row][walker][word], read and written without conversion.  L > 32: bit words
// [row][walker] (a nibble copy would not fit next to the table), converted per row.
template <int L>
struct SmemRows {
    static constexpr bool kNibbles = (L <= 32);
    static constexpr int NW = row_words(L);
    using RowT = typename RowOf<L>::type;
    __host__ __device__ static constexpr size_t bytes_per_walker()
    {
        return kNibbles ? (size_t)L * NW * 4 : (size_t)L * sizeof(RowT);
    }

    unsigned char *base;
    int wpb, tid;

    __device__ __forceinline__ void load(int y, uint32_t (&n)[NW]) const
    {
        if (kNibbles) {
            const uint32_t *p = reinterpret_cast<const uint32_t *>(base) + ((size_t)y * wpb + tid) * NW;
#pragma unroll
            for (int i = 0; i < NW; ++i)
                n[i] = p[i];
        } else {
            to_nibbles<L>(reinterpret_cast<const RowT *>(base)[(size_t)y * wpb + tid], n);
        }
    }
    __device__ __forceinline__ void store(int y, const uint32_t (&n)[NW]) const
    {
        if (kNibbles) {
            uint32_t *p = reinterpret_cast<uint32_t *>(base) + ((size_t)y * wpb + tid) * NW;
#pragma unroll
            for (int i = 0; i < NW; ++i)
                p[i] = n[i];
        } else {
            reinterpret_cast<RowT *>(base)[(size_t)y * wpb + tid] = from_nibbles<L>(n);
        }
    }
    __device__ __forceinline__ void store_bits(int y, RowT r) const
    {
        uint32_t n[NW];
        if (kNibbles) {
            to_nibbles<L>(r, n);
            store(y, n);
        } else {
            reinterpret_cast<RowT *>(base)[(size_t)y * wpb + tid] = r;
        }
    }
    __device__ __forceinline__ RowT load_bits(int y) const
    {
        if (kNibbles) {
            uint32_t n[NW];
            load(y, n);
            return from_nibbles<L>(n);
        }
        return reinterpret_cast<const RowT *>(base)[(size_t)y * wpb + tid];
    }
};

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// Histogram record of one attempt: one count for the post-decision energy, added to the
// histogram word (offset 20) of its table row.  Launches that do not record count too and
// leave the words behind: the reduction keeps the threshold loads of later attempts in
// place, and without it the compiler's order of the attempt loop measured 56 against 47
// cycles per attempt (one warp per sub-partition); a reduction under a predicate becomes
// a branch (58).
__device__ __forceinline__ void hist_add_one(uint32_t E)
{
    asm volatile("red.shared.add.u32 [%0+20], 1;" :: "r"(E));
}

// Random words of the current row, four attempts at a time.  The words of the row's first
// block are computed during the previous row (advance(), called during its last block)
// and kept in carry, so that a new row does not start by waiting for a whole Philox
// evaluation.
template <int L>
struct PhiloxSource {
    const PhiloxKeys &pk;
    uint32_t blk;            // counter word 0 of column 0's block
    uint4 carry;             // words of block blk, then of the next row's first block
    __device__ __forceinline__ static uint4 words(uint32_t b, const PhiloxKeys &k) { return block_words(block_head(b, k), k); }
    __device__ __forceinline__ uint4 get(int xb) const { return xb == 0 ? carry : words(blk + (uint32_t)(xb / 4), pk); }
    __device__ __forceinline__ void advance() { carry = words(blk + (uint32_t)(L / 4), pk); }
};

// The right and left neighbours' spins of every site of a row in its nibble fields.
template <int L>
__device__ __forceinline__ uint32_t right_of(const uint32_t (&C)[row_words(L)], int i)
{
    constexpr int NW = row_words(L);
    if (L % 8 != 0 && i == NW - 1)
        return (C[i] >> 4) | (C[0] << 12);
    return __funnelshift_r(C[i], C[(i + 1) % NW], 4);
}

template <int L>
__device__ __forceinline__ uint32_t left_of(const uint32_t (&C)[row_words(L)], int i)
{
    constexpr int NW = row_words(L);
    const uint32_t before = i > 0 ? C[i - 1] : L % 8 != 0 ? C[NW - 1] << 16 : C[NW - 1];
    return __funnelshift_l(before, C[i], 4);
}

// Antiparallel-neighbour counts of a row, original spins, as byte fields of four sites per
// word: word 2 i holds sites 8 i + 0, 2, 4, 6, word 2 i + 1 sites 8 i + 1, 3, 5, 7.  One
// dp4a (a four-byte dot product) adds a constant multiple of one site's count to an
// address: one instruction on the multiply pipe where a shift, a mask and an addition
// took three on the integer ALU, the pipe with the most instructions of this loop.
template <int L, bool SHIFTED = false>
struct RowCounts {
    static constexpr int NW = row_words(L);
    uint32_t k0[2 * NW];   // if the left neighbour did not flip
    uint32_t k1[2 * NW];   // if it did

    __device__ __forceinline__ RowCounts(const uint32_t (&U)[NW], const uint32_t (&C)[NW], const uint32_t (&D)[NW])
    {
        uint32_t hr[NW];   // right disagreements; shifted by a site they are the left ones
#pragma unroll
        for (int i = 0; i < NW; ++i)
            hr[i] = C[i] ^ right_of<L>(C, i);
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            const uint32_t kb = (U[i] ^ C[i]) + (D[i] ^ C[i]) + hr[i];
            const uint32_t h0 = SHIFTED ? left_of<L>(hr, i) : C[i] ^ left_of<L>(C, i);
            const uint32_t a = kb + h0, b = kb + 0x11111111u - h0;
            k0[2 * i] = a & 0x0F0F0F0Fu;
            k0[2 * i + 1] = (a >> 4) & 0x0F0F0F0Fu;
            k1[2 * i] = b & 0x0F0F0F0Fu;
            k1[2 * i + 1] = (b >> 4) & 0x0F0F0F0Fu;
        }
    }
    __device__ __forceinline__ uint32_t word0(int x) const { return k0[(x >> 3) * 2 + (x & 1)]; }
    __device__ __forceinline__ uint32_t word1(int x) const { return k1[(x >> 3) * 2 + (x & 1)]; }
    // Site L - 1's right neighbour is site 0: how its counts move if site 0 flips (minus
    // one if the two disagree, plus one if they agree), in its byte.
    static __device__ __forceinline__ uint32_t last_step(const uint32_t (&C)[NW])
    {
        constexpr int f = (L - 1) & 7, byte = 8 * (f >> 1);
        const bool differ = (((C[NW - 1] >> (4 * f)) ^ C[0]) & 1u) != 0u;
        return (differ ? 0xFFFFFFFFu : 1u) << byte;
    }
    __device__ __forceinline__ void add_to_last(uint32_t v)
    {
        k0[2 * (NW - 1) + 1] += v;
        k1[2 * (NW - 1) + 1] += v;
    }
};

// w with the bit flipped if acc: one predicated instruction instead of a select and an
// exclusive-or.
__device__ __forceinline__ uint32_t flip_if(uint32_t w, uint32_t bit, bool acc)
{
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p xor.b32 %0, %0, %2;\n\t}" : "+r"(w) : "r"(acc ? 1u : 0u), "r"(bit));
    return w;
}

// acc + m * (count of site x in its count word w), m in [-128, 127].
__device__ __forceinline__ uint32_t add_count(uint32_t w, int x, int m, uint32_t acc)
{
    return (uint32_t)__dp4a((int)w, (int)(((uint32_t)m & 0xFFu) << (8 * ((x & 7) >> 1))), (int)acc);
}

// ---------------------------------------------------------------------------------
// Continuous attempt stream over the whole rows of a range.  The two threshold
// candidates of every attempt are loaded two attempts ahead, across row ends as well:
// the first two sites of the next row have as neighbours the current row's first two
// sites (final after its attempts 0 and 1) and rows that the current row does not
// change, so their counts, and the candidates of the next row's attempts 0 and 1, are
// known during the current row's attempts L - 2 and L - 1.  A new row then starts with
// its first two decisions ready instead of waiting for its counts and loads.
//
// What bounds it: instruction issue.  A warp alone on its SM sub-partition issues one
// half-rate instruction per two cycles whatever its pipe (a wide multiply takes four), so
// at one warp the attempt costs twice its ALU and multiply instructions; with two warps
// the pipes overlap in part.  A chain warp whose words come from other warps (muca_pair.cuh)
// has half the instructions and is bound by the latency of its chain instead.  EARLY says
// how much is formed for both outcomes before a decision and selected by it: 0 nothing,
// 1 the row address if the next attempt flips, 2 also the address of its flipped candidate:
// each step shortens the chain and adds instructions.  The histogram's reduction comes
// after the loads, which it would delay.  Measured, us per sweep (EARLY 0 / 1 / 2):
//   L = 32, 16 384 walkers, one warp per sub-partition      24.7 / 24.4 / 24.5
//   L = 32, 38 912 walkers, two warps                       41.9 / 41.8 / 43.4
//   L = 64, 32 768 walkers, 1.75 warps                      166  / 168  / 176
//   L = 32, 4096 walkers, chain warps with generators       18.7 / 18.2 / 17.7
//   L = 64, 4096 walkers, the same                          74.8 / 74.2 / 72.1
//   L = 8, 128 walkers, the same                            1.23 / 1.16 / 1.28
// (side by side, before the lattices' and the table's loads took their present form: the
// chain warps of L = 64 now take 73.4.  At 16 384 walkers 24.9 with selects and exclusive-ors
// for the flips and the reduction first; 25.6 with shifted and masked count fields, 31.1
// instructions per attempt.)
// ---------------------------------------------------------------------------------
template <int L, int STRIDE, int EARLY>
struct AttemptStream {
    using Counts = RowCounts<L, EARLY == 0 && (L > 32)>;
    static constexpr int NW = row_words(L);
    static constexpr int kStep = -4 * STRIDE;          // row step of a flip: 4 STRIDE (2 - k) bytes
    static constexpr uint32_t kTwo = 8u * STRIDE;
    uint32_t E;                      // table row address of the current energy
    uint32_t Eacc;                   // the same if the next attempt flips
    bool prev_acc;                   // the previous attempt flipped
    uint32_t T0n, T1n, T0nn, T1nn;   // candidates of the next two attempts

    // First row of a launch: the candidates of its attempts 0 and 1.
    __device__ __forceinline__ void start(const uint32_t (&U)[NW], const uint32_t (&C)[NW], const uint32_t (&D)[NW],
                                          uint32_t E0)
    {
        const Counts k(U, C, D);
        E = E0;
        prev_acc = false;
        Eacc = add_count(k.word0(0), 0, kStep, E0 + kTwo);
        T0n = T1n = lds_u32(add_count(k.word0(0), 0, 4, E0));
        T0nn = lds_u32(add_count(k.word0(1), 1, 4, E0));
        T1nn = lds_u32(add_count(k.word1(1), 1, 4, Eacc));
    }

    // One row (U above, C updated in place, D below, D2 the row below D); on return the
    // candidates of the next row's attempts 0 and 1 are loaded.
    template <class Src>
    __device__ __forceinline__ void row(const uint32_t (&U)[NW], uint32_t (&C)[NW], const uint32_t (&D)[NW],
                                        const uint32_t (&D2)[NW], Src &src)
    {
        Counts k(U, C, D);
        uint32_t n0e = 0u, n0o = 0u, n1o = 0u;   // counts of the next row's sites 0 (n0e) and 1 (n0o, n1o)
        const uint32_t adj_if_flip = Counts::last_step(C);
#pragma unroll
        for (int xb = 0; xb < L; xb += 4) {
            const uint4 rw = src.get(xb);
            if (xb == L - 4)
                src.advance();
            const uint32_t words[4] = {rw.x, rw.y, rw.z, rw.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int x = xb + u;
                // counts for the step of attempt x + 1 (0: if x stays, 1: if it flips) and for the
                // candidates of attempt x + 2, in this row or the next (site 0's left neighbour
                // comes later)
                const uint32_t s0 = x + 1 == L ? n0e : k.word0(x + 1), s1 = x + 1 == L ? n0e : k.word1(x + 1);
                const uint32_t j0 = x + 2 < L ? k.word0(x + 2) : x + 2 == L ? n0e : n0o;
                const uint32_t j1 = x + 2 < L ? k.word1(x + 2) : x + 2 == L ? n0e : n1o;
                uint32_t stay = 0u, move = 0u, at_stay = 0u, at_move = 0u;
                if (EARLY >= 1) {
                    stay = add_count(s0, (x + 1) % L, kStep, E + kTwo);
                    move = add_count(s1, (x + 1) % L, kStep, Eacc + kTwo);
                }
                if (EARLY >= 2) {
                    at_stay = add_count(j1, (x + 2) % L, 4, stay);
                    at_move = add_count(j1, (x + 2) % L, 4, move);
                }
                const uint32_t T = prev_acc ? T1n : T0n;
                const bool acc = words[u] < T;
                E = acc ? Eacc : E;
                C[x >> 3] = flip_if(C[x >> 3], 1u << (4 * (x & 7)), acc);
                if (x == 0)
                    k.add_to_last(acc ? adj_if_flip : 0u);
                if (x == (L > 4 ? L - 5 : L - 3)) {
                    // the current row's sites 0 and 1 are final: the next row's first counts
                    const uint32_t kb = (C[0] ^ D[0]) + (D2[0] ^ D[0]) + (D[0] ^ right_of<L>(D, 0));
                    const uint32_t h0 = D[0] ^ left_of<L>(D, 0);
                    n0e = (kb + h0) & 0x0Fu;
                    n0o = ((kb + h0) >> 4) & 0x0Fu;
                    n1o = ((kb + 0x11111111u - h0) >> 4) & 0x0Fu;
                }
                if (EARLY >= 1)
                    Eacc = acc ? move : stay;
                else
                    Eacc = add_count(acc ? s1 : s0, (x + 1) % L, kStep, E + kTwo);
                T0n = T0nn;
                T1n = T1nn;
                T0nn = lds_u32(add_count(j0, (x + 2) % L, 4, E));
                if (EARLY >= 2)
                    T1nn = lds_u32(acc ? at_move : at_stay);
                else
                    T1nn = lds_u32(add_count(j1, (x + 2) % L, 4, Eacc));
                hist_add_one(E);
                prev_acc = acc;
            }
        }
    }
};

// ---------------------------------------------------------------------------------
// The same rows without the look-ahead: each attempt loads its one threshold once the
// attempt before it is decided.  The chain of an attempt (address, load, compare, select)
// then holds the load's latency, which other warps have to cover, but an attempt is 22.8
// instructions instead of 28.6 (L = 32, counted by ncu over 20 sweeps).  The decision enters as a factor 0 or 1: the step of the
// energy row and the flip bit are multiply-adds, on the pipe with room, where a select
// each would load the ALU.  Measured at L = 32, 48 640 walkers (2.5 warps per SM
// sub-partition) 57.9 us per sweep against 61.5 with the look-ahead; L = 16, 77 824 walkers
// (4 warps) 18.2 against 20.8; at one warp 33 against 24.5, at two 41 and 42 (L = 32, 38 912
// walkers): launches of more than two warps per sub-partition take it.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t mad32(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

template <int L, int STRIDE>
struct DirectStream {
    static constexpr int NW = row_words(L);
    uint32_t E;   // table row address of the current energy

    __device__ __forceinline__ void start(const uint32_t (&)[NW], const uint32_t (&)[NW], const uint32_t (&)[NW],
                                          uint32_t E0)
    {
        E = E0;
    }

    // One row (U above, C updated in place, D below).
    template <class Src>
    __device__ __forceinline__ void row(const uint32_t (&U)[NW], uint32_t (&C)[NW], const uint32_t (&D)[NW],
                                        const uint32_t (&)[NW], Src &src)
    {
        RowCounts<L> k(U, C, D);
        const uint32_t adj_if_flip = RowCounts<L>::last_step(C);
        uint32_t flips[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i)
            flips[i] = 0u;
        uint32_t kw = k.word0(0);
#pragma unroll
        for (int xb = 0; xb < L; xb += 4) {
            const uint4 rw = src.get(xb);
            if (xb == L - 4)
                src.advance();
            const uint32_t words[4] = {rw.x, rw.y, rw.z, rw.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int x = xb + u;
                const uint32_t T = lds_u32(add_count(kw, x, 4, E));
                const uint32_t step = add_count(kw, x, -4 * STRIDE, 8u * STRIDE);
                const bool acc = words[u] < T;
                uint32_t m = acc ? 1u : 0u;
                asm volatile("" : "+r"(m));   // kept as a number
                E = mad32(m, step, E);
                flips[x >> 3] = mad32(m, 1u << (4 * (x & 7)), flips[x >> 3]);
                if (x == 0)
                    k.add_to_last(acc ? adj_if_flip : 0u);
                if (x + 1 < L)
                    kw = acc ? k.word1(x + 1) : k.word0(x + 1);
                hist_add_one(E);
            }
        }
#pragma unroll
        for (int i = 0; i < NW; ++i)
            C[i] ^= flips[i];
    }
};

// nrows whole rows of one walker as one continuous attempt stream, from row y (wrapping to
// row 0 after row L - 1) whose column 0 lies in Philox block b.  Counter word 1 must stay
// at pk.c1 for the whole range.  The row below the next one is loaded from shared memory
// when a row starts (the current row does not change it).
template <int L, class Stream>
__device__ __forceinline__ uint32_t stream_rows(const SmemRows<L> &rows, uint32_t E, uint32_t b, int y, uint64_t nrows,
                                                const PhiloxKeys &pk)
{
    constexpr int NW = row_words(L);
    uint32_t U[NW], C[NW], D[NW];
    rows.load(y == 0 ? L - 1 : y - 1, U);
    rows.load(y, C);
    rows.load(y + 1 == L ? 0 : y + 1, D);
    PhiloxSource<L> src{pk, b};
    src.carry = PhiloxSource<L>::words(src.blk, pk);
    Stream st;
    st.start(U, C, D, E);
#pragma unroll 1
    for (uint64_t r = 0; r < nrows; ++r) {
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
        src.blk += (uint32_t)(L / 4);
        y = (y + 1 == L) ? 0 : y + 1;
    }
    return st.E;
}

// Attempts [x, x_end) of row y on its bit rows, one by one: the cut rows at the ends of a
// range (at most two per range, so the code is kept small).
template <int L, int STRIDE>
__device__ __forceinline__ uint32_t cut_row(const SmemRows<L> &rows, uint32_t E, int y, int x, int x_end, uint32_t blk,
                                            const PhiloxKeys &pk)
{
    using RowT = typename RowOf<L>::type;
    const RowT U = rows.load_bits(y == 0 ? L - 1 : y - 1), D = rows.load_bits(y + 1 == L ? 0 : y + 1);
    RowT C = rows.load_bits(y);
    uint4 rw = block_words(block_head(blk + (uint32_t)(x >> 2), pk), pk);
#pragma unroll 1
    for (; x < x_end; ++x) {
        const uint32_t s = bit_at(C, x);
        const uint32_t k = (s ^ bit_at(U, x)) + (s ^ bit_at(D, x)) + (s ^ bit_at(C, x == 0 ? L - 1 : x - 1)) +
                           (s ^ bit_at(C, x + 1 == L ? 0 : x + 1));
        const uint32_t u = (uint32_t)x & 3u;
        const uint32_t w = u == 0 ? rw.x : u == 1 ? rw.y : u == 2 ? rw.z : rw.w;
        if (w < lds_u32(E + 4u * k)) {
            C ^= (RowT)1 << x;
            E += (2u - k) * (4u * STRIDE);
        }
        hist_add_one(E);
        if (u == 3u)
            rw = block_words(block_head(blk + (uint32_t)(x >> 2) + 1u, pk), pk);
    }
    rows.store_bits(y, C);
    return E;
}

// The attempts of a plan.  One loop for the three parts: one inlined copy of the cut rows'
// code (an out-of-line call in it measured slower in the rows between).
template <int L, int STRIDE, class Stream>
__device__ __forceinline__ uint32_t run_plan(const SmemRows<L> &rows, uint32_t E, const RowPlan &p, uint64_t seed,
                                             uint32_t walker)
{
    const PhiloxKeys pk = make_keys(seed, walker, p.c1);
#pragma unroll 1
    for (int part = 0; part < 3; ++part) {
        if (part == 1) {
            if (p.rows > 0)
                E = stream_rows<L, Stream>(rows, E, p.blk1, p.y1, p.rows, pk);
        } else {
            const int x0 = part == 0 ? p.x0 : 0, x1 = part == 0 ? p.x0_end : p.tail;
            if (x0 < x1)
                E = cut_row<L, STRIDE>(rows, E, part == 0 ? p.y0 : p.y2, x0, x1, part == 0 ? p.blk0 : p.blk2, pk);
        }
    }
    return E;
}

// The launch's plans, made by the host: kernel parameters, so that the block counter that
// follows from them stays on the uniform data path (the heads of the Philox blocks then
// cost no vector issue: 47 against 50 cycles per attempt at one warp per sub-partition).
struct HostPlans {
    const LaunchPlan &plan;
    template <int L, int STRIDE, class Stream>
    __device__ __forceinline__ uint32_t run(const SweepArgs &a, int phase, const SmemRows<L> &rows, uint32_t E,
                                            uint32_t walker) const
    {
        return run_plan<L, STRIDE, Stream>(rows, E, plan.phase[phase], a.seed, walker);
    }
};

// Plans made on the device (batches, whose ranges come from memory); ranges that cross a
// step of Philox counter word 1 (t >> 34) run in parts, so that each part has it fixed.
struct DevicePlans {
    template <int L, int STRIDE, class Stream>
    __device__ __forceinline__ uint32_t run(const SweepArgs &a, int phase, const SmemRows<L> &rows, uint32_t E,
                                            uint32_t walker) const
    {
        uint64_t t0 = phase == 0 ? a.t0 : a.t0 + a.n_therm, n = phase == 0 ? a.n_therm : a.n;
#pragma unroll 1
        while (n > 0) {
            const uint64_t m = same_word1(t0, n);
            E = run_plan<L, STRIDE, Stream>(rows, E, row_plan(L, t0, m), a.seed, walker);
            t0 += m;
            n -= m;
        }
        return E;
    }
};

// The thresholds into the block's table rows as asynchronous 4-byte copies (the caller
// waits for them before its barrier), the counts zeroed, and the thresholds of the rows
// outside energies 0..N (row G holds energy 0).  A thread takes whole rows: no division per
// word, which made this loop 9 us of a launch at L = 64.  It is not unrolled: that changed
// the compiler's schedule of the attempts far below it (L = 32, 16384 walkers: 25.5 us per
// sweep instead of 24.5).
template <int NB, int NR, int G, int STRIDE>
__device__ __forceinline__ void load_table(uint32_t *sTab, const uint32_t *table, int tid, int nthr)
{
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sTab);
#pragma unroll 1
    for (int e = tid; e < NB; e += nthr) {
        const uint32_t at = sbase + (uint32_t)((e + G) * (4 * STRIDE));
#pragma unroll
        for (int k = 0; k < 5; ++k)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(at + 4u * k), "l"(table + e * 5 + k) : "memory");
        sTab[(e + G) * STRIDE + kHistSlot] = 0u;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int i = tid; i < (NR - NB) * STRIDE; i += nthr) {
        const int r = i / STRIDE;
        sTab[(r < G ? r : r + NB) * STRIDE + (i - r * STRIDE)] = 0u;
    }
}

// A walker's lattice (warp-cooperatively where the warp is full) into shared memory, and
// back.  Every lane of the warp calls them; lanes without a walker get an empty lattice.
// Bound by latency: few warps run, so each keeps many loads in flight - 16 packed rows, RB
// rows of bytes, a whole row of a ragged walker count (L = 64, 9000 walkers of bytes: what a
// launch takes besides its sweeps went from 174 to 87 us; 16384 packed ones, 36 to 23).
template <int L, int RB = 4>
__device__ __forceinline__ void load_lattice(const SweepArgs &a, const SmemRows<L> &rows, int64_t w, bool active,
                                             bool warp_full, int lane)
{
    using RowT = typename RowOf<L>::type;
    if (a.layout == MUCA_LAYOUT_PACKED) {
#pragma unroll 16
        for (int y = 0; y < L; ++y)
            rows.store_bits(y, active ? reinterpret_cast<const RowT *>(a.lattice)[(size_t)y * a.W + w] : (RowT)0);
    } else if (warp_full) {
        // RB rows per batch of loads
        for (int y = 0; y < L; y += RB) {
            RowT r[RB];
            warp_load_rows_int8<L, RB, RowT>(reinterpret_cast<const int8_t *>(a.lattice), a.W, w - lane, y, lane, r);
#pragma unroll
            for (int i = 0; i < RB; ++i)
                rows.store_bits(y + i, r[i]);
        }
    } else {
        const int8_t *g = reinterpret_cast<const int8_t *>(a.lattice);
        for (int y = 0; y < L; ++y) {
            RowT r = 0;
            if (active) {
#pragma unroll
                for (int x = 0; x < L; ++x)   // unrolled: a row's loads are in flight together
                    r |= (RowT)(g[(size_t)(y * L + x) * a.W + w] < 0) << x;
            }
            rows.store_bits(y, r);
        }
    }
}

template <int L>
__device__ __forceinline__ void store_lattice(const SweepArgs &a, const SmemRows<L> &rows, int64_t w, bool active,
                                              bool warp_full, int lane)
{
    using RowT = typename RowOf<L>::type;
    if (a.layout == MUCA_LAYOUT_PACKED) {
        if (active)
            for (int y = 0; y < L; ++y)
                reinterpret_cast<RowT *>(a.lattice)[(size_t)y * a.W + w] = rows.load_bits(y);
    } else if (warp_full) {
        // a walker whose energy is off the grid kept its lattice in shared memory unchanged
        for (int y = 0; y < L; ++y)
            warp_store_row_int8<L, RowT>(reinterpret_cast<int8_t *>(a.lattice), a.W, w - lane, y, lane, rows.load_bits(y));
    } else if (active) {
        int8_t *g = reinterpret_cast<int8_t *>(a.lattice);
        for (int y = 0; y < L; ++y) {
            const RowT r = rows.load_bits(y);
            for (int x = 0; x < L; ++x)
                g[(size_t)(y * L + x) * a.W + w] = bit_at(r, x) ? (int8_t)-1 : (int8_t)1;
        }
    }
}

// One block's share of a launch: walkers wbase .. wbase + wpb - 1 of the instance in
// `a` (warps from wpb on idle), all of the launch's attempts.  Every thread of the block
// calls it.  Shared memory: the table, one more row of zeros, then the rows of the wpb
// walkers.  A recording launch may carry a thermalization
// phase in front (n_therm attempts): its counts go to the histogram words too and are
// cleared before the recorded phase, so that the launch equals a thermalization launch
// followed by a recording one.  GUARD adds kTableGuard zero rows on both sides of the
// table, for energies that come from the caller and need not match the lattices (the
// library's own energies always do).
//
// The lanes of a warp stay together: a lane without a walker, or whose energy is off the
// grid, sits on the row of zeros, where no attempt is accepted and the counts are read by
// nobody, and so keeps its lattice.
template <int L, bool GUARD, int STRIDE, class Stream, class Plans>
__device__ __forceinline__ void sweep_block(const SweepArgs &a, const Plans &plans, int64_t wbase, int wpb,
                                            unsigned char *smem, bool record)
{
    if (a.skip && *a.skip)   // an iteration run on the device has finished
        return;
    constexpr int N = L * L;
    constexpr int NB = N + 1;
    constexpr int G = GUARD ? kTableGuard : 0;
    constexpr int NR = NB + 2 * G + 1;   // table rows: energies -G .. N + G, and the row of zeros
    const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    uint32_t *sTab = reinterpret_cast<uint32_t *>(smem);
    const SmemRows<L> rows{smem + align_up((size_t)NR * STRIDE * 4, 16), wpb, tid};
    const int64_t w = wbase + tid;
    const bool warp_on = tid < wpb && w - lane < a.W;   // uniform over the warp
    bool active = warp_on && w < a.W;
    const bool warp_full = warp_on && (w - lane + 32 <= a.W) && (a.W % 16 == 0);

    load_table<NB, NR, G, STRIDE>(sTab, a.table, tid, nthr);
    int32_t e = 0;
    if (warp_on) {
        load_lattice<L>(a, rows, w, active, warp_full, lane);
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

    const uint32_t tbase = (uint32_t)__cvta_generic_to_shared(sTab) + G * STRIDE * 4u;
    uint32_t E = tbase + (active ? (uint32_t)e : (uint32_t)(NB + G)) * (4u * STRIDE);
    const bool fused = record && a.n_therm > 0;   // uniform over the launch
#pragma unroll 1
    for (int phase = fused ? 0 : 1; phase < 2; ++phase) {
        if (warp_on)
            E = plans.template run<L, STRIDE, Stream>(a, phase, rows, E, a.walker0 + (uint32_t)w);
        if (phase == 0) {
            __syncthreads();
            for (int i = tid; i < NB; i += nthr)
                sTab[(i + G) * STRIDE + kHistSlot] = 0u;
            __syncthreads();
        }
    }
    if (active) {
        e = (int32_t)((E - tbase) / (4u * STRIDE));
        if (E < tbase || e > N || (E - tbase) % (4u * STRIDE) != 0u)   // corrupted energy address
            atomicOr(a.err, kErrEnergyRange);
    }
    __syncthreads();
    if (record)
        for (int i = tid; i < NB; i += nthr) {
            const uint32_t v = sTab[(i + G) * STRIDE + kHistSlot];
            if (v)
                atomicAdd(&a.hist[i], (unsigned long long)v);
        }
    if (warp_on)
        store_lattice<L>(a, rows, w, active, warp_full, lane);
    if (active)
        a.energy[w] = e;
}

// A batched work item.  Out of line: inlined into one kernel, the six sizes' loops came out
// with twice the fixed-latency stalls (four L = 32 instances of 9728 walkers: 6.8 against
// 7.5 x 10^11 attempts/s).
template <int L, bool GUARD = false, int STRIDE = kTableStride>
__device__ __noinline__ void batch_item(const SweepArgs &a, const BatchItem &it, unsigned char *smem, bool record)
{
    sweep_block<L, GUARD, STRIDE, AttemptStream<L, STRIDE, 0>>(a, DevicePlans{}, it.wbase, it.wpb, smem, record);
}

}  // namespace
}  // namespace muca
