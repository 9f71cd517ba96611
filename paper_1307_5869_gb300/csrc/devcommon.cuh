// Device helpers shared by the generation and jump kernels: exact modular
// arithmetic for the moduli of Sec. 5.1-5.2, SplitMix64 seed expansion, the
// float epilogue, and vectorised output emission.
#pragma once

#include <type_traits>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "prand_internal.h"

namespace prand {

constexpr unsigned kFull = 0xFFFFFFFFu;

// ---------------------------------------------------------------- SplitMix64
// Seed expansion (Steele, Lea & Flood 2014); the same published definition on
// both sides of any comparison, used only to turn a 64-bit seed into states.
__host__ __device__ inline uint64_t splitmix64_next(uint64_t &s)
{
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// ---------------------------------------------------------------- mod m1, m2
// a * b mod m for m = 2^32 - c (c = 209 or 22853), a, b < 2^32: fold the high
// word twice with 2^32 = c (mod m).
template <uint32_t C>
__device__ __forceinline__ uint32_t mulmod_2p32_minus(uint32_t a, uint32_t b)
{
    constexpr uint64_t m = (1ull << 32) - C;
    uint64_t p = (uint64_t)a * b;
    uint64_t t = (p & 0xFFFFFFFFull) + (uint64_t)C * (p >> 32);   // < 2^32 (1 + C)
    t = (t & 0xFFFFFFFFull) + (uint64_t)C * (t >> 32);            // < 2^32 + C (C+1)
    if (t >= m) t -= m;
    return (uint32_t)t;
}

__device__ __forceinline__ uint32_t addmod_u32(uint32_t a, uint32_t b, uint32_t m)
{
    uint64_t s = (uint64_t)a + b;
    return (uint32_t)(s >= m ? s - m : s);
}

// ---------------------------------------------------------------- mod p (GM/GQ)
// Full products of residues modulo the five primes of Table 2.
template <int KIND>
__device__ __forceinline__ uint64_t reduce_prod(uint64_t lo, uint64_t hi);

// p = 2^19 - 1: product < 2^38 (hi = 0)
template <>
__device__ __forceinline__ uint64_t reduce_prod<P19>(uint64_t lo, uint64_t)
{
    constexpr uint64_t p = (1ull << 19) - 1;
    uint64_t r = (lo & p) + (lo >> 19);   // < 2^20
    r = (r & p) + (r >> 19);              // <= p + 1
    return r >= p ? r - p : r;
}
// p = 2^29 - 3: product < 2^58 (hi = 0); 2^29 = 3 (mod p)
template <>
__device__ __forceinline__ uint64_t reduce_prod<P29>(uint64_t lo, uint64_t)
{
    constexpr uint64_t p = (1ull << 29) - 3, m = (1ull << 29) - 1;
    uint64_t r = (lo & m) + 3 * (lo >> 29);   // < 2^29 + 3 * 2^29
    r = (r & m) + 3 * (r >> 29);              // < 2^29 + 12
    return r >= p ? r - p : r;
}
// p = 2^31 - 1: product < 2^62 (hi = 0)
template <>
__device__ __forceinline__ uint64_t reduce_prod<P31>(uint64_t lo, uint64_t)
{
    constexpr uint64_t p = (1ull << 31) - 1;
    uint64_t r = (lo & p) + (lo >> 31);   // < 2^32
    r = (r & p) + (r >> 31);
    return r >= p ? r - p : r;
}
// p = 2^51 - 129: product < 2^102; 2^51 = 129 (mod p)
template <>
__device__ __forceinline__ uint64_t reduce_prod<P51>(uint64_t lo, uint64_t hi)
{
    constexpr uint64_t p = (1ull << 51) - 129, m = (1ull << 51) - 1;
    uint64_t h = (hi << 13) | (lo >> 51);         // < 2^51
    uint64_t r = (lo & m) + 129 * h;              // < 2^51 + 2^59
    r = (r & m) + 129 * (r >> 51);                // < 2^51 + 2^17
    return r >= p ? r - p : r;
}
// p = 2^61 - 1: product < 2^122
template <>
__device__ __forceinline__ uint64_t reduce_prod<P61>(uint64_t lo, uint64_t hi)
{
    constexpr uint64_t p = (1ull << 61) - 1;
    uint64_t r = (lo & p) + ((hi << 3) | (lo >> 61));   // < 2^62
    r = (r & p) + (r >> 61);
    return r >= p ? r - p : r;
}

template <int KIND>
__device__ __forceinline__ uint64_t mulmod_p(uint64_t a, uint64_t b)
{
    if (KIND == P51 || KIND == P61) return reduce_prod<KIND>(a * b, __umul64hi(a, b));
    return reduce_prod<KIND>(a * b, 0);
}

template <int KIND>
__device__ __forceinline__ uint64_t prime_of()
{
    return KIND == P19 ? (1ull << 19) - 1 : KIND == P29 ? (1ull << 29) - 3 : KIND == P31 ? (1ull << 31) - 1
         : KIND == P51 ? (1ull << 51) - 129 : (1ull << 61) - 1;
}

template <int KIND>
__device__ __forceinline__ uint64_t addmod_p(uint64_t a, uint64_t b)
{
    uint64_t s = a + b;   // both < p < 2^62
    return s >= prime_of<KIND>() ? s - prime_of<KIND>() : s;
}

// ---------------------------------------------------------------- floats
// f32 = (u >> 8) * 2^-24, formed as (u & 0xFFFFFF00) * 2^-32: the masked word
// has at most 24 significant bits, so it converts exactly (in any rounding
// mode), and the scale is a power of two whose product stays normal (the
// smallest nonzero value is 2^-24).  The mask folds into the logic operation
// that forms u in the cheapest generators (LFSR113's XOR of its components),
// so no shift is spent on either integer pipe.
__device__ __forceinline__ float u32_to_f32(uint32_t u) { return __uint2float_rz(u & 0xFFFFFF00u) * 0x1p-32f; }

// f64 = u * 2^-32, assembled from the bits (exact) to stay off the FP64 pipe.
__device__ __forceinline__ double u32_to_f64(uint32_t u)
{
    if (u == 0) return 0.0;
    int lz = __clz(u);                         // MSB at bit 31 - lz
    uint32_t m = (u << lz) << 1;               // fraction bits, MSB dropped
    uint32_t hi = ((uint32_t)(1022 - lz) << 20) | (m >> 12);
    uint32_t lo = m << 20;
    return __hiloint2double((int)hi, (int)lo);
}

// MRG32K3A f64 = z * RN(1 / (m1 + 1)), one round-to-nearest multiply, done in
// integer arithmetic so it stays off the FP64 pipe.  The constant is
// M 2^-84 with M = 0x1000000D00000B (53 bits, high word 2^20), so the exact
// product is P 2^-84 with P = z 2^52 + z Ml (Ml = M mod 2^32, one wide
// multiply).  With top = P >> 32 of bit length L, the double keeps the 53 bits
// P >> s, s = L - 21, rounded to nearest even on the s dropped bits, and its
// bits are ((s + 990) << 52) + mantissa (a round-up to 2^53 carries into the
// exponent by itself).  z = 0 gives 0.
__device__ __forceinline__ double mrg_to_f64(uint32_t z)
{
    const uint64_t zm = (uint64_t)z * 0x0D00000Bu;               // z Ml < 2^60
    const uint32_t w0 = (uint32_t)zm;                             // P mod 2^32
    const uint64_t top = ((uint64_t)z << 20) + (zm >> 32);        // P >> 32 < 2^53
    const uint32_t th = (uint32_t)(top >> 32), tl = (uint32_t)top;
    const int L = th ? 64 - __clz(th) : 32 - __clz(tl);           // 21..53 for z >= 1
    const int sh = L - 21;                                        // bits dropped, 0..32
    uint32_t mlo, mhi;
    asm("shf.r.clamp.b32 %0, %2, %3, %4;\n\t"
        "shf.r.clamp.b32 %1, %3, %5, %4;"
        : "=r"(mlo), "=r"(mhi) : "r"(w0), "r"(tl), "r"(sh), "r"(th));
    // the dropped bits, left-aligned (0 when nothing is dropped); round up above
    // one half, or at one half when the kept part is odd
    const uint32_t rem = sh ? w0 << (32 - sh) : 0u;
    const uint32_t up = rem > 0x80000000u - (mlo & 1u) ? 1u : 0u;
    const uint64_t m = (((uint64_t)mhi << 32) | mlo) + up;
    const uint64_t bits = ((uint64_t)(sh + 990) << 52) + m;
    return z ? __longlong_as_double((long long)bits) : 0.0;
}

// ---------------------------------------------------------------- output
// Conversion of one 32-bit output to the requested element type.
template <typename OutT, bool MRG = false>
struct Cvt;
template <bool MRG>
struct Cvt<uint32_t, MRG> { __device__ __forceinline__ static uint32_t f(uint32_t u) { return u; } };
template <bool MRG>
struct Cvt<float, MRG> { __device__ __forceinline__ static float f(uint32_t u) { return u32_to_f32(u); } };
template <>
struct Cvt<double, false> { __device__ __forceinline__ static double f(uint32_t u) { return u32_to_f64(u); } };
template <>
struct Cvt<double, true> { __device__ __forceinline__ static double f(uint32_t u) { return mrg_to_f64(u); } };

// Store two consecutive elements at p (aligned to both).
template <typename OutT>
__device__ __forceinline__ void store2(OutT *p, OutT a, OutT b)
{
    struct alignas(2 * sizeof(OutT)) Two { OutT a, b; };
    *reinterpret_cast<Two *>(p) = Two{ a, b };
}

// Store four consecutive elements at p (16-byte aligned for 4-byte types,
// 32-byte aligned for doubles when vec is true).
template <typename OutT>
__device__ __forceinline__ void store4(OutT *p, OutT a, OutT b, OutT c, OutT d);
template <>
__device__ __forceinline__ void store4<uint32_t>(uint32_t *p, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    *reinterpret_cast<uint4 *>(p) = make_uint4(a, b, c, d);
}
template <>
__device__ __forceinline__ void store4<float>(float *p, float a, float b, float c, float d)
{
    *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}
template <>
__device__ __forceinline__ void store4<double>(double *p, double a, double b, double c, double d)
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(a, b);
    reinterpret_cast<double2 *>(p)[1] = make_double2(c, d);
}

// Store four consecutive elements at p, aligned to all of them: doubles as one 32-byte
// store, so that a sector leaves whole.
template <typename OutT>
__device__ __forceinline__ void store4_whole(OutT *p, OutT a, OutT b, OutT c, OutT d)
{
    if constexpr (sizeof(OutT) == 8) *reinterpret_cast<double4_32a *>(p) = make_double4_32a(a, b, c, d);
    else store4<OutT>(p, a, b, c, d);
}

// ---------------------------------------------------------------- row staging
// Thread-per-stream generators produce one row of outputs per lane; written
// directly, a warp store would scatter 32 small pieces over 32 rows.  Instead
// each lane stages ROWB bytes (128 or 256) of its row in a padded shared-memory
// tile (pitch ROWB + 16, so 16-byte accesses are bank-conflict free on both
// sides) and the warp writes the tile out as whole ROWB-byte row segments,
// 512 / ROWB rows per store.  Longer segments suit HBM better; shorter ones
// need half the shared memory.
template <typename OutT, int ROWB = 128>
struct RowFill {
    static constexpr int K = ROWB / (int)sizeof(OutT);  // outputs per row chunk
    static constexpr int E = 16 / (int)sizeof(OutT);    // outputs per 16-byte vector
    static constexpr int PITCH = ROWB + 16;             // tile bytes per row
    static constexpr int TILE = 32 * PITCH;             // tile bytes per warp
    static constexpr int PIECES = ROWB / 16;            // 16-byte pieces per row segment
    static constexpr int ROWS = 32 / PIECES;            // row segments per warp store
};
constexpr int kTileBytes = RowFill<uint32_t, 128>::TILE;  // per warp, 128-byte segments

// Emits `len` outputs of this lane's stream to dst (aligned to an output), all
// 32 lanes of the warp taking part (lanes with len 0 only help store).
// next() returns the next 32-bit output; cvt converts it.  tile: the warp's
// RowFill<OutT, ROWB>::TILE bytes of shared memory.
// Rows on 16-byte boundaries are cut from their start.  Where a row of the warp is not on
// one, every row is cut at multiples of ROWB in memory, so that every chunk but its first
// and last leaves as whole lines in 16-byte stores (2^20 rows of 777: LFSR113 f32 742 us,
// MRG32K3A u32 920, by each thread's own stores 3436 and 3385).  The chunks that every
// lane has whole are a loop of their own; tests in it cost MRG32K3A 2 % of its bulk fill.
// ENDS: lanes may be idle or their rows end apart by whole chunks (a batch's request of
// fewer than 32 sections); the chunks between two ends go through that loop too, by the lanes
// that have them (3000 requests of 3000 LFSR113 u32 317 us without, 172).  Fills do without: it
// costs rows of 32 to 100 outputs 4 to 6 %, and their idle lanes repeat the last section.
// ROLL: keep the loop over a chunk's 16-byte pieces rolled (for generators
// whose next() is long, where unrolling a whole chunk would outgrow the
// instruction cache).  A generator may offer next(k) as well, for output k of a
// whole chunk (k a constant, in order from 0).
template <typename OutT, int ROWB = 128, bool ROLL = false, bool ENDS = false, typename Next, typename Conv>
__device__ __forceinline__ void fill_rows(Next &&next, Conv &&cvt, OutT *dst, uint64_t len, unsigned char *tile, int lane)
{
    using RF = RowFill<OutT, ROWB>;
    constexpr int K = RF::K, E = RF::E, PITCH = RF::PITCH, PIECES = RF::PIECES, ROWS = RF::ROWS;
    const bool on_vectors = __all_sync(kFull, len == 0 || (uintptr_t)dst % 16 == 0);
    const uint32_t phase = on_vectors ? 0u : (uint32_t)((uintptr_t)dst % ROWB) / (uint32_t)sizeof(OutT);
    OutT *const base = dst - phase;          // the row in whole chunks, from its first output's
    const uint64_t end = len ? phase + len : 0;
    // (a row in memory is fewer than 2^32 chunks; 64-bit lengths by shuffles took 1 to 2 % of
    // the bulk fills)
    const uint32_t nch = __reduce_max_sync(kFull, (uint32_t)((end + K - 1) / K));
    const uint32_t whole = (uint32_t)(end / K);  // up to where this lane's chunks are whole
    const uint32_t whole0 = on_vectors ? 0 : 1, whole1 = ENDS ? 0u : __reduce_min_sync(kFull, whole);  // those every lane has whole
    unsigned char *myrow = tile + lane * PITCH;
    const int piece = lane % PIECES;
    // a whole chunk's outputs of this lane into the tile
    auto make = [&]() {
#pragma unroll (ROLL ? 1 : PIECES)
        for (int v = 0; v < PIECES; ++v) {
            OutT vals[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if constexpr (std::is_invocable<Next, int>::value) vals[e] = cvt(next(v * E + e));
                else vals[e] = cvt(next());
            }
            *reinterpret_cast<uint4 *>(myrow + 16 * v) = *reinterpret_cast<const uint4 *>(vals);
        }
    };
    // (by the whole warp) the tile's rows out, from their places in a chunk (mydst): `cols` outputs of those in `rows`
    auto leave = [&](unsigned long long mydst, auto all, uint32_t rows, int cols) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < PIECES; ++i) {
            const int r = ROWS * i + lane / PIECES;
            OutT *rd = (OutT *)__shfl_sync(kFull, mydst, r);
            if (decltype(all)::value || (piece * E < cols && ((rows >> r) & 1u)))
                *reinterpret_cast<uint4 *>(rd + piece * E) = *reinterpret_cast<const uint4 *>(tile + r * PITCH + 16 * piece);
        }
        __syncwarp();
    };
    for (uint32_t ch = 0; ch < nch; ++ch) {
        if (!ENDS && ch >= whole0 && ch < whole1) {
            // no per-output tests, and every row segment of the tile is stored whole
            do {
                const unsigned long long mydst = (unsigned long long)(base + (uint64_t)ch * K);
                make();
                leave(mydst, std::true_type{}, kFull, K);
            } while (++ch < whole1);
            if (ch >= nch) return;
        }
        // this lane's outputs of the chunk: columns lo .. hi - 1
        const uint32_t lo = ch ? 0u : phase;
        const uint32_t hi = end > (uint64_t)ch * K ? (uint32_t)min((uint64_t)K, end - (uint64_t)ch * K) : 0u;
        const unsigned long long mydst = (unsigned long long)(base + (uint64_t)ch * K);
        if constexpr (ENDS) {
            if (__all_sync(kFull, hi == 0 || (lo == 0 && hi == (uint32_t)K))) {
                const uint32_t rows = __ballot_sync(kFull, hi != 0), stop = __reduce_min_sync(kFull, hi ? whole : nch);
                for (;;) {
                    if (hi) make();
                    const unsigned long long to = (unsigned long long)(base + (uint64_t)ch * K);
                    if (rows == kFull) leave(to, std::true_type{}, kFull, K);
                    else leave(to, std::false_type{}, rows, K);
                    if (ch + 1 >= stop) break;
                    ++ch;
                }
                continue;
            }
        }
        const uint32_t hi0 = ENDS ? __reduce_max_sync(kFull, hi) : __shfl_sync(kFull, hi, 0);
        if (hi0 % E == 0 && __all_sync(kFull, (ENDS && hi == 0) || (lo == 0 && hi == hi0))) {
            // every lane has the same whole pieces (or none): short rows, or the end of rows
            const uint32_t rows = ENDS ? __ballot_sync(kFull, hi != 0) : kFull;
            if (!ENDS || hi) {
#pragma unroll 4
                for (int v = 0; v < (int)(hi0 / E); ++v) {
                    OutT vals[E];
#pragma unroll
                    for (int e = 0; e < E; ++e) vals[e] = cvt(next());
                    *reinterpret_cast<uint4 *>(myrow + 16 * v) = *reinterpret_cast<const uint4 *>(vals);
                }
            }
            leave(mydst, std::false_type{}, rows, (int)hi0);
            continue;
        }
        // a row's first or last chunk, or rows of several lengths: rolled (a warp comes here
        // once or twice a row, with cold code: unrolled it took 2 us a chunk)
#pragma unroll 2
        for (int v = 0; v < PIECES; ++v) {
            if ((uint32_t)(v * E) >= hi) continue;
            OutT vals[E];
#pragma unroll
            for (uint32_t e = 0; e < E; ++e) vals[e] = v * E + e >= lo && v * E + e < hi ? cvt(next()) : OutT(0);
            *reinterpret_cast<uint4 *>(myrow + 16 * v) = *reinterpret_cast<const uint4 *>(vals);
        }
        __syncwarp();
#pragma unroll 1
        for (int i = 0; i < PIECES; ++i) {
            const int r = ROWS * i + lane / PIECES;
            OutT *rd = (OutT *)__shfl_sync(kFull, mydst, r);
            const uint32_t rl = __shfl_sync(kFull, lo, r), rh = __shfl_sync(kFull, hi, r), col = piece * E;
            const unsigned char *src = tile + r * PITCH + 16 * piece;
            if (col >= rl && col + E <= rh) {
                *reinterpret_cast<uint4 *>(rd + col) = *reinterpret_cast<const uint4 *>(src);
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (col + e >= rl && col + e < rh) rd[col + e] = reinterpret_cast<const OutT *>(src)[e];
            }
        }
        __syncwarp();
    }
}

// Whether a fill of n rows of nper outputs (nsec sections of seclen each) leaves through
// fill_rows or by each thread's own stores, whose lines L2 puts together while the fill
// fits there.  Rows on 16-byte boundaries: staged from 96 MiB on, and below if sections
// are own_len or longer (32 for the lighter steps; never for MRG32K3A, whose stores then
// hide behind its steps), but not for less than a warp of sections.  Others: staged beyond
// L2 when long: from off_len outputs (64; 512 for the thread-per-stream ensembles, whose
// first and last chunks, made for all lanes, are half a chunk's long steps lost each: GQ58.3
// u32 2^20 x 98 820 us, by own stores 636; 65536 x 777, x 1821 384 and 389, 797 and 909).
// host: the rows are in host memory, where no cache puts a thread's stores together on the
// way over the link (MRG32K3A u32 65536 x 256 366 staged, 1610 own; 3 x 100000 23 / 36): staged
// from 192 KiB on at the latest when they are on 16-byte boundaries (MRG32K3A 63 x 80 f64 20 / 15).
// Measured on the device, us, staged / own:
//   on 16 bytes: MRG32K3A one stream of 10^6 f64 10.3 / 8.2, 65536 x 300 u32 32.7 / 30.8,
//     x 500 f32 51 / 71; LFSR113 f32 2^20 x 16 30.8 / 22.6, 2^18 x 32 12.6 / 13.3, 65536 x
//     320 26.7 / 32.8; one stream of 64: LFSR113 u32 8.2 / 4.2, GQ58.3 18.5 / 12.3
//   others: MRG32K3A u32 2^20 x 47 162 / 152, x 63 180 / 212, x 777 920 / 3385, 65536 x
//     777 88 / 187, x 301 47 / 32
template <typename OutT>
inline bool staged_rows(const OutT *out, uint64_t n, uint64_t nper, uint32_t nsec, uint64_t seclen, uint64_t own_len, bool host = false,
                        uint64_t off_len = 64)
{
    constexpr uint64_t E = RowFill<OutT>::E;
    const uint64_t mib = n * nper / ((1ull << 20) / sizeof(OutT));
    if ((uintptr_t)out % 16 == 0 && nper % E == 0 && seclen % E == 0)
        return mib >= 96 || (n * nsec >= 32 && (seclen >= own_len || (host && n * nper * sizeof(OutT) >= 192u << 10)));
    return nper >= off_len && mib >= 144;
}

// Resident threads of a kernel launched with BS-thread blocks on the current
// device, computed once per kernel and device (ID tells the kernels apart: the
// generator id for the per-handle fills, 100 and up for the others).
template <int ID, int BS = 256, typename K>
inline uint64_t resident_threads(K kernel)
{
    constexpr int kDevs = 64;
    static std::atomic<uint64_t> cache[kDevs];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < kDevs) {
        const uint64_t c = cache[dev].load(std::memory_order_relaxed);
        if (c) return c;
    }
    const int sms = device_sm_count();
    int bps = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, BS, 0) != cudaSuccess || bps < 1) bps = 1;
    const uint64_t c = (uint64_t)sms * bps * BS;
    if (dev >= 0 && dev < kDevs) cache[dev].store(c, std::memory_order_relaxed);
    return c;
}

// Big offsets.
__device__ __forceinline__ int u256_bit(const U256 &e, int b) { return (int)((e.w[b >> 6] >> (b & 63)) & 1u); }

}  // namespace prand
