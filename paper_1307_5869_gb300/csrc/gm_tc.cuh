// GM/GQ generation on the tensor cores (tcgen05.mma): the lane-per-point
// ensembles (v = 1) and the 8-point ensembles with v = 4.
//
// The map is linear: with X0 = x^(n) and X1 = x^(n+m) (m = 64), every value of the
// block between them is x^(n+j) = a_j X0 + b_j X1 (mod p), with constants a_j, b_j
// that are the same for every point of every stream; and the next block's pair
// needs only X2 = x^(n+2m) = V X1 - q^m X0 (eq. (rec2)).  What a step outputs is
// floor(2^v x / p), the top bits of the fraction x / p, and a fraction needs no
// reduction: with X0 and X1 cut into limbs f_k at bits i_k (bytes or nibbles),
// x^(n+j) / p = sum_k f_k W_jk (mod 1), W_jk = (c 2^(i_k) mod p) / p (c = a_j or b_j)
// rounded to 24 bits.  W in two balanced digits of 12 bits makes that a product of
// small integers,
//     [128 points x 16 or 32 slots] x [slots x 128 digit columns],
// one or two tcgen05.mma (f16 inputs, f32 accumulators in tensor memory) per block
// of 64 steps of 128 points.  It is exact: limbs and digits are f16 integers (a limb
// is a subnormal f16, put in place by a byte permute; a digit is scaled by 2^4), and
// every partial sum stays below 2^24 units.  A bias of 1.5 2^23 units (one slot of
// each value is 1.0) fixes the exponent of every sum, so the bits of the accumulator
// are the integer sum, and t = 2^20 d0 + 2^8 d1 (mod 2^32) is the fraction, its top v
// bits the output.
//
// t is off by at most a margin of 37 to 314 units of 2^-24 (the rounding of W, bounded
// on the host when the tables are built); a second bias adds the margin, so a
// fraction that close to a strip boundary shows as (t mod 1/2^v) < 2 margins.  Every
// t is checked (one running minimum per point and half block); a point with such a
// value (one in 2 to 12 % of a warp's half blocks) is computed again, exactly in 64
// bits.  Outputs are therefore those of the recurrence, bit for bit.
//
// What bounds it: the arithmetic after the product, per point step two multiply-adds
// (FMA-heavy pipe, 2 cycles each), one funnel shift and half a three-input minimum
// (ALU, 2 cycles each), against four 32x32->64 products and a fold (about 24 cycles)
// by the recurrence; issue slots 70 % busy, both pipes 57 %, the tensor pipe 12 to 22 %.
// GB300, 65536 streams x 4096 u32, G words/s, lane-per-point or thread-per-stream
// kernel (gm_impl.cuh) / this one: GM61 51 / 126, GM31 88 / 145, GQ58.1 74 / 143, GM55
// 134 / 387, GQ58.4 250 / 462, GM19 128 / 146, GM29 135 / 143.  Measured on the way
// (GM31 / GM61): three digits and m = 32, 100 / 87; the same with m = 64 and two
// blocks per SM, 59 / 56 (two warps per scheduler cannot hide the latencies); two
// digits, m = 32, eight blocks of 64 registers, 108 / 88 (constants recomputed); m =
// 64 with a warp group per half, 64 registers, 107 / 95; this form without the next
// tile's product behind the last block, 139 / 119.
#pragma once
#include "batch.cuh"
#include "gm_impl.cuh"
#include "gm_tc_table.h"

namespace prand {

constexpr int kTcThreads = 128;  // one thread per point row of the product (M)
constexpr int kTcTmem = 128;     // tensor-memory columns per block of threads: one product's accumulators
constexpr int kTcCtas = 4;       // resident blocks per SM: tensor memory has 512 columns
// Dynamic shared memory: B and A, and enough more that no fifth block is put on
// an SM, where it would wait for tensor memory.
constexpr unsigned kTcSmem = 46 * 1024;

template <int GEN>
struct GmTc {
    using P = GmT<GEN>;
    static constexpr bool kUse = P::s == 32 || P::s == 8;
    static constexpr bool kNibbles = tc_nibbles(P::kind, P::v);
    static constexpr int kSlots = 2 * tc_value_slots(P::kind, P::v);       // K
    static constexpr int kImage = kTcCols * kSlots * 2;                    // bytes of a product's B
    static constexpr int kACol = kTcThreads * 16;                          // bytes of a 16-byte column of A
    static constexpr int kA = kSlots / 8 * kACol;                          // bytes of A
    static constexpr int kRegs = P::v;                                     // registers of strips per point and half
    static constexpr uint32_t kNear = 2 * tc_margin(P::kind, P::v) << (P::v == 1 ? 8 : 8 + P::v);  // of TcStrips' minimum
    static constexpr int kStreams = kTcThreads / (P::s == 32 ? 32 : 8);    // sections per block of threads
    static_assert(2 * kTcCols <= kTcTmem && kTcCtas * kTcTmem <= 512 && 2 * kImage + kA <= (int)kTcSmem, "operands fit");
};

// ------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t tc_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, K-major without swizzle: 8-row x 16-byte
// core matrices, `lbo` bytes apart along K and `sbo` bytes apart along M / N.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}

// Where `go`: D = A B over K slots (kind::f16, D f32, A and B f16, both K-major;
// 16 slots per instruction), its completion signalled on `mbar`.  For one thread
// of the block; predicated, since in diverged code the operands would go to the
// uniform registers they need through a loop over the lanes.
template <int N, int K>
__device__ __forceinline__ void tc_mma(bool go, uint32_t d, uint64_t a, uint64_t b, uint32_t mbar)
{
    constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(N / 8) << 17) | ((uint32_t)(kTcThreads / 16) << 24);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
    for (int k = 0; k < K; k += 16)
        asm volatile("{\n\t"
                     ".reg .pred p, q;\n\t"
                     "setp.ne.u32 p, %4, 0;\n\t"
                     "setp.ne.u32 q, %5, 0;\n\t"
                     "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
                     "}" :: "r"(d), "l"(a + (uint64_t)(k / 8 * kTcThreads * 16 >> 4)), "l"(b + (uint64_t)(k / 8 * 128 >> 4)),
                     "r"(idesc), "r"((uint32_t)k), "r"((uint32_t)go) : "memory");
    asm volatile("{\n\t"
                 ".reg .pred q;\n\t"
                 "setp.ne.u32 q, %1, 0;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t"
                 "}" :: "r"(mbar), "r"((uint32_t)go) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Lane 0 counts its warp in (acquire and release), from 0 to 3 and round again;
// returns the count before it.  (An increment with a limit: an addition the compiler
// would turn into one over the warp's lanes, at a dozen instructions more.)
__device__ __forceinline__ uint32_t tc_count(bool go, uint32_t addr)
{
    uint32_t old = 0;
    asm volatile("{\n\t"
                 ".reg .pred q;\n\t"
                 "setp.ne.u32 q, %2, 0;\n\t"
                 "@q atom.acq_rel.cta.shared::cta.inc.u32 %0, [%1], 3;\n\t"
                 "}" : "+r"(old) : "r"(addr), "r"((uint32_t)go) : "memory");
    return old;
}
__device__ __forceinline__ bool tc_try(uint32_t mbar, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n\t"
                 ".reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t"
                 "}" : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
    return done != 0;
}
// Wait for the phase of `mbar`, with a limit (about a second; a wait that
// reaches it sets *err and *late, and later ones do not wait).  Every wait of the kernel
// inside its loop is one of these, so the kernel always ends.
__device__ __forceinline__ void tc_wait(uint32_t mbar, uint32_t parity, bool &dead, volatile uint32_t *err, uint32_t *late)
{
    if (tc_try(mbar, parity) || dead) return;
    for (uint32_t i = 0; i < (1u << 20); ++i)
        if (tc_try(mbar, parity)) return;
    dead = true;
    *late = 1u;
    *err = 1u;
}

// 16 steps' accumulator columns of the warp's 32 points into registers.
#define PRAND_TC_R8(O) "=r"((O)[0]), "=r"((O)[1]), "=r"((O)[2]), "=r"((O)[3]), "=r"((O)[4]), "=r"((O)[5]), "=r"((O)[6]), "=r"((O)[7])
__device__ __forceinline__ void tc_ld(uint32_t (&r)[32], uint32_t taddr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : PRAND_TC_R8(r), PRAND_TC_R8(r + 8), PRAND_TC_R8(r + 16), PRAND_TC_R8(r + 24) : "r"(taddr));
}
#undef PRAND_TC_R8
// The registers of a load hold their values only after this; they are its
// operands so that no use of them can be moved before it.
__device__ __forceinline__ void tc_ld_wait(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) asm volatile("" : "+r"(r[i]));
}

// ------------------------------------------------------------------ pieces
// A value as the block recurrence takes it: for the 51- and 61-bit primes split at
// bit 26 or 31, where every sum of partial products fits 64 bits (at bit 32 the
// low one would not).  Lazy residues: below p + 8 (p + 2^18 for GM55).
template <int GEN>
struct TcValue {
    using P = GmT<GEN>;
    static constexpr bool kWide = P::kind == P51 || P::kind == P61;
    static constexpr int kCut = P::kind == P61 ? 31 : 26;
    uint32_t lo, hi;
    __device__ __forceinline__ TcValue() : lo(0), hi(0) {}
    __device__ __forceinline__ explicit TcValue(uint64_t x)
    {
        lo = kWide ? (uint32_t)x & ((1u << kCut) - 1) : (uint32_t)x;
        hi = kWide ? (uint32_t)(x >> kCut) : 0u;
    }
    __device__ __forceinline__ uint64_t whole() const { return kWide ? ((uint64_t)hi << kCut) + lo : (uint64_t)lo; }
};

// The block recurrence X2 = v X1 + q X0 (mod p), once per block and point: eight
// 32x32->64 multiply-adds without carries between them (two for a 32-bit prime)
// and one fold, no comparison.
template <int GEN>
struct TcBlockStep {
    using P = GmT<GEN>;
    using V = TcValue<GEN>;
    V v, q;
    __device__ __forceinline__ TcBlockStep(uint64_t v_, uint64_t q_) : v(v_), q(q_) {}
    __device__ __forceinline__ uint64_t operator()(const V &a, const V &b) const
    {
        if constexpr (P::kind == P61) {
            constexpr uint64_t p = P::p;
            // 2^62 = 2 (mod p): the high product joins the low one, doubled
            const uint64_t L = (uint64_t)v.lo * a.lo + (uint64_t)q.lo * b.lo + (uint64_t)(2 * v.hi) * a.hi + (uint64_t)(2 * q.hi) * b.hi;
            const uint64_t M = (uint64_t)v.lo * a.hi + (uint64_t)v.hi * a.lo + (uint64_t)q.lo * b.hi + (uint64_t)q.hi * b.lo;
            // M 2^31 = (M >> 30) + (M mod 2^30) 2^31; the sum is below 2^64
            const uint64_t S = L + (M >> 30) + ((M & ((1ull << 30) - 1)) << 31);
            return (S & p) + (S >> 61);
        } else if constexpr (P::kind == P51) {
            constexpr uint64_t m = (1ull << 51) - 1;
            const uint64_t L = (uint64_t)v.lo * a.lo + (uint64_t)q.lo * b.lo;
            const uint64_t M = (uint64_t)v.lo * a.hi + (uint64_t)v.hi * a.lo + (uint64_t)q.lo * b.hi + (uint64_t)q.hi * b.lo;
            const uint64_t H = (uint64_t)v.hi * a.hi + (uint64_t)q.hi * b.hi;
            // 2^52 = 258, M 2^26 = 129 (M >> 25) + (M mod 2^25) 2^26 (mod p); the sum is below 2^61
            const uint64_t S = L + 258 * H + 129 * (M >> 25) + ((M & ((1ull << 25) - 1)) << 26);
            return (S & m) + 129 * (S >> 51);
        } else {
            const uint64_t s = (uint64_t)v.lo * a.lo + (uint64_t)q.lo * b.lo;
            if constexpr (P::kind == P31) {
                const uint64_t r = (s & P::p) + (s >> 31);  // < 2^34
                return (uint32_t)(r & P::p) + (uint32_t)(r >> 31);
            } else if constexpr (P::kind == P29) {
                const uint32_t r = (uint32_t)(s & ((1u << 29) - 1)) + 3u * (uint32_t)(s >> 29);  // < 2^32
                return (r & ((1u << 29) - 1)) + 3u * (r >> 29);
            } else {
                const uint32_t r = (uint32_t)(s & P::p) + (uint32_t)(s >> 19);  // < 2^22
                return (uint32_t)(r & P::p) + (r >> 19);
            }
        }
    }
};

// A value's f16 slots, 16 bytes at a time: limbs f as subnormals f 2^-24, and 1.0 in
// the last slot, the bias slot.  Bytes: the four bytes, three empty slots.  Nibbles:
// even and odd ones of the low word, then those of the high word with its top byte
// (bits 56 and up) among them.
template <int GEN>
struct TcLimbs {
    static constexpr bool kTwo = GmT<GEN>::p >= (1ull << 32);  // the second half varies (else: empty slots and 1.0)
    uint4 a, b;
    __device__ __forceinline__ TcLimbs() {}
    __device__ __forceinline__ explicit TcLimbs(uint64_t x)
    {
        const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
        if constexpr (!GmTc<GEN>::kNibbles) {
            a = make_uint4(__byte_perm(lo, 0, 0x4140), __byte_perm(lo, 0, 0x4342), 0, 0x3C000000u);
        } else {
            const uint32_t e = lo & 0x0F0F0F0Fu, o = (lo >> 4) & 0x0F0F0F0Fu;
            a = make_uint4(__byte_perm(e, 0, 0x4140), __byte_perm(e, 0, 0x4342), __byte_perm(o, 0, 0x4140), __byte_perm(o, 0, 0x4342));
            if constexpr (kTwo) {
                const uint32_t he = hi & 0x000F0F0Fu, ho = (hi >> 4) & 0x000F0F0Fu;  // (their top bytes are zero bytes to fill with)
                b = make_uint4(__byte_perm(he, 0, 0x3130), __byte_perm(he, hi, 0x3732), __byte_perm(ho, 0, 0x3130),
                               __byte_perm(ho, 0x3C000000u, 0x7332));
            }
        }
    }
    // into value v (0, 1) of a copy of A, at this thread's row
    __device__ __forceinline__ void store(unsigned char *row, int v) const
    {
        constexpr int kCol = GmTc<GEN>::kACol, kValue = GmTc<GEN>::kA / 2;
        *reinterpret_cast<uint4 *>(row + v * kValue) = a;
        if constexpr (kTwo) *reinterpret_cast<uint4 *>(row + v * kValue + kCol) = b;
    }
};

// Transpose a G x G matrix of VB-bit fields held one row per lane (G = 32 / VB
// lanes, field f at bit VB f): lane i's field f becomes lane f's field i.  A stage
// exchanges VB d bits with the lane d away: 16 and 8 bits by one byte permute, fewer
// by a rotation and a select; the lane's constants are kept in registers.
template <int VB>
struct TcTranspose {
    static constexpr int G = 32 / VB;
    uint32_t perm[2], keep[3], rot[3];
    __device__ __forceinline__ explicit TcTranspose(int lane)
    {
        constexpr uint32_t low[3] = { 0x0F0F0F0Fu, 0x33333333u, 0x55555555u };
        perm[0] = lane & (16 / VB) ? 0x3276u : 0x5410u;
        perm[1] = lane & (8 / VB) ? 0x3715u : 0x6240u;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int w = 4 >> k;
            const bool up = w >= VB && (lane & (w / VB));
            keep[k] = up ? ~low[k] : low[k];
            rot[k] = up ? 32 - w : w;
        }
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const
    {
        x = __byte_perm(x, __shfl_xor_sync(kFull, x, 16 / VB), perm[0]);
        x = __byte_perm(x, __shfl_xor_sync(kFull, x, 8 / VB), perm[1]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int w = 4 >> k;
            if (w < VB) break;
            const uint32_t y = __shfl_xor_sync(kFull, x, w / VB);
            x = (x & keep[k]) | (__funnelshift_l(y, y, rot[k]) & ~keep[k]);
        }
        return x;
    }
};

// What a point gathers over a half of a block: strips and the running minimum of the
// checks.  Column group g of half h is step 1 + 2 (31 - g) + h (v = 1), or step
// 1 + 32 h + 4 (7 - g % 8) + g / 8 (v = 4), so each register fills by funnel shifts
// from its top field down and ends with step 1 + 2 f + h in field f (v = 1), or step
// 1 + 32 h + 4 f + r in field f of register r (v = 4).
template <int GEN>
struct TcStrips {
    static constexpr int V = GmT<GEN>::v;
    uint32_t acc[GmTc<GEN>::kRegs];
    // v = 1: the smallest |t| with t read as an f32, whose sign is the output bit
    // and whose magnitude orders like the 31 bits below it (a NaN pattern is a
    // large value, and fminf drops it): one three-input minimum per two steps.
    // v = 4: the smallest t 2^4 mod 2^32.
    float lowf;
    uint32_t low;
    __device__ __forceinline__ bool near() const { return (V == 1 ? __float_as_uint(lowf) : low) < GmTc<GEN>::kNear; }
    template <int Q>  // the first or the last 16 groups
    __device__ __forceinline__ void take(const uint32_t (&d)[32])
    {
        if constexpr (Q == 0) {
            lowf = __int_as_float(0x7F800000);
            low = 0xFFFFFFFFu;
        }
        uint32_t t[16];
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            t[s] = d[2 * s] * (1u << 20) + d[2 * s + 1] * (1u << 8);
            const int r = V == 1 ? 0 : 2 * Q + s / 8;
            acc[r] = __funnelshift_l(t[s], acc[r], V);
        }
#pragma unroll
        for (int s = 0; s < 16; s += 2) {
            if constexpr (V == 1) lowf = fminf(fminf(lowf, fabsf(__uint_as_float(t[s]))), fabsf(__uint_as_float(t[s + 1])));
            else low = min(min(low, t[s] << V), t[s + 1] << V);
        }
    }
};

// Half h of the points in `near` (a ballot) again, exactly, from their X1 and X2: one
// point at a time, by the whole warp, lane j computing the half's j-th step.
template <int GEN>
__device__ __noinline__ uint4 tc_exact_half(const uint64_t *al_s, const uint64_t *be_s, uint32_t near, int h, uint4 acc, TcValue<GEN> v1, TcValue<GEN> v2)
{
    using P = GmT<GEN>;
    const int lane = threadIdx.x & 31;
    const int at = 2 + (P::v == 1 ? 2 * lane + h : kTcRow * h + lane);
    const uint64_t al = al_s[at], be = be_s[at];
    while (near) {
        const int l = __ffs(near) - 1;
        near &= near - 1;
        TcValue<GEN> a, b;
        a.lo = __shfl_sync(kFull, v1.lo, l); a.hi = __shfl_sync(kFull, v1.hi, l);
        b.lo = __shfl_sync(kFull, v2.lo, l); b.hi = __shfl_sync(kFull, v2.hi, l);
        const uint64_t x = gm_lin<GEN>(al, a.whole(), be, b.whole());
        uint4 r = make_uint4(0, 0, 0, 0);
        if constexpr (P::v == 1) {
            r.x = __ballot_sync(kFull, x >= (P::p + 1) / 2);
        } else {
            const uint32_t strip = gm_strip_insert<GEN, 0>((GmZ<GEN>)x, 0u);
#pragma unroll
            for (int k = 0; k < 4; ++k) {  // bit k of lane 4 f + u's strip: bit 4 f + k of register u
                const uint32_t bits = __ballot_sync(kFull, (strip >> k) & 1u);
                r.x |= (bits & 0x11111111u) << k;
                r.y |= ((bits >> 1) & 0x11111111u) << k;
                r.z |= ((bits >> 2) & 0x11111111u) << k;
                r.w |= ((bits >> 3) & 0x11111111u) << k;
            }
        }
        if (lane == l) acc = r;
    }
    return acc;
}

// A block's words to `to` (this lane's first word): w[half][register], `words` of them
// in the whole block, `first` the lane's first.  VEC: rows are aligned for stores of
// two (v = 1) or four (v = 4) elements.  (A block that ends early by vectors too: more
// registers' worth of code, GM55 65536 x 64 u32 24.9 to 26.9 us.)  Four doubles leave as one
// store: as two, half a sector each, they took 1.3 to 1.6 times as long into host memory
// (GQ58.4 4096 x 1000 f64 320 us, as one 209, staged by the other kernel 201).
template <int GEN, typename OutT, bool VEC>
__device__ __forceinline__ void tc_put(const uint32_t (&w)[2][GmTc<GEN>::kRegs], OutT *to, uint32_t words, uint32_t first)
{
    constexpr int V = GmT<GEN>::v;
    if (VEC && words == (uint32_t)kTcSteps) {
        if constexpr (V == 1) {
            store2<OutT>(to, Cvt<OutT>::f(w[0][0]), Cvt<OutT>::f(w[1][0]));
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h)
                store4_whole<OutT>(to + kTcRow * h, Cvt<OutT>::f(w[h][0]), Cvt<OutT>::f(w[h][1]), Cvt<OutT>::f(w[h][2]), Cvt<OutT>::f(w[h][3]));
        }
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int r = 0; r < GmTc<GEN>::kRegs; ++r) {
                const int at = V == 1 ? h : kTcRow * h + r;
                if (first + at < words) to[at] = Cvt<OutT>::f(w[h][r]);
            }
    }
}

// ------------------------------------------------------------------ sections
// Where a kernel's sections come from: tiles of kStreams sections of nearly equal
// length, `at` a section's place in its tile (0: the longest).

// A fill's: unit g is section g / nstreams of stream g % nstreams (in order, so only
// the last section of a stream is shorter).  units = nstreams x nsec < 2^32, seclen <
// 2^32.  The last section of a stream leaves its next state in state_out.
template <int GEN, typename OutT, bool VEC>
struct TcFill {
    using P = GmT<GEN>;
    static constexpr int S = P::s, N = GmTc<GEN>::kStreams;
    static constexpr bool kNextState = true;
    const uint64_t *state_in;
    uint64_t *state_out;
    uint64_t stride, nper, seclen;
    uint32_t nstreams, units;
    OutT *out;
    struct Section {
        uint64_t start = 0;
        uint32_t j = 0, len = 0;
    };
    __device__ __forceinline__ uint32_t tiles() const { return (units + N - 1) / N; }
    __device__ __forceinline__ Section section(uint32_t tile, int at) const
    {
        Section s;
        const uint32_t g = tile * N + at;
        if (g >= units) return s;
        const uint32_t sec = units == nstreams ? 0 : g / nstreams;
        s.j = g - sec * nstreams;
        s.start = sec * seclen;
        s.len = s.start < nper ? (uint32_t)min(seclen, nper - s.start) : 0u;
        return s;
    }
    __device__ __forceinline__ void load(const Section &s, int li, uint64_t &prev, uint64_t &cur) const
    {
        prev = cur = 0;
        if (!s.len) return;
        prev = state_in[(uint64_t)s.j * S + li];
        cur = state_in[(stride + s.j) * S + li];
    }
    __device__ __forceinline__ void advance(const uint64_t *jump, const Section &s, uint64_t &zc, uint64_t &zp) const
    {
        if (units != nstreams) gm_apply<GEN>(gm_pow_group<GEN, S, false>(jump, s.start, 0), zc, zp);
    }
    __device__ __forceinline__ unsigned char *row(const Section &s) const
    {
        return reinterpret_cast<unsigned char *>(out + s.j * nper + s.start);
    }
    __device__ __forceinline__ int form(const Section &) const { return 0; }
    __device__ __forceinline__ static uint32_t bytes(int) { return sizeof(OutT); }
    __device__ __forceinline__ static void put(const uint32_t (&w)[2][GmTc<GEN>::kRegs], unsigned char *to, uint32_t words, uint32_t first, int)
    {
        tc_put<GEN, OutT, VEC>(w, reinterpret_cast<OutT *>(to), words, first);
    }
    __device__ __forceinline__ bool ends(const Section &s) const { return s.len && s.start + s.len == nper; }
    __device__ __forceinline__ void next_state(const Section &s, int li, uint64_t zp, uint64_t zc) const
    {
        state_out[(uint64_t)s.j * S + li] = zp << P::t;
        state_out[(stride + s.j) * S + li] = zc << P::t;
    }
};

// A batch's: a tile is up to kStreams sections of one request, from the seeded base
// advanced by stream x L + the section's offset (an exponent of up to 128 bits).
template <int GEN>
struct TcBatch {
    using P = GmT<GEN>;
    static constexpr int S = P::s;
    static constexpr bool kNextState = false;
    const BatchTile *list;
    uint32_t n;
    const uint64_t *base;
    struct Section {
        uint64_t lo = 0, hi = 0;
        unsigned char *out = nullptr;
        uint32_t len = 0;
        int form = 0;
    };
    __device__ __forceinline__ uint32_t tiles() const { return n; }
    __device__ __forceinline__ Section section(uint32_t tile, int at) const
    {
        const BatchTile &T = list[tile];
        Section s;
        const uint64_t off = (uint64_t)at * T.seclen;
        if (off >= T.len) return s;
        s.len = (uint32_t)min((uint64_t)T.seclen, T.len - off);
        const uint64_t add = T.start + off, klo = T.stream * P::L_;
        s.lo = klo + add;
        s.hi = __umul64hi(T.stream, P::L_) + (s.lo < klo ? 1u : 0u);
        s.form = T.dtype + (T.flags & kTileVec ? 4 : 0);
        s.out = reinterpret_cast<unsigned char *>(T.out) + off * bytes(s.form);
        return s;
    }
    __device__ __forceinline__ void load(const Section &s, int li, uint64_t &prev, uint64_t &cur) const
    {
        prev = base[li];
        cur = base[S + li];
    }
    __device__ __forceinline__ void advance(const uint64_t *jump, const Section &s, uint64_t &zc, uint64_t &zp) const
    {
        gm_apply<GEN>(gm_pow_group<GEN, S, true>(jump, s.lo, s.hi), zc, zp);
    }
    __device__ __forceinline__ unsigned char *row(const Section &s) const { return s.out; }
    __device__ __forceinline__ int form(const Section &s) const { return s.form; }
    __device__ __forceinline__ static uint32_t bytes(int form) { return (form & 3) == PRAND_DTYPE_F64 ? 8 : 4; }
    __device__ __forceinline__ static void put(const uint32_t (&w)[2][GmTc<GEN>::kRegs], unsigned char *to, uint32_t words, uint32_t first, int form)
    {
        auto as = [&](auto *p) {
            using T = typename std::remove_pointer<decltype(p)>::type;
            if (form & 4) tc_put<GEN, T, true>(w, p, words, first);
            else tc_put<GEN, T, false>(w, p, words, first);
        };
        if ((form & 3) == PRAND_DTYPE_U32) as(reinterpret_cast<uint32_t *>(to));
        else if ((form & 3) == PRAND_DTYPE_F32) as(reinterpret_cast<float *>(to));
        else as(reinterpret_cast<double *>(to));
    }
    __device__ __forceinline__ bool ends(const Section &) const { return false; }
    __device__ __forceinline__ void next_state(const Section &, int, uint64_t, uint64_t) const {}
};

// ------------------------------------------------------------------ kernel
// Persistent blocks of 128 threads; a tile is kStreams sections (one per warp
// for v = 1, one per 8 lanes for v = 4), thread = point.  Per block of 64 steps a
// thread computes X2 while the product runs; then it writes the next
// block's limbs to A, finishes the previous block's words under the first load of
// columns, and takes the columns 16 steps at a time, each load under the arithmetic
// of the steps before.  The last of the four warps to have its columns in registers
// issues the next product, so no warp waits for a slower one but at the product
// itself.  The next block of a tile's last one is the next tile's first, so the
// tensor cores run on from tile to tile.  The strips are transposed across the
// lanes, so lane l ends with words 2 l and 2 l + 1 (v = 1) or words 4 i .. 4 i + 3 of
// either half of its stream's block (v = 4), and rows leave 256 or 128 bytes at a time.
// err: a word in host memory, set if a wait ran out (DevTables::wait_failed: the call
// reports it if it waits for the outputs, else the next one does).
template <int GEN, typename Src>
__device__ __forceinline__ void gm_tc_run(const GmTcTable *__restrict__ tab, const uint64_t *__restrict__ jump, const Src &src,
                                          volatile uint32_t *err)
{
    using P = GmT<GEN>;
    using C = GmTc<GEN>;
    using Val = TcValue<GEN>;
    constexpr int S = P::s, M = kTcSteps;         // lanes per stream, steps per block
    extern __shared__ __align__(128) unsigned char sm[];
    unsigned char *smB = sm;                      // B: the first half's columns, then the second's
    unsigned char *smA = sm + 2 * C::kImage;      // A: 16-byte columns of 128 rows
    __shared__ __align__(8) uint64_t mbar_s;      // the product is done
    __shared__ uint32_t count_s;                  // warps that have its columns
    __shared__ uint32_t late_s;                   // a wait was given up
    __shared__ uint32_t tmem_s;
    __shared__ uint64_t al_s[kTcCoefs], be_s[kTcCoefs];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, li = tid % S;
    const uint32_t mbar = tc_smem(&mbar_s), count = tc_smem(&count_s);
    unsigned char *myA = smA + (tid >> 3) * 128 + (tid & 7) * 16;

    for (int i = tid; i < 2 * C::kImage / 16; i += kTcThreads)
        reinterpret_cast<uint4 *>(smB)[i] = reinterpret_cast<const uint4 *>(&tab->image[i >= C::kImage / 16][0])[i % (C::kImage / 16)];
    if (tid < kTcCoefs) {
        al_s[tid] = tab->al[tid];
        be_s[tid] = tab->be[tid];
    }
    const uint64_t to_a = tab->a, to_b = tab->b;
    if constexpr (C::kNibbles && !TcLimbs<GEN>::kTwo) {
#pragma unroll
        for (int k = 0; k < 2; ++k) *reinterpret_cast<uint4 *>(myA + (2 * k + 1) * C::kACol) = make_uint4(0, 0, 0, 0x3C000000u);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(tc_smem(&tmem_s)), "n"(kTcTmem) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        count_s = 0;
        late_s = 0;
    }

    // X0 and X1 of a section from its stream's state (prev, cur) = (zm, zc)
    auto pair = [&](const typename Src::Section &sec, uint64_t &zc, uint64_t &zm) {
        uint64_t zp = reduce_prod<P::kind>(zm >> P::t, 0);
        zc = reduce_prod<P::kind>(zc >> P::t, 0);
        src.advance(jump, sec, zc, zp);
        zm = gm_lin<GEN>(to_a, zc, to_b, zp);
    };

    const uint32_t tiles = src.tiles();
    uint32_t tile = blockIdx.x;
    typename Src::Section sec = src.section(tile, tid / S);
    Val x0, x1;
    TcLimbs<GEN> limbs;
    {
        uint64_t zc, zm;
        src.load(sec, li, zm, zc);
        pair(sec, zc, zm);
        TcLimbs<GEN>(zc).store(myA, 0);
        limbs = TcLimbs<GEN>(zm);
        limbs.store(myA, 1);
        x0 = Val(zc);
        x1 = Val(zm);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_s;
    const uint32_t cols = tmem + ((uint32_t)(32 * warp) << 16);
    const uint64_t descA = tc_desc(tc_smem(smA), C::kACol, 128);
    const uint64_t descB = tc_desc(tc_smem(smB), 128, 16 * C::kSlots);
    auto issue = [&](bool go) { tc_mma<2 * kTcCols, C::kSlots>(go, tmem, descA, descB, mbar); };
    if (warp == 0) issue(lane == 0);
    const TcBlockStep<GEN> next_pair(tab->v, tab->q);
    const TcTranspose<P::v> transpose(lane);
    uint32_t parity = 0;
    bool dead = false;

    TcStrips<GEN> T[2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int r = 0; r < C::kRegs; ++r) T[h].acc[r] = 0;
    // the block whose strips are in T: where its words go (this lane's first), how many
    // it has, and in which form
    const uint32_t first = P::v == 1 ? 2 * lane : 4 * li;
    unsigned char *to = nullptr;
    uint32_t words = 0;
    int to_form = 0;
    auto emit = [&]() {
        uint32_t w[2][C::kRegs];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int r = 0; r < C::kRegs; ++r) w[h][r] = transpose(T[h].acc[r]);
        src.put(w, to, words, first, to_form);
    };

    int form = src.form(sec);
    unsigned char *o = src.row(sec) + first * src.bytes(form);
    uint32_t left = sec.len;       // outputs of the section not yet made
    bool ends = src.ends(sec);     // the stream's next state is due after them
    uint32_t next = 0;             // (in a tile's last block) the next tile, if any
    bool on = true;
    // One block; LAST: the tile's last one.
    auto block = [&](auto last_block) {
        constexpr bool LAST = decltype(last_block)::value;
        const uint64_t z2 = next_pair(x1, x0);
        const Val x2(z2);
        typename Src::Section nsec;
        uint64_t zc = 0, zm = 0;
        if constexpr (LAST) {
            next = tile + gridDim.x;
            on = next < tiles;
            if (on) {  // the next tile's states, on their way from here on
                nsec = src.section(next, tid / S);
                src.load(nsec, li, zm, zc);
            }
        }
        uint32_t d0[32], d1[32];
        tc_wait(mbar, parity, dead, err, &late_s);
        parity ^= 1u;
        tc_fence_after();
        tc_ld(d0, cols);
        if constexpr (!LAST) {
            limbs.store(myA, 0);
            limbs = TcLimbs<GEN>(z2);
            limbs.store(myA, 1);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        emit();
        tc_ld_wait(d0);
        tc_ld(d1, cols + 32);
        T[0].template take<0>(d0);
        tc_ld_wait(d1);
        tc_ld(d0, cols + 64);
        T[0].template take<1>(d1);
        tc_ld_wait(d0);
        tc_ld(d1, cols + 96);
        T[1].template take<0>(d0);
        tc_ld_wait(d1);
        // this block's words (none once the section has ended)
        to = o;
        to_form = form;
        words = min((uint32_t)M, left);
        left -= words;
        o += M * src.bytes(form);
        if constexpr (LAST) {
            if (on) {  // A: the next tile's first pair
                pair(nsec, zc, zm);
                TcLimbs<GEN>(zc).store(myA, 0);
                limbs = TcLimbs<GEN>(zm);
                limbs.store(myA, 1);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
        }
        // this warp's columns are in registers and its rows of A hold the next block
        tc_fence_before();
        __syncwarp();
        const uint32_t before = tc_count(lane == 0, count);
        T[1].template take<1>(d1);
        const bool issuer = lane == 0 && before == 3 && (!LAST || on);
        if (__any_sync(kFull, issuer)) issue(issuer);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t near = __ballot_sync(kFull, T[h].near() && (P::v == 1 ? h : kTcRow * h) < words);
            if (near) {
                uint4 e = make_uint4(T[h].acc[0], 0, 0, 0);
                if constexpr (P::v != 1) e = make_uint4(T[h].acc[0], T[h].acc[1], T[h].acc[2], T[h].acc[3]);
                e = tc_exact_half<GEN>(al_s, be_s, near, h, e, x1, x2);
                T[h].acc[0] = e.x;
                if constexpr (P::v != 1) { T[h].acc[1] = e.y; T[h].acc[2] = e.z; T[h].acc[3] = e.w; }
            }
        }
        if (Src::kNextState && ends && left == 0) {
            // the stream ends here for this fill: x^(n + words - 1), x^(n + words)
            src.next_state(sec, li, gm_lin<GEN>(al_s[words], x1.whole(), be_s[words], z2),
                           gm_lin<GEN>(al_s[words + 1], x1.whole(), be_s[words + 1], z2));
            ends = false;
        }
        if constexpr (LAST) {
            if (!on) return;
            tile = next;
            sec = nsec;
            form = src.form(sec);
            o = src.row(sec) + first * src.bytes(form);
            left = sec.len;
            ends = src.ends(sec);
            x0 = Val(zc);
            x1 = Val(zm);
        } else {
            x0 = x1;
            x1 = x2;
        }
    };
    while (on) {
        // (the tile's first section is its longest)
        for (uint32_t b = (src.section(tile, 0).len + M - 1) / M; b > 1; --b) block(std::false_type{});
        block(std::true_type{});
    }
    emit();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        // products of waits given up may still be on their way into the tensor memory: a second
        // more (by a word in shared memory: the threads' own state, kept to the end, cost
        // doubles 3 % by its registers)
        if (late_s)
            for (int i = 0; i < 1024; ++i) __nanosleep(1000000);
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "n"(kTcTmem) : "memory");
    }
}

template <int GEN, typename OutT, bool VEC>
__global__ void __launch_bounds__(kTcThreads, kTcCtas) gm_tc_kernel(const GmTcTable *__restrict__ tab,
                                                                   const uint64_t *__restrict__ jump,
                                                                   const __grid_constant__ TcFill<GEN, OutT, VEC> fill,
                                                                   volatile uint32_t *err)
{
    gm_tc_run<GEN>(tab, jump, fill, err);
}

template <int GEN>
__global__ void __launch_bounds__(kTcThreads, kTcCtas) gm_tc_batch_kernel(const GmTcTable *__restrict__ tab,
                                                                         const uint64_t *__restrict__ jump,
                                                                         const __grid_constant__ TcBatch<GEN> batch,
                                                                         volatile uint32_t *err)
{
    gm_tc_run<GEN>(tab, jump, batch, err);
}

}  // namespace prand
