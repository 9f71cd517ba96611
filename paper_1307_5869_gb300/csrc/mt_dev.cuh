// Device routines of MT19937 (Matsumoto & Nishimura 1998; Sec. 5.4) shared by
// the per-handle kernels and the batched persistent kernel: the recurrence
// word, tempering, the fused twist-and-emit of one block, and the polynomial
// jump of eq. (g_v) applied by one block.
#pragma once
#include "devcommon.cuh"

namespace prand {

__device__ __forceinline__ uint32_t mt_recur(uint32_t xt, uint32_t xt1, uint32_t xt397)
{
    uint32_t y = (xt & 0x80000000u) | (xt1 & 0x7FFFFFFFu);
    return xt397 ^ (y >> 1) ^ ((y & 1u) ? 0x9908B0DFu : 0u);
}

// Copy one 624-word state with a warp: all of a lane's 20 loads are issued
// before any of its stores, so the copy costs one memory latency rather than
// twenty.  Each lane moves its own words (src and dst may be the same buffer).
__device__ __forceinline__ void mt_copy_state_warp(const uint32_t *src, uint32_t *dst, int lane)
{
    constexpr int R = (kMtN + 31) / 32;  // 20
    uint32_t r[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int i = lane + 32 * k;
        r[k] = i < kMtN ? src[i] : 0u;
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int i = lane + 32 * k;
        if (i < kMtN) dst[i] = r[k];
    }
}

__device__ __forceinline__ uint32_t mt_temper(uint32_t y)
{
    y ^= y >> 11;
    y ^= (y << 7) & 0x9D2C5680u;
    y ^= (y << 15) & 0xEFC60000u;
    y ^= y >> 18;
    return y;
}

// Twist of a whole block out of place (old block -> new block, both in shared
// memory) fused with the tempered output: every new word is tempered and
// stored straight from registers while it is written to the new block.  New
// word k reads old words k, k+1 (new word 0 for k = 623) and old word k + 397
// (k < 227) or new word k - 227 (k >= 227).  So the block is made in 20 chunks
// of 32 words in order.  The loop is unrolled completely so each chunk knows
// its case at compile time (only chunk 7 mixes the two partner sources and
// only chunk 19 is partly empty).  A word read from the new block was written
// at least seven chunks earlier, so a warp sync every fourth chunk orders
// every such read after its write.  Words k < emit are written to o[k]; FULL
// (emit == 624) drops that test.
template <typename OutT, bool FULL>
__device__ __forceinline__ void mt_twist_emit_chunks(const uint32_t *__restrict__ ob, uint32_t *__restrict__ nb,
                                                     int lane, OutT *o, uint32_t emit)
{
#pragma unroll
    for (int c = 0; c < 20; ++c) {
        const int k = 32 * c + lane;
        if (c < 19 || lane < kMtN - 32 * 19) {
            const uint32_t a = ob[k];
            const uint32_t b = (c < 19 || lane < kMtN - 32 * 19 - 1) ? ob[k + 1] : nb[0];
            const uint32_t p = c < 7 ? ob[k + 397] : c > 7 ? nb[k - 227] : (lane < 3 ? ob[k + 397] : nb[k - 227]);
            const uint32_t x = mt_recur(a, b, p);
            nb[k] = x;
            if (FULL || (uint32_t)k < emit) o[k] = Cvt<OutT>::f(mt_temper(x));
        }
        if ((c & 3) == 3) __syncwarp();
    }
}

// The same twist by a team of TEAM warps that make up the whole block, in rounds of 227
// words (or of one per thread): a word reads new words 227 or more before it, i.e. from
// earlier rounds, so one block barrier per round orders every such read after its
// write; the last one publishes the new block.  All TEAM warps call it.
template <typename OutT, int TEAM>
__device__ __forceinline__ void mt_twist_emit_team(const uint32_t *__restrict__ ob, uint32_t *__restrict__ nb, OutT *o,
                                                   uint32_t emit)
{
    constexpr int ROUND = 32 * TEAM < kMtN - kMtM ? 32 * TEAM : kMtN - kMtM;
#pragma unroll
    for (int a = 0; a < kMtN; a += ROUND) {
        const int k = a + threadIdx.x;
        if (threadIdx.x < ROUND && k < kMtN) {
            const uint32_t nxt = k + 1 < kMtN ? ob[k + 1] : nb[0];
            const uint32_t p = k < kMtN - kMtM ? ob[k + kMtM] : nb[k - (kMtN - kMtM)];
            const uint32_t x = mt_recur(ob[k], nxt, p);
            nb[k] = x;
            if ((uint32_t)k < emit) o[k] = Cvt<OutT>::f(mt_temper(x));
        }
        __syncthreads();
    }
}

template <typename OutT>
__device__ __forceinline__ void mt_twist_emit(const uint32_t *__restrict__ ob, uint32_t *__restrict__ nb, int lane,
                                              OutT *o, uint32_t emit)
{
    if (emit >= (uint32_t)kMtN) mt_twist_emit_chunks<OutT, true>(ob, nb, lane, o, emit);
    else mt_twist_emit_chunks<OutT, false>(ob, nb, lane, o, emit);
}

// ------------------------------------------------------------------ jump
// state := g(A) state for one stream, by one block (eq. (g_v)).
//
// With the state in window form x_0..x_623, A^i of it is the window x_i..x_{i+623}, so
// result word m is R_m = sum over the set coefficients g_i of x_{i+m} over GF(2): a
// product of a Toeplitz matrix with the coefficient vector.  It is split once in the
// manner of Karatsuba.  Take coefficients and results in blocks of K = 320 (two blocks
// of results, the last 16 unused); with G_q the q-th block of coefficients and
// G_q * X_s the K results sum_r g_{Kq+r} x_{Ks+r+m}, a pair q, q + 1 (q even) adds
//   to results 0..319:    G_q * X_q     + G_{q+1} * X_{q+1} = A + B
//   to results 320..639:  G_q * X_{q+1} + G_{q+1} * X_{q+2} = A + C
// with A = (G_q + G_{q+1}) * X_{q+1}, B = G_q * Y_q, C = G_{q+1} * Y_{q+1} and
// Y_s = X_s + X_{s+1}, i.e. y_i = x_i ^ x_{i+320}: three products of half the size each
// way instead of four.
//
// One warp computes (a share of the coefficients of) one of the three products: lane l
// owns the W = 10 consecutive results from 10 l, and keeps the sequence words from
// there on in registers as a window that slides by four words per group of four
// coefficients (two 8-byte shared-memory loads, free of bank conflicts at this stride).
// A group costs, per result, 1.25 logic operations on average over its 16 patterns of
// coefficients (0, 1 or 2 three-input XORs), selected by a tree of branches that are
// uniform over the warp.  The window's P = 16 registers come round every 16
// coefficients, so the loop is unrolled over a chunk of 16; wider windows are slower,
// because the 16 patterns of every group of the chunk no longer fit the instruction
// caches (21 results per lane and groups of four: 30 KB of code, warps stalled on
// instruction fetch for half of the time).
// The block goes through the coefficients in steps of one pair (640): the next step's
// 640 sequence words are made by the whole block (a word needs the one 227 before it,
// so three rounds of 227) into the other buffer, then every warp takes its share of
// the step.
//
// Bound by instruction issue: 32 steps x 3 products x 80 groups per stream, each 12.5
// logic operations (two-cycle ones: 5.4 ms of the ALU pipe for 32768 streams), two loads
// and about 20 instructions of branches, uniform tests and moves.  32768 streams: 8.4 ms
// (82 % of the issue slots), where one warp per stream over the unsplit sum, in groups of
// two coefficients, took 12.7 ms; one stream alone 85 us with 12 warps and 24 us by a
// cluster of eight blocks, where that took 670 us.  Groups of two coefficients 10.1 ms; a
// switch instead of the tree 8.7 ms; branches the compiler does not know to be uniform
// 9.7 ms.
constexpr int kMtK = 320, kMtStep = 2 * kMtK, kMtSteps = (kMtDeg + kMtStep - 1) / kMtStep;  // 32 steps
constexpr int kMtW = 10, kMtP = 16, kMtG = 4;
constexpr int kMtCluster = 8;  // blocks per stream when the streams are few

struct MtJumpSmem {
    uint32_t x[2][2 * kMtStep];       // x_{640 Q} .. x_{640 Q + 1279} of step Q, in buffer Q & 1
    uint32_t y[2][3 * kMtK];          // y_i = x_i ^ x_{i + 320}
    uint32_t poly[kMtStep / 32 * kMtSteps];
    uint32_t state[kMtStep];
};

template <int U, int BIT, int PAT>
__device__ __forceinline__ void mt_poly_tree(uint32_t bits, uint32_t (&acc)[kMtW], const uint32_t (&x)[kMtP])
{
    if constexpr (BIT >= 0) {
        if (bits & (1u << (U + BIT))) mt_poly_tree<U, BIT - 1, PAT | (1 << BIT)>(bits, acc, x);
        else mt_poly_tree<U, BIT - 1, PAT>(bits, acc, x);
    } else if constexpr (PAT != 0) {
#pragma unroll
        for (int j = 0; j < kMtW; ++j)
#pragma unroll
            for (int t = 0; t < kMtG; ++t)
                if ((PAT >> t) & 1) acc[j] ^= x[(U + j + t) % kMtP];
    }
}

template <int U>
__device__ __forceinline__ void mt_poly_groups(uint32_t bits, const uint32_t *run, uint32_t (&acc)[kMtW], uint32_t (&x)[kMtP])
{
    if constexpr (U < kMtP) {
#pragma unroll
        for (int t = 0; t < kMtG; t += 2) {  // words U + 10 .. U + 13; the last is ahead of its use
            const uint2 v = *reinterpret_cast<const uint2 *>(run + U + kMtW + t);
            x[(U + kMtW + t) % kMtP] = v.x;
            x[(U + kMtW + t + 1) % kMtP] = v.y;
        }
        mt_poly_tree<U, kMtG - 1, 0>(bits, acc, x);
        mt_poly_groups<U + kMtG>(bits, run, acc, x);
    }
}

// Barrier over the CS blocks of a cluster (the block alone for CS = 1), and a word of a
// shared variable of one of its blocks.
template <int CS>
__device__ __forceinline__ void mt_cluster_sync()
{
    if constexpr (CS == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
template <int CS>
__device__ __forceinline__ uint32_t mt_cluster_rank()
{
    uint32_t r = 0;
    if constexpr (CS > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
template <int CS>
__device__ __forceinline__ uint32_t mt_cluster_word(const uint32_t *p, uint32_t rank)
{
    if constexpr (CS == 1) {
        return *p;
    } else {
        uint32_t at, v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
        return v;
    }
}

// All 32 NW threads of the block call it, and of all CS blocks of the cluster: each takes
// a run of the steps (making the words before it on its own), the parts are summed
// through distributed shared memory, and every block ends with the new state.
// S.state holds the state before and after (a barrier at the end publishes it).
// poly: g's 624 coefficient words.  NW is a multiple of 3 whose third divides the 20
// chunks of a block of coefficients.
template <int NW, int CS = 1>
__device__ __forceinline__ void mt_jump_block(MtJumpSmem &S, const uint32_t *__restrict__ poly)
{
    constexpr int NT = 32 * NW, SHARE = kMtK / (NW / 3), ROUND = NT < 227 ? NT : 227;
    static_assert(NW % 3 == 0 && SHARE * (NW / 3) == kMtK && SHARE % kMtP == 0, "shares of whole chunks");
    static_assert(kMtSteps % CS == 0, "whole steps per block");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int role = warp % 3, c0 = SHARE * (warp / 3);
    const int q0 = kMtSteps / CS * (int)mt_cluster_rank<CS>(), q1 = q0 + kMtSteps / CS;
    __syncthreads();  // S.state written by the caller, or by the last jump
    for (int i = tid; i < kMtN; i += NT) S.x[0][i] = S.state[i];
    for (int i = tid; i < (int)(sizeof(S.poly) / 4); i += NT) S.poly[i] = i < kMtPolyWords ? poly[i] : 0u;
    __syncthreads();
    for (int i = tid; i < kMtStep; i += NT) S.state[i] = 0;
    for (int a = kMtN; a < 2 * kMtStep; a += ROUND) {  // the rest of the first step's words
        const int n = a + tid;
        if (tid < ROUND && n < 2 * kMtStep)
            S.x[0][n] = mt_recur(S.x[0][n - kMtN], S.x[0][n - kMtN + 1], S.x[0][n - (kMtN - kMtM)]);
        __syncthreads();
    }
    // the words of step Q + 1 from those of step Q (each other's buffer): the first 640 are
    // step Q's last, and the first round of the others reads those where they are
    auto advance = [&](int Q) {
        const uint32_t *ob = S.x[Q & 1] + kMtStep;
        uint32_t *nb = S.x[(Q & 1) ^ 1];
        if (tid < ROUND) nb[kMtStep + tid] = mt_recur(ob[kMtStep - kMtN + tid], ob[kMtStep - kMtN + 1 + tid], ob[kMtStep - (kMtN - kMtM) + tid]);
        for (int i = tid; i < kMtStep; i += NT) nb[i] = ob[i];
        __syncthreads();
#pragma unroll 1
        for (int a = kMtStep + ROUND; a < 2 * kMtStep; a += ROUND) {
            const int n = a + tid;
            if (tid < ROUND && n < 2 * kMtStep) nb[n] = mt_recur(nb[n - kMtN], nb[n - kMtN + 1], nb[n - (kMtN - kMtM)]);
            __syncthreads();
        }
    };
    auto sums = [&](int b) {
        for (int i = tid; i < 3 * kMtK; i += NT) S.y[b][i] = S.x[b][i] ^ S.x[b][i + kMtK];
    };
    if constexpr (CS > 1) {
#pragma unroll 1
        for (int Q = 0; Q < q0; ++Q) advance(Q);
    }
    sums(q0 & 1);
    uint32_t acc[kMtW], x[kMtP];
#pragma unroll
    for (int j = 0; j < kMtW; ++j) acc[j] = 0;
#pragma unroll 1
    for (int Q = q0; Q < q1; ++Q) {
        const int b = Q & 1;
        __syncthreads();  // this step's words are written; buffer b ^ 1 is read no more
        if (Q + 1 < q1) {
            advance(Q);
            sums(b ^ 1);
        }
        // coefficients 640 Q + (320 for C) + c, c0 <= c < c1, none past the polynomial's end
        const int left = kMtDeg - (kMtStep * Q + (role == 2 ? kMtK : 0));
        const int c1 = min(c0 + SHARE, left);
        const uint32_t *run = (role == 0 ? S.x[b] + kMtK : role == 1 ? S.y[b] : S.y[b] + kMtK) + c0 + kMtW * lane;
        const uint32_t *g = S.poly + (kMtStep / 32) * Q;
#pragma unroll
        for (int j = 0; j < kMtW; j += 2) {
            const uint2 v = *reinterpret_cast<const uint2 *>(run + j);
            x[j] = v.x;
            x[j + 1] = v.y;
        }
#pragma unroll 1
        for (int c = c0; c < c1; c += kMtP) {
            uint32_t bits = role < 2 ? g[c >> 5] : 0u;
            if (role != 1) bits ^= g[(kMtK + c) >> 5];
            // (a reduction's result is uniform to the compiler, and so are the branches on it)
            bits = __reduce_or_sync(kFull, bits >> (c & 16));
            mt_poly_groups<0>(bits, run, acc, x);
            run += kMtP;
        }
    }
#pragma unroll
    for (int j = 0; j < kMtW; ++j) {  // (result 640 and on do not exist: 320 + 319 is the last)
        if (role != 2) atomicXor(&S.state[kMtW * lane + j], acc[j]);
        if (role != 1) atomicXor(&S.state[kMtK + kMtW * lane + j], acc[j]);
    }
    mt_cluster_sync<CS>();
    if constexpr (CS > 1) {
        constexpr int R = (kMtN + NT - 1) / NT;
        uint32_t sum[R] = {};
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (tid + NT * r < kMtN)
                for (uint32_t k = 0; k < CS; ++k) sum[r] ^= mt_cluster_word<CS>(&S.state[tid + NT * r], k);
        mt_cluster_sync<CS>();  // every block has read every part
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (tid + NT * r < kMtN) S.state[tid + NT * r] = sum[r];
        __syncthreads();
    }
}

// Launch of a kernel whose blocks are in clusters of CS.
template <typename... Args>
inline prand_status_t mt_cluster_launch(void (*kernel)(Args...), unsigned blocks, unsigned threads, unsigned cs, cudaStream_t st, Args... args)
{
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeClusterDimension;
    a.val.clusterDim.x = cs;
    a.val.clusterDim.y = a.val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(blocks);
    c.blockDim = dim3(threads);
    c.stream = st;
    c.attrs = &a;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, args...) == cudaSuccess ? launch_check() : PRAND_ERR_CUDA;
}

}  // namespace prand
