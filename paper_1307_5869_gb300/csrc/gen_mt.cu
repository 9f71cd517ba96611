// MT19937 (Matsumoto & Nishimura 1998; Sec. 5.4): seeding, warp-cooperative
// generation and the polynomial jump-ahead of eq. (g_v).
//
// One warp owns one stream.  The 624-word state lives in shared memory and is
// twisted by the 32 lanes in the three dependency phases of the recurrence
// x_{t+624} = x_{t+397} ^ twist(x_t^u | x_{t+1}^l): words 0..226 read only old
// words, words 227..453 read words 0..226 of the new block, words 454..623 read
// words 227..396 of the new block (Table 5 uses 227 threads per stream for the
// same reason).  Each new word leaves tempered straight from registers, 32
// consecutive words per store instruction.
//
// State layout: stream j at state[j * 624 .. j * 624 + 623].  All streams of a
// handle share the position inside the current block (the handle's index), so
// the index is kept on the host.
//
// Jump (Sec. 5.4): A^v Y = g_v(A) Y = sum_i a_i A^(i-1) Y with g_v = x^v mod phi.
// With Y in window form (x_t..x_{t+623}), A^i Y is the window starting at
// x_{t+i}, so the sum is a sliding-window XOR over the stream's next 20560
// words, taken at the set coefficients of g_v (mt_jump_block).
#include <type_traits>

#include "mt_dev.cuh"

namespace prand {

constexpr int kMtWarpsPerBlock = 4;

// ------------------------------------------------------------------ seeding
// seed < 2^32: init_genrand(seed); wider seeds: init_by_array({lo32, hi32});
// PRAND_SEED_DEFAULT: init_genrand(5489).  One thread (the recurrence is serial).
__global__ void mt_seed_kernel(uint32_t *base, uint64_t seed)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    auto genrand_init = [&](uint32_t s) {
        base[0] = s;
        for (uint32_t i = 1; i < kMtN; ++i) base[i] = 1812433253u * (base[i - 1] ^ (base[i - 1] >> 30)) + i;
    };
    if (seed == PRAND_SEED_DEFAULT) { genrand_init(5489u); return; }
    if (seed <= 0xFFFFFFFFull) { genrand_init((uint32_t)seed); return; }
    const uint32_t key[2] = { (uint32_t)seed, (uint32_t)(seed >> 32) };
    genrand_init(19650218u);
    int i = 1, j = 0;
    for (int k = kMtN; k; --k) {
        base[i] = (base[i] ^ ((base[i - 1] ^ (base[i - 1] >> 30)) * 1664525u)) + key[j] + (uint32_t)j;
        ++i; ++j;
        if (i >= kMtN) { base[0] = base[kMtN - 1]; i = 1; }
        if (j >= 2) j = 0;
    }
    for (int k = kMtN - 1; k; --k) {
        base[i] = (base[i] ^ ((base[i - 1] ^ (base[i - 1] >> 30)) * 1566083941u)) - (uint32_t)i;
        ++i;
        if (i >= kMtN) { base[0] = base[kMtN - 1]; i = 1; }
    }
    base[0] = 0x80000000u;
}

// ------------------------------------------------------------------ generation
template <typename OutT>
__global__ void __launch_bounds__(32 * kMtWarpsPerBlock) mt_gen_kernel(uint32_t *state, uint64_t nstreams, uint32_t idx0,
                                                                       uint64_t nper, OutT *__restrict__ out)
{
    __shared__ uint32_t sm[kMtWarpsPerBlock][2][kMtN];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t j = (uint64_t)blockIdx.x * kMtWarpsPerBlock + w;
    if (j >= nstreams) return;  // whole warp
    uint32_t *b0 = sm[w][0], *b1 = sm[w][1];
    const uint32_t *src = state + j * kMtN;
    mt_copy_state_warp(src, b0, lane);
    __syncwarp();
    OutT *o = out + j * nper;
    uint64_t done = 0;
    // the rest of the current block
    if (idx0 < (uint32_t)kMtN) {
        const uint32_t cnt = (uint32_t)min((uint64_t)(kMtN - idx0), nper);
        for (uint32_t t = lane; t < cnt; t += 32) o[t] = Cvt<OutT>::f(mt_temper(b0[idx0 + t]));
        done = cnt;
    }
    // whole new blocks, each twisted once and emitted as it is made; the loop
    // is unrolled by two so both calls see fixed shared-memory buffers
    bool in_b0 = true;
    while (done < nper) {
        uint64_t rem = nper - done;
        uint32_t emit = rem < (uint64_t)kMtN ? (uint32_t)rem : (uint32_t)kMtN;
        mt_twist_emit<OutT>(b0, b1, lane, o + done, emit);
        done += emit;
        in_b0 = false;
        if (done >= nper) break;
        rem = nper - done;
        emit = rem < (uint64_t)kMtN ? (uint32_t)rem : (uint32_t)kMtN;
        mt_twist_emit<OutT>(b1, b0, lane, o + done, emit);
        done += emit;
        in_b0 = true;
    }
    const uint32_t *cur = in_b0 ? b0 : b1;
    uint32_t *dst = state + j * kMtN;
    mt_copy_state_warp(cur, dst, lane);
}

// Few streams: a block per stream, which makes each block of words in three rounds
// (mt_twist_emit_team) where one warp takes twenty steps: one stream of 10^6 u32 415 us
// (1376); short fills are bound by their call (96 x 1001 f32 4.1 us by calls in C, 5.7, but
// 6.6 and 6.7 from Python).  With six streams or more per SM the warps fill it by
// themselves (10^4 outputs of 608 streams 12.3 and 18.5 us, of 1216 20.5 and 20.5, of 2432
// 35.9 and 27.6).
constexpr int kMtGenTeam = 8;
constexpr uint64_t kMtTeamStreams = 6;

template <typename OutT>
__global__ void __launch_bounds__(32 * kMtGenTeam) mt_gen_team_kernel(uint32_t *state, uint32_t idx0, uint64_t nper, OutT *__restrict__ out)
{
    __shared__ uint32_t sm[2][kMtN];
    uint32_t *s = state + blockIdx.x * (uint64_t)kMtN;
    for (int i = threadIdx.x; i < kMtN; i += 32 * kMtGenTeam) sm[0][i] = s[i];
    __syncthreads();
    OutT *o = out + blockIdx.x * nper;
    uint64_t done = 0;
    if (idx0 < (uint32_t)kMtN) {  // the rest of the current block
        done = min((uint64_t)(kMtN - idx0), nper);
        for (uint32_t t = threadIdx.x; t < (uint32_t)done; t += 32 * kMtGenTeam) o[t] = Cvt<OutT>::f(mt_temper(sm[0][idx0 + t]));
    }
    int cur = 0;
    for (; done < nper; cur ^= 1) {
        const uint32_t emit = (uint32_t)min(nper - done, (uint64_t)kMtN);
        mt_twist_emit_team<OutT, kMtGenTeam>(sm[cur], sm[cur ^ 1], o + done, emit);
        done += emit;
    }
    for (int i = threadIdx.x; i < kMtN; i += 32 * kMtGenTeam) s[i] = sm[cur][i];
}

// ------------------------------------------------------------------ jump
// Blocks of 12 warps, four to an SM (40 registers): one wave holds 608 streams, and 65536
// streams take 17.4 ms (before the rounds of the next step's words were three instead of
// four: 18.2; 6 warps 18.1, 3 warps 21.5, 15 warps 19.7, 30 warps 28.0).  Few streams are
// latency, so each takes a cluster of blocks (kMtCluster): the first stream of a
// handle, a chain of one jump per set bit, 0.22 ms for nine jumps (one block 0.80,
// clusters of four 0.30; 15 or 30 warps a block the same), a level of up to 16 streams
// 26 us (90).
constexpr int kMtJumpWarps = 12;

// Doubling level: dst stream (off + j) := g(A) (src stream j), one block or cluster per stream.
template <int NW, int MB, int CS>
__global__ void __launch_bounds__(32 * NW, MB) mt_level_kernel(const uint32_t *poly, uint32_t *state, uint64_t off)
{
    __shared__ __align__(16) MtJumpSmem S;
    const uint64_t j = blockIdx.x / CS;
    for (int i = threadIdx.x; i < kMtN; i += 32 * NW) S.state[i] = state[j * kMtN + i];
    mt_jump_block<NW, CS>(S, poly);
    if (mt_cluster_rank<CS>() == 0)
        for (int i = threadIdx.x; i < kMtN; i += 32 * NW) state[(off + j) * kMtN + i] = S.state[i];
}

// Every stream advanced by the set bits of a 512-bit offset (one polynomial
// x^(2^b) mod phi per set bit b, applied one after another), one block or cluster per stream.
struct MtBits { uint64_t w[8]; };

template <int NW, int MB, int CS>
__global__ void __launch_bounds__(32 * NW, MB) mt_multi_kernel(const uint32_t *polys, uint32_t *state, MtBits e)
{
    __shared__ __align__(16) MtJumpSmem S;
    uint32_t *s = state + (uint64_t)(blockIdx.x / CS) * kMtN;
    for (int i = threadIdx.x; i < kMtN; i += 32 * NW) S.state[i] = s[i];
    for (int b = 0; b < 512; ++b)
        if ((e.w[b >> 6] >> (b & 63)) & 1u) mt_jump_block<NW, CS>(S, polys + (size_t)b * kMtPolyWords);
    // (every block of a cluster has read the state before the first jump's barrier)
    if (mt_cluster_rank<CS>() == 0)
        for (int i = threadIdx.x; i < kMtN; i += 32 * NW) s[i] = S.state[i];
}

// ------------------------------------------------------------------ host
static unsigned grid_warps(uint64_t n) { return (unsigned)((n + kMtWarpsPerBlock - 1) / kMtWarpsPerBlock); }

// One block per stream, or a cluster of them when every block then has an SM to itself.
template <typename... Args>
static prand_status_t mt_jump_launch(void (*block)(Args...), void (*cluster)(Args...), uint64_t n, cudaStream_t st, Args... args)
{
    if (n * kMtCluster > (uint64_t)device_sm_count()) {
        block<<<(unsigned)n, 32 * kMtJumpWarps, 0, st>>>(args...);
        return launch_check();
    }
    return mt_cluster_launch(cluster, (unsigned)n * kMtCluster, 32 * kMtJumpWarps, kMtCluster, st, args...);
}

prand_status_t mt_seed(uint64_t seed, void *d_base, cudaStream_t st)
{
    mt_seed_kernel<<<1, 32, 0, st>>>((uint32_t *)d_base, seed);
    return launch_check();
}

// streams j = 0..n-1 := base advanced by (first + j) * 2^shift (2^432 in the
// Table 4 layout): stream 0 by the bits of first, then a doubling tree
// (stream 2^b + j from stream j by 2^(shift + b)).
prand_status_t mt_init(const DevTables *T, const void *d_base, void *d_state, uint64_t first, uint64_t n, cudaStream_t st,
                       int shift)
{
    uint32_t *state = (uint32_t *)d_state;
    if (cudaMemcpyAsync(state, d_base, kMtN * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return PRAND_ERR_CUDA;
    if (first) {
        MtBits e = {};
        // first * 2^shift: bits shift .. shift + 63
        for (int b = 0; b < 64; ++b)
            if ((first >> b) & 1u) e.w[(shift + b) >> 6] |= 1ull << ((shift + b) & 63);
        prand_status_t s = mt_jump_launch(mt_multi_kernel<kMtJumpWarps, 4, 1>, mt_multi_kernel<kMtJumpWarps, 1, kMtCluster>, 1, st, (const uint32_t *)T->mt, state, e);
        if (s != PRAND_OK) return s;
    }
    for (int b = 0; b < 64 && (1ull << b) < n; ++b) {
        uint64_t have = 1ull << b;
        uint64_t count = min(have, n - have);
        prand_status_t s = mt_jump_launch(mt_level_kernel<kMtJumpWarps, 4, 1>, mt_level_kernel<kMtJumpWarps, 1, kMtCluster>, count, st,
                                          (const uint32_t *)T->mt + (size_t)(shift + b) * kMtPolyWords, state, have);
        if (s != PRAND_OK) return s;
    }
    return PRAND_OK;
}

// Skip ahead: consume the rest of the current block, then jump by polynomials.
// Every stream += off (512 bits, off < 2^512 as for the paper's a 2^b form):
// the rest of the current block is used up by moving the index, the remainder
// is one polynomial x^(2^b) mod phi per set bit.
prand_status_t mt_skip512(const DevTables *T, void *d_state, uint64_t n, uint32_t *idx, const uint64_t off_in[8],
                          cudaStream_t st)
{
    MtBits e = {};
    for (int i = 0; i < 8; ++i) e.w[i] = off_in[i];
    if (*idx < (uint32_t)kMtN) {
        uint64_t rem = kMtN - *idx;
        bool small = true;
        for (int i = 1; i < 8; ++i) small = small && !e.w[i];
        if (small && e.w[0] < rem) { *idx += (uint32_t)e.w[0]; return PRAND_OK; }
        uint64_t borrow = rem;
        for (int i = 0; i < 8 && borrow; ++i) {
            uint64_t before = e.w[i];
            e.w[i] -= borrow;
            borrow = before < borrow ? 1 : 0;
        }
        *idx = kMtN;
    }
    bool any = false;
    for (int i = 0; i < 8; ++i) any = any || e.w[i];
    if (!any) return PRAND_OK;
    return mt_jump_launch(mt_multi_kernel<kMtJumpWarps, 4, 1>, mt_multi_kernel<kMtJumpWarps, 1, kMtCluster>, n, st, (const uint32_t *)T->mt,
                          (uint32_t *)d_state, e);
}

prand_status_t mt_skip(const DevTables *T, void *d_state, uint64_t n, uint32_t *idx, const U256 &off, cudaStream_t st)
{
    const uint64_t w[8] = { off.w[0], off.w[1], off.w[2], off.w[3], 0, 0, 0, 0 };
    return mt_skip512(T, d_state, n, idx, w, st);
}

prand_status_t mt_gen(void *d_state, uint64_t nstreams, uint32_t *idx, void *out, int dtype, uint64_t nper, cudaStream_t st)
{
    uint32_t *state = (uint32_t *)d_state;
    const auto launch = [&](auto *o) {
        using OutT = std::remove_pointer_t<decltype(o)>;
        if (nstreams <= kMtTeamStreams * (uint64_t)device_sm_count())
            mt_gen_team_kernel<<<(unsigned)nstreams, 32 * kMtGenTeam, 0, st>>>(state, *idx, nper, o);
        else
            mt_gen_kernel<OutT><<<grid_warps(nstreams), 32 * kMtWarpsPerBlock, 0, st>>>(state, nstreams, *idx, nper, o);
    };
    if (dtype == PRAND_DTYPE_U32) launch((uint32_t *)out);
    else if (dtype == PRAND_DTYPE_F32) launch((float *)out);
    else launch((double *)out);
    prand_status_t s = launch_check();
    if (s != PRAND_OK) return s;
    // the index after nper outputs: the rest of the current block, then whole blocks
    uint64_t avail = kMtN - *idx;
    if (nper <= avail) *idx += (uint32_t)nper;
    else *idx = (uint32_t)((nper - avail - 1) % kMtN + 1);
    return PRAND_OK;
}

}  // namespace prand
