// Host side of the GM/GQ ensembles: launches of the kernels of gm_impl.cuh and
// gm_tc.cuh, instantiated one translation unit per generator.
#pragma once
#include <algorithm>

#include "gm_tc.cuh"

namespace prand {

template <int GEN>
inline prand_status_t gm_build_table_t(uint64_t *tab, cudaStream_t st)
{
    gm_table_kernel<GEN><<<1, 32, 0, st>>>(tab);
    gm_window_kernel<GEN><<<kGmDigits, 256, 0, st>>>(tab);
    return launch_check();
}

inline unsigned gm_grid_for(uint64_t n, unsigned block) { return (unsigned)((n + block - 1) / block); }

// Streams from which a thread-per-stream fill takes its states through shared memory.
constexpr uint64_t kWholeStates = 64;

template <int GEN>
struct GmHost {
    static prand_status_t seed(const uint64_t *tab, uint64_t *base, uint64_t seed, const Variant &V, cudaStream_t st)
    {
        gm_seed_kernel<GEN><<<1, 32, 0, st>>>(tab, base, seed, V.D[0], V.D[1]);
        return launch_check();
    }
    static prand_status_t init(const uint64_t *tab, const uint64_t *base, uint64_t *state, uint64_t first, uint64_t n,
                               const Variant &V, cudaStream_t st)
    {
        gm_init_kernel<GEN><<<gm_grid_for(n, kGmInitThreads), kGmInitThreads, 0, st>>>(tab, base, state, first, n, V.L[0], V.L[1]);
        return launch_check();
    }
    static prand_status_t skip(const uint64_t *tab, uint64_t *state, uint64_t n, const U256 &off, cudaStream_t st)
    {
        const unsigned B = 128;
        gm_skip_kernel<GEN><<<gm_grid_for(n * GmT<GEN>::s, B), B, 0, st>>>(tab, state, n, off);
        return launch_check();
    }
    // Sections per stream: whole waves of the kernel's resident sections (warps, threads
    // or groups of lanes: cap), of at least min_len outputs, on multiples of `align`;
    // a section's fixed work is worth `fixed` outputs.
    static void pick(uint64_t nstreams, uint64_t nper, uint64_t cap, uint64_t align, uint64_t min_len, uint64_t fixed,
                     uint32_t *nsec, uint64_t *seclen)
    {
        split(nper, pick_nsec(nstreams, cap, nper / min_len, nper, fixed), align, nsec, seclen);
    }
    // About s sections, on multiples of `align`.
    static void split(uint64_t nper, uint64_t s, uint64_t align, uint32_t *nsec, uint64_t *seclen)
    {
        uint64_t len = (nper + s - 1) / s;
        len = (len + align - 1) / align * align;
        if (len == 0) len = align;
        *seclen = len;
        *nsec = (uint32_t)((nper + len - 1) / len);
        if (*nsec == 0) *nsec = 1;
    }
    // Sections per stream of a thread-per-stream fill, of at least 256 outputs; wave: the
    // threads of one block per SM.  An SM's blocks share its pipes, so a fill takes as long as
    // the SM with the most of them, whatever is resident: blocks per SM that come out whole,
    // and three of them where there is a choice (a step takes 1.37 times as long with three
    // as with two, 0.6 times with one).  A section's start is worth some 30 outputs.  GQ58.3,
    // u32, us: 86625 x 1000 by one section 608, by three 484; 2 x 11348014 (f32) by 44328 181, by
    // 38912 146.
    static uint64_t thread_sections(uint64_t nstreams, uint64_t nper, uint64_t wave)
    {
        const uint64_t max_s = std::min<uint64_t>(std::max<uint64_t>(nper / 256, 1), kMaxSections);
        uint64_t best = 1;
        double best_score = 0;
        auto consider = [&](uint64_t s) {
            if (s < 1 || s > max_s) return;
            const uint64_t units = nstreams * s, blocks = (units + wave - 1) / wave;
            const double shared = blocks == 1 ? 0.76 : blocks == 2 ? 0.91 : 1.0;
            const double score = shared * (double)units / (double)(blocks * wave) / (1.0 + 32.0 * (double)s / (double)nper);
            if (score > best_score) { best_score = score; best = s; }
        };
        for (uint64_t s = 1; s <= 16; ++s) consider(s);
        for (uint64_t k = 1; k <= 6; ++k) consider(k * wave / nstreams);
        consider(max_s);
        return best;
    }
    // Whether a fill goes to the tensor-core kernel (cap: its resident sections) or to
    // this file's other one.  By the work of a row: the tensor-core kernel
    // makes whole blocks of 64 outputs and spends 0.9 block's time per row besides, the
    // other one 14 outputs' time, and an output takes r / 100 times as long there, r from
    // both kernels over 1 to 10^6 rows of 8 to 400 outputs (us, other / this):
    //   8 points: r falls with the bytes of an output; with fewer streams than the other
    //     kernel has threads its time stays and this one's falls (`few`).  GM55 u32
    //     300000 x 48, x 40, 20000 x 32: 0.87, 1.02, 0.87; f64 300000 x 96, x 80, 20000 x
    //     40: 0.96, 1.17, 0.79; GQ58.4 f32 300000 x 128, x 100, 20000 x 48: 0.87, 1.11, 0.99
    //     (this / other).  In one wave the chain of steps counts, 300 ns each there.
    //   32 points: up to four waves the last, partly empty one counts and the lines are
    //     measured ones: GM61 2500 x 36 u32 10.4 us here, 7.3 there, 2432 x 80 10.5 / 8.5,
    //     3500 x 96 1.0, 5000 x 64 0.86; GM31 2432 x 128 9.6 / 8.5, 3500 x 112 1.0; GM29
    //     3500 x 700 30.7 / 25.0.  Beyond: GM61 65536 x 40 0.94, x 36 1.03; GM31 12345 x
    //     60, x 80 1.0, 1.02.
    // A fill of more than a wave into host memory is bound by the link, which takes the
    // lane-per-point kernel's rows (9728 at once, out of step) 1 to 2 % faster than this
    // one's 2432 (65536 x 1024 f32: GM61 1439 / 1459 us, GM31 1413 / 1442; stores of 4, 8
    // or 16 bytes per lane alike).
    template <typename OutT>
    static bool use_tc(uint64_t nstreams, uint64_t nper, uint64_t cap, bool host)
    {
        constexpr bool kF64 = std::is_same<OutT, double>::value, kF32 = std::is_same<OutT, float>::value;
        constexpr bool kGm61 = GEN == PRAND_GM61, kGm31 = GEN == PRAND_GM31 || GEN == PRAND_GQ58_1;
        const uint64_t row = (nper + kTcSteps - 1) / kTcSteps * kTcSteps + 56, other = nper + 14;
        const uint64_t waves = (nstreams + cap - 1) / cap;
        const bool nearly_full = 8 * nstreams > 7 * cap;  // (one wave)
        if constexpr (GmT<GEN>::v == 4) {
            if (waves == 1) return nper >= (GEN == PRAND_GQ58_4 && nearly_full ? 32 : 24);
            if (nper > 65536) return true;
            constexpr bool kGm55 = GEN == PRAND_GM55;
            constexpr uint64_t few = kF64 ? 11000 : 7300;
            // doubles: a block that ends early leaves by single ones
            const uint64_t cost = row + (kF64 && nper % kTcSteps ? 16 : 0);
            uint64_t r = kGm55 ? (kF64 ? 188 : kF32 ? 188 : 217) : (kF64 ? 150 : kF32 ? 146 : 162);
            if (nper % 4 && nper > 64) r += !kF64 ? r / 8 : kGm55 ? r * 2 / 7 : 0;  // the other kernel's rows by its threads' own stores
            return 100 * cost * nstreams < r * other * (nstreams + few);
        }
        if (waves == 1) {
            if (kGm61) return nper >= 88;
            return kGm31 && (nstreams < 8 ? nper >= 192 : nearly_full ? nper >= 256 || 100 * row < 125 * other : nper >= 120);
        }
        if (host) return false;
        if (nper > 65536) return true;
        if (kGm61) {
            if (waves == 2) return nper >= (4 * nstreams > 5 * cap ? 88 : 80);
            return nper >= (waves <= 4 ? 56 : 0) && 100 * row < (waves <= 4 ? 215 : waves <= 16 ? 222 : 240) * other;
        }
        if (kGm31) return nper >= (waves == 2 ? 112 : waves <= 4 ? 96 : 0) && 100 * row < 164 * other;
        return waves == 2 && 4 * nstreams > 5 * cap ? nper >= 2048 : 100 * row < 109 * other;
    }
    // A batch's tiles (plan_request) from the seeded base.
    static prand_status_t batch(const uint64_t *tab, const GmTcTable *tc, volatile uint32_t *failed, const BatchTile *tiles,
                                uint32_t n, const uint64_t *base, cudaStream_t st)
    {
        if constexpr (GmTc<GEN>::kUse) {
            if (*failed) return PRAND_ERR_TIMEOUT;
            const uint32_t ctas = (uint32_t)device_sm_count() * kTcCtas;
            gm_tc_batch_kernel<GEN><<<n < ctas ? n : ctas, kTcThreads, kTcSmem, st>>>(tc, tab, TcBatch<GEN>{ tiles, n, base }, failed);
            return launch_check();
        }
        return PRAND_ERR_ARG;  // not a generator of this form
    }
    template <typename OutT>
    static prand_status_t gen(const uint64_t *tab, const GmTcTable *tc, volatile uint32_t *failed, uint64_t *state,
                              uint64_t *spare, StreamRange &R, OutT *out, uint64_t nper, cudaStream_t st)
    {
        using P = GmT<GEN>;
        const unsigned B = 256;
        const uint64_t off = R.j0 * P::s;
        const uint64_t *sin = state + off;
        if constexpr (GmTc<GEN>::kUse) {
            const uint64_t ctas = (uint64_t)device_sm_count() * kTcCtas;
            // Into host memory the 8-point rows' single elements (outputs off its vectors of four,
            // ends of rows) are a third of the link's rate and less; where they are many, the
            // other kernel's staged rows (GM55 f64 68929 x 60 818 us, 236; 105 x 34250 690, 260),
            // which take its chain of up to 256 steps, 70 us.
            const bool single = R.host && GmT<GEN>::v == 4 && (uintptr_t)out % 16 == 0 && nper % RowFill<OutT>::E == 0 &&
                                (nper % 4 || nper % kTcSteps > nper / 4) &&
                                R.count * nper * sizeof(OutT) >= (16u << 10) * std::min<uint64_t>(nper, 256);
            if (!single && use_tc<OutT>(R.count, nper, ctas * GmTc<GEN>::kStreams, R.host)) {
                if (*failed) return PRAND_ERR_TIMEOUT;
                if (R.nsec == 0) pick(R.count, nper, ctas * GmTc<GEN>::kStreams, kTcSteps, 256, 256, &R.nsec, &R.seclen);
                const uint32_t nsec = R.nsec;
                const uint64_t seclen = R.seclen, units = R.count * nsec;
                if (units <= UINT32_MAX && seclen <= UINT32_MAX) {
                    uint64_t *sout = (nsec > 1 ? spare : state) + off;
                    // stores of two (v = 1) or four elements (sections start on multiples of 64)
                    constexpr uint64_t V = GmT<GEN>::v == 1 ? 2 : 4;
                    const bool vec = (uintptr_t)out % (sizeof(OutT) * V) == 0 && nper % V == 0;
                    const uint64_t tiles = (units + GmTc<GEN>::kStreams - 1) / GmTc<GEN>::kStreams;
                    const unsigned grid = (unsigned)(tiles < ctas ? tiles : ctas);
                    auto launch = [&](auto v) {
                        constexpr bool VEC = decltype(v)::value;
                        const TcFill<GEN, OutT, VEC> fill = { sin, sout, R.stride, nper, seclen, (uint32_t)R.count, (uint32_t)units, out };
                        gm_tc_kernel<GEN, OutT, VEC><<<grid, kTcThreads, kTcSmem, st>>>(tc, tab, fill, failed);
                    };
                    if (vec) launch(std::true_type{});
                    else launch(std::false_type{});
                    return launch_check();
                }
            }
        }
        if constexpr (P::lanes == 32) {
            if (R.nsec == 0) pick(R.count, nper, resident_threads<GEN>(gm_gen_kernel<GEN, OutT, true>) / 32, 128, 512, 128, &R.nsec, &R.seclen);
            const uint32_t nsec = R.nsec;
            const uint64_t seclen = R.seclen, nstreams = R.count;
            uint64_t *sout = (nsec > 1 ? spare : state) + off;
            // section starts are multiples of 128, so rows start 16-byte aligned
            // when the output is aligned and n_per_stream is a multiple of 4
            const bool vec = ((uintptr_t)out % (sizeof(OutT) == 8 ? 32 : 16)) == 0 && nper % 4 == 0;
            const unsigned grid = gm_grid_for(nstreams * nsec * 32, B);
            auto launch = [&](auto v, auto few) {
                gm_gen_kernel<GEN, OutT, decltype(v)::value, decltype(few)::value><<<grid, B, 0, st>>>(tab, sin, sout, nstreams, R.stride, nper, nsec, seclen, out);
            };
            auto by_vec = [&](auto few) {
                if (vec) launch(std::true_type{}, few);
                else launch(std::false_type{}, few);
            };
            if (gm_blocks_per_sm<GEN>() > 6 && grid <= 3 * (unsigned)device_sm_count()) by_vec(std::integral_constant<bool, (gm_blocks_per_sm<GEN>() > 6)>{});
            else by_vec(std::false_type{});
        } else {
            if (R.nsec == 0) split(nper, thread_sections(R.count, nper, (uint64_t)B * device_sm_count()), 32, &R.nsec, &R.seclen);
            const uint32_t nsec = R.nsec;
            const uint64_t seclen = R.seclen, nstreams = R.count;
            uint64_t *sout = (nsec > 1 ? spare : state) + off;
            const bool rows = staged_rows(out, nstreams, nper, nsec, seclen, 32, R.host, 512);
            const unsigned grid = gm_grid_for(nstreams * nsec, B);
            const bool whole = nsec == 1 && nstreams >= kWholeStates;
            auto launch = [&](auto kernel) { kernel<<<grid, B, 0, st>>>(tab, sin, sout, nstreams, R.stride, nper, nsec, seclen, out, whole); };
            // blocks per SM: two for long rows by own stores (GQ58.3's only where streams are whole)
            if (rows) launch(gmt_gen_kernel<GEN, OutT, true>);
            else if (nper < 32 || (GEN == PRAND_GQ58_3 && nsec > 1)) launch(gmt_gen_kernel<GEN, OutT, false>);
            else launch(gmt_gen_kernel<GEN, OutT, false, 2>);
        }
        return launch_check();
    }
};


// Per-generator entry points, instantiated one translation unit per generator.
#define PRAND_GM_INSTANTIATE(GEN, NAME)                                                                          \
    prand_status_t NAME##_table(uint64_t *tab, cudaStream_t st) { return gm_build_table_t<GEN>(tab, st); }      \
    prand_status_t NAME##_seed(const uint64_t *tab, uint64_t *base, uint64_t seed, const Variant &V,           \
                               cudaStream_t st)                                                               \
    {                                                                                                         \
        return GmHost<GEN>::seed(tab, base, seed, V, st);                                                     \
    }                                                                                                         \
    prand_status_t NAME##_init(const uint64_t *tab, const uint64_t *base, uint64_t *state, uint64_t first,     \
                               uint64_t n, const Variant &V, cudaStream_t st)                                 \
    {                                                                                                         \
        return GmHost<GEN>::init(tab, base, state, first, n, V, st);                                          \
    }                                                                                                         \
    prand_status_t NAME##_skip(const uint64_t *tab, uint64_t *state, uint64_t n, const U256 &off,             \
                               cudaStream_t st)                                                               \
    {                                                                                                         \
        return GmHost<GEN>::skip(tab, state, n, off, st);                                                     \
    }                                                                                                         \
    prand_status_t NAME##_batch(const DevTables *T, const BatchTile *tiles, uint32_t n, const uint64_t *base,   \
                                cudaStream_t st)                                                              \
    {                                                                                                         \
        return GmHost<GEN>::batch(T->gm[GEN - PRAND_GM19], T->gm_tc[GEN - PRAND_GM19], T->wait_failed, tiles,  \
                                  n, base, st);                                                               \
    }                                                                                                         \
    prand_status_t NAME##_gen(const DevTables *T, uint64_t *state, uint64_t *spare, StreamRange &R,            \
                              void *out, int dtype, uint64_t nper, cudaStream_t st)                            \
    {                                                                                                         \
        const uint64_t *tab = T->gm[GEN - PRAND_GM19];                                                        \
        const GmTcTable *tc = T->gm_tc[GEN - PRAND_GM19];                                                     \
        if (dtype == PRAND_DTYPE_U32)                                                                         \
            return GmHost<GEN>::template gen<uint32_t>(tab, tc, T->wait_failed, state, spare, R, (uint32_t *)out, nper, st); \
        if (dtype == PRAND_DTYPE_F32)                                                                         \
            return GmHost<GEN>::template gen<float>(tab, tc, T->wait_failed, state, spare, R, (float *)out, nper, st);  \
        return GmHost<GEN>::template gen<double>(tab, tc, T->wait_failed, state, spare, R, (double *)out, nper, st);    \
    }

}  // namespace prand
