// Batched generation: thousands of requests (generator, stream index, length,
// element type, output pointer) of mixed generators and uneven lengths in one
// persistent launch, with each request's jump-ahead (block splitting, Table 4,
// plus the offset of its section) fused in front of its generation.
//
// Work unit: a tile, run by one warp.  MRG32K3A / LFSR113 tiles are up to 32
// sections of one request (one lane each, rows written through the staged
// 128-byte row stores); GQ58.3 tiles likewise; the other GM/GQ requests go to the
// tensor-core kernels in tiles of 4 or 16 sections (in the server, whose tiles start
// from state slots, to tiles of up to 32 / lanes sections); MT19937 tiles are one whole request (the jump is a chain of
// polynomial applications by the warp, Sec. 5.4).  Warps claim tiles from an
// atomic counter, so short and long tiles balance across the GPU; tiles are
// ordered longest first.
//
// The same kernel serves the resident-stream server: a tile may start from a
// state slot instead of the seeded base, and the tile that ends a request
// writes the stream's next state back to its slot.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "batch_kernel.cuh"

namespace prand {

constexpr int kBatchThreads = 64;  // the wide build: small blocks (a warp on a long tile holds little besides itself)

// One MT19937 stream for the per-request form: stream k = base advanced by
// k 2^432, one window polynomial per nonzero byte of k (the same jump the
// batched MT19937 tiles take), by one block.
__global__ void __launch_bounds__(32 * kMtTeam) mt_window_init_kernel(const uint32_t *base, const uint32_t *win, uint64_t k,
                                                                      uint32_t *dst)
{
    __shared__ __align__(16) MtJumpSmem S;
    for (int i = threadIdx.x; i < kMtN; i += 32 * kMtTeam) S.state[i] = base[i];
    for (int i = 0; i < kMtWinPositions; ++i) {
        const uint32_t d = (uint32_t)(k >> (kMtWinBits * i)) & (uint32_t)(kMtWinDigits - 1);
        if (d) mt_jump_block<kMtTeam>(S, win + ((size_t)i * kMtWinDigits + d) * kMtPolyWords);
    }
    for (int i = threadIdx.x; i < kMtN; i += 32 * kMtTeam) dst[i] = S.state[i];
}


// ------------------------------------------------------------------ host: engine
namespace {

size_t esize(int dtype) { return dtype == PRAND_DTYPE_F64 ? 8 : 4; }

struct Engine {
    int device = -1;
    DevTables *T = nullptr;
    std::mutex bases_mu;
    std::vector<BasesRef> bases;  // small cache, most recent last
    BatchTile *d_tiles = nullptr;
    size_t d_cap = 0;
    BatchTile *h_tiles = nullptr;  // pinned staging
    size_t h_cap = 0;
    cudaEvent_t staged = nullptr;  // the last copy out of h_tiles
    cudaEvent_t done = nullptr;    // the last batch on d_tiles, d_counter and br
    uint32_t *d_counter = nullptr;
    BatchParams params;
    int sms = 1, blocks_per_sm[kModes] = { 1, 1, 1 };  // the wide build's (the others keep their own)
    int mt_team_bps = 1;                               // MT19937 build: a team of warps per tile
    int rest_bps[kRestVariants] = { 1, 1, 1, 1 };      // the rest build's variants
    Branches br;                                  // side branches of mixed launches
    std::mutex run_mu;  // one call of prand_batch_run at a time uses the buffers, the events and br
    std::atomic<bool> ready{ false };
};

constexpr int kMaxDev = 64;
Engine *const g_eng = new Engine[kMaxDev];  // never destroyed: its device memory may outlive CUDA at exit
std::mutex g_eng_mu;

// A device's engine: set up by the first call, under the lock, for any number of threads.
// What a failed set-up has made is kept for the next attempt.
prand_status_t engine_set_up(Engine &E, int dev)
{
    std::lock_guard<std::mutex> lk(g_eng_mu);
    if (E.ready.load(std::memory_order_relaxed)) return PRAND_OK;
    E.device = dev;
    prand_status_t s = get_tables(PRAND_MT19937, &E.T);
    if (s != PRAND_OK) return s;
    if (!E.d_counter && !dev_alloc(&E.d_counter, 64)) { E.d_counter = nullptr; return PRAND_ERR_NOMEM; }
    for (cudaEvent_t *e : { &E.staged, &E.done })
        if (!*e && cudaEventCreateWithFlags(e, cudaEventDisableTiming) != cudaSuccess) { *e = nullptr; return PRAND_ERR_CUDA; }
    E.sms = device_sm_count();
    {
        int bps = 0;
        const cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, batch_kernel<kModeWide, kBatchThreads, 128>, kBatchThreads, 0);
        E.blocks_per_sm[kModeWide] = (e == cudaSuccess && bps >= 1) ? bps : 1;
    }
    for (int v = 0; v < kRestVariants; ++v) E.rest_bps[v] = rest_blocks_per_sm(v);
    {
        int bps = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &bps, batch_kernel<kModeMt, 32 * kMtTeam, 128>, 32 * kMtTeam, 0);
        E.mt_team_bps = (e == cudaSuccess && bps >= 1) ? bps : 1;
    }
    if (E.br.create() != PRAND_OK) { E.br.destroy(); return PRAND_ERR_CUDA; }
    const char *path = getenv("PRAND_TUNE_CACHE");
    if (path) {
        FILE *f = fopen(path, "r");
        if (f) {
            unsigned a = 0, b = 0, c = 0, d = 0;
            if (fscanf(f, "{\"seclen_mrg_lfsr\": %u, \"seclen_gm\": %u, \"block\": %u, \"row_bytes\": %u", &a, &b,
                       &c, &d) == 4 && a && b && a % 4 == 0 && b % 4 == 0 && (c == 64 || c == 128) &&
                (d == 128 || d == 256)) {
                E.params.seclen_mrg_lfsr = a;
                E.params.seclen_gm = b;
                E.params.block = c;
                E.params.row_bytes = d;
            }
            fclose(f);
        }
    }
    E.ready.store(true, std::memory_order_release);
    return PRAND_OK;
}

prand_status_t engine_get(Engine **out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return PRAND_ERR_CUDA;
    Engine &E = g_eng[dev];
    if (!E.ready.load(std::memory_order_acquire)) {
        const prand_status_t s = engine_set_up(E, dev);
        if (s != PRAND_OK) return s;
    }
    *out = &E;
    return PRAND_OK;
}

// Base states of all eleven generators for one seed (computed on the device).  The
// cache keeps the last four seeds'; what was handed out stays until its last user (a
// plan, a server, a call under way) lets go of it.
prand_status_t engine_bases(Engine &E, uint64_t seed, cudaStream_t st, BasesRef *out)
{
    BasesRef dropped;  // freed after the lock is: cudaFree waits for the device, and so for batches that read it
    std::lock_guard<std::mutex> lk(E.bases_mu);
    for (const BasesRef &b : E.bases)
        if (b->seed == seed) { *out = b; return PRAND_OK; }
    const std::shared_ptr<SeedBases> B = std::make_shared<SeedBases>();
    B->seed = seed;
    size_t total = 0;
    for (int g = 0; g < PRAND_NUM_GENERATORS; ++g) {
        B->off[g] = total;
        total += (state_bytes_per_stream(g) + 255) & ~(size_t)255;
    }
    if (!dev_alloc(&B->dev, total)) { B->dev = nullptr; return PRAND_ERR_NOMEM; }
    prand_status_t s = PRAND_OK;
    for (int g = 0; g < PRAND_NUM_GENERATORS && s == PRAND_OK; ++g) {
        void *p = (char *)B->dev + B->off[g];
        if (g == PRAND_MT19937) s = mt_seed(seed, p, st);
        else if (is_gm(g)) { Variant V; variant_params(g, 0, &V); s = gm_seed(g, E.T, seed, V, p, st); }
        else s = mrg_lfsr_seed(g, seed, p, st);
    }
    // wait once, so later batches on any stream see the bases
    if (s == PRAND_OK && cudaStreamSynchronize(st) != cudaSuccess) s = PRAND_ERR_CUDA;
    if (s != PRAND_OK) return s;
    if (E.bases.size() >= 4) {
        dropped = std::move(E.bases.front());
        E.bases.erase(E.bases.begin());
    }
    E.bases.push_back(B);
    *out = B;
    return PRAND_OK;
}

}  // namespace

SeedBases::~SeedBases()
{
    if (dev) cudaFree(dev);
}

prand_status_t batch_ctx(uint64_t seed, cudaStream_t st, BatchCtx *ctx, BasesRef *bases, DevTables **T)
{
    Engine *E;
    prand_status_t s = engine_get(&E);
    if (s != PRAND_OK) return s;
    if ((s = engine_bases(*E, seed, st, bases)) != PRAND_OK) return s;
    memset(ctx, 0, sizeof *ctx);
    ctx->mrg_tab = E->T->mrg;
    ctx->lfsr_tab = E->T->lfsr;
    ctx->mt_polys = E->T->mt;
    if ((s = get_mt_window(E->T)) != PRAND_OK) return s;
    ctx->mt_win = E->T->mt_win;
    for (int g = 0; g < 8; ++g) ctx->gm_tab[g] = E->T->gm[g];
    for (int g = 0; g < PRAND_NUM_GENERATORS; ++g) ctx->base[g] = (const char *)(*bases)->dev + (*bases)->off[g];
    if (T) *T = E->T;
    return PRAND_OK;
}

BatchParams batch_params()
{
    Engine *E;
    if (engine_get(&E) != PRAND_OK) return BatchParams();
    return E->params;
}

// Split one request into tiles (appended to `out`).  from_slot: continue the
// state in `slot`; else start from the seeded base advanced to the request's
// stream.  wslot >= 0: the request's last tile writes the next state there.
// Section length (outputs per lane) of r's tiles: the tuned default, made
// longer for long requests so that r yields at most max_tiles tiles (a
// multiple of 128 outputs).
// The thread-per-section GM/GQ tiles: at most kWideSection.  A step of theirs is 8 or 12
// points' work of one thread, so a section is long in time, and its start costs 16
// products: 10^4 mixed requests, GQ58.3 alone, 1.38 ms at 2048, 0.84 at 1024, 0.58 at
// 512 and 256; 100 requests without MT19937 0.59, 0.35, 0.32, 0.32 ms.
constexpr uint64_t kWideSection = 512;
static uint64_t section_length(const prand_request_t &r, const BatchParams &P, uint32_t max_tiles)
{
    const uint64_t lanes_per_tile = is_gm(r.gen) ? (uint64_t)(32 / gm_params(r.gen).lanes) : 32ull;
    // one section per warp (lane-per-point GM/GQ) or one per lane (the rest)
    uint64_t sec = lanes_per_tile == 1 ? P.seclen_gm : P.seclen_mrg_lfsr;
    if (is_gm(r.gen) && lanes_per_tile == 32 && sec > kWideSection) sec = kWideSection;
    if (max_tiles) {
        const uint64_t need = (r.length + lanes_per_tile * max_tiles - 1) / (lanes_per_tile * max_tiles);
        if (need > sec) sec = (need + 127) & ~127ull;
    }
    return sec;
}

uint64_t plan_tile_count(const prand_request_t &r, const BatchParams &P, uint32_t max_tiles)
{
    if (r.length == 0) return 0;
    if (r.gen == PRAND_MT19937) return 1;
    const uint64_t lanes_per_tile = is_gm(r.gen) ? (uint64_t)(32 / gm_params(r.gen).lanes) : 32ull;
    const uint64_t per_tile = section_length(r, P, max_tiles) * lanes_per_tile;
    return (r.length + per_tile - 1) / per_tile;
}

// Tensor-core tiles: the 4 (v = 1) or 16 (v = 4) sections of a tile are made in step by
// one block, each from its own jump, so a tile's sections are of one length, whole
// blocks of 64 outputs, at most seclen_gm (4096 before the tuner has run): long enough that
// a jump is a small part of a section, short enough that the longest requests still
// spread over tens of blocks (10^4 mixed requests, the part's five larger generators alone:
// 2.33 ms at 512, 2.11 at 1024, 1.99 at 2048, 1.93 at 4096; 100 requests without MT19937:
// 0.56, 0.56, 0.59, 0.58 ms).  Requests of a fraction of a tile's four sections stay with
// the lane-per-point tiles, a warp each (10^4 requests of one length, u32, us, these / those:
// GM61 10 outputs 79 / 54, 64 79 / 66, 128 79 / 79; GM31 10 56 / 44, 64 56 / 52; GM29 10 60 / 46, 160 60 / 57).
static bool tc_request(const prand_request_t &r)
{
    if (!is_gm(r.gen) || r.gen == PRAND_GQ58_3) return false;
    if (gm_params(r.gen).v != 1) return true;
    return r.length >= (r.gen == PRAND_GM29 ? 192u : r.gen == PRAND_GM19 ? 160u : r.gen == PRAND_GM61 ? 120u : 96u);
}

static void plan_tc(const prand_request_t &r, const BatchParams &P, std::vector<BatchTile> &out)
{
    const GmParams &G = gm_params(r.gen);
    const uint64_t n = G.s == 32 ? 4 : 16, es = esize(r.dtype);
    const uint64_t most = std::min<uint64_t>((P.seclen_gm + 63ull) & ~63ull, 1u << 20);
    const uint64_t tiles = (r.length + n * most - 1) / (n * most);
    const uint64_t sec = ((r.length + n * tiles - 1) / (n * tiles) + 63) & ~63ull, per_tile = sec * n;
    for (uint64_t off = 0; off < r.length; off += per_tile) {
        BatchTile t = {};
        t.stream = r.stream; t.start = off; t.len = std::min(per_tile, r.length - off);
        t.out = (uintptr_t)r.dev_out + off * es;
        t.seclen = (uint32_t)sec; t.gen = (uint8_t)r.gen; t.dtype = (uint8_t)r.dtype; t.slot = t.wslot = -1;
        t.flags = (uint16_t)(kTileTc | ((uintptr_t)r.dev_out % (es * (G.v == 1 ? 2 : 4)) == 0 ? kTileVec : 0u));
        out.push_back(t);
    }
}

void plan_request(const prand_request_t &r, int32_t slot, int32_t wslot, bool from_slot, const BatchParams &P,
                  std::vector<BatchTile> &out, uint32_t max_tiles, bool tc)
{
    if (r.length == 0) return;
    const int gen = r.gen;
    const size_t es = esize(r.dtype);
    const uintptr_t base = (uintptr_t)r.dev_out;
    if (tc && tc_request(r)) return plan_tc(r, P, out);
    auto vec_ok = [&](uint64_t seclen) { return base % 16 == 0 && (seclen * es) % 16 == 0 && seclen % 4 == 0; };
    const uint16_t fs = from_slot ? (uint16_t)kTileFromSlot : (uint16_t)0;
    if (gen == PRAND_MT19937) {
        BatchTile t = {};
        t.stream = r.stream; t.start = 0; t.len = r.length; t.out = base;
        t.seclen = 0; t.gen = (uint8_t)gen; t.dtype = (uint8_t)r.dtype; t.slot = slot; t.wslot = wslot;
        t.flags = (uint16_t)(fs | (wslot >= 0 ? kTileLast : 0u));
        out.push_back(t);
        return;
    }
    const uint64_t lanes_per_tile = is_gm(gen) ? (uint64_t)(32 / gm_params(gen).lanes) : 32ull;
    const uint64_t sec = section_length(r, P, max_tiles);
    const uint64_t per_tile = sec * lanes_per_tile;
    for (uint64_t off = 0; off < r.length; off += per_tile) {
        BatchTile t = {};
        t.stream = r.stream; t.start = off; t.len = std::min(per_tile, r.length - off);
        t.out = base + off * es;
        t.seclen = (uint32_t)sec; t.gen = (uint8_t)gen; t.dtype = (uint8_t)r.dtype; t.slot = slot; t.wslot = wslot;
        t.flags = (uint16_t)(fs | (vec_ok(sec) ? kTileVec : 0u) |
                             ((wslot >= 0 && off + t.len == r.length) ? kTileLast : 0u));
        out.push_back(t);
    }
}

size_t slot_words(int gen)
{
    if (gen == PRAND_MT19937) return kMtN + 1;
    return state_bytes_per_stream(gen) / 4;
}

bool wide_tile_gen(int gen) { return is_gm(gen) && gm_params(gen).lanes == 1; }

// The parts of BatchParts in order; longest first within each part (MT19937 jump
// chains are the longest).
static uint64_t tile_cost(const BatchTile &t)
{
    if (t.gen == PRAND_MT19937) return (3ull << 60) + t.len;
    if (t.flags & kTileTc) return ((uint64_t)(PRAND_NUM_GENERATORS - t.gen) << 44) + std::min<uint64_t>(t.len, 1ull << 40);
    if (wide_tile_gen(t.gen)) return (2ull << 60) + t.len;
    return (1ull << 60) + t.len / (t.gen == PRAND_MRG32K3A || t.gen == PRAND_LFSR113 ? 32 : 1);
}

void order_tiles(std::vector<BatchTile> &tiles)
{
    std::stable_sort(tiles.begin(), tiles.end(),
                     [](const BatchTile &a, const BatchTile &b) { return tile_cost(a) > tile_cost(b); });
}

prand_status_t validate_requests(const prand_request_t *reqs, size_t n)
{
    if (!reqs && n) return PRAND_ERR_ARG;
    for (size_t i = 0; i < n; ++i) {
        const prand_request_t &r = reqs[i];
        if (r.gen < 0 || r.gen >= PRAND_NUM_GENERATORS || r.dtype < 0 || r.dtype > 2) return PRAND_ERR_ARG;
        if (r.length && !r.dev_out) return PRAND_ERR_ARG;
        if ((uintptr_t)r.dev_out % esize(r.dtype)) return PRAND_ERR_ALIGN;
        uint64_t bytes;
        if (__builtin_mul_overflow(r.length, (uint64_t)esize(r.dtype), &bytes)) return PRAND_ERR_ARG;
    }
    return PRAND_OK;
}

// Persistent grid of a build: enough blocks for the tiles, at most the
// resident blocks of the whole GPU.
static unsigned batch_grid(uint32_t ntiles, uint32_t block, int blocks_per_sm)
{
    Engine *E;
    if (engine_get(&E) != PRAND_OK) return 1;
    uint64_t warps_needed = ntiles, per_block = block / 32;
    uint64_t g = std::min<uint64_t>((warps_needed + per_block - 1) / per_block, (uint64_t)E->sms * blocks_per_sm);
    return (unsigned)std::max<uint64_t>(g, 1);
}

BatchParts batch_parts(const std::vector<BatchTile> &tiles)
{
    BatchParts p;
    for (const BatchTile &t : tiles) {
        if (t.gen == PRAND_MT19937) ++p.mt;
        else if (t.flags & kTileTc) ++p.tc[t.gen - PRAND_GM19];
        else if (wide_tile_gen(t.gen)) ++p.wide;
        else ++p.rest;
    }
    return p;
}

prand_status_t Branches::create()
{
    for (int b = 0; b < kBranches; ++b)
        if (cudaStreamCreateWithFlags(&st[b], cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&fork[b], cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&join[b], cudaEventDisableTiming) != cudaSuccess)
            return PRAND_ERR_CUDA;
    return PRAND_OK;
}

void Branches::destroy()
{
    for (int b = 0; b < kBranches; ++b) {
        if (st[b]) cudaStreamDestroy(st[b]);
        if (fork[b]) cudaEventDestroy(fork[b]);
        if (join[b]) cudaEventDestroy(join[b]);
        st[b] = nullptr;
        fork[b] = join[b] = nullptr;
    }
}

// The parts' launches, MT19937's, the thread-per-stream and the tensor-core tiles on
// their branches' streams (st where there is none).
static prand_status_t launch_parts(const Engine &E, const BatchTile *d_tiles, const BatchParts &parts, uint32_t *d_counter,
                                   const BatchCtx &ctx, cudaStream_t st, const cudaStream_t (&on)[kBranches])
{
    const uint32_t nmt = parts.mt, nwide = parts.wide, nrest = parts.rest;
    prand_status_t s = PRAND_OK;
    if (nmt) {
        // few tiles: a cluster of blocks each, while every block has an SM to itself (a
        // stream of eight jumps and 1000 outputs: 175 us, by one block 669; 19 such 199)
        if ((uint64_t)nmt * kMtCluster <= (uint64_t)E.sms) {
            s = mt_cluster_launch(batch_kernel<kModeMt, 32 * kMtTeam, 128, kMtCluster>, nmt * kMtCluster, 32 * kMtTeam, kMtCluster, on[0],
                                  d_tiles, nmt, d_counter, ctx);
            if (s != PRAND_OK) return s;
        } else {
            const unsigned g = batch_grid(nmt, 32, E.mt_team_bps);  // one tile per block
            batch_kernel<kModeMt, 32 * kMtTeam, 128><<<g, 32 * kMtTeam, 0, on[0]>>>(d_tiles, nmt, d_counter, ctx);
            if ((s = launch_check()) != PRAND_OK) return s;
        }
    }
    if (nwide) {
        const unsigned g = batch_grid(nwide, kBatchThreads, E.blocks_per_sm[kModeWide]);
        batch_kernel<kModeWide, kBatchThreads, 128><<<g, kBatchThreads, 0, on[1]>>>(d_tiles + nmt, nwide, d_counter + 2, ctx);
        if ((s = launch_check()) != PRAND_OK) return s;
    }
    const BatchTile *tc_tiles = d_tiles + nmt + nwide + nrest;
    for (int g = 0; g < 8; ++g) {
        if (!parts.tc[g]) continue;
        s = gm_batch(PRAND_GM19 + g, E.T, tc_tiles, parts.tc[g], ctx.base[PRAND_GM19 + g], on[2]);
        if (s != PRAND_OK) return s;
        tc_tiles += parts.tc[g];
    }
    if (nrest) {
        const int v = rest_variant(E.params.block, E.params.row_bytes);
        rest_launch(v, batch_grid(nrest, rest_block(v), E.rest_bps[v]), st, d_tiles + nmt + nwide, nrest,
                    d_counter + 1, ctx);
        if ((s = launch_check()) != PRAND_OK) return s;
    }
    return PRAND_OK;
}

// d_counter: [0] MT19937, [1] the rest, [2] thread-per-stream tiles.  Whatever comes of
// it, `st` goes on only behind every branch that was forked: the caller's buffers are
// free when its work in `st` is done.
prand_status_t launch_batch(const BatchTile *d_tiles, const BatchParts &parts, uint32_t *d_counter, const BatchCtx &ctx,
                            cudaStream_t st, const Branches *br)
{
    Engine *E;
    prand_status_t s = engine_get(&E);
    if (s != PRAND_OK) return s;
    if (cudaMemsetAsync(d_counter, 0, 3 * sizeof(uint32_t), st) != cudaSuccess) return PRAND_ERR_CUDA;
    if (!parts.all()) return PRAND_OK;
    const uint32_t nmt = parts.mt, nwide = parts.wide, nrest = parts.rest, ntc = parts.tc_all();
    // a part goes to its branch when a later part runs beside it
    const bool on_branch[kBranches] = { br && nmt && (nwide || nrest || ntc), br && nwide && (nrest || ntc), br && ntc && nrest };
    bool forked[kBranches] = {};
    cudaStream_t on[kBranches];
    for (int b = 0; b < kBranches; ++b) {
        on[b] = on_branch[b] ? br->st[b] : st;
        if (!on_branch[b] || s != PRAND_OK) continue;
        if (cudaEventRecord(br->fork[b], st) != cudaSuccess || cudaStreamWaitEvent(br->st[b], br->fork[b], 0) != cudaSuccess)
            s = PRAND_ERR_CUDA;
        else forked[b] = true;
    }
    if (s == PRAND_OK) s = launch_parts(*E, d_tiles, parts, d_counter, ctx, st, on);
    for (int b = 0; b < kBranches; ++b)
        if (forked[b] && (cudaEventRecord(br->join[b], br->st[b]) != cudaSuccess ||
                          cudaStreamWaitEvent(st, br->join[b], 0) != cudaSuccess) && s == PRAND_OK)
            s = PRAND_ERR_CUDA;
    return s;
}

// The tile list into the engine's buffer, on `st` behind the last batch that reads it
// (which may be on another stream).  The engine's run_mu is held until that batch's
// successor is launched and recorded.
static prand_status_t upload_tiles(Engine *E, const std::vector<BatchTile> &tiles, cudaStream_t st)
{
    const size_t n = tiles.size();
    if (cudaStreamWaitEvent(st, E->done, 0) != cudaSuccess) return PRAND_ERR_CUDA;
    if (cudaEventSynchronize(E->staged) != cudaSuccess) return PRAND_ERR_CUDA;  // staging free again
    if (n > E->h_cap) {
        if (E->h_tiles) cudaFreeHost(E->h_tiles);
        E->h_cap = std::max<size_t>(n, 2 * E->h_cap);
        if (!host_alloc(&E->h_tiles, E->h_cap * sizeof(BatchTile))) { E->h_cap = 0; E->h_tiles = nullptr; return PRAND_ERR_NOMEM; }
    }
    if (n > E->d_cap) {
        if (E->d_tiles) { cudaEventSynchronize(E->done); cudaFree(E->d_tiles); }
        E->d_cap = std::max<size_t>(n, 2 * E->d_cap);
        if (!dev_alloc(&E->d_tiles, E->d_cap * sizeof(BatchTile))) { E->d_cap = 0; E->d_tiles = nullptr; return PRAND_ERR_NOMEM; }
    }
    if (n) {
        memcpy(E->h_tiles, tiles.data(), n * sizeof(BatchTile));
        if (cudaMemcpyAsync(E->d_tiles, E->h_tiles, n * sizeof(BatchTile), cudaMemcpyHostToDevice, st) != cudaSuccess)
            return PRAND_ERR_CUDA;
        if (cudaEventRecord(E->staged, st) != cudaSuccess) return PRAND_ERR_CUDA;
    }
    return PRAND_OK;
}

}  // namespace prand

using namespace prand;

// ------------------------------------------------------------------ C ABI
struct prand_batch_plan_s {
    int device = -1;
    BatchTile *d_tiles = nullptr;
    BatchParts parts;
    Branches br;  // the side branches while capturing
    uint32_t *d_counter = nullptr;
    BatchCtx ctx;
    BasesRef bases;  // ctx's base states
    DevTables *T = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

extern "C" {

prand_status_t prand_batch_run(const prand_request_t *reqs, size_t n, uint64_t seed, prand_stream_t stream)
{
    prand_status_t s = validate_requests(reqs, n);
    if (s != PRAND_OK || n == 0) return s;
    cudaStream_t st = (cudaStream_t)stream;
    BatchCtx ctx;
    BasesRef bases;
    if ((s = batch_ctx(seed, st, &ctx, &bases, nullptr)) != PRAND_OK) return s;
    const BatchParams P = batch_params();
    std::vector<BatchTile> tiles;
    tiles.reserve(n * 2);
    for (size_t i = 0; i < n; ++i) plan_request(reqs[i], -1, -1, false, P, tiles, 0, true);
    order_tiles(tiles);
    if (tiles.size() > 0xFFFFFFFFull) return PRAND_ERR_ARG;
    Engine *E;
    if ((s = engine_get(&E)) != PRAND_OK) return s;
    std::lock_guard<std::mutex> lk(E->run_mu);
    if ((s = upload_tiles(E, tiles, st)) != PRAND_OK) return s;
    s = launch_batch(E->d_tiles, batch_parts(tiles), E->d_counter, ctx, st, &E->br);
    if (cudaEventRecord(E->done, st) != cudaSuccess && s == PRAND_OK) s = PRAND_ERR_CUDA;
    return s;
}

prand_status_t prand_batch_plan_create(prand_batch_plan_t *out, const prand_request_t *reqs, size_t n, uint64_t seed)
{
    if (!out) return PRAND_ERR_ARG;
    *out = nullptr;
    prand_status_t s = validate_requests(reqs, n);
    if (s != PRAND_OK) return s;
    prand_batch_plan_t p = new (std::nothrow) prand_batch_plan_s;
    if (!p) return PRAND_ERR_NOMEM;
    cudaGetDevice(&p->device);
    cudaStream_t cap = nullptr;
    auto fail = [&](prand_status_t e) {
        if (cap) cudaStreamDestroy(cap);
        p->br.destroy();
        if (p->exec) cudaGraphExecDestroy(p->exec);
        if (p->graph) cudaGraphDestroy(p->graph);
        if (p->d_tiles) cudaFree(p->d_tiles);
        if (p->d_counter) cudaFree(p->d_counter);
        delete p;
        return e;
    };
    if ((s = batch_ctx(seed, 0, &p->ctx, &p->bases, &p->T)) != PRAND_OK) return fail(s);
    const BatchParams P = batch_params();
    std::vector<BatchTile> tiles;
    for (size_t i = 0; i < n; ++i) plan_request(reqs[i], -1, -1, false, P, tiles, 0, true);
    order_tiles(tiles);
    if (tiles.size() > 0xFFFFFFFFull) return fail(PRAND_ERR_ARG);
    p->parts = batch_parts(tiles);
    if (!dev_alloc(&p->d_counter, 64)) return fail(PRAND_ERR_NOMEM);
    if (p->br.create() != PRAND_OK) return fail(PRAND_ERR_CUDA);
    if (!tiles.empty()) {
        if (!dev_alloc(&p->d_tiles, tiles.size() * sizeof(BatchTile))) return fail(PRAND_ERR_NOMEM);
        if (cudaMemcpy(p->d_tiles, tiles.data(), tiles.size() * sizeof(BatchTile), cudaMemcpyHostToDevice) != cudaSuccess)
            return fail(PRAND_ERR_CUDA);
    }
    if (cudaStreamSynchronize(0) != cudaSuccess) return fail(PRAND_ERR_CUDA);
    // capture: counter reset + the persistent launches (the MT19937 and
    // thread-per-stream parts forked onto the plan's branch streams and joined back)
    if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) return fail(PRAND_ERR_CUDA);
    if (cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return fail(PRAND_ERR_CUDA);
    prand_status_t ls = launch_batch(p->d_tiles, p->parts, p->d_counter, p->ctx, cap, &p->br);
    cudaGraph_t g = nullptr;
    cudaError_t ce = cudaStreamEndCapture(cap, &g);
    p->graph = g;
    if (ls != PRAND_OK) return fail(ls);
    if (ce != cudaSuccess) return fail(PRAND_ERR_CUDA);
    if (cudaGraphInstantiate(&p->exec, p->graph, 0) != cudaSuccess) return fail(PRAND_ERR_CUDA);
    cudaStreamDestroy(cap);
    cap = nullptr;
    *out = p;
    return PRAND_OK;
}

prand_status_t prand_batch_plan_launch(prand_batch_plan_t p, prand_stream_t stream)
{
    if (!p || !p->exec) return PRAND_ERR_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != p->device) return PRAND_ERR_STATE;
    if (p->parts.tc_all() && *p->T->wait_failed) return PRAND_ERR_TIMEOUT;  // (the graph launches without a look)
    g_launches.fetch_add(p->parts.all() ? 1 : 0, std::memory_order_relaxed);
    return cudaGraphLaunch(p->exec, (cudaStream_t)stream) == cudaSuccess ? PRAND_OK : PRAND_ERR_CUDA;
}

prand_status_t prand_batch_plan_destroy(prand_batch_plan_t p)
{
    if (!p) return PRAND_OK;
    // the first cudaFree waits for the device (cudaDeviceSynchronize would end a capture
    // under way in another thread)
    if (p->d_counter) cudaFree(p->d_counter);
    if (p->exec) cudaGraphExecDestroy(p->exec);
    if (p->graph) cudaGraphDestroy(p->graph);
    if (p->d_tiles) cudaFree(p->d_tiles);
    p->br.destroy();
    delete p;
    return PRAND_OK;
}

prand_status_t prand_batch_autotune(const prand_request_t *reqs, size_t n, uint64_t seed, prand_stream_t stream,
                                    uint32_t *seclen_mrg_lfsr, uint32_t *seclen_gm, uint32_t *block,
                                    uint32_t *row_bytes, float *best_ms)
{
    prand_status_t s = validate_requests(reqs, n);
    if (s != PRAND_OK) return s;
    Engine *E;
    if ((s = engine_get(&E)) != PRAND_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    const BatchParams keep = E->params;
    BatchParams best = keep;
    float best_t = 1e30f;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    // one candidate: a graph plan with these parameters, one warm-up launch,
    // the mean of three timed launches
    auto try_params = [&](const BatchParams &c) {
        E->params = c;
        prand_batch_plan_t plan;
        if ((s = prand_batch_plan_create(&plan, reqs, n, seed)) != PRAND_OK) return;
        prand_batch_plan_launch(plan, stream);
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; ++r) prand_batch_plan_launch(plan, stream);
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        ms /= 3;
        prand_batch_plan_destroy(plan);
        if (ms < best_t) { best_t = ms; best = c; }
    };
    // coordinate search: the two section lengths (outputs per lane and per
    // tensor-core section), then the rest build's threads per block and staged row
    // size (outputs per row store) at the best lengths
    const uint32_t cand[] = { 2048, 8192, 32768 };
    for (uint32_t a : cand)
        for (uint32_t b : cand) {
            if (s != PRAND_OK) break;
            BatchParams c = keep;
            c.seclen_mrg_lfsr = a;
            c.seclen_gm = b;
            try_params(c);
        }
    const BatchParams lengths = best;
    for (uint32_t bs : { 64u, 128u })
        for (uint32_t rb : { 128u, 256u }) {
            if (s != PRAND_OK) break;
            BatchParams c = lengths;
            c.block = bs;
            c.row_bytes = rb;
            if (bs != lengths.block || rb != lengths.row_bytes) try_params(c);
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    E->params = s == PRAND_OK ? best : keep;
    if (s != PRAND_OK) return s;
    if (seclen_mrg_lfsr) *seclen_mrg_lfsr = best.seclen_mrg_lfsr;
    if (seclen_gm) *seclen_gm = best.seclen_gm;
    if (block) *block = best.block;
    if (row_bytes) *row_bytes = best.row_bytes;
    if (best_ms) *best_ms = best_t;
    const char *path = getenv("PRAND_TUNE_CACHE");
    if (path) {
        FILE *f = fopen(path, "w");
        if (f) {
            fprintf(f, "{\"seclen_mrg_lfsr\": %u, \"seclen_gm\": %u, \"block\": %u, \"row_bytes\": %u, \"ms\": %.4f}\n",
                    best.seclen_mrg_lfsr, best.seclen_gm, best.block, best.row_bytes, best_t);
            fclose(f);
        }
    }
    return PRAND_OK;
}

prand_status_t prand_batch_set_params(uint32_t seclen_mrg_lfsr, uint32_t seclen_gm, uint32_t block, uint32_t row_bytes)
{
    if (seclen_mrg_lfsr == 0 || seclen_gm == 0 || seclen_mrg_lfsr % 4 || seclen_gm % 4 || (block != 64 && block != 128) ||
        (row_bytes != 128 && row_bytes != 256))
        return PRAND_ERR_ARG;
    Engine *E;
    prand_status_t s = engine_get(&E);
    if (s != PRAND_OK) return s;
    E->params.seclen_mrg_lfsr = seclen_mrg_lfsr;
    E->params.seclen_gm = seclen_gm;
    E->params.block = block;
    E->params.row_bytes = row_bytes;
    return PRAND_OK;
}

// Per-request plain launches (for comparison with the fused form): for every
// request, the ordinary stream-initialisation launch(es) and generation launch
// on one stream, with no fusion and no persistent scheduling.
prand_status_t prand_batch_run_per_request(const prand_request_t *reqs, size_t n, uint64_t seed, prand_stream_t stream)
{
    prand_status_t s = validate_requests(reqs, n);
    if (s != PRAND_OK || n == 0) return s;
    cudaStream_t st = (cudaStream_t)stream;
    BatchCtx ctx;
    BasesRef bases;
    DevTables *T;
    if ((s = batch_ctx(seed, st, &ctx, &bases, &T)) != PRAND_OK) return s;
    size_t maxb = 0;
    for (int g = 0; g < PRAND_NUM_GENERATORS; ++g) maxb = std::max(maxb, state_bytes_per_stream(g));
    void *scratch = nullptr;
    if (n && !dev_alloc(&scratch, 2 * maxb * n)) return PRAND_ERR_NOMEM;
    for (size_t i = 0; i < n && s == PRAND_OK; ++i) {
        const prand_request_t &r = reqs[i];
        if (!r.length) continue;
        void *a = (char *)scratch + 2 * maxb * i, *b = (char *)a + maxb;
        StreamRange R;
        R.stride = R.count = 1;
        uint32_t idx = kMtN;
        if (r.gen == PRAND_MT19937) {
            mt_window_init_kernel<<<1, 32 * kMtTeam, 0, st>>>((const uint32_t *)ctx.base[r.gen], ctx.mt_win, r.stream,
                                                    (uint32_t *)a);
            s = launch_check();
            if (s == PRAND_OK) s = mt_gen(a, 1, &idx, r.dev_out, r.dtype, r.length, st);
        } else if (is_gm(r.gen)) {
            Variant V;
            variant_params(r.gen, 0, &V);
            s = gm_init(r.gen, T, ctx.base[r.gen], a, r.stream, 1, V, st);
            if (s == PRAND_OK) s = gm_gen(r.gen, T, a, b, R, r.dev_out, r.dtype, r.length, st);
        } else {
            Variant V;
            variant_params(r.gen, 0, &V);
            s = mrg_lfsr_init(r.gen, T, ctx.base[r.gen], a, r.stream, 1, V, st);
            if (s == PRAND_OK) s = mrg_lfsr_gen(r.gen, T, a, b, R, r.dev_out, r.dtype, r.length, st);
        }
    }
    // scratch is freed in stream order (the runtime defers it until the work is done)
    cudaStreamSynchronize(st);
    if (scratch) cudaFree(scratch);
    for (size_t i = 0; i < n && s == PRAND_OK; ++i)
        if (is_gm(reqs[i].gen) && T->gm_tc[reqs[i].gen - PRAND_GM19] && *T->wait_failed) s = PRAND_ERR_TIMEOUT;
    return s;
}

}  // extern "C"
