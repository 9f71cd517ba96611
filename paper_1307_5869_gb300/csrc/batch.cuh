// Shared declarations of the batched persistent kernel (batch.cu) and the
// resident-stream server built on it (serve.cpp).
#pragma once

#include <memory>
#include <vector>

#include "prand_internal.h"

namespace prand {

constexpr uint32_t kTileLast = 1u;      // the tile holds the request's last output: write the next state to wslot
constexpr uint32_t kTileVec = 2u;       // every row start is 16-byte aligned: vector / staged-row stores
constexpr uint32_t kTileFromSlot = 4u;  // start from the state in slot (else from the seeded base + stream * L)
constexpr uint32_t kTileTc = 8u;        // a tile of the tensor-core kernels (gm_tc.cuh): seclen outputs per section

// One unit of work for one warp (64 bytes).
struct BatchTile {
    uint64_t stream;  // stream index k (block splitting: base advanced by k L)
    uint64_t start;   // offset of the tile's first output inside the request
    uint64_t len;     // outputs in the tile
    uint64_t out;     // device address of the tile's first output
    uint32_t seclen;  // outputs per lane (MRG32K3A, LFSR113) or per lane group (GM/GQ)
    int32_t slot;     // state slot read with kTileFromSlot
    int32_t wslot;    // state slot written with kTileLast (a different buffer than slot)
    uint8_t gen, dtype;
    uint16_t flags;
    uint32_t req;     // index of the tile's request in its batch (completion tracking)
    uint32_t pad_[3];
};
static_assert(sizeof(BatchTile) == 64, "tile layout");

struct BatchCtx {
    const uint32_t *mrg_tab, *lfsr_tab, *mt_polys;
    const uint32_t *mt_win;                  // stream jumps by byte: [8][256][624] (digit 0 unused)
    const uint64_t *gm_tab[8];
    const void *base[PRAND_NUM_GENERATORS];  // base states of the batch's seed
    void *slots[PRAND_NUM_GENERATORS];       // resident-state arenas (server)
    uint32_t *tiles_left;                    // per request: tiles not finished (server), or null
    volatile uint32_t *done_list;            // mapped host memory: request index + 1, in completion order
    uint32_t *done_count;                    // device counter of done_list entries (zero at launch)
};

struct BatchParams {
    // outputs per lane section (thread-per-section tiles), chosen by the tuner; before it
    // has run, its choice for 10^4 mixed requests (11.3 ms at 8192, 10.1 at 2048)
    uint32_t seclen_mrg_lfsr = 2048;
    uint32_t seclen_gm = 4096;        // outputs per section of the tensor-core tiles, and per warp of the lane-per-point ones
    uint32_t block = 64;              // threads per block of the rest-of-generators build (64 or 128)
    uint32_t row_bytes = 128;         // its staged row size (128 or 256 bytes: 32 or 64 u32 outputs per row store)
};

// One seed's base states of all generators, in device memory.  Kernels read them by the
// raw pointers of a BatchCtx, so whoever keeps one (a plan, a server) keeps the bases too.
struct SeedBases {
    uint64_t seed = 0;
    void *dev = nullptr;
    size_t off[PRAND_NUM_GENERATORS] = {};
    SeedBases() = default;
    SeedBases(const SeedBases &) = delete;
    ~SeedBases();
};
using BasesRef = std::shared_ptr<const SeedBases>;

prand_status_t batch_ctx(uint64_t seed, cudaStream_t st, BatchCtx *ctx, BasesRef *bases, DevTables **T);
BatchParams batch_params();
// tc: GM/GQ requests may go to the tensor-core kernels (from the seeded base only).
void plan_request(const prand_request_t &r, int32_t slot, int32_t wslot, bool from_slot, const BatchParams &P,
                  std::vector<BatchTile> &out, uint32_t max_tiles = 0, bool tc = false);
// Number of tiles plan_request() makes for r (without planning it).
uint64_t plan_tile_count(const prand_request_t &r, const BatchParams &P, uint32_t max_tiles = 0);
size_t slot_words(int gen);  // 32-bit words per state slot
void order_tiles(std::vector<BatchTile> &tiles);
prand_status_t validate_requests(const prand_request_t *reqs, size_t n);
// A tile list runs in parts, each a persistent launch of its own kernel build, in
// this order (order_tiles): MT19937 tiles (many registers, shared memory), the
// thread-per-stream GM/GQ tiles (GM55, GQ58.3, GQ58.4: their points need more
// registers than the next build allows), every other generator's (few registers,
// many resident warps), and the tensor-core tiles, generator by generator.
// With side branches (Branches), the MT19937, thread-per-stream and tensor-core
// parts each run on a branch stream of their own, forked from and joined back
// into `st`, so all share the GPU at once; without them (the server's flights, one
// stream each) the parts run one after the other.
struct BatchParts {
    uint32_t mt = 0, wide = 0, rest = 0, tc[8] = {};  // tc: by generator, PRAND_GM19 first
    uint32_t tc_all() const
    {
        uint32_t n = 0;
        for (uint32_t t : tc) n += t;
        return n;
    }
    uint32_t all() const { return mt + wide + rest + tc_all(); }
};
BatchParts batch_parts(const std::vector<BatchTile> &tiles);  // of an ordered list
constexpr int kBranches = 3;
struct Branches {
    cudaStream_t st[kBranches] = {};  // MT19937, thread-per-stream GM/GQ and tensor-core tiles
    cudaEvent_t fork[kBranches] = {}, join[kBranches] = {};
    prand_status_t create();
    void destroy();
};
bool wide_tile_gen(int gen);
// Warps per MT19937 tile: one block applies each jump polynomial and twists each output
// block together, for batches and the server alike.
constexpr int kMtTeam = 12;

prand_status_t launch_batch(const BatchTile *d_tiles, const BatchParts &parts, uint32_t *d_counter, const BatchCtx &ctx,
                            cudaStream_t st, const Branches *br = nullptr);

// The tensor-core tiles of one generator (gm_tc.cuh), from its seeded base.
prand_status_t gm_batch(int gen, const DevTables *T, const BatchTile *tiles, uint32_t n, const void *base, cudaStream_t st);

}  // namespace prand
