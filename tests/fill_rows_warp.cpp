// A warp on the host: 32 threads run fill_rows (cut out of devcommon.cuh into
// fill_rows.inc), meeting at every warp operation, each of which checks that all
// 32 lanes came to the same one.
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <thread>
#include <type_traits>
#include <vector>

#define __device__
#define __forceinline__ inline
struct alignas(16) uint4 { uint32_t x, y, z, w; };
using std::min;
constexpr uint32_t kFull = 0xFFFFFFFFu;

static std::barrier<> meet(32);
static unsigned long long value[32];
static int at[32];
static thread_local int me;

static void vote(int where, unsigned long long v)
{
    value[me] = v;
    at[me] = where;
    meet.arrive_and_wait();
    for (int i = 0; i < 32; ++i)
        if (at[i] != where) {
            fprintf(stderr, "lane %d at line %d, lane %d at line %d\n", me, where, i, at[i]);
            _Exit(3);
        }
}
static void done() { meet.arrive_and_wait(); }
template <typename F> static auto gather(int where, unsigned long long v, F f)
{
    vote(where, v);
    auto r = f();
    done();
    return r;
}
static int all(int where, bool p) { return gather(where, p, [] { for (auto v : value) if (!v) return 0; return 1; }); }
static uint32_t ballot(int where, bool p) { return gather(where, p, [] { uint32_t r = 0; for (int i = 0; i < 32; ++i) r |= (uint32_t)(value[i] != 0) << i; return r; }); }
static uint32_t least(int where, uint32_t x) { return gather(where, x, [] { uint32_t r = ~0u; for (auto v : value) r = std::min(r, (uint32_t)v); return r; }); }
static uint32_t most(int where, uint32_t x) { return gather(where, x, [] { uint32_t r = 0; for (auto v : value) r = std::max(r, (uint32_t)v); return r; }); }
template <typename T> static T from(int where, T x, int lane) { return gather(where, (unsigned long long)x, [&] { return (T)value[lane & 31]; }); }
#define __all_sync(m, p) all(__LINE__, p)
#define __ballot_sync(m, p) ballot(__LINE__, p)
#define __reduce_min_sync(m, x) least(__LINE__, x)
#define __reduce_max_sync(m, x) most(__LINE__, x)
#define __shfl_sync(m, x, l) from(__LINE__, x, l)
#define __syncwarp() (vote(__LINE__, 0), done())

#include "fill_rows.inc"

static uint32_t word(int lane, uint64_t i) { return (uint32_t)(lane * 0x9E3779B1u + i * 0x85EBCA77u + 1); }

struct Plain {
    int lane;
    uint64_t n = 0;
    uint32_t operator()() { return word(lane, n++); }
};
struct Chunked : Plain {  // as a generator that makes whole chunks of outputs by their place
    uint32_t operator()() { return Plain::operator()(); }
    uint32_t operator()(int k)
    {
        if (k == 0) first = n;
        if (first + k != n) { fprintf(stderr, "output %d of a chunk out of order\n", k); _Exit(4); }
        return word(lane, n++);
    }
    uint64_t first = 0;
};

template <typename OutT, int ROWB, bool ROLL, bool ENDS, typename Gen>
static void run(const std::vector<uint64_t> &len, int offset)
{
    using RF = RowFill<OutT, ROWB>;
    uint64_t pitch = 0;
    for (uint64_t l : len) pitch = std::max(pitch, l);
    // rows one behind another, as a fill's are, or with room between them
    std::vector<uint64_t> start(32);
    uint64_t total = 64 + offset;
    for (int i = 0; i < 32; ++i) { start[i] = total; total += len[i]; }
    OutT *buf = (OutT *)aligned_alloc(256, (total + 512) * sizeof(OutT) / 256 * 256 + 256);
    const OutT guard = (OutT)12345;
    for (uint64_t i = 0; i < total + 64; ++i) buf[i] = guard;
    alignas(16) static unsigned char tile[RF::TILE];
    uint64_t made[32];
    std::vector<std::thread> warp;
    for (int l = 0; l < 32; ++l)
        warp.emplace_back([&, l] {
            me = l;
            Gen g;
            g.lane = l;
            fill_rows<OutT, ROWB, ROLL, ENDS>(g, [](uint32_t u) { return (OutT)u; }, buf + start[l], len[l], tile, l);
            made[l] = g.n;
        });
    for (auto &t : warp) t.join();
    std::vector<OutT> want(total + 64, guard);
    for (int l = 0; l < 32; ++l)
        for (uint64_t i = 0; i < len[l]; ++i) want[start[l] + i] = (OutT)word(l, i);
    for (uint64_t i = 0; i < total + 64; ++i)
        if (buf[i] != want[i]) { fprintf(stderr, "wrong at %llu\n", (unsigned long long)i); _Exit(5); }
    for (int l = 0; l < 32; ++l)
        if (made[l] != len[l]) { fprintf(stderr, "lane %d made %llu of %llu\n", l, (unsigned long long)made[l], (unsigned long long)len[l]); _Exit(6); }
    free(buf);
}

template <typename OutT, int ROWB, bool ROLL, bool ENDS, typename Gen>
static void shapes(int seed)
{
    std::mt19937 rng(seed);
    const uint64_t K = RowFill<OutT, ROWB>::K, E = RowFill<OutT, ROWB>::E;
    auto same = [](uint64_t n, int live, uint64_t last) {
        std::vector<uint64_t> v(32, 0);
        for (int i = 0; i < live; ++i) v[i] = i + 1 == live ? last : n;
        return v;
    };
    for (int live : { 32, 31, 2, 1 })
        for (uint64_t n : { E, K - E, K, K + E, 3 * K, 3 * K + 2 * E }) {
            run<OutT, ROWB, ROLL, ENDS, Gen>(same(n, live, n), 0);
            run<OutT, ROWB, ROLL, ENDS, Gen>(same(n, live, std::max<uint64_t>(n / 2, 1)), (int)E);
        }
    for (uint64_t n : { (uint64_t)1, K - 1, K + 1, 2 * K + 3 })
        for (int offset : { 0, 1, 3 }) run<OutT, ROWB, ROLL, ENDS, Gen>(same(n, 29, n), offset);
    for (int k = 0; k < 6; ++k) {  // rows that end anywhere, idle lanes among them
        std::vector<uint64_t> v(32);
        for (auto &x : v) x = rng() % 4 ? rng() % (3 * K) : 0;
        if (k % 2) for (auto &x : v) x = x / E * E;
        run<OutT, ROWB, ROLL, ENDS, Gen>(v, k / 2);
    }
}

int main()
{
    shapes<uint32_t, 128, false, false, Plain>(1);
    shapes<uint32_t, 128, false, true, Plain>(2);
    shapes<uint32_t, 256, false, true, Chunked>(3);
    shapes<uint32_t, 256, false, false, Chunked>(4);
    shapes<double, 128, true, true, Plain>(5);
    shapes<double, 256, false, false, Chunked>(6);
    shapes<float, 128, true, false, Plain>(7);
    puts("ok");
}
