// Tiles that the library plans for one request: argv gen, length, seclen_mrg_lfsr,
// seclen_gm; one line per tile: start, len, seclen, flags.
#include <cstdio>
#include <cstdlib>

#include "batch.cuh"

int main(int, char **argv)
{
    prand_request_t r = {};
    r.gen = atoi(argv[1]);
    r.length = strtoull(argv[2], nullptr, 10);
    r.dev_out = (void *)0x1000;
    prand::BatchParams P;
    if (atoi(argv[3])) P.seclen_mrg_lfsr = (uint32_t)strtoul(argv[3], nullptr, 10);
    if (atoi(argv[4])) P.seclen_gm = (uint32_t)strtoul(argv[4], nullptr, 10);
    std::vector<prand::BatchTile> tiles;
    prand::plan_request(r, -1, -1, false, P, tiles, 0, true);
    for (const prand::BatchTile &t : tiles)
        printf("%llu %llu %u %u %llu\n", (unsigned long long)t.start, (unsigned long long)t.len, t.seclen, t.flags, (unsigned long long)t.out);
}
