// Host construction of the tensor-core generation's constants (gm_tc.cuh): the
// digit matrices of one block of steps, the block recurrence and the maps
// from a block's pair to any of its values, all modulo the prime p.
#include <string.h>

#include "gm_tc_table.h"

namespace prand {
namespace {

using u128 = unsigned __int128;
using i128 = __int128;

struct Field {
    uint64_t p;
    uint64_t mul(uint64_t a, uint64_t b) const { return (uint64_t)((u128)a * b % p); }
    uint64_t add(uint64_t a, uint64_t b) const { return (uint64_t)(((u128)a + b) % p); }
    uint64_t sub(uint64_t a, uint64_t b) const { return add(a, p - b % p); }
    uint64_t pow(uint64_t a, uint64_t e) const
    {
        uint64_t r = 1 % p;
        for (; e; e >>= 1, a = mul(a, a))
            if (e & 1) r = mul(r, a);
        return r;
    }
    uint64_t inv(uint64_t a) const { return pow(a, p - 2); }  // p is prime
};

// Values x^(n+j), j = -1 .. 2 m, as r[0] x^(n) + r[1] x^(n+1).
struct Rows {
    const Field &F;
    uint64_t r[2 * kTcSteps + 2][2];
    Rows(const Field &F_, uint64_t k, uint64_t q) : F(F_)
    {
        for (int i = 0; i < 2; ++i) {
            r[1][i] = i == 0;
            r[2][i] = i == 1;
            r[0][i] = F.mul(F.sub(F.mul(k, r[1][i]), r[2][i]), F.inv(q));  // q x^(n-1) = k x^(n) - x^(n+1)
            for (int j = 3; j < 2 * kTcSteps + 2; ++j) r[j][i] = F.sub(F.mul(k, r[j - 1][i]), F.mul(q, r[j - 2][i]));
        }
    }
    const uint64_t *at(int j) const { return r[j + 1]; }
};

// x^(n+j) = al x^(n+s) + be x^(n+t) for any j; ok: whether the pair determines the values.
struct Through {
    const Rows &R;
    const uint64_t *a, *b;
    uint64_t inv;
    bool ok;
    Through(const Rows &R_, int s, int t) : R(R_), a(R_.at(s)), b(R_.at(t))
    {
        const uint64_t det = R.F.sub(R.F.mul(a[0], b[1]), R.F.mul(a[1], b[0]));
        ok = det != 0;
        inv = R.F.inv(det);
    }
    void operator()(int j, uint64_t *al, uint64_t *be) const
    {
        const uint64_t *r = R.at(j);
        const Field &F = R.F;
        *al = F.mul(F.sub(F.mul(r[0], b[1]), F.mul(r[1], b[0])), inv);
        *be = F.mul(F.sub(F.mul(a[0], r[1]), F.mul(a[1], r[0])), inv);
    }
};

// f16 bits of n 2^e (|n| <= 2048, result a normal or subnormal f16, exact).
uint16_t half_bits(int n, int e)
{
    if (!n) return 0;
    const uint16_t sign = n < 0 ? 0x8000u : 0u;
    uint32_t m = (uint32_t)(n < 0 ? -n : n);
    while (m < 1024u && e > -24) { m <<= 1; --e; }  // 11-bit significand, or the subnormal exponent
    while (m > 2047u) { m >>= 1; ++e; }             // (2048 only: exact)
    if (m < 1024u) return (uint16_t)(sign | m);     // subnormal: m 2^-24
    return (uint16_t)(sign | (uint32_t)(e + 25) << 10 | (m & 1023u));
}

}  // namespace

bool gm_tc_build(int gen, GmTcTable *T)
{
    const GmParams &G = gm_params(gen);
    const Field F{ G.p };
    memset(T, 0, sizeof *T);
    const int m = kTcSteps;
    const Rows rows(F, G.k, G.q);
    const Through recent(rows, 0, -1), ends(rows, 0, m), later(rows, m, 2 * m);
    if (!recent.ok || !ends.ok || !later.ok) return false;
    recent(m, &T->a, &T->b);
    ends(2 * m, &T->q, &T->v);
    for (int j = -1; j <= m; ++j) later(j, &T->al[j + 1], &T->be[j + 1]);

    // bit position and width of the limb in each slot of a value (tc_limbs; width 0: none)
    static const int byte_pos[8] = { 0, 8, 16, 24 };
    static const int nib_pos[16] = { 0, 8, 16, 24, 4, 12, 20, 28, 32, 40, 48, 56, 36, 44, 52 };
    const bool nib = tc_nibbles(G.kind, G.v);
    const int per = tc_value_slots(G.kind, G.v);
    uint64_t fmax[16] = {};
    int pos[16] = {};
    for (int s = 0; s < per - 1; ++s) {
        const int width = nib ? (s == 11 ? 6 : 4) : s < 4 ? 8 : 0;
        pos[s] = nib ? nib_pos[s] : byte_pos[s];
        // (the kernel's residues are lazy: below p + 2^18 or p + 8; they stay below 2^32 where p does)
        const uint64_t top = (G.p + (G.kind == P51 ? 1u << 18 : 8u)) >> pos[s], full = (1ull << width) - 1;
        fmax[s] = top < full ? top : full;
    }
    auto digits = [](uint32_t w, int *d) {  // two balanced digits of 12 bits, modulo 2^24
        d[1] = (int)((w + 2048u) & 4095u) - 2048;
        w = (w - (uint32_t)d[1]) >> 12;
        d[0] = (int)((w + 2048u) & 4095u) - 2048;
    };
    for (int c = 0; c < m; ++c) {
        // the step made by column group c % 32 of half c / 32 (see the kernel)
        const int h = c / kTcRow, g = c % kTcRow;
        const int step = 1 + (G.v == 1 ? 2 * (kTcRow - 1 - g) + h : kTcRow * h + 4 * (7 - g % 8) + g / 8);
        uint64_t coef[2];
        ends(step, &coef[0], &coef[1]);
        int dig[2][16][2];
        i128 centre = 0;   // sum of fmax eps (units 1 / (2 p)): twice the error at the limbs' mid values
        u128 spread = 0;   // sum of fmax |eps|
        for (int x = 0; x < 2; ++x)
            for (int s = 0; s < per - 1; ++s) {
                dig[x][s][0] = dig[x][s][1] = 0;
                if (!fmax[s]) continue;
                const u128 num = (u128)F.mul(coef[x], F.pow(2, (uint64_t)pos[s])) << 24;
                const u128 W = (num + G.p / 2) / G.p;  // 2^24 c / p, rounded
                const i128 eps = (i128)(W * G.p) - (i128)num;
                centre += (i128)fmax[s] * eps;
                spread += (u128)fmax[s] * (u128)(eps < 0 ? -eps : eps);
                digits((uint32_t)W, dig[x][s]);
            }
        // error of t after centring: at most spread / (2 p) + 1/2
        const uint32_t margin = tc_margin(G.kind, G.v);
        if (spread / (2 * (u128)G.p) + 1 > margin) return false;
        const i128 shift = centre >= 0 ? (centre + (i128)G.p) / (2 * (i128)G.p) : -((-centre + (i128)G.p) / (2 * (i128)G.p));
        // the bias of 12.0 adds its f32 bits to the last digit (to the first, a
        // multiple of 2^12): take them away, add the margin
        int bias[2];
        digits(margin - (uint32_t)(int64_t)shift - 0x41400000u, bias);
        for (int d = 0; d < 2; ++d) {
            // every partial sum of the products stays within 2^22 units of the 1.5 2^23 that 12.0 is
            int64_t hi = bias[d] > 0 ? bias[d] : 0, lo = bias[d] < 0 ? bias[d] : 0;
            for (int x = 0; x < 2; ++x)
                for (int s = 0; s < per - 1; ++s) (dig[x][s][d] > 0 ? hi : lo) += (int64_t)fmax[s] * dig[x][s][d];
            if (hi >= (1 << 22) || lo < -(1 << 22)) return false;
            const int n = 2 * g + d;  // column
            for (int slot = 0; slot < 2 * per; ++slot) {
                const int x = slot / per, s = slot % per;
                // limbs are f 2^-24 and digits w 2^4, so a unit is 2^-20; the bias slots hold 1.0
                const uint16_t hb = s < per - 1 ? half_bits(dig[x][s][d], 4) : x == 0 ? half_bits(12, 0) : half_bits(bias[d], -20);
                // 8 x 16-byte core matrices, those of 8 columns together
                const size_t off = (size_t)(n >> 3) * (32 * per) + (size_t)(slot >> 3) * 128 + (size_t)(n & 7) * 16 + 2 * (slot & 7);
                memcpy(&T->image[h][off], &hb, 2);
            }
        }
    }
    return true;
}

}  // namespace prand
