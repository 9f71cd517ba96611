// Constants of the GM/GQ tensor-core generation (gm_tc.cuh), built on the host.
#pragma once
#include "prand_internal.h"

namespace prand {

constexpr int kTcSteps = 64;            // m: steps per block
constexpr int kTcRow = 32;              // steps per half of a block: v = 1 every second one, v = 4 consecutive ones
constexpr int kTcCols = 2 * kTcRow;     // accumulator columns of a half: two digits per step
constexpr int kTcCoefs = kTcSteps + 2;  // j = -1 .. 64

// How a value is cut into limbs, by the prime and the strip width v: its four
// bytes (32-bit primes, v = 1; 8 operand slots), or nibbles (16 slots).  The last
// slot of a value is the bias slot.
constexpr bool tc_nibbles(int kind, int v) { return kind == P51 || kind == P61 || v != 1; }
constexpr int tc_value_slots(int kind, int v) { return tc_nibbles(kind, v) ? 16 : 8; }
constexpr int kTcImage = kTcCols * 64;  // bytes of the largest B operand: 64 columns x 32 slots x 2

// Bound on the error of a fraction t in units of 2^-24, checked when the table is built.
constexpr uint32_t tc_margin(int kind, int v)
{
    return kind == P61 ? 82u : kind == P51 ? 62u : v != 1 ? 37u : kind == P19 ? 212u : 314u;
}

// One generator's constants, kept per device.  image[h]: B of half h's steps on
// [limbs of X0 | limbs of X1].
struct GmTcTable {
    unsigned char image[2][kTcImage];
    uint64_t v, q;                        // X2 = v X1 + q X0 (mod p)
    uint64_t a, b;                        // x^(n+m) = a x^(n) + b x^(n-1)
    uint64_t al[kTcCoefs], be[kTcCoefs];  // x^(n+j) = al X1 + be X2 (mod p), j = index - 1
};

// False if the constants do not meet the bounds the kernel relies on.
bool gm_tc_build(int gen, GmTcTable *T);

}  // namespace prand
