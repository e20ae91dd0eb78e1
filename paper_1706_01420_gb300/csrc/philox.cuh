// Philox-4x32-10 (Salmon, Moraes, Dror and Shaw, "Parallel random numbers: as
// easy as 1, 2, 3", SC'11), written out here.  Every draw is a pure function of (counter, key), so the
// generators address their random numbers by (index, toy, call) and the
// result of a draw does not depend on which thread makes it.
#pragma once

#include <stdint.h>

#include "ipa_internal.cuh"

namespace ipa {

constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;

struct U4 {
    uint32_t x, y, z, w;
};

// Ten rounds.  Round: (hi0, lo0) = M0 * c0, (hi1, lo1) = M1 * c2,
// c <- (hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0); key bumped by (W0, W1) between rounds.
__device__ __forceinline__ U4 philox(U4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += kPhiloxW0;
            k1 += kPhiloxW1;
        }
        const uint32_t lo0 = kPhiloxM0 * c.x, hi0 = __umulhi(kPhiloxM0, c.x);
        const uint32_t lo1 = kPhiloxM1 * c.z, hi1 = __umulhi(kPhiloxM1, c.z);
        c = U4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
    }
    return c;
}

// The ten rounds' keys laid out beforehand, for kernels that take them as a
// parameter and read them from the parameter bank (an operand of the rounds'
// exclusive-ors instead of two additions per round).
struct PhiloxKeys {
    uint32_t k[20];
    PhiloxKeys() = default;
    explicit PhiloxKeys(uint64_t seed) {
        for (int r = 0; r < 10; ++r) {
            k[2 * r] = (uint32_t)seed + (uint32_t)r * kPhiloxW0;
            k[2 * r + 1] = (uint32_t)(seed >> 32) + (uint32_t)r * kPhiloxW1;
        }
    }
};
// Rounds R to 9.
template <int R>
__device__ __forceinline__ U4 keyed_from(const PhiloxKeys& keys, U4 c) {
#pragma unroll
    for (int r = R; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)kPhiloxM0 * c.x, p1 = (unsigned long long)kPhiloxM1 * c.z;
        c = U4{(uint32_t)(p1 >> 32) ^ c.y ^ keys.k[2 * r], (uint32_t)p1,
               (uint32_t)(p0 >> 32) ^ c.w ^ keys.k[2 * r + 1], (uint32_t)p0};
    }
    return c;
}
__device__ __forceinline__ U4 keyed(const PhiloxKeys& keys, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) {
    return keyed_from<0>(keys, U4{c0, c1, c2, c3});
}

// The first two rounds apart, for draws of all pairs of some (c0, c3) with some (c1, c2):
// after them the counter is (a ^ y, b, c ^ h, w), with (a, b, c) from c0 and c3 alone
// and (y, h, w) from c1 and c2 alone; four of the twenty products less per draw.
struct PhiloxRow {       // of (c0, c3)
    uint32_t a, b, c;
};
struct PhiloxCol {       // of (c1, c2)
    uint32_t y, h, w;
};
__device__ __forceinline__ PhiloxRow philox_row(const PhiloxKeys& keys, uint32_t c0, uint32_t c3) {
    const unsigned long long p = (unsigned long long)kPhiloxM0 * c0;
    const unsigned long long q = (unsigned long long)kPhiloxM1 * ((uint32_t)(p >> 32) ^ c3 ^ keys.k[1]);
    return PhiloxRow{(uint32_t)(q >> 32) ^ keys.k[2], (uint32_t)q, (uint32_t)p ^ keys.k[3]};
}
__device__ __forceinline__ PhiloxCol philox_col(const PhiloxKeys& keys, uint32_t c1, uint32_t c2) {
    const unsigned long long p = (unsigned long long)kPhiloxM1 * c2;
    const unsigned long long q = (unsigned long long)kPhiloxM0 * ((uint32_t)(p >> 32) ^ c1 ^ keys.k[0]);
    return PhiloxCol{(uint32_t)p, (uint32_t)(q >> 32), (uint32_t)q};
}

// Counter (idx lo32, idx hi32, toy, call) with key (k0, k1).
__device__ __forceinline__ U4 draw(uint64_t idx, uint32_t toy, uint32_t call, uint32_t k0, uint32_t k1) {
    return philox(U4{(uint32_t)idx, (uint32_t)(idx >> 32), toy, call}, k0, k1);
}

}  // namespace ipa
