// gb_wheel210.cuh -- the mod-210 wheel of the large primes' strikes, shared by
// the carried primes (gb_large.cu) and the batched ones (gb_batch.cu).
//
// The multiples m p with m divisible by 3, 5 or 7 are cleared by the stamp, so
// only m coprime to 210 is struck (48 of every 105 odd m).  From one coprime
// residue of m mod 210 to the next the bit index (m p - b) / 2 advances by p
// times half the gap (1 to 5); the tables, built at compile time, hold those
// half gaps, the inverse of p mod 210 and, for an odd residue, the next coprime
// one.
#pragma once

#include "gb_internal.cuh"

namespace gb {
namespace {

constexpr uint32_t kWheelPos = 48;          // residues mod 210 coprime to 210

constexpr bool coprime210(int r) { return r % 2 != 0 && r % 3 != 0 && r % 5 != 0 && r % 7 != 0; }

struct Wheel210 {
    uint8_t hgap[kWheelPos];    // half gap from wheel position w to w + 1 (position 47 -> 0: 209 -> 211)
    uint8_t inv[210];           // p^-1 mod 210 for p coprime to 210 (0 elsewhere)
    uint16_t next[210];         // odd r: position of the first coprime residue >= r | half the distance << 6
};

constexpr Wheel210 make_wheel210()
{
    Wheel210 t{};
    int res[kWheelPos + 1] = {};
    int n = 0;
    for (int r = 1; r < 210; ++r)
        if (coprime210(r)) res[n++] = r;
    res[kWheelPos] = 211;                   // 1 + 210: the first residue of the next period
    for (int w = 0; w < (int)kWheelPos; ++w) t.hgap[w] = (uint8_t)((res[w + 1] - res[w]) / 2);
    for (int p = 1; p < 210; ++p)
        if (coprime210(p))
            for (int u = 1; u < 210; ++u)
                if (p * u % 210 == 1) t.inv[p] = (uint8_t)u;
    for (int r = 1; r < 210; r += 2) {
        int w = 0;
        while (res[w] < r) ++w;             // res[48] = 211 >= every r
        t.next[r] = (uint16_t)((w % (int)kWheelPos) | (((res[w] - r) / 2) << 6));
    }
    return t;
}
__constant__ Wheel210 kWheel210 = make_wheel210();

// the wheel tables in shared memory (lanes read different entries)
struct WheelShared {
    uint8_t hgap[kWheelPos];
    uint8_t inv[210];
    uint16_t next[210];
};
__device__ __forceinline__ void load_wheel(WheelShared& ws)
{
    for (uint32_t t = threadIdx.x; t < 210; t += blockDim.x) {
        ws.inv[t] = kWheel210.inv[t];
        ws.next[t] = kWheel210.next[t];
        if (t < kWheelPos) ws.hgap[t] = kWheel210.hgap[t];
    }
}

// The wheel entry of the multiple b + 2 i of p (odd, i.e. m = (b + 2 i) / p
// odd), from b mod 210: the position of the first coprime residue >= m, half
// the distance to it << 6.
__device__ __forceinline__ uint32_t wheel_entry(const WheelShared& ws, uint32_t p, uint32_t b_mod210, uint32_t i)
{
    const uint32_t r = (b_mod210 + 2u * (i % 105u)) % 210u;
    return ws.next[(r * (uint32_t)ws.inv[p % 210u]) % 210u];
}

}  // namespace
}  // namespace gb
