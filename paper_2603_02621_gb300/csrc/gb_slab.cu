// gb_slab.cu -- the segment sieve of a long window, one shared-memory slab of
// 13 * 2^17 odd numbers (208 KB, nearly all an SM has) per CTA at a time: stamp,
// every sieving prime below 2^20, store -- the tile sieve and the slices
// (gb_sieve.cu) in one pass, for windows that give every SM its slabs
// (GoldbachGPU, arXiv 2603.02621, Sec. 2.3.1 and 4.5; layout of Sec. 2.2).
//
// Against tiles of 2^18 bits and slices of 1.75 * 2^20 read back from memory:
// the window is written once and not read; a prime is started once per slab
// instead of once per tile, or once more per slice; and a warp-struck prime
// leaves each lane enough strikes (104 and more below 512) that all of them can
// start in distinct banks (below).
//
// Work inside a slab is taken from one queue by the warps, longest first, between
// two barriers: the smallest primes one warp each, then 32 primes to a warp (a
// thread each, up to 1700 strikes), then, from 2^13 on, 128 primes to a warp,
// four starts per thread overlapping.  A slab is stored and the next one stamped
// over it in one pass.
//
// Bound: instruction issue and shared-memory wavefronts together (70 and 78 % of
// their peaks at 5e11).  2^33 odd numbers near 5e11 on a
// GB300: 3.77 ms by tiles and slices, 3.53 ms.  The strike loops are unrolled and
// their ends masked rather than branched around: as plain loops, with a branch
// per strike, the pass took 5.1 ms.
#include <algorithm>

#include "gb_internal.cuh"
#include "gb_sieve_tile.cuh"

namespace gb {

namespace {

constexpr int kNT = 1024;

// The stamp tables in shared memory, each 96 words longer than its period needs:
// a thread reads four words of a warp's 128 at one offset (rows of 32 words,
// 1024 bits apart), so that a table's offset is advanced and its word address
// and shift computed once per four words.
constexpr uint32_t kRows = 4;
constexpr uint32_t kExt = 32 * (kRows - 1);
constexpr uint32_t kM[4] = {kWheelM1, kWheelM2, kWheelM3, kWheelM4};
constexpr uint32_t kW[4] = {kWheelW1, kWheelW2, kWheelW3, kWheelW4};
constexpr uint32_t kAt[4] = {0, kWheelW1, kWheelW1 + kWheelW2, kWheelW1 + kWheelW2 + kWheelW3};   // in the global tables
constexpr uint32_t kTabWords = (kWheelWords + 4 * kExt + 3) & ~3u;
constexpr uint32_t kTab[4] = {kAt[0], kAt[1] + kExt, kAt[2] + 2 * kExt, kAt[3] + 3 * kExt};     // in shared memory
static_assert(kTabWords * 4 + kSlabBits / 8 + 1024 <= 227 * 1024, "shared memory");

template <int T>
__device__ __forceinline__ void load_table(uint32_t* tab, const uint32_t* wheel)
{
    constexpr uint32_t M = kM[T], W = kW[T], from = kAt[T], to = kTab[T];
    for (uint32_t i = threadIdx.x; i < W + kExt; i += kNT) {
        const uint32_t x = 32 * i % M;                      // the word's first bit, in the first period
        tab[to + i] = stamp_word(wheel + from, x);          // (W words hold M + 64 bits)
    }
}

// four words' patterns of table T at offset a, anded into v
template <int T>
__device__ __forceinline__ void stamp4(const uint32_t* tab, uint32_t a, uint32_t (&v)[kRows])
{
    constexpr uint32_t at = kTab[T];
    const uint32_t* t = tab + at + (a >> 5);
#pragma unroll
    for (uint32_t r = 0; r < kRows; ++r) v[r] &= __funnelshift_r(t[32 * r], t[32 * r + 1], a & 31);
}

// The numbers below 44 of the window: the stamped primes are prime, numbers
// below 2 are not.
__device__ __noinline__ void fix_small(uint32_t* sm, int64_t b, uint32_t nw)
{
    for (uint32_t w = threadIdx.x; w < nw; w += kNT) {
        const int64_t v0 = b + 64 * (int64_t)w;
        if (v0 > 43) break;
        uint32_t v = sm[w];
        for (uint32_t k = 0; k < 32; ++k) {
            const int64_t num = v0 + 2 * (int64_t)k;
            if (num < 2) v &= ~(1u << k);
            else if (num <= 43 && num != 9 && num != 15 && num != 21 && num != 25 && num != 27 && num != 33 &&
                     num != 35 && num != 39)
                v |= 1u << k;
        }
        sm[w] = v;
    }
}

// first multiple of p to strike in the slab whose first number is b: the first
// odd one, from p^2 on; 0xffffffff when p^2 is beyond the slab
__device__ __forceinline__ uint32_t slab_start(int64_t b, int64_t last, bool squares, uint32_t p, uint64_t m)
{
    uint32_t i;
    if (b > 0) {                                            // (p < 2^20)
        const uint32_t r = neg_mod_low((uint64_t)b, p, m);
        i = (r + ((r & 1u) ? p : 0u)) >> 1;
    } else {
        i = first_odd_multiple(b, p, m);
    }
    if (squares) {
        const int64_t pp = (int64_t)((uint64_t)p * p);
        if (pp > last) return 0xffffffffu;
        if (pp > b) i = max(i, (uint32_t)((uint64_t)(pp - b) >> 1));    // same residue class mod p
    }
    return i;
}

// and to a word of the slab, by shared-memory byte address (sa: the slab's)
__device__ __forceinline__ void clear_bits(uint32_t sa, uint32_t addr, uint32_t mask)
{
    if (!GB_DCHECK(addr - sa < kSlabBits / 8, kDbgTileStrike)) return;
    (void)sa;
    asm volatile("red.shared.and.b32 [%0], %1;" :: "r"(addr), "r"(mask) : "memory");
}

// clear bit i of the slab (its word's address by a shift and a shift-and-add)
__device__ __forceinline__ void strike_bit(uint32_t sa, uint32_t i)
{
    clear_bits(sa, sa + ((i >> 5) << 2), __funnelshift_l(0xfffffffeu, 0xfffffffeu, i));
}

// clear bit i of the slab if i < nb, without a branch
__device__ __forceinline__ void strike_if(uint32_t sa, uint32_t i, uint32_t nb)
{
    asm volatile("{ .reg .pred p; setp.lt.u32 p, %0, %1; @p red.shared.and.b32 [%2], %3; }"
                 :: "r"(i), "r"(nb), "r"(sa + ((i >> 5) << 2)), "r"(__funnelshift_l(0xfffffffeu, 0xfffffffeu, i))
                 : "memory");
}

}  // namespace

template <bool COUNT>
__global__ void __launch_bounds__(kNT, 1) k_slab(const SlabArgs a)
{
    extern __shared__ uint32_t smem[];
    uint32_t* const tab = smem;
    uint32_t* const sm = smem + kTabWords;                  // 16-byte aligned
    __shared__ uint32_t s_next, s_below;
    const uint32_t slab_bits = a.slab_bits;
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(sm);
    const int lane = threadIdx.x & 31;
    const uint32_t warp = threadIdx.x >> 5;
    load_table<0>(tab, a.wheel);
    load_table<1>(tab, a.wheel);
    load_table<2>(tab, a.wheel);
    load_table<3>(tab, a.wheel);
    const uint32_t n_single = (a.n_quad - a.n_warp + 31) / 32;          // 32-prime items
    const uint32_t n_items = a.n_warp + n_single + (a.n_primes - a.n_quad + 127) / 128;
    // first item whose primes are all from wheel_below on
    const uint32_t item_plain = a.n_warp + n_single + (a.n_plain > a.n_quad ? (a.n_plain - a.n_quad + 127) / 128 : 0);
    const uint64_t slabs = (a.nbits + slab_bits - 1) / slab_bits;
    unsigned long long nstrike = 0;
    uint32_t cnt = 0;

    // 1. stamp of 3..43 of the slab at t0, by rows of 32 words, warp w taking the
    // words 128 w .. 128 w + 127, then 128 kNT / 32 further on.  The slab before
    // it, at `done` (a whole one), leaves in the same pass: each thread stores a
    // word of it, if the words are wanted, and stamps the next slab over it.
    auto stamp = [&](uint64_t t0, bool leave, uint64_t done) {
        const int64_t b = a.B + 2 * (int64_t)t0;            // number of the slab's bit 0
        if (threadIdx.x == 0) {
            s_next = 0;
            // primes with p^2 <= b: of the rest, few, the squares are looked at
            uint32_t lo = 0, hi = b > 0 ? a.n_primes : 0u;
            if (hi && (uint64_t)b >= a.p_max2) lo = hi;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) / 2;
                const uint64_t p = a.primes[mid];
                if ((int64_t)(p * p) <= b) lo = mid + 1;
                else hi = mid;
            }
            s_below = lo;
        }
        const int64_t x0 = (b - 1) / 2 + 32 * (int64_t)(128 * warp + lane);     // (number - 1) / 2 of the thread's first bit
        constexpr uint32_t step = 32u * 128u * (kNT / 32);
        constexpr uint32_t m0 = kM[0], m1 = kM[1], m2 = kM[2], m3 = kM[3];
        constexpr uint32_t s0 = step % m0, s1 = step % m1, s2 = step % m2, s3 = step % m3;
        uint32_t a0 = pmod_u32(x0, m0), a1 = pmod_u32(x0, m1), a2 = pmod_u32(x0, m2), a3 = pmod_u32(x0, m3);
        uint32_t* const dst = leave && a.out ? a.out + done / 32 : nullptr;
        for (uint32_t w = 128 * warp + lane; w < slab_bits / 32; w += 128 * (kNT / 32)) {
            uint32_t v[kRows];
            if (leave) {
#pragma unroll
                for (uint32_t r = 0; r < kRows; ++r) v[r] = sm[w + 32 * r];
                if (dst)
#pragma unroll
                    for (uint32_t r = 0; r < kRows; ++r) dst[w + 32 * r] = v[r];
                if (a.popcount)
#pragma unroll
                    for (uint32_t r = 0; r < kRows; ++r) cnt += __popc(v[r]);
            }
#pragma unroll
            for (uint32_t r = 0; r < kRows; ++r) v[r] = 0xffffffffu;
            stamp4<0>(tab, a0, v);
            stamp4<1>(tab, a1, v);
            stamp4<2>(tab, a2, v);
            stamp4<3>(tab, a3, v);
#pragma unroll
            for (uint32_t r = 0; r < kRows; ++r) sm[w + 32 * r] = v[r];
            a0 += s0; if (a0 >= m0) a0 -= m0;
            a1 += s1; if (a1 >= m1) a1 -= m1;
            a2 += s2; if (a2 >= m2) a2 -= m2;
            a3 += s3; if (a3 >= m3) a3 -= m3;
        }
        __syncthreads();
        if (b <= 43) {
            fix_small(sm, b, slab_bits / 32);
            __syncthreads();
        }
    };

    __syncthreads();                                        // tables loaded
    if (blockIdx.x < slabs) stamp((uint64_t)blockIdx.x * slab_bits, false, 0);
    for (uint64_t s = blockIdx.x; s < slabs; s += gridDim.x) {
        const uint64_t t0 = s * slab_bits;
        const uint64_t rem = a.nbits - t0;
        const uint32_t nb = rem < slab_bits ? (uint32_t)rem : slab_bits;
        const int64_t b = a.B + 2 * (int64_t)t0;            // number of the slab's bit 0
        const int64_t last = b + 2 * (int64_t)(nb - 1);

        // 2. strikes
        const uint32_t below = s_below;
        const uint32_t bmod30 = pmod_u32(b, 30);
        const bool whole = !COUNT && nb == slab_bits;
        const uint32_t bh = (uint32_t)((uint64_t)b >> 32), bl = (uint32_t)b;
        for (;;) {
            uint32_t item = 0;
            if (lane == 0) item = atomicAdd(&s_next, 1u);
            item = __shfl_sync(0xffffffffu, item, 0);
            if (item >= n_items) break;
            if (item < a.n_warp) {
                // one prime, the warp's: lane l strikes j0 + l q + 32 q t, whole
                // words apart, so its mask is fixed.  It starts at the strike
                // t = rot whose word lies in bank l, runs to the end and strikes
                // rot - 1 .. 0 after: at every step the 32 lanes' words are in 32
                // distinct banks (each lane's bank moves by q, or by -q, per step)
                const uint32_t q = a.primes[item];
                const uint32_t j0 = slab_start(b, last, item >= below, q, a.recip[item]);
                if (j0 >= nb) continue;
                if (COUNT && lane == 0) nstrike += (nb - 1 - j0) / q + 1;
                const uint32_t i = j0 + (uint32_t)lane * q;
                if (i < nb) {
                    const uint32_t mask = __funnelshift_l(0xfffffffeu, 0xfffffffeu, i);
                    const uint32_t w0 = i >> 5;
                    const uint32_t end = (nb - (i & 31u) + 31u) >> 5;     // words whose bit i & 31 is < nb
                    const uint32_t qinv = q * (2u - q * q);               // q^-1 mod 64 (q odd)
                    uint32_t rot = (((uint32_t)lane - w0) * qinv) & 31u;
                    if (w0 + rot * q >= end) rot = 0;                     // a short (last) slab
                    const uint32_t q4 = 4 * q, stop = sa + 4 * end;       // byte addresses
                    const uint32_t from = sa + 4 * (w0 + rot * q);
                    uint32_t x = from;
                    for (; x + 7 * q4 < stop; x += 8 * q4) {
                        uint32_t y = x;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            clear_bits(sa, y, mask);
                            y += q4;
                        }
                    }
                    for (; x < stop; x += q4) clear_bits(sa, x, mask);
                    x = from;
                    for (; rot >= 4; rot -= 4) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            x -= q4;
                            clear_bits(sa, x, mask);
                        }
                    }
                    for (; rot > 0; --rot) {
                        x -= q4;
                        clear_bits(sa, x, mask);
                    }
                }
                continue;
            }
            constexpr int U = 4;
            if (whole && item >= item_plain && a.n_quad + 128 * (item - a.n_warp - n_single) + 128 <= below) {
                // 128 primes from wheel_below on, a whole slab past their squares: four
                // starts per thread, then as many strikes as every lane of the 32 has,
                // unconditionally, and the one or two more that some have
                const uint32_t k = a.n_quad + 128 * (item - a.n_warp - n_single) + lane;
                uint32_t p[U], i[U], g[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    p[u] = __ldg(a.primes + k + 32 * u);
                    const uint64_t m = __ldg(a.recip + k + 32 * u);
                    const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
                    // as neg_mod_low with a quotient 1 to 5 above floor(b / p): q p - b,
                    // in (0, 5p], is already the negative
                    const uint32_t q = bh * mh + 5u + mulhi_u32(bh, ml) + mulhi_u32(bl, mh);
                    uint32_t t = q * p[u] - bl;
                    t = __viaddmin_u32(t, 0u - 2 * p[u], t);              // (wraps above t when t < 2p)
                    t = __viaddmin_u32(t, 0u - 2 * p[u], t);
                    t = __viaddmin_u32(t, 0u - p[u], t);                  // < p
                    i[u] = (t + (t & 1u) * p[u]) >> 1;
                    g[u] = mulhi_u32(slab_bits, __shfl_sync(0xffffffffu, mh, 31));   // <= slab / largest p
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    uint32_t n = g[u];
                    for (; n >= 4; n -= 4)
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            strike_bit(sa, i[u]);
                            i[u] += p[u];
                        }
                    for (; n; --n) {
                        strike_bit(sa, i[u]);
                        i[u] += p[u];
                    }
                    do {
                        strike_if(sa, i[u], slab_bits);
                        i[u] += p[u];
                    } while (__any_sync(0xffffffffu, i[u] < slab_bits));
                }
                continue;
            }
            // a thread each: 32 primes, or four times 32 from n_quad on
            const bool quad = item >= a.n_warp + n_single;
            const uint32_t k0 = quad ? a.n_quad + 128 * (item - a.n_warp - n_single) : a.n_warp + 32 * (item - a.n_warp);
            const uint32_t k_end = quad ? a.n_primes : a.n_quad;
            uint32_t p[U], j[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t k = k0 + 32 * u + lane;
                p[u] = 0;
                j[u] = 0xffffffffu;
                if ((u == 0 || quad) && k < k_end) {
                    p[u] = a.primes[k];
                    j[u] = slab_start(b, last, k >= below, p[u], a.recip[k]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                uint32_t i = j[u];
                if (i >= nb) continue;
                if (p[u] < a.wheel_below) {
                    // only m p with m coprime to 30 (the stamp cleared the multiples
                    // of 3 and 5): see kHalfGaps30
                    const uint32_t jr = wheel30_at(p[u], bmod30, i % 15u);
                    i += p[u] * wheel30_skip(jr);                                   // < 2^21 + 4 * 2^20
                    uint32_t g = wheel30_gaps(jr);
                    // four at a time: three consecutive half gaps sum to 7 at most
                    while (i + 7 * p[u] < nb) {
                        const uint32_t i1 = i + p[u] * (g & 15u), i2 = i1 + p[u] * ((g >> 4) & 15u),
                                       i3 = i2 + p[u] * ((g >> 8) & 15u);
                        strike_bit(sa, i);
                        strike_bit(sa, i1);
                        strike_bit(sa, i2);
                        strike_bit(sa, i3);
                        i = i3 + p[u] * ((g >> 12) & 15u);
                        g = __funnelshift_r(g, g, 16);
                        if (COUNT) nstrike += 4;
                    }
#pragma unroll
                    for (int t = 0; t < 5; ++t) {           // (i + 7p >= nb, five half gaps sum to 8 at least)
                        if (COUNT) nstrike += i < nb;
                        strike_if(sa, i, nb);
                        i += p[u] * (g & 15u);
                        g >>= 4;
                    }
                } else {
                    if (COUNT) nstrike += (nb - 1 - i) / p[u] + 1;
                    const uint32_t p1 = p[u];
                    do {                                    // four at a time, the last ones masked
                        strike_if(sa, i, nb);
                        strike_if(sa, i + p1, nb);
                        strike_if(sa, i + 2 * p1, nb);
                        strike_if(sa, i + 3 * p1, nb);
                        i += 4 * p1;
                    } while (i < nb);
                }
            }
            __syncwarp();
        }
        __syncthreads();

        // 3. on to the CTA's next slab, or clear the bits past the window's end,
        // store and count
        if (s + gridDim.x < slabs) {
            stamp((s + gridDim.x) * slab_bits, true, t0);
            continue;
        }
        const uint32_t nw = ((nb + 63) / 64) * 2;           // whole 64-bit words
        for (uint32_t w = threadIdx.x; w < nw; w += kNT) {
            uint32_t v = sm[w];
            if (32 * w >= nb) v = 0;
            else if (nb - 32 * w < 32) v &= (1u << (nb - 32 * w)) - 1u;
            cnt += __popc(v);
            if (a.out) a.out[t0 / 32 + w] = v;
        }
    }
    if (COUNT) {
        for (int o = 16; o; o >>= 1) nstrike += __shfl_xor_sync(0xffffffffu, nstrike, o);
        if (lane == 0 && nstrike) atomicAdd(a.strikes, nstrike);
    }
    if (a.popcount) {
        unsigned long long c = cnt;
        for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0 && c) atomicAdd(a.popcount, c);
    }
}

cudaError_t launch_slab(const SlabArgs& a0, cudaStream_t s)
{
    if (a0.nbits == 0) return cudaSuccess;
    if (!a0.primes || !a0.recip || !a0.wheel || a0.n_warp > a0.n_quad || a0.n_quad > a0.n_primes) return cudaErrorInvalidValue;
    // as many rounds of slabs as the window needs, of equal length (whole blocks
    // of 128 words, the stamp's)
    SlabArgs a = a0;
    const uint64_t sms = device_sms(), rounds = (a.nbits + kSlabBits * sms - 1) / (kSlabBits * sms);
    a.slab_bits = (uint32_t)std::min<uint64_t>(kSlabBits, (a.nbits / (rounds * sms) + 4096) / 4096 * 4096);
    const size_t smem = kTabWords * 4 + kSlabBits / 8;
    const uint64_t slabs = (a.nbits + a.slab_bits - 1) / a.slab_bits;
    auto k = a.strikes ? k_slab<true> : k_slab<false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)(slabs < sms ? slabs : sms), kNT, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace gb
