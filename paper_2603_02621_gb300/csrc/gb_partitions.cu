// gb_partitions.cu -- Goldbach partition counts r(n): the number of prime
// pairs p <= q with p + q = n (GoldbachGPU, arXiv 2603.02621, Sec. 4.5: the
// counting of all representations named as future work).
//
// With P the odd-only prime bitset of [1, M) (bit i <-> 2i + 1) and
// m = (n - 2) / 2, the odd pairs are the i <= m / 2 with P[i] and P[m - i]:
// r(n) = popcount over i <= m/2 of P[i] & P[m - i] (n = 4 = 2 + 2 is added
// apart).  P[m - i] is read from the bit-reversed copy Rev (Rev[k] =
// P[Mp - 1 - k], Mp = 32 * words), where it is bit s + i with s = Mp - 1 - m:
// one funnel shift per 32-bit word aligns 32 partners at once, so a word
// step is a funnel shift, an AND and a popcount for 32 pairs.  A warp takes 32
// consecutive n (one per lane) and a run of words; runs of the same n-block
// add into the counts with one atomic per lane.
//
// Many n with long sums go by residues mod 15 of i (mod 30 of the odd number):
// 8 of the 15 hold all primes above 5, and for a given n an i of residue c meets
// a partner of residue c' = m - c, so only the c with both among the 8 count --
// 64 of the 225 pairs (n, c), 0.28 of the words.  As in the block cover, a word
// of one residue is merged from streams: with 15 O words of P and O prime to
// 15, the words k, k + O, ..., k + 14 O hold residue c at 15 different phases,
// which fill the 32 bits of one merged word; the reversed bits are merged at the
// same stride, so that a pair stays a pair under the shift between them.  Then
// the words, not the n, are spread over the lanes: a lane holds three words of
// residue c and the 16 words of residue c' they meet for 32 n whose m are 15
// apart (so that all have the same c'), whose shifts 0, 15, ..., 465 are
// compile-time constants; three words' counts go through a carry-save adder to
// two popcounts.
//
// Bound: ALU and popcount pipes of that step (8 ALU, 2 popcounts, 2
// multiply-adds for 96 pairs of one n).  A call for 2000 n near 1e9 on a GB300,
// its sieve of 0.16 ms included: 7.75 ms by k_partitions alone, 1.48 ms.
#include <algorithm>
#include <utility>

#include "gb_internal.cuh"

namespace gb {

__global__ void __launch_bounds__(256) k_reverse_bits(const uint32_t* P, uint32_t* rev, uint64_t words)
{
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= words; v += (uint64_t)gridDim.x * blockDim.x)
        rev[v] = v < words ? __brev(P[words - 1 - v]) : 0u;          // one zero word past the end
}

// REST: of a stretch whose first words are counted by residues, the words from
// w_first on and the pairs that no residue holds (a kernel of its own: the loop of
// the plain counts was 4 % slower with it, 33 n near 1e9 612 us against 584)
template <bool REST>
__global__ void __launch_bounds__(256) k_partitions(const PartitionArgs a)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t warp_id = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t item = warp_id;
    if (item >= (uint64_t)a.n_blocks * a.runs) return;
    const uint64_t blk = item / a.runs, run = item - blk * a.runs;
    const uint64_t j = blk * 32 + lane;                              // n index in the range
    const bool valid = j < a.count;
    const uint64_t n = a.lo + 2 * j;
    const uint64_t m = valid ? (n - 2) / 2 : 0;
    const uint64_t imax = m / 2;                                     // i <= m / 2
    const uint64_t s = (uint64_t)a.words * 32 - 1 - m;              // Rev bit of P[m]
    const uint64_t w0 = (REST ? a.w_first : 0) + run * a.run_words;
    uint64_t w1 = w0 + a.run_words;
    const uint64_t wlast = imax / 32;                                // this lane's last word
    uint32_t cnt = 0;
    if (valid && n >= 6) {
        if (w1 > wlast + 1) w1 = wlast + 1;
        const uint32_t sh = (uint32_t)(s & 31);
        const uint64_t sw = s >> 5;
        for (uint64_t w = w0; w < w1; ++w) {
            const uint32_t pw = __ldg(a.P + w);
            const uint32_t lo_w = __ldg(a.rev + sw + w), hi_w = __ldg(a.rev + sw + w + 1);
            uint32_t x = pw & __funnelshift_r(lo_w, hi_w, sh);
            if (w == wlast) {
                const uint32_t b = (uint32_t)(imax & 31);            // bits 0..b of the last word
                x &= b == 31 ? 0xffffffffu : ((2u << b) - 1u);
            }
            cnt += __popc(x);
        }
    }
    if (run == 0 && valid && n == 4) cnt += 1;                       // 4 = 2 + 2
    if (REST && run == 0 && valid) {
        // the pairs of 3 and 5, which are in no residue prime to 30 (n > 16)
        cnt += (__ldg(a.P + ((m - 1) >> 5)) >> ((m - 1) & 31)) & 1u;
        cnt += (__ldg(a.P + ((m - 2) >> 5)) >> ((m - 2) & 31)) & 1u;
    }
    if (valid && cnt) atomicAdd(a.counts + j, cnt);
}

namespace {

// residues i mod 15 with 2 i + 1 prime to 30, and the place of each among them
// (4 bits each; place 15: not among them)
constexpr uint64_t kResidues = 0xeb986530ull;               // 0, 3, 5, 6, 8, 9, 11, 14
constexpr uint64_t make_places()
{
    uint64_t t = 0;
    for (uint32_t r = 0; r < 15; ++r) {
        uint64_t v = 15;
        for (uint32_t k = 0; k < 8; ++k)
            if (((kResidues >> (4 * k)) & 15u) == r) v = k;
        t |= v << (4 * r);
    }
    return t;
}
constexpr uint64_t kPlaces = make_places();
__device__ __forceinline__ uint32_t residue(uint32_t c) { return (uint32_t)(kResidues >> (4 * c)) & 15u; }
__device__ __forceinline__ uint32_t place(uint32_t r) { return (uint32_t)(kPlaces >> (4 * r)) & 15u; }

// bits b = phi (mod 15) of a word, phi in 0 .. 14
__device__ __forceinline__ uint32_t phase15(uint32_t phi) { return 0x40008001u << phi; }

}  // namespace

// Merged words: y[c][k], k < O, bit b = P[x + 32 O j] with x = 32 k + b and the
// one stream j that makes it the c-th residue mod 15; z[c][k], bit b = P[m_max -
// x - 32 O j], the one index that is the c-th residue.  One thread per k, all residues.
__global__ void __launch_bounds__(128) k_part_merge(const PartCorrArgs a)
{
    const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = 32 * (uint64_t)a.O;
    if (k < a.ny) {
        uint32_t acc[8] = {};
        if (k < a.O)
            for (uint32_t j = 0; j < 15; ++j) {
                const uint64_t x = 32 * k + stride * j;     // < 480 O: in P
                const uint32_t v = a.P[x >> 5], x15 = (uint32_t)(x % 15);
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[c] |= v & phase15((residue(c) + 15 - x15) % 15);
            }
#pragma unroll
        for (int c = 0; c < 8; ++c) a.y[c * a.ny + k] = acc[c];
    }
    if (k < a.nz) {
        uint32_t acc[8] = {};
        for (uint32_t j = 0; j < 15; ++j) {
            const int64_t top = (int64_t)a.m_max - (int64_t)(32 * k + stride * j);     // the word's bit 0
            if (top < 0) break;
            // bits top, top - 1, ..., top - 31 (those below 0 are not there)
            const int64_t bot = top - 31;
            uint32_t v;
            if (bot >= 0) {
                const uint32_t w = (uint32_t)(bot >> 5);
                const uint32_t sh = (uint32_t)bot & 31;
                v = __funnelshift_r(a.P[w], sh ? a.P[w + 1] : 0u, sh);
            } else {
                v = a.P[0] << (uint32_t)(-bot);
            }
            v = __brev(v);
            const uint32_t t15 = (uint32_t)(top % 15);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] |= v & phase15((t15 + 15 - residue(c)) % 15);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) a.z[c * a.nz + k] = acc[c];
    }
}

namespace {

template <int T>
__device__ __forceinline__ void corr_step(const uint32_t (&y)[3], const uint32_t (&w)[3][16], uint32_t (&cum)[32],
                                          uint32_t w1, uint32_t w2)
{
    constexpr int q = (15 * T) >> 5, sh = (15 * T) & 31;
    uint32_t p[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        p[i] = (sh ? __funnelshift_r(w[i][q], w[i][sh ? q + 1 : q], sh) : w[i][q]) & y[i];
    const uint32_t x = p[0] ^ p[1] ^ p[2], c = (p[0] & p[1]) | (p[2] & (p[0] | p[1]));
    cum[T] = __popc(x) * w1 + cum[T];
    cum[T] = __popc(c) * w2 + cum[T];
}

template <int... T>
__device__ __forceinline__ void corr_steps(std::integer_sequence<int, T...>, const uint32_t (&y)[3],
                                           const uint32_t (&w)[3][16], uint32_t (&cum)[32], uint32_t w1, uint32_t w2)
{
    (corr_step<T>(y, w, cum, w1, w2), ...);
}

}  // namespace

// A warp takes 32 n of one m mod 15 (m = m_top - 15 t) and a run of merged words,
// over the residues c that meet a residue.
__global__ void __launch_bounds__(128, 4) k_part_corr(const PartCorrArgs a)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t item = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (item >= (uint64_t)a.blocks * 15 * a.runs) return;
    const uint32_t run = (uint32_t)(item % a.runs), bl = (uint32_t)(item / a.runs), g = bl / 15, d = bl % 15;
    // m of the block's first n: m_max - d - 480 g, and s = m_max - m
    if (a.m_max < (uint64_t)d + 480ull * g + a.m_min) return;           // no n of the range in the block
    const uint64_t m_top = a.m_max - d - 480ull * g;
    const uint32_t r15 = (uint32_t)(m_top % 15);
    const uint32_t k0 = run * a.run_words, k1 = min(a.ny, k0 + a.run_words);      // multiples of 96
    uint32_t cum[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) cum[t] = 0;
    for (uint32_t c = 0; c < 8; ++c) {
        const uint32_t o = place((r15 + 15 - residue(c)) % 15);
        if (o == 15) continue;
        const uint32_t* y = a.y + (uint64_t)c * a.ny + lane;
        const uint32_t* z = a.z + (uint64_t)o * a.nz + 15 * g + lane;
        for (uint32_t k = k0; k < k1; k += 96) {
            uint32_t v[3], w[3][16];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                v[i] = __ldg(y + k + 32 * i);
                uint32_t lo = __ldg(z + k + 32 * i);
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const uint32_t hi = __ldg(z + k + 32 * i + q + 1);
                    w[i][q] = __funnelshift_r(lo, hi, d);
                    lo = hi;
                }
            }
            corr_steps(std::make_integer_sequence<int, 32>{}, v, w, cum, a.w1, a.w2);
        }
    }
    // the lanes' counts: at each stage a lane keeps half of them, lane t ends with the t-th
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int h = 16 >> st;
        const bool up = (lane & (uint32_t)h) != 0;
#pragma unroll
        for (int t = 0; t < h; ++t) {
            const uint32_t send = up ? cum[t] : cum[t + h], keep = up ? cum[t + h] : cum[t];
            cum[t] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    }
    const uint64_t off = 15ull * lane;
    if (m_top >= off + a.m_min && cum[0]) atomicAdd(a.counts + (m_top - off - a.m_min), cum[0]);
}

uint64_t part_stream_words(uint64_t i_end)
{
    uint64_t o = i_end / 480;
    while (o && (o % 3 == 0 || o % 5 == 0)) --o;
    return o;
}

cudaError_t launch_part_corr(const PartCorrArgs& a0, cudaStream_t s)
{
    PartCorrArgs a = a0;
    if (!a.P || !a.y || !a.z || !a.counts || a.O == 0 || a.O % 3 == 0 || a.O % 5 == 0 || a.ny % 96 || a.ny < a.O ||
        a.m_max < a.m_min || a.run_words % 96 || a.run_words == 0)
        return cudaErrorInvalidValue;
    a.blocks = (uint32_t)((a.m_max - a.m_min) / 480 + 1);
    a.runs = (a.ny + a.run_words - 1) / a.run_words;
    if (a.nz < a.ny + 15ull * a.blocks + 17) return cudaErrorInvalidValue;
    a.w1 = 1;
    a.w2 = 2;
    const uint64_t words = std::max<uint64_t>(a.ny, a.nz);
    k_part_merge<<<(unsigned)((words + 127) / 128), 128, 0, s>>>(a);
    const uint64_t ctas = ((uint64_t)a.blocks * 15 * a.runs + 3) / 4;
    if (ctas > 0x7fffffffull) return cudaErrorInvalidValue;
    k_part_corr<<<(unsigned)ctas, 128, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_reverse_bits(const uint32_t* P, uint32_t* rev, uint64_t words, cudaStream_t s)
{
    if (!P || !rev) return cudaErrorInvalidValue;
    const uint64_t blocks = (words + 1 + 255) / 256;
    const uint64_t cap = (uint64_t)device_sms() * 32;
    k_reverse_bits<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, s>>>(P, rev, words);
    return cudaGetLastError();
}

cudaError_t launch_partitions(const PartitionArgs& a, cudaStream_t s)
{
    const uint64_t warps = (uint64_t)a.n_blocks * a.runs;
    if (warps == 0) return cudaSuccess;
    if (!a.P || !a.rev || !a.counts || a.runs == 0) return cudaErrorInvalidValue;
    const uint64_t blocks = (warps + 7) / 8;
    if (blocks > 0x7fffffffull) return cudaErrorInvalidValue;
    if (a.w_first) k_partitions<true><<<(unsigned)blocks, 256, 0, s>>>(a);
    else k_partitions<false><<<(unsigned)blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace gb
