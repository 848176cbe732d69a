// gb_cover_fast.cu -- block form of the loop-inverted Goldbach cover.
//
// Same computation as the generic cover (gb_cover.cu): for p = 3, 5, 7, ... <= P
// in ascending order, every even n whose partner n - p is prime and that no
// smaller p covered gets p_min(n) = p (GoldbachGPU, arXiv 2603.02621, Sec.
// 2.3.1-2.3.2, in the bitwise form of Sec. 4.3).  Only the schedule differs.
//
// Classes mod 3.  For half of the primes p the partner of an n not divisible by
// 3 is a multiple of 3, and a step over a word of consecutive n works for two
// n in three.  So the n are taken by their residue v mod 3, each class with its
// own useful primes: for v = 0 all from 5 on, for v = 1 those = 2 (mod 3) and 3,
// for v = 2 those = 1 (mod 3) and 3 (the partner 3 itself is p_min's only for
// n = 6, set apart like n = 4 = 2 + 2).  A word of one class comes from three
// places: a chunk of the window is cut into three streams of O words each, O not
// a multiple of 3, and since 32 = 2 (mod 3) the bits of one residue sit at three
// different phases in the words k, k + O and k + 2 O; an AND with the phase's
// mask and an OR put them side by side into one word, at the bit positions they
// had.  That is done once per chunk for the q of residue 1 and 2 (2 logic
// operations per word; q divisible by 3 drop out), into shared memory.  A shift
// by (p - 3)/2 bits then means the same in the merged words as in the window's,
// so a step is what it was, over words of 32 n of one class, and only two thirds
// of the steps are left.
//
// Steps.  With the halo chosen so that d_3 = (H - 4)/2 is a multiple of 32, the
// partner bits of word w for the prime p start at bit 32(w + d_3/32) - (p-3)/2 of
// Q: the word offset and the shift of every step are compile-time constants, and
// the few words a lane needs sit in registers.  A step is then
//     s = funnel-shift of two window registers,  C |= s,  cum_k += popc(C)
// and the histogram follows from the cumulative counts:
// #{n : p_min(n) = p_k} = cum_k - cum_{k-1} (three counts per register, added
// by multiply-adds with the field weights).  Block 0 (L0 useful primes) runs on
// every word of the class, three consecutive words per lane sharing one window;
// the words it leaves open (about one in four after 32 useful primes near 5e11)
// go to per-warp lists in shared memory, and blocks of 16 run on the open words
// alone, each leaving a shorter list.
//
// Probing.  The few n open after the last block, or in the last few words of a
// list, are taken one at a time by a warp: lane t probes the bit of Q at j + d_k
// for k = k0 + t, and the lowest set bit of the ballot is p_min.  An n still open
// after K primes goes to the retry pass (or counts as unresolved).
//
// The largest p_min, with its smallest n, of a warp's words of a class comes
// from the probing when any n reached it: every n of the class covered by the
// blocks has a smaller one.  Where a later block covers all that was open, its
// input list is still there and is run once more, recording it; where block 0
// does (a few words only), or no probed n is covered (a small bound), the merged
// words are, unless the blocks' last prime is below the chunk's maximum so far.
//
// Bound: the ALU pipe and the popcounts of block 0 (a step on three words is 8
// ALU, 2 popcount and 3 multiply-add instructions).  2^32 n from 4 on, 2^33
// near 5e11, 2^31 near 1e15 and 2^32 below 4e18 on a GB300: 1.69, 3.86, 1.26 and
// 3.13 ms without the classes (48 or 64 primes over every word, blocks of 32),
// 1.15, 2.64, 0.87 and 2.02 ms with them.
#include <algorithm>
#include <type_traits>
#include <utility>

#include "gb_internal.cuh"
#include "gb_sieve_tile.cuh"

namespace gb {

// cumulative counts are kept three per register (10-bit fields): a lane adds
// at most 96 per round of three words and runs at most ten rounds, or at most
// 32 per listed word and handles at most 30 of them (960 < 2^10)
constexpr int kCumBits = 10;
constexpr uint32_t kCumMask = (1u << kCumBits) - 1;
constexpr uint32_t kMaxRounds = 10;

// schedule: block 0 of L0 useful primes, then at most kMaxLater blocks of kLater
constexpr int kLater = 16;
constexpr int kMaxUseful = 128;
constexpr int kMaxPrefix = 256;
// a list this short is probed rather than run through another block (a block
// costs about 150 warp instructions, an open n about 40; 2^33 n near 5e11: 2.66
// ms with 1, 2.64 with 3, 2.71 with 8, 2.86 with 16)
constexpr uint32_t kProbeWords = 3;

// Threads per CTA, and rounds of merged words (96 per warp) per class and chunk.
// Two CTAs of 512 per SM, each warp through one class after the other: their
// sixteen warps are mostly in the same code (see block0_class).  A chunk has
// fixed costs (the counts' flushes, the merging's ends, the last words' probing),
// so it is as long as shared memory allows, five rounds (103 KB) -- 2^33 n near
// 5e11 take 2.83 ms with four and 2.64 with five; 2.65 with 256 threads, four
// CTAs and a barrier between the classes, 2.97 with 1024 -- unless the call is
// too small to give every SM its chunks.
constexpr int kCoverNT = 512, kFusedNT = 256;
constexpr int kCoverCtas = 2;                               // per SM
// Chunks of at most 96 merged words (segments of 2^11 .. 2^13, batches of ranges of
// at most 9216 n) are one warp per class: CTAs of 128, eight per SM.  2^24 n near
// 1e12, segments of 2^11, 2^12 and 2^13: 72, 39 and 25 us (319, 166 and 98 with CTAs
// of 512 whose first warp took the three classes one after the other); a batch of
// 1000 ranges of 1000 n near 1e9: 22 us (37).
constexpr int kShortNT = 128;
constexpr int kMaxWarps = kCoverNT / 32;
constexpr uint32_t kShortStream = 96;
constexpr uint32_t kRounds = 5;
constexpr uint32_t kFusedRounds = 3;                        // (the fused tile holds no more)
static_assert(kRounds <= kMaxRounds, "10-bit counters");
// words per chunk: three streams of 3 NT R - 1 words (not a multiple of 3)
uint32_t cover_chunk_words(uint64_t words, bool fused)
{
    if (fused) return 3 * (3 * kFusedNT * kFusedRounds - 1);
    const uint64_t round = 9ull * kCoverNT, slots = (uint64_t)kCoverCtas * device_sms();
    const uint64_t r = std::min<uint64_t>(std::max<uint64_t>((words + round * slots - 1) / (round * slots), 1), kRounds);
    return (uint32_t)(3 * (3 * kCoverNT * r - 1));
}

// useful primes of the classes: p[v][i], k[v][i] = its index among the odd primes
struct ClassPrimes {
    uint16_t p[3][kMaxUseful], k[3][kMaxUseful];
};
constexpr ClassPrimes make_class_primes()
{
    ClassPrimes t{};
    int n[3] = {0, 0, 0};
    int k = 0;
    for (uint32_t c = 3; n[0] < kMaxUseful || n[1] < kMaxUseful || n[2] < kMaxUseful; c += 2) {
        bool prime = true;
        for (uint32_t d = 3; d * d <= c; d += 2)
            if (c % d == 0) { prime = false; break; }
        if (!prime) continue;
        for (uint32_t v = 0; v < 3; ++v)
            if (c % 3 != v && n[v] < kMaxUseful) {
                t.p[v][n[v]] = (uint16_t)c;
                t.k[v][n[v]] = (uint16_t)k;
                ++n[v];
            }
        ++k;
    }
    return t;
}
constexpr ClassPrimes kClass = make_class_primes();
__constant__ ClassPrimes kClassDev = make_class_primes();

// step I of class V: the prime's (p - 3)/2, the word offset of its partner bits
// and the residue of the partners
constexpr uint32_t use_e(int V, int I) { return (kClass.p[V][I] - 3u) / 2; }
constexpr int use_c(int V, int I) { return (int)((use_e(V, I) + 31) / 32); }
constexpr int use_rho(int V, int I) { return (V + 3 - kClass.p[V][I] % 3) % 3; }
template <int V, int I>
struct Step {
    static constexpr int c = use_c(V, I), rho = use_rho(V, I);
    static constexpr uint32_t sh = 32u * (uint32_t)use_c(V, I) - use_e(V, I);
};

// window of the steps [I0, I0 + L) of class V in the merged words of residue
// rho: word offsets lo .. lo + n - 1 below the word's own
constexpr int win_lo(int V, int I0, int L, int rho)
{
    int lo = 1 << 20;
    for (int i = I0; i < I0 + L; ++i)
        if (use_rho(V, i) == rho && use_c(V, i) - 1 < lo) lo = use_c(V, i) - 1;
    return lo < 0 || lo == 1 << 20 ? 0 : lo;
}
constexpr int win_n(int V, int I0, int L, int rho)
{
    int hi = -1;
    for (int i = I0; i < I0 + L; ++i)
        if (use_rho(V, i) == rho && use_c(V, i) > hi) hi = use_c(V, i);
    return hi < 0 ? 0 : hi - win_lo(V, I0, L, rho) + 1;
}
template <int V, int I0, int L, int RHO>
struct Win {
    static constexpr int lo = win_lo(V, I0, L, RHO), n = win_n(V, I0, L, RHO);
};

// bits b = phi (mod 3) of a word, phi in 0 .. 2
__device__ __forceinline__ uint32_t phase_mask(uint32_t phi) { return 0x49249249u << phi; }
__device__ __forceinline__ uint32_t mod3(uint32_t x) { return x % 3u; }

// add one block's histogram to the class's bins, from the block's first on.  The lanes' cumulative counts
// are summed over the warp by a transposed butterfly: two counts per register as
// 16-bit fields (a lane's counts are at most 960, a warp's at most 30720), and
// at each of five shuffle stages a lane keeps half of its registers and sends
// the other half to its partner, so that lane l ends with the warp totals of
// the count pair l (L > 32: registers padded to 32), l / 2 (L > 16) or l / 4.
// The bins are the differences of consecutive totals.
template <int L, int KH>
__device__ __forceinline__ void flush_block(const uint32_t (&cum)[KH], uint32_t init_pop, uint32_t* first_bin, int lane)
{
    constexpr int NP = L / 2;                               // count pairs
    constexpr int NR = NP <= 8 ? 8 : NP <= 16 ? 16 : 32;    // registers, a power of two
    constexpr int SH = NR == 8 ? 2 : NR == 16 ? 1 : 0;      // lane >> SH is the lane's pair
    static_assert(L % 2 == 0 && NP <= NR, "block length");
    uint32_t P[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        if (r < NP) {
            const uint32_t lo = (cum[(2 * r) / 3] >> (kCumBits * ((2 * r) % 3))) & kCumMask;
            const uint32_t hi = (cum[(2 * r + 1) / 3] >> (kCumBits * ((2 * r + 1) % 3))) & kCumMask;
            P[r] = lo | (hi << 16);
        } else {
            P[r] = 0;
        }
    }
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const unsigned o = 16u >> st;
        const int m = NR >> (st + 1);                       // registers kept after this stage
        if (m > 0) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int r = 0; r < (m > 0 ? m : 1); ++r) {
                const uint32_t send = up ? P[r] : P[r + m];
                const uint32_t keep = up ? P[r + m] : P[r];
                P[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        } else {
            P[0] += __shfl_xor_sync(0xffffffffu, P[0], o);
        }
    }
    const uint32_t pi = (uint32_t)lane >> SH;               // this lane's pair
    const uint32_t t_lo = P[0] & 0xffffu, t_hi = P[0] >> 16;
    const uint32_t before = __reduce_add_sync(0xffffffffu, init_pop);       // total before the block
    const uint32_t up_hi = __shfl_up_sync(0xffffffffu, t_hi, 1 << SH);
    const uint32_t prev = pi == 0 ? before : up_hi;
    if (pi < (uint32_t)NP && (lane & ((1 << SH) - 1)) == 0) {
        const uint32_t d_lo = t_lo - prev, d_hi = t_hi - t_lo;
        uint32_t* bins = first_bin + 2 * pi;
        if (d_lo) atomicAdd(bins, d_lo);
        if (d_hi) atomicAdd(bins + 1, d_hi);
    }
}

// one step on one word of a later block: R1, R2 = windows of the merged words
// of residue 1 and 2 (R[t] = word w - lo - t)
template <int V, int I, int I0, int N1, int N2, int KH>
__device__ __forceinline__ void later_step(const uint32_t (&R1)[N1], const uint32_t (&R2)[N2], uint32_t& C,
                                           uint32_t (&cum)[KH], const uint32_t (&wt)[3])
{
    constexpr int rho = Step<V, I>::rho, t = Step<V, I>::c - Win<V, I0, kLater, rho>::lo;
    constexpr uint32_t sh = Step<V, I>::sh;
    uint32_t s;
    if constexpr (rho == 1) s = sh == 0 ? R1[t] : __funnelshift_r(R1[t], R1[t > 0 ? t - 1 : 0], sh);
    else s = sh == 0 ? R2[t] : __funnelshift_r(R2[t], R2[t > 0 ? t - 1 : 0], sh);
    C |= s;
    constexpr int j = I - I0;
    cum[j / 3] = __popc(C) * wt[j % 3] + cum[j / 3];
}

template <int V, int I0, int N1, int N2, int KH, int... J>
__device__ __forceinline__ void run_later(std::integer_sequence<int, J...>, const uint32_t (&R1)[N1],
                                          const uint32_t (&R2)[N2], uint32_t& C, uint32_t (&cum)[KH],
                                          const uint32_t (&wt)[3])
{
    (later_step<V, I0 + J, I0, N1, N2, KH>(R1, R2, C, cum, wt), ...);
}

// ---------------------------------------------------------------------------
// block 0 on three consecutive words per lane: one window serves the three
// words, so a step is three funnel shifts and three ORs, then the three
// words' popcounts added into the step's counter through a carry-save adder:
// popc(C0) + popc(C1) + popc(C2) = popc(x) + 2 popc(y) with x the sum bits and
// y the carry bits, two popcounts instead of three for two more logic ops
// (the popcounts bound the step: measured 8.15 against 9.19 ms for the cover
// of 2^34 even n near 5e11, before the classes).
// Window: R[t] = merged word w + 2 - t for the lane's first word w (block 0
// starts at offset 0).
//
// The counts reach the 10-bit fields by integer multiply-adds with the field
// weights 1, 2^10, 2^20 held as runtime values (not constants, which the
// compiler would turn into shifts): the multiply-adds run on the FMA pipe and
// leave the ALU pipe to the shifts and ORs, the popcounts run on the XU pipe.
// ---------------------------------------------------------------------------
template <int T, uint32_t SH, int N>
__device__ __forceinline__ void or3(const uint32_t (&R)[N], uint32_t& C0, uint32_t& C1, uint32_t& C2)
{
    static_assert(T + 2 < N, "window too small");
    if constexpr (SH == 0) {
        C0 |= R[T + 2];
        C1 |= R[T + 1];
        C2 |= R[T];
    } else {
        C0 |= __funnelshift_r(R[T + 2], R[T + 1], SH);
        C1 |= __funnelshift_r(R[T + 1], R[T], SH);
        C2 |= __funnelshift_r(R[T], R[T - 1], SH);
    }
}

template <int V, int I, int N1, int N2, int KH>
__device__ __forceinline__ void step3(const uint32_t (&R1)[N1], const uint32_t (&R2)[N2], uint32_t& C0, uint32_t& C1,
                                      uint32_t& C2, uint32_t (&cum)[KH], const uint32_t (&wt)[3])
{
    constexpr int t = Step<V, I>::c;
    constexpr uint32_t sh = Step<V, I>::sh;
    if constexpr (Step<V, I>::rho == 1) or3<t, sh>(R1, C0, C1, C2);
    else or3<t, sh>(R2, C0, C1, C2);
    const uint32_t w = wt[I % 3];
    const uint32_t x = C0 ^ C1 ^ C2;                        // sum bits
    const uint32_t y = (C0 & C1) | (C2 & (C0 | C1));        // carry bits (majority)
    const uint32_t py = __popc(y);
    cum[I / 3] = __popc(x) * w + cum[I / 3];
    cum[I / 3] = py * w + cum[I / 3];                       // twice: weight 2
    cum[I / 3] = py * w + cum[I / 3];
}

template <int V, int N1, int N2, int KH, int... J>
__device__ __forceinline__ void run_block0(std::integer_sequence<int, J...>, const uint32_t (&R1)[N1],
                                           const uint32_t (&R2)[N2], uint32_t& C0, uint32_t& C1, uint32_t& C2,
                                           uint32_t (&cum)[KH], const uint32_t (&wt)[3])
{
    (step3<V, J, N1, N2, KH>(R1, R2, C0, C1, C2, cum, wt), ...);
}

// a word of the q window: read-only global load, or a shared-memory load when
// the window is a tile the same CTA has just sieved (fused kernel)
template <bool SQ>
__device__ __forceinline__ uint32_t ldq(const uint32_t* p)
{
    if constexpr (SQ) return *p;
    else return __ldg(p);
}

// what the functions below need of the chunk
struct Chunk {
    const uint32_t* Qc;         // window word of the chunk's first coverage word
    const uint32_t* Y1;         // merged words of the q = 1 and = 2 (mod 3) in shared memory:
    const uint32_t* Y2;         // Y[k] holds the partners of p = 3 for the merged n word k
    uint32_t O;                 // words per stream
    uint32_t o3;                // O mod 3 (1 or 2)
    uint32_t na3;               // the chunk's first n, mod 3
    uint32_t n_end;             // n of the chunk
    uint32_t preset;            // bits of word 0: n = 4 and n = 6
    uint64_t w_begin;           // the chunk's first word in the slab
    uint32_t j_cta, seg;
    uint32_t k_first;           // this warp's first merged word (then every 96 NW words on)
    uint32_t* lc;               // this warp's list: coverage, merged word index
    uint16_t* lw;
    uint32_t* shist;            // the CTA's bins [3][kMaxUseful]
};

// the n of the chunk's plain word W that are there to cover
__device__ __forceinline__ uint32_t valid_bits(const Chunk& c, uint32_t W)
{
    const uint32_t j0 = 32 * W;
    uint32_t v = j0 >= c.n_end ? 0u : c.n_end - j0 >= 32 ? 0xffffffffu : (1u << (c.n_end - j0)) - 1u;
    if (W == 0) v &= ~c.preset;
    return v;
}

// phase of the n = v (mod 3) in the chunk's plain word W: n = n_a + 2 (32 W + b)
// = n_a + W + 2 b (mod 3), so b = 2 v + n_a + W
__device__ __forceinline__ uint32_t n_phase(const Chunk& c, uint32_t v, uint32_t W) { return mod3(2 * v + c.na3 + W); }

// coverage of merged word k of class v before the first prime: all but its valid n
__device__ __forceinline__ uint32_t init_c(const Chunk& c, uint32_t v, uint32_t k)
{
    if (k >= c.O) return 0xffffffffu;
    const uint32_t f = n_phase(c, v, k);
    return ~((valid_bits(c, k) & phase_mask(f)) | (valid_bits(c, k + c.O) & phase_mask(mod3(f + c.o3))) |
             (valid_bits(c, k + 2 * c.O) & phase_mask(mod3(f + 2 * c.o3))));
}

// The code of a chunk is kept small: of all that is unrolled, only the steps are
// there once per class and block, behind uniform branches; the lists, the
// counts' flush and the probing are there once (with everything unrolled per
// class, 110 KB of code, the warps waited for instructions 60 % of the time and
// the cover was slower than without the classes).

// steps of block 0 of class v on the lane's words at .. at + 2
template <int L0, int KH, int V>
__device__ __forceinline__ void block0_class(const uint32_t* Y1, const uint32_t* Y2, uint32_t& C0, uint32_t& C1,
                                             uint32_t& C2, uint32_t (&cum)[KH], const uint32_t (&wt)[3])
{
    static_assert(Win<V, 0, L0, 1>::lo == 0 && Win<V, 0, L0, 2>::lo == 0, "block 0 starts at offset 0");
    constexpr int N1 = Win<V, 0, L0, 1>::n + 2, N2 = Win<V, 0, L0, 2>::n + 2;
    uint32_t R1[N1], R2[N2];
#pragma unroll
    for (int t = 0; t < N1; ++t) R1[t] = Y1[2 - t];
#pragma unroll
    for (int t = 0; t < N2; ++t) R2[t] = Y2[2 - t];
    run_block0<V, N1, N2, KH>(std::make_integer_sequence<int, L0>{}, R1, R2, C0, C1, C2, cum, wt);
}

// steps of the later block I0 of class V on one word
template <int V, int I0, int KH>
__device__ __forceinline__ void later_class(const uint32_t* Y1, const uint32_t* Y2, uint32_t& C, uint32_t (&cum)[KH],
                                            const uint32_t (&wt)[3])
{
    constexpr int L = kLater;
    constexpr int n1 = Win<V, I0, L, 1>::n, n2 = Win<V, I0, L, 2>::n, lo1 = Win<V, I0, L, 1>::lo, lo2 = Win<V, I0, L, 2>::lo;
    constexpr int N1 = n1 ? n1 : 1, N2 = n2 ? n2 : 1;
    uint32_t R1[N1], R2[N2];
    R1[0] = R2[0] = 0;
#pragma unroll
    for (int t = 0; t < n1; ++t) R1[t] = Y1[-lo1 - t];
#pragma unroll
    for (int t = 0; t < n2; ++t) R2[t] = Y2[-lo2 - t];
    run_later<V, I0, N1, N2, KH>(std::make_integer_sequence<int, L>{}, R1, R2, C, cum, wt);
}

// later block b (from 1) of a schedule with block 0 of L0 primes
template <int V, int L0, int KH, int B = 1>
__device__ __forceinline__ void later_at(int b, const uint32_t* Y1, const uint32_t* Y2, uint32_t& C,
                                         uint32_t (&cum)[KH], const uint32_t (&wt)[3])
{
    if constexpr (L0 + kLater * B <= kMaxUseful) {
        if (b == B) later_class<V, L0 + kLater * (B - 1), KH>(Y1, Y2, C, cum, wt);
        else later_at<V, L0, KH, B + 1>(b, Y1, Y2, C, cum, wt);
    }
}

__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long key)
{
    const uint32_t khi = (uint32_t)(key >> 32);
    const uint32_t mhi = __reduce_max_sync(0xffffffffu, khi);
    const uint32_t klo = khi == mhi ? (uint32_t)key : 0u;
    const uint32_t mlo = __reduce_max_sync(0xffffffffu, klo);
    return ((unsigned long long)mhi << 32) | mlo;
}

// bit b of merged word k of class v as a chunk-relative n index: the stream st
// the bit came from has st O = b - f (mod 3), f the class's phase in word k
__device__ __forceinline__ uint32_t merged_n(const Chunk& c, uint32_t f, uint32_t k, uint32_t b)
{
    const uint32_t d = mod3(b + 3 - f), st = c.o3 == 1 ? d : mod3(2 * d);
    return 32 * (k + st * c.O) + b;
}

// Probing over a warp's list: the warp takes the open n one at a time, lane t
// probing the prime k + t; the lowest set bit of the ballot is p_min.
template <bool SQ>
__device__ __forceinline__ void probe_warp(const CoverArgs& a, const Chunk& c, uint32_t v, uint32_t n_in,
                                           uint32_t k_first, unsigned long long& best, uint32_t& nsteps)
{
    const int lane = threadIdx.x & 31;
    for (uint32_t e = 0; e < n_in; ++e) {
        const uint32_t wk = c.lw[e];
        const uint32_t f = n_phase(c, v, wk);
        uint32_t mm = ~c.lc[e];
        while (mm) {
            const uint32_t b = __ffs(mm) - 1;
            mm &= mm - 1;
            const uint32_t rel = merged_n(c, f, wk, b);      // CTA-relative n index
            uint32_t k = k_first;
            for (;;) {
                const uint32_t kt = k + (uint32_t)lane;
                uint32_t bit = 0;
                if (kt < a.K) {
                    const uint32_t i = rel + ((a.H - __ldg(a.primes + 1 + kt) - 1) >> 1);
                    bit = (ldq<SQ>(c.Qc + (i >> 5)) >> (i & 31)) & 1u;
                }
                const unsigned hb = __ballot_sync(0xffffffffu, bit);
                if (lane == 0) nsteps += 32;
                if (hb) {
                    const uint32_t kk = k + (__ffs(hb) - 1);
                    if (lane == 0) {
                        atomicAdd(&a.hist[(uint64_t)c.seg * a.hist_stride + kk + 1], 1u);
                        const unsigned long long key =
                            ((unsigned long long)(kk + 2) << 32) | (0xffffffffull - (c.j_cta + rel));
                        if (key > best) best = key;
                    }
                    break;
                }
                k += 32;
                if (k >= a.K) {
                    // open after every prime of this pass
                    if (lane == 0) {
                        const uint64_t jn = 32 * c.w_begin + rel;        // slab-relative n index
                        bool queued = false;
                        if (a.retry) {
                            const unsigned int slot = atomicAdd(a.retry_count, 1u);
                            if (slot < a.retry_cap) {
                                a.retry[slot].w = jn >> 6;
                                a.retry[slot].C = ~(1ull << (jn & 63));
                                queued = true;
                            }
                        }
                        if (!queued) atomicAdd(&a.unresolved[c.seg], 1ull);
                    }
                    break;
                }
            }
        }
    }
}

// The key of the largest p_min, with its smallest n, that the useful primes I0 ..
// I1 - 1 give the n open in merged word k of class v (C: its coverage before them;
// 0: none).  From the merged words in shared memory, every lane a word of its own.
__device__ __forceinline__ unsigned long long track_word(const Chunk& c, uint32_t v, uint32_t k, uint32_t C, uint32_t I0,
                                                         uint32_t I1)
{
    const uint32_t f = n_phase(c, v, k);
    uint32_t last = 0, bits = 0;
    for (uint32_t i = I0; i < I1 && C != 0xffffffffu; ++i) {
        const uint32_t p = kClassDev.p[v][i], d = (p - 3) >> 1, w = (d + 31) >> 5;
        const uint32_t* y = ((v + 3 - p % 3) % 3 == 1 ? c.Y1 : c.Y2) + k - w;
        const uint32_t nw = ((d & 31) ? __funnelshift_r(y[0], y[1], 32 - (d & 31)) : y[0]) & ~C;
        C |= nw;
        if (nw) {
            last = i + 1;
            bits = nw;
        }
    }
    if (!last) return 0;
    // the smallest n of the bits: of each stream's lowest
    uint32_t n = 0xffffffffu;
    for (uint32_t m = bits; m; m &= m - 1) n = min(n, merged_n(c, f, k, __ffs(m) - 1));
    return ((unsigned long long)(kClassDev.k[v][last - 1] + 2) << 32) | (0xffffffffull - (c.j_cta + n));
}

// The largest p_min, with its smallest n, that the block of kLater useful primes
// from I0 on gives the n open in the list (which it covers entirely, so that the
// list is still there as it was before).
__device__ __forceinline__ unsigned long long track_block(const Chunk& c, uint32_t v, uint32_t n_in, uint32_t I0)
{
    unsigned long long best = 0;
    for (uint32_t e = threadIdx.x & 31; e < n_in; e += 32) {
        const unsigned long long key = track_word(c, v, c.lw[e], c.lc[e], I0, I0 + kLater);
        if (key > best) best = key;
    }
    return warp_max_key(best);
}

// Class v of a chunk: block 0 over the warp's merged words, the later blocks
// over its open ones, probing.  best: the largest key of what block 0 left open
// (0: none of that was covered); returns the number of useful primes in the blocks
// run (the last of them bounds the others' p_min).
template <int NW, int L0, bool SQ>
__device__ __forceinline__ uint32_t cover_class(const CoverArgs& a, const Chunk& c, uint32_t v,
                                                unsigned long long& best, uint32_t& nsteps, const uint32_t (&wt)[3])
{
    const int lane = threadIdx.x & 31;
    uint32_t n_open = 0;
    uint32_t* const bins = c.shist + v * kMaxUseful;
    {
        constexpr int KH = (L0 + 2) / 3;
        uint32_t cum[KH];
#pragma unroll
        for (int k = 0; k < KH; ++k) cum[k] = 0;
        uint32_t init_pop = 0;
        for (uint32_t wbase = c.k_first; wbase < c.O; wbase += 96 * NW) {
            const uint32_t wl = wbase + 3 * (uint32_t)lane;           // the lane's first word
            uint32_t C0 = 0, C1 = 0, C2 = 0;
            if (wl + 2 >= c.O || 32 * (wl + 3 + 2 * c.O) > c.n_end || (wl == 0 && c.preset)) {
                C0 = init_c(c, v, wl);
                C1 = init_c(c, v, wl + 1);
                C2 = init_c(c, v, wl + 2);
                init_pop += __popc(C0) + __popc(C1) + __popc(C2);
            }
            const bool active = wl < c.O;
            nsteps += active ? 3 * L0 : 0;
            // (a lane past the stream reads the window of word 0: its C are full)
            const uint32_t at = active ? wl : 0;
            const uint32_t *Y1 = c.Y1 + at, *Y2 = c.Y2 + at;
            if (v == 0) block0_class<L0, KH, 0>(Y1, Y2, C0, C1, C2, cum, wt);
            else if (v == 1) block0_class<L0, KH, 1>(Y1, Y2, C0, C1, C2, cum, wt);
            else block0_class<L0, KH, 2>(Y1, Y2, C0, C1, C2, cum, wt);
            const uint32_t Cw[3] = {C0, C1, C2};
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const bool open = Cw[i] != 0xffffffffu;
                const unsigned m = __ballot_sync(0xffffffffu, open);
                if (open) {
                    const uint32_t slot = n_open + __popc(m & ((1u << lane) - 1u));
                    c.lw[slot] = (uint16_t)(wl + i);
                    c.lc[slot] = Cw[i];
                }
                n_open += __popc(m);
            }
        }
        flush_block<L0, KH>(cum, init_pop, bins, lane);
    }
    __syncwarp();
    // later blocks over the list, in batches of 32 words (one per lane); the
    // words still open move up in it (each batch is read before its outputs land)
    const int n_later = (int)(v == 0 ? a.n_later[0] : v == 1 ? a.n_later[1] : a.n_later[2]);
    int b = 1;
    for (; b <= n_later && n_open > kProbeWords; ++b) {
        constexpr int KH = (kLater + 2) / 3;
        uint32_t cum[KH];
#pragma unroll
        for (int j = 0; j < KH; ++j) cum[j] = 0;
        uint32_t init_pop = 0, n_out = 0;
        for (uint32_t e0 = 0; e0 < n_open; e0 += 32) {
            const uint32_t e = e0 + lane;
            const bool active = e < n_open;
            uint32_t C = 0xffffffffu, k = 0;                // (an inactive lane reads word 0's window)
            if (active) {
                k = c.lw[e];
                C = c.lc[e];
            }
            __syncwarp();
            init_pop += __popc(C);
            nsteps += active ? kLater : 0;
            const uint32_t *Y1 = c.Y1 + k, *Y2 = c.Y2 + k;
            if (v == 0) later_at<0, L0, KH>(b, Y1, Y2, C, cum, wt);
            else if (v == 1) later_at<1, L0, KH>(b, Y1, Y2, C, cum, wt);
            else later_at<2, L0, KH>(b, Y1, Y2, C, cum, wt);
            const bool open = C != 0xffffffffu;
            const unsigned m = __ballot_sync(0xffffffffu, open);
            if (open) {
                const uint32_t slot = n_out + __popc(m & ((1u << lane) - 1u));
                c.lw[slot] = (uint16_t)k;
                c.lc[slot] = C;
            }
            n_out += __popc(m);
        }
        __syncwarp();
        flush_block<kLater, KH>(cum, init_pop, bins + L0 + kLater * (b - 1), lane);
        if (n_out == 0) best = track_block(c, v, n_open, L0 + kLater * (b - 1));
        n_open = n_out;
    }
    const uint32_t used = (uint32_t)(L0 + kLater * (b - 1));
    probe_warp<SQ>(a, c, v, n_open, kClassDev.k[v][used - 1] + 1u, best, nsteps);
    __syncwarp();                                           // the list is the next class's
    return used;
}

// dynamic shared memory of a CTA: the merged words of both residues, then the
// warps' lists
struct CoverSmem {
    uint32_t stream;            // words per stream, at most
    uint32_t halo;              // merged words below a chunk's first
    __host__ __device__ constexpr uint32_t merged() const { return (stream + halo + 2 + 3) & ~3u; }
    __host__ __device__ constexpr uint32_t cap(int NW) const { return (stream + 96 * NW - 1) / (96 * NW) * 96; }
    __host__ __device__ constexpr uint32_t bytes(int NW) const { return 8 * merged() + (uint32_t)NW * cap(NW) * 6; }
};
__host__ __device__ constexpr uint32_t stream_words(uint32_t words)
{
    const uint32_t o = (words + 2) / 3;
    return o % 3 == 0 ? o + 1 : o;
}
// the most dynamic shared memory a CTA is launched with: the longest chunk, the
// longest halo (what the launchers allow, whatever the call's own size)
constexpr uint32_t max_halo()
{
    int c = 0;
    for (int v = 0; v < 3; ++v)
        if (use_c(v, kMaxUseful - 1) > c) c = use_c(v, kMaxUseful - 1);
    return (uint32_t)c;
}
constexpr uint32_t max_cover_bytes(int NT, uint32_t rounds)
{
    return CoverSmem{stream_words(3 * (3 * (uint32_t)NT * rounds - 1)), max_halo()}.bytes(NT / 32);
}

// shared counters of a CTA
struct CoverShared {
    uint32_t hist[3 * kMaxUseful];
    unsigned long long smax;
    uint32_t top;               // 2 + the index of the largest p_min known when these are gone through
    uint32_t any;               // 1: some of these
    uint8_t used[3][kMaxWarps]; // per class and warp (by its words) whose probing covered nothing: cover_class's value
};

// One chunk of coverage words [w_begin, w_end) (32-bit words of the window a.Q,
// 32 even n each) whose first n is n0, all in segment (row) seg, where it has
// index j_cta.  Qc is the window's word w_begin, of which words below q_lim may
// be read.  The classes [v0, v1) of it.  Called by every thread of the CTA.
template <int NT, int L0, bool SQ>
__device__ __forceinline__ void cover_chunk(const CoverArgs& a, const uint32_t* Qc, uint32_t q_lim, uint64_t n0,
                                            uint32_t seg, uint64_t w_begin, uint64_t w_end, uint32_t j_cta,
                                            uint32_t* smem, CoverShared& sh, uint32_t v0 = 0, uint32_t v1 = 3)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const CoverSmem lay{stream_words(a.cta_words), a.halo_words};
    const uint32_t nw_cta = (uint32_t)(w_end > w_begin ? w_end - w_begin : 0);
    const uint32_t wt[3] = {a.cum_wt[0], a.cum_wt[1], a.cum_wt[2]};   // 1, 2^10, 2^20
    uint32_t* const y1 = smem;
    uint32_t* const y2 = smem + lay.merged();
    uint32_t* const lists = smem + 2 * lay.merged();

    Chunk c;
    c.Qc = Qc;
    c.Y1 = y1 + a.halo_words;
    c.Y2 = y2 + a.halo_words;
    c.O = stream_words(nw_cta);
    c.o3 = c.O % 3;
    c.na3 = (uint32_t)(n0 % 3);
    const uint64_t n_left = nw_cta ? a.n_count - 32 * w_begin : 0;     // n from the chunk's first to the window end
    c.n_end = (uint32_t)(n_left < 32ull * nw_cta ? n_left : 32ull * nw_cta);
    c.preset = n0 == 4 ? 3u : n0 == 6 ? 1u : 0u;
    c.w_begin = w_begin;
    c.j_cta = j_cta;
    c.seg = seg;
    c.lc = lists + (uint32_t)warp * lay.cap(NW);
    c.lw = reinterpret_cast<uint16_t*>(lists + NW * lay.cap(NW)) + (uint32_t)warp * lay.cap(NW);
    c.shist = sh.hist;

    __syncthreads();                                        // shared memory free (previous chunk)
    for (uint32_t k = threadIdx.x; k < 3 * kMaxUseful; k += NT) sh.hist[k] = 0;
    if (threadIdx.x == 0) {
        sh.smax = 0;
        sh.any = 0;
    }
    if (threadIdx.x < 3 * kMaxWarps) (&sh.used[0][0])[threadIdx.x] = 0;
    {
        // merged words: the window words of the three streams, from halo words
        // below the first coverage word's partner of p = 3 on; q = Bc + 2 (32 W + b)
        // with Bc = n0 - H + 1, so the bits of residue r are b = 2 r + Bc + W (mod 3)
        const uint32_t base = (((a.H - 4) >> 1) >> 5) - a.halo_words;
        const uint32_t bc3 = (c.na3 + 3u - a.H % 3u + 1u) % 3u;
        const uint32_t total = c.O + a.halo_words + 2;
        for (uint32_t t = threadIdx.x; t < total; t += NT) {
            const uint32_t wa = base + t, wb = wa + c.O, wc = wb + c.O;
            const uint32_t A = wa < q_lim ? ldq<SQ>(Qc + wa) : 0u, B = wb < q_lim ? ldq<SQ>(Qc + wb) : 0u,
                           D = wc < q_lim ? ldq<SQ>(Qc + wc) : 0u;
            const uint32_t f = mod3(2 + bc3 + wa);
            const uint32_t m0 = phase_mask(f), m1 = phase_mask(mod3(f + 1)), m2 = ~(m0 | m1);    // phases f, f + 1, f + 2
            // residue 1 has phase f in A, f + O in B, f + 2 O in D; residue 2 two more
            const uint32_t B1 = c.o3 == 1 ? B : D, D1 = c.o3 == 1 ? D : B;
            y1[t] = (A & m0) | (B1 & m1) | (D1 & m2);
            y2[t] = (A & m2) | (B1 & m0) | (D1 & m1);
        }
    }
    __syncthreads();

    uint32_t nsteps = 0;
    // In a short chunk most warps would have no words, and the others the three classes
    // one after the other: there each class has warps of its own (2^24 n near 1e12 in
    // segments of 2^14: 59 -> 35 us).
    c.k_first = 96 * (uint32_t)warp;
    const uint32_t busy = (c.O + 95) / 96;
    if (v1 - v0 == 3 && 3 * busy <= (uint32_t)NW) {
        const uint32_t own = (uint32_t)warp / busy;
        c.k_first -= 96 * busy * own;
        v0 = own;
        v1 = own < 3 ? own + 1 : own;
    } else if (c.k_first >= c.O) {
        v1 = v0;
    }
#pragma unroll 1
    for (uint32_t v = v0; v < v1; ++v) {
        unsigned long long best = 0;
        const uint32_t used = cover_class<NW, L0, SQ>(a, c, v, best, nsteps, wt);
        best = __shfl_sync(0xffffffffu, best, 0);           // (the probing's lane)
        if (lane == 0) {
            if (best) {
                atomicMax(&sh.smax, best);
            } else {
                sh.used[v][c.k_first / 96] = (uint8_t)used;
                sh.any = 1;
            }
        }
    }
    if (threadIdx.x == 0 && c.preset && v0 == 0) {          // (thread 0 has the first class of a whole chunk)
        // n = 4 = 2 + 2 and n = 6 = 3 + 3
        uint32_t* hrow = a.hist + (uint64_t)seg * a.hist_stride;
        if (n0 == 4) {
            atomicAdd(&hrow[0], 1u);
            atomicMax(&sh.smax, (1ull << 32) | (0xffffffffull - j_cta));
        }
        const uint32_t j6 = n0 == 4 ? 1u : 0u;
        if (j6 < c.n_end) {
            atomicAdd(&hrow[1], 1u);
            atomicMax(&sh.smax, (2ull << 32) | (0xffffffffull - (j_cta + j6)));
        }
    }
    __syncthreads();
    // Warps and classes of which no probed n was covered: the maximum lies in the
    // blocks.  Where it may be the chunk's and the segment's, the whole CTA goes
    // through their merged words once more (10^4 n near 1e15 with the bound 1024:
    // 18 us; 30 by the warp itself, 176 from the window's words in global memory, a
    // load's latency per prime).
    if (sh.any) {
        // (one value for all warps, which share out the words by it)
        if (threadIdx.x == 0)
            sh.top = max((uint32_t)(sh.smax >> 32), (uint32_t)(*(volatile unsigned long long*)&a.maxkey[seg] >> 32));
        __syncthreads();
        const uint32_t top = sh.top;
#pragma unroll 1
        for (uint32_t v = 0; v < 3; ++v) {
            // the class's last prime that covered an n of the chunk
            uint32_t last = 0;
            for (uint32_t i = lane; i < (uint32_t)kMaxUseful; i += 32)
                if (c.shist[v * kMaxUseful + i]) last = i + 1;
            last = __reduce_max_sync(0xffffffffu, last);
            uint32_t n = lane < kMaxWarps ? min(last, (uint32_t)sh.used[v][lane]) : 0u;
            if (n && kClassDev.k[v][n - 1] + 2u < top) n = 0;
            const unsigned redo = __ballot_sync(0xffffffffu, n != 0);
            if (!redo) continue;
            // a third of a flagged warp's 96 words to each warp of the CTA
            const uint32_t thirds = 3 * ((c.O + 96 * NW - 1) / (96 * NW));
            unsigned long long key = 0;
            for (uint32_t u = warp; u < __popc(redo) * thirds; u += NW) {
                const uint32_t slot = __fns(redo, 0, (int)(u / thirds) + 1), r = u % thirds;
                const uint32_t k = 96 * (slot + NW * (r / 3)) + 32 * (r % 3) + lane;
                if (k >= c.O) continue;
                const unsigned long long t = track_word(c, v, k, init_c(c, v, k), 0, last);
                if (t > key) key = t;
            }
            key = warp_max_key(key);
            if (lane == 0 && key) atomicMax(&sh.smax, key);
        }
    }
    __syncthreads();

    if (a.iters) {
        // unrolled word steps plus probes
        unsigned long long t = nsteps;
        for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0 && t) atomicAdd(a.iters, t);
    }
    uint32_t* hrow = a.hist + (uint64_t)seg * a.hist_stride;
    for (uint32_t x = threadIdx.x; x < 3 * kMaxUseful; x += NT)
        if (sh.hist[x]) atomicAdd(&hrow[kClassDev.k[x / kMaxUseful][x % kMaxUseful] + 1], sh.hist[x]);
    if (threadIdx.x == 0 && sh.smax) atomicMax(&a.maxkey[seg], sh.smax);
}

bool cover_prefix_valid(int KA) { return KA >= 48 && KA <= kMaxPrefix && KA % 16 == 0; }

// block-cover fields of the arguments, and the length of block 0 (0: not to be
// run).  The prefix KA counts primes; a class of n not divisible by 3 uses every
// other one, so the blocks hold KA / 2 + 8 useful primes.  Block 0 takes 24 where
// the pass has no more than the 48 primes that hold them, 48 near 1e17 and above
// (KA = 240), 32 otherwise (2^33 n near 5e11: 2.69 ms with 28, 2.64 with 32, 2.67
// with 36, 2.72 with 40; 2^31 near 1e15: 0.89, 0.87, 0.86, 0.85).
// A bound below about 900 cuts the blocks short, each class's on its own: every n that
// they leave open is probed, 32 primes to a warp, whether or not a prime is useful to
// it.  There the n divisible by 3, to which every prime is useful, go through KA of them,
// and block 0 takes 24 where whole blocks after it then reach further in the other
// classes (10^8 n near 1e12 with P = 227, 300, 512 and 700: 2.39, 1.44, 0.20 and 0.08
// ms; 2.68, 1.78, 0.47 and 0.11 with the blocks that all three classes have room for;
// with P = 900 near 1e15 0.090 and 0.113, from 1024 on equal).
constexpr uint32_t kSmallK = 160;
static int cover_schedule(CoverArgs& a, int KA, int NW)
{
    if (!cover_prefix_valid(KA) || (uint32_t)KA > a.K || a.cta_words == 0) return 0;
    if (stream_words(a.cta_words) > kMaxRounds * 96u * (uint32_t)NW) return 0;
    int room[3];                                            // useful primes of the class in the pass
    for (int v = 0; v < 3; ++v) {
        room[v] = 0;
        while (room[v] < kMaxUseful && kClass.k[v][room[v]] < a.K) ++room[v];
    }
    const int least = std::min(room[0], std::min(room[1], room[2]));
    const int want = KA / 2 + 8;
    auto later = [&](int have, int L0, int to) {            // whole blocks after block 0
        return std::max(0, std::min((to - L0 + kLater - 1) / kLater, (have - L0) / kLater));
    };
    int L0 = KA >= 240 && least >= 48 ? 48 : least >= 32 ? 32 : least >= 24 ? 24 : 0;
    if (!L0) return 0;
    const bool small = a.K < kSmallK &&
                       L0 + kLater * later(std::min(room[1], room[2]), L0, want) < want;
    if (small && L0 == 32 &&
        later(room[1], 24, want) + later(room[2], 24, want) > later(room[1], 32, want) + later(room[2], 32, want))
        L0 = 24;
    a.halo_words = 0;
    for (int v = 0; v < 3; ++v) {
        const int n = small ? later(room[v], L0, v == 0 ? KA : want) : later(least, L0, want);
        a.n_later[v] = (uint32_t)n;
        a.halo_words = std::max<uint32_t>(a.halo_words, (uint32_t)use_c(v, L0 + kLater * n - 1));
    }
    if (((a.H - 4) >> 6) < a.halo_words) return 0;
    a.cum_wt[0] = 1; a.cum_wt[1] = 1u << kCumBits; a.cum_wt[2] = 1u << (2 * kCumBits);
    return L0;
}

template <int NT, int L0>
__global__ void __launch_bounds__(NT, kCoverCtas * kCoverNT / NT) k_cover_fast(const CoverArgs a)
{
    extern __shared__ uint32_t smem[];
    __shared__ CoverShared sh;
    // this CTA's words, all in one segment
    const uint64_t wps = 2ull * a.words_per_seg;
    const uint32_t seg = blockIdx.x / a.chunks_per_seg;
    const uint32_t chunk = blockIdx.x % a.chunks_per_seg;
    const uint64_t seg_w0 = (uint64_t)seg * wps;
    const uint64_t w_begin = seg_w0 + (uint64_t)chunk * a.cta_words;
    uint64_t w_end = w_begin + a.cta_words;
    const uint64_t n_words32 = (a.n_count + 31) / 32;
    if (w_end > seg_w0 + wps) w_end = seg_w0 + wps;
    if (w_end > n_words32) w_end = n_words32;
    if (w_begin >= w_end) return;
    const uint64_t q_words = 2 * (a.n_words + a.H / 128 + 2);
    const uint64_t lim = q_words - w_begin;
    cover_chunk<NT, L0, false>(a, reinterpret_cast<const uint32_t*>(a.Q) + w_begin,
                               lim < 0xffffffffull ? (uint32_t)lim : 0xffffffffu, a.A0 + 64 * w_begin, seg, w_begin, w_end,
                               (uint32_t)(32 * (w_begin - seg_w0)), smem, sh, gridDim.y == 3 ? blockIdx.y : 0,
                               gridDim.y == 3 ? blockIdx.y + 1 : 3);
}

// Sieve and cover fused per CTA: the CTA sieves the q bits its chunk of
// coverage words reads into shared memory with the tile sieve and runs the
// block cover on them there; Q never goes through global memory.  The cover
// reads window words from w_begin + off_w (the partner offset of the largest
// prime of the pass, (H - P1 - 1) / 2 bits) to w_end + (H - 4) / 64 + 2, so
// the tile starts at word w_begin + off_w.
template <int NT, int L0>
__global__ void __launch_bounds__(NT, 2) k_seg_cover(const CoverArgs a, const SieveArgs sv, uint32_t off_w)
{
    extern __shared__ uint32_t smem[];                      // [cover | stamp tables | tile]
    __shared__ CoverShared sh;
    constexpr int NW = NT / 32;
    const CoverSmem lay{stream_words(a.cta_words), a.halo_words};
    uint32_t* wt = smem + ((lay.bytes(NW) / 4 + 3) & ~3u);
    uint32_t* tile = wt + ((kWheelWords + 3 + 3) & ~3u);    // 16-byte aligned
    const uint64_t wps = 2ull * a.words_per_seg;
    const uint32_t seg = blockIdx.x / a.chunks_per_seg;
    const uint32_t chunk = blockIdx.x % a.chunks_per_seg;
    const uint64_t seg_w0 = (uint64_t)seg * wps;
    const uint64_t w_begin = seg_w0 + (uint64_t)chunk * a.cta_words;
    uint64_t w_end = w_begin + a.cta_words;
    const uint64_t n_words32 = (a.n_count + 31) / 32;
    if (w_end > seg_w0 + wps) w_end = seg_w0 + wps;
    if (w_end > n_words32) w_end = n_words32;
    if (w_begin >= w_end) return;
    for (uint32_t i = threadIdx.x; i < kWheelWords; i += NT) wt[i] = sv.wheel[i];
    // tile word k is window word w_begin + off_w + k; the cover's Qc[k] is
    // window word w_begin + k and is only read at k >= off_w
    const uint64_t t0 = 32ull * (w_begin + off_w);
    sieve_tile<NT>(sv, t0, wt, tile);
    const uint64_t have = (sv.nbits - t0 + 31) / 32;
    const uint32_t tile_words = have < kFusedTileBits / 32 ? (uint32_t)have : kFusedTileBits / 32;
    cover_chunk<NT, L0, true>(a, tile - off_w, off_w + tile_words, a.A0 + 64 * w_begin, seg, w_begin, w_end,
                              (uint32_t)(32 * (w_begin - seg_w0)), smem, sh);
}

uint32_t seg_cover_offset(uint32_t H, uint32_t P1)
{
    const uint32_t bits = P1 + 1 < H ? (H - P1 - 1) / 2 : 0;
    return bits >= 64 ? bits / 32 - 1 : 0;
}

template <int L0>
static cudaError_t launch_seg_l0(const CoverArgs& a, const SieveArgs& sv, uint32_t off_w, cudaStream_t s)
{
    constexpr int NT = kFusedNT;
    const unsigned grid = a.nseg * a.chunks_per_seg;
    if (grid == 0) return cudaSuccess;
    const CoverSmem lay{stream_words(a.cta_words), a.halo_words};
    constexpr size_t rest = ((kWheelWords + 3 + 3) & ~3u) * 4 + kFusedTileBits / 8;
    const size_t smem = (((size_t)lay.bytes(NT / 32) / 4 + 3) & ~size_t(3)) * 4 + rest;
    auto k = k_seg_cover<NT, L0>;
    cudaError_t e = allow_shared(k, ((max_cover_bytes(NT, kFusedRounds) + 15) & ~size_t(15)) + rest);
    if (e != cudaSuccess) return e;
    k<<<grid, NT, smem, s>>>(a, sv, off_w);
    return cudaGetLastError();
}

cudaError_t launch_seg_cover(const CoverArgs& a0, const SieveArgs& sv, int KA, uint32_t P1, cudaStream_t s)
{
    // the tile must hold the chunk's words and the partner halo read past
    // them, from the offset of the pass's largest prime on
    const uint32_t off_w = seg_cover_offset(a0.H, P1);
    const uint64_t need_words = a0.cta_words + ((a0.H - 4) >> 6) + 3 - off_w;
    if (need_words * 32 > kFusedTileBits || sv.tile_bits != kFusedTileBits || sv.out || sv.popcount)
        return cudaErrorInvalidValue;
    CoverArgs a = a0;
    switch (cover_schedule(a, KA, kFusedNT / 32)) {
    case 24: return launch_seg_l0<24>(a, sv, off_w, s);
    case 32: return launch_seg_l0<32>(a, sv, off_w, s);
    case 48: return launch_seg_l0<48>(a, sv, off_w, s);
    default: return cudaErrorInvalidValue;
    }
}

// persistent: CTAs take (range, chunk) items from the queue until it is empty;
// row r of the histograms, keys and counts is range r
template <int NT, int L0>
__global__ void __launch_bounds__(NT, kCoverCtas * kCoverNT / NT) k_cover_items(const CoverItemsArgs a)
{
    extern __shared__ uint32_t smem[];
    __shared__ CoverShared sh;
    __shared__ uint32_t s_item;
    const uint32_t n_items = *a.n_items;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(a.head, 1u);
        __syncthreads();
        const uint32_t part = s_item, item = part / a.split, v = part - item * a.split;
        __syncthreads();
        if (item >= n_items) break;
        const uint32_t ri = a.item_range[item];
        const BatchRange r = a.ranges[ri];
        CoverArgs c = a.base;
        c.n_count = r.n;
        const uint64_t w_begin = (uint64_t)a.item_chunk[item] * c.cta_words;
        uint64_t w_end = w_begin + c.cta_words;
        const uint64_t nw32 = (r.n + 31) / 32;
        if (w_end > nw32) w_end = nw32;
        const uint64_t lim = r.nbits / 32 - w_begin;
        cover_chunk<NT, L0, false>(c, reinterpret_cast<const uint32_t*>(a.Q + r.q_off) + w_begin,
                                   lim < 0xffffffffull ? (uint32_t)lim : 0xffffffffu, r.lo + 64 * w_begin, ri, w_begin,
                                   w_end, (uint32_t)(32 * w_begin), smem, sh, v, a.split == 3 ? v + 1 : 3);
    }
}

template <int NT, int L0>
static cudaError_t launch_items_nt(const CoverItemsArgs& a, cudaStream_t s)
{
    const size_t smem = CoverSmem{stream_words(a.base.cta_words), a.base.halo_words}.bytes(NT / 32);
    auto k = k_cover_items<NT, L0>;
    cudaError_t e = allow_shared(k, max_cover_bytes(NT, kRounds));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NT, smem)) != cudaSuccess) return e;
    k<<<(unsigned)(device_sms() * (per_sm > 0 ? per_sm : 1)), NT, smem, s>>>(a);
    return cudaGetLastError();
}

template <int L0>
static cudaError_t launch_items_l0(const CoverItemsArgs& a, cudaStream_t s)
{
    return stream_words(a.base.cta_words) <= kShortStream ? launch_items_nt<kShortNT, L0>(a, s)
                                                          : launch_items_nt<kCoverNT, L0>(a, s);
}

cudaError_t launch_cover_items(const CoverItemsArgs& a0, int KA, cudaStream_t s)
{
    CoverItemsArgs a = a0;
    a.split = 3ull * a.n_items_host <= (uint64_t)kCoverCtas * device_sms() ? 3u : 1u;     // (as launch_nt)
    switch (cover_schedule(a.base, KA, kCoverNT / 32)) {
    case 24: return launch_items_l0<24>(a, s);
    case 32: return launch_items_l0<32>(a, s);
    case 48: return launch_items_l0<48>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

int cover_fast_phase_primes(uint32_t K, uint64_t n_hi)
{
    // by magnitude: 144 primes below 1e14, 176 below 1e17, 240 above
    int ka = n_hi < 100000000000000ull ? 144 : n_hi < 100000000000000000ull ? 176 : 240;
    while (ka >= 48 && (uint32_t)ka > K) ka -= 32;
    if (ka < 48 && K >= 48) ka = 48;                        // the shortest schedule
    return ka >= 48 ? ka : 0;
}

template <int NT, int L0>
static cudaError_t launch_nt(const CoverArgs& a, cudaStream_t s)
{
    unsigned grid = a.nseg * a.chunks_per_seg;
    if (grid == 0) return cudaSuccess;
    const size_t smem = CoverSmem{stream_words(a.cta_words), a.halo_words}.bytes(NT / 32);
    auto k = k_cover_fast<NT, L0>;
    cudaError_t e = allow_shared(k, max_cover_bytes(NT, kRounds));
    if (e != cudaSuccess) return e;
    // one segment: only the chunks that hold some n
    if (a.nseg == 1) {
        const uint64_t have = ((a.n_count + 31) / 32 + a.cta_words - 1) / a.cta_words;
        if (have < grid) grid = (unsigned)have;
    }
    // a call of few chunks gives each class a CTA of its own: the chunk's time is a
    // warp's way through the classes' blocks and probings (2^16 n near 1e15: 22 ->
    // 12 us)
    const bool few = 3ull * grid <= (uint64_t)kCoverCtas * device_sms();
    k<<<dim3(grid, few ? 3u : 1u), NT, smem, s>>>(a);
    return cudaGetLastError();
}

template <int L0>
static cudaError_t launch_l0(const CoverArgs& a, cudaStream_t s)
{
    return stream_words(a.cta_words) <= kShortStream ? launch_nt<kShortNT, L0>(a, s) : launch_nt<kCoverNT, L0>(a, s);
}

cudaError_t launch_cover_fast(const CoverArgs& a0, int KA, cudaStream_t s)
{
    CoverArgs a = a0;
    switch (cover_schedule(a, KA, kCoverNT / 32)) {
    case 24: return launch_l0<24>(a, s);
    case 32: return launch_l0<32>(a, s);
    case 48: return launch_l0<48>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace gb
