// gb_query.cu -- single-n queries: the minimal Goldbach prime p_min(n) of an
// arbitrary even n < 2^63 (GoldbachGPU, arXiv 2603.02621, Sec. 2.4: the
// single-number check, here returning the minimal p and run on the GPU).
//
// One warp per query.  Candidates p are the odd primes in ascending order, in
// windows of 2 * kQueryBits consecutive integers.  For each window the warp
// first sieves the partners q = n - p in shared memory by the filter primes
// f <= kFilterMax (bit t <-> p = pl + 2t is cleared when f | q and q != f);
// the candidates that survive are gathered, 32 at a time, one per lane, and
// each lane takes the strong probable-prime test of its q to base 2.  The
// smallest p that passes is then settled by the whole warp: lane i tests its q
// to the i-th of the bases 3, 5, ..., 37 (with 2 the first 12 primes: no
// composite below 3.3e24 passes them all; Sorenson and Webster, Math. Comp.
// 2017).  The windows stop at the first hit or at p > P.
//
// Bound: a query alone is a chain of two modular powers, base 2 and then the
// eleven others side by side (before: twelve in sequence, in one thread); a
// batch is bound by issue slots, of which the two powers take most.  On a
// GB300, n uniform below 4e18, the calls timed from Python, both kernels in turn on
// one box: one query 197 to 274 us (with the n) -> 53 to 56, a batch of 4096 from
// host memory 1786 -> 135 us (one CTA of 128 threads per query, every survivor
// tested to all twelve bases by its own thread, before).
#include "gb_internal.cuh"

namespace gb {

namespace {

// window: 2048 consecutive integers of p.  At n near 4e18 it holds 308
// candidates, of which about 45 survive and 14 have a prime partner; the first
// 32 survivors miss all of them once in 10^5 queries.
constexpr uint32_t kQueryBits = 1024;
constexpr uint32_t kFilterMax = 2048;      // filter primes f <= 2048 (q with no factor <= 2048 and q < 2048^2 is prime)
constexpr int kQueryThreads = 128;         // four queries per CTA

// Montgomery multiplication modulo an odd N < 2^63 (Montgomery, Math. Comp.
// 1985): for a, b < N returns a b R^-1 mod N with R = 2^64; ninv = -N^-1 mod
// 2^64.  a b + m N is divisible by R with m = (a b mod R) ninv mod R; its low
// word a b + m N (mod R) is 0, so the carry out of the low word is (lo != 0).
__device__ __forceinline__ uint64_t mont_mul(uint64_t a, uint64_t b, uint64_t N, uint64_t ninv)
{
    const uint64_t lo = a * b, hi = __umul64hi(a, b);
    const uint64_t m = lo * ninv;
    const uint64_t t = hi + __umul64hi(m, N) + (lo != 0 ? 1ull : 0ull);   // < 2N < 2^64
    return t >= N ? t - N : t;
}

// Montgomery constants of an odd q, 2048^2 < q < 2^63
struct Mont {
    uint64_t q, ninv, one;                            // one = 2^64 mod q
    __device__ __forceinline__ explicit Mont(uint64_t q_) : q(q_)
    {
        // -q^-1 mod 2^64 by Newton's iteration x <- x (2 - q x): q is its own
        // inverse mod 8 (3 bits), each step doubles the correct bits
        uint64_t x = q;
#pragma unroll
        for (int i = 0; i < 5; ++i) x *= 2 - q * x;
        ninv = 0 - x;
        one = (0 - q) % q;
    }
    __device__ __forceinline__ uint64_t add(uint64_t a, uint64_t b) const
    {
        const uint64_t t = a + b;                     // < 2q < 2^64
        return t >= q ? t - q : t;
    }
    __device__ __forceinline__ uint64_t mul(uint64_t a, uint64_t b) const { return mont_mul(a, b, q, ninv); }
};

// strong probable-prime test of q to the small base b (2 <= b < 64)
template <bool TWO>
__device__ __forceinline__ bool strong_test(const Mont& m, uint32_t b)
{
    uint64_t a = m.add(m.one, m.one);                 // Montgomery form of 2
    if constexpr (!TWO) {
        // b times one, by doubling and adding from b's top bit down
        a = 0;
#pragma unroll
        for (int i = 5; i >= 0; --i) {
            a = m.add(a, a);
            if ((b >> i) & 1) a = m.add(a, m.one);
        }
    }
    const uint64_t minus_one = m.q - m.one;
    const int s = __ffsll((long long)(m.q - 1)) - 1;
    const uint64_t d = (m.q - 1) >> s;
    // a^d by left-to-right binary exponentiation from d's top bit (times 2 is
    // an addition)
    uint64_t y = a;
    for (int bit = 62 - __clzll((long long)d); bit >= 0; --bit) {
        y = m.mul(y, y);
        if ((d >> bit) & 1) y = TWO ? m.add(y, y) : m.mul(y, a);
    }
    bool pass = y == m.one || y == minus_one;
    for (int i = 1; i < s && !pass; ++i) {
        y = m.mul(y, y);
        pass = y == minus_one;
    }
    return pass;
}

}  // namespace

__global__ void __launch_bounds__(kQueryThreads) k_query(const QueryArgs a)
{
    constexpr uint32_t kAll = 0xffffffffu;
    __shared__ uint32_t s_win[kQueryThreads / 32][kQueryBits / 32];
    __shared__ uint32_t s_cand[kQueryThreads / 32][64];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* win = s_win[warp];
    uint32_t* cand = s_cand[warp];
    const uint32_t warps = gridDim.x * (blockDim.x / 32);
    for (uint32_t qi = blockIdx.x * (blockDim.x / 32) + warp; qi < a.count; qi += warps) {
        const uint64_t n = a.n ? a.n[qi] : a.n_inline;
        if ((n & 1) || n < 4 || n >= (1ull << 63)) {           // not a valid query: no work, flagged
            if (lane == 0) {
                a.out[qi] = 0;
                if (a.bad) atomicAdd(a.bad, 1u);
            }
            continue;
        }
        uint32_t best = n == 4 ? 2u : 0u;                       // 4 = 2 + 2, the only even prime partner
        uint32_t k = 1;                                         // next candidate: primes[k]
        uint64_t pl = 3;                                        // window's first p
        while (!best && k <= a.K && pl + 3 <= n) {
            const uint64_t ph = pl + 2 * kQueryBits;
            // pre-sieve of the partners: bit t <-> p = pl + 2t, q = n - pl - 2t
            for (uint32_t w = lane; w < kQueryBits / 32; w += 32) win[w] = kAll;
            __syncwarp();
            const uint64_t top = n - pl;                        // q of bit 0 (pl <= n - 3)
            for (uint32_t j0 = 1; j0 <= a.n_filter; j0 += 32) {
                // 32 filter primes' first bits, a lane each: 2t = top (mod f)
                const uint32_t j = j0 + lane;
                uint32_t f = 0, t = kQueryBits;
                if (j <= a.n_filter) {
                    f = a.primes[j];
                    const uint32_t r = barrett_mod(top, f, a.recip[j]);
                    t = (r & 1u) ? (r + f) >> 1 : r >> 1;
                }
                if (j0 == 1) {
                    // the smallest primes' many strikes are shared by the warp
                    for (int src = 0; src < 32; ++src) {
                        const uint32_t fs = __shfl_sync(kAll, f, src), ts = __shfl_sync(kAll, t, src);
                        if (fs == 0) break;
                        for (uint32_t i = ts + lane * fs; i < kQueryBits; i += 32 * fs)
                            if (top - 2ull * i != fs) atomicAnd(&win[i >> 5], ~(1u << (i & 31)));
                    }
                } else {
                    for (; t < kQueryBits; t += f)
                        if (top - 2ull * t != f) atomicAnd(&win[t >> 5], ~(1u << (t & 31)));
                }
            }
            __syncwarp();
            // candidates of this window in ascending order: the survivors, 32 at a
            // time, one per lane
            uint32_t have = 0;
            for (bool more = true; more && !best;) {
                while (have < 32) {
                    const uint32_t kk = k + lane;
                    const uint32_t p = kk <= a.K ? a.primes[kk] : kAll;
                    const bool in = p < ph;
                    bool live = false;
                    if (in && (uint64_t)p + 3 <= n) {
                        const uint32_t t = (uint32_t)((p - pl) >> 1);
                        live = (win[t >> 5] >> (t & 31)) & 1u;
                    }
                    const unsigned m_in = __ballot_sync(kAll, in), m_live = __ballot_sync(kAll, live);
                    if (live) cand[have + __popc(m_live & ((1u << lane) - 1u))] = p;
                    have += __popc(m_live);                     // < 32 + 32
                    k += __popc(m_in);
                    if (m_in != kAll) {                         // the window's last candidates
                        more = false;
                        break;
                    }
                }
                __syncwarp();
                const uint32_t mine = lane < have ? cand[lane] : 0u;
                const uint32_t next = 32 + lane < have ? cand[32 + lane] : 0u;
                // q below 2048^2 without a factor up to 2048 is prime; larger ones
                // are tested to base 2
                const uint64_t q = n - mine;
                const bool small = q < (uint64_t)kFilterMax * kFilterMax;
                bool pass = mine && small;
                if (mine && !small) pass = strong_test<true>(Mont(q), 2);
                unsigned m_pass = __ballot_sync(kAll, pass);
                const unsigned m_small = __ballot_sync(kAll, pass && small);
                while (m_pass) {
                    // the smallest p that passed: the bases 3 .. 37, a lane each
                    const int src = __ffs(m_pass) - 1;
                    const uint32_t p = __shfl_sync(kAll, mine, src);
                    bool ok = true;
                    if (!((m_small >> src) & 1u)) {
                        // bases 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37 = primes[1 .. 11]
                        if (lane < 11) ok = strong_test<false>(Mont(n - p), a.primes[1 + lane]);
                    }
                    if (__all_sync(kAll, ok)) {
                        best = p;
                        break;
                    }
                    m_pass &= m_pass - 1;
                }
                have = have > 32 ? have - 32 : 0;
                __syncwarp();
                if (lane < have) cand[lane] = next;
                __syncwarp();
                if (have) more = true;                          // a remainder to test
                else if (!more) break;
            }
            pl = ph;
        }
        if (lane == 0) a.out[qi] = best;
        __syncwarp();
    }
}

cudaError_t launch_query(const QueryArgs& a, cudaStream_t s)
{
    if (a.count == 0) return cudaSuccess;
    if ((!a.n && a.count != 1) || !a.primes || !a.recip || !a.out) return cudaErrorInvalidValue;
    // a warp per query; fewer queries than SMs x 4 spread out, one warp to a CTA
    const uint32_t sms = device_sms();
    const uint32_t threads = a.count <= 4 * sms ? 32 : kQueryThreads;
    const uint32_t need = (a.count + threads / 32 - 1) / (threads / 32), cap = sms * 12u;
    k_query<<<need < cap ? need : cap, threads, 0, s>>>(a);
    return cudaGetLastError();
}

uint32_t query_filter_max() { return kFilterMax; }

}  // namespace gb
