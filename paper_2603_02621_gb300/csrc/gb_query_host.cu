// gb_query_host.cu -- gb_query / gb_query_batch (GoldbachGPU, arXiv
// 2603.02621, Sec. 2.4) and gb_partitions (Sec. 4.5): argument checks,
// staging and the launches of the kernels in gb_query.cu and
// gb_partitions.cu.
#include "gb_runtime.cuh"

extern "C" {

int gb_query_batch(gb_ctx* ctx, const uint64_t* n, uint32_t count, uint32_t P, uint32_t* p_min)
{
    if (!ctx || (count && (!n || !p_min))) return fail(GB_EINVAL, "NULL argument");
    if (count == 0) return GB_OK;
    const gb_config& cfg = ctx->cfg;
    const uint32_t Pq = P ? P : std::max(cfg.p1, cfg.p2);
    if (Pq < 3 || Pq > ctx->L) return fail(GB_EINVAL, "P must be in [3, base primes]");
    if (ctx->L < gb::query_filter_max()) return fail(GB_EINVAL, "queries need base primes to 2048");
    GB_CUDA(cudaSetDevice(cfg.device));
    cudaStream_t s = ctx->stream;
    const bool n_dev = is_device_ptr(n), out_dev = is_device_ptr(p_min);
    if (!n_dev)
        for (uint32_t i = 0; i < count; ++i)
            if ((n[i] & 1) || n[i] < 4 || n[i] >= (1ull << 63)) return fail(GB_EINVAL, "n must be even, 4 <= n < 2^63");
    // host arrays go through pinned staging, one transfer each way (a single n
    // as a kernel argument); device ones are used in place, with a count of
    // the invalid n (host n were checked above)
    constexpr uint32_t kStaged = 1u << 16;            // larger batches are copied as they are
    const bool stage = count <= kStaged;
    int rc;
    if ((!n_dev && count > 1 && (rc = ctx->qn.ensure((size_t)count * 8))) ||
        (rc = ctx->qout.ensure((size_t)count * 4 + 16)) ||
        (stage && (rc = ctx->hstage.ensure((size_t)count * 12 + 16))))
        return rc;
    unsigned char* const h_n = static_cast<unsigned char*>(ctx->hstage.p);
    uint32_t* const h_out = reinterpret_cast<uint32_t*>(h_n + (size_t)count * 8);   // out, then the invalid count
    gb::QueryArgs qa{};
    qa.n = n;
    if (!n_dev) {
        qa.n = ctx->qn.as<uint64_t>();
        if (count == 1) {
            qa.n = nullptr;
            qa.n_inline = n[0];
        } else {
            if (stage) std::memcpy(h_n, n, (size_t)count * 8);
            GB_CUDA(ctx->copy(ctx->qn.p, stage ? (const void*)h_n : n, (size_t)count * 8, cudaMemcpyHostToDevice, s));
        }
    }
    uint32_t* const d_out = ctx->qout.as<uint32_t>();
    qa.bad = n_dev ? d_out + count : nullptr;
    if (n_dev) GB_CUDA(cudaMemsetAsync(qa.bad, 0, 4, s));
    qa.count = count;
    qa.primes = ctx->base->primes.as<uint32_t>();
    qa.recip = ctx->base->recip.as<uint64_t>();
    qa.n_filter = (uint32_t)(ctx->pi(gb::query_filter_max()) - 1);
    qa.K = (uint32_t)(ctx->pi(Pq) - 1);
    qa.out = out_dev ? p_min : d_out;
    GB_LAUNCH(gb::launch_query(qa, s));
    unsigned int h_bad = 0;
    unsigned int* const bad_to = stage ? h_out + count : &h_bad;
    if (!out_dev && n_dev && stage) {
        GB_CUDA(ctx->copy(h_out, d_out, (size_t)count * 4 + 4, cudaMemcpyDeviceToHost, s));
    } else {
        if (n_dev) GB_CUDA(ctx->copy(bad_to, qa.bad, 4, cudaMemcpyDeviceToHost, s));
        if (!out_dev)
            GB_CUDA(ctx->copy(stage ? h_out : p_min, d_out, (size_t)count * 4, cudaMemcpyDeviceToHost, s));
    }
    GB_CUDA(cudaStreamSynchronize(s));
    if (!out_dev && stage) std::memcpy(p_min, h_out, (size_t)count * 4);
    if (n_dev && stage) h_bad = *bad_to;
    if (h_bad) return fail(GB_EINVAL, "n must be even, 4 <= n < 2^63 (device input)");
    return GB_OK;
}


}  // extern "C"

namespace {

// A stretch [a, b) of the n of a partition call: the pairs i < 480 O of all its n
// by residues mod 15 (O = 0: none), the rest by the plain kernel
struct Stretch {
    uint64_t a, b, O;
    uint32_t ny() const { return (uint32_t)((O + 95) / 96 * 96); }
    uint32_t nz() const { return (uint32_t)(ny() + 15 * (((b - 4) / 2 - (a - 2) / 2) / 480 + 1) + 17); }
};

// Sums over many words for more than two warps of n go by residues mod 15, a
// sixty-fourth of the way to the next multiple of lo at a time (the i up to
// the first n's half are common to all, the rest is left to the plain
// kernel); a residue's n come in blocks of 32, so fewer than 96 n would
// mostly fill them with none (about 64 is where the two meet).
// A stretch is three launches, some 60 us together where the sums are short: there
// it takes 2^17 n, at most an eighth of the way.  2*10^5 n from 2^20 and from 2^21 on:
// 0.47 and 0.63 ms; 1.43 and 1.28 by sixty-fourths, 1.20 and 2.03 by the plain
// kernel (2*10^6 from 2^20: 6.6, 12.2, 24.9; stretches of 2^16 n 7.4, of 2^19 6.4; from
// 2^24 on the sixty-fourth is as long).
std::vector<Stretch> partition_stretches(uint64_t lo, uint64_t hi)
{
    std::vector<Stretch> out;
    for (uint64_t a = lo; a < hi;) {
        uint64_t b = hi, O = 0;
        if (a < (1u << 20)) b = std::min<uint64_t>(hi, 1u << 20);       // short sums: the plain kernel
        if (a >= (1u << 20) && (hi - a) / 2 >= 96) {
            b = std::min(hi, a + std::max<uint64_t>(a / 64 / 2 * 2, std::min<uint64_t>(a / 8 / 2 * 2, 1u << 18)));
            if (hi - b < 192) b = hi;
            O = gb::part_stream_words((a - 2) / 2 / 2 + 1);
        }
        out.push_back(Stretch{a, b, O});
        a = b;
    }
    return out;
}

}  // namespace

extern "C" {

int gb_partitions(gb_ctx* ctx, uint64_t lo, uint64_t hi, uint32_t* counts)
{
    if (!ctx || (hi > lo && !counts)) return fail(GB_EINVAL, "NULL argument");
    if ((lo & 1) || (hi & 1) || lo < 4 || hi < lo) return fail(GB_EINVAL, "range must be even, lo >= 4, hi >= lo");
    if (hi > (1ull << 34)) return fail(GB_EINVAL, "partition counts need hi <= 2^34");
    const uint64_t count = (hi - lo) / 2;
    if (count == 0) return GB_OK;
    if (count > (1ull << 28)) return fail(GB_EINVAL, "at most 2^28 even n per call");
    GB_CUDA(cudaSetDevice(ctx->cfg.device));
    cudaStream_t s = ctx->stream;
    // P covers the odd numbers 1 .. the largest m = (hi - 4) / 2 index
    const uint64_t mmax = (hi - 4) / 2;
    const uint64_t words = ((mmax + 1 + 63) / 64) * 2;                  // whole 64-bit words
    const bool out_dev = is_device_ptr(counts);
    int rc;
    if ((rc = ctx->part_p.ensure(words * 4)) || (rc = ctx->part_rev.ensure((words + 1) * 4)) ||
        (!out_dev && (rc = ctx->part_out.ensure(count * 4))))
        return rc;
    // the residues' merged words, sized once for the stretch that needs most; without
    // memory for them the plain kernel does the whole call
    std::vector<Stretch> stretches = partition_stretches(lo, hi);
    uint64_t ny = 0, nz = 0;
    for (const Stretch& t : stretches)
        if (t.O) {
            ny = std::max<uint64_t>(ny, t.ny());
            nz = std::max<uint64_t>(nz, t.nz());
        }
    if (ctx->part_y.ensure(32 * ny) || ctx->part_z.ensure(32 * nz)) {
        ctx->part_y.release();
        ctx->part_z.release();
        stretches.assign(1, Stretch{lo, hi, 0});
    }
    if ((rc = run_sieve(ctx, 1, words * 32, ctx->part_p.as<uint32_t>(), nullptr))) return rc;
    GB_LAUNCH(gb::launch_reverse_bits(ctx->part_p.as<uint32_t>(), ctx->part_rev.as<uint32_t>(), words, s));
    uint32_t* d_out = out_dev ? counts : ctx->part_out.as<uint32_t>();
    GB_CUDA(cudaMemsetAsync(d_out, 0, count * 4, s));
    gb::PartitionArgs pa{};
    pa.P = ctx->part_p.as<uint32_t>();
    pa.rev = ctx->part_rev.as<uint32_t>();
    pa.words = words;
    pa.run_words = 4096;
    for (const Stretch& t : stretches) {
        if (t.O) {
            gb::PartCorrArgs ca{};
            ca.P = pa.P;
            ca.m_min = (t.a - 2) / 2;
            ca.m_max = (t.b - 4) / 2;
            ca.O = (uint32_t)t.O;
            ca.ny = t.ny();
            ca.nz = t.nz();
            ca.run_words = 96 * 16;
            ca.y = ctx->part_y.as<uint32_t>();
            ca.z = ctx->part_z.as<uint32_t>();
            ca.counts = d_out + (t.a - lo) / 2;
            GB_LAUNCH(gb::launch_part_corr(ca, s));
            ctx->kernels += 1;                                          // (two kernels)
        }
        pa.lo = t.a;
        pa.count = (t.b - t.a) / 2;
        pa.n_blocks = (pa.count + 31) / 32;
        pa.counts = d_out + (t.a - lo) / 2;
        pa.w_first = 15 * t.O;
        const uint64_t need = ((t.b - 4) / 2) / 2 / 32 + 1 - pa.w_first;    // words of the largest n
        pa.runs = std::max<uint64_t>(1, (need + pa.run_words - 1) / pa.run_words);
        GB_LAUNCH(gb::launch_partitions(pa, s));
    }
    if (!out_dev) GB_CUDA(ctx->copy(counts, d_out, count * 4, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return GB_OK;
}


int gb_query(gb_ctx* ctx, uint64_t n, uint32_t* p_min)
{
    if (!ctx || !p_min) return fail(GB_EINVAL, "NULL argument");
    return gb_query_batch(ctx, &n, 1, 0, p_min);
}

}  // extern "C"
