// gb_verify.cu -- gb_verify_range: exhaustive verification of a range of
// even n (GoldbachGPU, arXiv 2603.02621, Sec. 2.3): the range is cut into
// segments of S even n (the unit of output) and slabs of whole segments (the
// unit of residency); per slab: segment sieve of the q window -> cover
// (p <= P1) -> retry (P1 < p <= P2) -> per-segment reduction; one copy of the
// results to the host at the end.
#include "gb_runtime.cuh"

// the first bytes of ctx->merged: what a call reads back besides its outputs;
// the merged histogram follows
struct RangeHead {
    gb::RangeTotals totals;
    unsigned int overflow;          // retry items that no list could hold
    unsigned int reserved[7];
};
static_assert(sizeof(RangeHead) == 64, "layout");
// histogram entries read back with the head (p_min up to 17863; more are copied apart)
constexpr uint32_t kHeadHist = 2048;

extern "C" {

int gb_verify_range(gb_ctx* ctx, uint64_t lo, uint64_t hi, uint32_t P, gb_range_result* out)
{
    if (!ctx || !out) return fail(GB_EINVAL, "NULL argument");
    NvtxRange call_range("gb_verify_range");
    if ((lo & 1) || (hi & 1) || lo < 4 || hi <= lo) return fail(GB_EINVAL, "range must be even, lo >= 4, hi > lo");
    if (hi > GB_MAX_HI) return fail(GB_EINVAL, "hi beyond 2^63 - 2^26");
    const gb_config& cfg = ctx->cfg;
    const uint32_t P1 = P ? P : cfg.p1;
    if (P1 < 2 || P1 > (1u << 24) || P1 > ctx->L) return fail(GB_EINVAL, "P out of range (2 .. min(2^24, base list))");
    const bool retry = cfg.p2 > P1;
    const uint32_t Pf = retry ? cfg.p2 : P1;
    const uint32_t K1 = (uint32_t)(ctx->pi(P1) - 1);      // odd primes <= P1
    const uint32_t Kf = (uint32_t)(ctx->pi(Pf) - 1);
    // halo: larger than every p of both passes, and H = 4 (mod 64) so that the
    // partner bits of p = 3 start on a 32-bit word boundary (two-phase cover)
    const uint32_t H = 64 * ((Pf + 1 - 4 + 63) / 64) + 4;
    const uint64_t S = cfg.seg_len;
    const uint64_t n_total = (hi - lo) / 2;
    const uint64_t nseg = (n_total + S - 1) / S;
    if (nseg > 0xffffffffull) return fail(GB_EINVAL, "too many segments");
    const uint64_t last_num = hi + 2 * 1024 + H;          // generous bound of the sieve window
    if (isqrt_u64(last_num) > ctx->L) return fail(GB_EINVAL, "hi beyond base_limit^2");
    const uint32_t hist_stride = Kf + 1;
    const uint64_t spb = std::max<uint64_t>(1, cfg.slab_bits / S);   // segments per slab
    GB_CUDA(cudaSetDevice(cfg.device));
    cudaStream_t s = ctx->stream;

    // where each output goes: caller device buffers are written in place,
    // host buffers through device staging and one copy at the end
    const bool want_rows = out->seg_hist && out->seg_hist_stride;
    const uint32_t row_stride = want_rows ? out->seg_hist_stride : 0;
    const uint64_t rows_n = want_rows ? (out->seg_cap ? std::min<uint64_t>(out->seg_cap, nseg) : nseg) : 0;
    const bool rows_dev = want_rows && is_device_ptr(out->seg_hist);
    const bool segs_dev = out->segs && is_device_ptr(out->segs);
    const bool pmin_dev = out->pmin && is_device_ptr(out->pmin);
    const bool hist_dev = out->hist && is_device_ptr(out->hist);
    int rc;
    const size_t merged_bytes = sizeof(RangeHead) + (size_t)hist_stride * 8;
    if ((rc = ctx->summary.ensure(nseg * sizeof(gb::SegSummary))) || (rc = ctx->merged.ensure(merged_bytes)) ||
        (rc = ctx->hstage.ensure(sizeof(RangeHead) + kHeadHist * 8)) ||
        (want_rows && !rows_dev && (rc = ctx->rows.ensure(std::max<uint64_t>(1, nseg * row_stride) * 8))) ||
        (out->segs && !segs_dev && (rc = ctx->records.ensure(nseg * sizeof(gb::SegRecord)))))
        return rc;
    RangeHead* const d_head = ctx->merged.as<RangeHead>();
    unsigned long long* const d_merged = reinterpret_cast<unsigned long long*>(d_head + 1);
    GB_CUDA(cudaMemsetAsync(ctx->merged.p, 0, merged_bytes, s));
    uint64_t* rows_base = want_rows ? (rows_dev ? out->seg_hist : ctx->rows.as<uint64_t>()) : nullptr;

    // per-slab buffers; what starts at zero is one array: segment keys,
    // unresolved counts, the retry list's count, histogram rows
    const uint64_t slab_n = std::min<uint64_t>(spb * S, n_total);
    const uint64_t slab_words = (slab_n + 63) / 64;
    const uint64_t slab_segs = std::min<uint64_t>(spb, nseg);
    const uint64_t q_words = slab_words + H / 128 + 2;
    const uint32_t retry_cap = (uint32_t)std::min<uint64_t>(slab_words, 1u << 21);
    if ((rc = ctx->q.ensure(q_words * 8)) || (rc = ctx->slab.ensure(slab_segs * (16 + (size_t)hist_stride * 4) + 16)) ||
        (retry && (rc = ctx->retry.ensure((size_t)retry_cap * sizeof(gb::RetryItem)))) ||
        (out->pmin && !pmin_dev && (rc = ctx->pmin.ensure(slab_n * 4))))
        return rc;

    // A short range is first sieved and covered with the first pass's halo; the
    // retry pass, whose halo may be many times the range, sieves its window only
    // when the first pass left some n open.  From P1 = 2^13 on that is rare (the
    // largest p_min up to 4e18 is 9781), and a range of 2^22 n or more hardly
    // notices the halo.
    const uint32_t H1 = 64 * ((P1 + 1 - 4 + 63) / 64) + 4;
    const bool lazy = retry && !ctx->fused && nseg <= spb && P1 >= (1u << 13) && n_total < (1u << 22);
    const uint32_t Hc = lazy ? H1 : H;                    // halo of the cover's window

    gb::ReduceArgs rd{};
    gb::RetryArgs ra{};
    for (uint64_t s0 = 0; s0 < nseg; s0 += spb) {
        const uint64_t ns = std::min<uint64_t>(spb, nseg - s0);
        const uint64_t A0 = lo + 2 * s0 * S;
        const uint64_t n_count = std::min<uint64_t>(ns * S, n_total - s0 * S);
        const uint64_t n_words = (n_count + 63) / 64;
        const uint64_t qw = n_words + Hc / 128 + 2;
        const int64_t B = (int64_t)A0 - (int64_t)Hc + 1;

        unsigned long long* const maxkey = ctx->slab.as<unsigned long long>();
        unsigned long long* const unres = maxkey + ns;
        unsigned int* const retry_count = reinterpret_cast<unsigned int*>(unres + ns);
        uint32_t* const hist = retry_count + 4;
        GB_CUDA(cudaMemsetAsync(ctx->slab.p, 0, ns * (16 + (size_t)hist_stride * 4) + 16, s));
        uint32_t* pm = nullptr;
        if (out->pmin) {
            pm = pmin_dev ? out->pmin + (s0 * S) : ctx->pmin.as<uint32_t>();
            GB_CUDA(cudaMemsetAsync(pm, 0, n_count * 4, s));
        }

        gb::CoverArgs ca{};
        ca.Q = ctx->q.as<uint64_t>();
        ca.H = Hc;
        ca.n_count = n_count;
        ca.n_words = n_words;
        ca.words_per_seg = (uint32_t)(S / 64);
        ca.cta_words = gb::cover_generic_words(n_words, S / 64);
        ca.chunks_per_seg = (uint32_t)((S / 64 + ca.cta_words - 1) / ca.cta_words);
        ca.nseg = (uint32_t)ns;
        ca.primes = ctx->base->primes.as<uint32_t>();
        ca.K = K1;
        ca.hist_stride = hist_stride;
        ca.hist = hist;
        ca.maxkey = maxkey;
        ca.unresolved = unres;
        ca.pmin = pm;
        ca.retry = retry ? ctx->retry.as<gb::RetryItem>() : nullptr;
        ca.retry_count = retry ? retry_count : nullptr;
        ca.retry_cap = retry_cap;
        ca.A0 = A0;
        ca.has_n4 = (A0 == 4);
        ca.iters = ctx->work_ptr(1);
        // two-phase kernel unless a p_min array is wanted (the generic kernel
        // writes it) or the pass has too few primes for its first phase
        int KA = (pm || ctx->generic_cover || cfg.cover_prefix == 1) ? 0 : gb::cover_fast_phase_primes(K1, A0 + 2 * n_count);
        if (KA && cfg.cover_prefix > 1 && cfg.cover_prefix <= K1) KA = (int)cfg.cover_prefix;
        if (KA) {
            const uint32_t seg_words = (uint32_t)(S / 32);
            ca.cta_words = std::min<uint32_t>(gb::cover_chunk_words((n_count + 31) / 32, ctx->fused), seg_words);
            ca.chunks_per_seg = (seg_words + ca.cta_words - 1) / ca.cta_words;
        }
        // fused sieve + cover (GB_FUSED=1): block cover, no large primes, the
        // chunk plus its partner halo within one shared-memory tile
        bool fused = false;
        gb::SieveArgs fsv{};
        const uint32_t P1max = ctx->base->h_primes[K1];           // largest prime of the first pass
        if (ctx->fused && KA &&
            ((uint64_t)ca.cta_words + (H - 4) / 64 + 3 - gb::seg_cover_offset(H, P1max)) * 32 <= gb::kFusedTileBits) {
            uint64_t np = 0, nsmall = 0;
            if ((rc = tile_sieve_args(ctx, B, qw * 64, fsv, np, nsmall))) return rc;
            fused = np <= nsmall;
            fsv.tile_bits = gb::kFusedTileBits;
        }
        bool q_in_hbm = false;
        if (!fused) {
            if ((rc = run_sieve(ctx, B, qw * 64, ctx->q.as<uint32_t>(), nullptr))) return rc;
            q_in_hbm = true;
        }
        ctx->prof_begin(kProfCover, n_count);
        if (fused) GB_LAUNCH(gb::launch_seg_cover(ca, fsv, KA, P1max, s));
        else if (KA) GB_LAUNCH(gb::launch_cover_fast(ca, KA, s));
        else GB_LAUNCH(gb::launch_cover(ca, (int)cfg.cta_threads, s));
        ctx->prof_end();

        if (retry && fused) {
            // the retry pass reads Q from global memory: sieve the slab there
            // only if some word was left open
            unsigned int cnt = 0;
            GB_CUDA(ctx->copy(&cnt, retry_count, 4, cudaMemcpyDeviceToHost, s));
            GB_CUDA(cudaStreamSynchronize(s));
            if (cnt) {
                if ((rc = run_sieve(ctx, B, qw * 64, ctx->q.as<uint32_t>(), nullptr))) return rc;
                q_in_hbm = true;
            }
        }
        if (retry) {
            ra.Q = ca.Q;
            ra.H = H;
            ra.words_per_seg = ca.words_per_seg;
            ra.primes = ca.primes;
            ra.K1 = K1;
            ra.K2 = Kf;
            ra.hist_stride = hist_stride;
            ra.hist = ca.hist;
            ra.maxkey = ca.maxkey;
            ra.unresolved = ca.unresolved;
            ra.pmin = pm;
            ra.items = ca.retry;
            ra.count = ca.retry_count;
            ra.cap = retry_cap;
            ra.overflow = &d_head->overflow;
            if (q_in_hbm && !lazy) {
                ctx->prof_begin(kProfRetry, n_count);
                GB_LAUNCH(gb::launch_retry(ra, s));
                ctx->prof_end();
            }
        }

        rd.nseg = (uint32_t)ns;
        rd.hist_stride = hist_stride;
        rd.hist = ca.hist;
        rd.maxkey = ca.maxkey;
        rd.unresolved = ca.unresolved;
        rd.primes = ca.primes;
        rd.summary = ctx->summary.as<gb::SegSummary>() + s0;
        rd.rows = (want_rows && s0 < rows_n) ? rows_base + s0 * row_stride : nullptr;
        rd.row_stride = row_stride;
        rd.nrows = (uint32_t)(want_rows ? std::min<uint64_t>(ns, rows_n > s0 ? rows_n - s0 : 0) : 0);
        rd.merged = d_merged;
        ctx->prof_begin(kProfReduce, ns);
        GB_LAUNCH(gb::launch_reduce(rd, s));
        ctx->prof_end();

        if (out->pmin && !pmin_dev && !lazy)
            GB_CUDA(ctx->copy(out->pmin + s0 * S, pm, n_count * 4, cudaMemcpyDeviceToHost, s));
    }

    gb::FinalizeArgs fa{};
    fa.lo = lo;
    fa.hi = hi;
    fa.S = S;
    fa.nseg = (uint32_t)nseg;
    fa.summary = ctx->summary.as<gb::SegSummary>();
    fa.records = out->segs ? (segs_dev ? reinterpret_cast<gb::SegRecord*>(out->segs) : ctx->records.as<gb::SegRecord>())
                           : nullptr;
    fa.nrecords = (uint32_t)(out->segs ? std::min<uint64_t>(out->seg_cap, nseg) : 0);
    fa.totals = &d_head->totals;
    fa.retry_count = lazy ? ra.count : nullptr;
    // the totals, with the first histogram entries, to pinned memory
    const uint32_t nh = out->hist ? std::min<uint32_t>(out->hist_cap, hist_stride) : 0;
    const uint32_t nh_head = hist_dev ? 0 : std::min<uint32_t>(nh, kHeadHist);
    RangeHead* const head = static_cast<RangeHead*>(ctx->hstage.p);
    auto finish = [&]() -> int {
        ctx->prof_begin(kProfReduce, nseg);
        GB_LAUNCH(gb::launch_finalize(fa, s));
        ctx->prof_end();
        GB_CUDA(ctx->copy(head, d_head, sizeof *head + (size_t)nh_head * 8, cudaMemcpyDeviceToHost, s));
        GB_CUDA(cudaStreamSynchronize(s));
        return GB_OK;
    };
    if ((rc = finish())) return rc;
    if (lazy && head->totals.open) {
        // n left open: the window with the retry pass's halo, the retry pass, and
        // the reductions once more
        const uint64_t qw = (n_total + 63) / 64 + H / 128 + 2;
        if ((rc = run_sieve(ctx, (int64_t)lo - (int64_t)H + 1, qw * 64, ctx->q.as<uint32_t>(), nullptr))) return rc;
        ra.H = H;
        ctx->prof_begin(kProfRetry, n_total);
        GB_LAUNCH(gb::launch_retry(ra, s));
        ctx->prof_end();
        GB_CUDA(cudaMemsetAsync(d_merged, 0, (size_t)hist_stride * 8, s));
        ctx->prof_begin(kProfReduce, nseg);
        GB_LAUNCH(gb::launch_reduce(rd, s));
        ctx->prof_end();
        if ((rc = finish())) return rc;
    }
    if (head->overflow) {
        // the retry list could not hold every word left open: redo in one pass to Pf
        gb_range_result again = *out;
        const uint32_t saved_p2 = ctx->cfg.p2;
        ctx->cfg.p2 = 0;
        rc = gb_verify_range(ctx, lo, hi, Pf, &again);
        ctx->cfg.p2 = saved_p2;
        if (rc && rc != GB_ERANGE) return rc;
        again.p_final = Pf;
        *out = again;
        return rc;
    }
    if (out->pmin && !pmin_dev && lazy)
        GB_CUDA(ctx->copy(out->pmin, ctx->pmin.p, n_total * 4, cudaMemcpyDeviceToHost, s));

    const gb::RangeTotals tot = head->totals;
    // histogram entries from hist_len on are zero (a device buffer is filled in place)
    const uint32_t nh_used = std::min<uint32_t>(nh, tot.hist_len);
    if (hist_dev) {
        GB_CUDA(cudaMemcpyAsync(out->hist, d_merged, (size_t)nh * 8, cudaMemcpyDeviceToDevice, s));
        if (out->hist_cap > nh) GB_CUDA(cudaMemsetAsync(out->hist + nh, 0, (size_t)(out->hist_cap - nh) * 8, s));
    } else if (nh_used) {
        std::memcpy(out->hist, head + 1, (size_t)std::min(nh_used, nh_head) * 8);
        if (nh_used > nh_head)
            GB_CUDA(ctx->copy(out->hist + nh_head, d_merged + nh_head, (size_t)(nh_used - nh_head) * 8,
                              cudaMemcpyDeviceToHost, s));
    }
    const uint64_t nrec = out->segs ? std::min<uint64_t>(out->seg_cap, nseg) : 0;
    if (nrec && !segs_dev)
        GB_CUDA(ctx->copy(out->segs, ctx->records.p, nrec * sizeof(gb::SegRecord), cudaMemcpyDeviceToHost, s));
    if (rows_n && !rows_dev)
        GB_CUDA(ctx->copy(out->seg_hist, ctx->rows.p, rows_n * row_stride * 8, cudaMemcpyDeviceToHost, s));
    if (out->hist && !hist_dev) std::memset(out->hist + nh_used, 0, (size_t)(out->hist_cap - nh_used) * 8);
    GB_CUDA(cudaStreamSynchronize(s));

    out->n_checked = n_total;
    out->n_segments = (uint32_t)nseg;
    out->p_final = Pf;
    out->unresolved = tot.unresolved;
    out->max_pmin = tot.max_pmin;
    out->max_pmin_n = tot.max_pmin_n;
    out->hist_len = tot.hist_len;

    // a segment histogram longer than the caller's row stride was truncated
    bool erange = (out->segs && out->seg_cap < nseg) || (want_rows && rows_n < nseg) ||
                  (out->hist && out->hist_cap < out->hist_len);
    if (want_rows && !erange && row_stride < hist_stride) {
        if (out->segs && !segs_dev) {
            for (uint64_t k = 0; k < nrec && !erange; ++k) erange = out->segs[k].hist_len > row_stride;
        } else {
            erange = tot.hist_len > row_stride;            // the longest row is the range maximum's
        }
    }
    if (erange) return fail(GB_ERANGE, "an output buffer was too small; what fit was written");
    return GB_OK;
}

}  // extern "C"
