// front.cu -- first pass of the search (Section IV): one thread per query.
//
// Most queries of a batch are decided by their k-mer bracket and one or two
// probes, so the first pass runs them straight through, one query per thread
// and no shared state:
//   * in input order the query's first 128 bases come from the packed batch
//     (five words of a 38-byte-per-100-bases array that the packing kernel
//     has just written) and, when the packing found a non-base byte in the
//     batch, its validity from the packing's bitmap; in k-mer order its record
//     in the list (bucket.cu) holds its first 192 bases, already checked;
//   * for m >= k one aligned 64-byte read of the k-mer entry of its first k
//     bases x gives the bracket (lo - 1, hi) of the suffixes that sort
//     between x and x + 1 and the suffix at the bracket's first pivot (its
//     position and first 192 bases), so the bracket and the first probe cost
//     one access;
//   * for m < k two entries' counts are the whole answer;
//   * further probes of the lockstep lower/upper bound, one 32-byte suffix
//     record each, as in the persistent kernel, up to `front_probes` probes
//     in all.
// A query still undecided after that (a bracket wider than the probes could
// resolve, an index without a k-mer table) is
// appended to a worklist -- a 64-byte record holding a bracket of both
// bounds, its length, index, reference, first base in the packed batch and
// first 160 bases -- which the persistent kernel of search.cu then finishes.
#include "first_pass.cuh"

namespace sa {

namespace {

constexpr int kFrontThreads = 256;

// The list slot of each lane's record j = base + lane of the k-mer-ordered
// list: region by region (in the largest bucket b whose regions before it hold
// at most j records), then the overflow region.  prefix: the exclusive sums of
// the regions' fills (kNumBuckets + 2 entries, the last their total); start:
// each region's first slot.  The warp finds base's bucket together (32 of the
// sums, then the 9 that follow the last that is small enough: two reads of
// shared memory against the eight a binary search makes one after the other),
// and the few lanes past its end step on from there.
__device__ __forceinline__ uint32_t list_slot(const uint32_t *prefix, const uint32_t *start, uint32_t ov_start,
                                              uint32_t base) {
    static_assert(kNumBuckets == 256, "the sums are looked through 9 at a time, 32 * 9 >= kNumBuckets + 1");
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t in_regions = prefix[kNumBuckets + 1], j = base + lane;
    const uint32_t coarse = 9u * lane;
    const unsigned below = __ballot_sync(0xFFFFFFFFu, coarse <= kNumBuckets && prefix[min(coarse, kNumBuckets)] <= base);
    const uint32_t group = 9u * (31u - __clz(below));  // (prefix[0] = 0: lane 0 votes)
    const uint32_t fine = group + lane;
    const unsigned in_group =
        __ballot_sync(0xFFFFFFFFu, lane < 9u && fine <= kNumBuckets && prefix[min(fine, kNumBuckets)] <= base);
    uint32_t b = group + 31u - __clz(in_group);
    if (j >= in_regions) return ov_start + (j - in_regions);
    while (prefix[b + 1] <= j) b++;
    return start[b] + (j - prefix[b]);
}

// kFromList: the queries come from the k-mer-ordered list of bucket.cu (one
// 64-byte record each: length, index, reference, first base in the packed
// batch and first 192 bases, already checked) instead of the batch's offsets.
// kOneProbe: the entry's pivot is the only probe (input order's default), in
// kernels of their own without the loop's registers (1 % of a call).
template <bool kSingle, bool kFromList, Bases kBases, bool kOneProbe = false>
__global__ void __launch_bounds__(kFrontThreads, 4) front_kernel(const __grid_constant__ SearchLaunch a) {
    __shared__ FrontDesc sdesc[SA_MAX_REFS];
    __shared__ uint4 s_stage[kFrontThreads / 32][32][4];  // worklist records staged per warp
    __shared__ uint32_t s_lprefix[kNumBuckets + 2];        // the list's numbering (list input)
    __shared__ uint32_t s_lstart[kNumBuckets + 1];
    constexpr bool kStrands = kBases != Bases::Packed;
    for (unsigned r = threadIdx.x; r < a.n_refs; r += blockDim.x) {
        sdesc[r] = front_desc(a.refs.r[r]);
    }
    if (kFromList) {
        for (unsigned i = threadIdx.x; i < kNumBuckets + 2; i += blockDim.x) s_lprefix[i] = a.bplan[kPlanPrefix + i];
        for (unsigned i = threadIdx.x; i <= kNumBuckets; i += blockDim.x) s_lstart[i] = a.bplan[kPlanStart + i];
    }
    const uint32_t ov_start = kFromList ? a.bplan[kPlanOvStart] : 0u;
    __syncthreads();

    const unsigned lane = threadIdx.x & 31u;
    const unsigned wib = threadIdx.x >> 5;
    const unsigned lanemask_lt = (1u << lane) - 1u;
    uint32_t staged = 0;  // warp-uniform: records in s_stage[wib]
    // Moves the warp's staged records to the worklist (one atomic).
    auto flush = [&](uint32_t cnt) {
        if (cnt == 0u) return;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(a.wl_count, cnt);
        at = __shfl_sync(0xFFFFFFFFu, at, 0);
        if (lane < cnt) {
            uint4 *dst = a.wrec + 4 * (size_t)(at + lane);
#pragma unroll
            for (int j = 0; j < 4; j++) dst[j] = s_stage[wib][lane][j];
        }
        __syncwarp();
    };
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t warp_first = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
    const uint64_t *__restrict__ tq = a.tq;
    bool any_bad = false, any_bad_ref = false;

    const uint64_t n_items = kFromList ? (uint64_t)*a.wl_in_count : a.n_q;
    // a batch without a non-base byte needs no per-query validity check
    const bool dirty = !kFromList && *a.batch_dirty != 0;
    // Offsets and reference of this lane's next query, read one query ahead.
    uint64_t nqa = 0, nqe = 0;
    uint32_t nr = 0;
    if (!kFromList && warp_first + lane < a.n_q) {
        nqa = __ldg(a.q_off + warp_first + lane);
        nqe = __ldg(a.q_off + warp_first + lane + 1);
        if (!kSingle) nr = __ldg(a.q_ref + warp_first + lane);
    }

    for (uint64_t base = warp_first; base < n_items; base += stride) {
        const bool live = base + lane < n_items;
        uint64_t q, qa;
        uint32_t r, m;
        bool ok, entry = true;
        uint64_t w[4];
        uint32_t lslot = 0;  // the record's slot in the list (list input)
        if (kFromList) {
            uint4 c0, c1, c2, c3;
            const uint32_t slot = list_slot(s_lprefix, s_lstart, ov_start, (uint32_t)base);
            if (live) lslot = slot;
            const uint4 *src = a.wrec_in + 4 * (size_t)lslot;
            ldg32_if(live, src, &c0, &c1);
            ldg32_if(live, src + 2, &c2, &c3);
            m = c0.x;
            q = c0.y;
            qa = place_of(c0.z, c0.w);
            r = ref_of(c0.w);
            entry = (c0.w & kListNeedsEntry) != 0u;
            w[0] = ((uint64_t)c1.y << 32) | c1.x;
            w[1] = ((uint64_t)c1.w << 32) | c1.z;
            w[2] = ((uint64_t)c2.y << 32) | c2.x;
            w[3] = ((uint64_t)c2.w << 32) | c2.z;
            ok = live;
        } else {
            q = base + lane;
            qa = nqa - a.first;
            const uint64_t qe = nqe - a.first;
            r = nr;
            if (base + stride + lane < a.n_q) {
                nqa = __ldg(a.q_off + base + stride + lane);
                nqe = __ldg(a.q_off + base + stride + lane + 1);
                if (!kSingle) nr = __ldg(a.q_ref + base + stride + lane);
            }
            const bool rc = kStrands && (a.revcomp || (a.strand_bits && (r & kStrandBit)));
            if (kStrands && a.strand_bits) r &= ~kStrandBit;
            const bool range_ok = live && qa <= qe && qe <= a.total && qe - qa < (1ull << 31);
            if (live && !range_ok) any_bad = true;
            ok = range_ok && r < a.n_refs;
            if (range_ok && r >= a.n_refs) any_bad_ref = true;
            m = ok ? (uint32_t)(qe - qa) : 0u;
            if (ok && m > 0 && dirty && !query_valid(a.tvb, a.tv, qa, m)) {
                ok = false;
                any_bad = true;
            }
            if (range_ok) qa = query_place(qa, qe, rc);
            query_windows<4, kStrands>(tq, ok ? qa : 0, 0, w);  // first 128 bases
        }

        FrontDesc d = sdesc[0];
        if (!kSingle && ok) d = sdesc[r];
        // Bracket and first pivot: the k-mer entry for m >= k, else (no k-mer
        // table, or a query it answers by itself) the whole array.
        const uint32_t kk = d.kmer_k;
        const bool look = ok && entry && m > 0 && d.krt != nullptr && m >= kk;
        const uint64_t x = look ? (w[0] >> (64u - 2u * kk)) : 0ull;
        uint4 h, e01, e23, e45;
        ldg64_pairs_if(look, d.krt + 4 * x, &h, &e01, &e23, &e45);
        Bounds bd;
        bd.start(look ? h.x - 1u : 0xFFFFFFFFu, look ? h.y : d.n);  // 0xFFFFFFFF stands for -1

        // A query's result waits in lo and hi for the end of the iteration, so
        // that the warp stores its lanes' results once.  (With that, one path
        // per compare and the list's slots found by the whole warp: 3.1 Gbp,
        // 4*10^7 x 150 bases 8044 -> 7683 us a call, 430 Mbp 1647 -> 1577 us.
        // Prefetching the next iteration's records into L2 cost 1.5 %.)
        bool done = !live || !ok || m == 0 || (look && bd.R - bd.L <= 1u);
        uint64_t lo = bd.R, hi = bd.R;  // a bracket without suffixes
        if (!ok) lo = hi = ~0ull;
        if (ok && m == 0) {
            lo = 0;
            hi = d.n;
        }
        if (ok && m > 0 && d.krt != nullptr && m < kk) {
            uint32_t l, u;
            brief_interval(d, w[0] >> (64u - 2u * m), m, &l, &u);
            lo = l;
            hi = u;
            done = true;
        }

        bool go = !done && look;
        // in list order, bases 128-191 are the record's last 16 bytes (read
        // again when a compare gets there: an L1 or L2 hit)
        const auto src = window_source<kBases>(a, qa, m);
        const RecordWindows<decltype(src)> qw{
            src, w[3], kFromList ? reinterpret_cast<const uint64_t *>(a.wrec_in + 4 * (size_t)lslot + 3) : nullptr,
            kFromList ? 2u : 0u};
        // One compare's outcome c at pivot M with common prefix l (lp, ln: the
        // pivot's own common prefixes with its neighbours).
        auto step = [&](int c, uint32_t M, uint32_t l, uint32_t lp, uint32_t ln) {
            if (bd.step(c, M, l, m, lp, ln)) {
                lo = bd.first();
                hi = bd.R;
                done = true;
                go = false;
            }
        };
        if (go) {  // the first probe: the entry's pivot
            const uint64_t e[6] = {((uint64_t)e01.y << 32) | e01.x, ((uint64_t)e01.w << 32) | e01.z,
                                   ((uint64_t)e23.y << 32) | e23.x, ((uint64_t)e23.w << 32) | e23.z,
                                   ((uint64_t)e45.y << 32) | e45.x, ((uint64_t)e45.w << 32) | e45.z};
            uint32_t l;
            const int c = cmp_entry(w, m, e, h.z, h.w & 0xFFu, d.n, d.text, qw, &l);
            step(c, bd.pivot(), l, (h.w >> 8) & 0xFFu, (h.w >> 16) & 0xFFu);
        }
        // Further probes, one suffix record each; queries without a k-mer
        // bracket go straight to the worklist (the persistent kernel descends
        // the shared-memory key table first).
        // A compare that ties on all a record holds goes on in the text.  In
        // k-mer order (several probes) it waits for the end of the probes, so
        // that the warp reads the text once for all its lanes that do, not once
        // per probe: 3.1 Gbp, 4*10^7 x 150 bases 2.82 -> 2.71 ms.
        bool pending = false;
        uint32_t pend_pos = 0, pend_lcps = 0;
        for (uint32_t p = 1; !kOneProbe && p < a.front_probes && __any_sync(0xFFFFFFFFu, go); p++) {
            const uint32_t M = bd.pivot();
            uint4 r0, r1;
            ldg32_if(go, d.rec + 2 * (size_t)M, &r0, &r1);
            if (go) {
                uint32_t l;
                bool und = false;
                int c = cmp_record(w, m, r0, r1, d.n, &l, &und);
                if (!kFromList && und)
                    c = cmp_suffix_qw(d.text, d.n, r1.w, qw, m, max(kRecBases, min(bd.lcpL, bd.lcpR)), &l);
                if (kFromList && und) {
                    pending = true;
                    pend_pos = r1.w;
                    pend_lcps = r1.z & 0xFFFFu;
                    go = false;
                } else {
                    step(c, M, l, (r1.z >> 8) & 0xFFu, r1.z & 0xFFu);
                }
            }
        }
        if (kFromList && pending) {
            uint32_t l;
            const int c = cmp_suffix_pairs(d.text, d.n, pend_pos, qw, m, max(kRecBases, min(bd.lcpL, bd.lcpR)), &l);
            step(c, bd.pivot(), l, pend_lcps >> 8, pend_lcps & 0xFFu);
        }

        if (live && done) store_result_sum(a, q, lo, hi);

        // The rest goes to the worklist with one bracket of both bounds:
        // phase 0 (L, R); phase 1 (L, HR) (lo in (L, M], hi in [M, HR));
        // phase 2 (lo - 1, R) (lo known, hi in (L, R) with L >= lo).  Records
        // are staged per warp in shared memory and flushed 32 at a time, so
        // the global count takes one atomic per 32 records.
        const bool rest = live && !done;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, rest);
        if (bal != 0u) {
            const uint32_t n_new = (uint32_t)__popc(bal);
            if (staged + n_new > 32u) {
                flush(staged);
                staged = 0;
            }
            if (rest) {
                const uint32_t slot = staged + __popc(bal & lanemask_lt);
                s_stage[wib][slot][0] = make_uint4(bd.phase == 2 ? bd.lo - 1u : bd.L,
                                                     bd.phase == 1 ? bd.HR : bd.R, m, (uint32_t)q);
                const uint64_t w4 = m > 128u ? qw(128u) : 0ull;  // bases 128-159 for the persistent pass
                s_stage[wib][slot][1] =
                    make_uint4((uint32_t)qa, place_high(qa, r), (uint32_t)w4, (uint32_t)(w4 >> 32));
                s_stage[wib][slot][2] =
                    make_uint4((uint32_t)w[0], (uint32_t)(w[0] >> 32), (uint32_t)w[1], (uint32_t)(w[1] >> 32));
                s_stage[wib][slot][3] =
                    make_uint4((uint32_t)w[2], (uint32_t)(w[2] >> 32), (uint32_t)w[3], (uint32_t)(w[3] >> 32));
            }
            staged += n_new;
            __syncwarp();
        }
    }
    flush(staged);
    if (!kFromList) {
        if (__any_sync(0xFFFFFFFFu, any_bad) && lane == 0) atomicOr(a.pack_err, 1);
        if (__any_sync(0xFFFFFFFFu, any_bad_ref) && lane == 0) atomicOr(a.bad_ref, 1);
    }
}

}  // namespace

cudaError_t launch_front(const SearchLaunch &L, cudaStream_t s) {
    if (L.n_q == 0) return cudaSuccess;
    const bool single = L.n_refs == 1 && L.q_ref == nullptr;
    const bool list = L.wrec_in != nullptr;
    static int per_sm[12][64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    using Kernel = void (*)(SearchLaunch);
    constexpr Bases P = Bases::Packed, S = Bases::PackedStrands;
    static const Kernel kernels[12] = {front_kernel<false, false, P>, front_kernel<true, false, P>,
                                       front_kernel<false, false, S>, front_kernel<true, false, S>,
                                       front_kernel<false, true, P>,  front_kernel<true, true, P>,
                                       front_kernel<false, true, S>,  front_kernel<true, true, S>,
                                       front_kernel<false, false, P, true>, front_kernel<true, false, P, true>,
                                       front_kernel<false, false, S, true>, front_kernel<true, false, S, true>};
    const int bases = L.revcomp || L.strand_bits ? 1 : 0;
    const int which = (single ? 1 : 0) + 2 * bases + (list ? 4 : L.front_probes == 1 ? 8 : 0);
    const Kernel kernel = kernels[which];
    int &bps = per_sm[which][dev];
    if (bps == 0) {
        int b = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kFrontThreads, 0);
        if (e != cudaSuccess) return e;
        bps = b > 0 ? b : 1;
    }
    const uint64_t warps = (L.n_q + 31) / 32;
    const uint64_t cap = (uint64_t)device_sm_count() * bps;
    uint64_t blocks = (warps + kFrontThreads / 32 - 1) / (kFrontThreads / 32);
    if (blocks > cap) blocks = cap;
    kernel<<<(unsigned)blocks, kFrontThreads, 0, s>>>(L);
    return cudaGetLastError();
}

}  // namespace sa
