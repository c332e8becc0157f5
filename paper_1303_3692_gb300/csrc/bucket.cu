// bucket.cu -- the worklist of a batch in k-mer order, for indexes larger
// than the GPU's address-translation reach.
//
// The probes of a search are random reads into the k-mer entries and suffix
// records (Section IV's binary search, with the exact shortcuts of this
// library).  On the GB300 such reads run at about 37-40 G sectors/s while the
// reads in flight across the GPU touch no more than ~64 GB; over a 190 GB
// index, with every lane at a random place, the rate falls to ~8 G/s.  A
// batch processed in the order of its queries' first k bases keeps the reads
// in flight inside a narrow slice of the index instead (measured: 40 G/s
// within 1 GB windows of a 192 GB buffer).  Ranks follow k-mer order, so a
// query's k-mer entry and every suffix record of its bracket lie in its
// slice.
//
// Four kernels (six for an unpacked batch) put the batch in that order before the
// first pass (front.cu), which then reads its queries from the list they write:
//   bucket_sample_kernel   every kListSampleStride-th query's bucket -- its
//                          first k bases as a fraction of all k-mer entries
//                          of the call's indexes, in kNumBuckets equal
//                          slices, or the extra bucket of queries with no
//                          k-mer bracket -- counted;
//   bucket_plan_kernel     one warp: from those counts each bucket's region
//                          of the list (9/8 of its estimated size plus 256
//                          records), in bucket order, and after them an
//                          overflow region with room for every query;
//   bucket_scatter_kernel (or, for an unpacked batch, bucket_scatter_ascii_kernel,
//                          and then for the few tiles it leaves out)
//                          per tile of queries: offsets, strand, reference,
//                          validity of every base when the packing found a
//                          non-base byte in the batch (invalid and empty
//                          queries get their results here) and bucket; each
//                          bucket's run reserved at once in its region (what
//                          does not fit goes to the overflow region), every
//                          query's 64-byte record (length, index, reference,
//                          first base in the packed batch, first 192 bases;
//                          flagged when it has a k-mer bracket to read) built
//                          in shared memory and the runs stored coalesced;
//   bucket_fill_kernel     one warp: the prefix sums of the regions' fills,
//                          by which the first pass numbers the records
//                          (region by region, then the overflow).
// The first pass and then the persistent kernel of search.cu take the queries
// in that order, so the reads in flight at any time stay in a few slices.
// Sizing the regions from a sample spares a pass over the whole batch that
// exact counts would need; the overflow region keeps the result exact
// whatever the sample missed.
#include "first_pass.cuh"

namespace sa {

namespace {

constexpr int kSampleThreads = 256;
constexpr uint16_t kNoQuery = 0xFFFFu;  // invalid or empty query: no list record

struct BucketRef {
    uint64_t kbase;   // k-mer entries of the earlier indexes of the call
    uint64_t n;
    uint32_t kmer_k;  // 0: no k-mer table
};

// The query's place in the packed batch (which names its strand), its length,
// its reference id (*r, the strand bit cleared) and whether the range and the
// reference id are usable.
template <bool kStrands>
__device__ __forceinline__ bool query_range(const SearchLaunch &a, uint64_t q, uint32_t *r, uint64_t *at_out,
                                            uint32_t *m_out, bool *bad_range, bool *bad_ref) {
    const uint64_t qa = __ldg(a.q_off + q) - a.first, qe = __ldg(a.q_off + q + 1) - a.first;
    const bool rc = kStrands && (a.revcomp || (a.strand_bits && (*r & kStrandBit)));
    if (kStrands && a.strand_bits) *r &= ~kStrandBit;
    const bool range_ok = qa <= qe && qe <= a.total && qe - qa < (1ull << 31);
    *bad_range = !range_ok;
    *bad_ref = range_ok && *r >= a.n_refs;
    *at_out = range_ok ? query_place(qa, qe, rc) : 0;
    *m_out = range_ok ? (uint32_t)(qe - qa) : 0u;
    return range_ok && *r < a.n_refs;
}

// The bucket of a usable query of length m >= 1 whose first 32 bases are w0.
__device__ __forceinline__ uint16_t bucket_of(const SearchLaunch &a, const BucketRef &d, uint32_t m, uint64_t w0) {
    if (d.kmer_k != 0 && m >= d.kmer_k) {
        const uint64_t x = w0 >> (64u - 2u * d.kmer_k);
        static_assert(kNumBuckets == 256, "the shift below");
        return (uint16_t)__umul64hi((d.kbase + x) << 8, a.kscale);  // about 256 (kbase + x) / ktotal
    }
    return (uint16_t)kNumBuckets;  // no k-mer bracket: the key-table descent
}

template <bool kSingle, Bases kBases>
__global__ void __launch_bounds__(kSampleThreads) bucket_sample_kernel(const __grid_constant__ SearchLaunch a) {
    __shared__ uint32_t hist[kNumBuckets + 1];
    __shared__ BucketRef sref[SA_MAX_REFS];
    for (unsigned i = threadIdx.x; i <= kNumBuckets; i += blockDim.x) hist[i] = 0;
    for (unsigned r = threadIdx.x; r < a.n_refs; r += blockDim.x) {
        const RefDesc &d = a.refs.r[r];
        sref[r] = BucketRef{d.kbase, d.n, d.krt != nullptr ? d.kmer_k : 0u};
    }
    __syncthreads();
    const uint64_t n_s = (a.n_q + kListSampleStride - 1) / kListSampleStride;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_s; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t q = i * kListSampleStride;
        uint32_t r = kSingle ? 0u : __ldg(a.q_ref + q);
        uint64_t at;
        uint32_t m;
        bool bad_range, bad_ref;
        // an estimate: the bases' validity is left to the scatter
        if (query_range<kBases != Bases::Packed>(a, q, &r, &at, &m, &bad_range, &bad_ref) && m > 0)
            atomicAdd(&hist[bucket_of(a, sref[kSingle ? 0u : r], m, window_source<kBases>(a, at, m)(0))], 1u);
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i <= kNumBuckets; i += blockDim.x)
        if (hist[i]) atomicAdd(a.bplan + kPlanSample + i, hist[i]);
}

// One warp: each bucket's region of the list and its cursor, then the
// overflow region.  A bucket sampled s times gets s * stride * 9/8 + 256
// records; the regions follow one another in bucket order.
__global__ void bucket_plan_kernel(const __grid_constant__ SearchLaunch a) {
    const unsigned lane = threadIdx.x;
    uint32_t *plan = a.bplan;
    uint32_t carry = 0;
    for (unsigned base = 0; base <= kNumBuckets; base += 32) {
        const unsigned i = base + lane;
        const uint32_t est = i <= kNumBuckets ? plan[kPlanSample + i] * kListSampleStride : 0u;
        const uint32_t v = i <= kNumBuckets ? est + est / 8u + 256u : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= (unsigned)o) x += y;
        }
        if (i <= kNumBuckets) {
            plan[kPlanStart + i] = carry + x - v;
            plan[kPlanCursor + i] = carry + x - v;
            plan[kPlanCap + i] = v;
        }
        carry += __shfl_sync(0xFFFFFFFFu, x, 31);
    }
    if (lane == 0) {
        plan[kPlanOvStart] = carry;
        plan[kPlanOvCursor] = carry;
    }
}

// Scatter: one CTA per tile of kScatterTile queries.  The tile's records are
// first built in shared memory in bucket order (each bucket's run of the
// tile contiguous), then copied out run by run: consecutive threads store
// consecutive 16-byte words of a run, so the stores coalesce (a record
// written straight to its slot from each lane would put the 32 lanes of a
// warp in 32 different runs).  Each bucket's run is reserved with one atomic
// on the bucket's cursor; the part past the region's end is reserved in the
// overflow region.
constexpr int kScatterThreads = 256;
constexpr int kScatterItems = 2;
static_assert(kScatterTile == (uint32_t)kScatterThreads * kScatterItems, "a tile's queries (32 KB of records)");
constexpr size_t kScatterSmem = (size_t)kScatterTile * 64;

// A tile's runs: exclusive scan of its counts (first warp), and each run's
// place in the list, reserved with one atomic per bucket.
__device__ __forceinline__ void reserve_runs(const SearchLaunch &a, const uint32_t *cnt, uint32_t *off, uint32_t *base,
                                             uint32_t *inreg, uint32_t *ovbase, uint32_t *n_valid) {
    if (threadIdx.x < 32) {
        const unsigned lane = threadIdx.x;
        uint32_t carry = 0;
        for (unsigned s0 = 0; s0 <= kNumBuckets; s0 += 32) {
            const unsigned i = s0 + lane;
            const uint32_t v = i <= kNumBuckets ? cnt[i] : 0u;
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= (unsigned)o) x += y;
            }
            if (i <= kNumBuckets) off[i] = carry + x - v;
            carry += __shfl_sync(0xFFFFFFFFu, x, 31);
        }
        if (lane == 0) *n_valid = carry;
    }
    for (unsigned i = threadIdx.x; i <= kNumBuckets; i += blockDim.x) {
        const uint32_t c = cnt[i];
        if (c == 0) continue;
        const uint32_t start = atomicAdd(a.bplan + kPlanCursor + i, c);
        const uint32_t end = a.bplan[kPlanStart + i] + a.bplan[kPlanCap + i];
        const uint32_t fit = start >= end ? 0u : (end - start < c ? end - start : c);
        base[i] = start;
        inreg[i] = fit;
        ovbase[i] = fit < c ? atomicAdd(a.bplan + kPlanOvCursor, c - fit) : 0u;
    }
}

// Whether the m > 0 bases from base qa on are all bases, by the bitmap alone and
// the bytes of the few words it marks; a very long query's by the whole warp.
// Called by all 32 lanes.
__device__ __forceinline__ bool spoiled_valid(const SearchLaunch &a, bool look, uint64_t qa, uint32_t m) {
    const uint8_t *ascii = reinterpret_cast<const uint8_t *>(a.ascii);
    const unsigned lane = threadIdx.x & 31u;
    constexpr uint32_t kByLane = 1u << 15;
    bool valid = true;
    for (unsigned left = __ballot_sync(0xFFFFFFFFu, look); left != 0u;) {
        // all lanes with a shorter query at once, then the others one by one
        const unsigned shorter = __ballot_sync(0xFFFFFFFFu, ((left >> lane) & 1u) && m <= kByLane);
        const int src = shorter ? (int)lane : __ffs(left) - 1;
        const uint64_t q0 = __shfl_sync(0xFFFFFFFFu, (unsigned long long)qa, src);
        const uint32_t len = __shfl_sync(0xFFFFFFFFu, m, src);
        const bool mine = shorter == 0u || ((shorter >> lane) & 1u);
        bool ok = true;
        if (mine) {
            const uint64_t w0 = q0 >> 5, w1 = (q0 + len - 1) >> 5;
            for (uint64_t g = (w0 >> 5) + (shorter ? 0u : lane); ok && g <= (w1 >> 5); g += shorter ? 1u : 32u) {
                uint32_t marked = __ldg(a.tvb + g);
                if (g == (w0 >> 5)) marked &= 0xFFFFFFFFu << (w0 & 31u);
                if (g == (w1 >> 5)) marked &= 0xFFFFFFFFu >> (31u - (uint32_t)(w1 & 31u));
                for (; ok && marked != 0u; marked &= marked - 1u) {
                    const uint64_t b0 = (g * 32 + (__ffs(marked) - 1)) * 32;
                    ok = bytes_valid(ascii, b0 > q0 ? b0 : q0, b0 + 32 < q0 + len ? b0 + 32 : q0 + len);
                }
            }
        }
        const bool all = __all_sync(0xFFFFFFFFu, ok);
        if (shorter) {
            valid = valid && ok;
            left &= ~shorter;
        } else {
            if ((int)lane == src) valid = all;
            left &= left - 1u;
        }
    }
    return valid;
}

// kListed: the tiles are those the scatter of an unpacked batch left out,
// packed since (fused launches; a few CTAs go through them).
template <bool kSingle, bool kStrands, bool kListed = false>
__global__ void __launch_bounds__(kScatterThreads, 5) bucket_scatter_kernel(const __grid_constant__ SearchLaunch a,
                                                                           uint4 *__restrict__ list) {
    extern __shared__ uint4 srec[];  // kScatterTile records of 4 uint4
    __shared__ uint32_t cnt[kNumBuckets + 1];
    __shared__ uint32_t off[kNumBuckets + 1];     // the run's first slot in the tile
    __shared__ uint32_t base[kNumBuckets + 1];    // its first slot in the list (in the bucket's region)
    __shared__ uint32_t inreg[kNumBuckets + 1];   // how many of the run fit the region
    __shared__ uint32_t ovbase[kNumBuckets + 1];  // the first overflow slot of the rest
    __shared__ uint16_t slot_bucket[kScatterTile];
    __shared__ BucketRef sref[SA_MAX_REFS];
    __shared__ uint32_t n_valid;
    for (unsigned r = threadIdx.x; r < a.n_refs; r += blockDim.x) {
        const RefDesc &d = a.refs.r[r];
        sref[r] = BucketRef{d.kbase, d.n, d.krt != nullptr ? d.kmer_k : 0u};
    }
    // a batch without a non-base byte needs no validity masks
    const bool dirty = *a.batch_dirty != 0;
    const uint32_t n_tiles = kListed ? *a.n_spoiled : gridDim.x;
    for (uint32_t ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
        for (unsigned i = threadIdx.x; i <= kNumBuckets; i += blockDim.x) cnt[i] = 0;
        const uint64_t tile = (uint64_t)(kListed ? a.spoiled[ti].x : ti) * kScatterTile;
        uint16_t b[kScatterItems];
        uint32_t rank[kScatterItems], r[kScatterItems], m[kScatterItems];
        uint64_t at[kScatterItems], w[kScatterItems][4];
        bool any_bad = false, any_bad_ref = false;
        __syncthreads();
        // Every item's loads are issued before the tile's bookkeeping, so that
        // their DRAM round trips overlap each other and the scans below.
#pragma unroll
        for (int it = 0; it < kScatterItems; it++) {
            const uint64_t q = tile + (uint64_t)it * kScatterThreads + threadIdx.x;
            r[it] = kSingle || q >= a.n_q ? 0u : __ldg(a.q_ref + q);
        }
#pragma unroll
        for (int it = 0; it < kScatterItems; it++) {
            const uint64_t q = tile + (uint64_t)it * kScatterThreads + threadIdx.x;
            at[it] = 0;
            m[it] = 0;
            b[it] = kNoQuery;
            if (q < a.n_q) {
                bool bad_range, bad_ref;
                const bool ok = query_range<kStrands>(a, q, &r[it], &at[it], &m[it], &bad_range, &bad_ref);
                any_bad |= bad_range;
                any_bad_ref |= bad_ref;
                b[it] = ok ? 0u : kNoQuery;  // usable so far; the bucket follows
            }
        }
#pragma unroll
        for (int it = 0; it < kScatterItems; it++) {
            const uint64_t q = tile + (uint64_t)it * kScatterThreads + threadIdx.x;
            // a query without a record reads the batch's first words (always there)
            const bool ok = b[it] != kNoQuery;
            query_windows<4, kStrands>(a.tq, ok ? at[it] : 0, 0, w[it]);
            const bool look = ok && m[it] > 0 && dirty;
            const uint64_t qa = place_first(at[it], m[it]);
            const bool valid = kListed ? spoiled_valid(a, look, qa, m[it]) : !look || query_valid(a.tvb, a.tv, qa, m[it]);
            if (q >= a.n_q) continue;
            if (!ok || !valid) {
                if (ok) any_bad = true;
                b[it] = kNoQuery;
                store_result_sum(a, q, ~0ull, ~0ull);
            } else if (m[it] == 0) {
                b[it] = kNoQuery;
                store_result_sum(a, q, 0, sref[kSingle ? 0u : r[it]].n);
            } else {
                b[it] = bucket_of(a, sref[kSingle ? 0u : r[it]], m[it], w[it][0]);
            }
        }
#pragma unroll
        for (int it = 0; it < kScatterItems; it++) rank[it] = b[it] != kNoQuery ? atomicAdd(&cnt[b[it]], 1u) : 0u;
        __syncthreads();
        reserve_runs(a, cnt, off, base, inreg, ovbase, &n_valid);
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kScatterItems; it++) {
            if (b[it] == kNoQuery) continue;
            const uint64_t q = tile + (uint64_t)it * kScatterThreads + threadIdx.x;
            const bool entry = b[it] < kNumBuckets;
            const uint32_t slot = off[b[it]] + rank[it];
            // bases 128-191 (the first pass then reads none of a query of up to
            // 192 bases from the batch)
            uint64_t t[2] = {0, 0};
            if (m[it] > 128u) query_windows<2, kStrands>(a.tq, at[it], 128u, t);
            uint4 *dst = srec + 4 * slot;
            dst[0] = make_uint4(m[it], (uint32_t)q, (uint32_t)at[it],
                                place_high(at[it], r[it]) | (entry ? kListNeedsEntry : 0u));
            dst[1] = make_uint4((uint32_t)w[it][0], (uint32_t)(w[it][0] >> 32), (uint32_t)w[it][1],
                                (uint32_t)(w[it][1] >> 32));
            dst[2] = make_uint4((uint32_t)w[it][2], (uint32_t)(w[it][2] >> 32), (uint32_t)w[it][3],
                                (uint32_t)(w[it][3] >> 32));
            dst[3] = make_uint4((uint32_t)t[0], (uint32_t)(t[0] >> 32), (uint32_t)t[1], (uint32_t)(t[1] >> 32));
            slot_bucket[slot] = b[it];
        }
        __syncthreads();
        // copy the runs out, 16 bytes per thread per step
        const uint32_t words = 4u * n_valid;
        for (uint32_t c = threadIdx.x; c < words; c += kScatterThreads) {
            const uint32_t slot = c >> 2;
            const uint32_t bk = slot_bucket[slot];
            const uint32_t k = slot - off[bk];
            const uint64_t g = k < inreg[bk] ? (uint64_t)base[bk] + k : (uint64_t)ovbase[bk] + (k - inreg[bk]);
            list[4 * g + (c & 3u)] = srec[c];
        }
        const unsigned lane = threadIdx.x & 31u;
        if (__any_sync(0xFFFFFFFFu, any_bad) && lane == 0) atomicOr(a.pack_err, 1);
        if (__any_sync(0xFFFFFFFFu, any_bad_ref) && lane == 0) atomicOr(a.bad_ref, 1);
        if (kListed) __syncthreads();  // the next tile's counts and records go over these
    }
}

// The scatter of a batch that is not packed (api.cu: kRecordBases).  The CTA
// packs its tile's bases itself, coalesced, into shared memory -- consecutive
// queries are one stretch of the batch -- and every 16-byte piece of a record
// is computed from there as it is stored, so the packed batch is neither
// written nor read back: per query of 150 bases 150 + 64 bytes of HBM traffic
// instead of 150 + 38 + 38 + 64.  What a record holds, the runs and their
// reservation are as above.  A tile with a query longer than compares read from
// its records writes its words to the packed batch for them.  One whose words
// do not fit -- a query far longer than the others -- is left to
// pack_spoiled_kernel and bucket_scatter_kernel (two launches, 4 us when there is
// none).  2^21 queries of 100 bases at 100 Mbp, us a call, with every compare
// past the records from the ASCII bases and every query of such a tile packed by
// one thread, and as it is: a tenth of them of 600 bases, 80 % copied, 750, 580;
// 400 of 10^5 random bases 1850, 320; one of 10^7 136,700, 298; none of either
// 275, 283.  Bound by the integer pipe (69 % busy; HBM 53 %):
// 4*10^7 x 150 bases 1.99 ms, where the packing and the scatter took 1.19 +
// 1.29 ms; 9*10^6 of 100-151 bases of both strands, some with an N, 0.47 ms for
// 0.24 + 0.33.  (The same in the first pass of input order, a tile per warp, was
// no faster at 100 bases, 586 us for 577, and slower at 20-250, 1263 for 1144:
// its warps wait for their reads in turn.)
constexpr uint32_t kTileWords = kScatterTile * 6;  // 192 bases per query
constexpr uint32_t kTileLead = 6, kTilePad = 8;
constexpr size_t kScatterAsciiSmem = (kTileLead + kTileWords + kTilePad) * 8 + kScatterTile * 16;
static_assert((kTileLead + kTileWords + kTilePad) * sizeof(uint2) % alignof(uint4) == 0,
              "the headers after the tile's words are read and written as uint4");

// 16 bases of a tile as a 32-bit word, base 0 on top: the tile holds its packed
// words' high halves before their low ones, so a window at any base is a funnel
// shift of two neighbours.
__device__ __forceinline__ uint32_t tile_window16(const uint32_t *half, int base) {
    const int i = base >> 4;
    return __funnelshift_l(half[i + 1], half[i], 2u * (uint32_t)(base & 15));
}

__device__ __forceinline__ uint32_t rc_window16(uint32_t x) {
    const uint32_t f = __brev(~x);
    return ((f >> 1) & 0x55555555u) | ((f & 0x55555555u) << 1);
}

// The N x 16 bases from base `off` of a query whose first base (for the other
// strand, one past its last) is base `at` of the tile.
template <int N>
__device__ __forceinline__ void tile_windows(const uint32_t *half, int at, bool rc, int off, uint32_t w[N]) {
    const int b = rc ? at - off - 16 * N : at + off;
    uint32_t t[N];
#pragma unroll
    for (int j = 0; j < N; j++) t[j] = tile_window16(half, b + 16 * j);
#pragma unroll
    for (int j = 0; j < N; j++) w[j] = rc ? rc_window16(t[N - 1 - j]) : t[j];
}

template <bool kSingle>
__global__ void __launch_bounds__(kScatterThreads, 5) bucket_scatter_ascii_kernel(const __grid_constant__ SearchLaunch a,
                                                                                 uint4 *__restrict__ list,
                                                                                 uint64_t *__restrict__ tq) {
    // the tile's words (kTileLead of no meaning before, kTilePad after), then its records' headers
    extern __shared__ __align__(16) uint2 stile[];
    uint2 *words = stile + kTileLead;
    const uint32_t *half = reinterpret_cast<const uint32_t *>(words);
    uint4 *head = reinterpret_cast<uint4 *>(stile + kTileLead + kTileWords + kTilePad);
    __shared__ uint32_t cnt[kNumBuckets + 1];
    __shared__ uint32_t off[kNumBuckets + 1];
    __shared__ uint32_t base[kNumBuckets + 1];
    __shared__ uint32_t inreg[kNumBuckets + 1];
    __shared__ uint32_t ovbase[kNumBuckets + 1];
    __shared__ uint32_t slot_to[kScatterTile];  // each slot's record in the list
    __shared__ uint32_t marks[kTileWords / 32];
    __shared__ BucketRef sref[SA_MAX_REFS];
    __shared__ uint32_t n_valid, w_first, w_last, any_marked, any_longer;
    for (unsigned i = threadIdx.x; i <= kNumBuckets; i += blockDim.x) cnt[i] = 0;
    for (unsigned r = threadIdx.x; r < a.n_refs; r += blockDim.x) {
        const RefDesc &d = a.refs.r[r];
        sref[r] = BucketRef{d.kbase, d.n, d.krt != nullptr ? d.kmer_k : 0u};
    }
    if (threadIdx.x == 0) {
        w_first = 0xFFFFFFFFu;
        w_last = 0;
        any_marked = 0;
        any_longer = 0;
    }
    const unsigned lane = threadIdx.x & 31u;
    const uint8_t *ascii = reinterpret_cast<const uint8_t *>(a.ascii);
    const bool aligned16 = ((uintptr_t)ascii & 15u) == 0;
    const uint64_t tile = (uint64_t)blockIdx.x * kScatterTile;
    uint16_t b[kScatterItems];
    uint32_t rank[kScatterItems], r[kScatterItems], m[kScatterItems];
    uint64_t at[kScatterItems];
    bool any_bad = false, any_bad_ref = false;
    uint32_t lo = 0xFFFFFFFFu, hi = 0;  // the words of this thread's queries
#pragma unroll
    for (int it = 0; it < kScatterItems; it++) {
        const uint64_t q = tile + (uint64_t)it * kScatterThreads + threadIdx.x;
        r[it] = kSingle || q >= a.n_q ? 0u : __ldg(a.q_ref + q);
        at[it] = 0;
        m[it] = 0;
        b[it] = kNoQuery;
        if (q < a.n_q) {
            bool bad_range, bad_ref;
            const bool ok = query_range<true>(a, q, &r[it], &at[it], &m[it], &bad_range, &bad_ref);
            any_bad |= bad_range;
            any_bad_ref |= bad_ref;
            if (ok) {
                b[it] = 0u;  // usable so far; the bucket follows
                if (m[it] > 0) {
                    const uint64_t qa = place_first(at[it], m[it]);
                    lo = min(lo, (uint32_t)(qa >> 5));
                    hi = max(hi, (uint32_t)((qa + m[it] - 1) >> 5));
                }
            }
        }
    }
    lo = __reduce_min_sync(0xFFFFFFFFu, lo);
    hi = __reduce_max_sync(0xFFFFFFFFu, hi);
    __syncthreads();
    if (lane == 0 && lo <= hi) {
        atomicMin(&w_first, lo);
        atomicMax(&w_last, hi);
    }
    __syncthreads();
    const uint32_t w_lo = w_first <= w_last ? w_first : 0u;
    const uint32_t n_words = w_first <= w_last ? w_last - w_first + 1u : 0u;
    if (n_words > kTileWords) {  // for pack_spoiled_kernel and bucket_scatter_kernel
        if (threadIdx.x == 0) a.spoiled[atomicAdd(a.n_spoiled, 1u)] = make_uint4(blockIdx.x, w_lo, n_words, 0u);
        return;
    }
    const uint64_t full = aligned16 ? a.total / 32 : 0;  // words that are two 16-byte loads
    for (uint32_t i0 = threadIdx.x - lane; i0 < n_words; i0 += kScatterThreads) {
        const uint32_t i = i0 + lane;
        const uint64_t w = (uint64_t)w_lo + i;
        uint32_t bad = 0;
        if (i < n_words) {
            const uint4 *from = reinterpret_cast<const uint4 *>(ascii + w * 32);
            const uint64_t x = w < full ? pack32(__ldg(from), __ldg(from + 1), &bad)
                                        : pack_edge_word(ascii, a.total, w, &bad);
            words[i] = make_uint2((uint32_t)(x >> 32), (uint32_t)x);
        }
        const unsigned marked = __ballot_sync(0xFFFFFFFFu, bad != 0u);
        if (lane == 0) {
            marks[i0 >> 5] = marked;
            if (marked != 0u) any_marked = 1u;
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kScatterItems; it++) {
        const uint64_t q = tile + (uint64_t)it * kScatterThreads + threadIdx.x;
        if (q >= a.n_q) continue;
        bool valid = b[it] != kNoQuery;
        uint64_t first = 0;  // the query's first 32 bases
        if (valid && m[it] > 0) {
            valid = any_marked == 0u || tile_valid(marks, w_lo, ascii, place_first(at[it], m[it]), m[it]);
            uint32_t f[2];
            tile_windows<2>(half, (int)((at[it] & ~kPlaceRc) - 32ull * w_lo), (at[it] & kPlaceRc) != 0, 0, f);
            first = ((uint64_t)f[0] << 32) | f[1];
            any_bad |= !valid;
        }
        if (!valid) {
            b[it] = kNoQuery;
            store_result_sum(a, q, ~0ull, ~0ull);
        } else if (m[it] == 0) {
            b[it] = kNoQuery;
            store_result_sum(a, q, 0, sref[kSingle ? 0u : r[it]].n);
        } else {
            b[it] = bucket_of(a, sref[kSingle ? 0u : r[it]], m[it], first);
            // (the worklist's records carry 160 bases; the key tables' descent
            // goes on in the text after 64)
            if (m[it] > (b[it] < kNumBuckets ? 160u : 64u)) any_longer = 1u;
        }
    }
#pragma unroll
    for (int it = 0; it < kScatterItems; it++) rank[it] = b[it] != kNoQuery ? atomicAdd(&cnt[b[it]], 1u) : 0u;
    __syncthreads();
    reserve_runs(a, cnt, off, base, inreg, ovbase, &n_valid);
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kScatterItems; it++) {
        if (b[it] == kNoQuery) continue;
        const uint64_t q = tile + (uint64_t)it * kScatterThreads + threadIdx.x;
        const uint32_t bk = b[it], slot = off[bk] + rank[it];
        head[slot] = make_uint4(m[it], (uint32_t)q, (uint32_t)at[it],
                                place_high(at[it], r[it]) | (bk < kNumBuckets ? kListNeedsEntry : 0u));
        slot_to[slot] = rank[it] < inreg[bk] ? base[bk] + rank[it] : ovbase[bk] + (rank[it] - inreg[bk]);
    }
    __syncthreads();
    // compares that go on past the records read the packed batch
    if (any_longer != 0u)
        for (uint32_t i = threadIdx.x; i < n_words; i += kScatterThreads)
            tq[(uint64_t)w_lo + i] = ((uint64_t)words[i].x << 32) | words[i].y;
    // the runs, 16 bytes per thread per step: the header, or 64 of the
    // record's 192 bases
    const uint32_t pieces = 4u * n_valid;
    for (uint32_t c = threadIdx.x; c < pieces; c += kScatterThreads) {
        const uint32_t slot = c >> 2, part = c & 3u;
        uint4 v = head[slot];
        if (part != 0u) {
            uint32_t w[4];
            tile_windows<4>(half, (int)(place_of(v.z, v.w & ~kRecordRc) - 32ull * w_lo), (v.w & kRecordRc) != 0,
                            64 * ((int)part - 1), w);
            v = make_uint4(w[1], w[0], w[3], w[2]);
        }
        list[4 * (uint64_t)slot_to[slot] + part] = v;
    }
    if (__any_sync(0xFFFFFFFFu, any_bad) && lane == 0) atomicOr(a.pack_err, 1);
    if (__any_sync(0xFFFFFFFFu, any_bad_ref) && lane == 0) atomicOr(a.bad_ref, 1);
}

// One warp: the exclusive prefix sums of the regions' fills (the records
// each bucket's region received), their total, and the list's record count
// (the regions' records, then the overflow's).
__global__ void bucket_fill_kernel(const __grid_constant__ SearchLaunch a) {
    const unsigned lane = threadIdx.x;
    uint32_t *plan = a.bplan;
    uint32_t carry = 0;
    for (unsigned s0 = 0; s0 <= kNumBuckets; s0 += 32) {
        const unsigned i = s0 + lane;
        uint32_t v = 0;
        if (i <= kNumBuckets) {
            const uint32_t used = plan[kPlanCursor + i] - plan[kPlanStart + i];
            v = used < plan[kPlanCap + i] ? used : plan[kPlanCap + i];
        }
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= (unsigned)o) x += y;
        }
        if (i <= kNumBuckets) plan[kPlanPrefix + i] = carry + x - v;
        carry += __shfl_sync(0xFFFFFFFFu, x, 31);
    }
    if (lane == 0) {
        plan[kPlanPrefix + kNumBuckets + 1] = carry;
        *a.wl_in_count = carry + (plan[kPlanOvCursor] - plan[kPlanOvStart]);
    }
}

}  // namespace

cudaError_t launch_bucketed_worklist(const SearchLaunch &L, uint4 *wrec_in, uint64_t *tq, uint32_t *tvb,
                                     cudaStream_t s) {
    if (L.n_q == 0) return cudaSuccess;
    const bool single = L.n_refs == 1 && L.q_ref == nullptr;
    const uint64_t n_s = (L.n_q + kListSampleStride - 1) / kListSampleStride;
    uint64_t sblocks = (n_s + kSampleThreads - 1) / kSampleThreads;
    const uint64_t scap = (uint64_t)device_sm_count() * 8;
    if (sblocks > scap) sblocks = scap;
    const bool strands = L.revcomp || L.strand_bits;
    constexpr Bases P = Bases::Packed, S = Bases::PackedStrands, A = Bases::Ascii;
    auto sample = single ? (L.fused ? bucket_sample_kernel<true, A>
                                    : strands ? bucket_sample_kernel<true, S> : bucket_sample_kernel<true, P>)
                         : (L.fused ? bucket_sample_kernel<false, A>
                                    : strands ? bucket_sample_kernel<false, S> : bucket_sample_kernel<false, P>);
    sample<<<(unsigned)sblocks, kSampleThreads, 0, s>>>(L);
    bucket_plan_kernel<<<1, 32, 0, s>>>(L);
    const unsigned tiles = (unsigned)scatter_tiles(L.n_q);
    cudaError_t e = cudaSuccess;
    auto packed = [&](auto kernel, unsigned blocks) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScatterSmem);
        if (e == cudaSuccess) kernel<<<blocks, kScatterThreads, kScatterSmem, s>>>(L, wrec_in);
    };
    if (L.fused) {
        auto scatter = single ? bucket_scatter_ascii_kernel<true> : bucket_scatter_ascii_kernel<false>;
        e = cudaFuncSetAttribute(scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScatterAsciiSmem);
        if (e != cudaSuccess) return e;
        scatter<<<tiles, kScatterThreads, kScatterAsciiSmem, s>>>(L, wrec_in, tq);
        if ((e = launch_pack_spoiled(L, tq, tvb, s)) != cudaSuccess) return e;
        const unsigned all = (unsigned)device_sm_count() * 5u, blocks = tiles < all ? tiles : all;
        if (single)
            strands ? packed(bucket_scatter_kernel<true, true, true>, blocks)
                    : packed(bucket_scatter_kernel<true, false, true>, blocks);
        else
            strands ? packed(bucket_scatter_kernel<false, true, true>, blocks)
                    : packed(bucket_scatter_kernel<false, false, true>, blocks);
    } else if (single) {
        strands ? packed(bucket_scatter_kernel<true, true>, tiles) : packed(bucket_scatter_kernel<true, false>, tiles);
    } else {
        strands ? packed(bucket_scatter_kernel<false, true>, tiles) : packed(bucket_scatter_kernel<false, false>, tiles);
    }
    if (e != cudaSuccess) return e;
    bucket_fill_kernel<<<1, 32, 0, s>>>(L);
    return cudaGetLastError();
}

}  // namespace sa
