// small.cu -- the search of a small batch (Section IV) in one kernel.
//
// A batch of some thousand queries does not fill the GPU, so what it costs is
// latency: the launches, the packing, the first and the persistent pass one
// after the other, and in those the dependent reads of the query with the
// longest binary search.  Here one kernel does it all:
//   * a thread packs its query's first bases from the ASCII itself and checks
//     them; a long query's bytes are checked by its warp, or by CTAs of a second
//     kernel (kLaneBases), so that none takes one thread long;
//   * the k-mer entry of its first k bases and up to kLaneProbes probes settle
//     most queries, as in the first pass (front.cu);
//   * a query that remains -- a wide bracket, an index without a k-mer table --
//     is finished by its whole warp: the 32 lanes probe 32 ranks spread over
//     the bracket at once, so a bracket of 1000 suffixes takes two rounds
//     of reads instead of ten, and one of 10^8 six instead of 27;
//   * a warp takes few queries when the batch is small (as many as give every
//     resident warp some), so that those rounds follow one another seldom.
// A round reads 32 records where a step of the binary search reads one: right
// while the GPU has nothing else to do, wrong for a large batch (api.cu:
// small_batch has the line between the two and both sides' times).
//
// Bound by the latency of a handful of dependent reads: 20 queries against 5
// Mbp 51 -> 24 us a call (of which a call that reads nothing takes about 20),
// 10^5 queries of 32 bases at 1 Mbp 57 -> 26 us, 20,011 of 20-300 bases of
// both strands over four genomes, with locate, 83 -> 47 us.  Random queries at
// 100 Mbp, with every byte checked by the query's lane, as it is, and by the
// other path, us a call: 20 of 10^5 bases 997, 45, 51; 20,000 of 20-300 and one
// of 10^6 9530, 45, 60; 5*10^5 of 100 and one of 10^7 131,700, 123, 94;
// 5*10^5 of 100 alone 66, 69, 92 (the second kernel).
#include "first_pass.cuh"

namespace sa {

namespace {

constexpr int kSmallThreads = 128;
constexpr int kSmallPerSm = 8;  // CTAs
constexpr uint32_t kLaneProbes = 2;
// Who checks that a query's bytes are bases: its lane up to kLaneBases, its
// warp beyond, and past kWarpBases in a batch that can hold far longer ones
// (SearchLaunch::check_longest) some CTAs of a second kernel.  A warp takes its
// longer queries one after the other, 0.6 us each, where its lanes check them
// side by side, 10 ns a base: with many that are not much longer (kWarpTurn)
// the lanes do.
constexpr uint32_t kLaneBases = 512;
constexpr uint32_t kWarpTurn = 128;
constexpr uint32_t kWarpBases = 1u << 15;
constexpr int kLongestThreads = 256;
constexpr uint32_t kLongestFound = 1024;  // queries a CTA notes; with more it goes through its share again

__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) {
    return __shfl_sync(0xFFFFFFFFu, (unsigned long long)v, src);
}

// Whether some of the m bytes at p is not a base, as thread t of the kThreads
// that check them sees it: the aligned 16-byte pieces dealt out in turn, eight
// loads of a thread in flight (past the end the last piece again: under a test
// the loads would wait for one another).
template <uint32_t kThreads>
__device__ __forceinline__ bool not_all_bases(const uint8_t *__restrict__ p, uint32_t m, uint32_t t) {
    constexpr uint32_t kInFlight = 8;
    const uint32_t to_aligned = (16u - ((uint32_t)(uintptr_t)p & 15u)) & 15u;
    const uint32_t head = min(m, to_aligned), pieces = (m - head) / 16u, tail = m - head - 16u * pieces;
    const uint4 *v = reinterpret_cast<const uint4 *>(p + head);
    uint32_t bad = 0;
    for (uint32_t i = t; i < pieces; i += kThreads * kInFlight) {
        uint4 x[kInFlight];
#pragma unroll
        for (uint32_t j = 0; j < kInFlight; j++) x[j] = __ldg(v + min(i + kThreads * j, pieces - 1u));
#pragma unroll
        for (uint32_t j = 0; j < kInFlight; j++) bad |= not_bases(x[j]);
    }
    if (t < head) bad |= base_code(__ldg(p + t)) > 3u;
    if (t < tail) bad |= base_code(__ldg(p + head + 16u * pieces + t)) > 3u;
    return bad != 0u;
}

// The same for each lane in `lanes`, whose query is the m bytes at byte qa of
// the batch, by the whole warp.  A function of its own, so that the kernel's
// registers stay its main path's: inlined, 5*10^5 queries of 100 bases took 33
// -> 38 us.
__device__ __noinline__ bool check_by_warp(const uint8_t *__restrict__ ascii, uint64_t qa, uint32_t m, unsigned lanes) {
    const unsigned lane = threadIdx.x & 31u;
    bool mine = false;
    for (; lanes != 0u; lanes &= lanes - 1u) {
        const int src = __ffs(lanes) - 1;
        const bool bad = not_all_bases<32>(ascii + shfl64(qa, src), __shfl_sync(0xFFFFFFFFu, m, src), lane);
        if (__any_sync(0xFFFFFFFFu, bad) && (int)lane == src) mine = true;
    }
    return mine;
}

// Query q (m bases, its first 128 in w, all in qw) against ranks (L, R) by the
// whole warp; every argument is the same in all lanes.  Each round's lanes
// probe ranks spread over what is open: while no rank with the query as prefix
// is known, all over (L, R); then the lower 16 over (loL, loR) and the upper
// 16 over (hiL, hiR), which hold the two ends of the interval.  known (in
// shared memory, of this warp: the registers are full) holds the query's common
// prefixes with the suffixes at the lowest and the highest bound as far as
// known: a compare in the text starts from what its lane's bounds share.
__device__ __forceinline__ void finish_by_warp(const FrontDesc &d, const AsciiWindows &qw, const uint64_t w[4],
                                               uint32_t m, uint32_t L, uint32_t R, volatile uint32_t *known,
                                               uint64_t *lo, uint64_t *hi) {
    const unsigned lane = threadIdx.x & 31u;
    bool split = false;  // a match is known: (L, R) is (loL, loR), and (hL, hR) the upper end's
    uint32_t hL = 0, hR = 0;
    for (;;) {
        const bool open_lo = R - L > 1u, open_hi = split && hR - hL > 1u;
        if (!open_lo && !open_hi) break;
        // this lane's interval and its place among the lanes that share it
        const bool both = open_lo && open_hi;
        const bool upper = both ? lane >= 16u : !open_lo;
        const uint32_t lanes = both ? 16u : 32u, at = both ? (lane & 15u) : lane;
        const uint32_t a = upper ? hL : L, b = upper ? hR : R;
        const uint32_t inside = b - a - 1u;  // ranks strictly between
        const bool live = at < inside;
        const uint32_t M = inside <= lanes ? a + 1u + at : a + (uint32_t)(((uint64_t)(b - a) * (at + 1u)) / (lanes + 1u));
        uint4 r0, r1;
        ldg32_if(live, d.rec + 2 * (size_t)M, &r0, &r1);
        int c = 2;
        uint32_t l = 0;
        if (live) {
            bool und = false;
            c = cmp_record(w, m, r0, r1, d.n, &l, &und);
            if (und) {
                const uint32_t share = upper ? known[1] : (split ? known[0] : min(known[0], known[1]));
                c = cmp_suffix_qw(d.text, d.n, r1.w, qw, m, max(kRecBases, share), &l);
            }
        }
        const uint32_t cut = min(m, kLcpCap);
        const unsigned match = __ballot_sync(0xFFFFFFFFu, c == CMP_PREFIX);
        const unsigned less = __ballot_sync(0xFFFFFFFFu, c == CMP_LESS);
        const unsigned greater = __ballot_sync(0xFFFFFFFFu, c == CMP_GREATER);
        // matches whose neighbour is known not to match settle an end
        const unsigned low_end = __ballot_sync(0xFFFFFFFFu, c == CMP_PREFIX && ((r1.z >> 8) & 0xFFu) < cut);
        const unsigned high_end = __ballot_sync(0xFFFFFFFFu, c == CMP_PREFIX && (r1.z & 0xFFu) < cut);
        auto rank_of = [&](int src) { return __shfl_sync(0xFFFFFFFFu, M, src); };
        const unsigned lo_lanes = both ? 0x0000FFFFu : (split && !open_lo ? 0u : 0xFFFFFFFFu);
        const unsigned hi_lanes = both ? 0xFFFF0000u : (split && open_lo ? 0u : (split ? 0xFFFFFFFFu : 0u));
        // the lower end's lanes (before the split: all lanes serve both ends)
        const unsigned g = greater & lo_lanes, p = match & lo_lanes, s = less & lo_lanes;
        const uint32_t last_g = rank_of(g ? 31 - __clz(g) : 0), first_p = rank_of(p ? __ffs(p) - 1 : 0);
        const uint32_t last_p = rank_of(p ? 31 - __clz(p) : 0), first_s = rank_of(s ? __ffs(s) - 1 : 0);
        // the new bounds' common prefixes (R's, or once split hR's: no rank
        // below R sorts after the query), for a query that goes on past a record
        if (m > kRecBases) {
            if (g && lane == 31u - __clz(g)) known[0] = l;
            if (less && lane == (unsigned)__ffs(less) - 1u) known[1] = l;
            __syncwarp();
        }
        const bool low_known = p && ((low_end >> (__ffs(p) - 1)) & 1u);
        const bool high_known = p && ((high_end >> (31 - __clz(p))) & 1u);
        // the upper end's lanes after the split
        const unsigned hp = match & hi_lanes, hs = less & hi_lanes;
        const uint32_t h_last_p = rank_of(hp ? 31 - __clz(hp) : 0), h_first_s = rank_of(hs ? __ffs(hs) - 1 : 0);
        const bool h_known = hp && ((high_end >> (31 - __clz(hp))) & 1u);
        if (g) L = last_g;
        if (!split) {
            if (p) {
                split = true;
                hL = last_p;
                hR = high_known ? last_p + 1u : (s ? first_s : R);
                R = first_p;
                if (low_known) L = first_p - 1u;
            } else if (s) {
                R = first_s;
            }
        } else {
            if (p) {
                R = first_p;
                if (low_known) L = first_p - 1u;
            }
            if (hs) hR = h_first_s;
            if (hp) {
                hL = h_last_p;
                if (h_known) hR = h_last_p + 1u;
            }
        }
    }
    *lo = R;
    *hi = split ? hR : R;
}

template <bool kSingle>
__global__ void __launch_bounds__(kSmallThreads, kSmallPerSm) small_kernel(const __grid_constant__ SearchLaunch a,
                                                                          uint32_t per_warp) {
    __shared__ FrontDesc sdesc[SA_MAX_REFS];
    __shared__ uint32_t s_known[kSmallThreads / 32][2];
    if (a.check_longest) asm volatile("griddepcontrol.launch_dependents;");
    const unsigned lane = threadIdx.x & 31u;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t q = warp * per_warp + lane;
    const bool live = lane < per_warp && q < a.n_q;
    uint64_t qa = 0, qe = 0;
    uint32_t r = 0;
    if (live) {
        qa = __ldg(a.q_off + q) - a.first;
        qe = __ldg(a.q_off + q + 1) - a.first;
        if (!kSingle) r = __ldg(a.q_ref + q);
    }
    for (unsigned i = threadIdx.x; i < a.n_refs; i += blockDim.x) sdesc[i] = front_desc(a.refs.r[i]);
    __syncthreads();
    if (warp * per_warp >= a.n_q) return;  // (whole warps)

    const bool rc = a.revcomp || (a.strand_bits && (r & kStrandBit));
    if (a.strand_bits) r &= ~kStrandBit;
    const bool range_ok = live && qa <= qe && qe <= a.total && qe - qa < (1ull << 31);
    bool ok = range_ok && r < a.n_refs;
    const bool bad_ref = range_ok && !ok;
    const uint32_t m = ok ? (uint32_t)(qe - qa) : 0u;
    const uint8_t *ascii = reinterpret_cast<const uint8_t *>(a.ascii);
    const bool elsewhere = a.check_longest && m > kWarpBases;
    unsigned by_warp = __ballot_sync(0xFFFFFFFFu, m > kLaneBases && !elsewhere);
    if (__reduce_max_sync(0xFFFFFFFFu, elsewhere ? 0u : m) < kWarpTurn * __popc(by_warp)) by_warp = 0u;
    uint32_t bad = by_warp != 0u && check_by_warp(ascii, qa, m, by_warp) ? 1u : 0u;
    const AsciiWindows qw{ascii, a.total, qa, m, rc};
    uint64_t w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < 4; j++)
        if (m > 32u * j) w[j] = qw.packed(32u * j, &bad);
    const bool by_lane = !elsewhere && !((by_warp >> lane) & 1u);
    for (uint32_t off = 128u; by_lane && off < m; off += 32u) (void)qw.packed(off, &bad);
    ok = ok && bad == 0u;

    FrontDesc d = sdesc[0];
    if (!kSingle && ok) d = sdesc[r];
    const uint32_t kk = d.kmer_k;
    const bool look = ok && m > 0 && d.krt != nullptr && m >= kk;
    uint4 h, e01, e23, e45;
    ldg64_pairs_if(look, d.krt + 4 * (look ? (w[0] >> (64u - 2u * kk)) : 0ull), &h, &e01, &e23, &e45);
    Bounds bd;
    bd.start(look ? h.x - 1u : 0xFFFFFFFFu, look ? h.y : d.n);
    bool done = !live || !ok || m == 0 || (look && bd.R - bd.L <= 1u);
    uint64_t lo = bd.R, hi = bd.R;  // a bracket without suffixes
    if (live && !ok) lo = hi = ~0ull;
    if (live && ok && m == 0) {
        lo = 0;
        hi = d.n;
    }
    if (live && ok && m > 0 && d.krt != nullptr && m < kk) {
        uint32_t l, u;
        brief_interval(d, w[0] >> (64u - 2u * m), m, &l, &u);
        lo = l;
        hi = u;
        done = true;
    }
    bool go = !done && look;
    auto step = [&](int c, uint32_t M, uint32_t l, uint32_t lp, uint32_t ln) {
        if (bd.step(c, M, l, m, lp, ln)) {
            lo = bd.first();
            hi = bd.R;
            done = true;
            go = false;
        }
    };
    if (go) {
        const uint64_t e[6] = {((uint64_t)e01.y << 32) | e01.x, ((uint64_t)e01.w << 32) | e01.z,
                               ((uint64_t)e23.y << 32) | e23.x, ((uint64_t)e23.w << 32) | e23.z,
                               ((uint64_t)e45.y << 32) | e45.x, ((uint64_t)e45.w << 32) | e45.z};
        uint32_t l;
        const int c = cmp_entry(w, m, e, h.z, h.w & 0xFFu, d.n, d.text, qw, &l);
        step(c, bd.pivot(), l, (h.w >> 8) & 0xFFu, (h.w >> 16) & 0xFFu);
    }
    for (uint32_t p = 0; p < kLaneProbes && __any_sync(0xFFFFFFFFu, go); p++) {
        const uint32_t M = bd.pivot();
        uint4 r0, r1;
        ldg32_if(go, d.rec + 2 * (size_t)M, &r0, &r1);
        if (go) {
            uint32_t l;
            bool und = false;
            int c = cmp_record(w, m, r0, r1, d.n, &l, &und);
            if (und) c = cmp_suffix_qw(d.text, d.n, r1.w, qw, m, max(kRecBases, min(bd.lcpL, bd.lcpR)), &l);
            step(c, M, l, (r1.z >> 8) & 0xFFu, r1.z & 0xFFu);
        }
    }
    // one bracket of both bounds, as for the worklist of front.cu
    const uint32_t L = bd.phase == 2 ? bd.lo - 1u : bd.L, R = bd.phase == 1 ? bd.HR : bd.R;
    unsigned rest = __ballot_sync(0xFFFFFFFFu, live && !done);
    while (rest != 0u) {
        const int src = __ffs(rest) - 1;
        rest &= rest - 1u;
        uint64_t wq[4];
#pragma unroll
        for (int j = 0; j < 4; j++) wq[j] = shfl64(w[j], src);
        const uint32_t mq = __shfl_sync(0xFFFFFFFFu, m, src), rq = __shfl_sync(0xFFFFFFFFu, r, src);
        const AsciiWindows qwq{qw.ascii, qw.total, shfl64(qa, src), mq, __shfl_sync(0xFFFFFFFFu, (int)rc, src) != 0};
        if ((int)lane == src) {
            s_known[threadIdx.x >> 5][0] = bd.phase == 2 ? 0u : bd.lcpL;
            s_known[threadIdx.x >> 5][1] = bd.phase == 1 ? bd.hlcpR : bd.lcpR;
        }
        __syncwarp();
        uint64_t l, u;
        finish_by_warp(sdesc[kSingle ? 0u : rq], qwq, wq, mq, __shfl_sync(0xFFFFFFFFu, L, src),
                       __shfl_sync(0xFFFFFFFFu, R, src), s_known[threadIdx.x >> 5], &l, &u);
        if ((int)lane == src) {
            lo = l;
            hi = u;
        }
    }
    if (live) store_result_sum(a, q, lo, hi);
    const bool any_bad = __any_sync(0xFFFFFFFFu, live && !ok && !bad_ref);
    const bool any_bad_ref = __any_sync(0xFFFFFFFFu, bad_ref);
    if (lane == 0 && any_bad && a.pack_err != nullptr) atomicOr(a.pack_err, 1);
    if (lane == 0 && any_bad_ref && a.bad_ref != nullptr) atomicOr(a.bad_ref, 1);
}

// The bytes of the queries of more than kWarpBases, whose results small_kernel
// stores as if they were bases.  `parts` CTAs look through the same share of the
// offsets, while small_kernel's last CTAs run, and each checks its part of the
// queries found.  The thread that is the first to find a byte that is not a
// base takes the result back.
__global__ void __launch_bounds__(kLongestThreads) check_longest_kernel(const __grid_constant__ SearchLaunch a,
                                                                       uint32_t parts) {
    __shared__ uint32_t found[kLongestFound];
    __shared__ uint32_t n_found;
    const uint64_t shares = gridDim.x / parts, share = (a.n_q + shares - 1) / shares;
    const uint64_t begin = blockIdx.x / parts * share;
    const uint64_t end = begin + share < a.n_q ? begin + share : a.n_q;
    const uint32_t part = blockIdx.x % parts;
    // the query's first byte and length, 0 unless the check is this kernel's
    auto longest = [&](uint64_t q, uint64_t *qa) {
        *qa = __ldg(a.q_off + q) - a.first;
        const uint64_t qe = __ldg(a.q_off + q + 1) - a.first;
        return *qa <= qe && qe <= a.total && qe - *qa < (1ull << 31) && qe - *qa > kWarpBases ? (uint32_t)(qe - *qa)
                                                                                              : 0u;
    };
    if (threadIdx.x == 0) n_found = 0;
    __syncthreads();
#pragma unroll 8
    for (uint64_t q = begin + threadIdx.x; q < end; q += kLongestThreads) {
        uint64_t qa;
        if (longest(q, &qa) != 0u) {
            const uint32_t at = atomicAdd(&n_found, 1u);
            if (at < kLongestFound) found[at] = (uint32_t)(q - begin);
        }
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");  // small_kernel's results are there
    const bool noted = n_found <= kLongestFound;  // (always, unless offsets go back)
    const uint64_t n = noted ? n_found : end - begin;
    for (uint64_t i = 0; i < n; i++) {
        const uint64_t q = begin + (noted ? found[i] : i);
        uint64_t qa;
        const uint32_t m = longest(q, &qa);
        if (m == 0u) continue;
        const uint32_t from = (uint32_t)((uint64_t)m * part / parts);
        const uint32_t to = (uint32_t)((uint64_t)m * (part + 1) / parts);
        if (!not_all_bases<kLongestThreads>(reinterpret_cast<const uint8_t *>(a.ascii) + qa + from, to - from, threadIdx.x))
            continue;
        const uint64_t count = __ldcg(&a.out[q].count);
        // (all ones already: a bad reference id, a byte small_kernel saw, or another thread here)
        if (atomicExch(reinterpret_cast<unsigned long long *>(&a.out[q].lo), ~0ull) == ~0ull) continue;
        a.out[q].hi = ~0ull;
        a.out[q].count = ~0ull;
        a.out[q].flags = SA_RESULT_INVALID;
        if (a.tile_kept != nullptr)
            atomicAdd(reinterpret_cast<unsigned long long *>(a.tile_kept) + (q >> a.tile_shift),
                      0ull - (count < a.trunc_cap ? count : a.trunc_cap));
        if (a.pack_err != nullptr) atomicOr(a.pack_err, 1);
    }
}

}  // namespace

cudaError_t launch_search_small(const SearchLaunch &L, cudaStream_t s) {
    if (L.n_q == 0) return cudaSuccess;
    // the fewest queries per warp (a power of two) with which the batch's
    // warps are all resident
    const uint64_t warps = (uint64_t)device_sm_count() * kSmallPerSm * (kSmallThreads / 32);
    uint32_t per_warp = 1;
    while (per_warp < 32 && per_warp * warps < L.n_q) per_warp *= 2;
    const uint64_t per_cta = (uint64_t)per_warp * (kSmallThreads / 32);
    const unsigned blocks = (unsigned)((L.n_q + per_cta - 1) / per_cta);
    if (L.n_refs == 1 && L.q_ref == nullptr)
        small_kernel<true><<<blocks, kSmallThreads, 0, s>>>(L, per_warp);
    else
        small_kernel<false><<<blocks, kSmallThreads, 0, s>>>(L, per_warp);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !L.check_longest) return e;
    // launched while small_kernel's last CTAs run; it waits for them itself
    uint32_t parts = 64;  // (all of them together read at most 2^22 offsets)
    while (parts > 8 && parts * L.n_q > (1u << 22)) parts /= 2;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(((unsigned)device_sm_count() * 4u / parts + 1u) * parts);
    cfg.blockDim = dim3(kLongestThreads);
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, check_longest_kernel, L, parts);
}

}  // namespace sa
