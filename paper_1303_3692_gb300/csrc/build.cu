// build.cu -- suffix-array construction on the GPU by prefix doubling (or the
// upload of one built on the host by DC3), and the sampled-key table.  Off the
// search path; timed apart from it.
//
// The paper builds its suffix array on the host (the straightforward sort or
// DC3, Section III).  Here the text is already packed in device memory, so
// the array is built there, by radix sorts of short keys that leave few
// suffixes to look at again (build_suffix_array):
//   1. all suffixes are sorted by their first 16 bases (a 32-bit key: 16 bytes
//      moved per suffix and pass, four passes);
//   2. a group of at most 32 suffixes that are still equal is ordered by
//      comparing them in the text, each with the others (refine_kernel), and
//      only larger groups, or suffixes that stay equal for long, go on;
//   3. those are sorted by (their group, their next ~20 bases), and refined
//      again, round by round, while that is cheaper than what follows;
//   4. what then remains (long repeats) goes through prefix doubling: the ranks
//      of all suffixes are written out, the remaining ones re-sorted by the
//      pair (rank[i], rank[i + h]), h the depth the order is known to, and h
//      doubles.  Ranks are the suffix-array position of the first member of
//      the group, so they order groups globally and a finished group's rank
//      is its final position.
// A suffix that ends within the compared bases is packed with A's (zeros)
// after its end; it sorts before every other suffix with the same key, the
// shorter of two such first (the order of Table I).  The first sort starts
// from descending text positions and every sort is stable, so they come in
// that order by themselves, and each counts as a group of its own.
// The radix sorts, scans and compactions come from CUB (a source-only library
// shipped with the CUDA toolkit); the rest are kernels here.
#include <cub/cub.cuh>
#include <thrust/iterator/counting_iterator.h>
#include <vector>

#include "dc3.h"
#include "sa_internal.cuh"

namespace sa {

namespace {

constexpr int kThreads = 256;

unsigned grid_for(uint64_t n) {
    uint64_t b = (n + kThreads - 1) / kThreads;
    const uint64_t cap = (uint64_t)device_sm_count() * 32;
    if (b > cap) b = cap;
    return (unsigned)(b ? b : 1);
}

#define GS_LOOP(i, n) \
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (uint64_t)gridDim.x * blockDim.x)

constexpr uint64_t kFirstBases = 16;

// The first sort's keys, from the last suffix to the first: 16 bases.
__global__ void init_keys_kernel(const uint64_t *__restrict__ T, uint64_t n, uint32_t *keys, uint32_t *vals) {
    GS_LOOP(t, n) {
        const uint64_t i = n - 1 - t;
        keys[t] = (uint32_t)(text_window(T, i) >> 32);
        vals[t] = (uint32_t)i;
    }
}

// The order of the suffixes at i and j (different; both longer than depth and
// equal so far) by up to `windows` further windows of 32 bases: -1 when S_j
// sorts before S_i, 1 after, 0 when they stay equal.
__device__ __forceinline__ int order_beyond(const uint64_t *__restrict__ T, uint64_t n, uint64_t i, uint64_t j,
                                            uint64_t depth, uint32_t windows) {
    const uint64_t shorter = n - (i > j ? i : j);  // bases of the shorter suffix
    for (uint32_t w = 0; w < windows; w++) {
        const uint64_t at = depth + 32ull * w;
        const uint64_t a = text_window(T, i + at), b = text_window(T, j + at), x = a ^ b;
        const uint64_t same = x ? (uint64_t)(__clzll((long long)x) >> 1) : 32u;
        const uint64_t left = shorter - at;
        if (same < left && same < 32) return b < a ? -1 : 1;
        if (left <= 32) return j > i ? -1 : 1;  // the shorter one ends first
    }
    return 0;
}

// One sort's outcome: items 0 .. cnt - 1 (suffix vals[t], going to suffix-array
// slot pos[t], or t itself when pos is null) ordered by key, equal keys (no
// suffix of the two ended within `depth` bases) being groups that share their
// first `depth` bases.  Writes every item to its slot: a group of one as it
// is; one of up to kSmallGroup members in the order the text gives, member by
// member the number of the others that sort before it (its compares read the
// same few lines of text as theirs); a larger one in the order it has.
// unresolved[t] marks the items of the list that are not settled, headb[slot]
// the first of each group of them.
// A block takes kRefineOut items with kSmallGroup more on each side, whose
// heads it needs to find the groups; one ballot per warp gives a word of
// heads.  A member's first window beyond depth is read once, into shared
// memory, where the others find it; only members equal there are compared in
// the text, over at most kRefineWindows windows per item in all.  Bound by
// those random reads and its members' compares: 1.4 ms for 10^8 human-like
// bases, of whose suffixes the first sort leaves about a third in groups, 10.4
// ms for 6*10^8 (2.0 and 20.3 with the rule for suffixes that end nearby in
// every compare).  Sorting by 64-bit keys of 29 bases instead, eight passes of 24 bytes,
// and prefix doubling for the rest took 15 ms in all at 10^8, this 9.
constexpr int kRefineThreads = 512;
constexpr int kSmallGroup = 32;
constexpr int kRefineOut = kRefineThreads - 2 * kSmallGroup;
constexpr uint32_t kRefineWindows = 64;

template <typename K>
__global__ void __launch_bounds__(kRefineThreads) refine_kernel(const K *__restrict__ keys,
                                                                const uint32_t *__restrict__ vals, uint64_t cnt,
                                                                const uint32_t *__restrict__ pos,
                                                                const uint64_t *__restrict__ T, uint64_t n,
                                                                uint64_t depth, uint32_t *sa, uint8_t *unresolved,
                                                                uint8_t *headb) {
    __shared__ uint32_t heads[kRefineThreads / 32];
    __shared__ uint64_t next[kRefineThreads];
    __shared__ uint32_t ends_near;  // some suffix of the tile ends within the next window
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint64_t tiles = (cnt + kRefineOut - 1) / kRefineOut;
    for (uint64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t t = (int64_t)(tile * kRefineOut) + threadIdx.x - kSmallGroup;
        const bool live = t >= 0 && t < (int64_t)cnt;
        uint32_t i = 0;
        bool head = t >= (int64_t)cnt;  // past the end: a boundary
        if (live) {
            i = vals[t];
            head = t == 0 || keys[t] != keys[t - 1] || n - i <= depth || n - vals[t - 1] <= depth;
        }
        const unsigned word = __ballot_sync(0xFFFFFFFFu, head);
        if (lane == 0) heads[warp] = word;
        if (threadIdx.x == 0) ends_near = 0;
        __syncthreads();
        // the group's start (at or before t) and end (after t)
        const uint32_t upto = word & (0xFFFFFFFFu >> (31u - lane));
        const uint32_t above = lane < 31u ? word & (0xFFFFFFFFu << (lane + 1u)) : 0u;
        const uint32_t before = warp > 0 ? heads[warp - 1] : 0u;
        const uint32_t after = warp < kRefineThreads / 32 - 1 ? heads[warp + 1] : 0u;
        uint32_t back = kSmallGroup, ahead = kSmallGroup + 1;  // members before t; distance to the end
        if (upto)
            back = lane - (31u - __clz(upto));
        else if (before)
            back = lane + 1u + __clz(before);
        if (above)
            ahead = (uint32_t)__ffs(above) - 1u - lane;
        else if (after)
            ahead = 31u - lane + (uint32_t)__ffs(after);
        const uint32_t size = back + ahead;
        // (of the items beside the block's own, those of a group that reaches
        // into it: no head between them and it)
        const bool left_of = warp == 0, right_of = warp == kRefineThreads / 32 - 1;
        const bool reaches = left_of ? above == 0u : !right_of || upto == 0u;
        if (live && reaches && size > 1u && size <= (uint32_t)kSmallGroup) {
            next[threadIdx.x] = text_window(T, (uint64_t)i + depth);
            if (n - i < depth + 32) ends_near = 1;
        }
        __syncthreads();
        if (live && !left_of && !right_of) {
            uint64_t at = t;  // the item's place in the list
            bool more = false, first = false;
            if (size > (uint32_t)kSmallGroup) {
                more = true;
                first = head;
            } else if (size > 1u) {
                const uint64_t a = t - back;
                const uint32_t windows = kRefineWindows / size;
                const uint64_t mine = next[threadIdx.x];
                uint32_t less = 0, ties = 0, ties_before = 0;
                const uint64_t *group = next + (threadIdx.x - back);
                if (!ends_near) {  // nearly always: the windows decide, but for equal ones
                    uint32_t equal = 0;  // members with the same window
                    for (uint32_t u = 0; u < size; u++) {
                        const uint64_t theirs = group[u];
                        less += theirs < mine ? 1u : 0u;
                        equal |= theirs == mine ? 1u << u : 0u;
                    }
                    for (equal &= ~(1u << back); equal != 0u; equal &= equal - 1u) {
                        const uint32_t u = __ffs(equal) - 1;
                        const uint32_t j = vals[a + u];
                        const bool ended = n - (i > j ? i : j) == depth + 32;
                        const int c = ended ? (j > i ? -1 : 1) : order_beyond(T, n, i, j, depth + 32, windows);
                        less += c < 0 ? 1u : 0u;
                        ties += c == 0 ? 1u : 0u;
                        ties_before += (c == 0 && u < back) ? 1u : 0u;
                    }
                } else {
                    for (uint32_t u = 0; u < size; u++) {
                        if (u == back) continue;
                        const uint64_t theirs = group[u];
                        int c = theirs < mine ? -1 : 1;
                        const uint32_t j = vals[a + u];
                        const uint64_t x = mine ^ theirs;
                        const uint64_t same = x ? (uint64_t)(__clzll((long long)x) >> 1) : 32u;
                        const uint64_t left = n - (i > j ? i : j) - depth;  // bases of the shorter one there
                        if (same >= left)
                            c = j > i ? -1 : 1;  // it ends first
                        else if (x == 0)
                            c = left > 32 ? order_beyond(T, n, i, j, depth + 32, windows) : (j > i ? -1 : 1);
                        less += c < 0 ? 1u : 0u;
                        ties += c == 0 ? 1u : 0u;
                        ties_before += (c == 0 && u < back) ? 1u : 0u;
                    }
                }
                at = a + less + ties_before;
                more = ties != 0u;
                first = ties_before == 0u;
            }
            const uint64_t slot = pos ? pos[at] : at;
            sa[slot] = i;
            unresolved[at] = more ? 1 : 0;
            if (more) headb[slot] = first ? 1 : 0;
        }
        __syncthreads();
    }
}

// 1 where the list's item t is the first of its group.
__global__ void group_heads_kernel(const uint32_t *__restrict__ pos, uint64_t cnt, const uint8_t *__restrict__ headb,
                                   uint32_t *g) {
    GS_LOOP(t, cnt) g[t] = headb[pos[t]];
}

// A later sort's keys: the item's group number (from 1, in list order) above
// its next `bases` bases from `depth` on.
__global__ void group_keys_kernel(const uint64_t *__restrict__ T, const uint32_t *__restrict__ pos, uint64_t cnt,
                                  const uint32_t *__restrict__ sa, const uint32_t *__restrict__ group,
                                  uint64_t depth, uint32_t bases, uint64_t *keys, uint32_t *vals) {
    GS_LOOP(t, cnt) {
        const uint32_t i = sa[pos[t]];
        keys[t] = ((uint64_t)(group[t] - 1u) << (2u * bases)) | (text_window(T, (uint64_t)i + depth) >> (64u - 2u * bases));
        vals[t] = i;
    }
}

// Prefix doubling starts from every suffix's rank: its slot, or for the
// suffixes still in groups the slot of their group's head.
__global__ void slot_ranks_kernel(const uint32_t *__restrict__ sa, uint64_t n, uint32_t *isa) {
    GS_LOOP(j, n) isa[sa[j]] = (uint32_t)j;
}

__global__ void head_slots_kernel(const uint32_t *__restrict__ pos, uint64_t cnt, const uint8_t *__restrict__ headb,
                                  uint32_t *hv) {
    GS_LOOP(t, cnt) hv[t] = headb[pos[t]] ? pos[t] : 0u;
}

__global__ void group_ranks_kernel(const uint32_t *__restrict__ pos, uint64_t cnt, const uint32_t *__restrict__ sa,
                                   const uint32_t *__restrict__ rank, uint32_t *isa) {
    GS_LOOP(t, cnt) isa[sa[pos[t]]] = rank[t];
}

// head value: pos[t] if item t starts a group of equal keys, else 0.
__global__ void head_values_kernel(const uint64_t *__restrict__ keys, uint64_t cnt,
                                   const uint32_t *__restrict__ pos, uint32_t *hv) {
    GS_LOOP(t, cnt) hv[t] = t == 0 || keys[t] != keys[t - 1] ? pos[t] : 0u;
}

// After the scan, rank[t] is the SA position of t's group head.  Writes the
// ranks, the suffix-array entries, and flags members of groups of size > 1.
__global__ void scatter_ranks_kernel(const uint64_t *__restrict__ keys, uint64_t cnt,
                                     const uint32_t *__restrict__ pos,   // SA positions
                                     const uint32_t *__restrict__ sorted_vals, const uint32_t *__restrict__ rank,
                                     uint32_t *isa, uint32_t *sa, uint8_t *unresolved) {
    GS_LOOP(t, cnt) {
        const uint32_t i = sorted_vals[t];
        sa[pos[t]] = i;
        isa[i] = rank[t];
        const bool head = t == 0 || keys[t] != keys[t - 1];
        const bool tail = t + 1 == cnt || keys[t + 1] != keys[t];
        unresolved[t] = (head && tail) ? 0 : 1;
    }
}

// Doubling key of the unresolved member at SA position pos[t].
__global__ void pair_keys_kernel(const uint32_t *__restrict__ pos, uint64_t cnt, const uint32_t *__restrict__ sa,
                                 const uint32_t *__restrict__ isa, uint64_t n, uint64_t h, uint64_t *keys,
                                 uint32_t *vals) {
    GS_LOOP(t, cnt) {
        const uint32_t i = sa[pos[t]];
        const uint64_t r1 = isa[i];
        const uint64_t r2 = (uint64_t)i + h < n ? (uint64_t)isa[i + h] + 1 : 0;
        keys[t] = (r1 << 32) | r2;
        vals[t] = i;
    }
}

__global__ void widen_kernel(const uint32_t *__restrict__ src, uint64_t n, uint64_t *dst) {
    GS_LOOP(i, n) dst[i] = src[i];
}

struct MaxOp {
    __device__ __forceinline__ uint32_t operator()(uint32_t a, uint32_t b) const { return a > b ? a : b; }
};

int bit_length(uint64_t x) {
    int b = 0;
    while (x) {
        b++;
        x >>= 1;
    }
    return b;
}

struct Pool {
    cudaStream_t s;
    Arena *arenas = nullptr;
    int n_arenas = 0;
    std::vector<void *> ptrs;
    cudaError_t err = cudaSuccess;
    template <typename T>
    T *get(size_t count) {
        void *p = nullptr;
        if (err != cudaSuccess) return nullptr;
        const size_t need = (count * sizeof(T) + 255) / 256 * 256;
        for (int i = 0; i < n_arenas; i++) {
            if (arenas[i].left < need) continue;
            p = arenas[i].at;
            arenas[i].at += need;
            arenas[i].left -= need;
            return reinterpret_cast<T *>(p);
        }
        err = scratch_alloc(&p, count * sizeof(T) + 16, s);
        if (err == cudaSuccess) ptrs.push_back(p);
        return reinterpret_cast<T *>(p);
    }
    ~Pool() {
        for (void *p : ptrs) scratch_free(p, s);
    }
};

}  // namespace

#define CK(x)                                   \
    do {                                        \
        cudaError_t e_ = (x);                   \
        if (e_ != cudaSuccess) return status_from_cuda(e_); \
    } while (0)

// Sorts by groups and next bases (step 3 above) are cheaper than prefix
// doubling, whose ranks cost one random write per suffix, as long as they
// handle few suffixes: at most half as many as the text has, in all, and at
// most one round per 2^22 suffixes (a round's launches and its read of the
// count take 0.1 ms, the ranks of 4*10^6 suffixes as long), 48 in the end.
constexpr uint64_t kRoundSuffixes = 1ull << 22;
constexpr uint64_t kMostRounds = 48;

int build_suffix_array(sa_index *idx, cudaStream_t s, Arena *arenas, int n_arenas) {
    const uint64_t n = idx->n;
    const uint64_t *T = idx->text;
    Pool pool{s, arenas, n_arenas};
    uint64_t *kA = pool.get<uint64_t>(n), *kB = pool.get<uint64_t>(n);
    uint32_t *vA = pool.get<uint32_t>(n), *vB = pool.get<uint32_t>(n);
    // the 32-bit array is built in place, a 64-bit one widened from scratch
    uint32_t *sa32 = idx->width == 4 ? reinterpret_cast<uint32_t *>(idx->sa) : pool.get<uint32_t>(n);
    uint32_t *isa = pool.get<uint32_t>(n), *hv = pool.get<uint32_t>(n);
    uint32_t *posA = pool.get<uint32_t>(n), *posB = pool.get<uint32_t>(n);
    uint8_t *flag = pool.get<uint8_t>(n), *headb = pool.get<uint8_t>(n);
    uint64_t *d_count = pool.get<uint64_t>(1);
    if (pool.err != cudaSuccess) return SA_ERR_NOMEM;
    uint32_t *group = isa;  // group numbers, before the ranks are needed

    // Temporary storage sized for the largest call of each CUB routine.
    size_t t_bytes = 0;
    thrust::counting_iterator<uint32_t> iota(0);
    cub::DoubleBuffer<uint32_t> kb32(reinterpret_cast<uint32_t *>(kA), reinterpret_cast<uint32_t *>(kB));
    {
        cub::DoubleBuffer<uint64_t> kb(kA, kB);
        cub::DoubleBuffer<uint32_t> vb(vA, vB);
        size_t t[6] = {};
        CK(cub::DeviceRadixSort::SortPairs(nullptr, t[0], kb, vb, n, 0, 64, s));
        CK(cub::DeviceRadixSort::SortPairs(nullptr, t[1], kb32, vb, n, 0, 32, s));
        CK(cub::DeviceScan::InclusiveScan(nullptr, t[2], hv, hv, MaxOp(), n, s));
        CK(cub::DeviceScan::InclusiveSum(nullptr, t[3], group, group, n, s));
        CK(cub::DeviceSelect::Flagged(nullptr, t[4], posA, flag, posB, d_count, n, s));
        CK(cub::DeviceSelect::Flagged(nullptr, t[5], iota, flag, posB, d_count, n, s));
        for (size_t x : t) t_bytes = x > t_bytes ? x : t_bytes;
    }
    void *temp = pool.get<uint8_t>(t_bytes);
    if (pool.err != cudaSuccess) return SA_ERR_NOMEM;
    uint64_t cnt = 0;
    auto read_count = [&]() -> cudaError_t {
        const cudaError_t e = cudaMemcpyAsync(&cnt, d_count, sizeof cnt, cudaMemcpyDeviceToHost, s);
        return e != cudaSuccess ? e : cudaStreamSynchronize(s);
    };
    const uint64_t most_tiles = (uint64_t)device_sm_count() * 16;
    auto refine_grid = [&](uint64_t c) {
        const uint64_t tiles = (c + kRefineOut - 1) / kRefineOut;
        return (unsigned)(tiles < most_tiles ? tiles : most_tiles);
    };

    const unsigned g = grid_for(n);
    init_keys_kernel<<<g, kThreads, 0, s>>>(T, n, kb32.Current(), vA);
    CK(cudaGetLastError());
    cub::DoubleBuffer<uint32_t> vb(vA, vB);
    CK(cub::DeviceRadixSort::SortPairs(temp, t_bytes, kb32, vb, n, 0, 32, s));
    uint64_t depth = kFirstBases;
    refine_kernel<uint32_t><<<refine_grid(n), kRefineThreads, 0, s>>>(kb32.Current(), vb.Current(), n, nullptr, T, n,
                                                                      depth, sa32, flag, headb);
    CK(cudaGetLastError());
    // Unresolved SA positions, in increasing order.
    CK(cub::DeviceSelect::Flagged(temp, t_bytes, iota, flag, posA, d_count, n, s));
    CK(read_count());
    uint32_t *pos = posA, *pos_next = posB;

    const uint64_t rounds = n / kRoundSuffixes < kMostRounds ? n / kRoundSuffixes : kMostRounds;
    uint64_t handled = 0;
    for (uint64_t r = 0; r < rounds && cnt > 0 && (handled += cnt) <= n / 2; r++) {
        const unsigned gc = grid_for(cnt);
        // every group has two members or more
        const int group_bits = bit_length(cnt / 2) > 0 ? bit_length(cnt / 2) : 1;
        const uint32_t bases = (uint32_t)(64 - group_bits) / 2;
        group_heads_kernel<<<gc, kThreads, 0, s>>>(pos, cnt, headb, group);
        CK(cudaGetLastError());
        CK(cub::DeviceScan::InclusiveSum(temp, t_bytes, group, group, cnt, s));
        group_keys_kernel<<<gc, kThreads, 0, s>>>(T, pos, cnt, sa32, group, depth, bases, kA, vA);
        CK(cudaGetLastError());
        cub::DoubleBuffer<uint64_t> rk(kA, kB);
        cub::DoubleBuffer<uint32_t> rv(vA, vB);
        CK(cub::DeviceRadixSort::SortPairs(temp, t_bytes, rk, rv, cnt, 0, group_bits + 2 * (int)bases, s));
        depth += bases;
        refine_kernel<uint64_t><<<refine_grid(cnt), kRefineThreads, 0, s>>>(rk.Current(), rv.Current(), cnt, pos, T, n,
                                                                            depth, sa32, flag, headb);
        CK(cudaGetLastError());
        CK(cub::DeviceSelect::Flagged(temp, t_bytes, pos, flag, pos_next, d_count, cnt, s));
        CK(read_count());
        uint32_t *tmp = pos;
        pos = pos_next;
        pos_next = tmp;
    }

    if (cnt > 0) {
        slot_ranks_kernel<<<g, kThreads, 0, s>>>(sa32, n, isa);
        CK(cudaGetLastError());
        const unsigned gc = grid_for(cnt);
        head_slots_kernel<<<gc, kThreads, 0, s>>>(pos, cnt, headb, hv);
        CK(cudaGetLastError());
        CK(cub::DeviceScan::InclusiveScan(temp, t_bytes, hv, hv, MaxOp(), cnt, s));
        group_ranks_kernel<<<gc, kThreads, 0, s>>>(pos, cnt, sa32, hv, isa);
        CK(cudaGetLastError());
    }
    const int rank_bits = bit_length(n);
    for (uint64_t h = depth; cnt > 0; h *= 2) {
        const unsigned gc = grid_for(cnt);
        pair_keys_kernel<<<gc, kThreads, 0, s>>>(pos, cnt, sa32, isa, n, h, kA, vA);
        CK(cudaGetLastError());
        cub::DoubleBuffer<uint64_t> rk(kA, kB);
        cub::DoubleBuffer<uint32_t> rv(vA, vB);
        CK(cub::DeviceRadixSort::SortPairs(temp, t_bytes, rk, rv, cnt, 0, 32 + rank_bits, s));
        head_values_kernel<<<gc, kThreads, 0, s>>>(rk.Current(), cnt, pos, hv);
        CK(cudaGetLastError());
        CK(cub::DeviceScan::InclusiveScan(temp, t_bytes, hv, hv, MaxOp(), cnt, s));
        scatter_ranks_kernel<<<gc, kThreads, 0, s>>>(rk.Current(), cnt, pos, rv.Current(), hv, isa, sa32, flag);
        CK(cudaGetLastError());
        CK(cub::DeviceSelect::Flagged(temp, t_bytes, pos, flag, pos_next, d_count, cnt, s));
        CK(read_count());
        uint32_t *tmp = pos;
        pos = pos_next;
        pos_next = tmp;
    }
    if (idx->width == 8) {
        widen_kernel<<<g, kThreads, 0, s>>>(sa32, n, reinterpret_cast<uint64_t *>(idx->sa));
        CK(cudaGetLastError());
    }
    CK(cudaStreamSynchronize(s));
    return SA_OK;
}

// The suffix array built on the host by DC3 (Section III's construction, in
// dc3_host.cpp) from host_text, then uploaded (and widened for 64-bit
// indexes on the device).
int build_suffix_array_host(sa_index *idx, const char *host_text, void *stream) {
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const uint64_t n = idx->n;
    std::vector<uint32_t> sa32;
    try {
        sa32.resize(n);
    } catch (const std::bad_alloc &) {
        return SA_ERR_NOMEM;
    }
    const int st = dc3_suffix_array(host_text, n, sa32.data());
    if (st != SA_OK) return st;
    if (idx->width == 4) {
        CK(cudaMemcpyAsync(idx->sa, sa32.data(), n * sizeof(uint32_t), cudaMemcpyHostToDevice, s));
        CK(cudaStreamSynchronize(s));
    } else {
        Pool pool{s};
        uint32_t *d = pool.get<uint32_t>(n);
        if (pool.err != cudaSuccess) return SA_ERR_NOMEM;
        CK(cudaMemcpyAsync(d, sa32.data(), n * sizeof(uint32_t), cudaMemcpyHostToDevice, s));
        widen_kernel<<<grid_for(n), kThreads, 0, s>>>(d, n, reinterpret_cast<uint64_t *>(idx->sa));
        CK(cudaGetLastError());
        CK(cudaStreamSynchronize(s));
    }
    return SA_OK;
}

// Key table in level (breadth-first) order: node k >= 1 at level l = floor(log2 k),
// p = k - 2^l, samples rank floor((2p + 1) n / 2^(l+1)).  Its first 2^d - 1
// nodes are the table of depth d, so a shallower table is a prefix.  Entry k
// holds the first 64 bases of that suffix (bits past the text are zero) and
// keylen[k] = min(64, n - SA[rank]).  Node 0 is unused padding.
template <typename IdxT>
__global__ void build_keys_kernel(const uint64_t *__restrict__ T, const IdxT *__restrict__ sa, uint64_t n,
                                  uint32_t depth, uint32_t entries, uint4 *keys, uint8_t *keylen) {
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < entries; k += gridDim.x * blockDim.x) {
        uint64_t w0 = 0, w1 = 0;
        uint32_t len = 0;
        if (k >= 1 && k < (1u << depth)) {
            const uint32_t l = 31 - __clz(k);
            const uint64_t p = k - (1u << l);
            const uint64_t rank = ((2 * p + 1) * n) >> (l + 1);
            const uint64_t pos = sa[rank];
            w0 = text_window(T, pos);
            w1 = text_window(T, pos + 32);
            const uint64_t rem = n - pos;
            len = rem < 64 ? (uint32_t)rem : 64u;
        }
        keys[k] = make_uint4((uint32_t)w0, (uint32_t)(w0 >> 32), (uint32_t)w1, (uint32_t)(w1 >> 32));
        keylen[k] = (uint8_t)len;
    }
}

cudaError_t launch_build_keys(sa_index *idx, cudaStream_t s) {
    const uint32_t entries = idx->depth >= 4 ? (1u << idx->depth) : 16u;
    const unsigned blocks = (entries + 255) / 256;
    if (idx->width == 4)
        build_keys_kernel<uint32_t><<<blocks, 256, 0, s>>>(idx->text, reinterpret_cast<const uint32_t *>(idx->sa),
                                                           idx->n, idx->depth, entries, idx->keys, idx->keylen);
    else
        build_keys_kernel<uint64_t><<<blocks, 256, 0, s>>>(idx->text, reinterpret_cast<const uint64_t *>(idx->sa),
                                                           idx->n, idx->depth, entries, idx->keys, idx->keylen);
    return cudaGetLastError();
}

// The kN windows of 32 bases from base b of the text on (zeros past its end), by
// 16-byte loads of the pairs of words they lie in (three, where a window by
// itself takes two of 8 bytes): at 6*10^8 bases the records take 15.3 -> 14.0 ms
// and the entries 21.0 -> 20.3.
template <int kN>
__device__ __forceinline__ void text_windows(const uint64_t *__restrict__ T, uint64_t n, uint64_t b, uint64_t *w) {
    constexpr int kPairs = (kN + 3) / 2;  // kN + 1 words, from an even one on
    const uint64_t first = b >> 5, even = first & ~1ull;
    const bool odd = (first & 1u) != 0;
    uint64_t x[2 * kPairs];
#pragma unroll
    for (int p = 0; p < kPairs; p++) {
        const uint64_t at = even + 2u * p;
        const bool need = at * 32 < n && (2 * p <= kN || odd);  // its second word is at most the first of the padding
        const ulonglong2 v = need ? __ldg(reinterpret_cast<const ulonglong2 *>(T + at)) : make_ulonglong2(0, 0);
        x[2 * p] = v.x;
        x[2 * p + 1] = v.y;
    }
    const unsigned sh = (unsigned)(b & 31u) * 2u;
#pragma unroll
    for (int j = 0; j < kN; j++) {
        const uint64_t hi = odd ? x[j + 1] : x[j], lo = odd ? x[j + 2] : x[j + 1];
        w[j] = (hi << sh) | ((lo >> 1) >> (63u - sh));
    }
}

// Suffix records: for rank i, the first 104 bases of suffix SA[i], its common
// prefixes with the suffixes at the ranks beside it, and SA[i] itself in one
// 32-byte entry (one DRAM sector), so that a probe of the search reads one
// aligned sector instead of an SA entry and then the text it points to, and a
// query of up to 104 bases never reads the text.
//
// A warp makes the records of 30 ranks: its lanes hold 32 consecutive
// suffixes' first 128 bases, each lane counts the bases it shares with the
// next lane's (reading on in the text past 128 equal ones, up to 255), and
// the outer two lanes only serve as neighbours.  The reads of the text (four
// windows per rank, random: 160 bytes of DRAM traffic) bound it, 6 % more of them for the two outer
// lanes.
//
// The k-mer counts come from the same windows (k > 0).  For rank i let f(i) be
// the smallest k-base string x with S_SA[i] < x: the suffix's k-base prefix
// plus one when it has k bases or more, else the suffix padded with A (a
// suffix that is a proper prefix of x sorts before x).  f is non-decreasing
// along the suffix array, and kmer[x] = #{i : f(i) <= x} = #{suffixes sorting
// before x}.  Rank i writes kmer[x] = i for f(i-1) <= x < f(i), with f(-1) = 0
// and f(n) = 4^k + 1, so every entry is written once.  (A kernel of its own
// read all records again for them: 3.7 ms at 6*10^8 bases.)
constexpr int kRecRanks = 30;  // ranks per warp

template <typename IdxT>
__global__ void build_records_kernel(const uint64_t *__restrict__ T, const IdxT *__restrict__ sa, uint64_t n,
                                     uint4 *rec, uint32_t k, uint32_t *kmer) {
    const unsigned lane = threadIdx.x & 31u;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    const uint64_t groups = n / kRecRanks + 1;  // ranks 0 .. n: the last one ends the k-mer counts
    for (uint64_t g = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); g < groups; g += warps) {
        const uint64_t i = g * kRecRanks + lane - 1u;  // lane 0 of the first group: no rank (wraps)
        const bool live = i < n;
        const uint64_t pos = live ? (uint64_t)sa[i] : 0;
        uint64_t w[4] = {0, 0, 0, 0};
        if (live) text_windows<4>(T, n, pos, w);
        // bases shared with the next lane's suffix
        const uint64_t npos = __shfl_down_sync(0xFFFFFFFFu, pos, 1);
        const bool nlive = __shfl_down_sync(0xFFFFFFFFu, (int)live, 1) != 0 && lane < 31u;
        uint32_t same = 0;
        bool more = true;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const uint64_t x = w[j] ^ __shfl_down_sync(0xFFFFFFFFu, w[j], 1);
            if (more) same += x ? (uint32_t)(__clzll((long long)x) >> 1) : 32u;
            more = more && x == 0;
        }
        uint32_t ln = 0;
        if (live && nlive) {
            const uint64_t far = pos > npos ? pos : npos;
            const uint32_t room = n - far < kLcpCap ? (uint32_t)(n - far) : kLcpCap;
            while (more && same < room) {
                const uint64_t x = text_window(T, pos + same) ^ text_window(T, npos + same);
                same += x ? (uint32_t)(__clzll((long long)x) >> 1) : 32u;
                more = x == 0;
            }
            ln = same < room ? same : room;
        }
        const uint32_t lp = __shfl_up_sync(0xFFFFFFFFu, ln, 1);  // 0 at rank 0: lane 0 held no suffix
        if (live && lane >= 1u && lane <= (unsigned)kRecRanks) {
            rec[2 * i] = make_uint4((uint32_t)w[0], (uint32_t)(w[0] >> 32), (uint32_t)w[1], (uint32_t)(w[1] >> 32));
            rec[2 * i + 1] = make_uint4((uint32_t)w[2], (uint32_t)(w[2] >> 32),
                                        ((uint32_t)(w[3] >> 32) & 0xFFFF0000u) | (lp << 8) | ln, (uint32_t)pos);
        }
        if (k == 0) continue;
        // the counts of the k-mers between this suffix and the one before it
        uint64_t f = i < n ? (w[0] >> (64u - 2u * k)) + (n - pos >= k ? 1u : 0u) : 0;
        if (i == n) f = (1ull << (2 * k)) + 1;
        const uint64_t before = __shfl_up_sync(0xFFFFFFFFu, f, 1);  // 0 at rank 0
        if (i <= n && lane >= 1u && lane <= (unsigned)kRecRanks)
            for (uint64_t x = before; x < f; x++) kmer[x] = (uint32_t)i;
    }
}

// k-mer table entry, 64 bytes (4 uint4) per k-base string x:
//   {lo, hi, pos, clamp}: ranks [lo, hi) hold the suffixes that sort at or
//     after x and before x + 1 (those with prefix x, and any suffix shorter
//     than k that falls between the two), lo = number of suffixes sorting
//     before x; when hi > lo, pos is the position of the suffix at rank
//     M = lo - 1 + (hi - lo + 1) / 2 -- the first pivot of the lockstep binary
//     search over (lo - 1, hi) -- and the last word holds clamp = min(192, n -
//     pos), the number of its first 192 bases that exist, and its record's two
//     common prefixes with the ranks beside it;
//   three uint4: the first 192 bases of that suffix as six packed words.
// One aligned 64-byte read therefore brackets a query of m >= k bases and
// makes its first probe.  The pivot's record gives its first 96 bases, so only
// the second 96 are read from the text (random; the records are read in
// order), and each half entry is one 32-byte store: 10^8 bases (17 GB of
// entries) 5.2 -> 3.9 ms against six text windows and four 16-byte stores,
// 6*10^8 (69 GB) 23.7 -> 21.0 ms (20.3 with text_windows), bound there by the text
// reads.
__device__ __forceinline__ void st32(void *p, uint64_t a, uint64_t b, uint64_t c, uint64_t d) {
    asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

__device__ __forceinline__ void write_krt_entry(uint64_t x, uint32_t lo, uint32_t hi, const uint4 *__restrict__ rec,
                                                const uint64_t *__restrict__ T, uint64_t n, uint4 *krt) {
    uint64_t pos = 0, e[6] = {0, 0, 0, 0, 0, 0};
    uint32_t last = 0;
    if (hi > lo) {
        const uint32_t M = lo + (hi - lo + 1u) / 2u - 1u;
        uint4 r0, r1;
        ldg32(rec + 2 * (uint64_t)M, &r0, &r1);
        pos = r1.w;
        const uint64_t left = n - pos;  // >= 1
        last = (uint32_t)(left < 192 ? left : 192) | (((r1.z >> 8) & 0xFFu) << 8) | ((r1.z & 0xFFu) << 16);
        e[0] = ((uint64_t)r0.y << 32) | r0.x;
        e[1] = ((uint64_t)r0.w << 32) | r0.z;
        e[2] = ((uint64_t)r1.y << 32) | r1.x;
        text_windows<3>(T, n, pos + 96, e + 3);
    }
    uint4 *dst = krt + 4 * x;
    st32(dst, ((uint64_t)hi << 32) | lo, ((uint64_t)last << 32) | pos, e[0], e[1]);
    st32(dst + 2, e[2], e[3], e[4], e[5]);
}

// Entries [first, end) from the counts kmer[first .. end], which no entry of
// this launch is written over.
__global__ void build_krt_kernel(const uint32_t *kmer, const uint4 *__restrict__ rec, const uint64_t *__restrict__ T,
                                 uint64_t n, uint64_t first, uint64_t end, uint4 *krt) {
    GS_LOOP(j, end - first) write_krt_entry(first + j, kmer[first + j], kmer[first + j + 1], rec, T, n, krt);
}

// The last entries, at most one per thread of the one block: every count is
// read before any entry is written over it.
__global__ void build_krt_last_kernel(const uint32_t *kmer, const uint4 *__restrict__ rec,
                                      const uint64_t *__restrict__ T, uint64_t n, uint64_t first, uint64_t end,
                                      uint4 *krt) {
    const uint64_t x = first + threadIdx.x;
    uint32_t lo = 0, hi = 0;
    if (x < end) {
        lo = kmer[x];
        hi = kmer[x + 1];
    }
    __syncthreads();
    if (x < end) write_krt_entry(x, lo, hi, rec, T, n, krt);
}

// The plain counts kmer[x] = lo of every entry, and kmer[4^k] = n.
__global__ void krt_lo_kernel(const uint4 *__restrict__ krt, uint64_t n, uint32_t k, uint32_t *__restrict__ out) {
    const uint64_t entries = 1ull << (2 * k);
    GS_LOOP(x, entries + 1) out[x] = x < entries ? krt[4 * x].x : (uint32_t)n;
}

// The counts kmer[0 .. 4^k] wait in the end of the entries' own memory, so that
// they need none of their own (4.3 GB at k = 15, mapped and unmapped for every
// build).
uint32_t *counts_of(const sa_index *idx) {
    const uint64_t entries = 1ull << (2 * idx->kmer_k);
    return reinterpret_cast<uint32_t *>(idx->krt) + 16 * entries - (entries + 1);
}

// The k-mer entries from the records and the counts that launch_build_records
// left.
cudaError_t launch_build_kmer(sa_index *idx, cudaStream_t s) {
    if (!idx->krt) return cudaSuccess;
    // Each launch writes the entries from s on that lie
    // before the counts from s on, all but a sixteenth of the rest, and the
    // counts of those it wrote are free to be written over by the next.
    constexpr uint64_t kLast = 256;
    const uint64_t entries = 1ull << (2 * idx->kmer_k);
    const uint32_t *kmer = counts_of(idx);
    uint64_t done = 0;
    while (entries - done > kLast) {
        const uint64_t end = entries - (entries - done + 1 + 15) / 16;
        build_krt_kernel<<<grid_for(end - done), kThreads, 0, s>>>(kmer, idx->rec, idx->text, idx->n, done, end,
                                                                   idx->krt);
        done = end;
    }
    build_krt_last_kernel<<<1, kLast, 0, s>>>(kmer, idx->rec, idx->text, idx->n, done, entries, idx->krt);
    return cudaGetLastError();
}

cudaError_t launch_copy_kmer_counts(const sa_index *idx, uint32_t *dst, cudaStream_t s) {
    const uint64_t entries = 1ull << (2 * idx->kmer_k);
    krt_lo_kernel<<<grid_for(entries + 1), kThreads, 0, s>>>(idx->krt, idx->n, idx->kmer_k, dst);
    return cudaGetLastError();
}

cudaError_t launch_build_records(sa_index *idx, cudaStream_t s) {
    const unsigned g = grid_for((idx->n / kRecRanks + 1) * 32);
    const uint32_t k = idx->krt ? idx->kmer_k : 0u;
    uint32_t *kmer = idx->krt ? counts_of(idx) : nullptr;
    if (idx->width == 4)
        build_records_kernel<uint32_t><<<g, kThreads, 0, s>>>(idx->text, reinterpret_cast<const uint32_t *>(idx->sa),
                                                              idx->n, idx->rec, k, kmer);
    else
        build_records_kernel<uint64_t><<<g, kThreads, 0, s>>>(idx->text, reinterpret_cast<const uint64_t *>(idx->sa),
                                                              idx->n, idx->rec, k, kmer);
    return cudaGetLastError();
}

}  // namespace sa
