// first_pass.cuh -- what the kernels that bracket a query by its k-mer entry
// share: front.cu (large batches) and small.cu (small ones).
#pragma once

#include "sa_internal.cuh"

namespace sa {

struct FrontDesc {
    const uint64_t *text;
    const uint4 *rec;
    const uint4 *krt;
    uint64_t tail;  // the text's last 32 bases (all, when it has fewer), the last in the low bits
    uint32_t n;
    uint32_t kmer_k;
};

__device__ __forceinline__ FrontDesc front_desc(const RefDesc &d) {
    const uint64_t tail = d.n >= 32 ? text_window(d.text, d.n - 32) : ldg_u64(d.text) >> (64u - 2u * (uint32_t)d.n);
    return FrontDesc{d.text, d.rec, d.krt, tail, (uint32_t)d.n, d.kmer_k};
}

// How many suffixes shorter than k equal the string q (qlen bases, as a
// number) followed by some A's.
__device__ __forceinline__ uint32_t short_suffixes(uint64_t tail, uint32_t n, uint32_t k, uint64_t q, uint32_t qlen) {
    uint32_t c = 0;
    for (uint32_t len = qlen; len < k && len <= n; len++)
        c += (tail & ((1ull << (2u * len)) - 1ull)) == (q << (2u * (len - qlen))) ? 1u : 0u;
    return c;
}

// The interval of a query of 1 <= m < k bases (p as a number), from the counts
// of two k-mer entries: kmer[x] is the number of suffixes that sort before the
// k-base string x.  P's first suffix comes before P A..A only as P, P A, P AA,
// ... at the text's end, so lo = kmer[P A..A] less those of them that are
// suffixes.  P's successor p + 1 is Q followed by A's, Q ending in the base
// that was raised; of the suffixes before (p + 1) A..A only Q, Q A, ... do not
// start with P or sort before it.  Two reads of random entries per query; the
// descent of a key table and the binary search below it took about 2 log2 of
// the count more (2*10^6 queries of 8-31 bases at 100 Mbp: 594 -> 375 us a
// call).
__device__ __forceinline__ void brief_interval(const FrontDesc &d, uint64_t p, uint32_t m, uint32_t *lo, uint32_t *hi) {
    const uint32_t k = d.kmer_k, up = 2u * (k - m);
    const uint64_t next = p + 1;
    const bool last = next == 1ull << (2u * m);  // P is T..T: no successor, every suffix from lo on
    const uint32_t klo = __ldg(reinterpret_cast<const uint32_t *>(d.krt + 4 * (p << up)));
    const uint32_t khi = last ? d.n : __ldg(reinterpret_cast<const uint32_t *>(d.krt + 4 * (next << up)));
    const uint32_t raised = ((uint32_t)__ffsll((long long)next) - 1u) >> 1;  // trailing A's of p + 1
    *lo = klo - short_suffixes(d.tail, d.n, k, p, m);
    *hi = last ? d.n : khi - short_suffixes(d.tail, d.n, k, next >> (2u * raised), m - raised);
}

// P (bases 0-127 in w, the rest from qw; length m >= 1) against the pivot of
// a k-mer entry: its first 192 bases in e (clamp of them exist), then the
// text from position pos + 192 when all 192 tie.
template <typename Windows>
__device__ __forceinline__ int cmp_entry(const uint64_t w[4], uint32_t m, const uint64_t e[6], uint32_t pos,
                                         uint32_t clamp, uint32_t n, const uint64_t *__restrict__ T,
                                         const Windows &qw, uint32_t *lcp) {
    bool undecided = false;
    int c = cmp_first(w, e, m, 128u, clamp, lcp, &undecided);
    if (!undecided) return c;
#pragma unroll
    for (uint32_t off = 128u; off < 192u; off += 32u) {
        c = cmp_window(qw(off), e[off / 32u], min(32u, m - off), clamp > off ? min(32u, clamp - off) : 0u, off, m, lcp);
        if (c != 2) return c;
    }
    return cmp_suffix_qw(T, n, pos, qw, m, 192u, lcp);
}

// The source of a record's query's windows, by where the kernel reads bases.
template <Bases kBases>
__device__ __forceinline__ auto window_source(const SearchLaunch &a, uint64_t at, uint32_t m) {
    if constexpr (kBases == Bases::Ascii)
        return AsciiWindows{reinterpret_cast<const uint8_t *>(a.ascii), a.total, place_first(at, m), m,
                            (at & kPlaceRc) != 0};
    else
        return PackedWindows<kBases == Bases::PackedStrands>{a.tq, at};
}

// Word w of the batch (bases 32 w .. 32 w + 31) where it is not full or not
// aligned.
__device__ __forceinline__ uint64_t pack_edge_word(const uint8_t *__restrict__ ascii, uint64_t total, uint64_t w,
                                                   uint32_t *bad) {
    const uint64_t b0 = w * 32;
    return pack_word(ascii, total, b0, total - b0 < 32 ? (uint32_t)(total - b0) : 32u, bad);
}

// Whether bytes [qa, qa + m) of the batch (m >= 1) are all bases, given the
// tile's bits of words that hold a byte that is not (bit i of marks[i / 32]:
// word w_lo + i, all of the query's words among them); the few marked words'
// bytes are looked at again.
__device__ __forceinline__ bool tile_valid(const uint32_t *marks, uint64_t w_lo, const uint8_t *__restrict__ ascii,
                                           uint64_t qa, uint32_t m) {
    const uint32_t w0 = (uint32_t)((qa >> 5) - w_lo), w1 = (uint32_t)(((qa + m - 1) >> 5) - w_lo);
    for (uint32_t g = w0 >> 5; g <= (w1 >> 5); g++) {
        uint32_t marked = marks[g];
        if (g == (w0 >> 5)) marked &= 0xFFFFFFFFu << (w0 & 31u);
        if (g == (w1 >> 5)) marked &= 0xFFFFFFFFu >> (31u - (w1 & 31u));
        for (; marked != 0u; marked &= marked - 1u) {
            const uint64_t b0 = (w_lo + g * 32u + (uint32_t)(__ffs(marked) - 1)) * 32;
            if (!bytes_valid(ascii, b0 > qa ? b0 : qa, b0 + 32 < qa + m ? b0 + 32 : qa + m)) return false;
        }
    }
    return true;
}

}  // namespace sa
