// sa_internal.cuh -- layouts and device helpers shared by the libsa kernels.
//
// Packed text layout (Section III alphabet, order A < C < G < T):
//   base b of a sequence lives in 64-bit word b / 32 at bits
//   [63 - 2*(b % 32), 62 - 2*(b % 32)], codes A=0 C=1 G=2 T=3.  Big-endian
//   placement makes unsigned integer comparison of two aligned windows equal
//   to lexicographic comparison of their bases.  Bits past the end are zero
//   and every packed text carries SA_PAD_WORDS zero words after its last
//   word, so a 32-base window starting at any base < n reads in bounds.
//
// Packed query batch: the bases of a whole batch (q_offsets[0] ..
// q_offsets[n_q]) packed like a text, 32 per word, with SA_TQ_PAD_WORDS zero
// words after the last and room for SA_TQ_LEAD_WORDS words of no meaning
// before the first.  Query q's bases start at base q_offsets[q] -
// q_offsets[0], so any of its 32-base windows is one window read; a window of
// its reverse complement is the window ending there, complemented and put in
// reverse order (QueryWindow helpers below), so one packing serves both
// strands.  A bitmap has bit w % 32 of word w / 32 set when packed word w
// holds a byte that is not in {A,C,G,T,a,c,g,t}, and only those words have a
// 32-bit mask, whose bit i marks base 32 w + i.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/sa.h"

#define SA_PAD_WORDS 2
#define SA_TQ_PAD_WORDS 6
#define SA_TQ_LEAD_WORDS 6
#define SA_MAX_REFS 64
#define SA_MAX_KEY_DEPTH 14

namespace sa {

// Device view of one index, passed to the kernels.
struct RefDesc {
    const uint64_t *text;   // packed text, nwords + SA_PAD_WORDS words
    const void *sa;         // n entries of width 4 or 8
    const uint4 *keys;      // 2^depth key entries: 64 bases as two words (x,y = w0; z,w = w1)
    const uint8_t *keylen;  // 2^depth clamp lengths min(64, n - SA[rank])
    const uint4 *rec;       // 2n uint4: n 32-byte suffix records, see sa_index::rec
    const uint4 *krt;       // 4^kmer_k 64-byte k-mer entries, see sa_index::krt (null: none)
    uint64_t n;
    uint32_t depth;         // key-table depth d of this index; K = 2^d - 1 samples
    uint32_t smem_off;      // byte offset of this table in the search kernel's shared memory
    uint32_t use_depth;     // depth the search uses (<= depth); 0 = no table
    uint32_t kmer_k;        // k of the k-mer table (0: none)
    uint64_t kbase;         // k-mer entries of the earlier indexes of the call (k-mer order buckets)
};

// k-mer order of a batch (bucket.cu): the slices of the k-mer entries of a
// call's indexes, plus one bucket for queries without a k-mer bracket.
constexpr uint32_t kNumBuckets = 256;
// The k-mer-ordered list's 64-byte records (bucket.cu writes, front.cu reads):
//   {m, q, at.lo, at.hi | ref << 16 | strand | kListNeedsEntry}  length, index,
//       place in the packed batch (at < 2^48, and kRecordRc for the other
//       strand), reference id (< 2^14), and whether the query has a k-mer
//       bracket to read
//   {w0, w1}, {w2, w3}, {w4, w5}  its first 192 bases as packed words (the
//       words past the query's end are not its bases)
constexpr uint32_t kListNeedsEntry = 0x80000000u;
constexpr uint32_t kRecordRc = 0x40000000u;  // in list and worklist records
constexpr uint64_t kListMaxBase = 1ull << 48;
// The list's plan (bucket.cu), 32-bit words: every kListSampleStride-th
// query's bucket counted; from those counts each bucket's region of the list
// (start, capacity) and a cursor; after the scatter, the exclusive prefix
// sums of the regions' fills (kNumBuckets + 2 words, the last the sum); and
// the overflow region that takes what does not fit a bucket's region.
constexpr uint32_t kListSampleStride = 32;
constexpr uint32_t kPlanSample = 0;
constexpr uint32_t kPlanStart = kPlanSample + kNumBuckets + 1;
constexpr uint32_t kPlanCap = kPlanStart + kNumBuckets + 1;
constexpr uint32_t kPlanCursor = kPlanCap + kNumBuckets + 1;
constexpr uint32_t kPlanPrefix = kPlanCursor + kNumBuckets + 1;
constexpr uint32_t kPlanOvStart = kPlanPrefix + kNumBuckets + 2;
constexpr uint32_t kPlanOvCursor = kPlanOvStart + 1;
constexpr uint32_t kPlanWords = kPlanOvCursor + 1;
// Records the list needs room for, at most: every bucket's region (the sample
// counts scaled up by 9/8, plus 256) and an overflow region for every query.
__host__ __device__ constexpr uint64_t list_capacity(uint64_t n_q) {
    return (n_q + kListSampleStride) * 9 / 8 + 256ull * (kNumBuckets + 1) + n_q;
}

// Queries per tile of the k-mer order's scatter (bucket.cu).
constexpr uint32_t kScatterTile = 512;
__host__ __device__ constexpr uint64_t scatter_tiles(uint64_t n_q) { return (n_q + kScatterTile - 1) / kScatterTile; }

// The compare outcome of the three cases of Section IV.
enum : int { CMP_LESS = -1, CMP_PREFIX = 0, CMP_GREATER = 1 };

__device__ __forceinline__ uint64_t ldg_u64(const uint64_t *p) { return __ldg(p); }

// 32 bases of the packed text starting at base position b (b < n + 32).
__device__ __forceinline__ uint64_t text_window(const uint64_t *__restrict__ T, uint64_t b) {
    const uint64_t w = b >> 5;
    const unsigned sh = (unsigned)(b & 31u) * 2u;
    const uint64_t a = ldg_u64(T + w);
    const uint64_t c = ldg_u64(T + w + 1);
    // (c >> 1) >> (63 - sh) is c >> (64 - sh) for sh > 0 and 0 for sh == 0.
    return (a << sh) | ((c >> 1) >> (63u - sh));
}

// Base code of an ASCII byte; returns 4 for a byte outside {ACGTacgt}.
__device__ __forceinline__ uint32_t base_code(uint32_t c) {
    const uint32_t u = c & 0xDFu;  // fold lower case
    const uint32_t x = (u >> 1) & 3u;  // A:0 C:1 G:3 T:2
    const uint32_t code = x ^ (x >> 1);  // A:0 C:1 G:2 T:3
    const bool ok = (u == 'A') | (u == 'C') | (u == 'G') | (u == 'T');
    return ok ? code : 4u;
}

// Marks a query that cannot be searched (a byte that is not a base,
// inconsistent offsets or an out-of-range reference id).
constexpr uint32_t kQueryInvalid = 0xFFFFFFFFu;

// Four ASCII bytes (little-endian in v) to four 2-bit codes in the low byte,
// first base in the top two bits.  Per byte, with u the case-folded byte:
// x = (u >> 1) & 3 is A0 C1 G3 T2 and c = x ^ (x >> 1) is A0 C1 G2 T3.  The
// codes sit at bits 0, 8, 16, 24; one multiply by 2^30 + 2^20 + 2^10 + 1
// moves them to bits 30, 28, 26, 24 without carries between the partial
// products.  The check rebuilds each letter from its code, 'A' + 2c + 2h +
// 11 (c & h) with h = c >> 1 (giving A, C, G, T for c = 0..3), and ORs any
// difference from u into *bad.
__device__ __forceinline__ uint32_t pack4_fast(uint32_t v, uint32_t *bad) {
    const uint32_t u = v & 0xDFDFDFDFu;
    const uint32_t x = (u >> 1) & 0x03030303u;
    const uint32_t h0 = (x >> 1) & 0x01010101u;
    const uint32_t c = x ^ h0;                     // per byte: A0 C1 G2 T3
    const uint32_t h = (c >> 1) & 0x01010101u;
    const uint32_t expect = 0x41414141u + 2u * c + 2u * h + 11u * (c & h);
    *bad |= u ^ expect;
    return (c * 0x40100401u) >> 24;
}

// A 32-base word from its 32 bytes; *bad becomes non-zero if one of them is not
// a base.  Bits 2-1 of a letter are A 00, C 01, G 11, T 10: four of them are
// put together by one multiply, and one x ^ (x >> 1) per word makes the codes.
// Of a base's other bits (case folded) 7 and 3 are clear, 6 is set, 4 is set
// exactly where bits 2-1 are 10 (T), and 0 is the opposite of 4; those are
// collected over the 32 bytes and looked at once.  The kernels that pack are
// bound by the integer pipe, so what can be a left shift is one (a multiply,
// on the other pipe): about 55 logic instructions per word, where pack4_fast
// on each four bytes takes 120.
__device__ __forceinline__ uint64_t pack32(uint4 v0, uint4 v1, uint32_t *bad) {
    const uint32_t v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
    uint32_t p[8], wrong = 0, any = 0, all = 0xFFFFFFFFu;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const uint32_t t = v[k] & ~(v[k] * 2u) & 0x04040404u;       // bit 2 of each byte: bits 2-1 are 10
        wrong |= (v[k] ^ (t * 4u)) | ~(v[k] ^ (v[k] * 16u));         // at bit 4
        any |= v[k];
        all &= v[k];
        p[k] = ((v[k] >> 1) & 0x03030303u) * 0x40100401u;           // the four pairs in its top byte
    }
    *bad |= (wrong & 0x10101010u) | (any & 0x88888888u) | (~all & 0x40404040u);
    const uint32_t hi = __byte_perm(__byte_perm(p[3], p[2], 0x0073), __byte_perm(p[1], p[0], 0x0073), 0x5410);
    const uint32_t lo = __byte_perm(__byte_perm(p[7], p[6], 0x0073), __byte_perm(p[5], p[4], 0x0073), 0x5410);
    const uint64_t x = ((uint64_t)hi << 32) | lo;
    return x ^ ((x >> 1) & 0x5555555555555555ull);
}

// Non-zero when one of 16 bytes is not a base (the check of pack32 alone).
__device__ __forceinline__ uint32_t not_bases(uint4 x) {
    const uint32_t v[4] = {x.x, x.y, x.z, x.w};
    uint32_t wrong = 0, any = 0, all = 0xFFFFFFFFu;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const uint32_t t = v[k] & ~(v[k] * 2u) & 0x04040404u;
        wrong |= (v[k] ^ (t * 4u)) | ~(v[k] ^ (v[k] * 16u));
        any |= v[k];
        all &= v[k];
    }
    return (wrong & 0x10101010u) | (any & 0x88888888u) | (~all & 0x40404040u);
}

// Packs the 32 ASCII bases starting at byte s of a (the first nb <= 32 belong
// to the query; the rest pack as A).  When nine aligned 32-bit words around
// them lie inside [a, a + total) they are read and aligned with funnel
// shifts; the check covers only the query's own nb bytes.  Otherwise (the
// batch's last bytes) the bytes are read one at a time.  Returns the word;
// *bad becomes non-zero if one of the nb bytes is not a base.
__device__ __forceinline__ uint64_t pack_word(const uint8_t *__restrict__ a, uint64_t total, uint64_t s,
                                              uint32_t nb, uint32_t *bad) {
    const uintptr_t lo_addr = ((uintptr_t)(a + s)) & ~(uintptr_t)3;
    uint64_t word = 0;
    if (lo_addr >= (uintptr_t)a && lo_addr + 36 <= (uintptr_t)(a + total)) {
        const uint32_t *p = reinterpret_cast<const uint32_t *>(lo_addr);
        const uint32_t sh = (uint32_t)(((uintptr_t)(a + s)) & 3u) * 8u;
        uint32_t v[9];
#pragma unroll
        for (int i = 0; i < 9; i++) v[i] = __ldg(p + i);
        uint32_t hi = 0, lo = 0, b = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            uint32_t gb = 0;
            const uint32_t g = pack4_fast(__funnelshift_r(v[i], v[i + 1], sh), &gb);
            const int own = (int)nb - 4 * i;  // bytes of this group that belong to the query
            b |= own >= 4 ? gb : (own > 0 ? gb & ((1u << (8 * own)) - 1u) : 0u);
            if (i < 4)
                hi = (hi << 8) | g;
            else
                lo = (lo << 8) | g;
        }
        *bad |= b;
        word = ((uint64_t)hi << 32) | lo;
        if (nb < 32) word &= ~0ull << (64u - 2u * nb);
    } else {
        for (uint32_t j = 0; j < 32; j++) {
            uint32_t code = 0;
            if (j < nb) {
                code = base_code(a[s + j]);
                if (code > 3) {
                    *bad |= 1u;
                    code = 0;
                }
            }
            word = (word << 2) | code;
        }
    }
    return word;
}

// q_ref bit 31 under SA_PARAM_STRAND_PER_QUERY: search the query's reverse complement.
constexpr uint32_t kStrandBit = 0x80000000u;

// A query's place in the packed batch: its first base, or for the other
// strand one past its last base with kPlaceRc set (base i of the reverse
// complement is the complement of base end - 1 - i).
constexpr uint64_t kPlaceRc = 1ull << 63;

__device__ __forceinline__ uint64_t query_place(uint64_t qa, uint64_t qe, bool rc) { return rc ? qe | kPlaceRc : qa; }

// The first base in the packed batch of a query of m bases at place at.
__device__ __forceinline__ uint64_t place_first(uint64_t at, uint32_t m) {
    return (at & kPlaceRc) ? (at & ~kPlaceRc) - m : at;
}

// The place's halves as list and worklist records hold them, with the reference.
__device__ __forceinline__ uint32_t place_high(uint64_t at, uint32_t ref) {
    return (uint32_t)((at & ~kPlaceRc) >> 32) | (ref << 16) | ((at & kPlaceRc) ? kRecordRc : 0u);
}
__device__ __forceinline__ uint64_t place_of(uint32_t lo, uint32_t hi) {
    return ((uint64_t)(hi & 0xFFFFu) << 32) | lo | ((hi & kRecordRc) ? kPlaceRc : 0ull);
}
__device__ __forceinline__ uint32_t ref_of(uint32_t hi) { return (hi >> 16) & 0x3FFFu; }

// The reverse complement of a window of 32 bases: every bit flipped and the
// bits reversed, then the two bits of each code swapped back.
__device__ __forceinline__ uint64_t rc_window(uint64_t x) {
    const uint64_t f = __brevll(~x);
    return ((f >> 1) & 0x5555555555555555ull) | ((f & 0x5555555555555555ull) << 1);
}

// The N 32-base windows of a query at bases off, off + 32, ... (N + 1 words
// read; bits past the query are not its bases).  The other strand's windows
// end at the query's place and may begin up to 31 + 32 (N - 1) bases before
// the query, in the words before it (or the batch's lead words).  kStrands:
// some query of the call may be of the other strand; a call of forward
// queries only runs kernels without that branch (with it, 1571 -> 1668 us a
// call of 1.6*10^7 queries over four genomes, 775 -> 819 us of 2^20 1024-base
// ones).
template <int N, bool kStrands>
__device__ __forceinline__ void query_windows(const uint64_t *__restrict__ tq, uint64_t at, uint32_t off,
                                              uint64_t w[N]) {
    const bool rc = kStrands && (at & kPlaceRc) != 0;
    const int64_t b = rc ? (int64_t)(at & ~kPlaceRc) - (int64_t)off - 32 * N : (int64_t)at + off;
    const uint64_t *p = tq + (b >> 5);
    const unsigned sh = (unsigned)(b & 31) * 2u;
    uint64_t t[N + 1];
#pragma unroll
    for (int i = 0; i <= N; i++) t[i] = ldg_u64(p + i);
#pragma unroll
    for (int j = 0; j < N; j++) w[j] = (t[j] << sh) | ((t[j + 1] >> 1) >> (63u - sh));
    if (rc) {
#pragma unroll
        for (int j = 0; j < (N + 1) / 2; j++) {
            const uint64_t x = rc_window(w[j]), y = rc_window(w[N - 1 - j]);
            w[j] = y;
            w[N - 1 - j] = x;
        }
    }
}

template <bool kStrands>
__device__ __forceinline__ uint64_t query_window(const uint64_t *__restrict__ tq, uint64_t at, uint32_t off) {
    uint64_t w[1];
    query_windows<1, kStrands>(tq, at, off, w);
    return w[0];
}

// Bits [lo, hi) of a 32-bit mask (0 <= lo <= hi <= 32).
__device__ __forceinline__ uint32_t bit_range(uint32_t lo, uint32_t hi) {
    const uint32_t upto = hi >= 32u ? 0xFFFFFFFFu : ((1u << hi) - 1u);
    return upto & ~((1u << lo) - 1u);
}

// Whether byte range [lo, hi) of the batch, within one of its words, is all bases.
__device__ __forceinline__ bool bytes_valid(const uint8_t *__restrict__ ascii, uint64_t lo, uint64_t hi) {
    for (uint64_t b = lo; b < hi; b++)
        if (base_code(__ldg(ascii + b)) > 3u) return false;
    return true;
}

// Whether all m >= 1 bases from base qa of the batch on are bases: the bits of
// their words in the bitmap tvb (one or two of its words for a query of up to
// 1024 bases), then the masks tv of the few words that are marked.
__device__ __forceinline__ bool query_valid(const uint32_t *__restrict__ tvb, const uint32_t *__restrict__ tv,
                                            uint64_t qa, uint32_t m) {
    const uint64_t w0 = qa >> 5, w1 = (qa + m - 1) >> 5;
    for (uint64_t g = w0 >> 5; g <= (w1 >> 5); g++) {
        uint32_t marked = __ldg(tvb + g);
        if (g == (w0 >> 5)) marked &= 0xFFFFFFFFu << (w0 & 31u);
        if (g == (w1 >> 5)) marked &= 0xFFFFFFFFu >> (31u - (uint32_t)(w1 & 31u));
        for (; marked != 0u; marked &= marked - 1u) {
            const uint64_t w = g * 32 + (__ffs(marked) - 1);
            const uint32_t lo = w == w0 ? (uint32_t)(qa & 31u) : 0u;
            const uint32_t hi = w == w1 ? (uint32_t)((qa + m - 1) & 31u) + 1u : 32u;
            if (__ldg(tv + w) & bit_range(lo, hi)) return false;
        }
    }
    return true;
}

// One query's result, written as one 32-byte store (a whole DRAM sector, so a
// result at a random slot needs no read-modify-write): [lo, hi), count and
// flags; lo = ~0 marks an invalid query (all-ones result).  trunc_cap: the
// call's locate cap (a count above it sets SA_RESULT_TRUNCATED), or ~0u.
__device__ __forceinline__ void store_result(sa_result *out, uint64_t q, uint64_t lo, uint64_t hi,
                                             uint32_t trunc_cap) {
    const bool bad = lo == ~0ull;
    const uint64_t count = bad ? ~0ull : hi - lo;
    const uint64_t flags = bad ? (uint64_t)SA_RESULT_INVALID
                               : (count > (uint64_t)trunc_cap ? (uint64_t)SA_RESULT_TRUNCATED : 0ull);
    asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(out + q), "l"(lo), "l"(hi), "l"(count),
                 "l"(flags)
                 : "memory");
}

// One 32-byte (one DRAM sector) read-only load; p must be 32-byte aligned.
// A single request per sector instead of two 16-byte ones, which the memory
// system would otherwise serve as two misses.
__device__ __forceinline__ void ldg32(const void *p, uint4 *lo, uint4 *hi) {
    unsigned long long a, b, c, d;
    asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p));
    *lo = make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
    *hi = make_uint4((uint32_t)c, (uint32_t)(c >> 32), (uint32_t)d, (uint32_t)(d >> 32));
}

template <typename IdxT>
__device__ __forceinline__ uint64_t sa_at(const void *sa, uint64_t i) {
    return (uint64_t)__ldg(reinterpret_cast<const IdxT *>(sa) + i);
}

// Predicated read-only loads: when pred is false nothing is read and the
// outputs keep their values.  p must be 32-byte (ldg32_if) or 16-byte
// (ldg16_if) aligned when pred is true.
__device__ __forceinline__ void ldg32_if(bool pred, const void *p, uint4 *lo, uint4 *hi) {
    unsigned long long a = 0, b = 0, c = 0, d = 0;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t"
        "@p ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];\n\t}"
        : "+l"(a), "+l"(b), "+l"(c), "+l"(d)
        : "l"(p), "r"((uint32_t)pred));
    *lo = make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
    *hi = make_uint4((uint32_t)c, (uint32_t)(c >> 32), (uint32_t)d, (uint32_t)(d >> 32));
}

__device__ __forceinline__ void ldg16_if(bool pred, const void *p, uint64_t *x, uint64_t *y) {
    unsigned long long a = 0, b = 0;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
        "@p ld.global.nc.v2.u64 {%0, %1}, [%2];\n\t}"
        : "+l"(a), "+l"(b)
        : "l"(p), "r"((uint32_t)pred));
    *x = a;
    *y = b;
}

// A 64-byte read-only record per lane, fetched by lane pairs: the two lanes
// of a pair read the even lane's record together (32 bytes each), then the
// odd lane's, and exchange the halves they hold for each other.  Random reads
// on the GB300 are limited per request, and the halves of a record that one
// instruction asks for are one request: 36.6 G random 64-byte records/s this
// way, 18.6 G/s when each lane reads its own halves in two instructions (over
// 64 GB).  Called by all 32 lanes; a lane with pred false reads nothing (its
// outputs are then zero).  p must be 64-byte aligned when pred is true.
__device__ __forceinline__ void ldg64_pairs_if(bool pred, const void *p, uint4 *a, uint4 *b, uint4 *c, uint4 *d) {
    const bool odd = threadIdx.x & 1u;
    const uint64_t mine = (uint64_t)p;
    const uint64_t other = __shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)mine, 1);
    const bool pred_other = __shfl_xor_sync(0xFFFFFFFFu, (int)pred, 1) != 0;
    const char *even_at = reinterpret_cast<const char *>(odd ? other : mine) + (odd ? 32 : 0);
    const char *odd_at = reinterpret_cast<const char *>(odd ? mine : other) + (odd ? 32 : 0);
    uint4 e0, e1, o0, o1;  // this lane's half of the even and of the odd lane's record
    ldg32_if(odd ? pred_other : pred, even_at, &e0, &e1);
    ldg32_if(odd ? pred : pred_other, odd_at, &o0, &o1);
    uint4 s0 = odd ? e0 : o0, s1 = odd ? e1 : o1;  // the half the other lane owns
    s0.x = __shfl_xor_sync(0xFFFFFFFFu, s0.x, 1);
    s0.y = __shfl_xor_sync(0xFFFFFFFFu, s0.y, 1);
    s0.z = __shfl_xor_sync(0xFFFFFFFFu, s0.z, 1);
    s0.w = __shfl_xor_sync(0xFFFFFFFFu, s0.w, 1);
    s1.x = __shfl_xor_sync(0xFFFFFFFFu, s1.x, 1);
    s1.y = __shfl_xor_sync(0xFFFFFFFFu, s1.y, 1);
    s1.z = __shfl_xor_sync(0xFFFFFFFFu, s1.z, 1);
    s1.w = __shfl_xor_sync(0xFFFFFFFFu, s1.w, 1);
    *a = odd ? s0 : e0;
    *b = odd ? s1 : e1;
    *c = odd ? o0 : s0;
    *d = odd ? o1 : s1;
}

// One window of a compare: q and t hold qlen and tlen bases (tlen may be 0)
// aligned at the top bits, starting at base `off` of the query; bits past
// qlen or tlen are ignored.  Returns 2 when the window does not decide, else
// the outcome with *lcp set.
__device__ __forceinline__ int cmp_window(uint64_t q, uint64_t t, uint32_t qlen, uint32_t tlen, uint32_t off,
                                          uint32_t m, uint32_t *lcp) {
    const uint64_t x = q ^ t;
    const uint32_t d = x ? ((uint32_t)__clzll((long long)x) >> 1) : 32u;
    if (d < min(qlen, tlen)) {
        *lcp = off + d;
        return q < t ? CMP_LESS : CMP_GREATER;
    }
    if (tlen < qlen) {
        *lcp = off + tlen;
        return CMP_GREATER;
    }
    if (off + qlen >= m) {
        *lcp = m;
        return CMP_PREFIX;
    }
    return 2;
}

// P (its first 128 bases in q; length m >= 1) against the first `known` <= 128
// bases of a suffix (t; zero past them) of `left` bases: the outcome with *lcp
// set, or CMP_PREFIX with *undecided when all known bases agree and both go
// on.  One path for every outcome -- the first differing word and the query's
// are picked by selects, and the highest differing bit tells the order -- as
// the lanes of a warp end in different words: a test per word, each taken by
// some lanes, cost twice the instructions, which bound the first pass (57 % of
// issue slots, 1300 instructions per 32 queries in k-mer order; 1040 with this
// and one result store per iteration).
__device__ __forceinline__ int cmp_first(const uint64_t q[4], const uint64_t t[4], uint32_t m, uint32_t known,
                                         uint32_t left, uint32_t *lcp, bool *undecided) {
    const uint64_t x0 = q[0] ^ t[0], x1 = q[1] ^ t[1], x2 = q[2] ^ t[2], x3 = q[3] ^ t[3];
    const bool low = (x0 | x1) != 0, first = (low ? x0 : x2) != 0;
    const uint64_t x = low ? (first ? x0 : x1) : (first ? x2 : x3);
    const uint64_t qx = low ? (first ? q[0] : q[1]) : (first ? q[2] : q[3]);
    const uint32_t z = (uint32_t)__clzll((long long)x);  // 64 when no word differs
    const uint32_t d = (low ? 0u : 64u) + (first ? 0u : 32u) + (z >> 1);
    const uint32_t have = min(known, left), lim = min(m, have);
    *lcp = min(d, lim);
    if (d < lim) return ((qx << (z & 63u)) >> 63) != 0 ? CMP_GREATER : CMP_LESS;
    if (have < m && have < known) return CMP_GREATER;  // the suffix ends first
    *undecided = m > known;
    return CMP_PREFIX;
}

// Bases a suffix record holds (8 fewer than without the neighbours' common
// prefixes: queries that tie on them read the text from 105 bases on, not 113.
// 8*10^6 copied queries at 100 Mbp, us a call at 104, 108, 112, 120 bases: 862,
// 868, 875, 938 with 112 bases and no prefixes, 594, 638, 641, 654 so).
constexpr uint32_t kRecBases = 104;

// P (its first 128 bases in q; length m >= 1) against a 32-byte suffix record
// (r0 = bases 0-63, r1 = bases 64-95, 96-103 with the neighbours' common
// prefixes, and the position).  Sets *undecided when all 104 bases agree, m >
// 104 and the suffix has 104 bases or more; the compare then continues in the
// text.
__device__ __forceinline__ int cmp_record(const uint64_t q[4], uint32_t m, uint4 r0, uint4 r1, uint32_t n,
                                          uint32_t *lcp, bool *undecided) {
    const uint64_t qm[4] = {q[0], q[1], q[2], q[3] & 0xFFFF000000000000ull};
    const uint64_t t[4] = {((uint64_t)r0.y << 32) | r0.x, ((uint64_t)r0.w << 32) | r0.z,
                           ((uint64_t)r1.y << 32) | r1.x, (uint64_t)(r1.z & 0xFFFF0000u) << 32};
    return cmp_first(qm, t, m, kRecBases, n - r1.w, lcp, undecided);
}

// The lengths of the common prefixes of the suffix at a rank with the
// suffixes at the ranks before and after it, as records and k-mer entries
// carry them: at most 255, which stands for 255 or more (0 where there is no
// such rank).
constexpr uint32_t kLcpCap = 255;
constexpr uint32_t kLcpUnknown = 0xFFFFFFFFu;

// The lower and the upper bound of one query (Section IV) moving in lockstep.
// Ranks are 32-bit modular: L = 0xFFFFFFFF stands for -1, and since every
// rank is in [-1, n] with n < 2^32 - 1, R - L and L + (R - L)/2 are exact.
// phase 0: both bounds share (L, R); a prefix match splits them into the
// lower bound in (L, R] (phase 1) and the upper bound in [HL, HR), kept until
// phase 1 ends (phase 2).  lcpL, lcpR, hlcpL, hlcpR: the query's common
// prefixes with the suffixes at L, R, HL, HR, as far as known.
struct Bounds {
    uint32_t L, R, HL, HR, lcpL, lcpR, hlcpL, hlcpR, lo, phase;

    __device__ __forceinline__ void start(uint32_t l, uint32_t r) {
        L = l;
        R = r;
        HL = HR = lcpL = lcpR = hlcpL = hlcpR = lo = phase = 0;
    }
    __device__ __forceinline__ uint32_t pivot() const { return L + ((R - L) >> 1); }

    // The outcome c of the compare at pivot M with l common bases; lp and ln:
    // the common prefixes of S_M with its neighbours (kLcpUnknown: not known).
    // They often settle the neighbour without reading it.  A neighbour shares
    // P's prefix m exactly when S_M has it and its common prefix with S_M is m
    // or more.  When P and S_M differ after l bases, a neighbour on P's side
    // of S_M that shares more than l bases with S_M differs from P in the same
    // way, and one that shares fewer lies beyond P: the bounds then meet.
    // (Probes per query beyond the entry's, on sampled 150-base queries with
    // at most one substitution: 2.07 without these, 1.37 with them, at 2.9
    // suffixes per k-mer; 0.29 and 0.16 at 0.37.  Four genomes, 1.6*10^7
    // queries of 20-250 bases: 1913 -> 1571 us a call; 3.1 Gbp, 4*10^7 of
    // 150: 8661 -> 7982 us.)
    // Returns whether both bounds are known.
    __device__ __forceinline__ bool step(int c, uint32_t M, uint32_t l, uint32_t m, uint32_t lp, uint32_t ln) {
        const bool known = lp != kLcpUnknown;
        if (c == CMP_PREFIX) {
            const uint32_t cut = min(m, kLcpCap);  // a value below it is exact and below m
            const bool prev_no = known && lp < cut, prev_yes = known && lp >= m;
            const bool next_no = known && ln < cut, next_yes = known && ln >= m;
            if (phase == 0) {
                HL = next_yes ? M + 1u : M;
                hlcpL = m;
                HR = next_no ? M + 1u : R;
                hlcpR = next_no ? ln : lcpR;
                phase = 1;
            }
            if (phase == 1) {
                if (prev_no) {
                    L = M - 1u;
                    lcpL = lp;
                }
                R = prev_yes ? M - 1u : M;
                lcpR = m;
            } else {
                if (next_no) {
                    R = M + 1u;
                    lcpR = ln;
                }
                L = next_yes ? M + 1u : M;
                lcpL = m;
            }
        } else if (c == CMP_LESS) {
            R = M;
            lcpR = l;
            if (known && l < lp) R = M - 1u;
            if (lp < kLcpCap && l > lp) {
                L = M - 1u;
                lcpL = lp;
            }
        } else {
            L = M;
            lcpL = l;
            if (known && l < ln) L = M + 1u;
            if (ln < kLcpCap && l > ln) {
                R = M + 1u;
                lcpR = ln;
            }
        }
        if (R - L > 1u) return false;
        if (phase == 1) {
            lo = R;
            L = HL;
            R = HR;
            lcpL = hlcpL;
            lcpR = hlcpR;
            phase = 2;
        }
        return R - L <= 1u;
    }
    // The result, once step() has returned true: [first(), R).
    __device__ __forceinline__ uint32_t first() const { return phase == 0 ? R : lo; }
};

// Where a kernel reads a query's bases beyond those its records carry: the
// packed batch (forward queries only, or of either strand), or the batch's
// ASCII bytes, of either strand.
enum class Bases { Packed, PackedStrands, Ascii };

// A query's 32-base window at base off (a multiple of 32 below m).
struct AsciiWindows {  // bytes [qa, qa + m) of the batch, or their reverse complement
    const uint8_t *ascii;
    uint64_t total;
    uint64_t qa;
    uint32_t m;
    bool rc;
    __device__ __forceinline__ uint64_t packed(uint32_t off, uint32_t *bad) const {
        const uint32_t nb = m - off < 32u ? m - off : 32u;
        if (!rc) return pack_word(ascii, total, qa + off, nb, bad);
        // the nb bytes that end off bases before the query's end
        return rc_window(pack_word(ascii, total, qa + (m - off - nb), nb, bad)) << (64u - 2u * nb);
    }
    __device__ __forceinline__ uint64_t operator()(uint32_t off) const {
        uint32_t bad = 0;
        return packed(off, &bad);
    }
};

template <bool kStrands>
struct PackedWindows {  // the query at place `at` of the packed batch
    const uint64_t *tq;
    uint64_t at;
    __device__ __forceinline__ uint64_t operator()(uint32_t off) const { return query_window<kStrands>(tq, at, off); }
};

// A query's windows from its record where that has them (off >= 96): base 96
// from w3 (its fourth packed word), bases 128 .. 128 + 32 tail_words - 1 from
// `tail` (later words its record carries, read again from the record when a
// compare gets there), the rest from src.
template <typename Source>
struct RecordWindows {
    Source src;
    uint64_t w3;
    const uint64_t *tail;
    uint32_t tail_words;
    __device__ __forceinline__ uint64_t operator()(uint32_t off) const {
        if (off == 96u) return w3;
        if (off >= 128u && ((off - 128u) >> 5) < tail_words) return __ldg(tail + ((off - 128u) >> 5));
        return src(off);
    }
};

// Query P (length m >= 1, its windows from qw) against the suffix at p of a
// text of n < 2^32 bases, from the 32-aligned base below `start` (< m; all
// bases before it known equal).
template <typename Windows>
__device__ __forceinline__ int cmp_suffix_qw(const uint64_t *__restrict__ T, uint32_t n, uint32_t p,
                                             const Windows &qw, uint32_t m, uint32_t start, uint32_t *lcp) {
    uint32_t off = start & ~31u;
    const uint32_t rem = n - p;
    for (;;) {
        const uint32_t qlen = min(32u, m - off);
        const uint32_t tlen = off < rem ? min(32u, rem - off) : 0u;
        const uint64_t q = qw(off);
        const uint64_t t = tlen ? text_window(T, (uint64_t)(p + off)) : 0ull;
        const int c = cmp_window(q, t, qlen, tlen, off, m, lcp);
        if (c != 2) return c;
        off += 32u;
    }
}

// The same with two windows a step, whose reads wait for each other's neither
// in the text nor in the query: for kernels with the registers for it (in the
// first pass of input order and in small.cu it spills or costs warps: 10^7
// reads 353 -> 373 us, 20,011 reads 29 -> 33 us).
template <typename Windows>
__device__ __forceinline__ int cmp_suffix_pairs(const uint64_t *__restrict__ T, uint32_t n, uint32_t p,
                                             const Windows &qw, uint32_t m, uint32_t start, uint32_t *lcp) {
    uint32_t off = start & ~31u;
    const uint32_t rem = n - p, sh = 2u * (p & 31u);
    for (;;) {
        const bool two = off + 32u < m;
        const uint64_t *at = T + ((p + off) >> 5);  // (off is a multiple of 32: the shift stays)
        const uint64_t q0 = qw(off), q1 = two ? qw(off + 32u) : 0ull;
        uint64_t t0 = 0, t1 = 0, t2 = 0;
        if (off < rem) {
            t0 = ldg_u64(at);
            t1 = ldg_u64(at + 1);
            if (two && off + 32u < rem) t2 = ldg_u64(at + 2);
        }
        int c = cmp_window(q0, (t0 << sh) | ((t1 >> 1) >> (63u - sh)), min(32u, m - off),
                           off < rem ? min(32u, rem - off) : 0u, off, m, lcp);
        if (c != 2) return c;
        off += 32u;
        c = cmp_window(q1, (t1 << sh) | ((t2 >> 1) >> (63u - sh)), min(32u, m - off),
                       off < rem ? min(32u, rem - off) : 0u, off, m, lcp);
        if (c != 2) return c;
        off += 32u;
    }
}

}  // namespace sa

// ---------------------------------------------------------------------------
// Host-side internals shared by the translation units.
// ---------------------------------------------------------------------------
struct sa_index {
    uint64_t n;
    uint32_t width;      // 4 or 8
    uint32_t depth;      // key-table depth
    int device;
    uint64_t nwords;     // packed words without padding
    uint64_t *text;      // device
    void *sa;            // device
    uint4 *keys;         // device, 2^depth entries
    uint8_t *keylen;     // device, 2^depth entries
    uint4 *rec;          // device, n 32-byte records in suffix-array order (2 uint4 each):
                         // the first 104 bases of suffix SA[i] as packed words w0, w1, w2
                         // (bases 0-95) and the 8 bases 96-103 in the top 16 bits of a 32-bit
                         // word w3, whose lower bytes hold the common prefixes (at most 255)
                         // with the suffixes at ranks i - 1 (bits 8-15) and i + 1 (bits 0-7),
                         // then SA[i]: {w0.lo, w0.hi, w1.lo, w1.hi}, {w2.lo, w2.hi, w3, SA[i]}
    uint4 *krt;          // device, 4^kmer_k k-mer entries of 64 bytes (4 uint4) for the k-base
                         // strings x (x as a 2k-bit number): {lo, hi, pos, clamp} -- the ranks
                         // [lo, hi) of the suffixes sorting at or after x and before x + 1,
                         // lo = number of suffixes that sort before x, and the position of the
                         // suffix at the first pivot lo - 1 + (hi - lo + 1) / 2 with, in bits
                         // 0-7 of the last word, clamp = min(192, n - pos) and above it that
                         // suffix's common prefixes with the ranks before (bits 8-15) and
                         // after it (bits 16-23), as in its record -- then the first 192 bases
                         // of that suffix as six packed words; null if none
    uint32_t kmer_k;
    uint64_t device_bytes;
};

namespace sa {

int status_from_cuda(cudaError_t e);
cudaMemPool_t scratch_pool(int device);
cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t s);
void scratch_free(void *p, cudaStream_t s);
int device_sm_count();

// Kernels launched from the API translation unit.
cudaError_t launch_pack_text(const char *ascii, uint64_t n, uint64_t *words, uint64_t nwords_padded,
                             int *err_flag, cudaStream_t s);
// A stretch of device memory a build may use as scratch (no longer than the call).
struct Arena {
    char *at;
    size_t left;
};
// Scratch comes from the arenas (may be null) while they last, then from the pool.
int build_suffix_array(sa_index *idx, cudaStream_t s, Arena *arenas, int n_arenas);
// The same array by the paper's DC3 construction, on the GPU (dc3_gpu.cu).
int build_suffix_array_dc3(sa_index *idx, cudaStream_t s);
cudaError_t launch_build_keys(sa_index *idx, cudaStream_t s);
cudaError_t launch_build_records(sa_index *idx, cudaStream_t s);
cudaError_t launch_build_kmer(sa_index *idx, cudaStream_t s);
cudaError_t launch_copy_kmer_counts(const sa_index *idx, uint32_t *dst, cudaStream_t s);

// Descriptors of every index a call uses, passed by value as a kernel
// parameter (64 x 80 bytes; kernel parameters may take up to 32 KB).
struct RefTable {
    RefDesc r[SA_MAX_REFS];
};

struct SearchLaunch {
    RefTable refs;
    uint32_t n_refs;
    uint32_t width;
    const char *ascii;        // query bases, indexed by q_off[q] - first
    const uint64_t *tq;       // packed batch: SA_TQ_LEAD_WORDS before it, nwords + SA_TQ_PAD_WORDS from it on
    const uint32_t *tvb;      // bitmap of the packed words that hold a byte that is not a base
    const uint32_t *tv;       // masks of those words: bit i set = base 32 w + i is not a base
    uint64_t nwords;          // ceil(total / 32)
    const uint64_t *q_off;    // n_q + 1 offsets
    uint64_t first;           // q_off[0]
    uint64_t total;           // q_off[n_q] - q_off[0]: query ranges past it are invalid
    const uint32_t *q_ref;    // null when n_refs == 1
    uint64_t n_q;
    uint4 *wrec;              // worklist records, 64 bytes (4 uint4) each, n_q of room
    uint32_t *wl_count;       // device: records in the worklist
    const uint4 *wrec_in;     // k-mer order: the batch's queries as records (first pass input), or null
    uint32_t *wl_in_count;    // k-mer order: records in wrec_in
    sa_result *out;
    int *pack_err;            // device flag: some query had a non-ACGT byte or bad offsets
    int *batch_dirty;         // device flag set by the packing: some byte of the batch is not a base
                              // (a clean batch's bitmap and masks need not be read)
    int *bad_ref;             // device flag: some query named a reference id >= n_refs
    unsigned long long *counter;
    int *status;
    uint32_t smem_bytes;      // shared-memory key tables
    uint32_t threads, blocks, chunk;
    uint32_t front_probes;    // probes per query in the first pass
    bool long_queries;        // the queries' average length is past what their records carry
    bool fused;               // k-mer order: the scatter packs its tiles' bases itself; tq holds only the
                              // words of tiles with longer queries, tv is null
    uint4 *spoiled;           // fused: the tiles that did not fit, {tile, first word, words, 0} each
    uint32_t *n_spoiled;      // fused: their number
    bool revcomp;             // search every query's reverse complement
    bool strand_bits;         // q_ref bit 31 selects each query's strand
    bool expire_waits;        // test hook: the bounded key-table wait gives up at once
    uint32_t trunc_cap;       // the locate cap of sa_search_locate (SA_RESULT_TRUNCATED), else ~0u
    // k-mer order (bucket.cu)
    uint64_t kscale;          // floor((2^64 - 1) / k-mer entries of all indexes of the call)
    uint32_t *bplan;          // the list's plan, kPlanWords words (see below; zeroed by the caller)
    // search + locate in one call: per 2^tile_shift queries, the sum of
    // min(count, trunc_cap) of their results (zeroed by the caller), or null
    uint64_t *tile_kept;
    uint32_t tile_shift;
    bool tile_sum_by_warp;    // input order: the lanes storing together mostly share a tile
    bool check_longest;       // small.cu: the longest queries' bytes are checked by a kernel of their own
};

// Queries per tile of the locate's scan (locate.cu): 4096, and 1024 for batches
// of up to 2^21 queries, whose 4096-query tiles would fill the GPU's 456
// resident CTAs a little more than once or not at all, and whose 1024-query
// tiles are few enough (kDirectTiles) to add up the sums of those before them
// without the scan's launch.  sa_locate, 1024 against 4096, us: 1.9*10^6 queries
// 80 against 88, 2^21 85 against 93; past it 2.2*10^6 91 against 93 and 87
// against 85 (14-base and 100-base queries), 3*10^6 113 against 107 and 106
// against 100, 9*10^6 273 against 269 and 254 against 259.
constexpr uint32_t kLocateTileShift = 12, kLocateSmallTileShift = 10;
inline uint32_t locate_tile_shift(uint64_t n_q) {
    return n_q <= (1ull << 21) ? kLocateSmallTileShift : kLocateTileShift;
}

// store_result for the search kernels; in a search + locate call it also
// adds the query's kept count min(count, cap) to its locate tile's sum, so
// the locate need not read every result to find the tile sums.
// In input order the lanes storing at the same time hold consecutive queries,
// so those sharing a tile add their counts with one atomic; in k-mer order
// each lane adds its own.  32 counts of up to trunc_cap may not fit 32 bits
// (an enormous cap and short or empty queries of a large text): the warp then
// adds their halves apart.
__device__ __forceinline__ void store_result_sum(const SearchLaunch &a, uint64_t q, uint64_t lo, uint64_t hi) {
    store_result(a.out, q, lo, hi, a.trunc_cap);
    if (a.tile_kept == nullptr) return;
    const uint64_t c = lo == ~0ull ? 0ull : hi - lo;
    const uint32_t k = c < (uint64_t)a.trunc_cap ? (uint32_t)c : a.trunc_cap;
    const uint64_t tile = q >> a.tile_shift;
    unsigned long long *sum_at = reinterpret_cast<unsigned long long *>(a.tile_kept) + tile;
    if (a.tile_sum_by_warp) {
        const unsigned same = __match_any_sync(__activemask(), tile);
        unsigned long long sum;
        if (a.trunc_cap <= 0xFFFFFFFFu / 32u)
            sum = __reduce_add_sync(same, k);
        else
            sum = __reduce_add_sync(same, k & 0xFFFFu) +
                  ((unsigned long long)__reduce_add_sync(same, k >> 16) << 16);
        if (sum != 0u && (threadIdx.x & 31u) == (unsigned)(__ffs(same) - 1)) atomicAdd(sum_at, sum);
    } else if (k != 0u) {
        atomicAdd(sum_at, (unsigned long long)k);
    }
}
// Worklist record of a query the first pass did not finish (64 bytes):
//   {L, R, m, q}            a bracket (L, R) holding both bounds (L = -1 is
//                           0xFFFFFFFF), the length and the query's index
//   {at.lo, at.hi | ref << 16 | strand, w4.lo, w4.hi}  its place in the packed
//                           batch (at < 2^48, and kRecordRc for the other
//                           strand), reference id (< 2^14), bases 128-159
//   {w0, w1}, {w2, w3}      its first 128 bases (packed words)
// Packs L.ascii; tvb is zero before, or null (then tv receives every word's mask).
cudaError_t launch_pack_batch(const SearchLaunch &L, uint64_t *tq, uint32_t *tvb, uint32_t *tv, cudaStream_t s);
// Packs the words of the tiles in L.spoiled, as above but without masks.
cudaError_t launch_pack_spoiled(const SearchLaunch &L, uint64_t *tq, uint32_t *tvb, cudaStream_t s);
cudaError_t launch_front(const SearchLaunch &L, cudaStream_t s);
// The batch's queries as records in k-mer order (wrec_in), the first pass's
// input in that order.
cudaError_t launch_bucketed_worklist(const SearchLaunch &L, uint4 *wrec_in, uint64_t *tq, uint32_t *tvb,
                                     cudaStream_t s);
cudaError_t launch_search(const SearchLaunch &L, cudaStream_t s);
// A small batch in one kernel, straight from its ASCII bases (L.tq, L.tv,
// L.wrec and the like are not used; L.pack_err and L.bad_ref may be null).
cudaError_t launch_search_small(const SearchLaunch &L, cudaStream_t s);
cudaError_t launch_search_plain(const SearchLaunch &L, cudaStream_t s);
// One thread: *dst = the call's status from its device flags (flags[1] a
// wait that ran out, flags[0] a query that is not bases, flags[3] a bad
// reference id), in that order of precedence.
cudaError_t launch_search_status(const int *flags, int *dst, cudaStream_t s);
// One thread each: fold one chunk's device flags into acc[0] (an atomic max
// of the status's precedence: 3 TIMEOUT, 2 BASE, 1 ARG, 0 OK), so that chunks
// on several streams fold into one word; then *dst = the status of acc[0], or
// SA_ERR_CAPACITY when that is SA_OK and check_overflow and acc[1] is set.
cudaError_t launch_fold_status(const int *flags, int *acc, cudaStream_t s);
cudaError_t launch_fold_final(const int *acc, bool check_overflow, int *dst, cudaStream_t s);
// One thread: *dst = SA_ERR_CAPACITY when *overflow is set and *dst is SA_OK.
cudaError_t launch_capacity_status(const int *overflow, int *dst, cudaStream_t s);
uint32_t search_table_bytes(uint32_t depth);  // shared-memory bytes of a depth-d key table

struct LocateLaunch {
    RefTable refs;
    uint32_t n_refs, width;
    const uint32_t *q_ref;
    const sa_result *res;
    uint64_t n_q;
    uint32_t cap;
    uint64_t *out_offsets;
    void *out_pos;
    uint64_t capacity;
    uint64_t *partials;       // scratch: one entry per scan tile + 1
    uint32_t tile_shift;      // kLocateTileShift or kLocateSmallTileShift
    bool presummed;           // partials already hold the tile sums (from the search kernels)
    int *overflow;            // optional device flag: a position fell at or beyond capacity
    const uint64_t *base_in;  // optional device value added to every offset (a chunk of a larger batch)
};
uint64_t locate_tiles(uint64_t n_q, uint32_t shift);
// Device address of the static scratch of sa_locate_noalloc on the current
// device (looked up once per device) and the number of partial sums it holds.
cudaError_t locate_static_partials(uint64_t **ptr, uint64_t *entries);
cudaError_t launch_locate(const LocateLaunch &L, cudaStream_t s);
// Copies positions [*first, *last) (clamped to capacity) of width bytes each
// from src to dst at the same indexes; dst may be host memory the device can
// address.
cudaError_t launch_copy_positions(const uint64_t *first, const uint64_t *last, const void *src, void *dst,
                                  uint32_t width, uint64_t capacity, cudaStream_t s);

}  // namespace sa
