// pack.cu -- ASCII bases to the 2-bit big-endian layout (Section III alphabet).
#include "sa_internal.cuh"

namespace sa {

// One thread per packed word; words past the text (padding) are zero.
__global__ void pack_text_kernel(const uint8_t *__restrict__ ascii, uint64_t n, uint64_t *__restrict__ words,
                                 uint64_t nwords_padded, int *err_flag, bool aligned16) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nwords_padded; w += stride) {
        const uint64_t b0 = w * 32;
        uint64_t word = 0;
        uint32_t bad = 0;
        if (b0 + 32 <= n && aligned16) {
            const uint4 v0 = __ldg(reinterpret_cast<const uint4 *>(ascii + b0));
            const uint4 v1 = __ldg(reinterpret_cast<const uint4 *>(ascii + b0 + 16));
            word = pack32(v0, v1, &bad);
        } else {
            for (int j = 0; j < 32; j++) {
                const uint64_t b = b0 + j;
                uint32_t code = 0;
                if (b < n) {
                    code = base_code(ascii[b]);
                    if (code > 3) {
                        bad |= 1u;
                        code = 0;
                    }
                }
                word = (word << 2) | code;
            }
        }
        words[w] = word;
        if (bad) atomicOr(err_flag, 1);
    }
}

cudaError_t launch_pack_text(const char *ascii, uint64_t n, uint64_t *words, uint64_t nwords_padded,
                             int *err_flag, cudaStream_t s) {
    const int threads = 256;
    const uint64_t want = (nwords_padded + threads - 1) / threads;
    const int blocks = (int)(want < (uint64_t)device_sm_count() * 16 ? want : (uint64_t)device_sm_count() * 16);
    const bool aligned = ((uintptr_t)ascii & 15u) == 0;
    pack_text_kernel<<<blocks > 0 ? blocks : 1, threads, 0, s>>>(reinterpret_cast<const uint8_t *>(ascii), n,
                                                                 words, nwords_padded, err_flag, aligned);
    return cudaGetLastError();
}

// Packs a whole query batch as one text (the layout of the reference) and
// records which of its bytes are not bases, so that the search reads any
// window of any query with one window read and checks a query's validity from
// its own bytes only.  One thread per word; a word that holds a non-base byte
// has its mask stored, its bit set in the bitmap of such words (zeroed by the
// caller) and the batch flag raised, so a batch of reads with a few Ns costs
// what a clean one does.  When the batch starts on a 16-byte boundary a full
// word is two 16-byte loads, so the reads are fully coalesced.  Words past the
// batch (padding) are zero.
//
// Bound by HBM (1.25 bytes moved per base): 1.6*10^7 queries of 135 bases
// 0.42 ms = 6.4 TB/s.  A second pass that stored every word's mask, over a
// batch that was not clean, took as long again, and a packing of the reverse
// complement beside it 1.25 times that (9*10^6 x 125 bases, both strands, a
// few Ns: 1.08 ms, now 0.22 ms).  Two words per thread in flight, or a ballot
// per warp that writes the bitmap whole, are 6-9 % slower.
__global__ void pack_batch_kernel(const uint8_t *__restrict__ ascii, uint64_t total, uint64_t nwords,
                                  uint64_t *__restrict__ tq, uint32_t *__restrict__ tvb, uint32_t *__restrict__ tv,
                                  bool aligned16, int *dirty) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nwords + SA_TQ_PAD_WORDS; w += stride) {
        if (w >= nwords) {
            tq[w] = 0;
            if (tvb == nullptr) tv[w] = 0;
            continue;
        }
        const uint64_t b0 = w * 32;
        uint64_t word;
        uint32_t bad = 0;
        if (aligned16 && b0 + 32 <= total) {
            const uint4 v0 = __ldg(reinterpret_cast<const uint4 *>(ascii + b0));
            const uint4 v1 = __ldg(reinterpret_cast<const uint4 *>(ascii + b0 + 16));
            word = pack32(v0, v1, &bad);
        } else {
            const uint64_t left = total - b0;
            word = pack_word(ascii, total, b0, left < 32 ? (uint32_t)left : 32u, &bad);
        }
        tq[w] = word;
        uint32_t mask = 0;
        if (bad) {  // rare: find which bytes are not bases
            for (uint32_t j = 0; j < 32 && b0 + j < total; j++)
                if (base_code(ascii[b0 + j]) > 3) mask |= 1u << j;
        }
        if (tvb == nullptr) {
            tv[w] = mask;
        } else if (mask != 0u) {
            tv[w] = mask;
            atomicOr(tvb + (w >> 5), 1u << (w & 31u));
            if (*(volatile int *)dirty == 0) atomicOr(dirty, 1);
        }
    }
}

cudaError_t launch_pack_batch(const SearchLaunch &L, uint64_t *tq, uint32_t *tvb, uint32_t *tv, cudaStream_t s) {
    const int threads = 256;
    const uint64_t want = (L.nwords + SA_TQ_PAD_WORDS + threads - 1) / threads;
    const uint64_t cap = (uint64_t)device_sm_count() * 8;
    const unsigned blocks = (unsigned)(want < cap ? want : cap);
    const bool aligned = ((uintptr_t)L.ascii & 15u) == 0;
    const uint8_t *ascii = reinterpret_cast<const uint8_t *>(L.ascii);
    pack_batch_kernel<<<blocks, threads, 0, s>>>(ascii, L.total, L.nwords, tq, tvb, tv, aligned, L.batch_dirty);
    return cudaGetLastError();
}

// Word w of the batch, packed; its bit in the bitmap when it holds a byte that
// is not a base.
__device__ __forceinline__ void pack_one(const SearchLaunch &a, uint64_t w, bool aligned16, uint64_t *__restrict__ tq,
                                         uint32_t *__restrict__ tvb) {
    const uint8_t *ascii = reinterpret_cast<const uint8_t *>(a.ascii);
    uint32_t bad = 0;
    if (aligned16 && w * 32 + 32 <= a.total) {
        const uint4 *from = reinterpret_cast<const uint4 *>(ascii + w * 32);
        tq[w] = pack32(__ldg(from), __ldg(from + 1), &bad);
    } else {
        const uint64_t left = a.total - w * 32;
        tq[w] = pack_word(ascii, a.total, w * 32, left < 32 ? (uint32_t)left : 32u, &bad);
    }
    if (bad) {
        atomicOr(tvb + (w >> 5), 1u << (w & 31u));
        if (*(volatile int *)a.batch_dirty == 0) atomicOr(a.batch_dirty, 1);
    }
}

// The words of the k-mer order's tiles whose bases did not fit the scatter's
// shared memory (bucket.cu): each tile's by one CTA, but those with a very long
// query's by all of them.  Tiles with more words than the batch in all (offsets
// that go back) have it packed once.  Nearly always there are none, and the
// launch costs 1.5 us.
constexpr uint32_t kPackThreads = 256;
constexpr uint32_t kOneCtaWords = 1u << 14;

__global__ void __launch_bounds__(kPackThreads) pack_spoiled_kernel(const __grid_constant__ SearchLaunch a,
                                                                   uint64_t *__restrict__ tq,
                                                                   uint32_t *__restrict__ tvb) {
    __shared__ unsigned long long in_all;
    __shared__ uint32_t larger[kPackThreads], n_larger;
    const bool aligned16 = ((uintptr_t)a.ascii & 15u) == 0;
    const uint32_t n = *a.n_spoiled;
    if (n == 0) return;
    if (threadIdx.x == 0) in_all = 0;
    __syncthreads();
    unsigned long long mine = 0;
    for (uint32_t e = threadIdx.x; e < n; e += kPackThreads) mine += a.spoiled[e].z;
    atomicAdd(&in_all, mine);
    __syncthreads();
    if (in_all >= a.nwords) {
        for (uint64_t w = (uint64_t)blockIdx.x * kPackThreads + threadIdx.x; w < a.nwords;
             w += (uint64_t)gridDim.x * kPackThreads)
            pack_one(a, w, aligned16, tq, tvb);
        return;
    }
    // a tile of ordinary size is one CTA's
    for (uint32_t e = blockIdx.x; e < n; e += gridDim.x) {
        const uint4 t = a.spoiled[e];
        for (uint32_t i = threadIdx.x; t.z <= kOneCtaWords && i < t.z; i += kPackThreads)
            pack_one(a, (uint64_t)t.y + i, aligned16, tq, tvb);
    }
    // the others are dealt out to all
    for (uint32_t e0 = 0; e0 < n; e0 += kPackThreads) {
        const bool large = e0 + threadIdx.x < n && a.spoiled[e0 + threadIdx.x].z > kOneCtaWords;
        if (!__syncthreads_or(large)) continue;
        if (threadIdx.x == 0) n_larger = 0;
        __syncthreads();
        if (large) larger[atomicAdd(&n_larger, 1u)] = e0 + threadIdx.x;
        __syncthreads();
        for (uint32_t j = 0; j < n_larger; j++) {
            const uint4 t = a.spoiled[larger[j]];
            for (uint64_t i = (uint64_t)blockIdx.x * kPackThreads + threadIdx.x; i < t.z;
                 i += (uint64_t)gridDim.x * kPackThreads)
                pack_one(a, t.y + i, aligned16, tq, tvb);
        }
        __syncthreads();
    }
}

cudaError_t launch_pack_spoiled(const SearchLaunch &L, uint64_t *tq, uint32_t *tvb, cudaStream_t s) {
    pack_spoiled_kernel<<<(unsigned)device_sm_count() * 8u, kPackThreads, 0, s>>>(L, tq, tvb);
    return cudaGetLastError();
}

}  // namespace sa
