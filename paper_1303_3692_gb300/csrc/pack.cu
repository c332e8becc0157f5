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

}  // namespace sa
