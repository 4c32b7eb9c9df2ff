// The FM index of a text filled on the device from a suffix array there
// (Section 2.3, Section 5 (1)-(2)): the BWT packed into occurrence blocks, the
// text-end array, and for collections the separator records and the sequence
// ends.  The layouts are those of ae_internal.h.
//
// On the host, one core took 2.0 s of the 2.14 s build of a 100 Mbp index (one
// cache miss per row for its BWT letter, then a copy of everything to the
// device); building a collection of 20 Mbp and searching it once took 744 ms
// and takes 18.3.  Here the rows are independent: a warp takes the 64 rows of a block,
// gathers their letters (random reads of one byte each, which bound the pass;
// the codes of a 100 Mbp text fit L2), packs them with ballots and counts them
// with population counts, and an exclusive scan over the blocks gives every
// block its counts.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "ae_device.cuh"
#include "ae_kernels.h"

namespace {
using namespace aedev;

struct BuildArgs {
    const uint8_t *s;        // codes of the text, or of the joined collection (0: separator, letters + 1)
    const int32_t *sa;       // J + 1 entries, suffix array of s reversed and the sentinel (may be tend itself)
    int64_t J;               // letters and separators
    const int64_t *starts;   // collections: first positions of the sequences in the text
    int32_t nseq;            // 0: one text
    uint32_t *occ, *sep;
    int32_t *tend;
    uint32_t *cnt;           // per letter, then separators: occurrences per block (stride nblocks)
    int64_t nblocks;
    int64_t *dollar;         // row of the sentinel
    int *bad;
};

// The last k < n with starts[k] + (joined ? k : 0) <= x (the first is 0)
__device__ __forceinline__ int32_t seq_of(const int64_t *starts, int32_t n, int64_t x, bool joined) {
    int32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int32_t mid = lo + ((hi - lo) >> 1);   // lo + hi may pass 2^31
        if (starts[mid] + (joined ? mid : 0) <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// The sequences' letters joined by separators: position p of sequence k goes to
// p + k (the separators' places are zero already)
__global__ void k_join(const uint8_t *codes, int64_t n, const int64_t *starts, int32_t nseq, uint8_t *joined) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
        joined[p + seq_of(starts, nseq, p, false)] = codes[p] + 1;
}

__global__ void k_seq_ends(const int64_t *starts, int32_t nseq, int64_t n, uint32_t *ends) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nseq; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = k + 1 < nseq ? starts[k + 1] : n;
        if (e > starts[k]) atomicOr(&ends[(e - 1) >> 5], 1u << ((e - 1) & 31));
    }
}

// 16 bits spread to the even bits of 32
__device__ __forceinline__ uint32_t spread16(uint32_t x) {
    x &= 0xFFFFu;
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}

// One warp per block of 64 rows: letters, text ends and per-block counts
template <int SIGMA>
__global__ void __launch_bounds__(256) k_bwt_blocks(BuildArgs a) {
    constexpr int BITS = SIGMA == 4 ? 2 : 5;
    constexpr int WORDS = SIGMA == 4 ? AE_DNA_BLOCK_WORDS : AE_PROT_BLOCK_WORDS;
    const int lane = threadIdx.x & 31;
    const int64_t N = a.J + 1;
    for (int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); b < a.nblocks;
         b += (int64_t)gridDim.x * (blockDim.x >> 5)) {
        uint32_t plane[2][BITS], counted[2], seps[2];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int64_t h = b * AE_ROWS_PER_BLOCK + half * 32 + lane;
            uint32_t code = 0;
            bool letter = false, sep = false;
            if (h < N) {
                const int64_t k = a.sa[h];
                if (k < 0 || k > a.J) {
                    *a.bad = 2;   // not a suffix array: an internal error
                } else {
                    if (k == 0) {
                        *a.dollar = h;   // the sentinel's row stores code 0
                    } else {
                        code = a.s[a.J - k];
                        letter = true;
                        if (a.nseq) {
                            sep = code == 0;
                            letter = !sep;
                            code = sep ? 0u : code - 1u;
                        }
                    }
                    // the substrings of row h end at position J - 1 - k
                    int64_t e = a.J - 1 - k;
                    if (a.nseq && e >= 0) {
                        const int32_t q = seq_of(a.starts, a.nseq, e, true);
                        e = (q + 1 < a.nseq && e == a.starts[q + 1] + q) ? -1 : e - q;   // -1: a separator
                    }
                    a.tend[h] = (int32_t)e;
                }
            }
#pragma unroll
            for (int t = 0; t < BITS; ++t) plane[half][t] = __ballot_sync(FULL, (code >> t) & 1u);
            counted[half] = __ballot_sync(FULL, letter);
            seps[half] = __ballot_sync(FULL, sep);
        }
        uint32_t *blk = a.occ + b * WORDS;
        if (SIGMA == 4) {
            if (lane < 4) {   // rows 16 lane .. 16 lane + 15, two bits each
                const int half = lane >> 1, sh = 16 * (lane & 1);
                const uint32_t lo = half ? plane[1][0] : plane[0][0], hi = half ? plane[1][1] : plane[0][1];
                blk[4 + lane] = spread16(lo >> sh) | (spread16(hi >> sh) << 1);
            }
        } else {
#pragma unroll
            for (int t = 0; t < BITS; ++t)
                if (lane < 2) blk[22 + 2 * t + lane] = lane ? plane[1][t] : plane[0][t];
        }
        if (lane < SIGMA) {
            uint32_t n = 0;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t eq = counted[half];
#pragma unroll
                for (int t = 0; t < BITS; ++t) eq &= ((lane >> t) & 1) ? plane[half][t] : ~plane[half][t];
                n += __popc(eq);
            }
            a.cnt[(int64_t)lane * a.nblocks + b] = n;
        } else if (lane == SIGMA) {
            a.cnt[(int64_t)SIGMA * a.nblocks + b] = __popc(seps[0]) + __popc(seps[1]);
        }
        if (a.nseq && lane < 2) a.sep[b * AE_SEP_BLOCK_WORDS + 1 + lane] = lane ? seps[1] : seps[0];
    }
}

// The scanned counts of `nl` letters from letter c0 on into the blocks
struct CountArgs {
    const uint64_t *off[5];
    uint32_t *dst[5];   // word of the first block
    int32_t stride[5];
};
__global__ void k_bwt_counts(CountArgs a, int nl, int64_t nblocks) {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nblocks; b += (int64_t)gridDim.x * blockDim.x)
        for (int c = 0; c < nl; ++c)
            if (a.dst[c]) a.dst[c][b * a.stride[c]] = (uint32_t)a.off[c][b];
}

unsigned blocks_for(int64_t n, int64_t per) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, 152 * 32));
}

}  // namespace

void ae_join_sequences(const uint8_t *codes, int64_t n, const int64_t *starts, int32_t nseq, uint8_t *joined,
                       uint32_t *ends, cudaStream_t st) {
    g_launches += 2;
    k_join<<<blocks_for(n, 256), 256, 0, st>>>(codes, n, starts, nseq, joined);
    k_seq_ends<<<blocks_for(nseq, 256), 256, 0, st>>>(starts, nseq, n, ends);
}

int64_t ae_fill_tmp_words(int64_t nblocks) { return ae_scan_tmp_words(nblocks, 5) + 5 * nblocks; }

void ae_fill_index(int sigma, const uint8_t *s, const int32_t *sa, int64_t J, const int64_t *starts, int32_t nseq,
                   uint32_t *occ, uint32_t *sep, int32_t *tend, int64_t nblocks, uint32_t *cnt, uint64_t *tmp,
                   uint64_t *totals, int64_t *dollar, int *bad, cudaStream_t st) {
    BuildArgs a;
    a.s = s;
    a.sa = sa;
    a.J = J;
    a.starts = starts;
    a.nseq = nseq;
    a.occ = occ;
    a.sep = sep;
    a.tend = tend;
    a.cnt = cnt;
    a.nblocks = nblocks;
    a.dollar = dollar;
    a.bad = bad;
    ++g_launches;
    if (sigma == 4) k_bwt_blocks<4><<<blocks_for(nblocks, 8), 256, 0, st>>>(a);
    else k_bwt_blocks<20><<<blocks_for(nblocks, 8), 256, 0, st>>>(a);
    // letters and, last, the separators, five arrays a scan (the last scan repeats
    // its last array when there are fewer)
    const int words = sigma == 4 ? AE_DNA_BLOCK_WORDS : AE_PROT_BLOCK_WORDS;
    for (int c0 = 0; c0 <= sigma; c0 += 5) {
        const uint32_t *in[5];
        uint64_t *out[5];
        CountArgs ca;
        const int nl = std::min(5, sigma + 1 - c0);
        for (int c = 0; c < 5; ++c) {
            const int l = c0 + std::min(c, nl - 1);
            in[c] = cnt + (int64_t)l * nblocks;
            out[c] = tmp + (int64_t)c * nblocks;
            ca.off[c] = out[c];
            ca.dst[c] = l < sigma ? occ + l : sep;
            ca.stride[c] = l < sigma ? words : AE_SEP_BLOCK_WORDS;
        }
        ae_scan_u32(in, out, 5, nblocks, totals + c0, tmp + 5 * nblocks, st);
        ++g_launches;
        k_bwt_counts<<<blocks_for(nblocks, 256), 256, 0, st>>>(ca, nl, nblocks);
    }
}
