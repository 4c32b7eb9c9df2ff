// Device kernels of exact local-alignment search on sm_103a.
//
// The search walks the suffix trie of T breadth-first through the FM index of
// the reversed text (Section 5): every trie node is an SA range [lo, hi) and
// appending a letter c to its substring is one backward-search step
// (lo' = C[c] + Occ(c, lo), hi' = C[c] + Occ(c, hi)).  Each node carries one
// sparse row of the Gotoh matrix M_X (Section 2.2): the live entries (j, M, G_a)
// sorted by query column j.  A child's row follows from its parent's by the
// three recurrences, where G_b (the in-row horizontal gap) is a max-plus prefix
// scan:  G_b(j) = s_g + j*s_s + max_{k<j} (M'(k) - k*s_s),  M' = max(D, G_a).
// An entry is kept only if its value exceeds
//     thr(j) = max{0, H - 1 - (m - 1 - j) * g_max}          (Theorem 2)
// (the text-length term of Theorem 2 is dropped: keeping more entries is always
// sound).  Starting the walk at depth q-1 from the query's (q-1)-grams is
// Theorem 3; depths beyond L_max (Theorem 1) never hold live entries.
//
// When a child has a single occurrence it leaves the trie: its row becomes an
// "injection" at its text end e.  The sweep kernel then follows such rows
// along the text (the next letter is T[e+1], read from the forward text),
// merging by maximum every row that reaches the same text position: rows of
// different trie paths ending at the same position have the same future, so
// only their per-entry maximum matters.  This is an order-free form of the
// global filter of Theorem 4 (a fork dominated by an alignment that already
// reaches its start cell is not followed separately).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "ae_device.cuh"
#include "ae_kernels.h"

#define FULL 0xffffffffu

// Kernel launches issued by the calling thread (reported as ae_stats.launches).
thread_local int64_t g_launches = 0;

namespace {
using namespace aedev;

// ------------------------------------------------------------------ scan

constexpr int SC_T = 256, SC_I = 8, SC_TILE = SC_T * SC_I;

template <typename In, int W>
struct InPtrs {
    const In *p[W];
};
template <int W>
struct OutPtrs {
    uint64_t *p[W];
};

template <typename In, int W>
__global__ void __launch_bounds__(SC_T) k_scan_reduce(InPtrs<In, W> in, int64_t N, uint64_t *bsum, int64_t nb) {
    __shared__ uint64_t red[W][SC_T / 32];
    const int64_t base = (int64_t)blockIdx.x * SC_TILE;
    uint64_t s[W];
#pragma unroll
    for (int w = 0; w < W; ++w) s[w] = 0;
    for (int i = 0; i < SC_I; ++i) {
        int64_t idx = base + (int64_t)i * SC_T + threadIdx.x;
        if (idx < N) {
#pragma unroll
            for (int w = 0; w < W; ++w) s[w] += (uint64_t)in.p[w][idx];
        }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint64_t v = s[w];
        for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(FULL, v, d);
        if ((threadIdx.x & 31) == 0) red[w][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    if (threadIdx.x < W) {
        uint64_t t = 0;
        for (int k = 0; k < SC_T / 32; ++k) t += red[threadIdx.x][k];
        bsum[(int64_t)threadIdx.x * nb + blockIdx.x] = t;
    }
}

template <typename In, int W>
__global__ void __launch_bounds__(SC_T) k_scan_down(InPtrs<In, W> in, OutPtrs<W> out, int64_t N,
                                                    const uint64_t *boff, int64_t nb, uint64_t *totals) {
    __shared__ uint64_t wsum[W][SC_T / 32];
    const int64_t base = (int64_t)blockIdx.x * SC_TILE + (int64_t)threadIdx.x * SC_I;
    uint64_t v[W][SC_I];
    uint64_t s[W];
#pragma unroll
    for (int w = 0; w < W; ++w) s[w] = 0;
#pragma unroll
    for (int i = 0; i < SC_I; ++i) {
        int64_t idx = base + i;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            v[w][i] = idx < N ? (uint64_t)in.p[w][idx] : 0;
            s[w] += v[w][i];
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t pre[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint64_t x = s[w];
        for (int d = 1; d < 32; d <<= 1) {
            uint64_t o = __shfl_up_sync(FULL, x, d);
            if (lane >= d) x += o;
        }
        if (lane == 31) wsum[w][wid] = x;
        pre[w] = x - s[w];
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint64_t add = boff ? boff[(int64_t)w * nb + blockIdx.x] : 0;
        for (int k = 0; k < wid; ++k) add += wsum[w][k];
        uint64_t run = pre[w] + add;
#pragma unroll
        for (int i = 0; i < SC_I; ++i) {
            int64_t idx = base + i;
            if (idx < N) out.p[w][idx] = run;
            run += v[w][i];
        }
        if (totals && blockIdx.x == gridDim.x - 1 && threadIdx.x == SC_T - 1) totals[w] = run;
    }
}

template <typename In, int W>
void scan_rec(const In *const *inp, uint64_t *const *outp, int64_t N, uint64_t *totals, uint64_t *tmp,
              cudaStream_t st) {
    InPtrs<In, W> in;
    OutPtrs<W> out;
    for (int w = 0; w < W; ++w) {
        in.p[w] = inp[w];
        out.p[w] = outp[w];
    }
    if (N <= 0) {
        if (totals) cudaMemsetAsync(totals, 0, sizeof(uint64_t) * W, st);
        return;
    }
    int64_t nb = (N + SC_TILE - 1) / SC_TILE;
    if (nb == 1) {
        ++g_launches;
        k_scan_down<In, W><<<1, SC_T, 0, st>>>(in, out, N, nullptr, 1, totals);
        return;
    }
    uint64_t *bsum = tmp, *boff = tmp + nb * W, *rest = tmp + 2 * nb * W;
    g_launches += 2;
    k_scan_reduce<In, W><<<(unsigned)nb, SC_T, 0, st>>>(in, N, bsum, nb);
    const uint64_t *bin[W];
    uint64_t *bout[W];
    for (int w = 0; w < W; ++w) {
        bin[w] = bsum + w * nb;
        bout[w] = boff + w * nb;
    }
    scan_rec<uint64_t, W>(bin, bout, nb, nullptr, rest, st);
    k_scan_down<In, W><<<(unsigned)nb, SC_T, 0, st>>>(in, out, N, boff, nb, totals);
}

// ------------------------------------------------------------------ radix sort
//
// Stable LSD sort of (key, value) pairs, 8 bits a pass.  A tile's pairs are
// ranked by digit in registers and put in digit order in shared memory, so that
// they leave in runs (16 pairs of a digit on average, 128 bytes of keys) instead
// of one scattered 8-byte store each.  10^7 pairs take 88 us in the scatter (240
// MB, 2.7 TB/s; bound by the ranking's votes and shared-memory chain) and 27 in
// the histogram, where one store per pair took 290 us a pass in all.  Up to
// RS_SMALL pairs one block does all passes in shared memory in one launch (the
// sorts of a small search were 5 passes of 3 launches, 24 us a pass).
constexpr int RS_T = 256, RS_I = 16, RS_TILE = RS_T * RS_I;
// Up to AE_RS_SPLIT pairs tiles of half the size are taken: a pass lasts as long
// as the few tiles an SM has one after the other.  Merges of 8,193 / 100 k / 1 M /
// 1.5 M records: 0.289 / 0.400 / 0.756 / 0.845 ms with half tiles, 0.313 / 0.431 /
// 0.788 / 0.825 with full ones.
#ifndef AE_RS_SPLIT
#define AE_RS_SPLIT (1 << 20)
#endif
constexpr int RS_ST = 1024, RS_SI = 8, RS_SMALL = RS_ST * RS_SI;

template <int T, int I>
struct RsSmem {
    uint64_t key[T * I];
    uint32_t val[T * I];
    uint32_t wcnt[T / 32][256];   // per warp and digit: pairs, then the pairs of earlier warps
    uint32_t first[256];          // the digit's first place in the tile
    uint32_t wsum[8];
};

template <int I>
__global__ void __launch_bounds__(RS_T) k_rs_hist(const uint64_t *keys, int64_t N, int shift, uint32_t *hist,
                                                  int64_t ntiles) {
    __shared__ uint32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (RS_T * I);
#pragma unroll
    for (int i = 0; i < I; ++i) {
        const int64_t idx = base + i * RS_T + threadIdx.x;
        if (idx < N) atomicAdd(&cnt[(keys[idx] >> shift) & 255], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

// A tile's pairs (thread order: warp, round, lane; the first n are there) into
// digit order in s.key / s.val; s.first holds each digit's first place
template <int T, int I>
__device__ __forceinline__ void rs_tile(RsSmem<T, I> &s, const uint64_t (&k)[I], const uint32_t (&v)[I], int n, int shift) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int d = lane; d < 256; d += 32) s.wcnt[wid][d] = 0;
    __syncwarp();
    uint32_t rank[I];   // among the warp's pairs of the same digit
#pragma unroll
    for (int i = 0; i < I; ++i) {
        const bool valid = wid * 32 * I + i * 32 + lane < n;
        const int d = (int)((k[i] >> shift) & 255);
        // the lanes with the same digit, bit by bit (eight votes: the match instruction
        // takes three times as long)
        unsigned peers = __ballot_sync(FULL, valid);
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const unsigned vote = __ballot_sync(FULL, (d >> x) & 1);
            peers &= ((d >> x) & 1) ? vote : ~vote;
        }
        const uint32_t c = valid ? s.wcnt[wid][d] : 0u;
        __syncwarp();
        rank[i] = c + __popc(peers & lt);
        if (valid && lane == __ffs(peers) - 1) s.wcnt[wid][d] = c + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        uint32_t sum = 0;
        for (int x = 0; x < T / 32; ++x) {
            const uint32_t c = s.wcnt[x][threadIdx.x];
            s.wcnt[x][threadIdx.x] = sum;
            sum += c;
        }
        const uint32_t incl = warp_incl_sum(sum);
        if (lane == 31) s.wsum[wid] = incl;
        s.first[threadIdx.x] = incl - sum;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        uint32_t before = 0;
        for (int x = 0; x < wid; ++x) before += s.wsum[x];
        s.first[threadIdx.x] += before;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < I; ++i) {
        if (wid * 32 * I + i * 32 + lane >= n) continue;
        const int d = (int)((k[i] >> shift) & 255);
        const uint32_t x = s.first[d] + s.wcnt[wid][d] + rank[i];
        s.key[x] = k[i];
        s.val[x] = v[i];
    }
    __syncthreads();
}

template <int I>
__global__ void __launch_bounds__(RS_T, 3) k_rs_scatter(const uint64_t *kin, const uint32_t *vin, uint64_t *kout,
                                                     uint32_t *vout, int64_t N, int shift, const uint64_t *offs,
                                                     int64_t ntiles) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    RsSmem<RS_T, I> &s = *reinterpret_cast<RsSmem<RS_T, I> *>(rs_smem);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * (RS_T * I);
    const int n = (int)min((int64_t)(RS_T * I), N - base);
    uint64_t k[I];
    uint32_t v[I];
#pragma unroll
    for (int i = 0; i < I; ++i) {
        const int x = wid * 32 * I + i * 32 + lane;
        k[i] = x < n ? kin[base + x] : 0;
        v[i] = x < n ? vin[base + x] : 0;
    }
    // where the tile's pairs of each digit go
    const uint64_t out0 = offs[(int64_t)threadIdx.x * ntiles + blockIdx.x];
    rs_tile<RS_T, I>(s, k, v, n, shift);
    uint64_t *out = reinterpret_cast<uint64_t *>(&s.wcnt[0][0]);   // no longer needed
    out[threadIdx.x] = out0 - s.first[threadIdx.x];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < I; ++i) {
        const int x = i * RS_T + threadIdx.x;
        if (x >= n) break;
        const uint64_t key = s.key[x];
        const uint64_t dst = out[(key >> shift) & 255] + x;
        kout[dst] = key;
        vout[dst] = s.val[x];
    }
}

// All passes of at most RS_SMALL pairs by one block, in place
__global__ void __launch_bounds__(RS_ST) k_rs_small(uint64_t *key, uint32_t *val, int n, int bits) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    RsSmem<RS_ST, RS_SI> &s = *reinterpret_cast<RsSmem<RS_ST, RS_SI> *>(rs_smem);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t k[RS_SI];
    uint32_t v[RS_SI];
#pragma unroll
    for (int i = 0; i < RS_SI; ++i) {
        const int x = wid * 32 * RS_SI + i * 32 + lane;
        k[i] = x < n ? key[x] : 0;
        v[i] = x < n ? val[x] : 0;
    }
    for (int shift = 0; shift < bits; shift += 8) {
        rs_tile<RS_ST, RS_SI>(s, k, v, n, shift);
#pragma unroll
        for (int i = 0; i < RS_SI; ++i) {
            const int x = wid * 32 * RS_SI + i * 32 + lane;
            if (x < n) {
                k[i] = s.key[x];
                v[i] = s.val[x];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < RS_SI; ++i) {
        const int x = wid * 32 * RS_SI + i * 32 + lane;
        if (x < n) {
            key[x] = k[i];
            val[x] = v[i];
        }
    }
}

// ------------------------------------------------------------------ queries

__global__ void k_encode(const uint8_t *ascii, uint8_t *codes, int64_t total, int alphabet, int *bad) {
    __shared__ uint8_t lut[256];
    for (int t = threadIdx.x; t < 256; t += blockDim.x) lut[t] = 255;
    __syncthreads();
    if (threadIdx.x == 0) {
        const char *a = alphabet == AE_DNA ? "ACGT" : "ARNDCQEGHILKMFPSTWYV";
        int s = alphabet == AE_DNA ? 4 : 20;
        for (int c = 0; c < s; ++c) lut[(uint8_t)a[c]] = (uint8_t)c;
    }
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint8_t c = lut[ascii[i]];
        if (c == 255) {
            atomicExch(bad, 1);
            c = 0;
        }
        codes[i] = c;
    }
}

// ------------------------------------------------------------------ seed (Theorem 3)

// The part of a seed subtree (its gram) when one search is split over ranks:
// a multiplicative hash spreads neighbouring grams over the parts.
__device__ __forceinline__ int fork_part(uint64_t gram, int parts) {
    return (int)((uint32_t)((gram * 0x9E3779B97F4A7C15ull) >> 32) % (uint32_t)parts);
}

__global__ void k_seed_keys(SeedArgs a, uint64_t *keys, uint32_t *vals) {
    const int bits = a.ix.sigma == 4 ? 2 : 5;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.npos;
         t += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = a.nitems;  // largest it with item_pos[it] <= t
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (a.item_pos[mid] <= t) lo = mid; else hi = mid;
        }
        const WorkItem it = a.items[lo];
        const int32_t y = it.c0 + (int32_t)(t - a.item_pos[lo]);
        const uint8_t *P = a.qv.codes + a.qv.off[it.qid];
        uint64_t gram = 0;
        for (int i = 0; i < a.d0; ++i) gram = (gram << bits) | P[y + i];
        keys[t] = ((uint64_t)lo << (bits * a.d0)) | gram;
        vals[t] = (uint32_t)y;
    }
}

__global__ void k_seed_flags(const uint64_t *keys, int64_t N, uint32_t *flags) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N; t += (int64_t)gridDim.x * blockDim.x)
        flags[t] = (t == 0 || keys[t] != keys[t - 1]) ? 1u : 0u;
}

template <int SIGMA>
__global__ void k_seed_nodes(SeedArgs a, const uint64_t *keys, const uint32_t *vals, int64_t N,
                             const uint32_t *flags, const uint64_t *flag_off, Node *nodes, int32_t *aj,
                             int32_t *aM, int32_t *aGa) {
    const int bits = SIGMA == 4 ? 2 : 5;
    const uint64_t gmask = (1ull << (bits * a.d0)) - 1ull;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N; t += (int64_t)gridDim.x * blockDim.x) {
        aj[t] = (int32_t)vals[t] + a.d0 - 1;
        // q-prefix domination (Lemma 1): when every occurrence of the gram in T is
        // preceded by the query letter before its start y, the fork starting at y
        // is matched letter for letter, one better, by the fork starting at y - 1
        // (the same text ends, one more match), so its entry starts dead
        int32_t M0 = a.d0 * a.sc.sa;
        bool dead = false;
        if (a.dom && vals[t] > 0) {
            const WorkItem it = a.items[(int32_t)(keys[t] >> (bits * a.d0))];
            const int prev = a.qv.codes[a.qv.off[it.qid] + vals[t] - 1];
            dead = __ldg(a.dom + (keys[t] & gmask)) == (1u << prev);
        }
        const unsigned dm = __ballot_sync(__activemask(), dead);
        // a search split over ranks keeps the seed subtrees of its own part
        if (a.parts > 1 && fork_part(keys[t] & gmask, a.parts) != a.part) dead = true;
        if (dead && a.dominated && (threadIdx.x & 31) == __ffs(dm) - 1)
            atomicAdd(a.dominated, (unsigned long long)__popc(dm));
        if (dead) M0 = AE_NEG;
        if (a.int16) {
            reinterpret_cast<uint32_t *>(aM)[t] = pack_mg(M0, AE_NEG);
        } else {
            aM[t] = M0;
            aGa[t] = AE_NEG;
        }
        if (flags[t]) {
            uint64_t key = keys[t];
            uint64_t gram = key & gmask;
            uint32_t lo = 0, hi = (uint32_t)a.ix.rows;
            for (int i = a.d0 - 1; i >= 0; --i) {
                int c = (int)((gram >> (bits * i)) & ((1u << bits) - 1u));
                lo = a.ix.C[c] + occ_of<SIGMA>(a.ix, c, lo);
                hi = a.ix.C[c] + occ_of<SIGMA>(a.ix, c, hi);
                if (hi <= lo) { lo = hi = 0; }
            }
            int64_t k = (int64_t)flag_off[t];
            Node nd;
            nd.lo = lo;
            nd.hi = hi;
            nd.item = a.items[(int32_t)(key >> (bits * a.d0))].qid;   // query id, 0 levels unique
            nd.cnt = 0;
            nd.off = (uint64_t)t;
            nodes[k] = nd;
        }
    }
}

// Predecessor masks of the d0-grams of T.  A gram is an occurrence only if it
// lies inside one sequence (collections); its predecessor is the letter before
// it, or `sigma` when it starts a sequence.  Small tables are merged per block
// in shared memory first (the grams of i.i.d. text hit every entry).
__global__ void k_dom_table(IndexView ix, int d0, int bits, uint32_t *mask, int64_t ngram) {
    extern __shared__ uint32_t sm_mask[];
    const bool local = ngram <= 4096;
    if (local) {
        for (int64_t g = threadIdx.x; g < ngram; g += blockDim.x) sm_mask[g] = 0;
        __syncthreads();
    }
    const int64_t last = ix.n - d0;   // last start position
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p <= last; p += (int64_t)gridDim.x * blockDim.x) {
        uint64_t gram = 0;
        bool inside = true;
        for (int i = 0; i < d0; ++i) {
            gram = (gram << bits) | ix.text[p + i];
            if (i + 1 < d0 && seq_end(ix, p + i)) inside = false;
        }
        if (!inside) continue;
        const int prev = (p > 0 && !seq_end(ix, p - 1)) ? (int)ix.text[p - 1] : ix.sigma;
        if (local) atomicOr(&sm_mask[gram], 1u << prev);
        else atomicOr(&mask[gram], 1u << prev);
    }
    if (local) {
        __syncthreads();
        for (int64_t g = threadIdx.x; g < ngram; g += blockDim.x)
            if (sm_mask[g]) atomicOr(&mask[g], sm_mask[g]);
    }
}

__global__ void k_seed_fix(Node *nodes, const uint64_t *nn_dev, int64_t N) {
    const int64_t nn = (int64_t)*nn_dev;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nn; i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t end = (i + 1 < nn) ? nodes[i + 1].off : (uint64_t)N;
        nodes[i].cnt = (uint32_t)(end - nodes[i].off);
    }
}

// ------------------------------------------------------------------ text-position sweep

__global__ void k_inject_keys(const Inject *inj, int64_t ninj, uint64_t *keys, uint32_t *vals) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ninj; t += (int64_t)gridDim.x * blockDim.x) {
        keys[t] = ((uint64_t)(uint32_t)inj[t].qid << 32) | (uint32_t)inj[t].e;
        vals[t] = (uint32_t)t;
    }
}

// Of the sorted keys: the range of each query's injections
__global__ void k_query_ranges(const uint64_t *keys, int64_t ninj, uint2 *range) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ninj; t += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t q = (uint32_t)(keys[t] >> 32);
        if (t == 0 || (uint32_t)(keys[t - 1] >> 32) != q) range[q].x = (uint32_t)t;
        if (t + 1 == ninj || (uint32_t)(keys[t + 1] >> 32) != q) range[q].y = (uint32_t)(t + 1);
    }
}

// Whether the injections of query q lie so close that they leave no gaps
__device__ __forceinline__ bool leaf_dense(const LeafArgs &a, int32_t q) {
    const uint64_t c = a.qrange ? a.qrange[q].y - a.qrange[q].x : (uint64_t)a.ninj;
    return (uint64_t)a.ix.n < AE_LEAF_DENSE * c;
}

// Where tasks of the sweep may start: for each multiple of seg, the first place
// before the next multiple at which the injections are cut (an offset, or
// LEAF_NO_CUT).  Rows injected close to each other, as along a homologous region,
// belong to one walk: cut apart, each part's walk would run on to the region's
// end beside the others, over the same cells.  So they are cut
// - where the query changes,
// - at gaps of more than AE_LEAF_GAP text positions, or one and a half times the
//   query's average gap where that is less (a fifth of the gaps of randomly placed
//   injections is longer; along a homolog they lie every few positions),
// - at multiples of a span of two to four query lengths, if there was no gap for
//   a span before.  A row lives about as long as its query, so a longer task only
//   walks one row after the other that could be walked side by side, as in a
//   tandem repeat that the query holds one copy of (3,000 copies of 171 letters,
//   613 bp query: sweep 17.3 ms without, 13.5 with this cut),
// - at every multiple of seg if the query's injections are dense.
// Cut at multiples of 32 injections instead, six homologous reads wrote 13 times
// the hit records (sweep 100 ms against 17).  One warp per multiple.
constexpr uint32_t LEAF_NO_CUT = 0xFFFFFFFFu;
__global__ void __launch_bounds__(256) k_leaf_cuts(LeafArgs a, const uint64_t *keys, uint32_t *cuts) {
    const int lane = threadIdx.x & 31;
    for (int64_t s = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); s < a.nseg;
         s += (int64_t)gridDim.x * (blockDim.x >> 5)) {
        const int64_t k0 = s * a.seg, k1 = min(k0 + a.seg, a.ninj);
        uint32_t at = LEAF_NO_CUT;
        for (int64_t k = k0; k < k1 && at == LEAF_NO_CUT; k += 32) {
            const int64_t x = k + lane;
            bool cut = false, past = false;
            uint64_t y = 0;
            uint32_t gap = 0;
            int span = 0;   // log2
            if (x < k1) {
                y = keys[x];
                const uint64_t z = x ? keys[x - 1] : ~0ull;
                const int32_t q = (int32_t)(y >> 32);
                const uint64_t c = a.qrange ? a.qrange[q].y - a.qrange[q].x : (uint64_t)a.ninj;
                gap = (uint32_t)min((uint64_t)AE_LEAF_GAP, 3 * (uint64_t)a.ix.n / (2 * c));
                span = min(max(33 - __clz(a.qv.m[q]), AE_LEAF_SPAN_MIN), AE_LEAF_SPAN_MAX);
                cut = (y >> 32) != (z >> 32) || (uint32_t)y - (uint32_t)z > gap || (x == k0 && leaf_dense(a, q));
                past = !cut && ((uint32_t)y >> span) != ((uint32_t)z >> span);
            }
            const unsigned bc = __ballot_sync(FULL, cut), bp = __ballot_sync(FULL, past);
            for (unsigned b = bc | bp; b && at == LEAF_NO_CUT; b &= b - 1) {   // in order
                const int l = __ffs(b) - 1;
                bool here = (bc >> l) & 1u;
                if (!here) {
                    // past a multiple of the span: a cut if no gap lies within a span before it
                    const uint64_t yl = __shfl_sync(FULL, y, l);
                    const uint32_t gl = __shfl_sync(FULL, gap, l), len = 1u << __shfl_sync(FULL, span, l);
                    unsigned ended = 0, broken = 0;
                    for (int64_t w = k + l - 1; !(ended | broken); w -= 32) {
                        const int64_t t = w - lane;
                        const uint64_t v = t >= 0 ? keys[t] : ~0ull, u = t > 0 ? keys[t - 1] : ~0ull;
                        const bool far = t >= 0 && (v >> 32) == (yl >> 32) && (uint32_t)yl - (uint32_t)v >= len;
                        ended = __ballot_sync(FULL, far);
                        broken = __ballot_sync(FULL, !far && ((u >> 32) != (v >> 32) || (uint32_t)v - (uint32_t)u > gl ||
                                                              t <= 0));
                    }
                    here = ended && (!broken || __ffs(ended) < __ffs(broken));
                }
                if (here) at = (uint32_t)(k - k0) + l;
            }
        }
        if (lane == 0) cuts[s] = at;
    }
}

struct Buf {
    int32_t *j, *M, *Ga;
};

__device__ __forceinline__ int64_t lower_bound_g(const int32_t *a, int64_t n, int32_t x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (a[mid] < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Hit records of the sweep are staged per warp in shared memory and appended
// to the global buffer LEAF_HS at a time, so that the walk along a homologous
// region (hits in most chunks) does not take an atomic on the shared counter
// per chunk.  A chunk with more than LEAF_HS hits reserves global space itself.
constexpr int LEAF_HS = 256;
constexpr int LEAF_WARPS = 4;   // k_leaf runs 128-thread blocks

struct HitStage {
    uint64_t *key;
    int32_t *score;
    uint32_t n;     // staged records (warp-uniform)
    uint32_t cap;   // records the stage holds
};

__device__ __forceinline__ void stage_flush(HitStage &hs, const LeafArgs &a, int lane) {
    __syncwarp();
    if (hs.n == 0) return;
    unsigned long long g = 0;
    if (lane == 0) g = atomicAdd(a.hit_count, (unsigned long long)hs.n);
    g = __shfl_sync(FULL, g, 0);
    if (g + hs.n <= a.hit_cap) {
        for (uint32_t i = lane; i < hs.n; i += 32) {
            a.hit_key[g + i] = hs.key[i];
            a.hit_score[g + i] = hs.score[i];
        }
    } else if (lane == 0) {
        atomicAdd(&a.stats->hit_overflow, 1ull);
    }
    __syncwarp();
    hs.n = 0;
}

// Slots for htot records of this chunk (warp-uniform call): in the stage
// (staged) or in the global buffer (ok = within its capacity).
__device__ __forceinline__ uint64_t stage_reserve(HitStage &hs, const LeafArgs &a, int lane, uint32_t htot,
                                                  bool &staged, bool &ok) {
    if (htot > hs.cap) {
        unsigned long long g = 0;
        if (lane == 0) g = atomicAdd(a.hit_count, (unsigned long long)htot);
        g = __shfl_sync(FULL, g, 0);
        staged = false;
        ok = g + htot <= a.hit_cap;
        if (!ok && lane == 0) atomicAdd(&a.stats->hit_overflow, 1ull);
        return g;
    }
    if (hs.n + htot > hs.cap) stage_flush(hs, a, lane);
    staged = true;
    ok = true;
    const uint64_t b = hs.n;
    hs.n += htot;
    return b;
}

__device__ __forceinline__ void hit_put(HitStage &hs, const LeafArgs &a, bool staged, uint64_t slot, uint64_t key,
                                        int32_t score) {
    if (staged) {
        hs.key[slot] = key;
        hs.score[slot] = score;
    } else {
        a.hit_key[slot] = key;
        a.hit_score[slot] = score;
    }
}

// Slots of one sweep entry (see slot_finish): slot A at the entry's column,
// slot B at the next column unless the next entry is there.
struct Slots {
    int32_t colA, MpA, GaA, MpB, Dp, Dk, next_col;
    bool hasB;
};

__device__ __forceinline__ void make_slots(const ScoreView &sc, const int8_t *smat, int c, const uint8_t *P, int32_t m,
                                           int32_t H, int32_t g, int32_t oe, bool valid, int32_t j, int32_t M,
                                           int32_t Ga, int32_t pj, int32_t pM, int32_t jn, Slots &s) {
    s.colA = m;
    s.MpA = s.GaA = s.MpB = s.Dp = s.Dk = AE_NEG;
    s.next_col = m;
    s.hasB = false;
    if (!valid) return;
    s.colA = j;
    const int32_t tA = thr_of(j, m, H, g);
    if (pj + 1 == j && pM > AE_NEG) {
        const int32_t D = pM + delta_of(sc, smat, c, P[j]);
        s.Dp = D > tA ? D : AE_NEG;
    }
    const int32_t gap = gap_from_i32(M, Ga, sc.ss, oe);
    s.GaA = gap > tA ? gap : AE_NEG;
    s.MpA = max(s.Dp, s.GaA);
    s.hasB = (j + 1 < m) && (j + 1 != jn);
    if (s.hasB) {
        const int32_t D = M + delta_of(sc, smat, c, P[j + 1]);
        s.Dk = D > thr_of(j + 1, m, H, g) ? D : AE_NEG;
        s.MpB = s.Dk;
    }
    s.next_col = jn;
}

// Merge the rows injected at (qid, p) into the walked row Rn (nlen entries), in
// place.  They are finished rows, and the union of two finished rows taken by
// maximum per column is again finished (each is closed under the horizontal-gap
// recurrence), so the merge needs no second finish.  Cells where an injected row
// brings a new or larger value report their hits here.
//
// Where most positions have an injection (protein at low thresholds) half of the
// sweep's rows are merged, so the walked row is touched as little as possible: a
// lane looks up one injected entry (the one search there is); columns both rows
// have are raised where they stand; for new columns the entries behind the first
// of them move up, 32 at a time from the row's end (each moves by the number of
// new columns before it, so none is overwritten before it is read).
// Against a merge through two copies of the row: protein, 5.1 M injections of 28
// entries into rows of 130, sweep 89 -> 69 ms.
// Used by the warp walk of k_leaf and, run by one warp, by the block walk of
// k_leaf_wide.
template <bool RUN>
__device__ __forceinline__ void leaf_merge(const LeafArgs &a, int lane, int32_t qid, int32_t p, int32_t H,
                                           uint64_t jmask, int64_t &k, int64_t kend, const Buf &Rn, int64_t &nlen,
                                           int64_t cap, bool &overflow, HitStage &hstage, unsigned long long &st_ent,
                                           unsigned long long &st_reused, unsigned long long &st_t0) {
    const unsigned lt = (1u << lane) - 1u;
    const uint64_t kq = ((uint64_t)qid << (a.be + a.bj)) | ((uint64_t)(uint32_t)p << a.bj);
    while (k < kend) {
        const Inject I = a.inj[a.order[k]];
        if (I.qid != qid || I.e != p) break;
        ++k;
        const int32_t *ij = a.lj + I.off, *iM = a.lM + I.off, *iGa = a.lGa + I.off;
        const int32_t icnt = (int32_t)I.cnt;
        // the entry of this lane, its place in the walked row and the values there
        int32_t n = (int32_t)nlen, y = 0, Mi = AE_NEG, Gi = AE_NEG, q = INT32_MAX, Mv = AE_NEG, Gv = AE_NEG;
        bool same = false;
        auto look = [&](int32_t idx) {
            q = INT32_MAX;
            same = false;
            Mi = Gi = Mv = Gv = AE_NEG;
            if (idx < icnt) {
                y = ij[idx];
                Mi = iM[idx];
                Gi = iGa[idx];
                int32_t lo = 0, hi = n;
                if (RUN && n > 0) {   // columns are consecutive along a homolog: look there first (2 % of such a walk)
                    const int32_t x = y - Rn.j[0];
                    if (x >= 0 && x < n && Rn.j[x] == y) lo = hi = x;
                }
                while (lo < hi) {
                    const int32_t mid = (lo + hi) >> 1;
                    if (Rn.j[mid] < y) lo = mid + 1; else hi = mid;
                }
                q = lo;
                same = q < n && Rn.j[q] == y;
                if (same) {
                    Mv = Rn.M[q];
                    Gv = Rn.Ga[q];
                }
            }
        };
        // an injected row whose every entry the walked row already has with
        // M and G_a at least as large changes nothing (its hits were reported
        // with the walked values): skip it.  Along a homologous region the row
        // walked from earlier starts usually dominates the later forks.
        bool dominated = true;
        int32_t at = 0;
        for (; dominated && at < icnt; at += 32) {
            look(at + lane);
            dominated = __all_sync(FULL, at + lane >= icnt || (same && Mv >= Mi && Gv >= Gi));
        }
        if (dominated) {
            st_reused += (unsigned long long)icnt;   // the whole row rides on the walked one
            continue;
        }
        if (nlen + icnt > cap) {
            overflow = true;
            break;
        }
        for (int32_t base = 0; base < icnt; base += 32) {
            if (at != 32 || base) look(base + lane);   // (the first 32 may have been looked up just now)
            const bool fresh = base + lane < icnt && !same;
            const bool hit = Mi > Mv && Mi >= H;
            if (same) {
                if (Mi > Mv) Rn.M[q] = Mi;
                if (Gi > Gv) Rn.Ga[q] = Gi;
            }
            const unsigned bf = __ballot_sync(FULL, fresh), bh = __ballot_sync(FULL, hit);
            __syncwarp();
            if (bf) {
                const int32_t first = __shfl_sync(FULL, q, __ffs(bf) - 1);
                for (int32_t c = (n - 1) & ~31; n > 0 && c >= (first & ~31); c -= 32) {
                    const int32_t x = c + lane;
                    const bool moves = x >= first && x < n;
                    int32_t vj = 0, vM = 0, vG = 0;
                    if (moves) {
                        vj = Rn.j[x];
                        vM = Rn.M[x];
                        vG = Rn.Ga[x];
                    }
                    int t = 0;   // injected entries with a place at or before x (places do not decrease)
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (__shfl_sync(FULL, q, t + step - 1) <= x) t += step;
                    if (__shfl_sync(FULL, q, t) <= x) ++t;
                    const int32_t d = x + __popc(bf & (t < 32 ? (1u << t) - 1u : ~0u));
                    __syncwarp();
                    if (moves) {
                        Rn.j[d] = vj;
                        Rn.M[d] = vM;
                        Rn.Ga[d] = vG;
                    }
                    __syncwarp();
                }
                if (fresh) {
                    const int32_t d = q + __popc(bf & lt);
                    Rn.j[d] = y;
                    Rn.M[d] = Mi;
                    Rn.Ga[d] = Gi;
                }
                n += __popc(bf);
                if (a.tiers && fresh) ++st_t0;
            }
            if (bh) {
                bool staged, hok;
                const uint64_t hbase = stage_reserve(hstage, a, lane, __popc(bh), staged, hok);
                if (hok && hit)
                    hit_put(hstage, a, staged, hbase + __popc(bh & lt), kq | ((uint64_t)y & jmask), Mi);
            }
            __syncwarp();
        }
        st_ent += (unsigned long long)(n - nlen);
        st_reused += (unsigned long long)(icnt - (n - nlen));   // columns both rows had
        nlen = n;
    }
}

// First injection of task s: the first cut at or behind the multiple of seg.  It
// depends on s alone and does not decrease.
__device__ __forceinline__ int64_t task_start(const LeafArgs &a, int lane, int64_t s) {
    if (!a.cuts || s == 0) return min(s * a.seg, a.ninj);
    for (int64_t t = s; t < a.nseg; t += 32) {
        const uint32_t c = t + lane < a.nseg ? a.cuts[t + lane] : LEAF_NO_CUT;
        const unsigned b = __ballot_sync(FULL, c != LEAF_NO_CUT);
        if (b) {
            const int l = __ffs(b) - 1;
            return (t + l) * a.seg + __shfl_sync(FULL, c, l);
        }
    }
    return a.ninj;
}

// One warp per task, a run of consecutive injections (sorted by query and text
// end; k_leaf_cuts).  The warp carries a row R along text positions p, p+1, ...:
//   candidates of row p+1 = the vertical and diagonal slots generated from R
//   with letter T[p+1], merged by maximum with every injected row at p+1;
//   then the horizontal-gap finish of Section 2.2 gives row p+1.
// The walk jumps to the next injection when R has no live entry.  Rows live
// in per-warp global scratch (cap entries per buffer); a row that outgrows it
// sets leaf_overflow and the host reruns with a larger cap.
// A walk whose row grows wide (LeafArgs says when) is handed on, with the rest of its
// task, to k_leaf_wide (a block of threads per walk); without a slot or room for its
// row the warp carries on itself.
// A step is a chain of scans and dependent loads, so the resident warps set the
// rate: 6 blocks per SM at one entry per lane (E = 1; 80 registers, 228 bytes of spills)
// against 3 at two entries (162 registers, 38 % of the issue slots used; 526
// warp instructions per 32 entries).  Sweeps of a protein batch, a 1 M-letter query
// and a batch with cheap gaps: 51.7 / 22.9 / 11.3 ms against 58.5 / 28.8 / 16.1
// (4 blocks 53.3 / 24.6 / 12.7; 8 blocks 53.2 / - / 11.3).  Where no walk moves to
// a block (tier counting, leaf_wide_rows 0, the fixed arena of the no-allocation
// entry point with its two blocks per SM) the longest walk sets the time, and two
// entries per lane without spills are faster (E = 2, 164 registers): a 400-letter
// homolog in the arena 1.81 ms against 2.36, 100 reads of 1,000 letters with tier
// counting 11.1 / 15.3, six of 4,000-12,000 letters 1,030 / 1,650.
#ifndef AE_LEAF_MINB
#define AE_LEAF_MINB 6
#endif
template <int E>
__global__ void __launch_bounds__(128, E == 1 ? AE_LEAF_MINB : 2) k_leaf(LeafArgs a) {
    __shared__ int8_t smat[AE_MAX_SIGMA * AE_MAX_SIGMA];
    __shared__ uint64_t s_hkey[LEAF_WARPS][LEAF_HS];
    __shared__ int32_t s_hscore[LEAF_WARPS][LEAF_HS];
    load_matrix(a.sc, smat);
    const int lane = threadIdx.x & 31;
    const int gw = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (gw >= a.nwarps) return;
    HitStage hstage = {s_hkey[(threadIdx.x >> 5) & (LEAF_WARPS - 1)], s_hscore[(threadIdx.x >> 5) & (LEAF_WARPS - 1)], 0u,
                       (uint32_t)LEAF_HS};
    const ScoreView &sc = a.sc;
    const int32_t u = -sc.ss, oe = sc.sg + sc.ss, g = sc.gmax;
    const int64_t cap = a.cap;
    int32_t *wb = a.scratch + (int64_t)gw * 6 * cap;
    Buf R = {wb, wb + cap, wb + 2 * cap};
    Buf Rn = {wb + 3 * cap, wb + 4 * cap, wb + 5 * cap};
    const uint64_t jmask = (1ull << a.bj) - 1ull;
    unsigned long long st_rows = 0, st_ent = 0, st_t0 = 0, st_t1 = 0, st_t2 = 0, st_reused = 0;
    bool overflow = false;
    bool tail = a.nseg <= a.last_warps;   // few warps still walk

    while (!overflow) {
        // one lane reads the counter and the overflow flag, which other warps write meanwhile:
        // the whole warp goes on or stops together
        unsigned long long s = 0;
        if (lane == 0)
            s = *(volatile unsigned long long *)&a.stats->leaf_overflow ? (unsigned long long)a.nseg
                                                                        : atomicAdd(a.next_seg, 1ull);
        s = __shfl_sync(FULL, s, 0);
        if (s >= (unsigned long long)a.nseg) break;
        int64_t k = task_start(a, lane, (int64_t)s);
        const int64_t kend = task_start(a, lane, (int64_t)s + 1);
        if (k >= kend) continue;
        int64_t rlen = 0;
        int32_t p = -1, qid = -1, m = 0, H = 0;
        const uint8_t *P = nullptr;
        unsigned long long seg_steps = 0, seg_width = 0;
        const long long task_t0 = clock64();
        // R lives in registers (lane i holds entry i) while it has <= 32 entries
        bool inreg = false;
        int32_t rj = 0, rM = AE_NEG, rGa = AE_NEG;
        // text window: lane i holds T[tw_base + i] (one coalesced 32-byte load per
        // 32 positions instead of a dependent random read per step)
        int64_t tw_base = -64;
        uint32_t tw = 0;
        // key (query, text end) of injection k, the next one to merge
        int32_t nk_qid = -1, nk_e = -1;
        if (k < kend) {
            const Inject In = a.inj[a.order[k]];
            nk_qid = In.qid;
            nk_e = In.e;
        }
        // row length at which the walk moves to a block, now and once few warps still walk
        const int dense = a.esc_by_density && leaf_dense(a, nk_qid);
        const int32_t esc_last = a.esc_last[dense];
        int32_t esc_at = tail ? esc_last : a.esc_min[dense];
        while (true) {
            if (rlen == 0 && k < kend) {
                // ---- jump to a lone injected row: it is already a finished row
                const Inject I0 = a.inj[a.order[k]];
                int32_t q2 = -1, e2 = -1;
                if (k + 1 < kend) {
                    const Inject I1 = a.inj[a.order[k + 1]];
                    q2 = I1.qid;
                    e2 = I1.e;
                }
                if (I0.cnt <= 32 && !(q2 == I0.qid && e2 == I0.e)) {
                    p = I0.e;
                    if (I0.qid != qid) {
                        qid = I0.qid;
                        m = a.qv.m[qid];
                        H = a.qv.H[qid];
                        P = a.qv.codes + a.qv.off[qid];
                    }
                    rlen = I0.cnt;
                    if (lane < rlen) {
                        rj = a.lj[I0.off + lane];
                        rM = a.lM[I0.off + lane];
                        rGa = a.lGa[I0.off + lane];
                    }
                    inreg = true;
                    ++k;
                    nk_qid = q2;
                    nk_e = e2;
                    const uint32_t h = (lane < rlen && rM >= H) ? 1u : 0u;
                    const uint32_t hi = warp_incl_sum(h);
                    const uint32_t htot = __shfl_sync(FULL, hi, 31);
                    if (htot) {
                        bool staged, hok;
                        const uint64_t hbase = stage_reserve(hstage, a, lane, htot, staged, hok);
                        if (hok && h) {
                            const uint64_t kq = ((uint64_t)qid << (a.be + a.bj)) | ((uint64_t)(uint32_t)p << a.bj);
                            hit_put(hstage, a, staged, hbase + hi - 1, kq | ((uint64_t)rj & jmask), rM);
                        }
                    }
                    if (a.tiers && lane == 0) st_t0 += (unsigned long long)rlen;   // warp-uniform count
                    ++st_rows;
                    ++seg_steps;
                    st_ent += (unsigned long long)rlen;
                    continue;
                }
            }
            if (rlen > 0 && inreg && p + 1 < a.ix.n && !seq_end(a.ix, p)) {
                const bool inj_next = nk_qid == qid && nk_e == p + 1;
                if (!inj_next) {
                    // ---- fast step: gen + horizontal finish in registers
                    ++p;
                    if (p < tw_base || p >= tw_base + 32) {
                        tw_base = p;
                        tw = (p + lane < a.ix.n) ? a.ix.text[p + lane] : 0u;
                    }
                    const int c = (int)__shfl_sync(FULL, tw, (int)(p - tw_base));
                    const bool valid = lane < rlen;
                    int32_t j = valid ? rj : m, M = valid ? rM : AE_NEG, Ga = valid ? rGa : AE_NEG;
                    int32_t jn = __shfl_down_sync(FULL, j, 1);
                    if (lane + 1 >= rlen) jn = m;
                    int32_t pjv = __shfl_up_sync(FULL, j, 1), pMv = __shfl_up_sync(FULL, M, 1);
                    if (lane == 0) {
                        pjv = -2;
                        pMv = AE_NEG;
                    }
                    int32_t colA = m, MpA = AE_NEG, GaA = AE_NEG, MpB = AE_NEG, next_col = m;
                    int32_t Dp = AE_NEG, Dk = AE_NEG;
                    bool hasB = false;
                    if (valid) {
                        colA = j;
                        const int32_t tA = thr_of(j, m, H, g);
                        if (pjv + 1 == j && pMv > AE_NEG) {
                            const int32_t D = pMv + delta_of(sc, smat, c, P[j]);
                            Dp = D > tA ? D : AE_NEG;
                        }
                        const int32_t gap = gap_from_i32(M, Ga, sc.ss, oe);
                        GaA = gap > tA ? gap : AE_NEG;
                        MpA = max(Dp, GaA);
                        hasB = (j + 1 < m) && (j + 1 != jn);
                        if (hasB) {
                            const int32_t D = M + delta_of(sc, smat, c, P[j + 1]);
                            Dk = D > thr_of(j + 1, m, H, g) ? D : AE_NEG;
                            MpB = Dk;
                        }
                        next_col = jn;
                    }
                    const int32_t keyA = MpA > AE_NEG ? MpA + colA * u : AE_KNEG;
                    const int32_t keyB = MpB > AE_NEG ? MpB + (colA + 1) * u : AE_KNEG;
                    const int32_t incl = warp_incl_max(max(keyA, keyB));
                    int32_t excl = __shfl_up_sync(FULL, incl, 1);
                    if (lane == 0) excl = AE_KNEG;
                    SlotOut o;
                    slot_finish(colA, MpA, hasB, MpB, next_col, excl, incl, sc, m, H, u, valid, o);
                    const uint32_t nA = o.aliveA, nB = o.aliveB, nR = (uint32_t)o.run_len;
                    const uint32_t cn = nA + nB + nR;
                    const uint32_t ci = warp_incl_sum(cn);
                    const uint32_t tot = __shfl_sync(FULL, ci, 31);
                    // hits
                    const uint32_t hA = o.aliveA && o.MA >= H, hB = o.aliveB && o.MB >= H;
                    const uint32_t hc = hA + hB + (uint32_t)o.run_hits;
                    const uint32_t hi = warp_incl_sum(hc);
                    const uint32_t htot = __shfl_sync(FULL, hi, 31);
                    bool staged = true, hok = true;
                    uint64_t hbase = 0;
                    if (htot) hbase = stage_reserve(hstage, a, lane, htot, staged, hok);
                    const uint64_t kq = ((uint64_t)qid << (a.be + a.bj)) | ((uint64_t)(uint32_t)p << a.bj);
                    const uint64_t h0 = hbase + hi - hc;
                    if (hok) {
                        if (hA) hit_put(hstage, a, staged, h0, kq | ((uint64_t)colA & jmask), o.MA);
                        if (hB) hit_put(hstage, a, staged, h0 + hA, kq | ((uint64_t)(colA + 1) & jmask), o.MB);
                    }
                    if (a.tiers) {
                        if (o.aliveA) {
                            const int tier = (Dp > AE_NEG) + (GaA > AE_NEG) + (o.GbA > thr_of(colA, m, H, g));
                            st_t0 += tier <= 1;
                            st_t1 += tier == 2;
                            st_t2 += tier >= 3;
                        }
                        if (o.aliveB) {
                            if ((Dk > AE_NEG) && (o.GbB > thr_of(colA + 1, m, H, g))) ++st_t1; else ++st_t0;
                        }
                        st_t0 += nR;
                    }
                    const int64_t e0 = (int64_t)(ci - cn);
                    if (tot > cap) {
                        overflow = true;
                        break;
                    }
                    // run hits and (for rows wider than a warp) run entries, cooperatively
                    unsigned rmask = __ballot_sync(FULL, nR > 0);
                    const bool spill = tot > 32;
                    while (rmask) {
                        const int L = __ffs(rmask) - 1;
                        rmask &= rmask - 1;
                        const int32_t s0 = __shfl_sync(FULL, o.run_start, L);
                        const int32_t rl = __shfl_sync(FULL, o.run_len, L);
                        const int32_t rh = __shfl_sync(FULL, o.run_hits, L);
                        const int32_t K = __shfl_sync(FULL, incl, L);
                        const int64_t d0 = __shfl_sync(FULL, e0 + nA + nB, L);
                        const uint64_t hd = __shfl_sync(FULL, h0 + hA + hB, L);
                        for (int32_t t = lane; t < rl; t += 32) {
                            const int32_t cc = s0 + t;
                            const int32_t v = sc.sg - cc * u + K;
                            if (spill) {
                                R.j[d0 + t] = cc;
                                R.M[d0 + t] = v;
                                R.Ga[d0 + t] = AE_NEG;
                            }
                            if (t < rh && hok) hit_put(hstage, a, staged, hd + t, kq | ((uint64_t)cc & jmask), v);
                        }
                    }
                    if (spill) {
                        if (o.aliveA) {
                            R.j[e0] = colA;
                            R.M[e0] = o.MA;
                            R.Ga[e0] = GaA;
                        }
                        if (o.aliveB) {
                            R.j[e0 + nA] = colA + 1;
                            R.M[e0 + nA] = o.MB;
                            R.Ga[e0 + nA] = AE_NEG;
                        }
                        inreg = false;
                    } else {
                        // output lane <- the lane whose slots/run produced output number `lane`
                        int s = 0;
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1) {
                            const uint32_t v = __shfl_sync(FULL, ci, s + step - 1);
                            if (v <= (uint32_t)lane) s += step;
                        }
                        const uint32_t ex_s = __shfl_sync(FULL, ci - cn, s);
                        const uint32_t nA_s = __shfl_sync(FULL, nA, s), nB_s = __shfl_sync(FULL, nB, s);
                        const int32_t col_s = __shfl_sync(FULL, colA, s), MA_s = __shfl_sync(FULL, o.MA, s);
                        const int32_t GaA_s = __shfl_sync(FULL, GaA, s), MB_s = __shfl_sync(FULL, o.MB, s);
                        const int32_t rs_s = __shfl_sync(FULL, o.run_start, s), K_s = __shfl_sync(FULL, incl, s);
                        const uint32_t r = (uint32_t)lane - ex_s;
                        if ((uint32_t)lane < tot) {
                            if (r < nA_s) {
                                rj = col_s;
                                rM = MA_s;
                                rGa = GaA_s;
                            } else if (r < nA_s + nB_s) {
                                rj = col_s + 1;
                                rM = MB_s;
                                rGa = AE_NEG;
                            } else {
                                rj = rs_s + (int32_t)(r - nA_s - nB_s);
                                rM = sc.sg - rj * u + K_s;
                                rGa = AE_NEG;
                            }
                        }
                    }
                    __syncwarp();
                    rlen = tot;
                    ++st_rows;
                    ++seg_steps;
                    st_ent += (unsigned long long)tot;
                    continue;
                }
            }
            if (inreg && rlen > 0) {   // the slow path reads R from scratch
                if (lane < rlen) {
                    R.j[lane] = rj;
                    R.M[lane] = rM;
                    R.Ga[lane] = rGa;
                }
                __syncwarp();
            }
            inreg = false;
            int64_t nlen = 0;   // length of the finished row at p, kept in Rn
            if (rlen == 0) {
                // a new walk: the row at p is the union of the rows injected there
                if (k >= kend) break;
                const Inject I0 = a.inj[a.order[k]];
                p = I0.e;
                if (I0.qid != qid) {
                    qid = I0.qid;
                    m = a.qv.m[qid];
                    H = a.qv.H[qid];
                    P = a.qv.codes + a.qv.off[qid];
                }
            } else {
                // the row ends with the text or its sequence: the walk goes on with
                // the next injection
                if (p + 1 >= a.ix.n || seq_end(a.ix, p)) {
                    rlen = 0;
                    continue;
                }
                ++p;
                if (p < tw_base || p >= tw_base + 32) {
                    tw_base = p;
                    tw = (p + lane < a.ix.n) ? a.ix.text[p + lane] : 0u;
                }
                const int c = (int)__shfl_sync(FULL, tw, (int)(p - tw_base));
                // ---- slots from R with letter c and the horizontal finish, straight
                // into Rn (the finished row at p) with its hits
                int32_t carry = AE_KNEG, prev_j = -2, prev_M = AE_NEG;
                // the next chunk's entries are loaded while this chunk is computed
                int32_t nj[E], nM[E], nG[E];
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int64_t x = (int64_t)lane * E + e;
                    const bool v = x < rlen;
                    nj[e] = v ? R.j[x] : m;
                    nM[e] = v ? R.M[x] : AE_NEG;
                    nG[e] = v ? R.Ga[x] : AE_NEG;
                }
                for (int64_t base = 0; base < rlen; base += 32 * E) {
                    const int64_t i0 = base + (int64_t)lane * E;
                    int32_t jj[E], MM[E], GG[E];
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        jj[e] = nj[e];
                        MM[e] = nM[e];
                        GG[e] = nG[e];
                        const int64_t x = i0 + 32 * E + e;
                        const bool v = x < rlen;
                        nj[e] = v ? R.j[x] : m;
                        nM[e] = v ? R.M[x] : AE_NEG;
                        nG[e] = v ? R.Ga[x] : AE_NEG;
                    }
                    // the first entry of the next chunk (lane 0's next load), m past the row
                    int32_t jnext = __shfl_down_sync(FULL, jj[0], 1);
                    const int32_t jfirst_next = __shfl_sync(FULL, nj[0], 0);
                    if (lane == 31) jnext = jfirst_next;
                    int32_t pj0 = __shfl_up_sync(FULL, jj[E - 1], 1), pM0 = __shfl_up_sync(FULL, MM[E - 1], 1);
                    if (lane == 0) {
                        pj0 = prev_j;
                        pM0 = prev_M;
                    }
                    Slots sl[E];
                    int32_t lk[E];   // the lane's keys up to and with entry e
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const bool v = i0 + e < rlen;
                        int32_t jn = e + 1 < E ? jj[e + 1 < E ? e + 1 : 0] : jnext;
                        if (i0 + e + 1 >= rlen) jn = m;
                        const int32_t pj = e ? jj[e ? e - 1 : 0] : pj0, pM = e ? MM[e ? e - 1 : 0] : pM0;
                        make_slots(sc, smat, c, P, m, H, g, oe, v, jj[e], MM[e], GG[e], pj, pM, jn, sl[e]);
                        const int32_t keyA = sl[e].MpA > AE_NEG ? sl[e].MpA + sl[e].colA * u : AE_KNEG;
                        const int32_t keyB = sl[e].MpB > AE_NEG ? sl[e].MpB + (sl[e].colA + 1) * u : AE_KNEG;
                        lk[e] = max(e ? lk[e ? e - 1 : 0] : AE_KNEG, max(keyA, keyB));
                    }
                    int32_t incl = warp_incl_max(lk[E - 1]);
                    int32_t excl = __shfl_up_sync(FULL, incl, 1);
                    if (lane == 0) excl = AE_KNEG;
                    incl = max(incl, carry);
                    excl = max(excl, carry);
                    SlotOut o[E];
                    int32_t ik[E];
                    uint32_t cl = 0, hl = 0;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int32_t ex = e ? max(excl, lk[e ? e - 1 : 0]) : excl;
                        ik[e] = max(excl, lk[e]);
                        slot_finish(sl[e].colA, sl[e].MpA, sl[e].hasB, sl[e].MpB, sl[e].next_col, ex, ik[e], sc, m, H,
                                    u, i0 + e < rlen, o[e]);
                        cl += (uint32_t)o[e].aliveA + (uint32_t)o[e].aliveB + (uint32_t)o[e].run_len;
                        hl += (uint32_t)(o[e].aliveA && o[e].MA >= H) + (uint32_t)(o[e].aliveB && o[e].MB >= H) +
                              (uint32_t)o[e].run_hits;
                    }
                    carry = __shfl_sync(FULL, incl, 31);
                    prev_j = __shfl_sync(FULL, jj[E - 1], 31);
                    prev_M = __shfl_sync(FULL, MM[E - 1], 31);
                    const uint32_t ci = warp_incl_sum(cl);
                    const uint32_t tot = __shfl_sync(FULL, ci, 31);
                    if (nlen + tot > cap) {
                        overflow = true;
                        break;
                    }
                    const uint32_t hi = warp_incl_sum(hl);
                    const uint32_t htot = __shfl_sync(FULL, hi, 31);
                    bool staged = true, hok = true;
                    uint64_t hbase = 0;
                    if (htot) hbase = stage_reserve(hstage, a, lane, htot, staged, hok);
                    const uint64_t kq = ((uint64_t)qid << (a.be + a.bj)) | ((uint64_t)(uint32_t)p << a.bj);
                    int64_t eo = nlen + (int64_t)(ci - cl);
                    uint64_t ho = hbase + hi - hl;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const uint32_t nA = o[e].aliveA, nB = o[e].aliveB, nR = (uint32_t)o[e].run_len;
                        const uint32_t hA = o[e].aliveA && o[e].MA >= H, hB = o[e].aliveB && o[e].MB >= H;
                        const int32_t j = jj[e];
                        if (nA) {
                            Rn.j[eo] = j;
                            Rn.M[eo] = o[e].MA;
                            Rn.Ga[eo] = sl[e].GaA;
                            if (hA && hok) hit_put(hstage, a, staged, ho, kq | ((uint64_t)j & jmask), o[e].MA);
                            if (a.tiers) {
                                const int tier = (sl[e].Dp > AE_NEG) + (sl[e].GaA > AE_NEG) + (o[e].GbA > thr_of(j, m, H, g));
                                st_t0 += tier <= 1;
                                st_t1 += tier == 2;
                                st_t2 += tier >= 3;
                            }
                        }
                        if (nB) {
                            Rn.j[eo + nA] = j + 1;
                            Rn.M[eo + nA] = o[e].MB;
                            Rn.Ga[eo + nA] = AE_NEG;
                            if (hB && hok) hit_put(hstage, a, staged, ho + hA, kq | ((uint64_t)(j + 1) & jmask), o[e].MB);
                            if (a.tiers) {
                                if ((sl[e].Dk > AE_NEG) && (o[e].GbB > thr_of(j + 1, m, H, g))) ++st_t1; else ++st_t0;
                            }
                        }
                        if (a.tiers) st_t0 += nR;
                        unsigned rmask = __ballot_sync(FULL, nR > 0);
                        while (rmask) {
                            const int L = __ffs(rmask) - 1;
                            rmask &= rmask - 1;
                            const int32_t s0 = __shfl_sync(FULL, o[e].run_start, L);
                            const int32_t rl = __shfl_sync(FULL, o[e].run_len, L);
                            const int32_t rh = __shfl_sync(FULL, o[e].run_hits, L);
                            const int32_t K = __shfl_sync(FULL, ik[e], L);
                            const int64_t d0 = __shfl_sync(FULL, eo + nA + nB, L);
                            const uint64_t hd = __shfl_sync(FULL, ho + hA + hB, L);
                            for (int32_t t = lane; t < rl; t += 32) {
                                const int32_t cc = s0 + t;
                                const int32_t v = sc.sg - cc * u + K;
                                Rn.j[d0 + t] = cc;
                                Rn.M[d0 + t] = v;
                                Rn.Ga[d0 + t] = AE_NEG;
                                if (t < rh && hok) hit_put(hstage, a, staged, hd + t, kq | ((uint64_t)cc & jmask), v);
                            }
                        }
                        eo += nA + nB + nR;
                        ho += hA + hB + (uint32_t)o[e].run_hits;
                    }
                    nlen += tot;
                }
                __syncwarp();
                if (overflow) break;
                st_ent += (unsigned long long)nlen;
            }
            leaf_merge<E == 2>(a, lane, qid, p, H, jmask, k, kend, Rn, nlen, cap, overflow, hstage, st_ent, st_reused, st_t0);
            if (overflow) break;
            if (k < kend) {
                const Inject In = a.inj[a.order[k]];
                nk_qid = In.qid;
                nk_e = In.e;
            } else {
                nk_qid = nk_e = -1;
            }
            Buf t = R;
            R = Rn;
            Rn = t;
            rlen = nlen;
            ++st_rows;
            ++seg_steps;
            seg_width = max(seg_width, (unsigned long long)nlen);
            // when tasks run out, warps fall idle while the last wide walks go on, and a block
            // each is the better use of the chip from narrower rows on.  A warp that finds no
            // task has counted next_seg past nseg.
            if (rlen > esc_last && esc_at > esc_last && (seg_steps & 7) == 0) {
                unsigned long long taken = 0;   // read once for the whole warp: the branches below are its
                if (lane == 0) taken = *(volatile unsigned long long *)a.next_seg;
                tail = (int64_t)__shfl_sync(FULL, taken, 0) >= a.nseg + max(a.nwarps - a.last_warps, 0);
                if (tail) esc_at = esc_last;
            }
            if (esc_at > 0 && rlen > esc_at) {
                // a wide row goes on on a whole block (k_leaf_wide), with the rest of
                // this task's injections; the warp takes its next task
                unsigned long long slot = 0, at = 0;
                if (lane == 0) {
                    // (a walk that finds no room leaves the counters past their ends; they are
                    // read first so that they cannot wrap)
                    slot = *(volatile unsigned long long *)a.esc_count;
                    at = *(volatile unsigned long long *)(a.esc_count + 1);
                    if (slot < (unsigned long long)(tail ? a.esc_max : a.esc_early) &&
                        at + rlen <= (unsigned long long)a.esc_pool_cap) {
                        at = atomicAdd(a.esc_count + 1, (unsigned long long)rlen);
                        slot = at + rlen <= (unsigned long long)a.esc_pool_cap ? atomicAdd(a.esc_count, 1ull)
                                                                               : (unsigned long long)a.esc_max;
                    } else {
                        slot = (unsigned long long)a.esc_max;
                    }
                }
                slot = __shfl_sync(FULL, slot, 0);
                at = __shfl_sync(FULL, at, 0);
                if (slot < (unsigned long long)a.esc_max) {
                    for (int64_t i = lane; i < rlen; i += 32) {
                        int32_t *x = a.esc_pool + 3 * ((int64_t)at + i);
                        x[0] = R.j[i];
                        x[1] = R.M[i];
                        x[2] = R.Ga[i];
                    }
                    if (lane == 0) {
                        EscWalk e;
                        e.qid = qid;
                        e.p = p;
                        e.rlen = rlen;
                        e.k = k;
                        e.kend = kend;
                        e.row = (int64_t)at;
                        a.esc[slot] = e;
                    }
                    __syncwarp();
                    rlen = 0;
                    k = kend;
                    continue;
                }
            }
            if (rlen <= 32) {
                if (lane < rlen) {
                    rj = R.j[lane];
                    rM = R.M[lane];
                    rGa = R.Ga[lane];
                }
                inreg = true;
            }
        }
        if (overflow && lane == 0) atomicAdd(&a.stats->leaf_overflow, 1ull);
        if (lane == 0) {
            atomicMax(&a.stats->leaf_max_steps, seg_steps);
            atomicMax(&a.stats->leaf_max_width, seg_width);
            atomicMax(&a.stats->leaf_max_cycles, (unsigned long long)(clock64() - task_t0));
        }
    }
    stage_flush(hstage, a, lane);
    unsigned long long t0 = st_t0, t1 = st_t1, t2 = st_t2;
    for (int d = 16; d > 0; d >>= 1) {
        t0 += __shfl_down_sync(FULL, t0, d);
        t1 += __shfl_down_sync(FULL, t1, d);
        t2 += __shfl_down_sync(FULL, t2, d);
    }
    if (lane == 0) {
        if (st_rows) atomicAdd(&a.stats->leaf_rows, st_rows);
        if (st_ent) {
            atomicAdd(&a.stats->entries, st_ent);
            atomicAdd(&a.stats->entries_leaf, st_ent);
        }
        if (t0) atomicAdd(&a.stats->tier[0], t0);
        if (t1) atomicAdd(&a.stats->tier[1], t1);
        if (t2) atomicAdd(&a.stats->tier[2], t2);
        if (st_reused) atomicAdd(&a.stats->reused, st_reused);
    }
}

// ------------------------------------------------------------------ wide sweep walks
//
// A walk whose row has grown wide is continued by a whole block: each step's
// entries are spread over the block's threads (WIDE_E consecutive entries
// each), the horizontal-gap keys and the output counts are block-wide scans.
// The values are those of the warp walk of k_leaf (the same make_slots /
// slot_finish per entry, the same merge); only the time per step differs.
//
// A walk is a chain of steps, one per text position, and a search waits for
// its longest one (thousands of positions along a homolog), so a step is built
// for latency: the two rows live in shared memory, a row of up to 512 entries
// is stepped one entry per thread, hits collect in a block-wide stage, and the
// next injections wait with their rows in a ring.  The rows injected at a
// position are looked up in the walked row by a warp each; those it dominates
// (nearly all along a homolog) are done with that, the others are merged by
// the whole block.  A row too long for shared memory moves to the block's
// buffers in global memory and back.  A step takes about 6,500 cycles at rows of
// 1,300 entries (load and slots 1,430, the key scan 820, finish 860, the count
// scan 1,110, writing 1,120, injected rows 1,100) and 3,800 at 200, where the
// warp walk takes 40,000 at 1,300; more entries per thread spill registers and
// are slower.
#ifndef AE_WIDE_T
#define AE_WIDE_T 512
#endif
constexpr int WIDE_T = AE_WIDE_T;     // threads
constexpr int WIDE_W = WIDE_T / 32;
constexpr int WIDE_E = 2;             // consecutive entries per thread at most
constexpr int WIDE_ROW = 6144;        // entries of a row in shared memory
constexpr int WIDE_HITS = 4096;       // staged hits
constexpr int WIDE_RING = 32;         // injections looked up ahead
constexpr int WIDE_RE = 8;            // entries of their rows held in the ring
constexpr int WIDE_HS = 64;           // hits staged by the merging warp

struct __align__(16) WideSmem {
    int32_t j[2][WIDE_ROW], M[2][WIDE_ROW], G[2][WIDE_ROW];
    int32_t hp[WIDE_HITS], hj[WIDE_HITS], hs[WIDE_HITS];   // hits: text position, column, score
    uint64_t mkey[WIDE_HS];
    int32_t mscore[WIDE_HS];
    __align__(16) int32_t smax[2][WIDE_W];
    __align__(16) uint32_t scnt[2][WIDE_W];
    __align__(16) uint32_t shit[2][WIDE_W];
    uint64_t roff[WIDE_RING];
    uint32_t rcnt[WIDE_RING];
    int32_t rqid[WIDE_RING], rpos[WIDE_RING];
    int32_t rj[WIDE_RING][WIDE_RE], rM[WIDE_RING][WIDE_RE], rG[WIDE_RING][WIDE_RE];
    int32_t dom[WIDE_RING];              // the walked row dominates the injected one
    int32_t mq[32], mM[32], mG[32];      // a merge: place in the row (new entries: ~place), values
    unsigned long long walk, hbase;
    int64_t nlen;
    int32_t overflow;
    int8_t mat[AE_MAX_SIGMA * AE_MAX_SIGMA];
};

// Over the values of the block's warps in sw: of those before warp w, and of all
__device__ __forceinline__ void wide_max(const int32_t *sw, int w, int32_t &pre, int32_t &all) {
    const int lane = threadIdx.x & 31;
    const int32_t v = lane < WIDE_W ? sw[lane] : AE_KNEG;
    pre = __reduce_max_sync(FULL, lane < w ? v : AE_KNEG);
    all = __reduce_max_sync(FULL, v);
}
__device__ __forceinline__ void wide_sum(const uint32_t *sw, int w, uint32_t &pre, uint32_t &all) {
    const int lane = threadIdx.x & 31;
    const uint32_t v = lane < WIDE_W ? sw[lane] : 0u;
    pre = __reduce_add_sync(FULL, lane < w ? v : 0u);
    all = __reduce_add_sync(FULL, v);
}

// The staged hits go out (all threads; hn is block-uniform)
__device__ __forceinline__ void wide_flush(const LeafArgs &a, WideSmem &s, int32_t qid, uint32_t &hn) {
    if (!hn) return;
    __syncthreads();
    if (threadIdx.x == 0) s.hbase = atomicAdd(a.hit_count, (unsigned long long)hn);
    __syncthreads();
    const uint64_t b = s.hbase;
    if (b + hn <= a.hit_cap) {
        const uint64_t kq = (uint64_t)qid << (a.be + a.bj);
        for (uint32_t i = threadIdx.x; i < hn; i += WIDE_T) {
            a.hit_key[b + i] = kq | ((uint64_t)(uint32_t)s.hp[i] << a.bj) | (uint64_t)(uint32_t)s.hj[i];
            a.hit_score[b + i] = s.hs[i];
        }
    } else if (threadIdx.x == 0) {
        atomicAdd(&a.stats->hit_overflow, 1ull);
    }
    __syncthreads();
    hn = 0;
}

__device__ __forceinline__ void wide_copy(const Buf &d, const Buf &r, int64_t n) {
    for (int64_t i = threadIdx.x; i < n; i += WIDE_T) {
        d.j[i] = r.j[i];
        d.M[i] = r.M[i];
        d.Ga[i] = r.Ga[i];
    }
}

__global__ void __launch_bounds__(WIDE_T, 1) k_leaf_wide(LeafArgs a) {
    extern __shared__ __align__(16) unsigned char wide_smem[];
    WideSmem &s = *reinterpret_cast<WideSmem *>(wide_smem);
    load_matrix(a.sc, s.mat);
    const unsigned long long nesc = min(*(volatile unsigned long long *)a.esc_count, (unsigned long long)a.esc_max);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    HitStage mstage = {s.mkey, s.mscore, 0u, (uint32_t)WIDE_HS};   // of the merging warp
    const ScoreView &sc = a.sc;
    const int32_t u = -sc.ss, oe = sc.sg + sc.ss, g = sc.gmax;
    const uint64_t jmask = (1ull << a.bj) - 1ull;
    int32_t *eb = a.wide_rows + (int64_t)blockIdx.x * 6 * a.wide_cap;
    // buffers 0 and 1: the rows in shared memory; 2 and 3: in global memory
    auto buf = [&](int x) {
        if (x < 2) return Buf{s.j[x], s.M[x], s.G[x]};
        int32_t *b = eb + (int64_t)(x - 2) * 3 * a.wide_cap;
        return Buf{b, b + a.wide_cap, b + 2 * (int64_t)a.wide_cap};
    };
    unsigned long long st_rows = 0, st_ent = 0, st_reused = 0, st_t0 = 0, width = 0;
    const long long t_start = clock64();
    bool stop = false;
    while (!stop) {
        // ---- the next walk handed on
        if (threadIdx.x == 0) {
            s.walk = *(volatile unsigned long long *)&a.stats->wide_overflow ? nesc : atomicAdd(a.esc_count + 2, 1ull);
            s.overflow = 0;
        }
        __syncthreads();
        if (s.walk >= nesc) break;
        const EscWalk e0 = a.esc[s.walk];
        const int64_t kend = e0.kend;
        int64_t k = e0.k, rlen = e0.rlen, ring = k;   // ring: first injection the ring holds
        int32_t p = e0.p;
        int32_t qid = e0.qid, m = a.qv.m[qid], H = a.qv.H[qid];
        const uint8_t *P = a.qv.codes + a.qv.off[qid];
        int cur = 0;                 // the row's buffer
        uint32_t hn = 0;             // staged hits
        if (rlen > WIDE_ROW) cur = 2;
        if (rlen > (cur ? (int64_t)a.wide_cap : (int64_t)WIDE_ROW)) {
            stop = true;
            break;
        }
        {
            const Buf B = buf(cur);
            for (int64_t i = threadIdx.x; i < rlen; i += WIDE_T) {
                const int32_t *x = a.esc_pool + 3 * (e0.row + i);
                B.j[i] = x[0];
                B.M[i] = x[1];
                B.Ga[i] = x[2];
            }
        }
        auto fill_ring = [&]() {     // injections [ring, ring + WIDE_RING)
            if (threadIdx.x < WIDE_RING) {
                const int64_t x = ring + threadIdx.x;
                s.rqid[threadIdx.x] = -1;
                if (x < kend) {
                    const Inject I = a.inj[a.order[x]];
                    s.rqid[threadIdx.x] = I.qid;
                    s.rpos[threadIdx.x] = I.e;
                    s.rcnt[threadIdx.x] = I.cnt;
                    s.roff[threadIdx.x] = I.off;
                }
            }
            __syncthreads();
            if (threadIdx.x < WIDE_RING * WIDE_RE) {
                const int r = threadIdx.x / WIDE_RE, x = threadIdx.x % WIDE_RE;
                if (s.rqid[r] >= 0 && (uint32_t)x < s.rcnt[r]) {
                    const uint64_t o = s.roff[r] + x;
                    s.rj[r][x] = a.lj[o];
                    s.rM[r][x] = a.lM[o];
                    s.rG[r][x] = a.lGa[o];
                }
            }
            __syncthreads();
        };
        // entry x of ring row r
        auto inj_entry = [&](int r, uint32_t x, int32_t &y, int32_t &M, int32_t &G) {
            if (x < WIDE_RE) {
                y = s.rj[r][x];
                M = s.rM[r][x];
                G = s.rG[r][x];
            } else {
                const uint64_t o = s.roff[r] + x;
                y = a.lj[o];
                M = a.lM[o];
                G = a.lGa[o];
            }
        };
        fill_ring();
        unsigned long long steps = 0;
        int ph = 0;                  // the scans' buffers alternate
        int c_next = p + 1 < a.ix.n ? (int)a.ix.text[p + 1] : 0;
        bool again = false;          // a step repeated in global memory
        while (true) {
            int64_t nlen = 0;
            int nxt = cur ^ 1;
            if (rlen == 0) {
                // a new walk: the row at p is the union of the rows injected there
                if (k >= kend) break;
                if (k >= ring + WIDE_RING) {
                    __syncthreads();
                    ring = k;
                    fill_ring();
                }
                p = s.rpos[k - ring];
                if (s.rqid[k - ring] != qid) {
                    wide_flush(a, s, qid, hn);   // staged hits are of one query
                    qid = s.rqid[k - ring];
                    m = a.qv.m[qid];
                    H = a.qv.H[qid];
                    P = a.qv.codes + a.qv.off[qid];
                }
                nxt = 0;
                c_next = p + 1 < a.ix.n ? (int)a.ix.text[p + 1] : 0;
            } else {
                if (!again) {
                    if (p + 1 >= a.ix.n || seq_end(a.ix, p)) {   // the walk ends with the text or its sequence
                        rlen = 0;
                        continue;
                    }
                    ++p;
                }
                again = false;
                const int c = c_next;
                const int c_after = p + 1 < a.ix.n ? (int)a.ix.text[p + 1] : 0;   // used one step on
                const Buf R = buf(cur), Rn = buf(nxt);
                const int64_t cap = cur < 2 ? (int64_t)WIDE_ROW : (int64_t)a.wide_cap;
                int32_t carry = AE_KNEG;
                bool full = false;
                // one chunk of the row: T * E entries from `base` on
                auto chunk = [&](int64_t base, auto ec) {
                    constexpr int E = decltype(ec)::value;
                    const int64_t i0 = base + (int64_t)threadIdx.x * E;
                    int32_t jj[E], MM[E], GG[E];
                    int32_t jnext = m, pj0 = -2, pM0 = AE_NEG;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        jj[e] = m;
                        MM[e] = GG[e] = AE_NEG;
                    }
                    if (i0 < rlen) {
#pragma unroll
                        for (int e = 0; e < E; ++e)
                            if (i0 + e < rlen) {
                                jj[e] = R.j[i0 + e];
                                MM[e] = R.M[i0 + e];
                                GG[e] = R.Ga[i0 + e];
                            }
                        if (i0 + E < rlen) jnext = R.j[i0 + E];
                        if (i0 > 0) {
                            pj0 = R.j[i0 - 1];
                            pM0 = R.M[i0 - 1];
                        }
                    }
                    // warps past the row only take part in the scans
                    const bool active = base + (int64_t)wid * 32 * E < rlen;
                    Slots sl[E];
                    int32_t lk[E];
#pragma unroll
                    for (int e = 0; e < E; ++e) lk[e] = AE_KNEG;
                    if (active)
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int32_t jn = (e + 1 < E) ? jj[e + 1] : jnext;
                        const int32_t pj = e ? jj[e - 1] : pj0, pM = e ? MM[e - 1] : pM0;
                        make_slots(sc, s.mat, c, P, m, H, g, oe, i0 + e < rlen, jj[e], MM[e], GG[e], pj, pM, jn, sl[e]);
                        const int32_t keyA = sl[e].MpA > AE_NEG ? sl[e].MpA + sl[e].colA * u : AE_KNEG;
                        const int32_t keyB = sl[e].MpB > AE_NEG ? sl[e].MpB + (sl[e].colA + 1) * u : AE_KNEG;
                        lk[e] = max(e ? lk[e - 1] : AE_KNEG, max(keyA, keyB));
                    }
                    const int32_t kincl = active ? warp_incl_max(lk[E - 1]) : AE_KNEG;
                    if (lane == 31) s.smax[ph][wid] = kincl;
                    int32_t lexcl = __shfl_up_sync(FULL, kincl, 1);
                    if (lane == 0) lexcl = AE_KNEG;
                    __syncthreads();
                    {
                        int32_t pre, all;
                        wide_max(s.smax[ph], wid, pre, all);
                        lexcl = max(max(lexcl, pre), carry);
                        carry = max(carry, all);
                    }
                    SlotOut o[E];
                    uint32_t cl = 0, hl = 0;
                    int32_t ik[E];
                    if (active)
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int32_t ex = e ? max(lexcl, lk[e - 1]) : lexcl;
                        ik[e] = max(lexcl, lk[e]);
                        slot_finish(sl[e].colA, sl[e].MpA, sl[e].hasB, sl[e].MpB, sl[e].next_col, ex, ik[e], sc, m, H, u,
                                    i0 + e < rlen, o[e]);
                        cl += (uint32_t)o[e].aliveA + (uint32_t)o[e].aliveB + (uint32_t)o[e].run_len;
                        hl += (uint32_t)(o[e].aliveA && o[e].MA >= H) + (uint32_t)(o[e].aliveB && o[e].MB >= H) +
                              (uint32_t)o[e].run_hits;
                    }
                    uint32_t ci = 0, hi = 0;
                    if (active) {
                        if (__any_sync(FULL, cl > 1023u)) {   // (no lane has more hits than outputs)
                            ci = warp_incl_sum(cl);
                            hi = warp_incl_sum(hl);
                        } else {
                            const uint32_t x = warp_incl_sum(cl | (hl << 16));
                            ci = x & 0xFFFFu;
                            hi = x >> 16;
                        }
                    }
                    if (lane == 31) {
                        s.scnt[ph][wid] = ci;
                        s.shit[ph][wid] = hi;
                    }
                    __syncthreads();
                    uint32_t cpre, ctot, hpre, htot;
                    wide_sum(s.scnt[ph], wid, cpre, ctot);
                    wide_sum(s.shit[ph], wid, hpre, htot);
                    ph ^= 1;
                    if (nlen + (int64_t)ctot > cap) {   // block-uniform
                        full = true;
                        return;
                    }
                    // hits: to the stage, or straight out where one chunk has more than it holds
                    if (hn + htot > WIDE_HITS) wide_flush(a, s, qid, hn);
                    const bool direct = htot > WIDE_HITS;
                    uint64_t ho = hn + hpre + hi - hl;
                    bool hok = true;
                    if (direct) {
                        if (threadIdx.x == 0) s.hbase = atomicAdd(a.hit_count, (unsigned long long)htot);
                        __syncthreads();
                        ho += s.hbase;
                        hok = s.hbase + htot <= a.hit_cap;
                        if (!hok && threadIdx.x == 0) atomicAdd(&a.stats->hit_overflow, 1ull);
                        __syncthreads();
                    } else {
                        hn += htot;
                    }
                    const uint64_t kq = ((uint64_t)qid << (a.be + a.bj)) | ((uint64_t)(uint32_t)p << a.bj);
                    auto put = [&](int32_t col, int32_t v) {
                        if (!direct) {
                            s.hp[ho] = p;
                            s.hj[ho] = col;
                            s.hs[ho] = v;
                        } else if (hok) {
                            a.hit_key[ho] = kq | ((uint64_t)col & jmask);
                            a.hit_score[ho] = v;
                        }
                        ++ho;
                    };
                    int64_t eo = nlen + (int64_t)(cpre + ci - cl);
                    if (active)
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int32_t colA = sl[e].colA;
                        if (o[e].aliveA) {
                            Rn.j[eo] = colA;
                            Rn.M[eo] = o[e].MA;
                            Rn.Ga[eo] = sl[e].GaA;
                            ++eo;
                            if (o[e].MA >= H) put(colA, o[e].MA);
                        }
                        if (o[e].aliveB) {
                            Rn.j[eo] = colA + 1;
                            Rn.M[eo] = o[e].MB;
                            Rn.Ga[eo] = AE_NEG;
                            ++eo;
                            if (o[e].MB >= H) put(colA + 1, o[e].MB);
                        }
                        for (int32_t r = 0; r < o[e].run_len; ++r) {
                            const int32_t cc = o[e].run_start + r;
                            const int32_t v = sc.sg - cc * u + ik[e];
                            Rn.j[eo] = cc;
                            Rn.M[eo] = v;
                            Rn.Ga[eo] = AE_NEG;
                            ++eo;
                            if (r < o[e].run_hits) put(cc, v);
                        }
                    }
                    nlen += (int64_t)ctot;
                };
                if (rlen <= WIDE_T) {
                    chunk(0, std::integral_constant<int, 1>());
                } else {
                    for (int64_t base = 0; base < rlen && !full; base += WIDE_T * WIDE_E)
                        chunk(base, std::integral_constant<int, WIDE_E>());
                }
                if (full) {
                    // past shared memory: the step is done again in global memory (hits it
                    // staged already are reported twice, which the per-cell maximum removes);
                    // past the block's buffers there: reported, the host runs the sweep again
                    if (cur >= 2 || rlen > a.wide_cap) {
                        stop = true;
                        break;
                    }
                    __syncthreads();
                    wide_copy(buf(2), buf(cur), rlen);
                    cur = 2;
                    again = true;
                    __syncthreads();
                    continue;
                }
                c_next = c_after;
                if (threadIdx.x == 0) st_ent += (unsigned long long)nlen;
                __syncthreads();   // the step's row is complete
            }
            // ---- the rows injected at (qid, p): those of the ring at once
            while (k < kend && !stop) {
                if (k >= ring + WIDE_RING) {
                    __syncthreads();
                    ring = k;
                    fill_ring();
                }
                const int r0 = (int)(k - ring);
                const bool here = r0 + lane < WIDE_RING && s.rqid[r0 + lane] == qid && s.rpos[r0 + lane] == p;
                const int nin = __ffs(~__ballot_sync(FULL, here)) - 1 < 0 ? 32 : __ffs(~__ballot_sync(FULL, here)) - 1;
                if (nin == 0) break;
                // an injected row whose every entry the walked row already has with M and G_a
                // at least as large changes nothing
                {
                    const Buf Rn = buf(nxt);
                    for (int r = r0 + wid; r < r0 + nin; r += WIDE_W) {
                        bool ok = nlen > 0;
                        for (uint32_t x = lane; x < s.rcnt[r] && ok; x += 32) {
                            int32_t y, M, G;
                            inj_entry(r, x, y, M, G);
                            // along a homolog the row's columns are consecutive: look there first
                            int64_t q = (int64_t)y - Rn.j[0];
                            if (q < 0 || q >= nlen || Rn.j[q] != y) q = lower_bound_g(Rn.j, nlen, y);
                            ok = q < nlen && Rn.j[q] == y && Rn.M[q] >= M && Rn.Ga[q] >= G;
                        }
                        ok = __all_sync(FULL, ok);
                        if (lane == 0) s.dom[r] = ok;
                    }
                }
                __syncthreads();
                for (int r = r0; r < r0 + nin && !stop; ++r, ++k) {
                    const uint32_t icnt = s.rcnt[r];
                    if (s.dom[r]) {
                        if (threadIdx.x == 0) st_reused += icnt;
                        continue;
                    }
                    if (icnt <= 32 && nxt < 2 && nlen + (int64_t)icnt <= WIDE_ROW) {
                        // ---- the union by maximum, into the other row buffer
                        if (hn + 32 > WIDE_HITS) wide_flush(a, s, qid, hn);
                        const Buf A = buf(nxt), D = buf(nxt ^ 1);
                        int32_t y = 0, M = AE_NEG, G = AE_NEG;
                        int64_t q = 0;
                        bool fresh = false, hit = false;
                        if ((uint32_t)lane < icnt) {
                            inj_entry(r, lane, y, M, G);
                            q = lower_bound_g(A.j, nlen, y);
                            fresh = !(q < nlen && A.j[q] == y);
                            hit = M >= H && (fresh || M > A.M[q]);
                        }
                        const unsigned bf = __ballot_sync(FULL, fresh), bh = __ballot_sync(FULL, hit);
                        const unsigned lt = (1u << lane) - 1u;
                        if (wid == 0) {
                            if ((uint32_t)lane < icnt) {
                                s.mq[lane] = fresh ? ~(int32_t)q : (int32_t)q;
                                s.mM[lane] = M;
                                s.mG[lane] = G;
                                if (fresh) {
                                    const int64_t d = q + __popc(bf & lt);
                                    D.j[d] = y;
                                    D.M[d] = M;
                                    D.Ga[d] = G;
                                }
                            }
                            if (hit) {
                                const uint32_t h = hn + __popc(bh & lt);
                                s.hp[h] = p;
                                s.hj[h] = y;
                                s.hs[h] = M;
                            }
                        }
                        hn += __popc(bh);
                        __syncthreads();
                        for (int64_t x = threadIdx.x; x < nlen; x += WIDE_T) {
                            int32_t Mx = A.M[x], Gx = A.Ga[x];
                            int64_t d = x;
                            for (uint32_t l = 0; l < icnt; ++l) {
                                const int32_t z = s.mq[l];
                                if (z < 0) {
                                    d += ~z <= x ? 1 : 0;   // a new entry goes before this one
                                } else if (z == x) {
                                    Mx = max(Mx, s.mM[l]);
                                    Gx = max(Gx, s.mG[l]);
                                }
                            }
                            D.j[d] = A.j[x];
                            D.M[d] = Mx;
                            D.Ga[d] = Gx;
                        }
                        nlen += __popc(bf);
                        if (threadIdx.x == 0) {
                            st_ent += __popc(bf);
                            st_reused += icnt - __popc(bf);
                        }
                        nxt ^= 1;
                        __syncthreads();
                        continue;
                    }
                    // long rows: the first warp merges, through the block's buffers in global memory
                    if (nxt < 2 && nlen <= a.wide_cap) {
                        wide_copy(buf(2), buf(nxt), nlen);
                        nxt = 2;
                        __syncthreads();
                    }
                    if (wid == 0) {
                        bool ovf = nxt < 2;   // longer than the buffers: reported
                        int64_t kk = k, nl = nlen;
                        if (!ovf)
                            leaf_merge<true>(a, lane, qid, p, H, jmask, kk, k + 1, buf(nxt), nl, (int64_t)a.wide_cap, ovf, mstage,
                                       st_ent, st_reused, st_t0);
                        if (lane == 0) {
                            s.nlen = nl;
                            if (ovf) s.overflow = 1;
                        }
                    }
                    __syncthreads();
                    if (s.overflow) {
                        stop = true;
                        break;
                    }
                    nlen = s.nlen;
                    __syncthreads();
                }
                __syncthreads();   // the ring's flags are read before the next group's are written
            }
            if (stop) break;
            cur = nxt;
            rlen = nlen;
            if (cur >= 2 && rlen <= WIDE_ROW / 2) {   // back to shared memory
                wide_copy(buf(0), buf(cur), rlen);
                cur = 0;
                __syncthreads();
            }
            ++st_rows;
            ++steps;
            width = max(width, (unsigned long long)rlen);
        }
        wide_flush(a, s, qid, hn);
        if (threadIdx.x == 0) atomicMax(&a.stats->leaf_max_steps, steps);
        __syncthreads();
    }
    if (wid == 0) stage_flush(mstage, a, lane);
    if (threadIdx.x == 0) {
        if (stop) atomicAdd(&a.stats->wide_overflow, 1ull);
        if (st_rows) atomicAdd(&a.stats->leaf_rows, st_rows);
        if (st_ent) {
            atomicAdd(&a.stats->entries, st_ent);
            atomicAdd(&a.stats->entries_leaf, st_ent);
        }
        if (st_reused) atomicAdd(&a.stats->reused, st_reused);
        atomicMax(&a.stats->leaf_max_width, width);
        atomicMax(&a.stats->leaf_max_cycles, (unsigned long long)(clock64() - t_start));
    }
}

// ------------------------------------------------------------------ locate + reduce

__global__ void k_locate_counts(const RangeHit *rh, int64_t n, uint32_t *cnt) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        cnt[t] = rh[t].hi - rh[t].lo;
}

__global__ void k_locate(const RangeHit *rh, int64_t n, const uint64_t *off, int64_t total, const int32_t *tend,
                         int be, int bj, uint64_t *key, int32_t *score) {
    const uint64_t jmask = (1ull << bj) - 1ull;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n;  // largest r with off[r] <= t
        while (hi - lo > 1) {
            int64_t mid = (lo + hi) >> 1;
            if ((int64_t)off[mid] <= t) lo = mid; else hi = mid;
        }
        const RangeHit r = rh[lo];
        const int64_t row = r.lo + (t - (int64_t)off[lo]);
        const int32_t e = tend[row];
        key[t] = ((uint64_t)(uint32_t)r.qid << (be + bj)) | ((uint64_t)(uint32_t)e << bj) | ((uint64_t)r.j & jmask);
        score[t] = r.score;
    }
}

// Keys (query, text end, query end) of result records to merge, their scores as values.
__global__ void k_merge_keys(const ae_hit *hits, const int32_t *qid, int64_t N, int be, int bj, uint64_t *key,
                             uint32_t *val) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N; t += (int64_t)gridDim.x * blockDim.x) {
        const ae_hit h = hits[t];
        key[t] = ((uint64_t)(uint32_t)qid[t] << (be + bj)) | ((uint64_t)h.text_end << bj) | (uint64_t)(uint32_t)h.query_end;
        val[t] = (uint32_t)h.score;
    }
}

__global__ void k_unique_flags(const uint64_t *key, int64_t N, uint32_t *flags) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N; t += (int64_t)gridDim.x * blockDim.x)
        flags[t] = (t == 0 || key[t] != key[t - 1]) ? 1u : 0u;
}

__global__ void k_unique_write(const uint64_t *key, const int32_t *score, int64_t N, const uint64_t *off, int be,
                               int bj, ae_hit *out, unsigned long long *qcount) {
    const uint64_t jmask = (1ull << bj) - 1ull, emask = (1ull << be) - 1ull;
    const int lane = threadIdx.x & 31;
    // the loop bound is uniform over a warp, so every lane reaches the per-query vote
    for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x; t0 < N; t0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = t0 + threadIdx.x;
        uint32_t q = 0xFFFFFFFFu;   // the query of a cell's first record, else none
        if (t < N) {
            const uint64_t k = key[t];
            if (!(t > 0 && key[t - 1] == k)) {
                int32_t best = score[t];
                for (int64_t u = t + 1; u < N && key[u] == k; ++u) best = max(best, score[u]);
                ae_hit h;
                h.text_end = (int64_t)((k >> bj) & emask);
                h.query_end = (int32_t)(k & jmask);
                h.score = best;
                out[off ? off[t] : t] = h;   // off NULL: the records are unique already
                q = (uint32_t)(k >> (be + bj));
            }
        }
        // per-query counts: one atomic per query present in the warp (the records are
        // sorted by query, so a warp usually holds one or two)
        const unsigned grp = __match_any_sync(FULL, q);
        if (q != 0xFFFFFFFFu && lane == __ffs(grp) - 1) atomicAdd(&qcount[q], (unsigned long long)__popc(grp));
    }
}

__global__ void k_unique_compact(const uint64_t *key, const int32_t *score, int64_t N, const uint64_t *off,
                                 uint64_t *okey, int32_t *oscore) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N; t += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = key[t];
        if (t > 0 && key[t - 1] == k) continue;
        int32_t best = score[t];
        for (int64_t u = t + 1; u < N && key[u] == k; ++u) best = max(best, score[u]);
        okey[off[t]] = k;
        oscore[off[t]] = best;
    }
}

inline unsigned grid_for(int64_t n, int threads, int64_t cap = 152 * 64) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

}  // namespace

// ------------------------------------------------------------------ launch wrappers

int64_t ae_launches_read() { return g_launches; }


int64_t ae_scan_tmp_words(int64_t N, int W) {
    int64_t words = 0;
    while (N > SC_TILE) {
        int64_t nb = (N + SC_TILE - 1) / SC_TILE;
        words += 2 * nb * W;
        N = nb;
    }
    return words + 8;
}

void ae_scan_u32(const uint32_t *const *in, uint64_t *const *out, int W, int64_t N, uint64_t *totals,
                 uint64_t *tmp, cudaStream_t st) {
    switch (W) {
        case 1: scan_rec<uint32_t, 1>(in, out, N, totals, tmp, st); break;
        case 2: scan_rec<uint32_t, 2>(in, out, N, totals, tmp, st); break;
        case 5: scan_rec<uint32_t, 5>(in, out, N, totals, tmp, st); break;
        default: break;
    }
}

int64_t ae_sort_tmp_words(int64_t N, bool halves) {
    // enough for any number of pairs up to N (short lists take smaller tiles)
    const int64_t half = halves ? std::min<int64_t>(N, AE_RS_SPLIT) : 0;
    const int64_t ntiles = std::max((N + RS_TILE - 1) / RS_TILE, (half + RS_TILE / 2 - 1) / (RS_TILE / 2));
    int64_t h = 256 * ntiles;
    // hist (u32, packed two per word) + offsets (u64) + scan tmp
    return (h + 1) / 2 + h + ae_scan_tmp_words(h, 1) + 8;
}

template <int I>
int rs_passes(uint64_t *k0, uint32_t *v0, uint64_t *k1, uint32_t *v1, int64_t N, int bits, uint64_t *tmp, cudaStream_t st) {
    const int smem = (int)sizeof(RsSmem<RS_T, I>);
    cudaFuncSetAttribute(k_rs_scatter<I>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    const int64_t ntiles = (N + RS_T * I - 1) / (RS_T * I);
    const int64_t h = 256 * ntiles;
    uint32_t *hist = reinterpret_cast<uint32_t *>(tmp);
    uint64_t *offs = tmp + (h + 1) / 2;
    uint64_t *stmp = offs + h;
    int which = 0;
    for (int shift = 0; shift < bits; shift += 8) {
        uint64_t *ki = which ? k1 : k0, *ko = which ? k0 : k1;
        uint32_t *vi = which ? v1 : v0, *vo = which ? v0 : v1;
        ++g_launches;
        k_rs_hist<I><<<(unsigned)ntiles, RS_T, 0, st>>>(ki, N, shift, hist, ntiles);
        const uint32_t *in[1] = {hist};
        uint64_t *out[1] = {offs};
        scan_rec<uint32_t, 1>(in, out, h, nullptr, stmp, st);
        ++g_launches;
        k_rs_scatter<I><<<(unsigned)ntiles, RS_T, smem, st>>>(ki, vi, ko, vo, N, shift, offs, ntiles);
        which ^= 1;
    }
    return which;
}

int ae_radix_sort(uint64_t *k0, uint32_t *v0, uint64_t *k1, uint32_t *v1, int64_t N, int bits, uint64_t *tmp,
                  cudaStream_t st, bool halves) {
    if (N <= 1 || bits <= 0) return 0;
    if (N <= RS_SMALL) {
        ++g_launches;
        const int smem = (int)sizeof(RsSmem<RS_ST, RS_SI>);
        cudaFuncSetAttribute(k_rs_small, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        k_rs_small<<<1, RS_ST, smem, st>>>(k0, v0, (int)N, bits);
        return 0;
    }
    return halves && N <= AE_RS_SPLIT ? rs_passes<RS_I / 2>(k0, v0, k1, v1, N, bits, tmp, st)
                            : rs_passes<RS_I>(k0, v0, k1, v1, N, bits, tmp, st);
}

void ae_encode_queries(const uint8_t *ascii, uint8_t *codes, int64_t total, int alphabet, int *bad,
                       cudaStream_t st) {
    if (total <= 0) return;
    ++g_launches;
    k_encode<<<grid_for(total, 256), 256, 0, st>>>(ascii, codes, total, alphabet, bad);
}

void ae_seed_keys(const SeedArgs &a, uint64_t *keys, uint32_t *vals, cudaStream_t st) {
    if (a.npos <= 0) return;
    ++g_launches;
    k_seed_keys<<<grid_for(a.npos, 256), 256, 0, st>>>(a, keys, vals);
}

void ae_seed_nodes(const SeedArgs &a, const uint64_t *keys, const uint32_t *vals, int64_t npos, int key_bits,
                   uint32_t *flags, uint64_t *flag_off, uint64_t *tmp, Node *nodes, int32_t *aj, int32_t *aM,
                   int32_t *aGa, uint64_t *nnodes_dev, cudaStream_t st) {
    (void)key_bits;
    if (npos <= 0) {
        cudaMemsetAsync(nnodes_dev, 0, sizeof(uint64_t), st);
        return;
    }
    ++g_launches;
    k_seed_flags<<<grid_for(npos, 256), 256, 0, st>>>(keys, npos, flags);
    const uint32_t *in[1] = {flags};
    uint64_t *out[1] = {flag_off};
    scan_rec<uint32_t, 1>(in, out, npos, nnodes_dev, tmp, st);
    ++g_launches;
    if (a.ix.sigma == 4)
        k_seed_nodes<4><<<grid_for(npos, 256), 256, 0, st>>>(a, keys, vals, npos, flags, flag_off, nodes, aj, aM, aGa);
    else
        k_seed_nodes<20><<<grid_for(npos, 256), 256, 0, st>>>(a, keys, vals, npos, flags, flag_off, nodes, aj, aM, aGa);
    ++g_launches;
    k_seed_fix<<<grid_for(npos, 256), 256, 0, st>>>(nodes, nnodes_dev, npos);
}

void ae_dom_table(const IndexView &ix, int d0, uint32_t *mask, cudaStream_t st) {
    const int bits = ix.sigma == 4 ? 2 : 5;
    const int64_t ngram = 1ll << (bits * d0);
    if (ix.n < d0) return;
    ++g_launches;
    const size_t smem = ngram <= 4096 ? (size_t)ngram * 4 : 0;
    k_dom_table<<<grid_for(ix.n, 256, 152 * 8), 256, smem, st>>>(ix, d0, bits, mask, ngram);
}

void ae_inject_keys(const Inject *inj, int64_t ninj, uint64_t *keys, uint32_t *vals, cudaStream_t st) {
    if (ninj <= 0) return;
    ++g_launches;
    k_inject_keys<<<grid_for(ninj, 256), 256, 0, st>>>(inj, ninj, keys, vals);
}

int ae_leaf_wide_blocks_per_sm() { return 1; }

int64_t ae_leaf_scratch_words(int32_t cap, int32_t nwarps) { return (int64_t)6 * cap * nwarps; }

void ae_leaf_cuts(const LeafArgs &a, const uint64_t *keys, uint2 *qrange, uint32_t *cuts, cudaStream_t st) {
    if (a.nseg <= 0) return;
    if (a.qrange) {
        ++g_launches;
        k_query_ranges<<<grid_for(a.ninj, 256), 256, 0, st>>>(keys, a.ninj, qrange);
    }
    ++g_launches;
    k_leaf_cuts<<<grid_for(a.nseg, 8), 256, 0, st>>>(a, keys, cuts);
}

void ae_leaf_sweep(const LeafArgs &a, int blocks, int threads, cudaStream_t st) {
    if (a.nseg <= 0) return;
    ++g_launches;
    if (a.few) k_leaf<2><<<blocks, threads, 0, st>>>(a);
    else k_leaf<1><<<blocks, threads, 0, st>>>(a);
    if (a.esc_max > 0) {   // the walks handed on to blocks
        ++g_launches;
        cudaFuncSetAttribute(k_leaf_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WideSmem));
        k_leaf_wide<<<a.wide_blocks, WIDE_T, sizeof(WideSmem), st>>>(a);
    }
}

void ae_locate_counts(const RangeHit *rh, int64_t nrh, uint32_t *cnt, cudaStream_t st) {
    if (nrh <= 0) return;
    ++g_launches;
    k_locate_counts<<<grid_for(nrh, 256), 256, 0, st>>>(rh, nrh, cnt);
}

void ae_locate(const RangeHit *rh, int64_t nrh, const uint64_t *off, int64_t total, const int32_t *tend, int be,
                 int bj, uint64_t *key, int32_t *score, cudaStream_t st) {
    if (total <= 0) return;
    ++g_launches;
    k_locate<<<grid_for(total, 256), 256, 0, st>>>(rh, nrh, off, total, tend, be, bj, key, score);
}

void ae_merge_keys(const ae_hit *hits, const int32_t *qid, int64_t N, int be, int bj, uint64_t *key, uint32_t *val,
                   cudaStream_t st) {
    if (N <= 0) return;
    ++g_launches;
    k_merge_keys<<<grid_for(N, 256), 256, 0, st>>>(hits, qid, N, be, bj, key, val);
}

void ae_unique_flags(const uint64_t *key, int64_t N, uint32_t *flags, cudaStream_t st) {
    if (N <= 0) return;
    ++g_launches;
    k_unique_flags<<<grid_for(N, 256), 256, 0, st>>>(key, N, flags);
}

void ae_unique_compact(const uint64_t *key, const int32_t *score, int64_t N, const uint64_t *flag_off, uint64_t *okey,
                       int32_t *oscore, cudaStream_t st) {
    if (N <= 0) return;
    ++g_launches;
    k_unique_compact<<<grid_for(N, 256), 256, 0, st>>>(key, score, N, flag_off, okey, oscore);
}

void ae_unique_write(const uint64_t *key, const int32_t *score, int64_t N, const uint64_t *flag_off, int be, int bj,
                     ae_hit *out, unsigned long long *qcount, cudaStream_t st) {
    if (N <= 0) return;
    ++g_launches;
    k_unique_write<<<grid_for(N, 256), 256, 0, st>>>(key, score, N, flag_off, be, bj, out, qcount);
}

// ------------------------------------------------------------------ suffix array by prefix doubling
//
// The suffix array of Section 2.3 (Section 5 (1) builds it over the reversed
// text), computed on the device by prefix doubling (Manber & Myers, 1993).
// Every suffix gets a key of its first L letters, b bits each (b for letters
// only: places past the text read 0), and a stable radix sort orders them.  A
// suffix's rank is the place of the first suffix with its key.  From then on
// only the suffixes that share their key are sorted (as Larsson & Sadakane,
// 2007, do): by (group, what follows h letters on), into the places their groups
// hold, which orders them by 2 h letters; new groups split and ranks follow.
// What follows h letters on is the rank there; a suffix that ends within h
// letters comes before all others of its key, shorter ones first.
//
// L is chosen so that about 1% of the suffixes of an i.i.d. text share a key:
// sorting these again costs less than a pass over all of them for longer keys.
// 10^7 letters: 4 passes over all suffixes and one round of some 10^4 of them
// (1.44 ms), where a 63-bit key and a 48-bit pair key for every suffix took 14
// passes (4.5 ms).  Only groups of several suffixes are numbered, so a text of few
// such groups sorts short pairs: 5 * 10^6 equal letters 8.7 ms, 12.8 with ranks as
// group numbers.  The flags and sums of a round lie over the sorted keys and the
// free pair, so that no other array of the text's length is needed.

namespace {

// s[k] = letter of the text (read backwards with `reversed`)
__global__ void k_sa_letters(const uint8_t *codes, int64_t n, int reversed, int sigma, uint8_t *s, int *bad) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const uint8_t c = codes[reversed ? n - 1 - k : k];
        if (c >= sigma) *bad = 1;
        s[k] = c;
    }
}

// key of suffix i: its first L letters, b bits each, first letter highest.  A
// thread takes eight suffixes in a row and reads their letters once.
constexpr int SA_KEYS = 8;
__global__ void __launch_bounds__(256) k_sa_first_keys(const uint8_t *s, int64_t n, int b, int L, uint64_t *keys,
                                                       uint32_t *vals) {
    const uint64_t mask = b * L >= 64 ? ~0ull : (1ull << (b * L)) - 1ull;
    const int64_t N = n + 1, nt = (N + SA_KEYS - 1) / SA_KEYS;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i0 = t * SA_KEYS;
        uint64_t key = 0;
        for (int x = 0; x < L - 1; ++x) key = (key << b) | (uint64_t)(i0 + x < n ? s[i0 + x] : 0);
        for (int q = 0; q < SA_KEYS && i0 + q < N; ++q) {
            const int64_t x = i0 + q + L - 1;
            key = ((key << b) | (uint64_t)(x < n ? s[x] : 0)) & mask;
            keys[i0 + q] = key;
            vals[i0 + q] = (uint32_t)(i0 + q);
        }
    }
}

// Of a sorted list of keys: whether a key is the first of several equal ones, and
// (upper half) whether it shares its value with a neighbour.  One scan adds up both.
__global__ void k_sa_groups(const uint64_t *keys, int64_t N, uint64_t *flags) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < N; p += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[p];
        const bool before = p > 0 && keys[p - 1] == k, after = p + 1 < N && keys[p + 1] == k;
        flags[p] = (uint64_t)(!before && after) | (uint64_t)(before || after) << 32;
    }
}

// The place in the suffix array of the first suffix of each group of several; the
// list's k-th element stands at place pos[k] (NULL: at k)
__global__ void k_sa_starts(const uint64_t *flags, const uint64_t *sums, const uint32_t *pos, int64_t N,
                            uint32_t *start) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < N; p += (int64_t)gridDim.x * blockDim.x)
        if ((uint32_t)flags[p]) start[(uint32_t)sums[p]] = pos ? pos[p] : (uint32_t)p;
}

// The list's suffixes at their places with their ranks.  The flags of an element
// that still shares its key become its group's number with its place in the
// upper half, vals[p] becomes 1 there and 0 elsewhere.
__global__ void k_sa_place(uint32_t *vals, uint64_t *flags, const uint64_t *sums, const uint32_t *start,
                           const uint32_t *pos, int64_t T, int64_t N, uint32_t *sa, uint32_t *rank, int *bad) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < T; p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = vals[p], at = pos ? pos[p] : (uint32_t)p;
        const uint64_t f = flags[p];
        const bool tied = f >> 32;
        vals[p] = tied;
        // the sum counts the groups that start before p: the element's own is that, or one less
        const uint32_t g = (uint32_t)sums[p] + (uint32_t)f - 1;
        if (tied) flags[p] = (uint64_t)g | ((uint64_t)at << 32);
        if ((int64_t)i >= N || (int64_t)at >= N) {
            *bad = 2;
            continue;
        }
        sa[at] = i;
        rank[i] = tied ? start[g] : at;
    }
}

// The next list: places and groups of the elements that are still tied
__global__ void k_sa_next(const uint32_t *tied, const uint64_t *sums, const uint64_t *group, int64_t T, uint32_t *pos,
                          uint32_t *ord) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < T; p += (int64_t)gridDim.x * blockDim.x)
        if (tied[p]) {
            const uint64_t o = sums[p] >> 32, g = group[p];
            pos[o] = (uint32_t)(g >> 32);
            ord[o] = (uint32_t)g;
        }
}

// keys of the tied suffixes (at places pos[0..T), in groups ord[0..T)) for the
// 2 h-letter order.  Groups are numbered along the list, in the order of their
// ranks: a text of few groups (one letter, a period) has short keys.
__global__ void k_sa_pair_keys(const uint32_t *sa, const uint32_t *pos, const uint32_t *ord, const uint32_t *rank, int64_t T,
                               int64_t n, int64_t h, int rb, uint64_t *keys, uint32_t *vals) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < T; p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = sa[pos[p]];
        const uint64_t second = i + h <= n ? (uint64_t)rank[i + h] + (uint64_t)h : (uint64_t)(n - i);
        keys[p] = ((uint64_t)ord[p] << rb) | second;
        vals[p] = i;
    }
}

int sa_bits_for(uint64_t maxval) {  // bits to hold values in [0, maxval]
    int b = 1;
    while (b < 64 && (maxval >> b) != 0) ++b;
    return b;
}

}  // namespace

ae_status ae_sa_doubling(const uint8_t *d_codes, int64_t n, int sigma, int reversed, int32_t *d_sa, int *rounds,
                         cudaStream_t st) {
    const int64_t N = n + 1;
    if (rounds) *rounds = 0;
    const int b = sa_bits_for((uint64_t)std::max(sigma - 1, 1));
    // letters of the first key: enough for about 100 N different ones, in whole passes
    int L = 1;
    for (double words = sigma; words < 100.0 * (double)N && (L + 1) * b <= 64; words *= std::max(sigma, 2)) ++L;
    L = std::min(64, (L * b + 7) / 8 * 8) / b;
    // one allocation for all buffers (ten of them cost 0.5 ms): 32 bytes a letter and the sort's
    const int64_t tmp_words = std::max(ae_sort_tmp_words(N), ae_scan_tmp_words(N, 1));
    const int64_t words = 2 * N + tmp_words + 2 + 2 * N;   // of eight bytes
    uint64_t *mem = nullptr;
    ae_status res = AE_OK;
    if (cudaMalloc(&mem, sizeof(uint64_t) * (size_t)words) != cudaSuccess) {
        cudaGetLastError();
        return AE_ENOMEM;
    }
    // total: groups of several and (upper half) tied suffixes, then an error flag
    uint64_t *k0 = mem, *k1 = k0 + N, *tmp = k1 + N, *total = tmp + tmp_words;
    uint32_t *v0 = reinterpret_cast<uint32_t *>(total + 2), *v1 = v0 + N, *rank = v1 + N, *pos = rank + N;
    int *bad = reinterpret_cast<int *>(total + 1);
    uint8_t *s = reinterpret_cast<uint8_t *>(k1);   // until the first sort
    int h_bad = 0;
    if (cudaMemsetAsync(total, 0, 2 * sizeof(uint64_t), st) != cudaSuccess) res = AE_ECUDA;
    if (res == AE_OK) {
        g_launches += 2;
        k_sa_letters<<<grid_for(n, 256), 256, 0, st>>>(d_codes, n, reversed, sigma, s, bad);
        k_sa_first_keys<<<grid_for((N + SA_KEYS - 1) / SA_KEYS, 256), 256, 0, st>>>(s, n, b, L, k0, v0);
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            res = AE_ECUDA;
        else if (h_bad)
            res = AE_EINVAL;
    }
    // (kr, vr): the sorted pairs of the current list; (kf, vf): the free pair
    uint64_t *kr = k0, *kf = k1;
    uint32_t *vr = v0, *vf = v1, *sa = reinterpret_cast<uint32_t *>(d_sa);
    int bits = b * L;
    int64_t h = L, T = N;   // T: length of the list, at first every suffix
    bool all = true;
    while (res == AE_OK) {
        if (ae_radix_sort(kr, vr, kf, vf, T, bits, tmp, st)) {
            std::swap(kr, kf);
            std::swap(vr, vf);
        }
        if (rounds) ++*rounds;
        // flags in the free keys, their sums over the sorted ones, which are done with; group
        // starts, and then the next list's groups, in the free values
        uint64_t *flags = kf, *sum = kr;
        const uint32_t *at = all ? nullptr : pos;
        g_launches += 4;
        k_sa_groups<<<grid_for(T, 256), 256, 0, st>>>(kr, T, flags);
        const uint64_t *in[1] = {flags};
        uint64_t *out[1] = {sum};
        scan_rec<uint64_t, 1>(in, out, T, total, tmp, st);
        k_sa_starts<<<grid_for(T, 256), 256, 0, st>>>(flags, sum, at, T, vf);
        k_sa_place<<<grid_for(T, 256), 256, 0, st>>>(vr, flags, sum, vf, at, T, N, sa, rank, bad);
        k_sa_next<<<grid_for(T, 256), 256, 0, st>>>(vr, sum, flags, T, pos, vf);
        uint64_t back[2] = {0, 0};
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(back, total, 2 * sizeof(uint64_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            res = AE_ECUDA;
            break;
        }
        const int64_t groups = (int64_t)(uint32_t)back[0], tied = (int64_t)(back[0] >> 32);
        if (back[1] || tied > T || 2 * groups > tied || (tied > 0 && groups < 1)) {
            res = AE_ECUDA;   // not a permutation: an internal error
            break;
        }
        if (tied == 0) break;
        if (!all && h / 2 >= N) {   // a round at h >= N orders everything left by its length
            res = AE_ECUDA;
            break;
        }
        T = tied;
        all = false;
        const int rb = sa_bits_for((uint64_t)(N - 1 + h));
        bits = rb + sa_bits_for((uint64_t)(groups - 1));
        if (bits > 64) {
            res = AE_EUNSUPPORTED;
            break;
        }
        ++g_launches;
        k_sa_pair_keys<<<grid_for(T, 256), 256, 0, st>>>(sa, pos, vf, rank, T, n, h, rb, kf, vr);
        std::swap(kr, kf);
        h *= 2;
    }
    if (res == AE_OK && cudaStreamSynchronize(st) != cudaSuccess) res = AE_ECUDA;
    if (res != AE_OK) cudaStreamSynchronize(st);
    cudaFree(mem);
    return res;
}
