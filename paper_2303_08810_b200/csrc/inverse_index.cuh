// Inverse routing index of one (image, routing head): for each key region the query regions whose rows list it, in
// entry order (query region, then slot) - the fixed order of the dK / dV sums - as CSR; and the key regions by falling
// length of their lists.  The dK / dV kernels start the longest first: where a map has a few kinds of content, the queries
// of a kind all pick the same few regions (2 x 100 x 167 tokens, S = 16: 264 us in map order, 172 us with evenly spread lists).
#pragma once

#include "bra_internal.h"

namespace bra {

constexpr int INVERSE_BITS_MAX = 40 * 1024;     // bytes of the bit matrix up to which it is used

inline int inverse_words(const Dims& d) { return (d.R + 31) / 32; }
inline bool inverse_uses_bits(const Dims& d) { return (size_t)d.R * inverse_words(d) * 4 <= INVERSE_BITS_MAX; }
// places in shared memory (words): counts [R + 1] and a flag, keys of the order, parts (where lists are cut: ListParts), bits
__host__ __device__ inline int inverse_key_at(int R) { return (R + 2 + 3) / 4 * 4; }
__host__ __device__ inline int inverse_bits_at(int R, bool cut) { return inverse_key_at(R) + (cut ? 2 : 1) * ((R + 3) / 4 * 4); }
inline size_t inverse_smem(const Dims& d, bool cut = false) {
    return sizeof(int32_t) * (inverse_bits_at(d.R, cut) + (inverse_uses_bits(d) ? (size_t)d.R * inverse_words(d) : 0));
}

// What the inverse index job writes besides the index, in place of the order, where lists are cut in parts (ListParts).
struct ListJobs {
    int2* jobs;             // [images, heads_i, p.jobs]: (region or -1, part)
    int32_t* done;          // counters to set to zero, `counters` per (image, routing head)
    int counters;
    ListParts p;
};

// The inverse index of the images of a piece.
struct InversePiece { int32_t *off, *list, *order; };
inline InversePiece inverse_piece(const Dims& d, const GridPiece& p, int32_t* off, int32_t* list, int32_t* order) {
    const size_t bh = (size_t)p.b0 * d.heads_i;
    return {off + bh * (d.R + 1), list + bh * d.R * d.topk, order + bh * d.R};
}
// Pieces of the dK / dV grids (heads, images, groups): all heads; `chunks` consecutive groups of warps are a region, several regions or a
// job (ListParts); launch(piece, g, groups) starts with the g-th of these in the order.
template <typename F>
inline cudaError_t group_pieces(const Dims& d, int groups, int chunks, F&& launch) {
    if (chunks > GRID_YZ) return cudaErrorInvalidConfiguration;        // (a region of millions of tokens)
    const int most = GRID_YZ / chunks * chunks;
    Dims images = d;
    images.heads = 1;                                       // x holds them all
    for (int g0 = 0; g0 < groups; g0 += most) {
        const cudaError_t e = grid_pieces(images, [&](GridPiece p) {
            p.heads = d.heads;
            p.stat = (size_t)p.b0 * d.heads * d.H0 * d.W0;
            return launch(p, g0 / chunks, groups - g0 < most ? groups - g0 : most);
        });
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// One CTA.  A row of the index seldom names a region twice, so what has to be inverted is a bit matrix (key region x
// query region): every entry sets a bit (atomics whose order does not matter), every key region counts and lists its
// bits in ascending order: work proportional to the entries, where comparing every entry with every region took
// 109 us at 256 regions, topk 4 and 41 us at 64 regions, topk 12.  A repeated entry (a caller's index may have them)
// or a matrix that does not fit: counts by atomics, then one warp puts the entries in their places in order, 32 at a time, the
// rank among equals of the 32 from a match.  (Every region comparing itself with every entry instead: 961 regions, topk 16,
// 2 heads, gradients 17.6 ms; 0.24 ms now.)
// Entries outside [0, R) are in no list.
__device__ __forceinline__ void inverse_index_job(const int32_t* __restrict__ index, int32_t* __restrict__ inv_off,
                                                  int32_t* __restrict__ inv_list, int32_t* __restrict__ order, int bh, int32_t* sm, bool use_bits, const Dims& dm,
                                                  const ListJobs& lj = {nullptr, nullptr, 0, {0, 0, 0, false}}) {
    const int tid = threadIdx.x, nthreads = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int entries = dm.R * dm.topk, words = (dm.R + 31) >> 5;
    const int32_t* idx = index + (size_t)bh * entries;
    int32_t* off = inv_off + (size_t)bh * (dm.R + 1);
    int32_t* list = inv_list + (size_t)bh * entries;
    int32_t* count = sm;                                    // [R + 1]
    // [R], then -1 to a multiple of four: 1024 times the length, less the region: a number per region (at most 1000 regions, lists of
    // at most 10^6 entries), greater than another's where the region comes before that one in the order
    int32_t* key = sm + inverse_key_at(dm.R);
    int32_t* parts = key + (dm.R + 3) / 4 * 4;              // [R], then 0 to a multiple of four
    uint32_t* bits = reinterpret_cast<uint32_t*>(sm + inverse_bits_at(dm.R, lj.p.most != 0));
    int* repeated = sm + dm.R + 1;                          // later: jobs
    bool by_bits = use_bits;
    if (lj.p.most)
        for (int e = tid; e < lj.counters; e += nthreads) lj.done[(size_t)bh * lj.counters + e] = 0;
    if (use_bits) {
        for (int e = tid; e < dm.R * words; e += nthreads) bits[e] = 0u;
        if (tid == 0) *repeated = 0;
        __syncthreads();
        for (int e = tid; e < entries; e += nthreads) {
            const int j = idx[e], i = e / dm.topk;
            if (j >= 0 && j < dm.R && (atomicOr(&bits[j * words + (i >> 5)], 1u << (i & 31)) >> (i & 31) & 1u)) *repeated = 1;
        }
        __syncthreads();
        by_bits = *repeated == 0;
    }
    if (by_bits) {
        for (int j = tid; j < dm.R; j += nthreads) {
            int n = 0;
            for (int w = 0; w < words; ++w) n += __popc(bits[j * words + w]);
            count[j] = n;
        }
    } else {
        for (int j = tid; j < dm.R; j += nthreads) count[j] = 0;
        __syncthreads();
        for (int e = tid; e < entries; e += nthreads) {
            const int j = idx[e];
            if (j >= 0 && j < dm.R) atomicAdd(count + j, 1);
        }
    }
    __syncthreads();
    if (warp == 0) {                                        // exclusive prefix sum
        int run = 0, jobs = 0;
        for (int j0 = 0; j0 < dm.R; j0 += 32) {
            const int j = j0 + lane, n = j < dm.R ? count[j] : 0;
            int incl = n;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, incl, s);
                if (lane >= s) incl += o;
            }
            if (j < dm.R) { count[j] = run + incl - n; key[j] = n * 1024 + 1023 - j; }
            if (lj.p.most) {
                const int m = j >= dm.R ? 0 : n > lj.p.most ? (n + lj.p.most - 1) / lj.p.most : 1;
                if (j < (dm.R + 3) / 4 * 4) parts[j] = m;
                jobs += m;
            }
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lj.p.most) jobs = __reduce_add_sync(0xffffffffu, jobs);
        if (lane == 0) { count[dm.R] = run; *repeated = jobs; }
        if (lane < 4 && dm.R + lane < (dm.R + 3) / 4 * 4) key[dm.R + lane] = -1;
    }
    __syncthreads();
    for (int j = tid; j <= dm.R; j += nthreads) off[j] = count[j];
    if (!lj.p.most) {
        for (int j = tid; j < dm.R; j += nthreads) {        // longest list first, ties to the lower region
            const int mine = key[j];
            int rank = 0;
            for (int o = 0; o < dm.R; o += 4) {
                const int4 k = *reinterpret_cast<const int4*>(key + o);
                rank += (k.x > mine) + (k.y > mine) + (k.z > mine) + (k.w > mine);
            }
            order[(size_t)bh * dm.R + rank] = j;
        }
    } else {
        int2* jobs = lj.jobs + (size_t)bh * lj.p.jobs;
        for (int j = tid; j < dm.R; j += nthreads) {        // the jobs in that order
            const int mine = key[j];
            int at = 0;
            for (int o = 0; o < dm.R; o += 4) {
                const int4 k = *reinterpret_cast<const int4*>(key + o), p = *reinterpret_cast<const int4*>(parts + o);
                at += (k.x > mine ? p.x : 0) + (k.y > mine ? p.y : 0) + (k.z > mine ? p.z : 0) + (k.w > mine ? p.w : 0);
            }
            for (int p = 0; p < parts[j]; ++p) jobs[at + p] = make_int2(j, p);
        }
        for (int e = *repeated + tid; e < lj.p.jobs; e += nthreads) jobs[e] = make_int2(-1, 0);
    }
    if (by_bits) {
        for (int j = tid; j < dm.R; j += nthreads) {
            int32_t* out = list + count[j];
            for (int w = 0; w < words; ++w)
                for (uint32_t m = bits[j * words + w]; m; m &= m - 1) *out++ = w * 32 + __ffs(m) - 1;
        }
    } else {
        __syncthreads();                                    // the offsets have been read: from here on the next free places
        if (warp != 0) return;
        int j = lane < entries ? idx[lane] : -1;
        for (int e0 = 0; e0 < entries; e0 += 32) {
            const int next = e0 + 32 + lane < entries ? idx[e0 + 32 + lane] : -1;
            const bool ok = j >= 0 && j < dm.R;
            const unsigned same = __match_any_sync(0xffffffffu, ok ? j : -1);
            const int at = ok ? count[j] : 0, rank = __popc(same & ((1u << lane) - 1u));
            if (ok) list[at + rank] = (e0 + lane) / dm.topk;
            __syncwarp();
            if (ok && rank == 0) count[j] = at + __popc(same);
            __syncwarp();
            j = next;
        }
    }
}

}  // namespace bra
