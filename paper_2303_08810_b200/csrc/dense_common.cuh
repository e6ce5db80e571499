// Shared by the kernels that attend to every token of a small map and weigh the scores by the routing index
// (attend_dense.cu, backward_dense.cu): bf16, head dim 32, at most 64 regions and 256 tokens.
//
// The late stages of a network route small regions to many others (2 x 2 tokens to 16 of 49 regions, single tokens to all
// 49).  A matrix tile of one region then uses 4 or 1 of its 16 rows.  Here a tile is any 16 tokens of the map and its keys
// are ALL tokens, masked by a 64-bit word per query region (bit j: the list names key region j).  A list with repeats (a
// caller's index may have them: they count twice) instead adds log2(count) to the scores.  Nothing is gathered and every
// warp of a CTA shares the slices, whose rows are the tokens region by region: with four tokens per region a mask bit
// covers the two columns a lane holds of an n-tile.
#pragma once

#include "direct_common.cuh"

namespace bra {

namespace dn {
constexpr int ST = 40;              // floats per staged token: eight rows of a fragment on different banks
}

struct DenseGeom {
    DirGeom g;                      // for the LCE: the whole map as one region, a chunk of its rows per CTA
    int rows, np;                   // tokens rounded up to 32 (slices), tiles of 16 per chunk
    int nw, rrc;                    // warps per CTA, region rows per chunk
    uint32_t mul_nr, mul_ws, mul_s, mul_k;
    int off_a, off_b, off_c, off_d; // slices
    int off_stat, off_mask, off_bias, off_reg, smem_bytes;
};

// slices: 2 (K, V) or 4 (Q, K, V, dO); a chunk is some rows of regions
inline DenseGeom dense_geom(const Dims& d, int slices, int region_rows) {
    DenseGeom q;
    q.rrc = region_rows;
    const int chunk_rows = region_rows * d.hs;
    DirGeom& g = q.g;
    g.planes = 1;
    g.hb = chunk_rows; g.chunks = (d.S + region_rows - 1) / region_rows;
    q.np = (chunk_rows * d.W + 15) / 16;
    q.nw = q.np <= 8 ? q.np : (q.np + 1) / 2;
    g.nw = q.nw; g.gpc = 1; g.gpi = g.chunks; g.tpc = q.np;
    g.halo_w = d.W + 4; g.halo_row = g.halo_w * 64 + 16;
    g.mul_hw = recip32(g.halo_w);
    q.mul_nr = recip32(d.n_r); q.mul_ws = recip32(d.ws); q.mul_s = recip32(d.S); q.mul_k = recip32(d.topk);
    q.rows = (d.N + 31) / 32 * 32;
    int off = 0;
    q.off_a = off; off += q.rows * 64;
    q.off_b = off; off += q.rows * 64;
    q.off_c = off; off += slices > 2 ? q.rows * 64 : 0;
    q.off_d = off; off += slices > 2 ? q.rows * 64 : 0;
    g.off_st = 0;                                                    // over the slices, once they have been read
    const int st = q.np * 16 * dn::ST * 4;
    if (off < st) off = st;
    g.off_halo = off; off += d.lce ? (chunk_rows + 7) * g.halo_row + 1024 : 0;   // tiles that stick out read (and discard) rows behind
    off = (off + 15) / 16 * 16;
    g.off_w = off;    off += d.lce ? 32 * 25 * 4 : 0;
    q.off_stat = off; off += slices > 2 ? q.rows * 8 : 0;
    q.off_mask = off; off += 2 * 64 * 8 + 16;
    q.off_bias = off; off += d.R * d.R * 4;
    q.off_reg = off;  off += q.rows;
    q.smem_bytes = off;
    return q;
}

inline bool dense_supported(const Dims& d, int dtype) {
    return dtype == BRA_BF16 && d.d == 32 && d.R <= 64 && d.N <= 256;
}

// slice row r, 16-byte chunk q: chunk index xor (r >> 1) & 3, conflict-free for ldmatrix and for 16-byte fragment reads
__device__ __forceinline__ uint32_t dense_at(int r, int q) { return r * 64 + ((q ^ ((r >> 1) & 3)) << 4); }

// token t (region by region) -> row and column of the padded map
__device__ __forceinline__ int2 dense_pos(const Dims& dm, const DenseGeom& gm, int t) {
    const int r = fdiv(t, dm.n_r, gm.mul_nr), tt = t - r * dm.n_r;
    const int ry = fdiv(r, dm.S, gm.mul_s), ty = fdiv(tt, dm.ws, gm.mul_ws);
    return make_int2((r - ry * dm.S) * dm.ws + tt - ty * dm.ws, ry * dm.hs + ty);
}
// 64-byte rows of a head for all tokens of the (padded) map; zeros in the padding and behind the last token
template <int SLICES>
__device__ __forceinline__ void dense_load_slices(const uint32_t (&dst)[SLICES], const uint8_t* const (&head)[SLICES], const Dims& dm,
                                                  const DenseGeom& gm, int tid, int nthreads) {
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
    for (int e = tid; e < gm.rows * 4; e += nthreads) {
        const int r = e >> 2, q = e & 3;
        const int2 at = dense_pos(dm, gm, r);
        const bool in = at.y < dm.H0 && at.x < dm.W0;
        const size_t off = in ? (size_t)(uint32_t)(at.y * dm.W0 + at.x) * tok_bytes + q * 16 : 0;
#pragma unroll
        for (int s = 0; s < SLICES; ++s) ptx::cp_async_16(dst[s] + dense_at(r, q), head[s] + off, in ? 16u : 0u);
    }
}
// token -> region (255 behind the last token)
__device__ __forceinline__ void dense_regions(uint8_t* reg, const Dims& dm, const DenseGeom& gm, int tid, int nthreads) {
    for (int t = tid; t < gm.rows; t += nthreads) reg[t] = t < dm.N ? (uint8_t)fdiv(t, dm.n_r, gm.mul_nr) : 255;
}
// mask[0 .. 63]: per query region the key regions; mask[64 .. 127]: per key region the query regions.  CTA-wide.
// True: some region is on a list more than once, see the table of log2(count) (-inf: not routed).
__device__ __forceinline__ bool dense_routes(unsigned long long* mask, float* bias, const int32_t* irows, int32_t* status, const Dims& dm,
                                             const DenseGeom& gm, int tid, int nthreads) {
    uint32_t* words = reinterpret_cast<uint32_t*>(mask);
    int* repeats = reinterpret_cast<int*>(mask + 128);
    if (!irows) {
        const unsigned long long all = dm.R == 64 ? ~0ull : (1ull << dm.R) - 1;
        for (int e = tid; e < 128; e += nthreads) mask[e] = all;
        __syncthreads();
        return false;
    }
    const int entries = dm.R * dm.topk;
    for (int e = tid; e < 257; e += nthreads) words[e] = 0u;
    __syncthreads();
    for (int e0 = tid; e0 < entries; e0 += 8 * nthreads) {
        int v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = e0 + u * nthreads < entries ? __ldcg(irows + e0 + u * nthreads) : -1;   // coherent: may come from the kernel this one overlaps
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * nthreads, j = v[u], i = fdiv(e, dm.topk, gm.mul_k);
            if (e >= entries) break;
            if (j < 0 || j >= dm.R) { record_error(status, BRA_ERR_INDEX, j); continue; }
            if (atomicOr(words + 2 * i + (j >> 5), 1u << (j & 31)) >> (j & 31) & 1u) *repeats = 1;
            atomicOr(words + 2 * (64 + j) + (i >> 5), 1u << (i & 31));
        }
    }
    __syncthreads();
    const bool weighted = *repeats != 0;
    if (weighted) {
        int32_t* cnt = reinterpret_cast<int32_t*>(bias);
        const int rr = dm.R * dm.R;
        for (int e = tid; e < rr; e += nthreads) cnt[e] = 0;
        __syncthreads();
        for (int e = tid; e < entries; e += nthreads) {
            const int j = __ldcg(irows + e);
            if (j >= 0 && j < dm.R) atomicAdd(cnt + e / dm.topk * dm.R + j, 1);
        }
        __syncthreads();
        for (int e = tid; e < rr; e += nthreads) bias[e] = cnt[e] == 0 ? -INFINITY : log2f((float)cnt[e]);
        __syncthreads();
    }
    return weighted;
}
// What is added to the scaled scores of a row for the columns of n-tiles, in blocks of tokens from 0 on: `yes` where the column's region
// is on the row's list, -inf elsewhere (and behind the last token).  NR: tokens per region - with four a bit of the mask covers the
// two columns a lane holds of an n-tile, with one it is the token's, 0 (any) goes by the table of regions.  (A bit per two or
// four scores, picked before the exponential: a test and a select per row and n-tile instead of per score behind it.  A bit of its own for
// a token, 64 x 7 x 7, 16 heads, topk 49: attention 15.1 -> 14.5 us, gradients 38.3 -> 36.4 against going by the table.)
constexpr int DENSE_ALL = -1;       // every region is on every list: nothing is picked, the kernel masks what is behind the last token
template <int NR>
struct DenseRow {
    unsigned long long m;
    DenseRow() = default;
    __device__ __forceinline__ DenseRow(unsigned long long mask, int t4) : m(NR == 4 ? mask >> (t4 >> 1) : NR == 1 ? mask >> (2 * t4) : mask) {}
    // n-tile j of the block from token k0 on, column 2 t4 + e
    __device__ __forceinline__ float pick(float yes, int j, int e, int k0, int t4, const uint8_t* reg) const {
        bool on;
        if (NR == DENSE_ALL) on = true;
        else if (NR == 4) on = (uint32_t)m >> (2 * j) & 1;
        else if (NR == 1) on = (uint32_t)m >> (8 * j + e) & 1;
        else {
            const int r = reg[k0 + 8 * j + 2 * t4 + e];
            on = r < 64 && (m >> r & 1);
        }
        return on ? yes : -INFINITY;
    }
    template <int TOKENS>
    __device__ __forceinline__ void next() {
        if (NR == 4) m >>= TOKENS / 4;
        if (NR == 1) m >>= TOKENS;
    }
};
// the same for lists with repeats, from row `at` of the table of log2(count)
__device__ __forceinline__ float dense_weight(const float* at, int r) { return r < 64 ? at[r] : -INFINITY; }

// Offsets of a lane in a slice: its 16-byte chunk of row g; rows lane % 16 for ldmatrix (exclusive or with 32: two chunks on).
// From a row that is a multiple of eight on.
__device__ __forceinline__ uint32_t dense_row_offset(int lane) { return dense_at(lane >> 2, lane & 3); }
__device__ __forceinline__ uint32_t dense_col_offset(int lane) { return dense_at(lane & 15, lane >> 4); }
__device__ __forceinline__ uint4 dense_chunk(uint32_t at) {
    const float4 f = ptx::lds_f32x4(at);
    return make_uint4(__float_as_uint(f.x), __float_as_uint(f.y), __float_as_uint(f.z), __float_as_uint(f.w));
}
__device__ __forceinline__ void dense_a(uint32_t (&a)[1][2][4], uint32_t at) {
    const uint4 lo[1] = {dense_chunk(at)}, up[1] = {dense_chunk(at + 512)};
    rows_to_a<1>(a, lo, up);
}
// The products run over every token of the map, with probability 0 where a pair is not routed: an infinity or NaN of a token
// then becomes a NaN in the accumulators of queries (keys) that do not list its region.  A CTA whose accumulators hold a NaN
// does its work again with the functions below (in attend_dense.cu and backward_dense.cu), a thread per token that
// looks at the routed pairs alone.  (That costs the kernels a few comparisons behind each walk.)
template <int RT>
__device__ __forceinline__ bool dense_any_nan(const float (&acc)[RT][4][4]) {
    bool nan = false;
#pragma unroll
    for (int x = 0; x < RT; ++x)
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) nan = nan || acc[x][n][e] != acc[x][n][e];
    return nan;
}
// row r of a slice
__device__ __forceinline__ void dense_row32(float (&v)[32], const uint8_t* slice, int r) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 u = *reinterpret_cast<const uint4*>(slice + dense_at(r, q));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[8 * q + 2 * j] = __uint_as_float(reg_of(u, j) << 16);
            v[8 * q + 2 * j + 1] = __uint_as_float(reg_of(u, j) & 0xffff0000u);
        }
    }
}
__device__ __forceinline__ float dense_dot(const float (&a)[32], const float (&b)[32]) {
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < 32; ++c) s = fmaf(a[c], b[c], s);
    return s;
}
// acc += the 5 x 5 correlation of a head's channels at (y, x), plus its bias; FLIP: with the flipped filter
template <bool FLIP>
__device__ __forceinline__ void dense_lce_row(float (&acc)[32], const __nv_bfloat16* in_head, const float* w, const float* bias, int y, int x, const Dims& dm) {
#pragma unroll 1
    for (int k = 0; k < 25; ++k) {
        const int yy = y + k / 5 - 2, xx = x + k % 5 - 2;
        if ((unsigned)yy >= (unsigned)dm.H0 || (unsigned)xx >= (unsigned)dm.W0) continue;
        float v[32];
        load_row<32>(in_head + (size_t)(uint32_t)(yy * dm.W0 + xx) * dm.C, v);
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[c] = fmaf(__ldg(w + c * 25 + (FLIP ? 24 - k : k)), v[c], acc[c]);
    }
    if (bias) {
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[c] += __ldg(bias + c);
    }
}

// acc (16 x 32) += A (16 x 16) * the 16 rows of a slice that start at `rows`
template <int RT>
__device__ __forceinline__ void dense_mma_tokens(float (*acc)[4][4], const uint32_t (*a)[4], uint32_t rows, uint32_t col_off) {
#pragma unroll
    for (int np = 0; np < 2; ++np) {
        uint32_t b[4];
        ldmatrix_x4_trans(rows + (col_off ^ (np * 32)), b);
#pragma unroll
        for (int x = 0; x < RT; ++x) {
            mma_bf16(acc[x][2 * np], a[x], b[0], b[1]);
            mma_bf16(acc[x][2 * np + 1], a[x], b[2], b[3]);
        }
    }
}

}  // namespace bra
