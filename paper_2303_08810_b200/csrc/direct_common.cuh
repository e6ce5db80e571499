// Shared by the warp-level tensor-core kernels whose operands come straight from global memory
// (attend_direct.cu, backward_direct.cu): geometry, token tables, operand fragments, LCE tiles.
//
// Fragments without shared memory.  A lane (g = lane / 4, t = lane % 4) loads 16 bytes - channels 8t .. 8t + 7 of a
// 32-channel plane - of token row g: four registers.  The contraction over channels of S = Q K^T may run in any order
// as long as both operands agree, so registers 0, 1 of a row are used as the k = 2t, 2t + 1 and k = 2t + 8, 2t + 9
// pairs of the first m16n8k16 step and registers 2, 3 as those of the second: rows as loaded ARE the A and B fragments.
// For a product that contracts over tokens (P V, dS K, ...) register i of eight token rows is an 8 x 8 matrix
// (token, channel); movmatrix transposes it into the B fragment whose column n is channel 8 (n / 2) + 2 i + n % 2,
// so that the accumulators of n-tiles i = 0 .. 3 are again channels 8t .. 8t + 7 of rows g and g + 8: results leave as
// 16-byte stores.
#pragma once

#include "fast_div.h"
#include "mma_common.cuh"

namespace bra {

namespace dk {
constexpr int TAB = 512;            // tokens a table holds (per group)
constexpr int TAB_WARP = 256;       // the same where a group is one warp
}  // namespace dk

struct DirGeom {
    int planes;
    int hb, chunks;        // region rows per chunk, chunks per region
    int tpc;               // 16-token tiles of a (full) chunk
    int nw, gpc;           // warps per CTA; groups (regions) per CTA: several when a region is one warp's work, else 1
    int gpi;               // CTAs per (image, head): the grid is (gpi, heads, images)
    int halo_w, halo_row;  // tokens and bytes of a halo row
    FastDiv by_nr;                                // positions in a walk pass n_r * n_r < 2^32; tokens of a region and regions do not
    uint32_t mul_ws, mul_s, mul_hw;
    int off_tab, off_w, off_halo, off_st, smem_bytes;
    int tab, tab_bytes, halo_bytes, st_bytes;     // per group; tab: entries
};

// entry_bytes: bytes of a table entry; rt: 16-token tiles of a warp
inline DirGeom direct_geom(const Dims& d, bool with_lce, int entry_bytes, int rt) {
    DirGeom g;
    g.planes = d.d / 32;
    g.hb = d.hs; g.chunks = 1;
    if (d.n_r > 128) {
        g.hb = 128 / d.ws;
        if (g.hb < 1) g.hb = 1;
        if (g.hb > 4) g.hb = g.hb / 4 * 4;             // whole LCE tiles
        if (g.hb > d.hs) g.hb = d.hs;
        g.chunks = (d.hs + g.hb - 1) / g.hb;
    }
    g.tpc = (g.hb * d.ws + 15) / 16;
    const int most = (g.planes == 2 ? 4 : 8) / rt;
    // two rounds of tiles per CTA only where there is a CTA for every SM (64 x 64, S = 2, topk 2, one head of 64: attention
    // 1 image 101 -> 56 us; 8 images, 256 CTAs, 141 -> 146)
    while (g.chunks > 1 && (g.tpc + rt - 1) / rt > most && g.hb > 1 && (long long)d.B * d.heads * d.R * g.chunks < kSMs) {
        g.hb = (g.hb + 1) / 2;
        g.chunks = (d.hs + g.hb - 1) / g.hb;
        g.tpc = (g.hb * d.ws + 15) / 16;
    }
    const int want = (g.tpc + rt - 1) / rt;
    if (want == 1 && g.chunks == 1) g.gpc = g.nw = most < 4 ? most : 4;
    else { g.gpc = 1; g.nw = want < most ? want : most; }
    g.gpi = (d.R + g.gpc - 1) / g.gpc * g.chunks;
    g.halo_w = d.ws + 4;
    g.halo_row = g.halo_w * 64 * g.planes + 16;        // tiles four rows apart start on different banks
    g.by_nr = fast_div(d.n_r); g.mul_ws = recip32(d.ws); g.mul_s = recip32(d.S); g.mul_hw = recip32(g.halo_w);
    g.tab = g.gpc > 1 ? dk::TAB_WARP : dk::TAB;
    const int need = (d.topk * d.n_r + 31) / 32 * 32;
    if (need < g.tab) g.tab = need;
    int off = 0;
    g.tab_bytes = (g.tab * entry_bytes + g.tab / 8 + 8 + 15) / 16 * 16;     // entries, a bit per entry, a counter; or three numbers
    g.off_tab = off;  off += g.gpc * g.tab_bytes;
    g.off_w = off;    off += with_lce ? 32 * g.planes * 25 * 4 : 0;
    off = (off + 15) / 16 * 16;
    g.halo_bytes = with_lce ? (g.hb + 4) * g.halo_row : 0;
    g.off_halo = off; off += g.gpc * g.halo_bytes;
    g.st_bytes = (g.tpc + rt - 1) / rt * rt * 16 * 128 * g.planes;
    g.off_st = off;   off += g.gpc * g.st_bytes;
    // LCE tiles that stick out of a chunk read (and discard) up to three halo rows behind it
    const int reach = g.off_halo + g.gpc * g.halo_bytes + (with_lce ? 3 * g.halo_row + 1024 : 0);
    g.smem_bytes = off > reach ? off : reach;
    return g;
}

// Regions of more than 128 tokens whose rows do not divide 128, lists of more than 256 regions and regions of tens of
// thousands of tokens: these problems used to run in fp32 on the CUDA cores, so the probabilities keep 16 bits of mantissa
// here (two MMAs).  The gradients of head dim 64 do so for every shape.
inline bool direct_exact(const Dims& d) {
    return (d.n_r > 128 && 128 % d.ws != 0) || d.topk > 256 || (long long)d.topk * d.n_r * d.n_r >= (1ll << 32);
}

// Tiles per warp in the forward kernel: two share every row that is loaded (and transposed) where regions have two and enough
// warps remain.  Measured, one / two tiles: 2 x 100 x 167 tokens, S = 16, topk 4, 6 heads 124 / 114 us; 2 x 112 x 112, S = 8: 98 / 88.
// Around the line each wave of CTAs is a step on either side: 35 x 35, 784 warps 11.7 / 13.1, 1176 13.9 / 15.7, 1372 20.6 / 15.8, 1764
// 22.7 / 24.0, 3626 42.1 / 37.6; 70 x 70, 1176 warps 12.1 / 12.2, 1568 19.0 / 14.5, 2352 22.5 / 21.9.
inline int direct_rt(const Dims& d) {
    const long long warps = (long long)d.B * d.heads * d.R * ((d.n_r + 31) / 32);
    return d.n_r > 16 && warps >= 8 * kSMs ? 2 : 1;
}

// ------------------------------------------------------------------ loads
// 16 bytes of the read-only input tensors; zero where `ok` is false (nothing is read)
__device__ __forceinline__ uint4 ld16_or_zero(const uint8_t* p, bool ok) {
    uint4 v;
    asm("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "mov.b32 %0, 0; mov.b32 %1, 0; mov.b32 %2, 0; mov.b32 %3, 0;\n\t"
        "@q ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "=&r"(v.x), "=&r"(v.y), "=&r"(v.z), "=&r"(v.w) : "l"(p), "r"((int)ok));
    return v;
}
__device__ __forceinline__ uint4 ld16(const uint8_t* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }
// A lane's chunks of the token whose row starts off16 * 16 bytes behind base.
template <int PL>
__device__ __forceinline__ void ld_token(uint4 (&v)[PL], const uint8_t* base, uint32_t off16) {
    const uint8_t* p = base + (size_t)off16 * 16;
#pragma unroll
    for (int q = 0; q < PL; ++q) v[q] = ld16(p + q * 64);
}
// the same for a row that may not exist
template <int PL>
__device__ __forceinline__ void ld_row(uint4 (&v)[PL], const uint8_t* base, int tok, uint32_t tok_bytes) {
    const uint8_t* p = base + (size_t)(uint32_t)tok * tok_bytes;
#pragma unroll
    for (int q = 0; q < PL; ++q) v[q] = ld16_or_zero(p + q * 64, tok >= 0);
}
__device__ __forceinline__ uint32_t movm(uint32_t x) {
    uint32_t y;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ uint32_t reg_of(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// A fragments of 16 rows: a[plane][k step] from the chunks of rows g (lo) and g + 8 (hi)
template <int PL>
__device__ __forceinline__ void rows_to_a(uint32_t (&a)[PL][2][4], const uint4 (&lo)[PL], const uint4 (&hi)[PL]) {
#pragma unroll
    for (int p = 0; p < PL; ++p) {
        a[p][0][0] = lo[p].x; a[p][0][1] = hi[p].x; a[p][0][2] = lo[p].y; a[p][0][3] = hi[p].y;
        a[p][1][0] = lo[p].z; a[p][1][1] = hi[p].z; a[p][1][2] = lo[p].w; a[p][1][3] = hi[p].w;
    }
}
// c (16 x 8) = A * B^T for eight token rows given as chunks
template <int PL>
__device__ __forceinline__ void mma_rows(float (&c)[4], const uint32_t (&a)[PL][2][4], const uint4 (&b)[PL]) {
    mma_bf16_zero(c, a[0][0], b[0].x, b[0].y);
    mma_bf16(c, a[0][1], b[0].z, b[0].w);
    if (PL == 2) {
        mma_bf16(c, a[PL - 1][0], b[PL - 1].x, b[PL - 1].y);
        mma_bf16(c, a[PL - 1][1], b[PL - 1].z, b[PL - 1].w);
    }
}
// A fragment of 16 x 16 probabilities (two n-tiles of accumulators) in bf16, and what the rounding left over
__device__ __forceinline__ void frag_hi(uint32_t (&a)[4], const float (&c0)[4], const float (&c1)[4]) {
    a[0] = pack2_bf16(c0[0], c0[1]); a[1] = pack2_bf16(c0[2], c0[3]);
    a[2] = pack2_bf16(c1[0], c1[1]); a[3] = pack2_bf16(c1[2], c1[3]);
}
__device__ __forceinline__ uint32_t left_over(uint32_t h, float x, float y) {
    return pack2_bf16(x - __uint_as_float(h << 16), y - __uint_as_float(h & 0xffff0000u));
}
__device__ __forceinline__ void frag_lo(uint32_t (&l)[4], const uint32_t (&a)[4], const float (&c0)[4], const float (&c1)[4]) {
    l[0] = left_over(a[0], c0[0], c0[1]); l[1] = left_over(a[1], c0[2], c0[3]);
    l[2] = left_over(a[2], c1[0], c1[1]); l[3] = left_over(a[3], c1[2], c1[3]);
}
// acc[x] (16 x 32 PL) += A[x] (16 x 16, fragments c[x][j0], c[x][j0 + 1]) * the 16 token rows lo (0-7), hi (8-15)
// EXACT: A = hi + lo parts (16 bits of mantissa), for problems whose products were fp32 before they had these kernels
template <int PL, bool EXACT, int RT, int J>
__device__ __forceinline__ void mma_tokens(float (&acc)[RT][PL][4][4], const float (&c)[RT][J][4], int j0, const uint4 (&lo)[PL], const uint4 (&hi)[PL]) {
    uint32_t a[RT][4], l[RT][4];
#pragma unroll
    for (int x = 0; x < RT; ++x) {
        frag_hi(a[x], c[x][j0], c[x][j0 + 1]);
        if (EXACT) frag_lo(l[x], a[x], c[x][j0], c[x][j0 + 1]);
    }
#pragma unroll
    for (int p = 0; p < PL; ++p)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t b0 = movm(reg_of(lo[p], i)), b1 = movm(reg_of(hi[p], i));
#pragma unroll
            for (int x = 0; x < RT; ++x) {
                mma_bf16(acc[x][p][i], a[x], b0, b1);
                if (EXACT) mma_bf16(acc[x][p][i], l[x], b0, b1);
            }
        }
}
// eight consecutive channels of one row (n-tiles 0..3, elements 2r, 2r + 1) times f, as bf16
__device__ __forceinline__ uint4 pack_row(const float (&acc)[4][4], int r, float f) {
    return make_uint4(pack2_bf16(acc[0][2 * r] * f, acc[0][2 * r + 1] * f), pack2_bf16(acc[1][2 * r] * f, acc[1][2 * r + 1] * f),
                      pack2_bf16(acc[2][2 * r] * f, acc[2][2 * r + 1] * f), pack2_bf16(acc[3][2 * r] * f, acc[3][2 * r + 1] * f));
}

// ------------------------------------------------------------------ groups and token tables
// Token (row-major in the caller's map) of token t of region r; -1 in the zero padding.
__device__ __forceinline__ int token_of(const Dims& dm, const DirGeom& gm, int r, int t) {
    const int ry = fdiv(r, dm.S, gm.mul_s), rx = r - ry * dm.S;
    const int ty = fdiv(t, dm.ws, gm.mul_ws), tx = t - ty * dm.ws;
    const int y = ry * dm.hs + ty, x = rx * dm.ws + tx;
    return y < dm.H0 && x < dm.W0 ? y * dm.W0 + x : -1;
}
// Dead rows (of a tile's rest, of a bad routing entry, of the zero padding) have the probability 0, but what is read in their
// place must be finite, or the product is NaN: a row of a region that nobody routes to would reach the results.  They read
// token 0, or, if that holds an infinity or NaN in one of the two tensors, the first token that does not (none: 0).
// spare_probe(), with a chunk of token 0 per lane, is called where its latency is hidden; both by whole warps.  (Zeroing the
// rows in the walk, or walking again when a NaN came out, costs registers there: forward + backward at 64 x 56 x 56 x 64
// 238 -> 264 and 252 us.)
template <int PL>
__device__ __forceinline__ uint4 spare_probe(const uint8_t* a, const uint8_t* b, int lane) {
    return ld16_or_zero((lane < 4 * PL ? a : b) + lane % (4 * PL) * 16, lane < 8 * PL);
}
// (0 times a finite number added to 0 is +0, anything else NaN: five instructions, which count where a warp's walk is short)
__device__ __forceinline__ bool finite_bf16x8(const uint4& v) {
    const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
    __nv_bfloat162 sum = zero;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t w = reg_of(v, i);
        sum = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w), zero, sum);
    }
    return *reinterpret_cast<const uint32_t*>(&sum) == 0u;
}
template <int PL>
__device__ __forceinline__ int spare_token(const uint4& probe, const uint8_t* a, const uint8_t* b, uint32_t tok_bytes, int tokens, int lane) {
    if (__all_sync(0xffffffffu, finite_bf16x8(probe))) return 0;
#pragma unroll 1
    for (int t0 = 0; t0 < tokens; t0 += 32) {
        const int t = t0 + lane;
        bool ok = t < tokens;
#pragma unroll 1
        for (int q = 0; ok && q < 8 * PL; ++q)
            ok = finite_bf16x8(ld16((q < 4 * PL ? a : b) + (size_t)(uint32_t)t * tok_bytes + q % (4 * PL) * 16));
        const uint32_t word = __ballot_sync(0xffffffffu, ok);
        if (word) return t0 + __ffs(word) - 1;
    }
    return 0;
}
// Table of the keys [k0, k0 + n) of a group: key kk is token kk % n_r of region irow[kk / n_r].  An entry is the
// offset of the token's row from the head's first byte, in units of 16 bytes.  Keys that are not rows of the map - entries
// beyond `total`, of a bad routing entry, of the zero padding - name the row of token `spare` and have their bit set in `dead`:
// the caller gives them the probability zero.  (A key of the zero padding has the score 0 and the value 0: all it does is
// count in the softmax's denominator.)  Returns how many keys of the zero padding this lane met.
__device__ __forceinline__ int fill_keys(uint32_t* tab, uint32_t* dead, const int32_t* irow, int k0, int n, int total, int spare, int lane0,
                                         int lanes, int32_t* status, const Dims& dm, const DirGeom& gm) {
    int zeros = 0;
    for (int e = lane0; e < n; e += lanes) {                         // whole warps: n and lanes are multiples of 32
        const int kk = min(k0 + e, total - 1);
        const int m = fdiv(kk, gm.by_nr);
        const int r = __ldcg(irow + m);  // coherent load: the index may come from the kernel this one overlaps
        bool ok = k0 + e < total;
        int tok = spare;
        if (r < 0 || r >= dm.R) {
            record_error(status, BRA_ERR_INDEX, r);
            ok = false;
        } else {
            tok = token_of(dm, gm, r, kk - m * dm.n_r);
            if (tok < 0) { zeros += ok; ok = false; }
            if (!ok) tok = spare;
        }
        tab[e] = (uint32_t)tok * (uint32_t)(dm.C >> 3);
        const uint32_t word = __ballot_sync(0xffffffffu, !ok);
        if ((e & 31) == 0) dead[e >> 5] = word;
    }
    return zeros;
}
// columns 8 j + 2 t4, + 1 (j = 0 .. J - 1) of the rows c[x] whose bits are set: value v
template <int RT, int J>
__device__ __forceinline__ void mask_columns(float (&c)[RT][J][4], uint32_t bits, int t4, float v) {
    bits >>= 2 * t4;
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int x = 0; x < RT; ++x) {
            if (bits >> (8 * j) & 1) c[x][j][0] = c[x][j][2] = v;
            if (bits >> (8 * j + 1) & 1) c[x][j][1] = c[x][j][3] = v;
        }
}

// ------------------------------------------------------------------ LCE
// LCE weights of a head, as they lie in memory: [32 PL channels][25]
__device__ __forceinline__ void load_lce_weights(float* s_w, const float* lce_w, int h, int n, int tid, int nthreads) {
    const float* w = lce_w + (size_t)h * n;
    for (int e = tid; e < n; e += nthreads) s_w[e] = __ldg(w + e);
}
// Rows y0 - 2 .. y0 + rows + 1, columns x0 - 2 .. x0 + ws + 1 of a head's channels: zero outside the map
template <int PL>
__device__ __forceinline__ void load_halo(uint32_t dst, const uint8_t* img, int y0, int x0, int rows, const Dims& dm,
                                          const DirGeom& gm, int lane0, int lanes) {
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
    const int n = (rows + 4) * gm.halo_w * 4 * PL;
    for (int e = lane0; e < n; e += lanes) {
        const int cell = e / (4 * PL), q = e % (4 * PL);
        const int hy = fdiv(cell, gm.halo_w, gm.mul_hw), hx = cell - hy * gm.halo_w;
        const int y = y0 + hy - 2, x = x0 + hx - 2;
        const bool in = (unsigned)y < (unsigned)dm.H0 && (unsigned)x < (unsigned)dm.W0;
        ptx::cp_async_16(dst + hy * gm.halo_row + hx * 64 * PL + q * 16, in ? img + (size_t)(uint32_t)(y * dm.W0 + x) * tok_bytes + q * 16 : img,
                         in ? 16u : 0u);
    }
}
// acc[TY][TX] += 5 x 5 depthwise correlation of a channel pair at TY x TX positions; halo: shared-memory address of
// the pair at the top left of the window.  FLIP: the flipped filter (the adjoint).
template <int PL, int TY, int TX, bool FLIP>
__device__ __forceinline__ void lce_tile(float2 (&acc)[TY][TX], uint32_t halo, int halo_row, const float2 (&wv)[25]) {
#pragma unroll
    for (int r = 0; r < TY + 4; ++r) {
        float2 v[TX + 4];
#pragma unroll
        for (int c = 0; c < TX + 4; ++c) {
            const uint32_t w = ptx::lds_u32(halo + c * 64 * PL);
            v[c] = make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
        }
        halo += halo_row;
#pragma unroll
        for (int yy = 0; yy < TY; ++yy) {
            const int ti = r - yy;
            if (ti < 0 || ti > 4) continue;
#pragma unroll
            for (int tj = 0; tj < 5; ++tj)
#pragma unroll
                for (int xx = 0; xx < TX; ++xx)
                    acc[yy][xx] = __ffma2_rn(wv[FLIP ? 24 - (ti * 5 + tj) : ti * 5 + tj], v[xx + tj], acc[yy][xx]);
        }
    }
}
// The LCE of a chunk (rows x ws tokens at (y0, x0)) by `gwarps` warps, added to the staged attention term
// (fp32 [token][32 PL channels]) and stored as bf16.
template <int PL, int TY, int TX, bool FLIP, int ST = 32 * PL>       // ST: floats per staged token
__device__ __forceinline__ void lce_chunk(const float* st, uint32_t halo, const float* s_w, const float* bias, bool lce, __nv_bfloat16* out_head,
                                          int y0, int x0, int rows, const Dims& dm, const DirGeom& gm, int gwarp, int gwarps, int lane) {
    const int cp = PL == 2 ? lane : lane & 15, sub = PL == 2 ? 0 : lane >> 4;
    const int nty = (rows + TY - 1) / TY, ntx = (dm.ws + TX - 1) / TX;
    // two tiles per warp pass where a head has 16 channel pairs: one below the other (on different banks), else side by side
    const bool vertical = nty > 1;
    const int items = PL == 2 ? nty * ntx : vertical ? (nty + 1) / 2 * ntx : (ntx + 1) / 2;
    if (gwarp >= items) return;
    float2 wv[25], b2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 25; ++q) wv[q] = lce ? make_float2(s_w[2 * cp * 25 + q], s_w[(2 * cp + 1) * 25 + q]) : make_float2(0.f, 0.f);
    if (bias) b2 = make_float2(__ldg(bias + 2 * cp), __ldg(bias + 2 * cp + 1));
    for (int it = gwarp; it < items; it += gwarps) {
        int ty, tx;
        if (PL == 2) { ty = it / ntx; tx = it - ty * ntx; }
        else if (vertical) { ty = it / ntx; tx = it - ty * ntx; ty = 2 * ty + sub; }
        else { ty = 0; tx = 2 * it + sub; }
        if (ty >= nty || tx >= ntx) continue;
        float2 acc[TY][TX];
#pragma unroll
        for (int yy = 0; yy < TY; ++yy)
#pragma unroll
            for (int xx = 0; xx < TX; ++xx) acc[yy][xx] = b2;
        if (lce) lce_tile<PL, TY, TX, FLIP>(acc, halo + ty * TY * gm.halo_row + tx * TX * 64 * PL + cp * 4, gm.halo_row, wv);
        const float* src = st + (ty * TY * dm.ws + tx * TX) * ST + 2 * cp;
        __nv_bfloat16* dst = out_head + (size_t)(uint32_t)((y0 + ty * TY) * dm.W0 + x0 + tx * TX) * dm.C + 2 * cp;
        const int ny = min(rows - ty * TY, dm.H0 - y0 - ty * TY), nx = min(dm.ws - tx * TX, dm.W0 - x0 - tx * TX);
#pragma unroll
        for (int yy = 0; yy < TY; ++yy) {
            if (yy >= ny) break;
#pragma unroll
            for (int xx = 0; xx < TX; ++xx) {
                if (xx >= nx) break;
                const float2 a = *reinterpret_cast<const float2*>(src + xx * ST);
                const float2 o = __fadd2_rn(a, acc[yy][xx]);
                *reinterpret_cast<uint32_t*>(dst + (size_t)xx * dm.C) = pack2_bf16(o.x, o.y);
            }
            src += dm.ws * ST;
            dst += (size_t)dm.W0 * dm.C;
        }
    }
}

// Columns of an LCE tile (four rows): the width that leaves the busiest warp the least to do (instructions of a tile:
// 8 rows of 3 per column of the window, 20 packed FMAs per position; about 60 more per tile).
inline int lce_tile_width(const DirGeom& g, const Dims& d) {
    int best = 4;
    long long best_cost = -1;
    for (int tx = 2; tx <= 4; ++tx) {
        const int nty = (g.hb + 3) / 4, ntx = (d.ws + tx - 1) / tx;
        const int items = g.planes == 2 ? nty * ntx : nty > 1 ? (nty + 1) / 2 * ntx : (ntx + 1) / 2;
        const int warps = g.gpc > 1 ? 1 : g.nw;
        const long long cost = (long long)((items + warps - 1) / warps) * (24 * (tx + 4) + 100 * tx + 60);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = tx; }
    }
    return best;
}

}  // namespace bra
