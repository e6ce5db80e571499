// Shared by the fp32-arithmetic kernels on CUDA cores (attend_simt.cu, backward.cu): fp32 problems (a result to 1e-5 and
// the precision of fp32 sums rule out bf16 / tf32 matrix instructions) and the shapes the tensor-core kernels do not take.
//
// Mapping.  A lane owns QT rows of this side (queries; keys in the dK / dV kernel) with all their channels and walks the
// rows of the other side, which all lanes of a region read from shared memory at once (a 16-byte read that several lanes
// share costs the SM two cycles: with QT = 1 those reads, not the FMA pipe, set the time of S and P V; with QT = 2 the two
// are level).  Dot products are single chains over the channels in increasing order.  Where a call has too few rows to
// fill the GPU, 2, 4 or 8 lanes share their rows and split the other side between them (`ksl`).
//
// The other side's rows reach shared memory by asynchronous copies: the whole (image, head) slice where it is small
// (`resident`: every routed row would otherwise be copied once per region that lists it), else a block of rows per region
// of the CTA, double-buffered.  Rows are padded by 16 bytes and so are the blocks of the regions, so that rows read at
// once (of several regions, or of several key shares) start on different banks.
#pragma once

#include "fast_div.h"
#include "mma_common.cuh"

namespace bra {

namespace sk {
constexpr int THREADS = 256;            // at most: enough for a region, which shares the copies (64 if that is enough: an even tail)
constexpr int RESIDENT_MAX = 100 * 1024;
constexpr int IDX_MAX = 4096;           // routing entries kept in shared memory per CTA
constexpr int SMEM_MAX = 220 * 1024;
}  // namespace sk

struct SimtGeom {
    int hb, cw;            // rows and columns of a chunk of a region (the whole region unless it is large)
    int cx, chunks;        // chunks per row of chunks, chunks per region
    int rpc, spr;          // regions per CTA; lane groups (QT rows each) per region (of a full chunk)
    int ksl;               // log2 of the lanes that share rows
    int threads, gpi;      // the grid is (gpi, heads, images)
    int far;               // rows straight from global memory (simt_far())
    int resident, dense;   // dense: topk == R, walk every region and weigh it by how often the list names it
    int kps, stages;       // rows of the other side per region and stage
    int span;              // dK / dV: entries of a list per walk (their rows are counted in 32 bits)
    FastDiv by_nr, by_ws, by_s;
    uint32_t mul_spr, mul_kps, mul_cw;
    int row;               // bytes of a row of one tensor in shared memory
    int reg;               // bytes from one region's rows of a stage to the next region's
    int zero;              // resident: offset of a row of zeros in either tensor's rows
    int off_a, off_b, off_stat, off_idx, off_cnt, off_w, off_st, smem_bytes;
    int stage_bytes;       // from one stage to the next (0: there is one)
};

enum SimtKind { SIMT_ATTEND, SIMT_DQ, SIMT_DKV };

// Attention over regions of one or two tokens: the lanes of a CTA share no rows of K and V, and rows staged for each of them leave
// an SM two to four warps.  They read their rows straight from global memory (attend_simt_kernel<T, D, true>), unless every
// region is routed to and the slice is resident.  Measured (B200, us, staged / straight / one thread per query without shared key
// lanes): 64 x 14 x 14, S = 14, topk 8: 1 head of 64 127 / 46 / 63, 1 head of 128 512 / 93 / 127, 2 heads of 32 (resident) 47 / 43 / 56;
// 64 x 16 x 16, S = 16, topk 4, 2 heads of 32 86 / 41 / 46; 64 x 28 x 14, S = 14, topk 8, 2 heads of 32 77 / 68 / 81.
inline bool simt_far(const Dims& d, SimtKind kind) { return kind == SIMT_ATTEND && d.n_r <= 2 && !(d.topk == d.R && d.R <= 64); }
// rows per lane: two where registers allow it (the dK / dV kernel keeps four rows of channels per key)
inline int simt_rows(const Dims& d, SimtKind kind) { return kind != SIMT_DKV && d.d <= 32 && !simt_far(d, kind) ? 2 : 1; }
// log2 of the lanes that hold a row's channels: a dK / dV lane with the four rows of 64 channels spilled 2 KB of registers
// (gradients at 64 x 14 x 14, 4 heads of 64, topk 16: 1048 us)
inline int simt_split(int head_dim, SimtKind kind) { return kind == SIMT_DKV && head_dim > 32 ? 1 : 0; }

// At most rpc_max regions per CTA; stages of the rows of the other side where they are not resident; threads that a CTA has
// unless one region wants more.
inline SimtGeom simt_geom(const Dims& d, SimtKind kind, int rpc_max, int stages, int threads = 64) {
    SimtGeom g;
    const int qt = simt_rows(d, kind);
    g.far = simt_far(d, kind);
    g.row = d.d * d.esize + 16;
    g.by_nr = fast_div(d.n_r); g.by_ws = fast_div(d.ws); g.by_s = fast_div(d.S);
    // lanes of this call against the lanes the GPU holds at once (12 warps per SM)
    // (dK / dV of larger maps: as if a half of the regions held the lists, a quarter with topk = 1, which is what clustered content
    // comes to.  By 8 / 4 / 2 / 1, gradients in us: 64 x 21 x 21, 2 heads, topk 8 400 / 316 / 279 / 276; 4 x 44 x 44, 4 heads, topk 4 354 /
    // 298 / 254 / 291; clustered, forward and gradients: 2 x 88 x 88, 2 heads, topk 1 448 / 447 / 563 / 731, 5 x 48 x 48, 4 heads, topk 4
    // 491 / 418 / 385 / 497)
    const int held = kind == SIMT_DKV && d.N > 400 ? (d.topk == 1 ? 4 : 2) : 1;
    const long long lanes = (long long)d.B * d.heads * d.R * ((d.n_r + qt - 1) / qt) / held;
    const int split = simt_split(d.d, kind);
    g.ksl = 0;
    while (g.ksl < 3 && (lanes << (g.ksl + split)) < kSMs * 256 && (qt * d.d >> (g.ksl + split + 1)) >= 4) ++g.ksl;    // sum_shares: whole float4s
    const int group = g.ksl + split;                                  // log2 of the lanes of a group
    while (threads < sk::THREADS && ((d.n_r + qt - 1) / qt << group) > threads) threads *= 2;
    const int most = threads >> group;                                // lane groups of a CTA
    g.hb = d.hs; g.cw = d.ws;
    if ((d.n_r + qt - 1) / qt > most) {
        if (g.cw > qt * most) g.cw = qt * most;
        g.hb = qt * most / g.cw;
        if (g.hb > d.hs) g.hb = d.hs;
    }
    g.cx = (d.ws + g.cw - 1) / g.cw;
    g.chunks = (d.hs + g.hb - 1) / g.hb * g.cx;
    g.mul_cw = recip32(g.cw);
    g.spr = (g.hb * g.cw + qt - 1) / qt;
    g.rpc = g.chunks > 1 ? 1 : most / g.spr;
    if (g.rpc < 1) g.rpc = 1;
    if (g.rpc > d.R) g.rpc = d.R;
    if (g.rpc > rpc_max) g.rpc = rpc_max;
    if ((long long)g.rpc * d.topk > sk::IDX_MAX) g.rpc = sk::IDX_MAX / d.topk > 0 ? sk::IDX_MAX / d.topk : 1;
    const int ctas = (d.R + g.rpc - 1) / g.rpc;                       // even out the regions over them
    g.rpc = (d.R + ctas - 1) / ctas;
    g.mul_spr = recip32(g.spr);
    g.threads = ((g.rpc * g.spr << group) + 31) / 32 * 32;
    g.gpi = ctas * g.chunks;
    const long long slice = 2ll * d.N * g.row;
    // copies of the slice against copies of the listed rows (a key region is listed topk times on average)
    g.resident = !g.far && slice <= sk::RESIDENT_MAX && (long long)g.rpc * d.topk * d.n_r >= d.N;
    g.dense = g.resident && d.topk == d.R && d.R <= 64;
    const int block = 4 << g.ksl;
    // about 64 rows of two tensors per stage (18 KB at D = 32, fp32), in whole blocks of four per lane
    g.kps = 64 / g.rpc / block * block;
    if (g.kps < block) g.kps = block;
    if (g.kps > 32) g.kps = 32;
    g.mul_kps = recip32(g.kps);
    g.span = (1 << 30) / d.n_r + 1;
    g.stages = g.resident ? 1 : stages;
    const int rows = g.far ? 0 : g.resident ? d.N : g.rpc * g.kps;    // of one stage
    g.reg = (g.kps * g.row + 111) / 128 * 128 + 16;                   // 16 modulo 128
    int off = 0;
    g.zero = g.far ? 0 : g.resident ? rows * g.row : g.rpc * g.reg;
    g.off_a = off;    off += g.zero + (g.resident ? g.row : 0);
    g.off_b = off;    off += g.zero + (g.resident ? g.row : 0);
    g.off_stat = off; off += kind == SIMT_DKV ? (rows * 8 + 15) / 16 * 16 : 0;     // lse, delta
    g.stage_bytes = g.stages == 2 ? off : 0;
    off *= g.stages;
    const int rows_end = off;
    g.off_idx = off;                                                  // (dK / dV: the lists are read through L1)
    if (kind != SIMT_DKV && (long long)g.rpc * d.topk <= sk::IDX_MAX) off += g.rpc * d.topk * 4;
    g.off_cnt = off;  off += g.dense ? g.rpc * d.R * 4 : 0;
    g.off_w = off;    off += kind != SIMT_DQ && d.lce ? 25 * d.d * 4 : 0;
    off = (off + 15) / 16 * 16;
    g.off_st = 0;                                                     // over the rows, once they have been read
    const int st = kind != SIMT_DQ ? g.rpc * qt * g.spr * (d.d + 4) * 4 : 0;
    if (st > rows_end) { g.off_st = off; off += st; }
    g.smem_bytes = off;
    return g;
}
// Two stages, so that the next rows arrive while these are used, if three CTAs of them fit on an SM.  Else one: more CTAs hide
// more than the second stage does (attention, one / two stages: 64 x 14 x 14, 2 heads of 128, topk 16: 247 / 511 us;
// 64 x 28 x 28, S = 14, 2 heads of 32: 91 / 138; below the line 16 x 64 x 64, S = 16, 2 heads of 32: 234 / 227; 64 x 40 x 24, S = 8,
// 2 heads of 64: 308 / 293).  Where a region is a few tokens, nearly every lane has rows of its own: as many regions as fit.
inline SimtGeom simt_geom(const Dims& d, SimtKind kind) {
    SimtGeom g = simt_geom(d, kind, sk::THREADS, 2);
    // resident: twice the threads make half the copies of the slice (64 x 14 x 14, 2 heads of 32, attention, S = 14, topk 8: 62 -> 47 us,
    // S = 7, topk 16: 43 -> 35; dK / dV, whose lists differ in length: 104 to 107 %)
    if ((g.resident && kind != SIMT_DKV) || g.far) g = simt_geom(d, kind, sk::THREADS, 2, 128);
    if (g.stages * g.stage_bytes > 72 * 1024) g = simt_geom(d, kind, sk::THREADS, 1);
    for (int rpc = sk::THREADS; g.smem_bytes > sk::SMEM_MAX && rpc > 0; rpc /= 2) g = simt_geom(d, kind, rpc, 1);
    return g;
}
inline bool simt_fits(const Dims& d, SimtKind kind) {
    // (token numbers and positions in a walk are ints)
    return (long long)d.H * d.W < (1ll << 31) - 65536 && simt_geom(d, kind).smem_bytes <= sk::SMEM_MAX;
}

// Token (row-major in the caller's map) of token t of region r; -1 in the zero padding.
__device__ __forceinline__ int simt_token(const Dims& dm, const SimtGeom& gm, int r, int t) {
    const int ry = fdiv(r, gm.by_s), rx = r - ry * dm.S;
    const int ty = fdiv(t, gm.by_ws), tx = t - ty * dm.ws;
    const int y = ry * dm.hs + ty, x = rx * dm.ws + tx;
    return y < dm.H0 && x < dm.W0 ? y * dm.W0 + x : -1;
}

// Chunk ck of a region: first row and column in the region, extent.
struct SimtChunk { int y, x, rows, cols; };
__device__ __forceinline__ SimtChunk simt_chunk(const Dims& dm, const SimtGeom& gm, int ck) {
    SimtChunk c;
    const int cy = ck / gm.cx;
    c.y = cy * gm.hb; c.x = (ck - cy * gm.cx) * gm.cw;
    c.rows = min(gm.hb, dm.hs - c.y); c.cols = min(gm.cw, dm.ws - c.x);
    return c;
}
// Token of row t of a chunk (gm.cw rows of this side per line) of region r; -1 outside the chunk or the map.
__device__ __forceinline__ int simt_row(const Dims& dm, const SimtGeom& gm, const SimtChunk& c, int r, int t) {
    const int ly = fdiv(t, gm.cw, gm.mul_cw), lx = t - ly * gm.cw;
    if (ly >= c.rows || lx >= c.cols) return -1;
    const int ry = fdiv(r, gm.by_s), rx = r - ry * dm.S;
    const int y = ry * dm.hs + c.y + ly, x = rx * dm.ws + c.x + lx;
    return y < dm.H0 && x < dm.W0 ? y * dm.W0 + x : -1;
}

// N channels of a row
template <typename T, int N>
__device__ __forceinline__ void lds_row(float (&v)[N], uint32_t a) {
    if (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const float4 f = ptx::lds_f32x4(a + 16 * i);
            v[4 * i] = f.x; v[4 * i + 1] = f.y; v[4 * i + 2] = f.z; v[4 * i + 3] = f.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < N / 8; ++i) {
            const float4 f = ptx::lds_f32x4(a + 16 * i);
            const uint32_t w[4] = {__float_as_uint(f.x), __float_as_uint(f.y), __float_as_uint(f.z), __float_as_uint(f.w)};
#pragma unroll
            for (int j = 0; j < 4; ++j) { v[8 * i + 2 * j] = __uint_as_float(w[j] << 16); v[8 * i + 2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u); }
        }
    }
}
template <typename T, int N>
__device__ __forceinline__ void ldg_row(float (&v)[N], const T* p, bool ok, float f) {
    if (ok) {
        load_row<N>(p, v);
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] *= f;
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = 0.f;
    }
}
// s[x][u] = q[x] . row at[u]: one chain each over the channels in increasing order, all chains interleaved (an FMA waits
// four cycles for the one before it in its chain)
template <typename T, int QT, int U, int N>
__device__ __forceinline__ void dots(float (&s)[QT][U], const float (&q)[QT][N], const uint32_t (&at)[U], int off) {
    constexpr int CH = 16 / (int)sizeof(T);
#pragma unroll
    for (int x = 0; x < QT; ++x)
#pragma unroll
        for (int u = 0; u < U; ++u) s[x][u] = 0.f;
#pragma unroll
    for (int c = 0; c < N; c += CH) {
        float k[U][CH];
#pragma unroll
        for (int u = 0; u < U; ++u) lds_row<T, CH>(k[u], at[u] + off + c * (int)sizeof(T));
#pragma unroll
        for (int i = 0; i < CH; ++i)
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int x = 0; x < QT; ++x) s[x][u] = fmaf(q[x][c + i], k[u][i], s[x][u]);
    }
}
// 16 bytes of a row in global memory; zeros if there is no row
template <typename T>
__device__ __forceinline__ void ldg_chunk(float (&v)[16 / sizeof(T)], const T* p, bool ok) {
    if (ok) load_row<16 / (int)sizeof(T)>(p, v);
    else
#pragma unroll
        for (int i = 0; i < 16 / (int)sizeof(T); ++i) v[i] = 0.f;
}
// s[x][u] = q[x] . row tok[u] of a head in global memory (no row: 0)
template <typename T, int QT, int U, int N>
__device__ __forceinline__ void dots_far(float (&s)[QT][U], const float (&q)[QT][N], const T* head, const int (&tok)[U], int C) {
    constexpr int CH = 16 / (int)sizeof(T);
#pragma unroll
    for (int x = 0; x < QT; ++x)
#pragma unroll
        for (int u = 0; u < U; ++u) s[x][u] = 0.f;
#pragma unroll
    for (int c = 0; c < N; c += CH) {
        float k[U][CH];
#pragma unroll
        for (int u = 0; u < U; ++u) ldg_chunk(k[u], head + (size_t)max(tok[u], 0) * C + c, tok[u] >= 0);
#pragma unroll
        for (int i = 0; i < CH; ++i)
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int x = 0; x < QT; ++x) s[x][u] = fmaf(q[x][c + i], k[u][i], s[x][u]);
    }
}
// acc[x] += sum of f[x][u] row tok[u]
template <typename T, int QT, int U, int N>
__device__ __forceinline__ void axpy_far(float (&acc)[QT][N], const float (&f)[QT][U], const T* head, const int (&tok)[U], int C) {
    constexpr int CH = 16 / (int)sizeof(T);
#pragma unroll
    for (int c = 0; c < N; c += CH) {
        float v[U][CH];
#pragma unroll
        for (int u = 0; u < U; ++u) ldg_chunk(v[u], head + (size_t)max(tok[u], 0) * C + c, tok[u] >= 0);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < CH; ++i)
#pragma unroll
                for (int x = 0; x < QT; ++x) acc[x][c + i] = fmaf(f[x][u], v[u][i], acc[x][c + i]);
    }
}
template <int N>
__device__ __forceinline__ float dot(const float (&a)[N], const float (&b)[N]) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) s = fmaf(a[i], b[i], s);
    return s;
}
// the same in four chains
template <int N>
__device__ __forceinline__ float dot4(const float (&a)[N], const float (&b)[N]) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < N; ++i) s[i & 3] = fmaf(a[i], b[i], s[i & 3]);
    return (s[0] + s[1]) + (s[2] + s[3]);
}
// acc += f b, two channels per instruction
template <int N>
__device__ __forceinline__ void axpy(float (&acc)[N], float f, const float (&b)[N]) {
    const float2 f2 = make_float2(f, f);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float2 r = __ffma2_rn(f2, make_float2(b[i], b[i + 1]), make_float2(acc[i], acc[i + 1]));
        acc[i] = r.x; acc[i + 1] = r.y;
    }
}
// Sums QT rows of N channels over 2^ksl neighbouring lanes, lane ks of them weighing its share by f[x]: every round a lane
// hands half of what it still holds to its partner and keeps the other half.  Afterwards the lane holds `held` consecutive
// values from `first` on of the QT x N values (row-major), at least four.
template <int QT, int N>
__device__ __forceinline__ void sum_shares(float (&v)[QT][N], int ksl, int ks, int* first, int* held) {
    float* w = &v[0][0];
    int at = 0, n = QT * N;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        constexpr int ALL = QT * N;
        const int half = ALL >> (r + 1);
        if (r < ksl) {
            const bool up = (ks >> r) & 1;
#pragma unroll
            for (int i = 0; i < ALL / 2; ++i) {
                if (i < half) {
                    const float give = up ? w[i] : w[i + half], keep = up ? w[i + half] : w[i];
                    w[i] = keep + __shfl_xor_sync(0xffffffffu, give, 1 << r);
                }
            }
            n = half;
            at += up ? half : 0;
        }
    }
    *first = at; *held = n;
}
// values 4 i .. 4 i + 3 of what sum_shares left, for all of them: f(x, channel, float4)
template <int QT, int N, typename F>
__device__ __forceinline__ void for_held(const float (&v)[QT][N], int first, int held, F&& f) {
    const float* w = &v[0][0];
#pragma unroll
    for (int i = 0; i < QT * N; i += 4) {
        if (i < held) {
            const int at = first + i;
            f(at / N, at % N, make_float4(w[i], w[i + 1], w[i + 2], w[i + 3]));
        }
    }
}
__device__ __forceinline__ void store4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float4& v) {
    *reinterpret_cast<uint2*>(p) = make_uint2(pack2_bf16(v.x, v.y), pack2_bf16(v.z, v.w));
}

// Rows 0 .. n - 1 of two tensors into shared memory; tok_at(row, at): token (-1 for a row of zeros) and the byte offset
// of the row from the start of its tensor's rows.
template <typename T, int D, typename TokAt>
__device__ __forceinline__ void simt_copy_rows(uint32_t dst_a, uint32_t dst_b, const T* A, const T* B, int C, int n, TokAt&& tok_at) {
    constexpr int CH = D * (int)sizeof(T) / 16;
    for (int e = threadIdx.x; e < n * 4; e += blockDim.x) {
        const int row = e >> 2;
        uint32_t at;
        const int tok = tok_at(row, at);
        const size_t off = (size_t)(tok < 0 ? 0 : tok) * C;
        const uint32_t bytes = tok < 0 ? 0u : 16u;
#pragma unroll
        for (int c0 = 0; c0 < CH; c0 += 4) {
            const int c = c0 + (e & 3);
            if (CH % 4 == 0 || c < CH) {
                ptx::cp_async_16(dst_a + at + c * 16, A + off + c * (16 / sizeof(T)), bytes);
                ptx::cp_async_16(dst_b + at + c * 16, B + off + c * (16 / sizeof(T)), bytes);
            }
        }
    }
}

// Keys (queries) that do not count have the probability 0 and must read zeros: 0 times an infinity or NaN of some other region's
// row would not be 0.  In a stage they have rows of zeros in their own places (tok_at() says -1); a resident slice has one here.
__device__ __forceinline__ void simt_zero_rows(uint8_t* smem, const SimtGeom& gm) {
    const int n = gm.row / 16;
    for (int e = threadIdx.x; e < 2 * n; e += blockDim.x)
        *reinterpret_cast<uint4*>(smem + (e < n ? gm.off_a + e * 16 : gm.off_b + (e - n) * 16) + gm.zero) = make_uint4(0, 0, 0, 0);
}

// Stage `it` of a walk has arrived (for this thread's copies) and, with two stages, the next one is on its way.
// load(i): starts the copies of stage i; stage 0 was started before.
template <typename F>
__device__ __forceinline__ void simt_advance(const SimtGeom& gm, int it, int n, F&& load) {
    const int next = it + gm.stages - 1;
    if (next > 0 && next < n) load(next);
    if (next > it && next < n) ptx::cp_async_wait<1>(); else ptx::cp_async_wait<0>();
}

// LCE weights of a head as they lie in memory: [D channels][25] (odd stride: lane = channel reads without conflicts)
__device__ __forceinline__ void simt_load_weights(float* s_w, const float* lce_w, int n) {
    for (int e = threadIdx.x; e < n; e += blockDim.x) s_w[e] = __ldg(lce_w + e);
}

__device__ __forceinline__ float simt_ld(const float* p) { return __ldg(p); }
__device__ __forceinline__ float simt_ld(const __nv_bfloat16* p) { return __bfloat162float(__ldg(p)); }
__device__ __forceinline__ void simt_st(float* p, float v) { *p = v; }
__device__ __forceinline__ void simt_st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// Adds the 5 x 5 depthwise correlation of `in` (FLIP: with the flipped filter) to the staged rows of the CTA's regions and
// stores them.  Lane = channel (32 at a time), TS x TS positions per pass: every input value is read once per tile.
// region_at[i]: region i of the CTA.
struct SimtFrom { int r0; __device__ int operator[](int i) const { return r0 + i; } };
template <typename T, int D, int TS, bool FLIP, typename RegionAt>
__device__ __forceinline__ void simt_lce(const float* st, const float* s_w, const float* bias, const T* in, T* out, RegionAt region_at, int nreg, int rows_per_region,
                                         const SimtChunk& c, const Dims& dm, const SimtGeom& gm) {
    constexpr int LANES = D < 32 ? D : 32, GROUPS = D / LANES, SUB = 32 / LANES;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int nty = (c.rows + TS - 1) / TS, ntx = (c.cols + TS - 1) / TS, tiles = nty * ntx;
    const int items = nreg * tiles * GROUPS;
    float w[25], b = 0.f;
    int loaded = -1;
    for (int it = warp * SUB + lane / LANES; it < items; it += nwarps * SUB) {
        const int cg = it % GROUPS, q = it / GROUPS;                  // GROUPS is a constant
        const int rl = q / tiles, tile = q - rl * tiles;
        const int ty = tile / ntx, tx = tile - ty * ntx;
        const int ch = cg * LANES + lane % LANES;
        if (cg != loaded) {
            loaded = cg;
#pragma unroll
            for (int k = 0; k < 25; ++k) w[k] = dm.lce ? s_w[ch * 25 + k] : 0.f;
            b = bias ? __ldg(bias + ch) : 0.f;
        }
        const int r = region_at[rl];
        const int ry = fdiv(r, gm.by_s), rx = r - ry * dm.S;
        const int ly0 = ty * TS, lx0 = tx * TS;                       // within the chunk
        const int y0 = ry * dm.hs + c.y + ly0, x0 = rx * dm.ws + c.x + lx0;
        float acc[TS][TS];
#pragma unroll
        for (int yy = 0; yy < TS; ++yy)
#pragma unroll
            for (int xx = 0; xx < TS; ++xx) acc[yy][xx] = b;
        if (dm.lce) {
            bool in_x[TS + 4];
#pragma unroll
            for (int cc = 0; cc < TS + 4; ++cc) in_x[cc] = (unsigned)(x0 + cc - 2) < (unsigned)dm.W0;
            const T* p = in + (ptrdiff_t)((y0 - 2) * dm.W0 + x0 - 2) * dm.C + ch;
#pragma unroll
            for (int rr = 0; rr < TS + 4; ++rr) {
                const bool in_y = (unsigned)(y0 + rr - 2) < (unsigned)dm.H0;
                float v[TS + 4];
#pragma unroll
                for (int cc = 0; cc < TS + 4; ++cc) v[cc] = in_y && in_x[cc] ? simt_ld(p + cc * dm.C) : 0.f;
                p += (ptrdiff_t)dm.W0 * dm.C;
#pragma unroll
                for (int yy = 0; yy < TS; ++yy) {
                    const int ti = rr - yy;
                    if (ti < 0 || ti > 4) continue;
#pragma unroll
                    for (int tj = 0; tj < 5; ++tj)
#pragma unroll
                        for (int xx = 0; xx < TS; ++xx) acc[yy][xx] = fmaf(w[FLIP ? 24 - (ti * 5 + tj) : ti * 5 + tj], v[xx + tj], acc[yy][xx]);
                }
            }
        }
#pragma unroll
        for (int yy = 0; yy < TS; ++yy)
#pragma unroll
            for (int xx = 0; xx < TS; ++xx)
                if (ly0 + yy < c.rows && lx0 + xx < c.cols && y0 + yy < dm.H0 && x0 + xx < dm.W0) {
                    const float a = st[(rl * rows_per_region + (ly0 + yy) * gm.cw + lx0 + xx) * (D + 4) + ch];
                    simt_st(out + (ptrdiff_t)((y0 + yy) * dm.W0 + x0 + xx) * dm.C + ch, a + acc[yy][xx]);
                }
    }
}

// How often each region is named by the list of each region of the CTA: cnt[rl][R], counted by count(add) where add(rl, region);
// true if every count is one.
template <typename Count>
__device__ __forceinline__ bool simt_counts(int32_t* cnt, int nreg, int R, Count&& count) {
    for (int e = threadIdx.x; e < nreg * R; e += blockDim.x) cnt[e] = 0;
    __syncthreads();
    count([&](int rl, int r) { atomicAdd(cnt + rl * R + r, 1); });
    __syncthreads();
    bool ones = true;
    for (int e = threadIdx.x; e < nreg * R; e += blockDim.x) ones = ones && cnt[e] == 1;
    return __syncthreads_and(ones);
}

}  // namespace bra
