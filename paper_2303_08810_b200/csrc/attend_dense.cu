// Attention + LCE on small maps with every token as a key (dense_common.cuh), bf16, head dim 32.
// CTA = (image, head, chunk of map rows); a warp owns RT tiles of 16 query tokens and walks all keys in blocks of 32:
// S by m16n8k16 MMAs on fragments read as 16-byte chunks, online softmax, O += P V with V through ldmatrix.  O^att goes
// to the LCE's thread mapping through shared memory (over the slices).
// Per 16 x 16 scores: eight MMAs (64 cycles of a scheduler's tensor pipe), eight exponentials per lane (64 cycles of its MUFU share)
// and about 60 instructions.  What bounds it at 64 x 14 x 14, 8 heads, topk 16: latency - 0.46 instructions per cycle and scheduler
// with 12 warps per SM (128 registers), per issue 1.6 cycles of fixed waits, 0.8 at barriers, 0.7 for loads, 0.7 for the MMA pipe;
// 1.73 waves of CTAs.
// Measured (B200): 64 x 7 x 7, 16 heads, topk 49: forward 161 us with routing -> 16.4 us; 64 x 14 x 14, 8 heads, topk 16:
// level with attend_img.cu (44 us); 46 -> 44 under ncu, bra_forward 55.9 -> 53.9, with the mask as the addend of the scaling.  The other
// side of the rule: dense_pays().
#include "dense_common.cuh"

#include <type_traits>

namespace bra {

using namespace ptx;

// The CTA's tokens one by one (dense_any_nan() says when and why).
__device__ __noinline__ void attend_dense_by_token(const __nv_bfloat16* Qg, const __nv_bfloat16* Vg, const float* lce_w, const float* lce_b,
                                                   __nv_bfloat16* O, float* lse, const uint8_t* smem, bool weighted, const Dims& dm, const DenseGeom& gm) {
    const int h = blockIdx.y, b = blockIdx.z;
    const int N0 = dm.H0 * dm.W0, y0 = blockIdx.x * gm.g.hb;
    const int q0 = y0 * dm.W, nq = min(gm.g.hb, dm.H - y0) * dm.W;
    const size_t head = (size_t)b * N0 * dm.C + (size_t)h * 32;
    const uint8_t* reg = smem + gm.off_reg;
    const float* bias = reinterpret_cast<const float*>(smem + gm.off_bias);
    const float sl2 = dm.scale * 1.4426950408889634f;
    for (int t = threadIdx.x; t < nq; t += blockDim.x) {
        const int2 at = dense_pos(dm, gm, q0 + t);
        if (at.y >= dm.H0 || at.x >= dm.W0) continue;
        const int i = reg[q0 + t], tok = at.y * dm.W0 + at.x;
        const unsigned long long m64 = reinterpret_cast<const unsigned long long*>(smem + gm.off_mask)[i];
        float q[32], o[32], v[32], m = -INFINITY, l = 0.f;
        load_row<32>(Qg + head + (size_t)(uint32_t)tok * dm.C, q);
#pragma unroll
        for (int c = 0; c < 32; ++c) o[c] = 0.f;
        auto score = [&](int j) {
            dense_row32(v, smem + gm.off_a, j);
            return dense_dot(q, v) * sl2 + (weighted ? bias[i * dm.R + reg[j]] : 0.f);
        };
#pragma unroll 1
        for (int j = 0; j < dm.N; ++j)
            if (m64 >> reg[j] & 1) m = fmaxf(m, score(j));
        const float mn = m == -INFINITY ? 0.f : m;
#pragma unroll 1
        for (int j = 0; j < dm.N; ++j)
            if (m64 >> reg[j] & 1) {
                const float p = exp2f(score(j) - mn);
                l += p;
                dense_row32(v, smem + gm.off_b, j);
#pragma unroll
                for (int c = 0; c < 32; ++c) o[c] = fmaf(p, v[c], o[c]);
            }
        const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
        for (int c = 0; c < 32; ++c) o[c] *= inv;
        if (lse) lse[((size_t)b * dm.heads + h) * N0 + tok] = (m + log2f(l)) * 0.6931471805599453f;
        if (dm.lce) dense_lce_row<false>(o, Vg + head, lce_w + (size_t)h * 32 * 25, lce_b ? lce_b + h * 32 : nullptr, at.y, at.x, dm);
        store_row<32>(O + head + (size_t)(uint32_t)tok * dm.C, o);
    }
}

template <int RT, int TX, int NR>
__global__ void __launch_bounds__(256, 2)
attend_dense_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg, const __nv_bfloat16* __restrict__ Vg,
                    const int32_t* index, const float* __restrict__ lce_w, const float* __restrict__ lce_b,
                    __nv_bfloat16* __restrict__ O, float* __restrict__ lse, int32_t* __restrict__ status,
                    const __grid_constant__ Dims dm, const __grid_constant__ DenseGeom gm) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthreads = blockDim.x;
    const int g = lane >> 2, t4 = lane & 3;
    const int h = blockIdx.y, b = blockIdx.z;
    const int y0 = blockIdx.x * gm.g.hb, rows = min(gm.g.hb, dm.H - y0);
    const int q0 = y0 * dm.W, nq = rows * dm.W;                       // the chunk's tokens: whole rows of regions
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
    const int N0 = dm.H0 * dm.W0;
    const size_t head_off = (size_t)b * N0 * tok_bytes + (size_t)h * 64;
    const uint8_t* Qh = reinterpret_cast<const uint8_t*>(Qg) + head_off;
    const uint8_t* Vh = reinterpret_cast<const uint8_t*>(Vg) + head_off;
    const uint32_t ks = sbase + gm.off_a, vs = sbase + gm.off_b;
    Dims map = dm;                                                    // the whole map as one region
    map.ws = dm.W;

    dense_load_slices<2>({ks, vs}, {reinterpret_cast<const uint8_t*>(Kg) + head_off, Vh}, dm, gm, tid, nthreads);
    cp_async_commit();
    float* s_w = reinterpret_cast<float*>(smem + gm.g.off_w);
    if (dm.lce) {
        load_lce_weights(s_w, lce_w, h, 32 * 25, tid, nthreads);
        load_halo<1>(sbase + gm.g.off_halo, Vh, y0, 0, rows, map, gm.g, tid, nthreads);
    }
    cp_async_commit();
    // Q fragments of this warp's tiles
    uint32_t qa[RT][1][2][4];
    int tok[RT][2];                                                   // token in the caller's map, -1: none
    uint32_t where[RT][2];                                            // region, position in the chunk
#pragma unroll
    for (int x = 0; x < RT; ++x) {
        uint4 v[2][1];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int t = (warp * RT + x) * 16 + g + 8 * r;
            const int2 at = dense_pos(dm, gm, q0 + min(t, nq - 1));
            tok[x][r] = t < nq && at.y < dm.H0 && at.x < dm.W0 ? at.y * dm.W0 + at.x : -1;
            where[x][r] = (uint32_t)fdiv(q0 + min(t, nq - 1), dm.n_r, gm.mul_nr) << 16 | (uint32_t)((at.y - y0) * dm.W + at.x);
            ld_row<1>(v[r], Qh + t4 * 16, tok[x][r], tok_bytes);
        }
        rows_to_a<1>(qa[x], v[0], v[1]);
    }
    uint8_t* reg = smem + gm.off_reg;
    float* bias = reinterpret_cast<float*>(smem + gm.off_bias);
    unsigned long long* mask = reinterpret_cast<unsigned long long*>(smem + gm.off_mask);
    dense_regions(reg, dm, gm, tid, nthreads);
    pdl_wait();          // in bra_forward the launch may overlap the tail of the routing kernel
    const int hi = dm.heads_i == 1 ? 0 : h;
    const bool repeats = dense_routes(mask, bias, index ? index + ((size_t)b * dm.heads_i + hi) * dm.R * dm.topk : nullptr, status, dm, gm,
                                      tid, nthreads);
    cp_async_wait<1>();
    __syncthreads();

    const float sl2 = dm.scale * 1.4426950408889634f;
    float m_run[RT][2], l_run[RT][2], o[RT][4][4];
#pragma unroll
    for (int x = 0; x < RT; ++x) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            m_run[x][r] = -INFINITY; l_run[x][r] = 0.f;
        }
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[x][n][e] = 0.f;
    }
    const uint32_t row_off = dense_row_offset(lane), col_off = dense_col_offset(lane);
    auto walk = [&](auto weighted) {
        DenseRow<NR> on[RT][2];
#pragma unroll
        for (int x = 0; x < RT; ++x)
#pragma unroll
            for (int r = 0; r < 2; ++r) on[x][r] = DenseRow<NR>(mask[where[x][r] >> 16], t4);
#pragma unroll 1
        for (int kb = 0; kb < dm.N; kb += 32) {
            float c[RT][4][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 kr[1] = {dense_chunk(ks + (kb + 8 * j) * 64 + row_off)};
#pragma unroll
                for (int x = 0; x < RT; ++x) mma_rows<1>(c[x][j], qa[x], kr);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int x = 0; x < RT; ++x)
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float a = weighted.value ? dense_weight(bias + (where[x][r] >> 16) * dm.R, reg[kb + 8 * j + 2 * t4 + e])
                                                           : on[x][r].pick(0.f, j, e, kb, t4, reg);
                            c[x][j][2 * r + e] = fmaf(c[x][j][2 * r + e], sl2, a);
                        }
#pragma unroll
            for (int x = 0; x < RT; ++x)
#pragma unroll
                for (int r = 0; r < 2; ++r) on[x][r].template next<32>();
            if (NR == DENSE_ALL && kb + 32 > dm.N) {                  // behind the last token
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (kb + 8 * j + 2 * t4 + (e & 1) >= dm.N)
#pragma unroll
                            for (int x = 0; x < RT; ++x) c[x][j][e] = -INFINITY;
            }
            uint32_t pa[2][RT][4];
#pragma unroll
            for (int x = 0; x < RT; ++x) {
                float mx[2];
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    mx[r] = fmaxf(fmax3(fmax3(c[x][0][2 * r], c[x][0][2 * r + 1], c[x][1][2 * r]), c[x][1][2 * r + 1], c[x][2][2 * r]),
                                  fmax3(c[x][2][2 * r + 1], c[x][3][2 * r], c[x][3][2 * r + 1]));
                if (__any_sync(0xffffffffu, mx[0] > m_run[x][0] || mx[1] > m_run[x][1])) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
                        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
                        const float mnew = fmaxf(m_run[x][r], mx[r]);
                        const float corr = mnew == -INFINITY ? 1.f : ex2_approx(m_run[x][r] - mnew);
                        m_run[x][r] = mnew;
                        l_run[x][r] *= corr;
#pragma unroll
                        for (int n = 0; n < 4; ++n) { o[x][n][2 * r] *= corr; o[x][n][2 * r + 1] *= corr; }
                    }
                }
                const float mn0 = m_run[x][0] == -INFINITY ? 0.f : m_run[x][0], mn1 = m_run[x][1] == -INFINITY ? 0.f : m_run[x][1];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    c[x][j][0] = ex2_approx(c[x][j][0] - mn0);
                    c[x][j][1] = ex2_approx(c[x][j][1] - mn0);
                    c[x][j][2] = ex2_approx(c[x][j][2] - mn1);
                    c[x][j][3] = ex2_approx(c[x][j][3] - mn1);
                    l_run[x][0] += c[x][j][0] + c[x][j][1];
                    l_run[x][1] += c[x][j][2] + c[x][j][3];
                }
                frag_hi(pa[0][x], c[x][0], c[x][1]);
                frag_hi(pa[1][x], c[x][2], c[x][3]);
            }
#pragma unroll
            for (int s = 0; s < 2; ++s) dense_mma_tokens<RT>(o, pa[s], vs + (kb + 16 * s) * 64, col_off);
        }
    };
    if (NR != DENSE_ALL && repeats) walk(std::true_type());
    else walk(std::false_type());
    cp_async_wait<0>();
    if (__syncthreads_or(dense_any_nan(o))) {                         // the slices have been read: staging takes their place
        attend_dense_by_token(Qg, Vg, lce_w, lce_b, O, lse, smem, repeats, dm, gm);
        return;
    }
    float* st = reinterpret_cast<float*>(smem + gm.g.off_st);
#pragma unroll
    for (int x = 0; x < RT; ++x)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float l = l_run[x][r];
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            if (tok[x][r] < 0) continue;
            const float inv = l > 0.f ? 1.f / l : 0.f;
            float* dst = st + (where[x][r] & 0xffffu) * dn::ST + 2 * t4;
#pragma unroll
            for (int n = 0; n < 4; ++n) *reinterpret_cast<float2*>(dst + 8 * n) = make_float2(o[x][n][2 * r] * inv, o[x][n][2 * r + 1] * inv);
            if (lse && t4 == 0) lse[((size_t)b * dm.heads + h) * N0 + tok[x][r]] = (m_run[x][r] + log2f(l)) * 0.6931471805599453f;
        }
    __syncthreads();
    lce_chunk<1, 4, TX, false, dn::ST>(st, sbase + gm.g.off_halo, s_w, dm.lce && lce_b ? lce_b + h * 32 : nullptr, dm.lce, O + head_off / 2, y0, 0,
                                       rows, map, gm.g, warp, gm.nw, lane);
}

// ------------------------------------------------------------------ host side
// Rows of regions per CTA: all of them where the (image, head) pairs fill the GPU, else about four map rows (an LCE tile).
static int chunk_rows(const Dims& d) {
    return (long long)d.B * d.heads < 2 * kSMs && d.hs < 4 && d.H > 4 ? (4 + d.hs - 1) / d.hs : d.S;
}

bool attend_dense_supported(const Dims& d, int dtype) {
    return dense_supported(d, dtype) && dense_geom(d, 2, chunk_rows(d)).smem_bytes <= 200 * 1024;
}

template <int RT, int TX, int NR>
static cudaError_t launch_t(const Dims& d, const DenseGeom& g, const void* Q, const void* K, const void* V, const int32_t* index,
                            const float* lce_w, const float* lce_b, void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    auto kernel = attend_dense_kernel<RT, TX, NR>;
    static PerDeviceMax smem_set;
    if (g.smem_bytes > 48 * 1024) {
        const cudaError_t e = smem_set.ensure(g.smem_bytes, [&] {
            return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, g.smem_bytes);
        });
        if (e != cudaSuccess) return e;
    }
    typedef __nv_bfloat16 bf;
    return grid_pieces(d, [&](const GridPiece& p) {
        count_launch();
        return launch_kernel(kernel, dim3(g.g.chunks, p.heads, p.images), dim3(g.nw * 32), (size_t)g.smem_bytes, st, after_own_kernel,
                             static_cast<const bf*>(Q) + p.tensor, static_cast<const bf*>(K) + p.tensor, static_cast<const bf*>(V) + p.tensor,
                             piece_of(index, p.index), piece_of(lce_w, p.channel * 25), piece_of(lce_b, p.channel), static_cast<bf*>(O) + p.tensor,
                             piece_of(lse, p.stat), status, d, g);
    });
}

cudaError_t launch_attend_dense(const Dims& d, const void* Q, const void* K, const void* V,
                                const int32_t* index, const float* lce_w, const float* lce_b,
                                void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    const DenseGeom g = dense_geom(d, 2, chunk_rows(d));
    Dims map = d;
    map.ws = d.W;
    const int tx = lce_tile_width(g.g, map);
#define BRA_GO(RT, TX, NR) return launch_t<RT, TX, NR>(d, g, Q, K, V, index, lce_w, lce_b, O, lse, status, st, after_own_kernel)
    // nothing to mask but what is behind the map (picked like any list: 24 x 12 x 12, 24 heads, S = 7, topk 49 33.3 -> 35.2 us, 64 x 7 x 7,
    // 16 heads 14.2 -> 14.5)
    if (!index) {
        if (g.np <= 8) { if (tx == 2) BRA_GO(1, 2, DENSE_ALL); BRA_GO(1, 4, DENSE_ALL); }
        if (tx == 2) BRA_GO(2, 2, DENSE_ALL);
        BRA_GO(2, 4, DENSE_ALL);
    }
    if (d.n_r == 1) { if (tx == 2) BRA_GO(1, 2, 1); BRA_GO(1, 4, 1); }                    // at most 64 tokens
    if (d.n_r == 4) {
        if (g.np <= 8) { if (tx == 2) BRA_GO(1, 2, 4); BRA_GO(1, 4, 4); }
        if (tx == 2) BRA_GO(2, 2, 4);
        BRA_GO(2, 4, 4);
    }
    if (g.np <= 8) { if (tx == 2) BRA_GO(1, 2, 0); BRA_GO(1, 4, 0); }
    if (tx == 2) BRA_GO(2, 2, 0);
    BRA_GO(2, 4, 0);
#undef BRA_GO
}

}  // namespace bra
