// Gradients of the routed attention for a fixed routing index on small maps with every token on the other side
// (dense_common.cuh), bf16, head dim 32: one launch, CTA = (image, head), the slices of Q, K, V and dO resident.
//   1. warp = 16 queries: delta = rowsum(P o dP) in a first walk over the keys, dQ = scale dS K in a second
//   2. warp = 16 keys: dK = scale dS^T Q and dV = P^T dO in one walk over the queries; dV + LCE adjoint
// P from the saved log-sum-exp, dP = dO V^T, dS = P o (dP - delta).  Who is routed where is the bit masks (with repeats a table
// of log2 of the counts), so no inverse index is needed.  Every sum has a fixed order.
// Bound: latency at 12 warps per SM (0.46 instructions per cycle and scheduler; per issue 1.3 cycles of fixed waits, 1.1 at
// barriers, 0.84 for the MMA pipe), 1.73 waves; the two walks over the keys in 1. make S and dP twice.  Measured (B200) against the kernels of
// backward_img.cu: 64 x 14 x 14, 8 heads, topk 16: 156 -> 103 us; 64 x 7 x 7, 16 heads, topk 49: 477 -> 39 us.  With the mask picked
// before the exponential, a walk of its own for lists with repeats and the slices' swizzle out of the walks (12.2 k -> 10.3 k
// instructions a warp): 96 -> 84 us, forward + backward 155.5 -> 142.2; 64 x 12 x 12 153.0 -> 138.4; 64 x 9 x 9, S = 3 69.8 -> 65.0.
#include "dense_common.cuh"

#include <type_traits>

namespace bra {

using namespace ptx;

// The gradients of an (image, head) token by token (dense_any_nan() says when and why).
__device__ __noinline__ void bwd_dense_by_token(const float* lce_w, const __nv_bfloat16* dOg, __nv_bfloat16* dQg, __nv_bfloat16* dKg, __nv_bfloat16* dVg,
                                                uint8_t* smem, bool weighted, const Dims& dm, const DenseGeom& gm) {
    const int h = blockIdx.y, b = blockIdx.z;
    const size_t head = (size_t)b * dm.H0 * dm.W0 * dm.C + (size_t)h * 32;
    const uint8_t *qs = smem + gm.off_a, *ks = smem + gm.off_b, *vs = smem + gm.off_c, *gs = smem + gm.off_d, *reg = smem + gm.off_reg;
    const float* bias = reinterpret_cast<const float*>(smem + gm.off_bias);
    const unsigned long long* mask = reinterpret_cast<const unsigned long long*>(smem + gm.off_mask);
    const float* l2 = reinterpret_cast<const float*>(smem + gm.off_stat);
    float* dl = reinterpret_cast<float*>(smem + gm.off_stat) + gm.rows;
    const float sl2 = dm.scale * 1.4426950408889634f;
    auto on_map = [&](const int2& at) { return at.y < dm.H0 && at.x < dm.W0; };
    auto store = [&](__nv_bfloat16* out, const int2& at, float (&v)[32], float f) {
#pragma unroll
        for (int c = 0; c < 32; ++c) v[c] *= f;
        store_row<32>(out + head + (size_t)(uint32_t)(at.y * dm.W0 + at.x) * dm.C, v);
    };
    for (int t = threadIdx.x; t < dm.N; t += blockDim.x) {            // queries
        const int2 at = dense_pos(dm, gm, t);
        if (!on_map(at)) continue;
        const int i = reg[t];
        float q[32], g[32], row[32], acc[32], delta = 0.f;
        dense_row32(q, qs, t);
        dense_row32(g, gs, t);
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[c] = 0.f;
#pragma unroll 1
        for (int it = 0; it < 2 * dm.N; ++it) {
            const int j = it < dm.N ? it : it - dm.N;
            if (!(mask[i] >> reg[j] & 1)) continue;
            dense_row32(row, vs, j);
            const float dp = dense_dot(g, row);
            dense_row32(row, ks, j);
            const float p = exp2f(dense_dot(q, row) * sl2 + (weighted ? bias[i * dm.R + reg[j]] : 0.f) - l2[t]);
            if (it < dm.N) { delta = fmaf(p, dp, delta); continue; }
            const float ds = p * (dp - delta);
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[c] = fmaf(ds, row[c], acc[c]);
        }
        dl[t] = delta;
        store(dQg, at, acc, dm.scale);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < dm.N; t += blockDim.x) {            // keys
        const int2 at = dense_pos(dm, gm, t);
        if (!on_map(at)) continue;
        const int j = reg[t];
        float k[32], v[32], row[32], gk[32], gv[32];
        dense_row32(k, ks, t);
        dense_row32(v, vs, t);
#pragma unroll
        for (int c = 0; c < 32; ++c) gk[c] = gv[c] = 0.f;
#pragma unroll 1
        for (int i = 0; i < dm.N; ++i) {
            if (!(mask[64 + j] >> reg[i] & 1)) continue;
            dense_row32(row, qs, i);
            const float p = exp2f(dense_dot(k, row) * sl2 + (weighted ? bias[reg[i] * dm.R + j] : 0.f) - l2[i]);
            float g[32];
            dense_row32(g, gs, i);
            const float ds = p * (dense_dot(v, g) - dl[i]);
#pragma unroll
            for (int c = 0; c < 32; ++c) { gk[c] = fmaf(ds, row[c], gk[c]); gv[c] = fmaf(p, g[c], gv[c]); }
        }
        store(dKg, at, gk, dm.scale);
        if (dm.lce) dense_lce_row<true>(gv, dOg + head, lce_w + (size_t)h * 32 * 25, nullptr, at.y, at.x, dm);
        store(dVg, at, gv, 1.f);
    }
}

template <int TX, int NR>
__global__ void __launch_bounds__(256, 2)
bwd_dense_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg, const __nv_bfloat16* __restrict__ Vg,
                 const int32_t* __restrict__ index, const float* __restrict__ lse, const __nv_bfloat16* __restrict__ dOg,
                 const float* __restrict__ lce_w, __nv_bfloat16* __restrict__ dQg, __nv_bfloat16* __restrict__ dKg,
                 __nv_bfloat16* __restrict__ dVg, int32_t* __restrict__ status, const __grid_constant__ Dims dm,
                 const __grid_constant__ DenseGeom gm) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthreads = blockDim.x;
    const int g = lane >> 2, t4 = lane & 3;
    const int h = blockIdx.y, b = blockIdx.z;
    const int N0 = dm.H0 * dm.W0;
    const size_t head_off = (size_t)b * N0 * dm.C * 2 + (size_t)h * 64;
    const uint8_t* Gh = reinterpret_cast<const uint8_t*>(dOg) + head_off;
    const uint32_t qs = sbase + gm.off_a, ks = sbase + gm.off_b, vs = sbase + gm.off_c, gs = sbase + gm.off_d;
    Dims map = dm;
    map.ws = dm.W;

    dense_load_slices<4>({qs, ks, vs, gs}, {reinterpret_cast<const uint8_t*>(Qg) + head_off, reinterpret_cast<const uint8_t*>(Kg) + head_off,
                                            reinterpret_cast<const uint8_t*>(Vg) + head_off, Gh}, dm, gm, tid, nthreads);
    cp_async_commit();
    float* s_w = reinterpret_cast<float*>(smem + gm.g.off_w);
    if (dm.lce) {
        load_lce_weights(s_w, lce_w, h, 32 * 25, tid, nthreads);
        load_halo<1>(sbase + gm.g.off_halo, Gh, 0, 0, dm.H, map, gm.g, tid, nthreads);
    }
    cp_async_commit();
    // lse * log2(e) and delta per token; a token behind the last has lse = inf (P = 0); one of the zero padding has zero rows
    // of Q and dO and lse = delta = 0: as a query it adds nothing
    float* s_l2 = reinterpret_cast<float*>(smem + gm.off_stat);
    float* s_dl = s_l2 + gm.rows;
    const float* lse_h = lse + ((size_t)b * dm.heads + h) * N0;
    for (int t = tid; t < gm.rows; t += nthreads) {
        const int2 at = dense_pos(dm, gm, t);
        s_l2[t] = t >= dm.N ? INFINITY : at.y < dm.H0 && at.x < dm.W0 ? __ldg(lse_h + at.y * dm.W0 + at.x) * 1.4426950408889634f : 0.f;
        s_dl[t] = 0.f;
    }
    uint8_t* reg = smem + gm.off_reg;
    float* bias = reinterpret_cast<float*>(smem + gm.off_bias);
    dense_regions(reg, dm, gm, tid, nthreads);
    const int hi = dm.heads_i == 1 ? 0 : h;
    unsigned long long* mask = reinterpret_cast<unsigned long long*>(smem + gm.off_mask);
    const bool repeats = dense_routes(mask, bias, index + ((size_t)b * dm.heads_i + hi) * dm.R * dm.topk, status, dm, gm, tid, nthreads);
    cp_async_wait<1>();
    __syncthreads();

    const float sl2 = dm.scale * 1.4426950408889634f;
    const int steps = (dm.N + 15) / 16;
    // token t in the caller's map, -1 in the padding
    auto token = [&](int t) -> int {
        const int2 at = dense_pos(dm, gm, t);
        return t < dm.N && at.y < dm.H0 && at.x < dm.W0 ? at.y * dm.W0 + at.x : -1;
    };

    // ---- queries: delta, dQ ----
    const uint32_t row_off = dense_row_offset(lane), col_off = dense_col_offset(lane);
    bool nan = false;
    auto queries = [&](auto weighted) {
#pragma unroll 1
        for (int tile = warp; tile < steps; tile += gm.nw) {
            const int r0 = tile * 16;
            uint32_t qa[1][2][4], ga[1][2][4];
            dense_a(qa, qs + r0 * 64 + row_off);
            dense_a(ga, gs + r0 * 64 + row_off);
            const float l0 = s_l2[r0 + g], l1 = s_l2[r0 + 8 + g];
            const int i0 = min((int)reg[r0 + g], dm.R - 1), i1 = min((int)reg[r0 + 8 + g], dm.R - 1);
            float delta[2] = {0.f, 0.f}, dq[1][4][4];
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) dq[0][n][e] = 0.f;
            // P and dP of 16 keys
            auto scores = [&](float (&c)[2][4], float (&dp)[2][4], DenseRow<NR>& on0, DenseRow<NR>& on1, int kb) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const uint4 kr[1] = {dense_chunk(ks + (kb + 8 * j) * 64 + row_off)}, vr[1] = {dense_chunk(vs + (kb + 8 * j) * 64 + row_off)};
                    mma_rows<1>(c[j], qa, kr);
                    mma_rows<1>(dp[j], ga, vr);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int r = weighted.value ? reg[kb + 8 * j + 2 * t4 + e] : 0;
                        const float a = weighted.value ? dense_weight(bias + i0 * dm.R, r) - l0 : on0.pick(-l0, j, e, kb, t4, reg);
                        const float b = weighted.value ? dense_weight(bias + i1 * dm.R, r) - l1 : on1.pick(-l1, j, e, kb, t4, reg);
                        c[j][e] = ex2_approx(fmaf(c[j][e], sl2, a));
                        c[j][2 + e] = ex2_approx(fmaf(c[j][2 + e], sl2, b));
                    }
                on0.template next<16>();
                on1.template next<16>();
            };
            {
                DenseRow<NR> on0(mask[i0], t4), on1(mask[i1], t4);
#pragma unroll 2
                for (int kb = 0; kb < dm.N; kb += 16) {
                    float c[2][4], dp[2][4];
                    scores(c, dp, on0, on1, kb);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        delta[0] = fmaf(c[j][0], dp[j][0], fmaf(c[j][1], dp[j][1], delta[0]));
                        delta[1] = fmaf(c[j][2], dp[j][2], fmaf(c[j][3], dp[j][3], delta[1]));
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                delta[r] += __shfl_xor_sync(0xffffffffu, delta[r], 1);
                delta[r] += __shfl_xor_sync(0xffffffffu, delta[r], 2);
            }
            {
                DenseRow<NR> on0(mask[i0], t4), on1(mask[i1], t4);
#pragma unroll 2
                for (int kb = 0; kb < dm.N; kb += 16) {
                    float c[2][4], dp[2][4];
                    scores(c, dp, on0, on1, kb);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        c[j][0] *= dp[j][0] - delta[0]; c[j][1] *= dp[j][1] - delta[0];
                        c[j][2] *= dp[j][2] - delta[1]; c[j][3] *= dp[j][3] - delta[1];
                    }
                    uint32_t sa[1][4];
                    frag_hi(sa[0], c[0], c[1]);
                    dense_mma_tokens<1>(dq, sa, ks + kb * 64, col_off);
                }
            }
            nan = nan || dense_any_nan(dq) || delta[0] != delta[0] || delta[1] != delta[1];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int t = r0 + g + 8 * r, tok = token(t);
                if (tok < 0) continue;                                    // delta of a padding row stays 0
                if (t4 == 0) s_dl[t] = delta[r];
                uint32_t* o = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(dQg) + head_off) + (size_t)(uint32_t)tok * (dm.C / 2) + t4;
#pragma unroll
                for (int n = 0; n < 4; ++n) o[4 * n] = pack2_bf16(dq[0][n][2 * r] * dm.scale, dq[0][n][2 * r + 1] * dm.scale);
            }
        }
    };
    if (repeats) queries(std::true_type());
    else queries(std::false_type());
    if (__syncthreads_or(nan)) {
        cp_async_wait<0>();
        bwd_dense_by_token(lce_w, dOg, dQg, dKg, dVg, smem, repeats, dm, gm);
        return;
    }

    // ---- keys: dK, dV (a warp has at most two tiles; dV is staged once all warps have read the slices) ----
    float dv[2][4][4];
    auto keys = [&](auto weighted) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int r0 = (warp + x * gm.nw) * 16;
            if (r0 >= steps * 16) continue;
            uint32_t ka[1][2][4], va[1][2][4];
            dense_a(ka, ks + r0 * 64 + row_off);
            dense_a(va, vs + r0 * 64 + row_off);
            const int k0 = min((int)reg[r0 + g], dm.R - 1), k1 = min((int)reg[r0 + 8 + g], dm.R - 1);
            DenseRow<NR> on0(mask[64 + k0], t4), on1(mask[64 + k1], t4);
            float dk[1][4][4];
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) dk[0][n][e] = dv[x][n][e] = 0.f;
#pragma unroll 2
            for (int qb = 0; qb < dm.N; qb += 16) {
                float c[2][4], dp[2][4];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const uint4 qr[1] = {dense_chunk(qs + (qb + 8 * j) * 64 + row_off)}, gr[1] = {dense_chunk(gs + (qb + 8 * j) * 64 + row_off)};
                    mma_rows<1>(c[j], ka, qr);
                    mma_rows<1>(dp[j], va, gr);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int q = qb + 8 * j + 2 * t4;
                    const float2 l2 = *reinterpret_cast<const float2*>(s_l2 + q), dl = *reinterpret_cast<const float2*>(s_dl + q);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float l = e ? l2.y : l2.x, d = e ? dl.y : dl.x;
                        const int r = weighted.value ? reg[q + e] : 0;
                        const float a = weighted.value ? (r < 64 ? bias[r * dm.R + k0] : -INFINITY) - l : on0.pick(-l, j, e, qb, t4, reg);
                        const float b = weighted.value ? (r < 64 ? bias[r * dm.R + k1] : -INFINITY) - l : on1.pick(-l, j, e, qb, t4, reg);
                        c[j][e] = ex2_approx(fmaf(c[j][e], sl2, a));
                        c[j][2 + e] = ex2_approx(fmaf(c[j][2 + e], sl2, b));
                        dp[j][e] -= d;
                        dp[j][2 + e] -= d;
                    }
                }
                on0.template next<16>();
                on1.template next<16>();
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) dp[j][e] *= c[j][e];
                uint32_t a[1][4];
                frag_hi(a[0], dp[0], dp[1]);
                dense_mma_tokens<1>(dk, a, qs + qb * 64, col_off);
                frag_hi(a[0], c[0], c[1]);
                dense_mma_tokens<1>(dv + x, a, gs + qb * 64, col_off);
            }
            nan = nan || dense_any_nan(dk) || dense_any_nan(reinterpret_cast<const float (&)[1][4][4]>(dv[x]));
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int tok = token(r0 + g + 8 * r);
                if (tok < 0) continue;
                uint32_t* o = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(dKg) + head_off) + (size_t)(uint32_t)tok * (dm.C / 2) + t4;
#pragma unroll
                for (int n = 0; n < 4; ++n) o[4 * n] = pack2_bf16(dk[0][n][2 * r] * dm.scale, dk[0][n][2 * r + 1] * dm.scale);
            }
        }
    };
    if (repeats) keys(std::true_type());
    else keys(std::false_type());
    cp_async_wait<0>();
    if (__syncthreads_or(nan)) {
        bwd_dense_by_token(lce_w, dOg, dQg, dKg, dVg, smem, repeats, dm, gm);
        return;
    }
    float* st = reinterpret_cast<float*>(smem + gm.g.off_st);
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int r0 = (warp + x * gm.nw) * 16;
        if (r0 >= steps * 16) continue;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int t = r0 + g + 8 * r;
            if (t >= dm.N) continue;
            const int2 at = dense_pos(dm, gm, t);
            float* dst = st + (at.y * dm.W + at.x) * dn::ST + 2 * t4;
#pragma unroll
            for (int n = 0; n < 4; ++n) *reinterpret_cast<float2*>(dst + 8 * n) = make_float2(dv[x][n][2 * r], dv[x][n][2 * r + 1]);
        }
    }
    __syncthreads();
    // ---- LCE adjoint + store of dV: correlation of dO with the flipped filter ----
    lce_chunk<1, 4, TX, true, dn::ST>(st, sbase + gm.g.off_halo, s_w, nullptr, dm.lce, dVg + head_off / 2, 0, 0, dm.H, map, gm.g, warp, gm.nw, lane);
}

// ------------------------------------------------------------------ host side
bool backward_dense_supported(const Dims& d, int dtype) {
    return dense_supported(d, dtype) && dense_geom(d, 4, d.S).smem_bytes <= 200 * 1024;
}

template <int TX, int NR>
static cudaError_t launch_t(const Dims& d, const DenseGeom& g, const void* Q, const void* K, const void* V, const int32_t* index,
                            const float* lce_w, const float* lse, const void* dO, void* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st) {
    auto kernel = bwd_dense_kernel<TX, NR>;
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
        return launch_kernel(kernel, dim3(1, p.heads, p.images), dim3(g.nw * 32), (size_t)g.smem_bytes, st, false,
                             static_cast<const bf*>(Q) + p.tensor, static_cast<const bf*>(K) + p.tensor, static_cast<const bf*>(V) + p.tensor,
                             index + p.index, lse + p.stat, static_cast<const bf*>(dO) + p.tensor, piece_of(lce_w, p.channel * 25),
                             static_cast<bf*>(dQ) + p.tensor, static_cast<bf*>(dK) + p.tensor, static_cast<bf*>(dV) + p.tensor, status, d, g);
    });
}

cudaError_t launch_backward_dense(const Dims& d, const void* Q, const void* K, const void* V, const int32_t* index, const float* lce_w,
                                  const float* lse, const void* dO, void* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st) {
    const DenseGeom g = dense_geom(d, 4, d.S);
    Dims map = d;
    map.ws = d.W;
    const bool narrow = lce_tile_width(g.g, map) == 2;
#define BRA_GO(TX, NR) return launch_t<TX, NR>(d, g, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, status, st)
    if (d.n_r == 4) { if (narrow) BRA_GO(2, 4); BRA_GO(4, 4); }
    if (d.n_r == 1) { if (narrow) BRA_GO(2, 1); BRA_GO(4, 1); }
    if (narrow) BRA_GO(2, 0);
    BRA_GO(4, 0);
#undef BRA_GO
}

}  // namespace bra
