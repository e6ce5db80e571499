// Gradients of the routed attention for a fixed routing index (Eq. 7 with Eq. 1) with warp-level tensor-core MMAs:
// head dim 32 or 64, bf16, any region shape, any topk, any map.  With P the softmax of Eq. 1 over a group's routed keys
// (recomputed from the saved log-sum-exp): dP = dO V^g^T, delta = rowsum(P o dP), dS = P o (dP - delta),
//   dQ = scale dS K^g                                    (query-centric kernel)
//   dK_j = scale sum dS^T Q, dV_j = sum P^T dO  over the query regions that routed to j,
//   in the fixed order of the inverse routing index      (key-centric kernel)
//   dV += LCE adjoint of dO (5x5 depthwise correlation with the flipped filter).
// The structure is the forward kernel's (attend_direct.cu): a warp owns 16 rows, the other side streams from global
// memory straight into MMA fragments, a table of token numbers per group, no barriers in the streaming loop.  A row
// that was loaded serves both products it takes part in: as loaded where the contraction runs over channels, through
// movmatrix where it runs over tokens.  No atomics: every sum has a fixed order, results are bit-identical from run
// to run.
#include "direct_common.cuh"
#include "inverse_index.cuh"

namespace bra {

using namespace ptx;

// ------------------------------------------------------------------ dQ and delta
// The CTAs of grid row 0 build the inverse routing index for the dK / dV kernel instead.
// SINGLE: all keys of a group (at most 64) in one block, S and dP computed once; otherwise one sweep for delta and
// one for dQ.
template <int PL, bool EXACT, bool SINGLE, bool ZEROS>
__global__ void __launch_bounds__(PL == 2 ? 128 : 256, PL == 2 ? 3 : 2)
bwd_dq_direct_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg,
                     const __nv_bfloat16* __restrict__ Vg, const int32_t* __restrict__ index,
                     const float* __restrict__ lse, const __nv_bfloat16* __restrict__ dOg,
                     __nv_bfloat16* __restrict__ dQg, float* __restrict__ delta_out,
                     int32_t* __restrict__ inv_off, int32_t* __restrict__ inv_list, bool inv_bits,
                     int32_t* __restrict__ status, Dims dm, DirGeom gm) {
    constexpr int KS = SINGLE ? 4 : 2;                                // 16-key steps per block
    extern __shared__ __align__(128) uint8_t smem[];
    // blockIdx.y = 0: the inverse index (one CTA per (image, routing head)); else head blockIdx.y - 1
    if (blockIdx.y == 0) {
        if ((int)blockIdx.x < dm.heads_i)
            inverse_index_job(index, inv_off, inv_list, blockIdx.z * dm.heads_i + blockIdx.x, reinterpret_cast<int32_t*>(smem), inv_bits, dm);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const bool one_warp = gm.gpc > 1;
    const int rest = blockIdx.x, h = blockIdx.y - 1, b = blockIdx.z;
    const int grp = one_warp ? warp : 0;
    const int ck = one_warp ? 0 : rest % gm.chunks;
    const int i = one_warp ? rest * gm.gpc + warp : rest / gm.chunks;
    const int gwarp = one_warp ? 0 : warp, gwarps = one_warp ? 1 : gm.nw;
    const int glane = one_warp ? lane : tid, glanes = gwarps * 32;
    if (i >= dm.R || rest >= gm.gpi) return;                                            // a whole warp of a CTA without CTA barriers
    auto group_sync = [&]() { if (one_warp) __syncwarp(); else __syncthreads(); };

    const int c0 = ck * gm.hb * dm.ws;                                // first token of the chunk in its region
    const int ntok = min(gm.hb, dm.hs - ck * gm.hb) * dm.ws;
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
    const int N0 = dm.H0 * dm.W0;
    const size_t head_off = (size_t)b * N0 * tok_bytes + (size_t)h * 64 * PL + t4 * 16;
    const uint8_t* Qb = reinterpret_cast<const uint8_t*>(Qg) + head_off;
    const uint8_t* Kb = reinterpret_cast<const uint8_t*>(Kg) + head_off;
    const uint8_t* Vb = reinterpret_cast<const uint8_t*>(Vg) + head_off;
    const uint8_t* Gb = reinterpret_cast<const uint8_t*>(dOg) + head_off;
    uint8_t* dQb = reinterpret_cast<uint8_t*>(dQg) + head_off;
    const size_t stat0 = ((size_t)b * dm.heads + h) * N0;
    const int hi = dm.heads_i == 1 ? 0 : h;
    const int32_t* irow = index + (((size_t)b * dm.heads_i + hi) * dm.R + i) * dm.topk;
    const int total = dm.topk * dm.n_r;
    uint32_t* tab = reinterpret_cast<uint32_t*>(smem + gm.off_tab) + grp * gm.tab;
    const float sl2 = dm.scale * 1.4426950408889634f;
    const int passes = (total + gm.tab - 1) / gm.tab;
    bool any_bad = false, filled = false;

    for (int tile = gwarp; tile - gwarp < gm.tpc; tile += gwarps) {
        const bool has = tile * 16 < ntok;
        int tok[2];
        float lse2[2];
        uint32_t qa[PL][2][4], ga[PL][2][4];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int tk = tile * 16 + g + 8 * r;
            tok[r] = tk < ntok ? token_of(dm, gm, i, c0 + tk) : -1;
            lse2[r] = tok[r] >= 0 ? __ldg(lse + stat0 + tok[r]) * 1.4426950408889634f : 0.f;
        }
        {
            uint4 lo[PL], up[PL];
            ld_row<PL>(lo, Qb, tok[0], tok_bytes); ld_row<PL>(up, Qb, tok[1], tok_bytes);
            rows_to_a<PL>(qa, lo, up);
            ld_row<PL>(lo, Gb, tok[0], tok_bytes); ld_row<PL>(up, Gb, tok[1], tok_bytes);
            rows_to_a<PL>(ga, lo, up);
        }
        float delta[2] = {0.f, 0.f};
        float dq[PL][4][4];
#pragma unroll
        for (int p = 0; p < PL; ++p)
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) dq[p][n][e] = 0.f;

#pragma unroll 1
        for (int it = 0; it < (SINGLE ? 1 : 2 * passes); ++it) {
            const int sweep = it >= passes ? 1 : 0, pass = it - sweep * passes;
            const int k0 = pass * gm.tab;
            const int nk = SINGLE ? 16 * KS : min(gm.tab, (total - k0 + 31) / 32 * 32);
            if (passes > 1 || !filled) {
                if (filled) group_sync();
                const bool bad = fill_keys(tab, irow, i, k0, nk, total, glane, glanes, status, dm, gm);
                any_bad = (one_warp ? __any_sync(0xffffffffu, bad) : __syncthreads_or(bad)) || any_bad;
                if (one_warp) __syncwarp();
                filled = true;
            }
            if (!has) continue;
#pragma unroll 1
            for (int kb = 0; kb < nk; kb += 16 * KS) {
                uint4 kr[KS][2][PL];
                float c[2 * KS][4], dp[2 * KS][4];
#pragma unroll
                for (int s = 0; s < KS; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t kt = tab[kb + 16 * s + 8 * e + g];
                        uint4 vr[PL];
                        ld_token<PL, ZEROS>(kr[s][e], Kb, kt);
                        ld_token<PL, ZEROS>(vr, Vb, kt);
                        mma_rows<PL>(c[2 * s + e], qa, kr[s][e]);
                        mma_rows<PL>(dp[2 * s + e], ga, vr);
                    }
                const bool mask = any_bad || k0 + kb + 16 * KS > total;
#pragma unroll
                for (int j = 0; j < 2 * KS; ++j) {
                    c[j][0] = ex2_approx(fmaf(c[j][0], sl2, -lse2[0]));
                    c[j][1] = ex2_approx(fmaf(c[j][1], sl2, -lse2[0]));
                    c[j][2] = ex2_approx(fmaf(c[j][2], sl2, -lse2[1]));
                    c[j][3] = ex2_approx(fmaf(c[j][3], sl2, -lse2[1]));
                }
                if (mask) {
#pragma unroll
                    for (int j = 0; j < 2 * KS; ++j) {
                        const int kk = k0 + kb + 8 * j + 2 * t4;
                        if (dead_key(kk, total, any_bad, irow, dm, gm)) { c[j][0] = 0.f; c[j][2] = 0.f; }
                        if (dead_key(kk + 1, total, any_bad, irow, dm, gm)) { c[j][1] = 0.f; c[j][3] = 0.f; }
                    }
                }
                if (SINGLE || sweep == 0) {
#pragma unroll
                    for (int j = 0; j < 2 * KS; ++j) {
                        delta[0] = fmaf(c[j][0], dp[j][0], fmaf(c[j][1], dp[j][1], delta[0]));
                        delta[1] = fmaf(c[j][2], dp[j][2], fmaf(c[j][3], dp[j][3], delta[1]));
                    }
                    if (SINGLE || (pass == passes - 1 && kb + 16 * KS >= nk)) {
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            delta[r] += __shfl_xor_sync(0xffffffffu, delta[r], 1);
                            delta[r] += __shfl_xor_sync(0xffffffffu, delta[r], 2);
                        }
                    }
                }
                if (SINGLE || sweep == 1) {
#pragma unroll
                    for (int j = 0; j < 2 * KS; ++j) {
                        c[j][0] *= dp[j][0] - delta[0]; c[j][1] *= dp[j][1] - delta[0];
                        c[j][2] *= dp[j][2] - delta[1]; c[j][3] *= dp[j][3] - delta[1];
                    }
#pragma unroll
                    for (int s = 0; s < KS; ++s) mma_tokens<PL, EXACT>(dq, c[2 * s], c[2 * s + 1], kr[s][0], kr[s][1]);
                }
            }
        }
        // ---- dQ = scale * acc, delta kept for the dK/dV kernel ----
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (tok[r] < 0) continue;
            uint8_t* o = dQb + (size_t)(uint32_t)tok[r] * tok_bytes;
#pragma unroll
            for (int p = 0; p < PL; ++p) *reinterpret_cast<uint4*>(o + p * 64) = pack_row(dq[p], r, dm.scale);
            if (t4 == 0) delta_out[stat0 + tok[r]] = delta[r];
        }
    }
    pdl_launch_dependents();
}

// ------------------------------------------------------------------ dK, dV
template <int PL, bool EXACT, bool ZEROS, int TY, int TX>
__global__ void __launch_bounds__(PL == 2 ? 128 : 256, PL == 2 ? 3 : 2)
bwd_dkv_direct_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg,
                      const __nv_bfloat16* __restrict__ Vg, const int32_t* inv_off,
                      const int32_t* inv_list, const float* __restrict__ lse,
                      const float* delta, const __nv_bfloat16* __restrict__ dOg,
                      const float* __restrict__ lce_w, __nv_bfloat16* __restrict__ dKg,
                      __nv_bfloat16* __restrict__ dVg, Dims dm, DirGeom gm) {
    constexpr int KS = PL == 2 ? 1 : 2;                               // 16-query steps per block
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const bool one_warp = gm.gpc > 1;
    const int rest = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int grp = one_warp ? warp : 0;
    const int ck = one_warp ? 0 : rest % gm.chunks;
    const int jr = one_warp ? rest * gm.gpc + warp : rest / gm.chunks;   // key region
    const int gwarp = one_warp ? 0 : warp, gwarps = one_warp ? 1 : gm.nw;
    const int glane = one_warp ? lane : tid, glanes = gwarps * 32;
    const bool live = jr < dm.R;
    auto group_sync = [&]() { if (one_warp) __syncwarp(); else __syncthreads(); };

    const int rj = live ? jr : 0;
    const int ry = fdiv(rj, dm.S, gm.mul_s), rx = rj - ry * dm.S;
    const int y0 = ry * dm.hs + ck * gm.hb, x0 = rx * dm.ws;
    const int rows = min(gm.hb, dm.hs - ck * gm.hb);
    const int ntok = rows * dm.ws, c0 = ck * gm.hb * dm.ws;
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
    const int N0 = dm.H0 * dm.W0;
    const size_t head_off = (size_t)b * N0 * tok_bytes + (size_t)h * 64 * PL;
    const uint8_t* Qb = reinterpret_cast<const uint8_t*>(Qg) + head_off + t4 * 16;
    const uint8_t* Kb = reinterpret_cast<const uint8_t*>(Kg) + head_off + t4 * 16;
    const uint8_t* Vb = reinterpret_cast<const uint8_t*>(Vg) + head_off + t4 * 16;
    const uint8_t* Gh = reinterpret_cast<const uint8_t*>(dOg) + head_off;
    const uint8_t* Gb = Gh + t4 * 16;
    uint8_t* dKb = reinterpret_cast<uint8_t*>(dKg) + head_off + t4 * 16;

    float* s_w = reinterpret_cast<float*>(smem + gm.off_w);
    if (dm.lce) {
        load_lce_weights(s_w, lce_w, h, 32 * PL * 25, tid, gm.nw * 32);
        if (live) load_halo<PL>(sbase + gm.off_halo + grp * gm.halo_bytes, Gh, y0, x0, rows, dm, gm, glane, glanes);
    }
    cp_async_commit();
    __syncthreads();                                                  // weights
    pdl_wait();          // delta and the inverse index come from the dQ kernel
    if (!live) return;

    const int hi = dm.heads_i == 1 ? 0 : h;
    const size_t bhi = (size_t)b * dm.heads_i + hi;
    const int e0 = __ldcg(inv_off + bhi * (dm.R + 1) + jr), e1 = __ldcg(inv_off + bhi * (dm.R + 1) + jr + 1);
    const int32_t* list = inv_list + bhi * dm.R * dm.topk + e0;      // query regions that list jr, fixed order
    const int total = (e1 - e0) * dm.n_r;
    const float* lse_h = lse + ((size_t)b * dm.heads + h) * N0;
    const float* delta_h = delta + ((size_t)b * dm.heads + h) * N0;
    uint32_t* tab = reinterpret_cast<uint32_t*>(smem + gm.off_tab) + grp * 3 * gm.tab;   // row offsets, lse * log2(e), delta
    float* s_l2 = reinterpret_cast<float*>(tab + gm.tab);
    float* s_dl = s_l2 + gm.tab;
    float* st = reinterpret_cast<float*>(smem + gm.off_st + grp * gm.st_bytes);
    const float sl2 = dm.scale * 1.4426950408889634f;
    const int passes = (total + gm.tab - 1) / gm.tab;
    // A query beyond the list repeats the last one with lse = inf: its P is zero.  One in the zero padding has zero rows
    // of Q and dO and lse = delta = 0: it adds nothing.
    auto fill_queries = [&](int k0, int n) {
        for (int e = glane; e < n; e += glanes) {
            const int kk = min(k0 + e, total - 1);
            const int m = fdiv(kk, dm.n_r, gm.mul_nr);
            const int tk = token_of(dm, gm, __ldcg(list + m), kk - m * dm.n_r);
            tab[e] = tk >= 0 ? (uint32_t)tk * (uint32_t)(dm.C >> 3) : dk::ZERO;
            s_l2[e] = k0 + e >= total ? INFINITY : tk >= 0 ? __ldg(lse_h + tk) * 1.4426950408889634f : 0.f;
            s_dl[e] = tk >= 0 ? __ldcg(delta_h + tk) : 0.f;
        }
    };
    bool filled = false;

    for (int tile = gwarp; tile - gwarp < gm.tpc; tile += gwarps) {
        const bool has = tile * 16 < ntok;
        int tok[2];
        uint32_t ka[PL][2][4], va[PL][2][4];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int tk = tile * 16 + g + 8 * r;
            tok[r] = tk < ntok ? token_of(dm, gm, jr, c0 + tk) : -1;
        }
        {
            uint4 lo[PL], up[PL];
            ld_row<PL>(lo, Kb, tok[0], tok_bytes); ld_row<PL>(up, Kb, tok[1], tok_bytes);
            rows_to_a<PL>(ka, lo, up);
            ld_row<PL>(lo, Vb, tok[0], tok_bytes); ld_row<PL>(up, Vb, tok[1], tok_bytes);
            rows_to_a<PL>(va, lo, up);
        }
        float dkx[PL][4][4], dvx[PL][4][4];
#pragma unroll
        for (int p = 0; p < PL; ++p)
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) { dkx[p][n][e] = 0.f; dvx[p][n][e] = 0.f; }

#pragma unroll 1
        for (int pass = 0; pass < passes; ++pass) {
            const int k0 = pass * gm.tab;
            const int nk = min(gm.tab, (total - k0 + 31) / 32 * 32);
            if (passes > 1 || !filled) {
                if (filled) group_sync();
                fill_queries(k0, nk);
                group_sync();
                filled = true;
            }
            if (!has) continue;
#pragma unroll 1
            for (int kb = 0; kb < nk; kb += 16 * KS) {
                uint4 qr[KS][2][PL], gr[KS][2][PL];
                float c[2 * KS][4], dp[2 * KS][4];
#pragma unroll
                for (int s = 0; s < KS; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t qt = tab[kb + 16 * s + 8 * e + g];
                        ld_token<PL, ZEROS>(qr[s][e], Qb, qt);
                        ld_token<PL, ZEROS>(gr[s][e], Gb, qt);
                    }
#pragma unroll
                for (int s = 0; s < KS; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        mma_rows<PL>(c[2 * s + e], ka, qr[s][e]);     // S^T = K Q^T
                        mma_rows<PL>(dp[2 * s + e], va, gr[s][e]);    // dP^T = V dO^T
                    }
#pragma unroll
                for (int j = 0; j < 2 * KS; ++j) {
                    const float2 l2 = *reinterpret_cast<const float2*>(s_l2 + kb + 8 * j + 2 * t4);
                    const float2 dl = *reinterpret_cast<const float2*>(s_dl + kb + 8 * j + 2 * t4);
                    c[j][0] = ex2_approx(fmaf(c[j][0], sl2, -l2.x));
                    c[j][1] = ex2_approx(fmaf(c[j][1], sl2, -l2.y));
                    c[j][2] = ex2_approx(fmaf(c[j][2], sl2, -l2.x));
                    c[j][3] = ex2_approx(fmaf(c[j][3], sl2, -l2.y));
                    dp[j][0] = c[j][0] * (dp[j][0] - dl.x);
                    dp[j][1] = c[j][1] * (dp[j][1] - dl.y);
                    dp[j][2] = c[j][2] * (dp[j][2] - dl.x);
                    dp[j][3] = c[j][3] * (dp[j][3] - dl.y);
                }
#pragma unroll
                for (int s = 0; s < KS; ++s) {
                    mma_tokens<PL, EXACT>(dkx, dp[2 * s], dp[2 * s + 1], qr[s][0], qr[s][1]);   // dK += dS^T Q
                    mma_tokens<PL, EXACT>(dvx, c[2 * s], c[2 * s + 1], gr[s][0], gr[s][1]);     // dV += P^T dO
                }
            }
        }
        // ---- dK = scale * acc; dV to the staging tile ----
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int tk = tile * 16 + g + 8 * r;
            if (tk >= ntok) continue;
            if (tok[r] >= 0) {
                uint8_t* o = dKb + (size_t)(uint32_t)tok[r] * tok_bytes;
#pragma unroll
                for (int p = 0; p < PL; ++p) *reinterpret_cast<uint4*>(o + p * 64) = pack_row(dkx[p], r, dm.scale);
            }
            float* dst = st + tk * 32 * PL + t4 * 8;
#pragma unroll
            for (int p = 0; p < PL; ++p)
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    *reinterpret_cast<float4*>(dst + p * 32 + 4 * q) =
                        make_float4(dvx[p][2 * q][2 * r], dvx[p][2 * q][2 * r + 1], dvx[p][2 * q + 1][2 * r], dvx[p][2 * q + 1][2 * r + 1]);
        }
    }
    cp_async_wait<0>();
    group_sync();
    // ---- LCE adjoint + store of dV: dV[y,x] += sum_ij w[i,j] dO[y-i+2, x-j+2] = correlation with the flipped filter ----
    lce_chunk<PL, TY, TX, true>(st, sbase + gm.off_halo + grp * gm.halo_bytes, s_w, nullptr, dm.lce, dVg + head_off / 2, y0, x0, rows, dm, gm,
                            gwarp, gwarps, lane);
}

// ------------------------------------------------------------------ host side
static DirGeom dq_geom(const Dims& d) {
    DirGeom g = direct_geom(d, false, 4);
    if (d.topk * d.n_r <= 64) g.tab = 64;                            // one block of 64 keys
    g.smem_bytes = g.off_tab + g.gpc * g.tab * 4;                    // the table only
    const int inv = (int)inverse_smem(d);
    if (g.smem_bytes < inv) g.smem_bytes = inv;
    return g;
}
static DirGeom dkv_geom(const Dims& d) {
    Dims full = d;
    full.topk = d.R;                                                 // a key region may be on every query region's list
    return direct_geom(full, d.lce, 12);
}

bool backward_direct_supported(const Dims& d, int dtype) {
    if (!attend_direct_supported(d, dtype)) return false;
    if ((long long)d.R * d.n_r * d.n_r >= (1ll << 32)) return false;
    return dkv_geom(d).smem_bytes <= 200 * 1024 && dq_geom(d).smem_bytes <= 200 * 1024 && d.R <= 8192;
}

template <typename F>
static cudaError_t allow_smem(PerDeviceMax& set, F kernel, int bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return set.ensure(bytes, [&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}

namespace {
struct BwdArgs {
    const __nv_bfloat16 *q, *k, *v, *go;
    const int32_t* index;
    int32_t *inv_off, *inv_list;
    const float *lce_w, *lse;
    __nv_bfloat16 *dq, *dk, *dv;
    float* delta;
    int32_t* status;
    cudaStream_t st;
};
}  // namespace

template <int PL, bool EXACT, bool SINGLE, bool ZEROS>
static cudaError_t launch_dq(const Dims& d, const BwdArgs& a) {
    const DirGeom g = dq_geom(d);
    auto kernel = bwd_dq_direct_kernel<PL, EXACT, SINGLE, ZEROS>;
    static PerDeviceMax set;
    const cudaError_t e = allow_smem(set, kernel, g.smem_bytes);
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_kernel(kernel, dim3(g.gpi > d.heads_i ? g.gpi : d.heads_i, d.heads + 1, d.B), dim3(g.nw * 32), (size_t)g.smem_bytes, a.st, false,
                         a.q, a.k, a.v, a.index, a.lse, a.go, a.dq, a.delta, a.inv_off, a.inv_list, inverse_uses_bits(d), a.status, d, g);
}

template <int PL, bool EXACT, bool ZEROS, int TY, int TX>
static cudaError_t launch_dkv(const Dims& d, const BwdArgs& a) {
    const DirGeom g = dkv_geom(d);
    auto kernel = bwd_dkv_direct_kernel<PL, EXACT, ZEROS, TY, TX>;
    static PerDeviceMax set;
    const cudaError_t e = allow_smem(set, kernel, g.smem_bytes);
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_kernel(kernel, dim3(g.gpi, d.heads, d.B), dim3(g.nw * 32), (size_t)g.smem_bytes, a.st, true,
                         a.q, a.k, a.v, a.inv_off, a.inv_list, a.lse, a.delta, a.go, a.lce_w, a.dk, a.dv, d, g);
}

template <bool ZEROS>
static cudaError_t launch_both(const Dims& d, const BwdArgs& a) {
    const bool single = d.topk * d.n_r <= 64, exact = direct_exact(d);
    const cudaError_t e = d.d == 64 ? launch_dq<2, true, false, ZEROS>(d, a)
                        : exact     ? launch_dq<1, true, false, ZEROS>(d, a)
                        : single    ? launch_dq<1, false, true, ZEROS>(d, a)
                                    : launch_dq<1, false, false, ZEROS>(d, a);
    if (e != cudaSuccess) return e;
    if (d.hs <= 2) return d.d == 64 ? launch_dkv<2, true, ZEROS, 2, 2>(d, a) : launch_dkv<1, false, ZEROS, 2, 2>(d, a);
    if (d.d == 64) return launch_dkv<2, true, ZEROS, 4, 4>(d, a);
    if (exact) return launch_dkv<1, true, ZEROS, 4, 3>(d, a);
    switch (lce_tile_width(dkv_geom(d), d)) {
        case 2: return launch_dkv<1, false, ZEROS, 4, 2>(d, a);
        case 3: return launch_dkv<1, false, ZEROS, 4, 3>(d, a);
        default: return launch_dkv<1, false, ZEROS, 4, 4>(d, a);
    }
}

cudaError_t launch_backward_direct(const Dims& d, const void* Q, const void* K, const void* V,
                                   const int32_t* index, int32_t* inv_off, int32_t* inv_list,
                                   const float* lce_w, const float* lse, const void* dO,
                                   void* dQ, void* dK, void* dV, float* delta, int32_t* status, cudaStream_t st) {
    typedef __nv_bfloat16 bf;
    const BwdArgs a = {static_cast<const bf*>(Q), static_cast<const bf*>(K), static_cast<const bf*>(V), static_cast<const bf*>(dO), index,
                       inv_off, inv_list, lce_w, lse, static_cast<bf*>(dQ), static_cast<bf*>(dK), static_cast<bf*>(dV), delta, status, st};
    return d.H != d.H0 || d.W != d.W0 ? launch_both<true>(d, a) : launch_both<false>(d, a);
}

}  // namespace bra
