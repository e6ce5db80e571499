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
// movmatrix where it runs over tokens.  Every sum has a fixed order, results are bit-identical from run to run: where a list of
// the inverse index is cut in parts (direct_grad_parts), each leaves its sums in scratch memory and the one that is done last, which
// an atomic counter tells, adds them up in the order of the parts.  (Two tiles per warp, which pay in the forward kernel, do not here: 8 warps per SM at 168 registers,
// dQ 140 -> 170 us and dK / dV 274 -> 331 us at 2 x 100 x 167, S = 16.  Fetching the next 16 rows ahead into registers:
// 140 -> 155 and 274 -> 286 us.)
// Bound: the latency of the listed rows at 12 - 16 warps per SM (0.53 instructions per cycle and scheduler at head dim 32; at head
// dim 64, 168 registers, 0.41 in dQ and 0.34 in dK / dV, 1.9 and 3.6 cycles per issue waiting for loads).
// Measured (B200), dQ / dK dV: 2 x 100 x 167, 6 heads: 193 / 322 -> 136 / 201 us, now, lists cut and clustered, 148 / 149 under ncu;
// 16 x 32 x 32, 12 heads of 64: 1998 / 2412 us (CUDA cores) -> 140 / 220 us.
#include "direct_common.cuh"
#include "inverse_index.cuh"

namespace bra {

using namespace ptx;

// ------------------------------------------------------------------ dQ and delta
// The CTAs of grid row 0 build the inverse routing index for the dK / dV kernel instead.
// SINGLE: all keys of a group (at most 64) in one block, S and dP computed once; otherwise one sweep for delta and
// one for dQ.
template <int PL, bool EXACT, bool SINGLE>
__global__ void __launch_bounds__(PL == 2 ? 128 : 256, PL == 2 ? 3 : 2)
bwd_dq_direct_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg,
                     const __nv_bfloat16* __restrict__ Vg, const int32_t* __restrict__ index,
                     const float* __restrict__ lse, const __nv_bfloat16* __restrict__ dOg,
                     __nv_bfloat16* __restrict__ dQg, float* __restrict__ delta_out,
                     int32_t* __restrict__ inv_off, int32_t* __restrict__ inv_list, int32_t* __restrict__ inv_order, bool inv_bits,
                     ListJobs lj, int32_t* __restrict__ status, Dims dm, DirGeom gm) {
    constexpr int RT = 1, KS = SINGLE ? 4 : 2;                        // tiles per warp, 16-key steps per block
    extern __shared__ __align__(128) uint8_t smem[];
    // blockIdx.y = 0: the inverse index (one CTA per (image, routing head)); else head blockIdx.y - 1
    if (blockIdx.y == 0) {
        if (inv_off && (int)blockIdx.x < dm.heads_i)
            inverse_index_job(index, inv_off, inv_list, inv_order, blockIdx.z * dm.heads_i + blockIdx.x, reinterpret_cast<int32_t*>(smem), inv_bits, dm, lj);
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
    const uint4 probe = spare_probe<PL>(Kb - t4 * 16, Vb - t4 * 16, lane);
    const size_t stat0 = ((size_t)b * dm.heads + h) * N0;
    const int hi = dm.heads_i == 1 ? 0 : h;
    const int32_t* irow = index + (((size_t)b * dm.heads_i + hi) * dm.R + i) * dm.topk;
    const int total = dm.topk * dm.n_r;
    uint32_t* tab = reinterpret_cast<uint32_t*>(smem + gm.off_tab + grp * gm.tab_bytes);
    uint32_t* dead = tab + gm.tab;
    const float sl2 = dm.scale * 1.4426950408889634f;
    const int passes = (total + gm.tab - 1) / gm.tab;
    const int spare = spare_token<PL>(probe, Kb - t4 * 16, Vb - t4 * 16, tok_bytes, N0, lane);
    bool filled = false;

    for (int tile = gwarp * RT; tile - gwarp * RT < gm.tpc; tile += gwarps * RT) {
        const bool has = tile * 16 < ntok;
        int tok[RT][2];
        float lse2[RT][2], delta[RT][2];
        uint32_t qa[RT][PL][2][4], ga[RT][PL][2][4];
        float dq[RT][PL][4][4];
#pragma unroll
        for (int x = 0; x < RT; ++x) {
            uint4 q[2][PL], go[2][PL];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int tk = (tile + x) * 16 + g + 8 * r;
                tok[x][r] = tk < ntok ? token_of(dm, gm, i, c0 + tk) : -1;
                lse2[x][r] = tok[x][r] >= 0 ? __ldg(lse + stat0 + tok[x][r]) * 1.4426950408889634f : 0.f;
                delta[x][r] = 0.f;
                ld_row<PL>(q[r], Qb, tok[x][r], tok_bytes);
                ld_row<PL>(go[r], Gb, tok[x][r], tok_bytes);
            }
            rows_to_a<PL>(qa[x], q[0], q[1]);
            rows_to_a<PL>(ga[x], go[0], go[1]);
#pragma unroll
            for (int p = 0; p < PL; ++p)
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) dq[x][p][n][e] = 0.f;
        }

#pragma unroll 1
        for (int it = 0; it < (SINGLE ? 1 : 2 * passes); ++it) {
            const int sweep = it >= passes ? 1 : 0, pass = it - sweep * passes;
            const int k0 = pass * gm.tab;
            const int nk = SINGLE ? 16 * KS : min(gm.tab, (total - k0 + 31) / 32 * 32);
            if (passes > 1 || !filled) {
                if (filled) group_sync();
                fill_keys(tab, dead, irow, k0, nk, total, spare, glane, glanes, status, dm, gm);
                group_sync();
                filled = true;
            }
            if (!has) continue;
#pragma unroll 1
            for (int kb = 0; kb < nk; kb += 16 * KS) {
                uint4 kr[KS][2][PL];
                float c[RT][2 * KS][4], dp[RT][2 * KS][4];
#pragma unroll
                for (int s = 0; s < KS; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t kt = tab[kb + 16 * s + 8 * e + g];
                        uint4 vr[PL];
                        ld_token<PL>(kr[s][e], Kb, kt);
                        ld_token<PL>(vr, Vb, kt);
#pragma unroll
                        for (int x = 0; x < RT; ++x) {
                            mma_rows<PL>(c[x][2 * s + e], qa[x], kr[s][e]);
                            mma_rows<PL>(dp[x][2 * s + e], ga[x], vr);
                        }
                    }
#pragma unroll
                for (int x = 0; x < RT; ++x)
#pragma unroll
                    for (int j = 0; j < 2 * KS; ++j) {
                        c[x][j][0] = ex2_approx(fmaf(c[x][j][0], sl2, -lse2[x][0]));
                        c[x][j][1] = ex2_approx(fmaf(c[x][j][1], sl2, -lse2[x][0]));
                        c[x][j][2] = ex2_approx(fmaf(c[x][j][2], sl2, -lse2[x][1]));
                        c[x][j][3] = ex2_approx(fmaf(c[x][j][3], sl2, -lse2[x][1]));
                    }
                // (keys of the zero padding add nothing to delta or dQ)
                if (SINGLE) {
                    const uint32_t b0 = dead[0], b1 = dead[1];
                    if (b0 | b1) {
                        const uint32_t w[2] = {b0 >> (2 * t4), b1 >> (2 * t4)};
#pragma unroll
                        for (int j = 0; j < 2 * KS; ++j)
#pragma unroll
                            for (int x = 0; x < RT; ++x) {
                                if (w[j >> 2] >> (8 * (j & 3)) & 1) c[x][j][0] = c[x][j][2] = 0.f;
                                if (w[j >> 2] >> (8 * (j & 3) + 1) & 1) c[x][j][1] = c[x][j][3] = 0.f;
                            }
                    }
                } else {
                    const uint32_t bits = dead[kb >> 5] >> (kb & 31);
                    if (bits) mask_columns<RT, 2 * KS>(c, bits, t4, 0.f);
                }
                if (SINGLE || sweep == 0) {
#pragma unroll
                    for (int x = 0; x < RT; ++x) {
#pragma unroll
                        for (int j = 0; j < 2 * KS; ++j) {
                            delta[x][0] = fmaf(c[x][j][0], dp[x][j][0], fmaf(c[x][j][1], dp[x][j][1], delta[x][0]));
                            delta[x][1] = fmaf(c[x][j][2], dp[x][j][2], fmaf(c[x][j][3], dp[x][j][3], delta[x][1]));
                        }
                        if (SINGLE || (pass == passes - 1 && kb + 16 * KS >= nk)) {
#pragma unroll
                            for (int r = 0; r < 2; ++r) {
                                delta[x][r] += __shfl_xor_sync(0xffffffffu, delta[x][r], 1);
                                delta[x][r] += __shfl_xor_sync(0xffffffffu, delta[x][r], 2);
                            }
                        }
                    }
                }
                if (SINGLE || sweep == 1) {
#pragma unroll
                    for (int x = 0; x < RT; ++x)
#pragma unroll
                        for (int j = 0; j < 2 * KS; ++j) {
                            c[x][j][0] *= dp[x][j][0] - delta[x][0]; c[x][j][1] *= dp[x][j][1] - delta[x][0];
                            c[x][j][2] *= dp[x][j][2] - delta[x][1]; c[x][j][3] *= dp[x][j][3] - delta[x][1];
                        }
#pragma unroll
                    for (int s = 0; s < KS; ++s) mma_tokens<PL, EXACT>(dq, c, 2 * s, kr[s][0], kr[s][1]);
                }
            }
        }
        // ---- dQ = scale * acc, delta kept for the dK/dV kernel ----
#pragma unroll
        for (int x = 0; x < RT; ++x)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (tok[x][r] < 0) continue;
                uint8_t* o = dQb + (size_t)(uint32_t)tok[x][r] * tok_bytes;
#pragma unroll
                for (int p = 0; p < PL; ++p) *reinterpret_cast<uint4*>(o + p * 64) = pack_row(dq[x][p], r, dm.scale);
                if (t4 == 0) delta_out[stat0 + tok[x][r]] = delta[x][r];
            }
        if (SINGLE) break;                                            // (at most 64 tokens: as many warps as tiles)
    }
    pdl_launch_dependents();
}

// ------------------------------------------------------------------ dK, dV
// dK = scale * acc of a tile's rows (tokens tok of the map), dV to the staging tile
template <int PL>
__device__ __forceinline__ void finish_rows(uint8_t* dKb, float* st, const float (&dk)[PL][4][4], const float (&dv)[PL][4][4], const int (&tok)[2], int tile,
                                            int ntok, int g, int t4, const Dims& dm) {
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int tk = tile * 16 + g + 8 * r;
        if (tk >= ntok) continue;
        if (tok[r] >= 0) {
            uint8_t* o = dKb + (size_t)(uint32_t)tok[r] * tok_bytes;
#pragma unroll
            for (int p = 0; p < PL; ++p) *reinterpret_cast<uint4*>(o + p * 64) = pack_row(dk[p], r, dm.scale);
        }
        float* dst = st + tk * 32 * PL + t4 * 8;
#pragma unroll
        for (int p = 0; p < PL; ++p)
#pragma unroll
            for (int q = 0; q < 2; ++q)
                *reinterpret_cast<float4*>(dst + p * 32 + 4 * q) = make_float4(dv[p][2 * q][2 * r], dv[p][2 * q][2 * r + 1],
                                                                               dv[p][2 * q + 1][2 * r], dv[p][2 * q + 1][2 * r + 1]);
    }
}
// The same for the sums of the parts of a cut list, added in the order of the parts
template <int PL>
__device__ __forceinline__ void sum_parts(const float* at, int nparts, size_t stride, uint8_t* dKb, float* st, int jr, int c0, int tile, int ntok, int lane,
                                          const Dims& dm, const DirGeom& gm) {
    const int g = lane >> 2, t4 = lane & 3;
    int tok[2];
    float dk[PL][4][4], dv[PL][4][4];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int tk = tile * 16 + g + 8 * r;
        tok[r] = tk < ntok ? token_of(dm, gm, jr, c0 + tk) : -1;
    }
#pragma unroll
    for (int p = 0; p < PL; ++p)
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) dk[p][n][e] = dv[p][n][e] = 0.f;
#pragma unroll 1
    for (int q = 0; q < nparts; ++q, at += stride) {
#pragma unroll
        for (int p = 0; p < PL; ++p)
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    dk[p][n][e] += __ldcg(at + ((p * 4 + n) * 4 + e) * 32);
                    dv[p][n][e] += __ldcg(at + ((PL * 4 + p * 4 + n) * 4 + e) * 32);
                }
    }
    finish_rows<PL>(dKb, st, dk, dv, tok, tile, ntok, g, t4, dm);
}
// CUT: long lists in parts (ListParts).
template <int PL, bool EXACT, bool CUT, int TY, int TX>
__device__ __forceinline__ void bwd_dkv_direct(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg,
                                               const __nv_bfloat16* __restrict__ Vg, const int32_t* inv_off,
                                               const int32_t* inv_list, const int32_t* inv_order, const float* __restrict__ lse,
                                               const float* delta, const __nv_bfloat16* __restrict__ dOg,
                                               const float* __restrict__ lce_w, __nv_bfloat16* __restrict__ dKg,
                                               __nv_bfloat16* __restrict__ dVg, const int2* jobs, const ListParts& parts, int32_t* done, float* sums,
                                               int job0, const Dims& dm, const DirGeom& gm) {
    constexpr int RT = 1, KS = PL == 2 ? 1 : 2;                       // tiles per warp, 16-query steps per block
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const bool one_warp = gm.gpc > 1;
    const int rest = blockIdx.z, h = blockIdx.x, b = blockIdx.y;      // longest lists of all (image, head) pairs first
    const int grp = one_warp ? warp : 0;
    const int ck = one_warp ? 0 : rest % gm.chunks;
    const int nth = one_warp ? rest * gm.gpc + warp : rest / gm.chunks;  // by falling length of the list
    const int gwarp = one_warp ? 0 : warp, gwarps = one_warp ? 1 : gm.nw;
    const int glane = one_warp ? lane : tid, glanes = gwarps * 32;
    const bool live = nth < (CUT ? parts.jobs : dm.R) - job0;
    auto group_sync = [&]() { if (one_warp) __syncwarp(); else __syncthreads(); };

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

    const uint4 probe = spare_probe<PL>(Qb - t4 * 16, Gh, lane);
    const int hi = dm.heads_i == 1 ? 0 : h;
    const size_t bhi = (size_t)b * dm.heads_i + hi;
    int2 job = make_int2(-1, 0);                                      // key region, part of its list
    // there are as many jobs as regions, or more
    if (CUT && !one_warp && job0 + nth >= dm.R) {
        pdl_wait();
        if (__ldcg(&jobs[bhi * parts.jobs + job0 + nth].x) < 0) return;
    }
    float* s_w = reinterpret_cast<float*>(smem + gm.off_w);
    if (dm.lce) load_lce_weights(s_w, lce_w, h, 32 * PL * 25, tid, gm.nw * 32);
    __syncthreads();                                                  // weights
    pdl_wait();          // delta, the inverse index and the order of the regions come from the dQ kernel
    if (CUT && live) job = __ldcg(jobs + bhi * parts.jobs + job0 + nth);
    if (CUT ? job.x < 0 : !live) return;
    if (!CUT) job.x = __ldcg(inv_order + bhi * dm.R + job0 + nth);
    const int spare = spare_token<PL>(probe, Qb - t4 * 16, Gh, tok_bytes, N0, lane);

    const int jr = job.x;
    const int ry = fdiv(jr, dm.S, gm.mul_s), rx = jr - ry * dm.S;
    const int y0 = ry * dm.hs + ck * gm.hb, x0 = rx * dm.ws;
    if (dm.lce) load_halo<PL>(sbase + gm.off_halo + grp * gm.halo_bytes, Gh, y0, x0, rows, dm, gm, glane, glanes);
    cp_async_commit();
    const int l0 = __ldcg(inv_off + bhi * (dm.R + 1) + jr), l1 = __ldcg(inv_off + bhi * (dm.R + 1) + jr + 1);
    const int nparts = CUT ? max(1, (l1 - l0 + parts.most - 1) / parts.most) : 1;
    const int per = !CUT ? 0 : parts.even ? (l1 - l0 + nparts - 1) / nparts : parts.most;
    const int e0 = CUT ? l0 + job.y * per : l0, e1 = CUT ? min(l1, e0 + per) : l1;
    // (parts, job, part): not needed before the end, so they wait behind the table; every thread writes them, for itself
    volatile int* s_job = reinterpret_cast<int*>(smem + gm.off_tab + grp * gm.tab_bytes) + 3 * gm.tab;
    if (CUT) { s_job[0] = nparts; s_job[1] = job0 + nth; s_job[2] = job.y; }
    const int32_t* list = inv_list + bhi * dm.R * dm.topk + e0;      // query regions that list jr, fixed order
    const long long total = (long long)(e1 - e0) * dm.n_r;           // a list with repeats may hold every entry of the index
    const float* lse_h = lse + ((size_t)b * dm.heads + h) * N0;
    const float* delta_h = delta + ((size_t)b * dm.heads + h) * N0;
    uint32_t* tab = reinterpret_cast<uint32_t*>(smem + gm.off_tab + grp * gm.tab_bytes);   // row offsets, lse * log2(e), delta
    float* s_l2 = reinterpret_cast<float*>(tab + gm.tab);
    float* s_dl = s_l2 + gm.tab;
    float* st = reinterpret_cast<float*>(smem + gm.off_st + grp * gm.st_bytes);
    const float sl2 = dm.scale * 1.4426950408889634f;
    const int passes = (int)((total + gm.tab - 1) / gm.tab);
    // A query beyond the list, or of the zero padding (zero rows of Q and dO: it adds nothing), names the row of token `spare`
    // with lse = inf: its P is zero.
    // (m0, t0): list entry and token of the table's first query; left: how many queries remain from there on.
    auto fill_queries = [&](int m0, int t0, int n, int left) {
        for (int e = glane; e < n; e += glanes) {
            const int u = t0 + min(e, left - 1), m = fdiv(u, gm.by_nr);
            const int tk = token_of(dm, gm, __ldcg(list + m0 + m), u - m * dm.n_r);
            const bool ok = e < left && tk >= 0;
            const int at = ok ? tk : spare;
            tab[e] = (uint32_t)at * (uint32_t)(dm.C >> 3);
            s_l2[e] = ok ? __ldg(lse_h + at) * 1.4426950408889634f : INFINITY;
            s_dl[e] = ok ? __ldcg(delta_h + at) : 0.f;
        }
    };
    bool filled = false;
    // where the sums of a tile of a job lie: 32 lanes times dK, dV as the lane holds them
    auto sum_at = [&](int j, int tile) { return (((((size_t)b * dm.heads + h) * parts.cut + j) * gm.chunks + ck) * gm.tpc + tile) * 1024 * PL + lane; };

    for (int tile = gwarp * RT; tile - gwarp * RT < gm.tpc; tile += gwarps * RT) {
        const bool has = tile * 16 < ntok;
        int tok[RT][2];
        uint32_t ka[RT][PL][2][4], va[RT][PL][2][4];
        float dkx[RT][PL][4][4], dvx[RT][PL][4][4];
#pragma unroll
        for (int x = 0; x < RT; ++x) {
            uint4 k[2][PL], v[2][PL];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int tk = (tile + x) * 16 + g + 8 * r;
                tok[x][r] = tk < ntok ? token_of(dm, gm, jr, c0 + tk) : -1;
                ld_row<PL>(k[r], Kb, tok[x][r], tok_bytes);
                ld_row<PL>(v[r], Vb, tok[x][r], tok_bytes);
            }
            rows_to_a<PL>(ka[x], k[0], k[1]);
            rows_to_a<PL>(va[x], v[0], v[1]);
#pragma unroll
            for (int p = 0; p < PL; ++p)
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) { dkx[x][p][n][e] = 0.f; dvx[x][p][n][e] = 0.f; }
        }

        int m0 = 0, t0 = 0;
#pragma unroll 1
        for (int pass = 0; pass < passes; ++pass) {
            const int left = (int)min((long long)gm.tab, total - (long long)pass * gm.tab);
            const int nk = (left + 31) / 32 * 32;                     // (the table's size is a multiple of 32)
            if (passes > 1 || !filled) {
                if (filled) group_sync();
                fill_queries(m0, t0, nk, left);
                const int u = t0 + gm.tab, m = fdiv(u, gm.by_nr);
                m0 += m; t0 = u - m * dm.n_r;
                group_sync();
                filled = true;
            }
            if (!has) continue;
#pragma unroll 1
            for (int kb = 0; kb < nk; kb += 16 * KS) {
                uint4 qr[KS][2][PL], gr[KS][2][PL];
                float c[RT][2 * KS][4], dp[RT][2 * KS][4];
#pragma unroll
                for (int s = 0; s < KS; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t qt = tab[kb + 16 * s + 8 * e + g];
                        ld_token<PL>(qr[s][e], Qb, qt);
                        ld_token<PL>(gr[s][e], Gb, qt);
                    }
#pragma unroll
                for (int s = 0; s < KS; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int x = 0; x < RT; ++x) {
                            mma_rows<PL>(c[x][2 * s + e], ka[x], qr[s][e]);       // S^T = K Q^T
                            mma_rows<PL>(dp[x][2 * s + e], va[x], gr[s][e]);      // dP^T = V dO^T
                        }
#pragma unroll
                for (int j = 0; j < 2 * KS; ++j) {
                    const float2 l2 = *reinterpret_cast<const float2*>(s_l2 + kb + 8 * j + 2 * t4);
                    const float2 dl = *reinterpret_cast<const float2*>(s_dl + kb + 8 * j + 2 * t4);
#pragma unroll
                    for (int x = 0; x < RT; ++x) {
                        c[x][j][0] = ex2_approx(fmaf(c[x][j][0], sl2, -l2.x));
                        c[x][j][1] = ex2_approx(fmaf(c[x][j][1], sl2, -l2.y));
                        c[x][j][2] = ex2_approx(fmaf(c[x][j][2], sl2, -l2.x));
                        c[x][j][3] = ex2_approx(fmaf(c[x][j][3], sl2, -l2.y));
                        dp[x][j][0] = c[x][j][0] * (dp[x][j][0] - dl.x);
                        dp[x][j][1] = c[x][j][1] * (dp[x][j][1] - dl.y);
                        dp[x][j][2] = c[x][j][2] * (dp[x][j][2] - dl.x);
                        dp[x][j][3] = c[x][j][3] * (dp[x][j][3] - dl.y);
                    }
                }
#pragma unroll
                for (int s = 0; s < KS; ++s) {
                    mma_tokens<PL, EXACT>(dkx, dp, 2 * s, qr[s][0], qr[s][1]);    // dK += dS^T Q
                    mma_tokens<PL, EXACT>(dvx, c, 2 * s, gr[s][0], gr[s][1]);     // dV += P^T dO
                }
            }
        }
        if (CUT && s_job[0] > 1) {                                    // the sums of a part: to scratch memory
            // (a warp whose last round has no tile for it: what would be its place is another part's)
            if (!has) continue;
            float* at = sums + sum_at(s_job[1], tile);
#pragma unroll
            for (int p = 0; p < PL; ++p)
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        __stcg(at + ((p * 4 + n) * 4 + e) * 32, dkx[0][p][n][e]);
                        __stcg(at + ((PL * 4 + p * 4 + n) * 4 + e) * 32, dvx[0][p][n][e]);
                    }
        } else {
            finish_rows<PL>(dKb, st, dkx[0], dvx[0], tok[0], tile, ntok, g, t4, dm);
        }
    }
    if (CUT && s_job[0] > 1) {                                        // the part that is done last adds them up
        const int nparts = s_job[0], first = s_job[1] - s_job[2];
        int last = 0;
        __threadfence();
        group_sync();
        if (glane == 0) last = atomicAdd(done + (((size_t)b * dm.heads + h) * dm.R + jr) * gm.chunks + ck, 1) == nparts - 1;
        last = one_warp ? __shfl_sync(0xffffffffu, last, 0) : __syncthreads_or(last);
        if (!last) { cp_async_wait<0>(); return; }
        __threadfence();
        for (int tile = gwarp; tile * 16 < ntok; tile += gwarps)
            sum_parts<PL>(sums + sum_at(first, tile), nparts, (size_t)gm.chunks * gm.tpc * 1024 * PL, dKb, st, jr, c0, tile, ntok, lane, dm, gm);
    }
    cp_async_wait<0>();
    group_sync();
    // ---- LCE adjoint + store of dV: dV[y,x] += sum_ij w[i,j] dO[y-i+2, x-j+2] = correlation with the flipped filter ----
    lce_chunk<PL, TY, TX, true>(st, sbase + gm.off_halo + grp * gm.halo_bytes, s_w, nullptr, dm.lce, dVg + head_off / 2, y0, x0, rows, dm, gm,
                            gwarp, gwarps, lane);
}

// Geometry in the parameters' own memory or held by value: the same code with other registers.  Whole lists with 16 + 16 bits of P at 32
// channels are better off with the second (30 x 80 x 80, 12 x 12 regions, spills 128 -> 108 bytes: gradients 446 -> 440 us), all others with the
// first (whole lists at 64 channels 16 x 32 x 32, 12 heads 377 -> 373 us, at 32 channels 4 x 11 x 11, 24 heads, topk 49 86.7 -> 85.5; spills of
// cut lists at 64 channels 136 -> 92 bytes).
template <int PL, bool EXACT, bool CUT, int TY, int TX>
__global__ void __launch_bounds__(PL == 2 ? 128 : 256, PL == 2 ? 3 : 2)
bwd_dkv_direct_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg, const __nv_bfloat16* __restrict__ Vg,
                      const int32_t* inv_off, const int32_t* inv_list, const int32_t* inv_order, const float* __restrict__ lse,
                      const float* delta, const __nv_bfloat16* __restrict__ dOg, const float* __restrict__ lce_w,
                      __nv_bfloat16* __restrict__ dKg, __nv_bfloat16* __restrict__ dVg, const int2* jobs, ListParts parts, int32_t* done,
                      float* sums, int job0, const __grid_constant__ Dims dm, const __grid_constant__ DirGeom gm) {
    bwd_dkv_direct<PL, EXACT, CUT, TY, TX>(Qg, Kg, Vg, inv_off, inv_list, inv_order, lse, delta, dOg, lce_w, dKg, dVg, jobs, parts, done, sums,
                                           job0, dm, gm);
}
template <int TY, int TX>
__global__ void __launch_bounds__(256, 2)
bwd_dkv_exact_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg, const __nv_bfloat16* __restrict__ Vg,
                     const int32_t* inv_off, const int32_t* inv_list, const int32_t* inv_order, const float* __restrict__ lse,
                     const float* delta, const __nv_bfloat16* __restrict__ dOg, const float* __restrict__ lce_w,
                     __nv_bfloat16* __restrict__ dKg, __nv_bfloat16* __restrict__ dVg, int job0, Dims dm, DirGeom gm) {
    bwd_dkv_direct<1, true, false, TY, TX>(Qg, Kg, Vg, inv_off, inv_list, inv_order, lse, delta, dOg, lce_w, dKg, dVg, nullptr, ListParts(),
                                            nullptr, nullptr, job0, dm, gm);
}

// ------------------------------------------------------------------ host side
static bool dq_single(const Dims& d) { return d.d == 32 && d.topk * d.n_r <= 64 && !direct_exact(d); }
static DirGeom dq_geom(const Dims& d) {
    Dims k = d;
    if (dq_single(d)) k.topk = (64 + d.n_r - 1) / d.n_r;             // one block of 64 keys
    DirGeom g = direct_geom(k, false, 4, 1);
    g.smem_bytes = g.off_tab + g.gpc * g.tab_bytes;                  // the table only
    const int inv = (int)inverse_smem(d, true);
    if (g.smem_bytes < inv) g.smem_bytes = inv;
    return g;
}
static DirGeom dkv_geom(const Dims& d) {
    Dims full = d;
    full.topk = d.R;                                                 // a key region may be on every query region's list
    return direct_geom(full, d.lce, 12, 1);
}

bool backward_direct_supported(const Dims& d, int dtype) {
    if (!attend_direct_supported(d, dtype)) return false;
    return dkv_geom(d).smem_bytes <= 200 * 1024 && dq_geom(d).smem_bytes <= 200 * 1024 && d.R <= 8192;
}

// A part is the fair share, what a group of warps would have if all were busy from the first to the last, and at least 256 queries and 8
// entries (parts of 8 entries of 2 x 2 tokens, 10 x 15 x 15, 3 heads of 64, S = 8, topk 12: 61 / 80 us, lists whole / cut).  Where it is much more
// than the fair share the parts of a list are of one length: a list of an entry more than a part does not wait for a part of one (1 x 48 x 63,
// 12 heads, S = 16, topk 4 35.8 -> 33.2 us, lists whole 34.2).  Parts of the fair share stay whole but for the last, the longest first
// (2 x 100 x 167, 6 heads, topk 4 clustered 285, of one length 303; 1 x 112 x 112, 2 heads, S = 8, topk 8, 8 entries to a share of 7, 192 / 207).
// Lists are cut where the longest possible one is four parts or more, in problems that have no other kernels, if besides
//   all groups of warps are on the GPU at once: the longest list is what they wait for;
//   or the longest list of a map with a few kinds of content is three fair shares: a third of R, where topk is large 8/3 topk up to half of R
//   (R = 49: 19 - 22 entries, 64: 23 - 36, 256: 73 - 89), and the regions outside the map, whose scores are 0 and which all list the same;
//   or regions have 128 tokens and more, beside which the sums of a part do not show, and R is five fair shares.
// Measured (B200, us, gradients, lists whole / cut).  Content in a few kinds: 2 x 100 x 167, 6 heads, S = 16, topk 4 (87 % of the lists are
// empty, the longest has 73 entries) 351 / 284, 1 x 123 x 99, 4 heads, topk 2 130 / 52, 4 x 32 x 32, 6 heads of 64, S = 8, topk 12 71 / 57,
// 2 x 96 x 96, 3 heads, S = 8, topk 4 215 / 198, 8 x 80 x 80, 3 heads, S = 7, topk 1 182 / 172, 3 x 27 x 27, 12 heads of 64, topk 12 105 / 95.  Evenly
// spread lists there: 284 / 287, 61 / 46, 63 / 55, 169 / 171, 169 / 171, 89 / 89; 2 x 85 x 137, 6 heads, S = 16, topk 2 117 / 120, 2 x 74 x 46, 12 heads,
// topk 8 76 / 78.  Not cut: 10 x 32 x 32, 3 heads of 64, topk 12 clustered 80 / 87, evenly 81 / 85; 10 x 32 x 32, 6 heads, S = 7, topk 4 65 / 69 and
// 67 / 67; 7 x 40 x 40 75 / 79 and 77 / 77; 9 x 44 x 44, 4 heads 93 / 97 and 94 / 96; 31 x 64 x 64, 2 heads, topk 1 223 / 227 and 235 / 235; 12 x 96 x 96,
// 3 heads 395 / 398 and 404 / 407.
ListParts direct_grad_parts(const Dims& d, int* chunks, size_t* sum_bytes) {
    ListParts p = {0, d.R, 0, false};
    *sum_bytes = 0;
    *chunks = 1;
    if (!backward_direct_supported(d, d.esize == 2 ? BRA_BF16 : BRA_F32) || (backward_one_supported(d, BRA_BF16) && one_grad_pays(d)) ||
        (backward_dense_supported(d, BRA_BF16) && dense_grad_pays(d)) || (backward_img_supported(d, BRA_BF16) && img_grad_pays(d)))
        return p;
    const DirGeom g = dkv_geom(d);
    *chunks = g.chunks;
    const int warps = g.planes == 2 ? 12 : 16;                        // of an SM
    const long long slots = (long long)kSMs * (g.gpc > 1 ? warps : warps / g.nw > 0 ? warps / g.nw : 1);
    const long long entries = (long long)d.R * d.topk, work = entries * d.B * d.heads * g.chunks;
    const long long fair = (work + slots - 1) / slots;
    long long most = fair;
    if (most < (256 + d.n_r - 1) / d.n_r) most = (256 + d.n_r - 1) / d.n_r;
    if (most < 8) most = 8;
    if (4 * most > d.R) return p;                                     // (a list is longer than R only where it repeats regions)
    const int outside = d.R - ((d.H0 + d.hs - 1) / d.hs) * ((d.W0 + d.ws - 1) / d.ws);
    const int half = d.R / 2 < 8 * d.topk / 3 ? d.R / 2 : 8 * d.topk / 3;
    const long long longest = (d.R / 3 > half ? d.R / 3 : half) + outside;
    if (work > d.topk * slots && 3 * work > longest * slots && (d.n_r < 128 || 5 * work > d.R * slots)) return p;
    p.most = (int)most;
    p.even = 4 * most >= 5 * fair;
    p.jobs = d.R + (int)(entries / most);
    p.cut = (int)(2 * entries / most);
    *sum_bytes = (size_t)d.B * d.heads * p.cut * g.chunks * g.tpc * 4096 * g.planes;
    return p;
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
    int32_t *inv_off, *inv_list, *inv_order;
    const float *lce_w, *lse;
    __nv_bfloat16 *dq, *dk, *dv;
    float* delta;
    ListParts parts;
    int chunks;
    int2* jobs;
    int32_t* done;
    float* sums;
    int32_t* status;
    cudaStream_t st;
};
}  // namespace

template <int PL, bool EXACT, bool SINGLE>
static cudaError_t launch_dq(const Dims& d, const BwdArgs& a) {
    const DirGeom g = dq_geom(d);
    auto kernel = bwd_dq_direct_kernel<PL, EXACT, SINGLE>;
    static PerDeviceMax set;
    const cudaError_t e = allow_smem(set, kernel, g.smem_bytes);
    if (e != cudaSuccess) return e;
    return grid_pieces(d, [&](const GridPiece& p) {
        const InversePiece inv = inverse_piece(d, p, a.inv_off, a.inv_list, a.inv_order);
        const int counters = (d.heads_i == 1 ? d.heads : 1) * d.R * a.chunks;
        const ListJobs lj = {a.jobs + (size_t)p.b0 * d.heads_i * a.parts.jobs, a.done + (size_t)p.b0 * d.heads_i * counters, counters, a.parts};
        count_launch();
        return launch_kernel(kernel, dim3(g.gpi > d.heads_i ? g.gpi : d.heads_i, p.heads + 1, p.images), dim3(g.nw * 32), (size_t)g.smem_bytes, a.st,
                             false, a.q + p.tensor, a.k + p.tensor, a.v + p.tensor, a.index + p.index, a.lse + p.stat, a.go + p.tensor,
                             a.dq + p.tensor, a.delta + p.stat, p.h0 ? nullptr : inv.off, inv.list, inv.order, inverse_uses_bits(d), lj, a.status, d, g);
    });
}

template <typename F>
static cudaError_t launch_dkv_pieces(const Dims& d, const BwdArgs& a, const DirGeom& g, F&& launch) {
    return group_pieces(d, (a.parts.jobs + g.gpc - 1) / g.gpc * g.chunks, g.chunks, [&](const GridPiece& p, int groups_before, int groups) {
        count_launch();
        return launch(p, inverse_piece(d, p, a.inv_off, a.inv_list, a.inv_order), dim3(p.heads, p.images, groups), groups_before * g.gpc);
    });
}
template <int PL, bool EXACT, bool CUT, int TY, int TX>
static cudaError_t launch_dkv_t(const Dims& d, const BwdArgs& a) {
    const DirGeom g = dkv_geom(d);
    auto kernel = bwd_dkv_direct_kernel<PL, EXACT, CUT, TY, TX>;
    static PerDeviceMax set;
    const cudaError_t e = allow_smem(set, kernel, g.smem_bytes);
    if (e != cudaSuccess) return e;
    return launch_dkv_pieces(d, a, g, [&](const GridPiece& p, const InversePiece& inv, dim3 grid, int job0) {
        const size_t bh = (size_t)p.b0 * d.heads;
        return launch_kernel(kernel, grid, dim3(g.nw * 32), (size_t)g.smem_bytes, a.st, true, a.q + p.tensor, a.k + p.tensor, a.v + p.tensor,
                             inv.off, inv.list, inv.order, a.lse + p.stat, a.delta + p.stat, a.go + p.tensor, a.lce_w, a.dk + p.tensor,
                             a.dv + p.tensor, a.jobs + (size_t)p.b0 * d.heads_i * a.parts.jobs, a.parts, a.done + bh * d.R * g.chunks,
                             a.sums + bh * a.parts.cut * g.chunks * g.tpc * 1024 * PL, job0, d, g);
    });
}
template <int TY, int TX>
static cudaError_t launch_dkv_exact(const Dims& d, const BwdArgs& a) {
    const DirGeom g = dkv_geom(d);
    auto kernel = bwd_dkv_exact_kernel<TY, TX>;
    static PerDeviceMax set;
    const cudaError_t e = allow_smem(set, kernel, g.smem_bytes);
    if (e != cudaSuccess) return e;
    return launch_dkv_pieces(d, a, g, [&](const GridPiece& p, const InversePiece& inv, dim3 grid, int job0) {
        return launch_kernel(kernel, grid, dim3(g.nw * 32), (size_t)g.smem_bytes, a.st, true, a.q + p.tensor, a.k + p.tensor, a.v + p.tensor,
                             inv.off, inv.list, inv.order, a.lse + p.stat, a.delta + p.stat, a.go + p.tensor, a.lce_w, a.dk + p.tensor,
                             a.dv + p.tensor, job0, d, g);
    });
}
template <int PL, bool EXACT, int TY, int TX>
static cudaError_t launch_dkv(const Dims& d, const BwdArgs& a) {
    if (a.parts.most) return launch_dkv_t<PL, EXACT, true, TY, TX>(d, a);
    if constexpr (PL == 1 && EXACT) return launch_dkv_exact<TY, TX>(d, a);
    else return launch_dkv_t<PL, EXACT, false, TY, TX>(d, a);
}

static cudaError_t launch_both(const Dims& d, const BwdArgs& a) {
    const bool exact = direct_exact(d);
    const cudaError_t e = d.d == 64      ? launch_dq<2, true, false>(d, a)
                        : exact          ? launch_dq<1, true, false>(d, a)
                        : dq_single(d)   ? launch_dq<1, false, true>(d, a)
                                         : launch_dq<1, false, false>(d, a);
    if (e != cudaSuccess) return e;
    if (d.d == 64) return d.hs <= 2 ? launch_dkv<2, true, 2, 2>(d, a) : launch_dkv<2, true, 4, 4>(d, a);
    if (exact) return d.hs <= 2 ? launch_dkv<1, true, 2, 2>(d, a) : launch_dkv<1, true, 4, 4>(d, a);
    if (d.hs <= 2) return launch_dkv<1, false, 2, 2>(d, a);
    switch (lce_tile_width(dkv_geom(d), d)) {
        case 2: return launch_dkv<1, false, 4, 2>(d, a);
        case 3: return launch_dkv<1, false, 4, 3>(d, a);
        default: return launch_dkv<1, false, 4, 4>(d, a);
    }
}

cudaError_t launch_backward_direct(const Dims& d, const void* Q, const void* K, const void* V, const int32_t* index, char* ws, const WsLayout& L,
                                   const float* lce_w, const float* lse, const void* dO, void* dQ, void* dK, void* dV, cudaStream_t st) {
    typedef __nv_bfloat16 bf;
    int chunks;
    size_t sum_bytes;
    const ListParts parts = direct_grad_parts(d, &chunks, &sum_bytes);
    auto at = [&](size_t off) { return reinterpret_cast<int32_t*>(ws + off); };
    const BwdArgs a = {static_cast<const bf*>(Q), static_cast<const bf*>(K), static_cast<const bf*>(V), static_cast<const bf*>(dO), index,
                       at(L.inv_off), at(L.inv_list), at(L.inv_order), lce_w, lse, static_cast<bf*>(dQ), static_cast<bf*>(dK), static_cast<bf*>(dV),
                       reinterpret_cast<float*>(ws + L.delta), parts, chunks, reinterpret_cast<int2*>(ws + L.jobs), at(L.done),
                       reinterpret_cast<float*>(ws + L.sums), at(L.status), st};
    return launch_both(d, a);
}

}  // namespace bra
