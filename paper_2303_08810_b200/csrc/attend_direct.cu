// Routed token-to-token attention + LCE with warp-level tensor-core MMAs (Eq. 6, Eq. 7 with Eq. 1):
// head dim 32 or 64, bf16, any region shape, any topk, any map (also one that S does not divide).
//
// A group is one region's tokens of one (image, head), each group with its own routed keys.  A warp owns 16 query rows
// of a group and streams the group's keys and values from global memory straight into MMA fragments (the layouts of
// direct_common.cuh): no staging tiles, no barriers in the key loop, registers the only limit on how many warps an SM
// holds.  The warps of a region find one another's keys in L1.  Regions of at most 16 tokens are one warp each.  What
// the routing index contributes is a table of token numbers in shared memory, built once per group (per 512 keys):
// K^g / V^g are never formed.  Online softmax in blocks of 32 keys.
// O^att goes through shared memory (fp32) to the LCE's thread mapping: lane = channel pair, 4 x 4 positions in
// registers, V from a halo tile copied while the attention ran.
//
// What bounds it: one m16n8k16 MMA takes 8 cycles of a scheduler's tensor pipe (16 per 16 queries x 64 keys x 32
// channels: S and P V) and the softmax needs about as many issue slots; with regions of few tokens, the L2 traffic of
// the routed keys (every group reads topk * n_r of them).  Counters at 2 x 100 x 167, S = 16, topk 4, 6 heads: 0.53
// instructions per cycle and scheduler, tensor pipe 14 %; at 16 x 32 x 32, 12 heads of 64: 0.40, 2.2 cycles per issue waiting
// for loads, 1.7 in fixed waits: latency at 12 warps per SM.
// Measured (B200) against staging keys and values in shared memory: 16 x 32 x 32, 12 heads of 64, topk 12: 278 -> 126 us;
// 2 x 100 x 167, 6 heads: 131 us and four padded copies -> 114 us and none.  Small maps: attend_img.cu
// where it has the CTAs (img_pays()).  A reference maximum that moves only for scores 8 above it: no faster, error
// 2.0e-3 -> 2.1e-3.
#include "direct_common.cuh"

namespace bra {

using namespace ptx;

template <int PL, bool EXACT, int RT, int TY, int TX>
__global__ void __launch_bounds__((PL == 2 ? 128 : 256) / RT, RT == 2 ? (PL == 2 ? 4 : 3) : PL == 2 ? 3 : 2)
attend_direct_kernel(const __nv_bfloat16* __restrict__ Qg, const __nv_bfloat16* __restrict__ Kg,
                     const __nv_bfloat16* __restrict__ Vg, const int32_t* index,
                     const float* __restrict__ lce_w, const float* __restrict__ lce_b,
                     __nv_bfloat16* __restrict__ O, float* __restrict__ lse,
                     int32_t* __restrict__ status, Dims dm, DirGeom gm) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3;

    // ---- which group (image, head, region) and chunk of its rows ----
    const bool one_warp = gm.gpc > 1;                                 // a group is one warp
    const int rest = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int grp = one_warp ? warp : 0;
    const int ck = one_warp ? 0 : rest % gm.chunks;
    const int i = one_warp ? rest * gm.gpc + warp : rest / gm.chunks;
    const int gwarp = one_warp ? 0 : warp, gwarps = one_warp ? 1 : gm.nw;
    const int glane = one_warp ? lane : tid, glanes = gwarps * 32;
    const bool live = i < dm.R;
    auto group_sync = [&]() { if (one_warp) __syncwarp(); else __syncthreads(); };

    const int ri = live ? i : 0;
    const int ry = fdiv(ri, dm.S, gm.mul_s), rx = ri - ry * dm.S;
    const int y0 = ry * dm.hs + ck * gm.hb, x0 = rx * dm.ws;          // first token of the chunk
    const int rows = min(gm.hb, dm.hs - ck * gm.hb);
    const int ntok = rows * dm.ws;
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
    const int N0 = dm.H0 * dm.W0;
    const size_t head_off = (size_t)b * N0 * tok_bytes + (size_t)h * 64 * PL;
    const uint8_t* Qb = reinterpret_cast<const uint8_t*>(Qg) + head_off + t4 * 16;
    const uint8_t* Kb = reinterpret_cast<const uint8_t*>(Kg) + head_off + t4 * 16;
    const uint8_t* Vh = reinterpret_cast<const uint8_t*>(Vg) + head_off;
    const uint8_t* Vb = Vh + t4 * 16;

    const uint4 probe = spare_probe<PL>(Kb - t4 * 16, Vh, lane);
    float* s_w = reinterpret_cast<float*>(smem + gm.off_w);
    if (dm.lce) {
        load_lce_weights(s_w, lce_w, h, 32 * PL * 25, tid, gm.nw * 32);
        if (live) load_halo<PL>(sbase + gm.off_halo + grp * gm.halo_bytes, Vh, y0, x0, rows, dm, gm, glane, glanes);
    }
    cp_async_commit();
    uint32_t* tab = reinterpret_cast<uint32_t*>(smem + gm.off_tab + grp * gm.tab_bytes);
    uint32_t* dead = tab + gm.tab;
    int* zeros = reinterpret_cast<int*>(dead + gm.tab / 32);          // keys of the zero padding
    if (glane == 0) *zeros = 0;
    __syncthreads();                                                  // weights
    pdl_wait();          // in bra_forward the launch may overlap the tail of the routing kernel
    if (!live) return;                                                // a whole warp (one_warp) and no barrier of the CTA follows
    const int spare = spare_token<PL>(probe, Kb - t4 * 16, Vh, tok_bytes, N0, lane);

    const int hi = dm.heads_i == 1 ? 0 : h;
    const int32_t* irow = index + (((size_t)b * dm.heads_i + hi) * dm.R + i) * dm.topk;
    const int total = dm.topk * dm.n_r;
    float* st = reinterpret_cast<float*>(smem + gm.off_st + grp * gm.st_bytes);
    const float sl2 = dm.scale * 1.4426950408889634f;
    const int passes = (total + gm.tab - 1) / gm.tab;
    for (int tile = gwarp * RT; tile - gwarp * RT < gm.tpc; tile += gwarps * RT) {    // every warp of the group takes the same number of rounds
        const bool has = tile * 16 < ntok;
        const bool first_round = tile == gwarp * RT;
        uint32_t qa[RT][PL][2][4];
        int tok[RT][2];
#pragma unroll
        for (int x = 0; x < RT; ++x) {
            uint4 v[2][PL];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int t = (tile + x) * 16 + g + 8 * r;
                tok[x][r] = t < ntok ? token_of(dm, gm, i, ck * gm.hb * dm.ws + t) : -1;
                ld_row<PL>(v[r], Qb, tok[x][r], tok_bytes);
            }
            rows_to_a<PL>(qa[x], v[0], v[1]);
        }
        float m_run[RT][2], l_run[RT][2], o[RT][PL][4][4];
#pragma unroll
        for (int x = 0; x < RT; ++x) {
            m_run[x][0] = m_run[x][1] = -INFINITY;
            l_run[x][0] = l_run[x][1] = 0.f;
#pragma unroll
            for (int p = 0; p < PL; ++p)
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[x][p][n][e] = 0.f;
        }

        for (int pass = 0; pass < passes; ++pass) {
            const int k0 = pass * gm.tab;
            const int nk = min(gm.tab, (total - k0 + 31) / 32 * 32);
            if (passes > 1 || first_round) {
                if (pass > 0 || !first_round) group_sync();           // the table before has been read
                int z = fill_keys(tab, dead, irow, k0, nk, total, spare, glane, glanes, status, dm, gm);
                if (first_round) {
                    z = __reduce_add_sync(0xffffffffu, z);
                    if (lane == 0 && z) atomicAdd(zeros, z);
                }
                group_sync();
            }
            if (!has) continue;
            uint4 kr[2][2][PL], vr[2][2][PL];                         // [16-key step][rows g, g + 8]
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int e = 0; e < 2; ++e) ld_token<PL>(kr[s][e], Kb, tab[16 * s + 8 * e + g]);
            for (int kb = 0; kb < nk; kb += 32) {
                float c[RT][4][4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int x = 0; x < RT; ++x) mma_rows<PL>(c[x][j], qa[x], kr[j >> 1][j & 1]);
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        ld_token<PL>(vr[s][e], Vb, tab[kb + 16 * s + 8 * e + g]);
                        if (kb + 32 < nk) ld_token<PL>(kr[s][e], Kb, tab[kb + 32 + 16 * s + 8 * e + g]);
                    }
                const uint32_t bits = dead[kb >> 5];
                if (bits) mask_columns<RT, 4>(c, bits, t4, -INFINITY);
                float mx[RT][2];
                bool up = false;
#pragma unroll
                for (int x = 0; x < RT; ++x)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        mx[x][r] = fmaxf(fmax3(fmax3(c[x][0][2 * r], c[x][0][2 * r + 1], c[x][1][2 * r]), c[x][1][2 * r + 1], c[x][2][2 * r]),
                                         fmax3(c[x][2][2 * r + 1], c[x][3][2 * r], c[x][3][2 * r + 1])) * sl2;
                        up = up || mx[x][r] > m_run[x][r];
                    }
                if (__any_sync(0xffffffffu, up)) {
#pragma unroll
                    for (int x = 0; x < RT; ++x)
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            mx[x][r] = fmaxf(mx[x][r], __shfl_xor_sync(0xffffffffu, mx[x][r], 1));
                            mx[x][r] = fmaxf(mx[x][r], __shfl_xor_sync(0xffffffffu, mx[x][r], 2));
                            const float mnew = fmaxf(m_run[x][r], mx[x][r]);
                            const float corr = mnew == -INFINITY ? 1.f : ex2_approx(m_run[x][r] - mnew);
                            m_run[x][r] = mnew;
                            l_run[x][r] *= corr;
#pragma unroll
                            for (int p = 0; p < PL; ++p)
#pragma unroll
                                for (int n = 0; n < 4; ++n) { o[x][p][n][2 * r] *= corr; o[x][p][n][2 * r + 1] *= corr; }
                        }
                }
#pragma unroll
                for (int x = 0; x < RT; ++x) {
                    const float mn0 = m_run[x][0] == -INFINITY ? 0.f : -m_run[x][0], mn1 = m_run[x][1] == -INFINITY ? 0.f : -m_run[x][1];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        c[x][j][0] = ex2_approx(fmaf(c[x][j][0], sl2, mn0));
                        c[x][j][1] = ex2_approx(fmaf(c[x][j][1], sl2, mn0));
                        c[x][j][2] = ex2_approx(fmaf(c[x][j][2], sl2, mn1));
                        c[x][j][3] = ex2_approx(fmaf(c[x][j][3], sl2, mn1));
                        l_run[x][0] += c[x][j][0] + c[x][j][1];
                        l_run[x][1] += c[x][j][2] + c[x][j][3];
                    }
                }
#pragma unroll
                for (int s = 0; s < 2; ++s) mma_tokens<PL, EXACT>(o, c, 2 * s, vr[s][0], vr[s][1]);
            }
        }
        // ---- keys of the zero padding; normalise; O^att to the staging tile; lse ----
        const int nz = *zeros;
#pragma unroll
        for (int x = 0; x < RT; ++x)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float l = l_run[x][r], m = m_run[x][r], f = 1.f;
                l += __shfl_xor_sync(0xffffffffu, l, 1);
                l += __shfl_xor_sync(0xffffffffu, l, 2);
                if (nz) {                                             // nz scores of 0
                    const float mnew = fmaxf(m, 0.f);
                    f = ex2_approx(m - mnew);
                    l = l * f + (float)nz * ex2_approx(-mnew);
                    m = mnew;
                }
                const int tk = (tile + x) * 16 + g + 8 * r;
                if (tk < ntok) {
                    const float inv = l > 0.f ? f / l : 0.f;
                    float* dst = st + tk * 32 * PL + t4 * 8;
#pragma unroll
                    for (int p = 0; p < PL; ++p)
#pragma unroll
                        for (int q = 0; q < 2; ++q)
                            *reinterpret_cast<float4*>(dst + p * 32 + 4 * q) =
                                make_float4(o[x][p][2 * q][2 * r] * inv, o[x][p][2 * q][2 * r + 1] * inv, o[x][p][2 * q + 1][2 * r] * inv,
                                            o[x][p][2 * q + 1][2 * r + 1] * inv);
                    if (lse && t4 == 0 && tok[x][r] >= 0) lse[((size_t)b * dm.heads + h) * N0 + tok[x][r]] = (m + log2f(l)) * 0.6931471805599453f;
                }
            }
    }
    cp_async_wait<0>();
    group_sync();
    lce_chunk<PL, TY, TX, false>(st, sbase + gm.off_halo + grp * gm.halo_bytes, s_w, dm.lce && lce_b ? lce_b + h * 32 * PL : nullptr, dm.lce,
                             O + head_off / 2, y0, x0, rows, dm, gm, gwarp, gwarps, lane);
}

// ------------------------------------------------------------------ host side
bool attend_direct_supported(const Dims& d, int dtype) {
    if (dtype != BRA_BF16 || (d.d != 32 && d.d != 64)) return false;
    if (d.ws > 128 || d.R > 65535 || d.n_r >= 1 << 25) return false;                      // fdiv() by ws and S
    if ((long long)d.H0 * d.W0 * d.C / 8 >= (1ll << 31)) return false;
    return direct_geom(d, d.lce, 4, 1).smem_bytes <= 200 * 1024;
}

template <int PL, bool EXACT, int RT, int TY, int TX>
static cudaError_t launch_t(const Dims& d, const DirGeom& g, const void* Q, const void* K, const void* V, const int32_t* index,
                            const float* lce_w, const float* lce_b, void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    auto kernel = attend_direct_kernel<PL, EXACT, RT, TY, TX>;
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
        return launch_kernel(kernel, dim3(g.gpi, p.heads, p.images), dim3(g.nw * 32), (size_t)g.smem_bytes, st, after_own_kernel,
                             static_cast<const bf*>(Q) + p.tensor, static_cast<const bf*>(K) + p.tensor, static_cast<const bf*>(V) + p.tensor,
                             index + p.index, piece_of(lce_w, p.channel * 25), piece_of(lce_b, p.channel), static_cast<bf*>(O) + p.tensor,
                             piece_of(lse, p.stat), status, d, g);
    });
}

cudaError_t launch_attend_direct(const Dims& d, const void* Q, const void* K, const void* V,
                                 const int32_t* index, const float* lce_w, const float* lce_b,
                                 void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    const int rt = direct_rt(d);
    const DirGeom g = direct_geom(d, d.lce, 4, rt);
#define BRA_GO(PL, EX, RT, TY, TX) return launch_t<PL, EX, RT, TY, TX>(d, g, Q, K, V, index, lce_w, lce_b, O, lse, status, st, after_own_kernel)
    if (g.planes == 2) {
        if (direct_exact(d)) { if (rt == 2) BRA_GO(2, true, 2, 4, 4); BRA_GO(2, true, 1, 4, 4); }
        if (rt == 2) BRA_GO(2, false, 2, 4, 4);
        if (d.hs <= 2) BRA_GO(2, false, 1, 2, 2);
        BRA_GO(2, false, 1, 4, 4);
    }
    if (direct_exact(d)) { if (rt == 2) BRA_GO(1, true, 2, 4, 4); BRA_GO(1, true, 1, 4, 4); }
    const int tx = lce_tile_width(g, d);
    if (rt == 2) { if (tx == 2) BRA_GO(1, false, 2, 4, 2); if (tx == 3) BRA_GO(1, false, 2, 4, 3); BRA_GO(1, false, 2, 4, 4); }
    if (d.hs <= 2) BRA_GO(1, false, 1, 2, 2);
    if (tx == 2) BRA_GO(1, false, 1, 4, 2);
    if (tx == 3) BRA_GO(1, false, 1, 4, 3);
    BRA_GO(1, false, 1, 4, 4);
#undef BRA_GO
}

}  // namespace bra
