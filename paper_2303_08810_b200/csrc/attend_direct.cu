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
// the routed keys (every group reads topk * n_r of them).
#include "direct_common.cuh"

#include <type_traits>

namespace bra {

using namespace ptx;

template <int PL, bool EXACT, bool ZEROS, int TY, int TX>
__global__ void __launch_bounds__(PL == 2 ? 128 : 256, PL == 2 ? 3 : 2)
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

    float* s_w = reinterpret_cast<float*>(smem + gm.off_w);
    if (dm.lce) {
        load_lce_weights(s_w, lce_w, h, 32 * PL * 25, tid, gm.nw * 32);
        if (live) load_halo<PL>(sbase + gm.off_halo + grp * gm.halo_bytes, Vh, y0, x0, rows, dm, gm, glane, glanes);
    }
    cp_async_commit();
    __syncthreads();                                                  // weights
    pdl_wait();          // in bra_forward the launch may overlap the tail of the routing kernel
    if (!live) return;                                                // a whole warp (one_warp) and no barrier of the CTA follows

    const int hi = dm.heads_i == 1 ? 0 : h;
    const int32_t* irow = index + (((size_t)b * dm.heads_i + hi) * dm.R + i) * dm.topk;
    const int total = dm.topk * dm.n_r;
    uint32_t* tab = reinterpret_cast<uint32_t*>(smem + gm.off_tab) + grp * gm.tab;
    float* st = reinterpret_cast<float*>(smem + gm.off_st + grp * gm.st_bytes);
    const float sl2 = dm.scale * 1.4426950408889634f;
    const int passes = (total + gm.tab - 1) / gm.tab;
    bool any_bad = false;

    for (int tile = gwarp; tile - gwarp < gm.tpc; tile += gwarps) {   // every warp of the group takes the same number of rounds
        const bool has = tile * 16 < ntok;
        uint32_t qa[PL][2][4];
        {
            uint4 lo[PL], hi4[PL];
            const int ta = tile * 16 + g, tb = ta + 8;
            ld_row<PL>(lo, Qb, ta < ntok ? token_of(dm, gm, i, ck * gm.hb * dm.ws + ta) : -1, tok_bytes);
            ld_row<PL>(hi4, Qb, tb < ntok ? token_of(dm, gm, i, ck * gm.hb * dm.ws + tb) : -1, tok_bytes);
            rows_to_a<PL>(qa, lo, hi4);
        }
        float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
        float o[PL][4][4];
#pragma unroll
        for (int p = 0; p < PL; ++p)
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[p][n][e] = 0.f;

        for (int pass = 0; pass < passes; ++pass) {
            const int k0 = pass * gm.tab;
            const int nk = min(gm.tab, (total - k0 + 31) / 32 * 32);
            if (passes > 1 || tile == gwarp) {
                if (pass > 0 || tile != gwarp) group_sync();          // the table before has been read
                const bool bad = fill_keys(tab, irow, i, k0, nk, total, glane, glanes, status, dm, gm);
                any_bad = (one_warp ? __any_sync(0xffffffffu, bad) : __syncthreads_or(bad)) || any_bad;
                if (one_warp) __syncwarp();
            }
            if (!has) continue;
            uint4 kr[2][2][PL], vr[2][2][PL];                         // [16-key step][rows g, g + 8]
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int e = 0; e < 2; ++e) ld_token<PL, ZEROS>(kr[s][e], Kb, tab[16 * s + 8 * e + g]);
            for (int kb = 0; kb < nk; kb += 32) {
                float c[4][4];
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_rows<PL>(c[j], qa, kr[j >> 1][j & 1]);
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        ld_token<PL, ZEROS>(vr[s][e], Vb, tab[kb + 16 * s + 8 * e + g]);
                        if (kb + 32 < nk) ld_token<PL, ZEROS>(kr[s][e], Kb, tab[kb + 32 + 16 * s + 8 * e + g]);
                    }
                if (any_bad || k0 + kb + 32 > total) {                // keys that do not count
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int kk = k0 + kb + 8 * j + 2 * t4;
                        if (dead_key(kk, total, any_bad, irow, dm, gm)) { c[j][0] = -INFINITY; c[j][2] = -INFINITY; }
                        if (dead_key(kk + 1, total, any_bad, irow, dm, gm)) { c[j][1] = -INFINITY; c[j][3] = -INFINITY; }
                    }
                }
                float mx[2];
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    mx[r] = fmaxf(fmax3(fmax3(c[0][2 * r], c[0][2 * r + 1], c[1][2 * r]), c[1][2 * r + 1], c[2][2 * r]),
                                  fmax3(c[2][2 * r + 1], c[3][2 * r], c[3][2 * r + 1])) * sl2;
                if (__any_sync(0xffffffffu, mx[0] > m_run[0] || mx[1] > m_run[1])) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
                        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
                        const float mnew = fmaxf(m_run[r], mx[r]);
                        const float corr = mnew == -INFINITY ? 1.f : ex2_approx(m_run[r] - mnew);
                        m_run[r] = mnew;
                        l_run[r] *= corr;
#pragma unroll
                        for (int p = 0; p < PL; ++p)
#pragma unroll
                            for (int n = 0; n < 4; ++n) { o[p][n][2 * r] *= corr; o[p][n][2 * r + 1] *= corr; }
                    }
                }
                const float mn0 = m_run[0] == -INFINITY ? 0.f : -m_run[0], mn1 = m_run[1] == -INFINITY ? 0.f : -m_run[1];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    c[j][0] = ex2_approx(fmaf(c[j][0], sl2, mn0));
                    c[j][1] = ex2_approx(fmaf(c[j][1], sl2, mn0));
                    c[j][2] = ex2_approx(fmaf(c[j][2], sl2, mn1));
                    c[j][3] = ex2_approx(fmaf(c[j][3], sl2, mn1));
                    l_run[0] += c[j][0] + c[j][1];
                    l_run[1] += c[j][2] + c[j][3];
                }
#pragma unroll
                for (int s = 0; s < 2; ++s) mma_tokens<PL, EXACT>(o, c[2 * s], c[2 * s + 1], vr[s][0], vr[s][1]);
            }
        }
        // ---- normalise; O^att to the staging tile; lse ----
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 1);
            l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 2);
            const int tk = tile * 16 + g + 8 * r;
            if (has && tk < ntok) {
                const float inv = l_run[r] > 0.f ? 1.f / l_run[r] : 0.f;
                float* dst = st + tk * 32 * PL + t4 * 8;
#pragma unroll
                for (int p = 0; p < PL; ++p)
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        *reinterpret_cast<float4*>(dst + p * 32 + 4 * q) =
                            make_float4(o[p][2 * q][2 * r] * inv, o[p][2 * q][2 * r + 1] * inv, o[p][2 * q + 1][2 * r] * inv, o[p][2 * q + 1][2 * r + 1] * inv);
                if (lse && t4 == 0) {
                    const int tok = token_of(dm, gm, i, ck * gm.hb * dm.ws + tk);
                    if (tok >= 0) lse[((size_t)b * dm.heads + h) * N0 + tok] = (m_run[r] + log2f(l_run[r])) * 0.6931471805599453f;
                }
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
    if (d.ws > 128 || d.R > 65535 || (long long)d.topk * d.n_r * d.n_r >= (1ll << 32)) return false;   // fast division by n_r
    if ((long long)d.H0 * d.W0 * d.C / 8 >= (1ll << 31) || d.heads > 65535 || d.B > 65535) return false;
    return direct_geom(d, d.lce, 4).smem_bytes <= 200 * 1024;
}

template <int PL, bool EXACT, bool ZEROS, int TY, int TX>
static cudaError_t launch_t(const Dims& d, const DirGeom& g, const void* Q, const void* K, const void* V, const int32_t* index,
                            const float* lce_w, const float* lce_b, void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    auto kernel = attend_direct_kernel<PL, EXACT, ZEROS, TY, TX>;
    static PerDeviceMax smem_set;
    if (g.smem_bytes > 48 * 1024) {
        const cudaError_t e = smem_set.ensure(g.smem_bytes, [&] {
            return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, g.smem_bytes);
        });
        if (e != cudaSuccess) return e;
    }
    count_launch();
    return launch_kernel(kernel, dim3(g.gpi, d.heads, d.B), dim3(g.nw * 32), (size_t)g.smem_bytes, st, after_own_kernel,
                         static_cast<const __nv_bfloat16*>(Q), static_cast<const __nv_bfloat16*>(K), static_cast<const __nv_bfloat16*>(V),
                         index, lce_w, lce_b, static_cast<__nv_bfloat16*>(O), lse, status, d, g);
}

cudaError_t launch_attend_direct(const Dims& d, const void* Q, const void* K, const void* V,
                                 const int32_t* index, const float* lce_w, const float* lce_b,
                                 void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    const DirGeom g = direct_geom(d, d.lce, 4);
    const bool zeros = d.H != d.H0 || d.W != d.W0;
    auto go = [&](auto z) -> cudaError_t {
        constexpr bool Z = decltype(z)::value;
#define BRA_GO(PL, EX, TY, TX) return launch_t<PL, EX, Z, TY, TX>(d, g, Q, K, V, index, lce_w, lce_b, O, lse, status, st, after_own_kernel)
        if (d.hs <= 2) { if (g.planes == 2) BRA_GO(2, false, 2, 2); BRA_GO(1, false, 2, 2); }
        if (g.planes == 2) BRA_GO(2, false, 4, 4);
        if (direct_exact(d)) BRA_GO(1, true, 4, 3);
        switch (lce_tile_width(g, d)) {
            case 2: BRA_GO(1, false, 4, 2);
            case 3: BRA_GO(1, false, 4, 3);
            default: BRA_GO(1, false, 4, 4);
        }
#undef BRA_GO
    };
    return zeros ? go(std::true_type()) : go(std::false_type());
}

}  // namespace bra
