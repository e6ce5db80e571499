// Gradients for topk = 1 in one launch: head dim 32, bf16, regions of 17 to 64 tokens, any map.
//
// A query region attends to ONE key region, so the CTA of a key region sees all keys of every query that lists it: S, dP, P,
// delta and dS are made once and serve dQ, dK and dV, where the kernels of backward_direct.cu make them once per side, and
// there is no delta to hand over, no inverse index and no second launch.  The sums are theirs: P and dS rounded to bf16 for
// the products, fp32 accumulation, a fixed order.
//
// CTA = (key region, head, image), a warp per 16 tokens.  K, V of the region and Q, dO of the listing regions (one ahead) arrive
// as bulk tensor copies: boxes in the swizzled order that ldmatrix reads without bank conflicts, zero outside the map.  Per
// listing region a warp takes 16 queries against all keys (up to 64 scores a row in registers), stores dQ and puts P and dS
// into shared memory; then it takes the 16 keys it owns against all queries, both operands transposed by ldmatrix.  The
// list is read off the index by the CTA itself.
// Rows of a tile that are no query (behind the region's last token, outside the map) are zero in shared memory and have lse = inf, so P = 0.
// As A fragments they read a token of the region that exists instead: a zero row beside a key with an infinity scores NaN, a query that
// exists does so only where its gradients are NaN by rights.
//
// Bound: latency and issue at 16 warps per SM (64 x 56 x 56, 2 heads: 0.53 instructions per cycle and scheduler; a third of the time
// is the LCE adjoint).  Measured (B200), there, LCE gradient beside it: dQ + dK / dV 58 + 114 -> 97 us; forward + backward
// 238.9 -> 171.4; 64 x 40 x 40 212 -> 174, 64 x 48 x 48 260 -> 214; 8 images, clustered lists 78 -> 66.  One Q, dO buffer instead of two:
// 78 -> 78 there.  Regions of more than 64 tokens, a tile's keys shared by two warps: 8 x 64 x 64 (100 tokens) 98 -> 104, with
// two passes over the keys 98 -> 102: they keep backward_direct.cu.
#include "smem_rows.cuh"

namespace bra {

using namespace ptx;

namespace one {
constexpr int ST = 40;           // floats of a staged token
constexpr uint32_t POLL_LIMIT = 4000000u;
}

struct OneGeom {
    int arr_bytes;               // a [16 KT tokens][32 channels] array
    int p_pitch, p_bytes;        // a row, and all rows, of P (dS lies behind P)
    int off_p, off_list, off_w, off_halo, off_bar, smem_bytes;
    uint32_t box_bytes;
};

__device__ __forceinline__ void stmatrix_x4(uint32_t addr, const uint32_t (&r)[4]) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}

// Regions of 16 KT tokens; fewer; the map ends inside the last ones.
enum OneEdge { ONE_FULL, ONE_REST, ONE_CUT };

template <int KT, int TX, OneEdge EDGE>
__global__ void __launch_bounds__(32 * KT, 16 / KT)
bwd_one_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
               const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_g,
               const int32_t* __restrict__ index, const float* __restrict__ lse, const __nv_bfloat16* __restrict__ dOg,
               const float* __restrict__ lce_w, __nv_bfloat16* __restrict__ dQg, __nv_bfloat16* __restrict__ dKg,
               __nv_bfloat16* __restrict__ dVg, int32_t* __restrict__ status, int h0, int b0, Dims dm, DirGeom gm, OneGeom og) {
    constexpr int ST = one::ST;
    constexpr int NT = 2 * KT;                                        // 8-key tiles
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const int h = blockIdx.x, j = blockIdx.y, b = blockIdx.z;
    const uint32_t s_k = sbase, s_v = s_k + og.arr_bytes, s_qg = s_v + og.arr_bytes;    // Q, dO of two regions
    const uint32_t s_p = sbase + og.off_p, s_ds = s_p + og.p_bytes;
    uint16_t* list = reinterpret_cast<uint16_t*>(smem + og.off_list);
    int* count = reinterpret_cast<int*>(smem + og.off_bar + 24);
    uint64_t* bar_kv = reinterpret_cast<uint64_t*>(smem + og.off_bar);
    uint64_t* bar_q = bar_kv + 1;                                     // one per buffer
    float* s_w = reinterpret_cast<float*>(smem + og.off_w);

    const int ry = fdiv(j, dm.S, gm.mul_s), rx = j - ry * dm.S;
    const int y0 = ry * dm.hs, x0 = rx * dm.ws, c0 = (h0 + h) * 32;
    const uint32_t tok_bytes = (uint32_t)dm.C * 2;
    const int N0 = dm.H0 * dm.W0;
    const size_t head_off = (size_t)b * N0 * tok_bytes + (size_t)h * 64;
    const float* lse_h = lse + ((size_t)b * dm.heads + h) * N0;
    const int32_t* irow = index + ((size_t)b * dm.heads_i + (dm.heads_i == 1 ? 0 : h)) * dm.R;
    const int own = __ldg(irow + j);                                  // the region that this one's queries attend to
    const bool cut = EDGE == ONE_CUT && (KT < 4 || dm.H != dm.H0 || dm.W != dm.W0);

    if (tid == 0) {
        mbar_init(bar_kv, 1);
        mbar_init(bar_q, 1);
        mbar_init(bar_q + 1, 1);
        fence_mbar_init();
        mbar_expect_tx(bar_kv, 2 * og.box_bytes);
        tma_load_4d(s_k, &map_k, bar_kv, c0, x0, y0, b0 + b);
        tma_load_4d(s_v, &map_v, bar_kv, c0, x0, y0, b0 + b);
    }
    // ---- the query regions that list this one, ascending ----
    auto fetch = [&](int it) {                                        // one thread: Q and dO of list[it]
        const int i = list[it], qy = fdiv(i, dm.S, gm.mul_s), qx = i - qy * dm.S;
        uint64_t* bar = bar_q + (it & 1);
        const uint32_t at = s_qg + (it & 1) * 2 * og.arr_bytes;
        mbar_expect_tx(bar, 2 * og.box_bytes);
        tma_load_4d(at, &map_q, bar, c0, qx * dm.ws, qy * dm.hs, b0 + b);
        tma_load_4d(at + og.arr_bytes, &map_g, bar, c0, qx * dm.ws, qy * dm.hs, b0 + b);
    };
    if (tid < 32) {
        int n = 0;
        for (int e0 = 0; e0 < dm.R; e0 += 128) {
            int r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) r[q] = e0 + 32 * q + lane < dm.R ? __ldg(irow + e0 + 32 * q + lane) : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                bool lists = r[q] == j;
                if (cut && lists) {                                   // not without a token
                    const int i = e0 + 32 * q + lane, qy = fdiv(i, dm.S, gm.mul_s);
                    lists = qy * dm.hs < dm.H0 && (i - qy * dm.S) * dm.ws < dm.W0;
                }
                const uint32_t m = __ballot_sync(0xffffffffu, lists);
                if (lists) list[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(e0 + 32 * q + lane);
                n += __popc(m);
            }
        }
        __syncwarp();
        if (lane == 0) {
            *count = n;
            if (n > 0) fetch(0);
            if (n > 1) fetch(1);
        }
    }
    if (dm.lce) {
        load_halo<1>(sbase + og.off_halo, reinterpret_cast<const uint8_t*>(dOg) + head_off, y0, x0, dm.hs, dm, gm, tid, blockDim.x);
        load_lce_weights(s_w, lce_w, h, 800, tid, blockDim.x);
    }
    cp_async_commit();
    // rows behind the last token: zero (the copies never write them)
    for (int e = dm.n_r * 4 + tid; e < KT * 64; e += KT * 32) {
        sts_f32x4(s_k + e * 16, 0.f, 0.f, 0.f, 0.f);
        sts_f32x4(s_v + e * 16, 0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 4; ++q) sts_f32x4(s_qg + q * og.arr_bytes + e * 16, 0.f, 0.f, 0.f, 0.f);
    }
    const int tk = warp * 16 + g;                                     // the lane's tokens of a region: tk, tk + 8
    int ty[2], tx[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) { ty[r] = fdiv(tk + 8 * r, dm.ws, gm.mul_ws); tx[r] = tk + 8 * r - ty[r] * dm.ws; }
    // row-major token of the map; -1: none
    auto token = [&](int r, int yy0, int xx0) {
        const int y = yy0 + ty[r], x = xx0 + tx[r];
        return tk + 8 * r < dm.n_r && y < dm.H0 && x < dm.W0 ? y * dm.W0 + x : -1;
    };
    if (own < 0 || own >= dm.R) {                                     // a bad entry: nothing is attended to
        if (tid == 0) record_error(status, BRA_ERR_INDEX, own);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int tok = token(r, y0, x0);
            if (tok >= 0) *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(dQg) + head_off + (size_t)(uint32_t)tok * tok_bytes + t4 * 16) = make_uint4(0, 0, 0, 0);
        }
    }
    __syncthreads();
    const int n = *count;

    float dk[4][4], dv[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) { dk[i][e] = 0.f; dv[i][e] = 0.f; }
    const uint32_t row_off = rows8_offset(lane), col_off = rows16_offset(lane);
    // the warp's 16 rows as A fragments
    const int row = warp * 16 + (lane & 15);
    uint32_t own_at = EDGE == ONE_FULL || row < dm.n_r ? warp * 1024 + col_off : col_off & 511u;    // (rows 0 .. 7: other banks)
    // P and dS: where a lane's row goes (16 queries x 16 keys), and as the transposed operand
    const uint32_t put_at = (warp * 16 + (lane & 15)) * og.p_pitch + (lane >> 4) * 16;
    const uint32_t get_at = ((lane & 7) + (lane >> 4) * 8) * og.p_pitch + warp * 32 + ((lane >> 3) & 1) * 16;
    auto put_rows = [&](uint8_t* base, int tok, const float (&acc)[4][4], int r) {   // a row of its sums, times the scale
        const uint4 v = pack_row_of_quad(acc, r, dm.scale, t4);
        if (tok >= 0) *reinterpret_cast<uint4*>(base + head_off + (size_t)(uint32_t)tok * tok_bytes + t4 * 16) = v;
    };
    const float sl2 = dm.scale * 1.4426950408889634f;
    const bool rest = EDGE != ONE_FULL && dm.n_r != 8 * NT;
    bool ok = true;
    if (n > 0 && !mbar_wait(bar_kv, 0, one::POLL_LIMIT)) ok = false;

#pragma unroll 1
    for (int it = 0; it < n; ++it) {
        const int i = list[it], qy = fdiv(i, dm.S, gm.mul_s), qx = i - qy * dm.S;
        const uint32_t s_q = s_qg + (it & 1) * 2 * og.arr_bytes, s_g = s_q + og.arr_bytes;
        int tok[2];
        float lse2[2], delta[2] = {0.f, 0.f};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            tok[r] = token(r, qy * dm.hs, qx * dm.ws);
            lse2[r] = tok[r] >= 0 ? __ldg(lse_h + tok[r]) * 1.4426950408889634f : INFINITY;
        }
        if (!mbar_try_wait(bar_q + (it & 1), it >> 1 & 1)) ok = mbar_wait(bar_q + (it & 1), it >> 1 & 1, ok ? one::POLL_LIMIT : 1u) && ok;
        if (cut) {
            const int y = fdiv(row, dm.ws, gm.mul_ws), x = row - y * dm.ws;
            own_at = row < dm.n_r && qy * dm.hs + y < dm.H0 && qx * dm.ws + x < dm.W0 ? warp * 1024 + col_off : (uint32_t)(lane >> 4) << 4;
        }
        float c[NT][4], dp[NT][4];
        {
            uint32_t qa[2][4], ga[2][4], f[4];
            ldmatrix_x4(s_q + own_at, qa[0]);
            ldmatrix_x4(s_q + (own_at ^ 32), qa[1]);
            if (KT == 4) {                                            // (one after the other: 109 -> 113 us at 64 x 56 x 56)
                ldmatrix_x4(s_g + own_at, ga[0]);
                ldmatrix_x4(s_g + (own_at ^ 32), ga[1]);
#pragma unroll
                for (int m = 0; m < NT; ++m) {
                    ldmatrix_x4(s_k + m * 512 + row_off, f);
                    mma_rows8(c[m], qa, f);
                    ldmatrix_x4(s_v + m * 512 + row_off, f);
                    mma_rows8(dp[m], ga, f);
                }
            } else {
#pragma unroll
                for (int m = 0; m < NT; ++m) {
                    ldmatrix_x4(s_k + m * 512 + row_off, f);
                    mma_rows8(c[m], qa, f);
                }
                ldmatrix_x4(s_g + own_at, ga[0]);
                ldmatrix_x4(s_g + (own_at ^ 32), ga[1]);
#pragma unroll
                for (int m = 0; m < NT; ++m) {
                    ldmatrix_x4(s_v + m * 512 + row_off, f);
                    mma_rows8(dp[m], ga, f);
                }
            }
        }
#pragma unroll
        for (int m = 0; m < NT; ++m) {
            c[m][0] = ex2_approx(fmaf(c[m][0], sl2, -lse2[0]));
            c[m][1] = ex2_approx(fmaf(c[m][1], sl2, -lse2[0]));
            c[m][2] = ex2_approx(fmaf(c[m][2], sl2, -lse2[1]));
            c[m][3] = ex2_approx(fmaf(c[m][3], sl2, -lse2[1]));
        }
        if (rest) {
            const int left = dm.n_r - 2 * t4;         // keys behind the region's last token
#pragma unroll
            for (int m = 0; m < NT; ++m) {
                if (8 * m >= left) c[m][0] = c[m][2] = 0.f;
                if (8 * m + 1 >= left) c[m][1] = c[m][3] = 0.f;
            }
        }
#pragma unroll
        for (int m = 0; m < NT; ++m) {
            delta[0] = fmaf(c[m][0], dp[m][0], fmaf(c[m][1], dp[m][1], delta[0]));
            delta[1] = fmaf(c[m][2], dp[m][2], fmaf(c[m][3], dp[m][3], delta[1]));
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            delta[r] += __shfl_xor_sync(0xffffffffu, delta[r], 1);
            delta[r] += __shfl_xor_sync(0xffffffffu, delta[r], 2);
        }
        float dq[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) dq[q][e] = 0.f;
#pragma unroll
        for (int s = 0; s < KT; ++s) {
            uint32_t a[4];
            frag_hi(a, c[2 * s], c[2 * s + 1]);
            stmatrix_x4(s_p + put_at + s * 32, a);
#pragma unroll
            for (int m = 2 * s; m < 2 * s + 2; ++m) {
                c[m][0] *= dp[m][0] - delta[0]; c[m][1] *= dp[m][1] - delta[0];
                c[m][2] *= dp[m][2] - delta[1]; c[m][3] *= dp[m][3] - delta[1];
            }
            frag_hi(a, c[2 * s], c[2 * s + 1]);
            stmatrix_x4(s_ds + put_at + s * 32, a);
#pragma unroll
            for (int q = 0; q < 2; ++q) {                             // dQ += dS K
                uint32_t f[4];
                ldmatrix_x4_trans(s_k + s * 1024 + (col_off ^ (q * 32)), f);
                mma_bf16(dq[2 * q], a, f[0], f[1]);
                mma_bf16(dq[2 * q + 1], a, f[2], f[3]);
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) put_rows(reinterpret_cast<uint8_t*>(dQg), tok[r], dq, r);
        __syncthreads();                                              // P and dS of all queries
#pragma unroll
        for (int s = 0; s < KT; ++s) {
            uint32_t a[4], f[4];
            ldmatrix_x4_trans(s_p + get_at + s * 16 * og.p_pitch, a);
#pragma unroll
            for (int q = 0; q < 2; ++q) {                        // dV += P^T dO
                ldmatrix_x4_trans(s_g + s * 1024 + (col_off ^ (q * 32)), f);
                mma_bf16(dv[2 * q], a, f[0], f[1]);
                mma_bf16(dv[2 * q + 1], a, f[2], f[3]);
            }
            ldmatrix_x4_trans(s_ds + get_at + s * 16 * og.p_pitch, a);
#pragma unroll
            for (int q = 0; q < 2; ++q) {                        // dK += dS^T Q
                ldmatrix_x4_trans(s_q + s * 1024 + (col_off ^ (q * 32)), f);
                mma_bf16(dk[2 * q], a, f[0], f[1]);
                mma_bf16(dk[2 * q + 1], a, f[2], f[3]);
            }
        }
        __syncthreads();                                              // read by all
        if (tid == 0 && it + 2 < n && ok) fetch(it + 2);
    }
    // ---- dK = scale * acc; dV to the staging tile ----
    float* st = reinterpret_cast<float*>(smem + og.off_p);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        put_rows(reinterpret_cast<uint8_t*>(dKg), token(r, y0, x0), dk, r);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *reinterpret_cast<float2*>(st + (tk + 8 * r) * ST + q * 8 + 2 * t4) = make_float2(dv[q][2 * r], dv[q][2 * r + 1]);
    }
    if (!ok && lane == 0) record_error(status, BRA_ERR_TIMEOUT, blockIdx.y);
    if (tid == 0 && !(n > 0 && ok)) {                                 // nothing in flight when the CTA leaves
        mbar_wait(bar_kv, 0, one::POLL_LIMIT);
        for (int it = max(0, n - 2); it < n; ++it) mbar_wait(bar_q + (it & 1), it >> 1 & 1, one::POLL_LIMIT);
    }
    cp_async_wait<0>();
    __syncthreads();
    // ---- LCE adjoint + store of dV: correlation of dO with the flipped filter ----
    lce_chunk<1, 4, TX, true, ST>(st, sbase + og.off_halo, s_w, nullptr, dm.lce, dVg + head_off / 2, y0, x0, dm.hs, dm, gm, warp, KT, lane);
}

// ------------------------------------------------------------------ host side
static bool one_geom(const Dims& d, DirGeom* gm, OneGeom* og) {
    if (d.d != 32 || d.topk != 1 || d.n_r <= 16 || d.n_r > 64 || d.R > 1024 || (long long)d.H0 * d.W0 * d.C / 8 >= (1ll << 31)) return false;
    DirGeom g = direct_geom(d, d.lce, 4, 1);                          // for the LCE: one chunk, a warp per 16 tokens
    OneGeom o;
    const int kt = (d.n_r + 15) / 16;
    o.arr_bytes = kt * 1024;
    o.p_pitch = kt * 32 + 16;
    o.p_bytes = kt * 16 * o.p_pitch;
    o.box_bytes = (uint32_t)d.n_r * 64;
    const int st_bytes = kt * 16 * one::ST * 4;
    int off = 6 * o.arr_bytes;
    o.off_p = off; off += 2 * o.p_bytes > st_bytes ? 2 * o.p_bytes : st_bytes;
    o.off_halo = off; off += g.halo_bytes;
    const int reach = off + (d.lce ? 3 * g.halo_row + 1024 : 0);     // LCE tiles read (and discard) what is behind the halo
    o.off_w = off; off += d.lce ? 3200 : 0;
    o.off_list = off; off += (d.R * 2 + 15) / 16 * 16;
    o.off_bar = off; off += 32;
    o.smem_bytes = off > reach ? off : reach;
    *gm = g; *og = o;
    return true;
}
bool backward_one_supported(const Dims& d, int dtype) {
    DirGeom g; OneGeom o;
    return dtype == BRA_BF16 && one_geom(d, &g, &o);
}

template <int KT, int TX, OneEdge EDGE>
static cudaError_t launch_edge(const Dims& d, const DirGeom& g, const OneGeom& o, const void* Q, const void* K, const void* V, const int32_t* index,
                            const float* lce_w, const float* lse, const void* dO, void* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st) {
    auto kernel = bwd_one_kernel<KT, TX, EDGE>;
    static PerDeviceMax set;
    const cudaError_t e = set.ensure(o.smem_bytes, [&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, o.smem_bytes); });
    if (e != cudaSuccess) return e;
    CUtensorMap mq, mk, mv, mg;
    const CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_64B;
    if (!make_map(&mq, Q, d, 32, d.ws, d.hs, sw) || !make_map(&mk, K, d, 32, d.ws, d.hs, sw) || !make_map(&mv, V, d, 32, d.ws, d.hs, sw) ||
        !make_map(&mg, dO, d, 32, d.ws, d.hs, sw))
        return cudaErrorInvalidValue;
    typedef __nv_bfloat16 bf;
    return grid_pieces(d, [&](const GridPiece& p) {
        count_launch();
        return launch_kernel(kernel, dim3(p.heads, d.R, p.images), dim3(KT * 32), (size_t)o.smem_bytes, st, false, mq, mk, mv, mg,
                             index + p.index, lse + p.stat, static_cast<const bf*>(dO) + p.tensor, piece_of(lce_w, p.channel * 25),
                             static_cast<bf*>(dQ) + p.tensor, static_cast<bf*>(dK) + p.tensor, static_cast<bf*>(dV) + p.tensor, status, p.h0, p.b0, d, g, o);
    });
}
template <int KT, int TX, typename... Args>
static cudaError_t launch_t(const Dims& d, Args... args) {
    if (d.H != d.H0 || d.W != d.W0) return launch_edge<KT, TX, ONE_CUT>(d, args...);
    if (d.n_r == 16 * KT) return launch_edge<KT, TX, ONE_FULL>(d, args...);
    // (four tiles: the instance that also asks for a cut map keeps everything in registers, this one alone does not)
    return launch_edge<KT, TX, KT == 4 ? ONE_CUT : ONE_REST>(d, args...);
}

cudaError_t launch_backward_one(const Dims& d, const void* Q, const void* K, const void* V, const int32_t* index, const float* lce_w,
                                const float* lse, const void* dO, void* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st) {
    DirGeom g; OneGeom o;
    if (!one_geom(d, &g, &o)) return cudaErrorInvalidConfiguration;
    const int kt = (d.n_r + 15) / 16, tx = lce_tile_width(g, d);
#define BRA_GO(KT, TX) return launch_t<KT, TX>(d, g, o, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, status, st)
#define BRA_GO_TX(KT) do { if (tx == 2) BRA_GO(KT, 2); if (tx == 3) BRA_GO(KT, 3); BRA_GO(KT, 4); } while (0)
    if (kt == 2) BRA_GO_TX(2);
    if (kt == 3) BRA_GO_TX(3);
    BRA_GO_TX(4);
#undef BRA_GO_TX
#undef BRA_GO
}

}  // namespace bra
