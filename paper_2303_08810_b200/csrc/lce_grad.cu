// Gradient of the LCE weights and bias (Eq. 7's depthwise 5 x 5 correlation):
//   d_lce_w[c, i, j] = sum over b, y, x of dO[b, y, x, c] * V[b, y + i - 2, x + j - 2, c],  d_lce_b[c] = sum of dO.
// Per-CTA partial sums, then a fixed-order final sum: results are bit-identical from run to run.
#include "sm100_ptx.cuh"
#include "tma_map.h"

namespace bra {

using namespace ptx;

namespace lg {
constexpr int THREADS = 128;
constexpr int CTAS_PER_SM = 4;
constexpr int SMEM_LIMIT = 55 * 1024;       // four CTAs per SM
constexpr uint32_t POLL_LIMIT = 4000000u;
}  // namespace lg

// A tile is tr x tc positions of one image and one block of channels.
struct LceGradGeom {
    int tr, tc;                // positions of a tile
    int vcols, gcols;          // columns of the V box (tc + 4, perhaps one more) and of the dO box
    int tiles_y, tiles_x, tiles;
    int off_g, off_bar, smem_bytes;
};

template <typename T> struct PairOf;
template <> struct PairOf<float> {
    static __device__ __forceinline__ float2 load(uint32_t a) { return lds_f32x2(a); }
};
template <> struct PairOf<__nv_bfloat16> {
    static __device__ __forceinline__ float2 load(uint32_t a) {
        const uint32_t w = lds_u32(a);
        return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
};

// Thread = (channel pair, row slot): for its row of the tile it slides along x with the 5 x 5 window of V in
// registers, so a position costs six shared-memory reads (five new V values, one dO) and 25 packed FMAs into 25
// sums that never leave the thread.  The tile (V with a border of two, dO) arrives as two bulk tensor copies,
// zero-filled outside the map: no bounds tests, and the addresses are a row base plus constants.
// Bound: the FMA pipe - 25 FMAs per token and channel, a packed FMA every two cycles and scheduler, the reads and
// the unpacking of bf16 pairs in the issue slots between them: 8.6 us at 64 x 56 x 56 x 64.
// Measured (B200): 24 us there, 114 us with a thread per (channel pair, tap row) that read global memory; the same mapping
// without the staged tiles, the window from global memory: 54 - 65 us.
template <typename T, int CB>
__global__ void __launch_bounds__(lg::THREADS, lg::CTAS_PER_SM)
lce_grad_partial_kernel(const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_g,
                        float* __restrict__ part, int32_t* __restrict__ status, LceGradGeom gm, int C) {
    constexpr int TB = CB * (int)sizeof(T);         // bytes of a token in shared memory
    constexpr int PB = CB / 2;                      // channel pairs
    constexpr int SUB = 32 / PB;                    // row slots per warp
    constexpr int SLOTS = lg::THREADS / PB;
    extern __shared__ __align__(128) uint8_t smem[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + gm.off_bar);
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31;
    const int lp = lane % PB, slot = (tid >> 5) * SUB + lane / PB;
    const uint32_t lane_off = lp * 2 * (uint32_t)sizeof(T);

    if (tid == 0) { mbar_init(bar, 1); fence_mbar_init(); }
    __syncthreads();

    float2 acc[25], accb = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 25; ++k) acc[k] = make_float2(0.f, 0.f);
    bool ok = true;
    uint32_t phase = 0;
    for (int tile = blockIdx.x; tile < gm.tiles; tile += gridDim.x) {
        if (tid == 0) {
            const int b = tile / (gm.tiles_y * gm.tiles_x), q = tile - b * (gm.tiles_y * gm.tiles_x);
            const int ty = q / gm.tiles_x, tx = q - ty * gm.tiles_x;
            mbar_expect_tx(bar, (uint32_t)((gm.tr + 4) * gm.vcols + gm.tr * gm.gcols) * TB);
            tma_load_4d(sbase, &map_v, bar, blockIdx.y * CB, tx * gm.tc - 2, ty * gm.tr - 2, b);
            tma_load_4d(sbase + gm.off_g, &map_g, bar, blockIdx.y * CB, tx * gm.tc, ty * gm.tr, b);
        }
        if (!mbar_wait(bar, phase, lg::POLL_LIMIT)) ok = false;
        phase ^= 1;
        if (__syncthreads_or(!ok)) { ok = false; break; }
        for (int r = slot; r < gm.tr; r += SLOTS) {
            uint32_t pv[5];
#pragma unroll
            for (int ti = 0; ti < 5; ++ti) pv[ti] = sbase + (uint32_t)((r + ti) * gm.vcols) * TB + lane_off;
            uint32_t pg = sbase + gm.off_g + (uint32_t)(r * gm.gcols) * TB + lane_off;
            float2 w[5][5];                                 // w[ti][s]: column s of the window ring
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int ti = 0; ti < 5; ++ti) w[ti][s] = PairOf<T>::load(pv[ti] + s * TB);
            auto position = [&](int u) {                    // ring slots u, u + 1, ..., u + 4 hold its window
                const float2 g = PairOf<T>::load(pg + u * TB);
#pragma unroll
                for (int ti = 0; ti < 5; ++ti) w[ti][(u + 4) % 5] = PairOf<T>::load(pv[ti] + (u + 4) * TB);
                accb = __fadd2_rn(accb, g);
#pragma unroll
                for (int ti = 0; ti < 5; ++ti)
#pragma unroll
                    for (int tj = 0; tj < 5; ++tj) acc[ti * 5 + tj] = __ffma2_rn(g, w[ti][(u + tj) % 5], acc[ti * 5 + tj]);
            };
            int x = 0;
            for (; x + 5 <= gm.tc; x += 5) {
#pragma unroll
                for (int u = 0; u < 5; ++u) position(u);
#pragma unroll
                for (int ti = 0; ti < 5; ++ti) pv[ti] += 5 * TB;
                pg += 5 * TB;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (x + u < gm.tc) position(u);
        }
        fence_proxy_async_smem();
        __syncthreads();                                    // read by all: the next tile may take its place
    }
    if (!ok) {
        if (tid == 0) {
            record_error(status, BRA_ERR_TIMEOUT, blockIdx.x);
            mbar_wait(bar, phase ^ 1, lg::POLL_LIMIT);      // nothing in flight when the CTA leaves
        }
        __syncthreads();
        return;
    }

    // row slots added in a fixed order; one partial per CTA, [26][C]
    float2* red = reinterpret_cast<float2*>(smem) + lp;
    if (slot > 0) {
#pragma unroll
        for (int k = 0; k < 25; ++k) red[((slot - 1) * 26 + k) * PB] = acc[k];
        red[((slot - 1) * 26 + 25) * PB] = accb;
    }
    __syncthreads();
    const int c = blockIdx.y * CB + 2 * lp;
    if (slot > 0 || c >= C) return;
#pragma unroll 1
    for (int s = 0; s < SLOTS - 1; ++s) {
#pragma unroll
        for (int k = 0; k < 25; ++k) acc[k] = __fadd2_rn(acc[k], red[(s * 26 + k) * PB]);
        accb = __fadd2_rn(accb, red[(s * 26 + 25) * PB]);
    }
    float* out = part + (size_t)blockIdx.x * 26 * C + c;
#pragma unroll
    for (int k = 0; k < 25; ++k) *reinterpret_cast<float2*>(out + (size_t)k * C) = acc[k];
    *reinterpret_cast<float2*>(out + (size_t)25 * C) = accb;
}

// Final sum over the partials: 32 outputs per CTA, 32 threads per output each taking every
// 32nd partial in order (four loads in flight); the slice sums are then added in order.
constexpr int LG_SLICES = 32;
__global__ void __launch_bounds__(32 * LG_SLICES)
lce_grad_final_kernel(const float* part, int blocks, float* __restrict__ d_lce_w, float* __restrict__ d_lce_b, int C) {
    __shared__ float sl[LG_SLICES][32];
    pdl_wait();
    const int o = blockIdx.x * 32 + threadIdx.x;   // (tap, channel)
    const int slice = threadIdx.y;
    const size_t stride = (size_t)C * 26;
    float s = 0.f;
    if (o < C * 26) {
        int p = slice;
        for (; p + 3 * LG_SLICES < blocks; p += 4 * LG_SLICES) {
            const float a0 = __ldcg(part + (size_t)p * stride + o), a1 = __ldcg(part + (size_t)(p + LG_SLICES) * stride + o);
            const float a2 = __ldcg(part + (size_t)(p + 2 * LG_SLICES) * stride + o), a3 = __ldcg(part + (size_t)(p + 3 * LG_SLICES) * stride + o);
            s += a0; s += a1; s += a2; s += a3;
        }
        for (; p < blocks; p += LG_SLICES) s += __ldcg(part + (size_t)p * stride + o);
    }
    sl[slice][threadIdx.x] = s;
    __syncthreads();
    if (slice == 0 && o < C * 26) {
        float t = sl[0][threadIdx.x];
#pragma unroll
        for (int q = 1; q < LG_SLICES; ++q) t += sl[q][threadIdx.x];
        const int k = o / C, c = o - k * C;
        if (k < 25) { if (d_lce_w) d_lce_w[c * 25 + k] = t; }
        else if (d_lce_b) d_lce_b[c] = t;
    }
}

// ------------------------------------------------------------------ host side
// 64 channels per CTA where they divide C (a warp reads 128 bytes of a token), else 32
static int channel_block(const Dims& d) { return d.esize == 2 && d.C % 64 == 0 ? 64 : 32; }

// Most partials (CTAs per block of channels) a call writes: one wave of the grid.
int lce_grad_partials(const Dims& d) {
    const int groups = (d.C + channel_block(d) - 1) / channel_block(d);
    const int n = kSMs * lg::CTAS_PER_SM / groups;
    return n > 0 ? n : 1;
}

// The tile that leaves the busiest CTA the least to do: positions per row slot, the window's start-up (about six
// positions' worth per row) and the wait for a tile's copies (about ten).
static LceGradGeom lce_grad_geom(const Dims& d) {
    const int cb = channel_block(d), tb = cb * d.esize;
    const int slots = lg::THREADS / (cb / 2);
    const int ctas = lce_grad_partials(d);
    LceGradGeom best = {};
    long long best_cost = -1;
    for (int tr = slots; tr <= 2 * slots; tr += slots) {
        for (int nx = (d.W0 + 39) / 40; nx <= d.W0; ++nx) {
            LceGradGeom g;
            g.tr = tr;
            g.tc = (d.W0 + nx - 1) / nx;
            // two rows per warp: an odd number of columns puts them on different banks
            g.vcols = slots > 4 ? (g.tc + 4) | 1 : g.tc + 4;
            g.gcols = slots > 4 ? g.tc | 1 : g.tc;
            g.off_g = ((g.tr + 4) * g.vcols * tb + 127) / 128 * 128;
            g.off_bar = (g.off_g + g.tr * g.gcols * tb + 127) / 128 * 128;
            const int red = (slots - 1) * 26 * (cb / 2) * 8;
            if (g.off_bar < red) g.off_bar = (red + 127) / 128 * 128;
            g.smem_bytes = g.off_bar + 16;
            if (g.smem_bytes > lg::SMEM_LIMIT || g.vcols > 256) continue;
            g.tiles_x = (d.W0 + g.tc - 1) / g.tc;
            g.tiles_y = (d.H0 + g.tr - 1) / g.tr;
            g.tiles = d.B * g.tiles_y * g.tiles_x;
            const long long cost = (long long)((g.tiles + ctas - 1) / ctas) * (tr / slots * (g.tc + 6) + 10);
            if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = g; }
            if (g.tc <= 4) break;
        }
    }
    return best;
}

template <typename T, int CB>
static cudaError_t launch_partial(const Dims& d, const LceGradGeom& g, int grid_x, const void* V, const void* dO, float* part,
                                  int32_t* status, cudaStream_t st) {
    static PerDeviceMax smem_set;
    cudaError_t e = smem_set.ensure(lg::SMEM_LIMIT, [] {
        cudaError_t a = cudaFuncSetAttribute(lce_grad_partial_kernel<T, CB>, cudaFuncAttributeMaxDynamicSharedMemorySize, lg::SMEM_LIMIT);
        if (a != cudaSuccess) return a;
        return cudaFuncSetAttribute(lce_grad_partial_kernel<T, CB>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    });
    if (e != cudaSuccess) return e;
    CUtensorMap mv, mg;
    if (!make_map(&mv, V, d, CB, g.vcols, g.tr + 4, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map(&mg, dO, d, CB, g.gcols, g.tr, CU_TENSOR_MAP_SWIZZLE_NONE))
        return cudaErrorInvalidValue;
    return launch_kernel(lce_grad_partial_kernel<T, CB>, dim3(grid_x, (d.C + CB - 1) / CB), dim3(lg::THREADS), (size_t)g.smem_bytes,
                         st, false, mv, mg, part, status, g, d.C);
}

cudaError_t launch_lce_grad(const Dims& d, int dtype, const void* V, const void* dO, float* part, float* d_lce_w, float* d_lce_b,
                            int32_t* status, cudaStream_t st) {
    const LceGradGeom g = lce_grad_geom(d);
    const int max_x = lce_grad_partials(d);
    const int grid_x = g.tiles < max_x ? g.tiles : max_x;
    cudaError_t e;
    if (dtype == BRA_F32) e = launch_partial<float, 32>(d, g, grid_x, V, dO, part, status, st);
    else if (channel_block(d) == 64) e = launch_partial<__nv_bfloat16, 64>(d, g, grid_x, V, dO, part, status, st);
    else e = launch_partial<__nv_bfloat16, 32>(d, g, grid_x, V, dO, part, status, st);
    if (e != cudaSuccess) return e;
    count_launch();
    e = launch_kernel(lce_grad_final_kernel, dim3((d.C * 26 + 31) / 32), dim3(32, LG_SLICES), 0, st, true,
                      static_cast<const float*>(part), grid_x, d_lce_w, d_lce_b, d.C);
    count_launch();
    return e;
}

}  // namespace bra
