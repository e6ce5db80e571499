// Internal declarations shared by the translation units of the BRA library.
// Nothing here is part of the C boundary (include/bra.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>
#include <stdlib.h>

#include <mutex>

#include "../../include/bra.h"

namespace bra {

// Problem with every derived quantity the kernels need, passed by value.
struct Dims {
    int B, H, W, C, heads, S, topk;
    int d;        // C / heads
    int R;        // S * S regions
    int hs, ws;   // region height / width in tokens
    int n_r;      // hs * ws tokens per region
    int N;        // H * W tokens per image
    int heads_i;  // heads of the routing index: heads, or 1 with shared routing
    int lce;      // 1: add LCE
    float scale;  // softmax scale (Eq. 1)
    // When S does not divide the caller's map, H and W above are the padded sizes (next multiples of S) and these
    // the sizes of the map in memory.  Kernels that take any map address it by H0, W0 and read zeros outside; the
    // others are given a padded copy and H0 = H, W0 = W.
    int H0, W0;
    int esize;    // bytes per element of Q, K, V, O
};

// A launch covers at most GRID_YZ heads, images or groups of regions (grid extents in y and z end at 65535, one row to spare);
// larger problems are launched piece by piece, every piece with pointers to its first head and image.
constexpr int GRID_YZ = 65534;
struct GridPiece {
    int heads, images;
    size_t tensor;      // elements from the start of Q, K, V, O and their gradients
    size_t index;       // entries from the start of the routing index
    size_t stat;        // floats from the start of lse and delta
    size_t channel;     // channels from the start of the LCE weights and bias
    int h0, b0;
};
template <typename F>
inline cudaError_t grid_pieces(const Dims& d, F&& launch) {
    for (int h0 = 0; h0 < d.heads; h0 += GRID_YZ)
        for (int b0 = 0; b0 < d.B; b0 += GRID_YZ) {
            GridPiece p;
            p.h0 = h0; p.b0 = b0;
            p.heads = d.heads - h0 < GRID_YZ ? d.heads - h0 : GRID_YZ;
            p.images = d.B - b0 < GRID_YZ ? d.B - b0 : GRID_YZ;
            p.channel = (size_t)h0 * d.d;
            p.tensor = (size_t)b0 * d.H0 * d.W0 * d.C + p.channel;
            p.index = ((size_t)b0 * d.heads_i + (d.heads_i == 1 ? 0 : h0)) * d.R * d.topk;
            p.stat = ((size_t)b0 * d.heads + h0) * d.H0 * d.W0;
            const cudaError_t e = launch(p);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}
template <typename T>
inline T* piece_of(T* p, size_t n) { return p ? p + n : nullptr; }

// Lists of the inverse routing index cut in parts (the dK / dV kernel of backward_direct.cu): a job is a key region and a part of at
// most `most` entries of its list, so that no CTA has much more to do than the others, however few regions hold most of the
// index.  Every part of a region that has several leaves its sums in scratch memory; the one that finishes last adds them up,
// in the order of the parts.  Jobs by falling length of their regions' lists: those of cut lists come first, and number their sums.
struct ListParts {
    int most;               // entries of a part; 0: lists are not cut
    int jobs, cut;          // jobs of an (image, routing head) and, of those, parts of cut lists, at most
    bool even;              // the parts of a list are of one length; else the last one has what is left
};

// Scratch layout (byte offsets from ws, all multiples of 256).
struct WsLayout {
    size_t status;      // int32[64]: [0] first device error, [1] detail
    size_t q_mean;      // fp32 [B,R,C]
    size_t k_mean;      // fp32 [B,R,C]
    size_t index;       // int32 [B,heads_i,R,topk] (bra_forward with index == NULL)
    size_t delta;       // fp32 [B,heads,N]  rowsum(P o dP) of the backward pass
    size_t inv_off;     // int32 [B,heads_i,R+1] CSR offsets of the inverse routing index
    size_t inv_list;    // int32 [B,heads_i,R*topk] query regions routed to each key region
    size_t inv_order;   // int32 [B,heads_i,R] key regions by falling length of their lists
    size_t jobs;        // int2 [B,heads_i,parts.jobs] key regions and parts of their lists
    size_t done;        // int32 [B,heads,R,chunks] parts of a region's list that are done
    size_t sums;        // fp32 dK and dV of the parts of cut lists, by job and tile
    size_t dw_part;     // fp32 [lce_grad_partials(d), 26*C] partial LCE weight / bias gradients
    size_t pad;         // padded maps only: seven [B,H,W,C] tensors of the padded size (Q, K, V, O / dO, dQ, dK, dV)
    size_t pad_lse;     // padded maps only: fp32 [B,heads,H*W] of the padded size
    size_t pad_tensor;  // bytes of one padded tensor
    size_t total;
};

constexpr int kSMs = 148;      // B200

WsLayout ws_layout(const Dims& d);

// Host-side bookkeeping of kernel launches for bra_last_launch_count().
void count_launch(int n = 1);
void reset_launch_count();

// Validate a problem statement and fill the derived dimensions.
bra_status check_problem(const bra_problem* p, Dims* out);

// ---- kernel launchers (each returns the cudaError of its launches) ----------
// Copies between the caller's [B,H0,W0,C] map and the zero-padded [B,H,W,C] map the kernels work on
// (to_padded: fill; else crop).  elem_bytes: bytes of one token (C * element size; a multiple of 4).
cudaError_t launch_pad_copy(const void* src, void* dst, long long images, int H0, int W0, int H, int W,
                            int token_bytes, bool to_padded, cudaStream_t st);
cudaError_t launch_pool(const Dims& d, int dtype, const void* Q, const void* K,
                        float* q_mean, float* k_mean, cudaStream_t st);
cudaError_t launch_route(const Dims& d, const float* q_mean, const float* k_mean,
                         int32_t* index, cudaStream_t st);
// true if this build has a routing kernel for the problem
bool route_supported(const Dims& d);

bool attend_simt_supported(const Dims& d);
cudaError_t launch_attend_simt(const Dims& d, int dtype, const void* Q, const void* K, const void* V,
                               const int32_t* index, const float* lce_w, const float* lce_b,
                               void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel);

bool attend_direct_supported(const Dims& d, int dtype);
cudaError_t launch_attend_direct(const Dims& d, const void* Q, const void* K, const void* V,
                              const int32_t* index, const float* lce_w, const float* lce_b,
                              void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel);

// after_own_kernel (here and below): the kernel before this one in the stream is the library's own
// routing kernel, so the launch may overlap its tail (programmatic dependent launch)
bool attend_tc_supported(const Dims& d, int dtype);
cudaError_t launch_attend_tc(const Dims& d, const void* Q, const void* K, const void* V,
                             const int32_t* index, const float* lce_w, const float* lce_b,
                             void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel);

// Algorithm 1 in one launch (pooling, routing and attention of 8 x 8-token regions, topk = 1)
bool forward_tc_supported(const Dims& d, int dtype);
cudaError_t launch_forward_tc(const Dims& d, const void* Q, const void* K, const void* V,
                              const float* lce_w, const float* lce_b, void* O, int32_t* index, float* lse,
                              float* q_mean, float* k_mean, int32_t* ctrl, int inject, cudaStream_t st);

bool attend_img_supported(const Dims& d, int dtype);
cudaError_t launch_attend_img(const Dims& d, const void* Q, const void* K, const void* V,
                              const int32_t* index, const float* lce_w, const float* lce_b,
                              void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel);
// Small maps, every token a key (index NULL: every query attends to every region once)
bool attend_dense_supported(const Dims& d, int dtype);
cudaError_t launch_attend_dense(const Dims& d, const void* Q, const void* K, const void* V,
                                const int32_t* index, const float* lce_w, const float* lce_b,
                                void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel);
// true if the dense kernels are the faster ones: they walk all tokens of the map for 16 queries at a time, the routed ones
// topk regions for a tile of one region, n_r of whose 16 rows are used.  Measured (B200, us, dense / direct).
// Above 64 tokens a CTA's walk is long and wants (image, head) pairs to fill the GPU.  14 x 14, 49 regions, topk 16: attention
// 64 pairs 10.6 / 14.6, 32 pairs 14 / 8; gradients 296 pairs 54 / 94, 128 pairs 53 / 46.
inline bool dense_fewer_rows(const Dims& d) { return (long long)d.N < (long long)d.topk * ((d.n_r + 15) / 16 * 16); }
inline bool dense_grad_pays(const Dims& d) {
    return dense_fewer_rows(d) && (d.N <= 64 || (long long)d.B * d.heads >= 2 * kSMs);   // up to 64 tokens, 4 pairs, topk 8: 11.2 / 12.0
}
// Up to 64 tokens: the direct kernel has a warp per region and is the faster one while they fit on the GPU at once (12 per SM):
// 7 x 7, topk 16: 16 pairs 8.2 / 6.2, 32 pairs 8.2 / 6.9, 48 pairs 8.3 / 11.2; 8 x 8, 2 x 2 regions, topk 8: 96 pairs 7.1 / 7.1,
// 192 pairs 7.6 / 12.2.  With every region on every list bra_forward has nothing to route for the dense kernel (7 x 7, topk 49,
// 16 pairs: 5.8 against 13 us), and bra_attend, whose results are the same bit for bit, takes it too (10.8 / 7.0).
inline bool dense_pays(const Dims& d) {
    const long long pairs = (long long)d.B * d.heads;
    if (!dense_fewer_rows(d)) return false;
    return d.N > 64 ? pairs >= 64 : d.topk == d.R || pairs * d.R * ((d.n_r + 15) / 16) > 12 * kSMs;
}
// true if the kernels with one CTA per (image, head) are: they are written for regions of 2 x 2 and 4 x 4 tokens (5 x 5, topk 6,
// 25 x 25, 256 pairs: attention 111 against 70 us, gradients 244 / 163; 3 x 3, topk 9: 59 / 33, 93 / 69), fill the GPU in waves of 148
// and, with a whole SM each, start only when the routing kernel is done.  bra_forward, resident / direct: 28 x 28, topk 4: 144 pairs
// 46.7 / 38.9, 160 46.8 / 41.1, 200 49.7 / 50.7, 256 49.7 / 58.1; 20 x 20, S = 5, topk 6: 160 29.7 / 26.8, 200 30.2 / 34.3; 14 x 14: topk 4,
// 256 pairs 47.5 / 42.1, 320 49.7 / 52.7, topk 12, 200 43.6 / 46.1.  The work: the blocks of 32 keys that the direct kernel walks.
// On the wrong side of it: 16 x 16, S = 8, topk 8, 256 pairs 62.9 / 53.3 and 20 x 20, S = 10, topk 8, 160 pairs 62.9 / 65.2.
// (Attention alone: 28 x 28 144 pairs 30.0 / 31.5; 32 x 32, S = 8, topk 4, 128 pairs 28.5 / 33.4, bra_forward 35.5 / 39.7.)
inline bool img_regions(const Dims& d) { return d.hs == d.ws && (d.hs == 2 || d.hs == 4); }
inline bool img_pays(const Dims& d) {
    const long long pairs = (long long)d.B * d.heads;
    return img_regions(d) && pairs >= 190 && pairs * d.R * ((d.topk * d.n_r + 31) / 32) >= 15000;
}
// Gradients: 28 x 28, topk 4: 144 pairs 57.5 / 58.6, 200 95 / 79, 256 99 / 103; 14 x 14, topk 8: 160 pairs 62 / 49, 256 65 / 72.
inline bool img_grad_pays(const Dims& d) { return img_regions(d) && (long long)d.B * d.heads >= 237; }
bool backward_dense_supported(const Dims& d, int dtype);
cudaError_t launch_backward_dense(const Dims& d, const void* Q, const void* K, const void* V, const int32_t* index, const float* lce_w,
                                  const float* lse, const void* dO, void* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st);
bool attend_tc_wide_supported(const Dims& d, int dtype);
cudaError_t launch_attend_tc_wide(const Dims& d, const void* Q, const void* K, const void* V,
                                  const int32_t* index, const float* lce_w, const float* lce_b,
                                  void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel);

bool backward_direct_supported(const Dims& d, int dtype);
// How it cuts lists; chunks: groups of a region, sum_bytes: what the parts of cut lists of the whole problem leave in scratch memory.
ListParts direct_grad_parts(const Dims& d, int* chunks, size_t* sum_bytes);
cudaError_t launch_backward_direct(const Dims& d, const void* Q, const void* K, const void* V, const int32_t* index, char* ws, const WsLayout& L,
                                const float* lce_w, const float* lse, const void* dO, void* dQ, void* dK, void* dV, cudaStream_t st);

bool backward_one_supported(const Dims& d, int dtype);
// It walks a list from end to end in one CTA, where the direct kernels cut long ones.  More regions make longer lists where a few kinds
// of content share them, and only many (image, head) pairs hide one.  Measured (B200, us, one launch / direct), evenly spread and
// clustered: 64 regions, 1 x 64 x 64, 2 heads 12 / 18 and 35 / 27, 8 images 27 / 35 and 51 / 42; 81 regions of 64, 4 pairs 17 / 24 and
// 45 / 32, 16 pairs 32 / 40 and 62 / 46, 32 pairs 52 / 71 and 82 / 74, 64 pairs 96 / 145 and 120 / 142; 256 regions of 49, 4 pairs 32 / 39 and
// 116 / 46, 16 pairs 77 / 106 and 173 / 108, 32 pairs 147 / 212 and 239 / 203, 64 pairs 272 / 428 and 365 / 393.
inline bool one_grad_pays(const Dims& d) { return d.R <= 64 || (long long)d.B * d.heads >= 32; }
cudaError_t launch_backward_one(const Dims& d, const void* Q, const void* K, const void* V, const int32_t* index, const float* lce_w,
                                const float* lse, const void* dO, void* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st);

bool backward_img_supported(const Dims& d, int dtype);
cudaError_t launch_backward_img(const Dims& d, const void* Q, const void* K, const void* V,
                                const int32_t* index, const int32_t* inv_off, const int32_t* inv_list,
                                const float* lce_w, const float* lse, const void* dO,
                                void* dQ, void* dK, void* dV, float* delta, int32_t* status, cudaStream_t st);

// A process may drive several GPUs, and kernel attributes are per device: the largest value already
// set for a kernel on the CURRENT device (dynamic shared-memory size, or 1 for "set-up done").  The
// set-up runs under a lock and is recorded only once it has succeeded, so concurrent host threads
// never launch before the attribute exists and a failed set-up is tried again.
struct PerDeviceMax {
    std::mutex lock;
    int v[64] = {};
    template <typename F>
    cudaError_t ensure(int want, F&& set) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return set();
        std::lock_guard<std::mutex> guard(lock);
        if (want <= v[dev]) return cudaSuccess;
        const cudaError_t e = set();
        if (e == cudaSuccess) v[dev] = want;
        return e;
    }
};
struct PerDeviceOnce {
    PerDeviceMax m;
    template <typename F>
    cudaError_t run(F&& set) { return m.ensure(1, set); }
};

// A helper stream per device and host thread, forked from and joined back into the caller's stream with
// events (created on first use; nullptr if that fails or BRA_NO_SIDE_STREAM is set: then the work stays in
// order on the caller's stream).
struct SideStream { cudaStream_t s; cudaEvent_t fork, join; };
SideStream* side_stream();

// Gradient of the LCE weights and bias from V and dO (part: lce_grad_partials(d) x 26 C floats of scratch).
int lce_grad_partials(const Dims& d);
cudaError_t launch_lce_grad(const Dims& d, int dtype, const void* V, const void* dO, float* part, float* d_lce_w, float* d_lce_b,
                            int32_t* status, cudaStream_t st);

bool backward_supported(const Dims& d, int dtype, int impl);
// true if the kernels launch_backward() takes for this problem work on maps that S does not divide
bool backward_any_map(const Dims& d, int dtype, int impl);
// impl: the bra_impl the caller asked for
cudaError_t launch_backward(const Dims& d, int dtype, int impl, const void* Q, const void* K, const void* V,
                            const int32_t* index, const float* lce_w, const float* lse,
                            const void* dO, void* dQ, void* dK, void* dV,
                            float* d_lce_w, float* d_lce_b,
                            char* ws, const WsLayout& L, cudaStream_t st);

// ---- device helpers -----------------------------------------------------------
#ifdef __CUDACC__
// Programmatic dependent launch: a kernel launched with launch_kernel(..., after_own_kernel = true)
// may start while the kernel before it in the stream is still running; pdl_wait() returns once
// that kernel has completed and its writes are visible (a no-op for an ordinary launch).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 bool after_own_kernel, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    static const bool pdl_off = getenv("BRA_NO_PDL") != nullptr;   // debugging aid: plain stream order
    cfg.numAttrs = (after_own_kernel && !pdl_off) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

__device__ __forceinline__ void record_error(int32_t* status, int code, int detail) {
    if (atomicCAS(status, 0, code) == 0) status[1] = detail;
}

// Load `n` consecutive elements (n multiple of 8 for bf16 / 4 for fp32, 16-byte aligned) as fp32.
template <int n>
__device__ __forceinline__ void load_row(const float* __restrict__ p, float* out) {
#pragma unroll
    for (int i = 0; i < n; i += 4) {
        float4 v = __ldg(reinterpret_cast<const float4*>(p + i));
        out[i] = v.x; out[i + 1] = v.y; out[i + 2] = v.z; out[i + 3] = v.w;
    }
}
template <int n>
__device__ __forceinline__ void load_row(const __nv_bfloat16* __restrict__ p, float* out) {
#pragma unroll
    for (int i = 0; i < n; i += 8) {
        uint4 v = __ldg(reinterpret_cast<const uint4*>(p + i));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            out[i + 2 * j] = __uint_as_float(w[j] << 16);
            out[i + 2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
        }
    }
}
template <int n>
__device__ __forceinline__ void store_row(float* p, const float* v) {
#pragma unroll
    for (int i = 0; i < n; i += 4)
        *reinterpret_cast<float4*>(p + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
}
template <int n>
__device__ __forceinline__ void store_row(__nv_bfloat16* p, const float* v) {
#pragma unroll
    for (int i = 0; i < n; i += 8) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[i + 2 * j], v[i + 2 * j + 1]);
            w[j] = *reinterpret_cast<uint32_t*>(&h);
        }
        *reinterpret_cast<uint4*>(p + i) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
#endif  // __CUDACC__

}  // namespace bra
