// Token-to-token attention over the routed regions plus LCE on CUDA cores (Eq. 6, Eq. 7 with Eq. 1), fp32 arithmetic
// throughout (simt_common.cuh has the mapping).  K^g / V^g are never formed: the routing index picks the rows that are
// copied to (or, with a resident slice, read from) shared memory.  Softmax is the one-pass running-max form in blocks of
// four keys per lane.
// Bound: the FMA pipe, 2 D FMAs per query and key (a packed FMA every two cycles and scheduler), in practice the latency of
// the dot-product chains (64 x 28 x 28, 4 heads, topk 4: 0.48 instructions per cycle and scheduler with 7.5 warps per SM, 255 registers).
// Measured (B200) against one thread per query with operands from global memory: 64 x 28 x 28,
// 4 heads, topk 4: 356 -> 144 us; 1 x 16 x 16, 1 head: 41 -> 11 us.
#include "simt_common.cuh"

#include <type_traits>

namespace bra {

using namespace ptx;

// FAR: rows of K and V straight from global memory (simt_far()).
template <typename T, int D, bool FAR>
__global__ void __launch_bounds__(FAR ? 128 : sk::THREADS, FAR ? (D <= 64 ? 3 : 2) : D <= 16 ? 2 : 1)
attend_simt_kernel(const T* __restrict__ Qg, const T* __restrict__ Kg, const T* __restrict__ Vg, const int32_t* index,
                   const float* __restrict__ lce_w, const float* __restrict__ lce_b, T* __restrict__ Og, float* __restrict__ lse,
                   int32_t* __restrict__ status, Dims dm, SimtGeom gm) {
    constexpr int QT = D <= 32 && !FAR ? 2 : 1, U = 4;                // simt_rows()
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x;
    const int h = blockIdx.y, b = blockIdx.z;
    const SimtChunk chunk = simt_chunk(dm, gm, blockIdx.x % gm.chunks);
    const int r0 = blockIdx.x / gm.chunks * gm.rpc;
    const int nreg = min(gm.rpc, dm.R - r0);
    const int N0 = dm.H0 * dm.W0;
    const size_t head = (size_t)b * N0 * dm.C + (size_t)h * D;
    const T* Q = Qg + head; const T* K = Kg + head; const T* V = Vg + head;
    float* s_w = reinterpret_cast<float*>(smem + gm.off_w);
    if (dm.lce) simt_load_weights(s_w, lce_w + (size_t)h * D * 25, 25 * D);
    if (!FAR && gm.resident) {
        simt_zero_rows(smem, gm);
        simt_copy_rows<T, D>(sbase + gm.off_a, sbase + gm.off_b, K, V, dm.C, dm.N, [&](int row, uint32_t& at) {
            const int r = fdiv(row, gm.by_nr);
            at = row * gm.row;
            return simt_token(dm, gm, r, row - r * dm.n_r);
        });
        cp_async_commit();
    }
    pdl_wait();          // in bra_forward the launch may overlap the tail of the routing kernel

    // ---- routing entries: -1 if out of range ----
    const int hi = dm.heads_i == 1 ? 0 : h;
    const int32_t* irow = index + (((size_t)b * dm.heads_i + hi) * dm.R + r0) * dm.topk;
    int32_t* s_idx = reinterpret_cast<int32_t*>(smem + gm.off_idx);
    const bool idx_staged = gm.rpc * dm.topk <= sk::IDX_MAX;
    auto checked = [&](int e) -> int {
        const int r = __ldcg(irow + e);  // coherent load: the index may come from the kernel this one overlaps
        if (r < 0 || r >= dm.R) { record_error(status, BRA_ERR_INDEX, r); return -1; }
        return r;
    };
    bool bad = !idx_staged;                                           // some key may not count
    if (idx_staged) for (int e = tid; e < nreg * dm.topk; e += blockDim.x) { s_idx[e] = checked(e); bad = bad || s_idx[e] < 0; }
    auto entry = [&](int e) -> int { return idx_staged ? s_idx[e] : checked(e); };
    bad = __syncthreads_or(bad);
    bool weighted = false;
    int32_t* cnt = reinterpret_cast<int32_t*>(smem + gm.off_cnt);
    if (!FAR && gm.dense)
        weighted = !simt_counts(cnt, nreg, dm.R, [&](auto add) {
            for (int e = tid; e < nreg * dm.topk; e += blockDim.x)
                if (s_idx[e] >= 0) add(e / dm.topk, s_idx[e]);
        });

    // ---- this lane's rows: QT queries of one region, a share of the keys ----
    const int KS = 1 << gm.ksl, ks = tid & (KS - 1), slot = tid >> gm.ksl;
    const int rl_raw = fdiv(slot, gm.spr, gm.mul_spr);
    const bool active = rl_raw < nreg;
    const int rl = active ? rl_raw : 0;
    const int t0 = active ? QT * (slot - rl_raw * gm.spr) : 0;
    float q[QT][D], o[QT][D], m_run[QT], l_run[QT];
    int tok[QT];
#pragma unroll
    for (int x = 0; x < QT; ++x) {
        tok[x] = active ? simt_row(dm, gm, chunk, r0 + rl, t0 + x) : -1;
        ldg_row<T, D>(q[x], Q + (size_t)(tok[x] < 0 ? 0 : tok[x]) * dm.C, tok[x] >= 0, dm.scale);
        m_run[x] = -INFINITY; l_run[x] = 0.f;
#pragma unroll
        for (int i = 0; i < D; ++i) o[x][i] = 0.f;
    }
    const int total = dm.topk * dm.n_r;

    // keys [k0, k1): rows from offset at0 on, in order (PLAIN), or row_of(kk, dead, wt): offset of the row in shared memory (of
    // zeros if the key does not count) and its weight.  The reference maximum follows the scores only when one lies 16 above it (P and its sums
    // are fp32: any reference gives the same relative precision), so that the sums are seldom rescaled.
    auto walk = [&](auto plain, uint32_t abase, uint32_t at0, int k0, int k1, auto&& row_of) {
        constexpr bool PLAIN = decltype(plain)::value;
        const int blocks = (k1 - k0 + U * KS - 1) / (U * KS);
        [[maybe_unused]] uint32_t next = abase + at0 + ks * gm.row;
#pragma unroll 1
        for (int blk = 0; blk < blocks; ++blk) {
            [[maybe_unused]] uint32_t at[U];
            [[maybe_unused]] int row[U];                              // FAR: token
            bool dead[U];
            float s[QT][U], wt[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int kk = k0 + (blk * U + u) * KS + ks;
                dead[u] = kk >= k1;
                if constexpr (FAR) {
                    row[u] = row_of(kk, dead[u], wt[u]);
                } else if constexpr (PLAIN) {
                    at[u] = dead[u] && gm.resident ? abase + gm.zero : next;
                    next += KS * gm.row;
                } else {
                    wt[u] = 1.f;
                    at[u] = abase + row_of(kk, dead[u], wt[u]);
                }
            }
            if constexpr (FAR) dots_far<T>(s, q, K, row, dm.C);
            else dots<T, QT, U, D>(s, q, at, gm.off_a);
#pragma unroll
            for (int x = 0; x < QT; ++x) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (dead[u]) s[x][u] = -INFINITY;
                const float mx = fmaxf(fmaxf(s[x][0], s[x][1]), fmaxf(s[x][2], s[x][3]));
                if (mx > m_run[x] + 16.f) {                           // always for the first keys that count
                    const float corr = expf(m_run[x] - mx);           // 0 then (m_run = -inf)
                    m_run[x] = mx;
                    l_run[x] *= corr;
#pragma unroll
                    for (int i = 0; i < D; ++i) o[x][i] *= corr;
                }
                const float mn = m_run[x] == -INFINITY ? 0.f : m_run[x];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    s[x][u] = expf(s[x][u] - mn);
                    if (!FAR && !PLAIN && weighted) s[x][u] *= wt[u];
                    l_run[x] += s[x][u];
                }
            }
            if constexpr (FAR) axpy_far<T>(o, s, V, row, dm.C);
            else {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float v[D];
                    lds_row<T, D>(v, at[u] + gm.off_b);
#pragma unroll
                    for (int x = 0; x < QT; ++x) axpy(o[x], s[x][u], v);
                }
            }
        }
    };
    if constexpr (FAR) {
        walk(std::false_type(), 0, 0, 0, total, [&](int kk, bool& dead, float&) -> int {
            if (dead) return -1;
            const int m = fdiv(kk, gm.by_nr), r = entry(rl * dm.topk + m);
            dead = r < 0;
            return dead ? -1 : simt_token(dm, gm, r, kk - m * dm.n_r);        // (-1 in the zero padding: a row of zeros that counts)
        });
    } else {
        const int nst = gm.resident ? 1 : (total + gm.kps - 1) / gm.kps;
        auto load_stage = [&](int st) {
            const uint32_t base = sbase + (st & 1) * gm.stage_bytes;
            simt_copy_rows<T, D>(base + gm.off_a, base + gm.off_b, K, V, dm.C, nreg * gm.kps, [&](int row, uint32_t& at) {
                const int l = fdiv(row, gm.kps, gm.mul_kps), kk = st * gm.kps + row - l * gm.kps;
                at = l * gm.reg + (row - l * gm.kps) * gm.row;
                if (kk >= total) return -1;
                const int m = fdiv(kk, gm.by_nr);
                const int r = entry(l * dm.topk + m);
                return r >= 0 ? simt_token(dm, gm, r, kk - m * dm.n_r) : -1;
            });
            cp_async_commit();
        };
        if (!gm.resident) load_stage(0);
        for (int st = 0; st < nst; ++st) {
            simt_advance(gm, st, nst, load_stage);
            __syncthreads();
            const uint32_t abase = sbase + (st & 1) * gm.stage_bytes;
            const int k0 = gm.resident ? 0 : st * gm.kps;
            if (gm.resident ? gm.dense && !weighted : !bad)
                walk(std::true_type(), abase, gm.resident ? 0 : rl * gm.reg, k0, gm.resident ? dm.N : min(total, k0 + gm.kps), 0);
            else
                walk(std::false_type(), abase, 0, k0, gm.dense ? dm.N : gm.resident ? total : min(total, k0 + gm.kps), [&](int kk, bool& dead, float& wt) -> int {
                    const int none = gm.resident ? gm.zero : rl * gm.reg + (kk - k0) * gm.row;
                    if (dead) return none;
                    const int m = fdiv(kk, gm.by_nr);
                    if (gm.dense) {
                        const int n = cnt[rl * dm.R + m];
                        wt = (float)n;
                        dead = n == 0;
                        return dead ? none : kk * gm.row;
                    }
                    const int r = entry(rl * dm.topk + m);
                    dead = r < 0;
                    return dead || !gm.resident ? none : (r * dm.n_r + kk - m * dm.n_r) * gm.row;
                });
            __syncthreads();
        }
    }

    // ---- merge the key shares; normalise; stage; lse ----
#pragma unroll
    for (int x = 0; x < QT; ++x) {
        float m = m_run[x];
        for (int off = 1; off < KS; off <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        float f = KS == 1 || m == -INFINITY ? 1.f : expf(m_run[x] - m), l = l_run[x] * f;
        for (int off = 1; off < KS; off <<= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        f *= l > 0.f ? 1.0f / l : 0.f;
#pragma unroll
        for (int i = 0; i < D; ++i) o[x][i] *= f;
        if (lse && tok[x] >= 0 && ks == 0) lse[((size_t)b * dm.heads + h) * N0 + tok[x]] = m + logf(l);
    }
    int first, held;
    sum_shares<QT, D>(o, gm.ksl, ks, &first, &held);
    __syncthreads();
    float* st = reinterpret_cast<float*>(smem + gm.off_st);
    if (active)
        for_held<QT, D>(o, first, held, [&](int x, int c, const float4& v) {
            *reinterpret_cast<float4*>(st + (rl * QT * gm.spr + t0 + x) * (D + 4) + c) = v;
        });
    __syncthreads();
    const float* bias = dm.lce && lce_b ? lce_b + h * D : nullptr;
    if (FAR ? dm.n_r == 1 : dm.hs <= 2) simt_lce<T, D, FAR ? 1 : 2, false>(st, s_w, bias, V, Og + head, SimtFrom{r0}, nreg, QT * gm.spr, chunk, dm, gm);
    else simt_lce<T, D, FAR ? 2 : 4, false>(st, s_w, bias, V, Og + head, SimtFrom{r0}, nreg, QT * gm.spr, chunk, dm, gm);
}

bool attend_simt_supported(const Dims& d) {
    return (d.d == 16 || d.d == 32 || d.d == 64 || d.d == 128) && simt_fits(d, SIMT_ATTEND);
}

template <typename T, int D, bool FAR>
static cudaError_t launch_t(const Dims& d, const void* Q, const void* K, const void* V,
                            const int32_t* index, const float* lce_w, const float* lce_b,
                            void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel, const SimtGeom& g) {
    static PerDeviceMax smem_set;
    if (g.smem_bytes > 48 * 1024) {
        const cudaError_t e = smem_set.ensure(g.smem_bytes, [&] {
            return cudaFuncSetAttribute(attend_simt_kernel<T, D, FAR>, cudaFuncAttributeMaxDynamicSharedMemorySize, g.smem_bytes);
        });
        if (e != cudaSuccess) return e;
    }
    return grid_pieces(d, [&](const GridPiece& p) {
        count_launch();
        return launch_kernel(attend_simt_kernel<T, D, FAR>, dim3(g.gpi, p.heads, p.images), dim3(g.threads), (size_t)g.smem_bytes, st, after_own_kernel,
                             static_cast<const T*>(Q) + p.tensor, static_cast<const T*>(K) + p.tensor, static_cast<const T*>(V) + p.tensor,
                             index + p.index, piece_of(lce_w, p.channel * 25), piece_of(lce_b, p.channel), static_cast<T*>(O) + p.tensor,
                             piece_of(lse, p.stat), status, d, g);
    });
}

template <typename T>
static cudaError_t launch_d(const Dims& d, const void* Q, const void* K, const void* V,
                            const int32_t* index, const float* lce_w, const float* lce_b,
                            void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    const SimtGeom g = simt_geom(d, SIMT_ATTEND);
#define BRA_GO(D)                                                                                                                     \
    case D: return g.far ? launch_t<T, D, true>(d, Q, K, V, index, lce_w, lce_b, O, lse, status, st, after_own_kernel, g)             \
                         : launch_t<T, D, false>(d, Q, K, V, index, lce_w, lce_b, O, lse, status, st, after_own_kernel, g)
    switch (d.d) { BRA_GO(16); BRA_GO(32); BRA_GO(64); BRA_GO(128); }
#undef BRA_GO
    return cudaErrorInvalidValue;
}

cudaError_t launch_attend_simt(const Dims& d, int dtype, const void* Q, const void* K, const void* V,
                               const int32_t* index, const float* lce_w, const float* lce_b,
                               void* O, float* lse, int32_t* status, cudaStream_t st, bool after_own_kernel) {
    if (dtype == BRA_BF16)
        return launch_d<__nv_bfloat16>(d, Q, K, V, index, lce_w, lce_b, O, lse, status, st, after_own_kernel);
    return launch_d<float>(d, Q, K, V, index, lce_w, lce_b, O, lse, status, st, after_own_kernel);
}

}  // namespace bra
