// Gradients of O = softmax(scale Q K^g^T) V^g + LCE(V) for a fixed routing index (Eq. 7 with Eq. 1; the index of Eq. 5 is
// a constant): choice of the kernels, and the kernels with fp32 arithmetic on CUDA cores (simt_common.cuh has their
// mapping).  Every sum has a fixed order: no atomics on the data path.
//
//   1. inverse index (inverse_index.cuh): for each key region, the list (in (query region, slot) order) of query regions
//      that routed to it, as CSR; built by extra CTAs of the dQ launch.
//   2. dQ kernel: delta = rowsum(P o dP) in a first walk over the keys, dQ = scale * sum_j P_j (dP_j - delta) K_j in a
//      second; delta is kept for step 3.
//   3. dK/dV kernel: rows are keys, the walk goes over the queries of the regions on the key region's list; P from the
//      saved log-sum-exp; then the LCE adjoint dV += sum_ij w[c,i,j] dO[y-i+2, x-j+2, c].
//   4. d_lce_w / d_lce_b: lce_grad.cu.
// Steps 1 to 3 run on the tensor cores instead (backward_one.cu, backward_dense.cu, backward_img.cu, backward_direct.cu) for bf16 with head
// dim 32 or 64.
#include "inverse_index.cuh"
#include "simt_common.cuh"

#include <type_traits>

namespace bra {

using namespace ptx;

// ------------------------------------------------------------ dQ and delta
// Grid row 0 builds the inverse index, row 1 + h is head h.
template <typename T, int D>
__global__ void __launch_bounds__(sk::THREADS, 1)
bwd_dq_simt_kernel(const T* __restrict__ Qg, const T* __restrict__ Kg, const T* __restrict__ Vg, const int32_t* __restrict__ index,
                   const float* __restrict__ lse, const T* __restrict__ dOg, T* __restrict__ dQg, float* __restrict__ delta,
                   int32_t* __restrict__ inv_off, int32_t* __restrict__ inv_list, int32_t* __restrict__ inv_order, bool inv_bits,
                   int32_t* __restrict__ status, Dims dm, SimtGeom gm) {
    constexpr int QT = D <= 32 ? 2 : 1, U = 2;                        // simt_rows()
    extern __shared__ __align__(128) uint8_t smem[];
    if (blockIdx.y == 0) {
        if (inv_off && (int)blockIdx.x < dm.heads_i)
            inverse_index_job(index, inv_off, inv_list, inv_order, blockIdx.z * dm.heads_i + blockIdx.x, reinterpret_cast<int32_t*>(smem), inv_bits, dm);
        return;
    }
    if ((int)blockIdx.x >= gm.gpi) return;
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x;
    const int h = blockIdx.y - 1, b = blockIdx.z;
    const SimtChunk chunk = simt_chunk(dm, gm, blockIdx.x % gm.chunks);
    const int r0 = blockIdx.x / gm.chunks * gm.rpc;
    const int nreg = min(gm.rpc, dm.R - r0);
    const int N0 = dm.H0 * dm.W0;
    const size_t head = (size_t)b * N0 * dm.C + (size_t)h * D;
    const T* K = Kg + head; const T* V = Vg + head;
    if (gm.resident) {
        simt_zero_rows(smem, gm);
        simt_copy_rows<T, D>(sbase + gm.off_a, sbase + gm.off_b, K, V, dm.C, dm.N, [&](int row, uint32_t& at) {
            const int r = fdiv(row, gm.by_nr);
            at = row * gm.row;
            return simt_token(dm, gm, r, row - r * dm.n_r);
        });
        cp_async_commit();
    }
    const int hi = dm.heads_i == 1 ? 0 : h;
    const int32_t* irow = index + (((size_t)b * dm.heads_i + hi) * dm.R + r0) * dm.topk;
    int32_t* s_idx = reinterpret_cast<int32_t*>(smem + gm.off_idx);
    const bool idx_staged = gm.rpc * dm.topk <= sk::IDX_MAX;
    auto checked = [&](int e) -> int {
        const int r = __ldg(irow + e);
        if (r < 0 || r >= dm.R) { record_error(status, BRA_ERR_INDEX, r); return -1; }
        return r;
    };
    bool bad = !idx_staged;
    if (idx_staged) for (int e = tid; e < nreg * dm.topk; e += blockDim.x) { s_idx[e] = checked(e); bad = bad || s_idx[e] < 0; }
    auto entry = [&](int e) -> int { return idx_staged ? s_idx[e] : checked(e); };
    bad = __syncthreads_or(bad);
    bool weighted = false;
    int32_t* cnt = reinterpret_cast<int32_t*>(smem + gm.off_cnt);
    if (gm.dense)
        weighted = !simt_counts(cnt, nreg, dm.R, [&](auto add) {
            for (int e = tid; e < nreg * dm.topk; e += blockDim.x)
                if (s_idx[e] >= 0) add(e / dm.topk, s_idx[e]);
        });

    const int KS = 1 << gm.ksl, ks = tid & (KS - 1), slot = tid >> gm.ksl;
    const int rl_raw = fdiv(slot, gm.spr, gm.mul_spr);
    const bool active = rl_raw < nreg;
    const int rl = active ? rl_raw : 0;
    const int t0 = active ? QT * (slot - rl_raw * gm.spr) : 0;
    float q[QT][D], go[QT][D], acc[QT][D], l[QT], dsum[QT];
    int tok[QT];
    const float* lse_h = lse + ((size_t)b * dm.heads + h) * N0;
#pragma unroll
    for (int x = 0; x < QT; ++x) {
        tok[x] = active ? simt_row(dm, gm, chunk, r0 + rl, t0 + x) : -1;
        const size_t at = head + (size_t)(tok[x] < 0 ? 0 : tok[x]) * dm.C;
        ldg_row<T, D>(q[x], Qg + at, tok[x] >= 0, dm.scale);
        ldg_row<T, D>(go[x], dOg + at, tok[x] >= 0, 1.f);
        l[x] = tok[x] >= 0 ? __ldg(lse_h + tok[x]) : 0.f;
        dsum[x] = 0.f;
#pragma unroll
        for (int i = 0; i < D; ++i) acc[x][i] = 0.f;
    }
    const int total = dm.topk * dm.n_r;
    auto walk = [&](auto plain, uint32_t abase, uint32_t at0, int k0, int k1, bool second, auto&& row_of) {
        constexpr bool PLAIN = decltype(plain)::value;
        const int blocks = (k1 - k0 + U * KS - 1) / (U * KS);
        uint32_t next = abase + at0 + ks * gm.row;
#pragma unroll 1
        for (int blk = 0; blk < blocks; ++blk) {
            uint32_t at[U];
            bool dead[U];
            float s[QT][U], dp[QT][U], wt[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int kk = k0 + (blk * U + u) * KS + ks;
                dead[u] = kk >= k1;
                if constexpr (PLAIN) {
                    at[u] = dead[u] && gm.resident ? abase + gm.zero : next;
                    next += KS * gm.row;
                } else {
                    wt[u] = 1.f;
                    at[u] = abase + row_of(kk, dead[u], wt[u]);
                }
            }
            dots<T, QT, U, D>(s, q, at, gm.off_a);
            dots<T, QT, U, D>(dp, go, at, gm.off_b);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int x = 0; x < QT; ++x) {
                    s[x][u] = dead[u] ? 0.f : expf(s[x][u] - l[x]);
                    if (!PLAIN && weighted) s[x][u] *= wt[u];
                    if (!second) dsum[x] = fmaf(s[x][u], dp[x][u], dsum[x]);
                    else s[x][u] *= dp[x][u] - dsum[x];
                }
            if (!second) continue;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float k[D];
                lds_row<T, D>(k, at[u] + gm.off_a);
#pragma unroll
                for (int x = 0; x < QT; ++x) axpy(acc[x], s[x][u], k);
            }
        }
    };
    auto end_of_first = [&]() {
        for (int off = 1; off < KS; off <<= 1)
#pragma unroll
            for (int x = 0; x < QT; ++x) dsum[x] += __shfl_xor_sync(0xffffffffu, dsum[x], off);
    };
    const int nst = gm.resident ? 1 : (total + gm.kps - 1) / gm.kps;
    auto load_stage = [&](int it) {
        const int st = it < nst ? it : it - nst;
        const uint32_t base = sbase + (it & 1) * gm.stage_bytes;
        simt_copy_rows<T, D>(base + gm.off_a, base + gm.off_b, K, V, dm.C, nreg * gm.kps, [&](int row, uint32_t& at) {
            const int lr = fdiv(row, gm.kps, gm.mul_kps), kk = st * gm.kps + row - lr * gm.kps;
            at = lr * gm.reg + (row - lr * gm.kps) * gm.row;
            if (kk >= total) return -1;
            const int m = fdiv(kk, gm.by_nr);
            const int r = entry(lr * dm.topk + m);
            return r >= 0 ? simt_token(dm, gm, r, kk - m * dm.n_r) : -1;
        });
        cp_async_commit();
    };
    if (!gm.resident) load_stage(0);
    for (int it = 0; it < 2 * nst; ++it) {
        simt_advance(gm, it, gm.resident ? 0 : 2 * nst, load_stage);
        __syncthreads();
        const int k0 = gm.resident ? 0 : (it < nst ? it : it - nst) * gm.kps;
        const uint32_t abase = sbase + (it & 1) * gm.stage_bytes;
        if (gm.resident ? gm.dense && !weighted : !bad)
            walk(std::true_type(), abase, gm.resident ? 0 : rl * gm.reg, k0, gm.resident ? dm.N : min(total, k0 + gm.kps), it >= nst, 0);
        else
            walk(std::false_type(), abase, 0, k0, gm.dense ? dm.N : gm.resident ? total : min(total, k0 + gm.kps), it >= nst, [&](int kk, bool& dead, float& wt) -> int {
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
        if (it == nst - 1) end_of_first();
        __syncthreads();
    }
    int first, held;
    sum_shares<QT, D>(acc, gm.ksl, ks, &first, &held);
    pdl_launch_dependents();
    if (!active) return;
    for_held<QT, D>(acc, first, held, [&](int x, int c, const float4& v) {
        const int tk = QT == 2 && x == 1 ? tok[QT - 1] : tok[0];
        if (tk >= 0) store4(dQg + head + (size_t)tk * dm.C + c, make_float4(v.x * dm.scale, v.y * dm.scale, v.z * dm.scale, v.w * dm.scale));
    });
#pragma unroll
    for (int x = 0; x < QT; ++x)
        if (tok[x] >= 0 && ks == 0) delta[((size_t)b * dm.heads + h) * N0 + tok[x]] = dsum[x];
}

// ------------------------------------------------------------ dK, dV
template <typename T, int D>
__global__ void __launch_bounds__(sk::THREADS, 1)
bwd_dkv_simt_kernel(const T* __restrict__ Qg, const T* __restrict__ Kg, const T* __restrict__ Vg, const int32_t* inv_off,
                    const int32_t* inv_list, const int32_t* inv_order, const float* __restrict__ lse, const float* delta, const T* __restrict__ dOg,
                    const float* __restrict__ lce_w, T* __restrict__ dKg, T* __restrict__ dVg, Dims dm, SimtGeom gm) {
    constexpr int SPLIT = D > 32 ? 1 : 0, DL = D >> SPLIT;            // simt_split(); channels of a lane
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x;
    const int h = blockIdx.x, b = blockIdx.y;                         // longest lists of all (image, head) pairs first
    const SimtChunk chunk = simt_chunk(dm, gm, blockIdx.z % gm.chunks);
    const int r0 = blockIdx.z / gm.chunks * gm.rpc;                   // regions r0 .. of the order
    const int nreg = min(gm.rpc, dm.R - r0);
    const int N0 = dm.H0 * dm.W0;
    const size_t head = (size_t)b * N0 * dm.C + (size_t)h * D;
    const T* Q = Qg + head; const T* dO = dOg + head;
    float* s_w = reinterpret_cast<float*>(smem + gm.off_w);
    if (dm.lce) simt_load_weights(s_w, lce_w + (size_t)h * D * 25, 25 * D);
    if (gm.resident) {
        simt_zero_rows(smem, gm);
        simt_copy_rows<T, D>(sbase + gm.off_a, sbase + gm.off_b, Q, dO, dm.C, dm.N, [&](int row, uint32_t& at) {
            const int r = fdiv(row, gm.by_nr);
            at = row * gm.row;
            return simt_token(dm, gm, r, row - r * dm.n_r);
        });
        cp_async_commit();
    }
    pdl_wait();          // delta and the inverse index come from the dQ kernel

    const int hi = dm.heads_i == 1 ? 0 : h;
    const size_t bhi = (size_t)b * dm.heads_i + hi;
    const int32_t* offs = inv_off + bhi * (dm.R + 1);
    const int32_t* order = inv_order + bhi * dm.R + r0;              // the CTA's key regions
    const int32_t* list = inv_list + bhi * dm.R * dm.topk;
    const float* lse_h = lse + ((size_t)b * dm.heads + h) * N0;
    const float* delta_h = delta + ((size_t)b * dm.heads + h) * N0;
    const int KS = 1 << gm.ksl, ks = tid & (KS - 1), slot = tid >> (gm.ksl + SPLIT);
    const int c0 = SPLIT ? (tid >> gm.ksl & 1) * DL : 0;              // this lane's first channel
    const int rl_raw = fdiv(slot, gm.spr, gm.mul_spr);
    const bool active = rl_raw < nreg;
    const int rl = active ? rl_raw : 0;
    const int jr = __ldcg(order + rl);                                // this lane's key region
    const int e0 = __ldcg(offs + jr), listed = __ldcg(offs + jr + 1) - e0;              // its query regions
    const int warp_listed = __reduce_max_sync(0xffffffffu, listed);
    bool weighted = false;
    int32_t* cnt = reinterpret_cast<int32_t*>(smem + gm.off_cnt);
    if (gm.dense) {
        __syncthreads();
        weighted = !simt_counts(cnt, nreg, dm.R, [&](auto add) {      // eight lanes per list
            for (int l = tid >> 3; l < nreg; l += blockDim.x >> 3) {
                const int j = __ldcg(order + l), end = __ldcg(offs + j + 1);
                for (int at = __ldcg(offs + j) + (tid & 7); at < end; at += 8) add(l, __ldcg(list + at));
            }
        });
    }
    const int t0 = active ? slot - rl_raw * gm.spr : 0;
    const int tok = active ? simt_row(dm, gm, chunk, jr, t0) : -1;
    float kr[DL], vr[DL], gk[1][DL], gv[1][DL];
    {
        const size_t at = head + (size_t)(tok < 0 ? 0 : tok) * dm.C + c0;
        ldg_row<T, DL>(kr, Kg + at, tok >= 0, dm.scale);
        ldg_row<T, DL>(vr, Vg + at, tok >= 0, 1.f);
#pragma unroll
        for (int i = 0; i < DL; ++i) gk[0][i] = gv[0][i] = 0.f;
    }
    // statistics of a row: lse and delta; a row that does not count has lse = inf (P = 0); a row of the zero padding has
    // zero Q and dO and lse = delta = 0 and adds nothing
    auto walk = [&](auto plain, uint32_t abase, uint32_t at0, int row0, int n, auto&& row_of) {
        constexpr bool PLAIN = decltype(plain)::value;
        uint32_t next = abase + at0 + ks * gm.row, next_stat = abase + gm.off_stat + (row0 + ks) * 8;
#pragma unroll 1
        for (int kb = 0; kb < n; kb += KS) {
            const int kk = kb + ks;
            uint32_t at = next, at_stat = next_stat;
            bool dead = kk >= n;
            float wt = 1.f;
            if constexpr (PLAIN) {
                if (dead && gm.resident) { at = abase + gm.zero; at_stat = abase + gm.off_stat; }
                next += KS * gm.row;
                next_stat += KS * 8;
            } else {
                const int row = dead ? -1 : row_of(kk, wt);
                dead = row < 0;
                at = abase + (dead ? gm.zero : row * gm.row);         // (resident: row number)
                at_stat = abase + gm.off_stat + (dead ? 0 : row) * 8;
            }
            const float2 stat = lds_f32x2(at_stat);
            float g[DL], qv[DL];
            lds_row<T, DL>(qv, at + gm.off_a + c0 * (int)sizeof(T));
            lds_row<T, DL>(g, at + gm.off_b + c0 * (int)sizeof(T));
            float dp = dot4(vr, g), s = dot(qv, kr);
            if (SPLIT) {
                dp += __shfl_xor_sync(0xffffffffu, dp, KS);
                s += __shfl_xor_sync(0xffffffffu, s, KS);
            }
            float p = expf(s - stat.x);
            if (!PLAIN && weighted) p *= wt;
            float ds = p * (dp - stat.y);
            if (dead) p = ds = 0.f;
            axpy(gk[0], ds, qv);
            axpy(gv[0], p, g);
        }
    };
    int most = 0;                                                     // entries of the CTA's longest list
    if (gm.resident) {
        float2* stat = reinterpret_cast<float2*>(smem + gm.off_stat);
        for (int row = tid; row < dm.N; row += blockDim.x) {
            const int r = fdiv(row, gm.by_nr);
            const int tk = simt_token(dm, gm, r, row - r * dm.n_r);
            stat[row] = tk >= 0 ? make_float2(__ldg(lse_h + tk), __ldcg(delta_h + tk)) : make_float2(0.f, 0.f);
        }
    } else {
        const int j = __ldcg(order);                                  // the first has the longest list
        most = __ldcg(offs + j + 1) - __ldcg(offs + j);
    }
    int first_entry = 0;                                              // of the walk
    auto load_stage = [&](int st) {
        const int off = (st & 1) * gm.stage_bytes;
        const uint32_t base = sbase + off;
        float2* stat = reinterpret_cast<float2*>(smem + off + gm.off_stat);
        simt_copy_rows<T, D>(base + gm.off_a, base + gm.off_b, Q, dO, dm.C, nreg * gm.kps, [&](int row, uint32_t& at) {
            const int lr = fdiv(row, gm.kps, gm.mul_kps), u = st * gm.kps + row - lr * gm.kps;
            at = lr * gm.reg + (row - lr * gm.kps) * gm.row;
            const int j = __ldcg(order + lr), m = fdiv(u, gm.by_nr), s0 = __ldcg(offs + j) + first_entry + m;
            int tk = -1;
            float2 v = make_float2(INFINITY, 0.f);
            if (s0 < __ldcg(offs + j + 1)) {
                tk = simt_token(dm, gm, __ldcg(list + s0), u - m * dm.n_r);
                v = tk >= 0 ? make_float2(__ldg(lse_h + tk), __ldcg(delta_h + tk)) : make_float2(0.f, 0.f);
            }
            if ((threadIdx.x & 3) == 0) stat[row] = v;
            return tk;
        });
        cp_async_commit();
    };
    do {
        const int nst = gm.resident ? 1 : (min(most - first_entry, gm.span) * dm.n_r + gm.kps - 1) / gm.kps;
        const int warp_total = min(warp_listed - first_entry, gm.span) * dm.n_r;
        if (!gm.resident) load_stage(0);
        for (int st = 0; st < nst; ++st) {
            simt_advance(gm, st, nst, load_stage);
            __syncthreads();
            const uint32_t abase = sbase + (st & 1) * gm.stage_bytes;
            if (!gm.resident) {
                const int rest = warp_total - st * gm.kps;
                if (rest > 0) walk(std::true_type(), abase, rl * gm.reg, rl * gm.kps, min(rest, gm.kps), 0);
            } else if (gm.dense && !weighted) {
                walk(std::true_type(), abase, 0, 0, dm.N, 0);
            } else {
                const int mine = listed * dm.n_r;                         // (a resident slice: a few hundred tokens)
                walk(std::false_type(), abase, 0, 0, gm.dense ? dm.N : warp_total, [&](int kk, float& wt) -> int {
                    const int m = fdiv(kk, gm.by_nr);
                    if (gm.dense) {
                        const int n = cnt[rl * dm.R + m];
                        wt = (float)n;
                        return n > 0 ? kk : -1;
                    }
                    return kk < mine ? __ldcg(list + e0 + m) * dm.n_r + kk - m * dm.n_r : -1;
                });
            }
            __syncthreads();
        }
        first_entry += gm.span;
    } while (first_entry < most);
    int first, held;
    sum_shares<1, DL>(gk, gm.ksl, ks, &first, &held);
    sum_shares<1, DL>(gv, gm.ksl, ks, &first, &held);
    cp_async_wait<0>();
    __syncthreads();
    float* st = reinterpret_cast<float*>(smem + gm.off_st);
    if (tok >= 0) {
        for_held<1, DL>(gk, first, held, [&](int, int c, const float4& v) {
            store4(dKg + head + (size_t)tok * dm.C + c0 + c, make_float4(v.x * dm.scale, v.y * dm.scale, v.z * dm.scale, v.w * dm.scale));
        });
        for_held<1, DL>(gv, first, held, [&](int, int c, const float4& v) {
            *reinterpret_cast<float4*>(st + (rl * gm.spr + t0) * (D + 4) + c0 + c) = v;
        });
    }
    __syncthreads();
    if (dm.hs <= 2) simt_lce<T, D, 2, true>(st, s_w, nullptr, dO, dVg + head, order, nreg, gm.spr, chunk, dm, gm);
    else simt_lce<T, D, 4, true>(st, s_w, nullptr, dO, dVg + head, order, nreg, gm.spr, chunk, dm, gm);
}

enum Family { FAMILY_SIMT, FAMILY_DIRECT, FAMILY_IMG, FAMILY_DENSE, FAMILY_ONE };

// bf16, head dim 32 or 64: tensor-core kernels.  Small maps with enough (image, head) pairs to fill the GPU keep a
// whole slice resident (head dim 32); the rest take their operands straight from global memory.
static Family choose_family(const Dims& d, int dtype, int impl) {
    if (dtype != BRA_BF16 || impl == BRA_IMPL_SIMT) return FAMILY_SIMT;
    if (impl == BRA_IMPL_AUTO && backward_dense_supported(d, dtype) && dense_grad_pays(d)) return FAMILY_DENSE;
    if (impl == BRA_IMPL_AUTO && backward_one_supported(d, dtype) && one_grad_pays(d)) return FAMILY_ONE;
    if (backward_img_supported(d, dtype) &&
        (impl == BRA_IMPL_IMG || (impl == BRA_IMPL_AUTO && img_grad_pays(d))))
        return FAMILY_IMG;
    return backward_direct_supported(d, dtype) ? FAMILY_DIRECT : FAMILY_SIMT;
}
bool backward_supported(const Dims& d, int dtype, int impl) {
    if ((d.d != 16 && d.d != 32 && d.d != 64) || d.R > 1000) return false;
    return choose_family(d, dtype, impl) != FAMILY_SIMT || (simt_fits(d, SIMT_DQ) && simt_fits(d, SIMT_DKV));
}
bool backward_any_map(const Dims& d, int dtype, int impl) { return choose_family(d, dtype, impl) != FAMILY_IMG; }

// The LCE weight gradient needs only V and dO, the attention gradients need neither of its results: the two
// run side by side (helper stream of bra_internal.h; everything stays on the caller's stream if there is none).
template <typename T, int D>
static cudaError_t launch_bwd_t(const Dims& d, int impl, const void* Q, const void* K, const void* V,
                                const int32_t* index, const float* lce_w, const float* lse,
                                const void* dO, void* dQ, void* dK, void* dV,
                                float* d_lce_w, float* d_lce_b, char* ws, const WsLayout& L,
                                cudaStream_t st) {
    int32_t* status = reinterpret_cast<int32_t*>(ws + L.status);
    float* delta = reinterpret_cast<float*>(ws + L.delta);
    int32_t* inv_off = reinterpret_cast<int32_t*>(ws + L.inv_off);
    int32_t* inv_list = reinterpret_cast<int32_t*>(ws + L.inv_list);
    int32_t* inv_order = reinterpret_cast<int32_t*>(ws + L.inv_order);
    float* part = reinterpret_cast<float*>(ws + L.dw_part);
    const T* q = static_cast<const T*>(Q); const T* k = static_cast<const T*>(K);
    const T* v = static_cast<const T*>(V); const T* go = static_cast<const T*>(dO);
    cudaError_t e;

    // ---- LCE weight / bias gradient, beside the attention gradients ----
    SideStream* ss = (d.lce || d_lce_b) ? side_stream() : nullptr;
    cudaStream_t dw_st = st;
    if (ss) {
        if (cudaEventRecord(ss->fork, st) != cudaSuccess || cudaStreamWaitEvent(ss->s, ss->fork, 0) != cudaSuccess) ss = nullptr;
        else dw_st = ss->s;
    }
    if (d.lce || d_lce_b) {
        if ((e = launch_lce_grad(d, sizeof(T) == 2 ? BRA_BF16 : BRA_F32, V, dO, part, d.lce ? d_lce_w : nullptr, d_lce_b,
                                 status, dw_st)) != cudaSuccess)
            return e;
    }
    if (ss && cudaEventRecord(ss->join, ss->s) != cudaSuccess) return cudaErrorUnknown;

    const Family family = choose_family(d, sizeof(T) == 2 ? BRA_BF16 : BRA_F32, impl);
    if (family == FAMILY_IMG) {
        // the dQ kernel of this family, of the direct and of the CUDA-core kernels also writes the inverse routing index
        if ((e = launch_backward_img(d, Q, K, V, index, inv_off, inv_list, lce_w, lse, dO, dQ, dK, dV,
                                     delta, status, st)) != cudaSuccess) return e;
    } else if (family == FAMILY_ONE) {
        if ((e = launch_backward_one(d, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, status, st)) != cudaSuccess) return e;
    } else if (family == FAMILY_DENSE) {
        if ((e = launch_backward_dense(d, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, status, st)) != cudaSuccess) return e;
    } else if (family == FAMILY_DIRECT) {
        if ((e = launch_backward_direct(d, Q, K, V, index, ws, L, lce_w, lse, dO, dQ, dK, dV, st)) != cudaSuccess) return e;
    } else {
        SimtGeom g = simt_geom(d, SIMT_DQ);
        const int inv = (int)inverse_smem(d);
        if (g.smem_bytes < inv) g.smem_bytes = inv;
        static PerDeviceMax set_q, set_kv;
        if (g.smem_bytes > 48 * 1024 && (e = set_q.ensure(g.smem_bytes, [&] {
                return cudaFuncSetAttribute(bwd_dq_simt_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, g.smem_bytes);
            })) != cudaSuccess)
            return e;
        e = grid_pieces(d, [&](const GridPiece& p) {
            const InversePiece inv = inverse_piece(d, p, inv_off, inv_list, inv_order);
            count_launch();
            return launch_kernel(bwd_dq_simt_kernel<T, D>, dim3(g.gpi > d.heads_i ? g.gpi : d.heads_i, p.heads + 1, p.images), dim3(g.threads),
                                 (size_t)g.smem_bytes, st, false, q + p.tensor, k + p.tensor, v + p.tensor, index + p.index, lse + p.stat,
                                 go + p.tensor, static_cast<T*>(dQ) + p.tensor, delta + p.stat, p.h0 ? nullptr : inv.off, inv.list, inv.order,
                                 inverse_uses_bits(d), status, d, g);
        });
        if (e != cudaSuccess) return e;
        const SimtGeom gk = simt_geom(d, SIMT_DKV);
        if (gk.smem_bytes > 48 * 1024 && (e = set_kv.ensure(gk.smem_bytes, [&] {
                return cudaFuncSetAttribute(bwd_dkv_simt_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, gk.smem_bytes);
            })) != cudaSuccess)
            return e;
        e = group_pieces(d, gk.gpi, gk.chunks, [&](const GridPiece& p, int regions_before, int groups) {
            const InversePiece inv = inverse_piece(d, p, inv_off, inv_list, inv_order);
            count_launch();
            return launch_kernel(bwd_dkv_simt_kernel<T, D>, dim3(p.heads, p.images, groups), dim3(gk.threads), (size_t)gk.smem_bytes, st, true,
                                 q + p.tensor, k + p.tensor, v + p.tensor, inv.off, inv.list, inv.order + regions_before, lse + p.stat,
                                 delta + p.stat, go + p.tensor, lce_w, static_cast<T*>(dK) + p.tensor, static_cast<T*>(dV) + p.tensor, d, gk);
        });
        if (e != cudaSuccess) return e;
    }

    if (ss && cudaStreamWaitEvent(st, ss->join, 0) != cudaSuccess) return cudaErrorUnknown;
    return cudaSuccess;
}

template <typename T>
static cudaError_t launch_bwd_d(const Dims& d, int impl, const void* Q, const void* K, const void* V,
                                const int32_t* index, const float* lce_w, const float* lse,
                                const void* dO, void* dQ, void* dK, void* dV,
                                float* d_lce_w, float* d_lce_b, char* ws, const WsLayout& L,
                                cudaStream_t st) {
    switch (d.d) {
        case 16: return launch_bwd_t<T, 16>(d, impl, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, d_lce_w, d_lce_b, ws, L, st);
        case 32: return launch_bwd_t<T, 32>(d, impl, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, d_lce_w, d_lce_b, ws, L, st);
        case 64: return launch_bwd_t<T, 64>(d, impl, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, d_lce_w, d_lce_b, ws, L, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_backward(const Dims& d, int dtype, int impl, const void* Q, const void* K, const void* V,
                            const int32_t* index, const float* lce_w, const float* lse,
                            const void* dO, void* dQ, void* dK, void* dV,
                            float* d_lce_w, float* d_lce_b,
                            char* ws, const WsLayout& L, cudaStream_t st) {
    if (dtype == BRA_BF16)
        return launch_bwd_d<__nv_bfloat16>(d, impl, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, d_lce_w, d_lce_b, ws, L, st);
    return launch_bwd_d<float>(d, impl, Q, K, V, index, lce_w, lse, dO, dQ, dK, dV, d_lce_w, d_lce_b, ws, L, st);
}

}  // namespace bra
