// fp32 backward for fp32 inputs on register-tiled FMA products, the counterpart of attn_fp32.cu (the
// paper trains through its kernel, Sec. 4.1, without describing the backward pass; this is the
// derivative of Algorithm 1's result).  One launch holds both directions:
//   mode 0: resident = 64 query rows;  over the keys they see:  dq_i += dS_ij k_j
//   mode 1: resident = 64 key rows;    over the queries that see them (the same ranges, the mask
//           being symmetric):  dk_j += dS_ij q_i,  dv_j += P_ij dO_i
// with P_ij = exp(s q_i.k_j - lse_i), dS_ij = P_ij (dO_i.v_j - delta_i).  Nothing is accumulated across
// CTAs but through a cluster's shared memory in rank order, so results are bit-reproducible.
// One pair of streamed tiles and three CTAs an SM (168 registers, 63 KB): their warps cover the waits for one
// another's tiles; two pairs and two CTAs took 193 instead of 186 us (32 x 32 + 64 tokens, 8 heads of 64, both passes).
#include <math.h>

#include "attn_fp32_tile.cuh"

namespace hilberta {

using namespace fp32t;

namespace {

constexpr int kDeltaRows = 4;

template <int D>
__global__ void __launch_bounds__(kDeltaRows * 32)
delta_fp32_kernel(const float *__restrict__ dout, const float *__restrict__ out, float *__restrict__ delta,
                  long long stride_b, long long stride_h, long long stride_s, int heads, int S) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bh = blockIdx.y, row = (int)blockIdx.x * kDeltaRows + warp;
    allow_next();
    wait_for_previous();
    if (row >= S) return;
    const long long off = (long long)(bh / heads) * stride_b + (long long)(bh % heads) * stride_h +
                          (long long)row * stride_s;
    float acc = 0.f;
#pragma unroll
    for (int e = 0; e < D / 32; ++e) acc = fmaf(dout[off + lane + 32 * e], out[off + lane + 32 * e], acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) delta[(long long)bh * S + row] = acc;
}

template <int D>
constexpr int bwd_smem() { return (2 * res_floats(D) + 2 * blk_floats(D) + BR * PS) * (int)sizeof(float); }

// One mode for one CTA.  r1 / t1: resident and streamed operand of the scores, r2 / t2: of dP.
template <int D, int MODE>
__device__ __forceinline__ void bwd_tile(const float *r1, const float *r2, const float *t1, const float *t2,
                                         const float *lse, const float *delta, float *out_a, float *out_b,
                                         long long stride_s, const WorkItem &it, const Share &share, float scale) {
    extern __shared__ float4 smem4[];
    constexpr int C = D / 8;
    float *sR1 = reinterpret_cast<float *>(smem4), *sR2 = sR1 + res_floats(D), *sT = sR2 + res_floats(D);
    float *sP = sT + 2 * blk_floats(D);
    const KeyList kl(it);
    const int nb = (kl.total + BC - 1) / BC;
    const int j0 = (int)((long long)nb * share.rank / share.parts), j1 = (int)((long long)nb * (share.rank + 1) / share.parts);
    const int lane = threadIdx.x & 31, rg = lane >> 3, cg = lane & 7;
    const int wrow = (threadIdx.x >> 5) * 16 + rg;

    load_rows<D>(sR1, r1, stride_s, it.q_start, it.q_rows, nullptr);
    load_rows<D>(sR2, r2, stride_s, it.q_start, it.q_rows, nullptr);
    float row_lse[4], row_delta[4];
    float a[4][C], b[4][C];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = wrow + 4 * i;
        row_lse[i] = MODE == 0 && r < it.q_rows ? lse[it.q_start + r] : 0.f;
        row_delta[i] = MODE == 0 && r < it.q_rows ? delta[it.q_start + r] : 0.f;
#pragma unroll
        for (int c = 0; c < C; ++c) a[i][c] = b[i][c] = 0.f;
    }
    const float one[4] = {1.f, 1.f, 1.f, 1.f};
    const bool busy = (int)(threadIdx.x >> 5) * 16 < it.q_rows;   // a warp without rows only helps with the loads
    const float *sT1 = sT, *sT2 = sT + blk_floats(D);
    auto load = [&](int j) {
        load_block<D>(sT, t1, stride_s, kl, j, nullptr);
        load_block<D>(sT + blk_floats(D), t2, stride_s, kl, j, nullptr);
    };
    if (j0 < j1) load(j0);
    cp_commit();   // also where this share has no block: the resident tiles' space holds the sums at the end
    for (int j = j0; j < j1; ++j) {
        const int valid = kl.total - j * BC;   // >= 1
        // the statistics belong to the QUERY of the pair: the streamed row in mode 1
        float col_lse[4], col_delta[4];
        if (MODE == 1) {
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                const int row = kl.row(8 * jj + cg < valid ? j * BC + 8 * jj + cg : 0);
                col_lse[jj] = __ldg(lse + row);
                col_delta[jj] = __ldg(delta + row);
            }
        }
        cp_wait<0>();
        __syncthreads();   // this block's tiles are in
        if (busy) {
            float p[4][4];
            dot_tile<D>(p, sR1 + wrow * (D + 4), sT1 + cg * (D + 4));
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj)
                    p[i][jj] = 8 * jj + cg < valid ? expf(fmaf(p[i][jj], scale, -(MODE == 0 ? row_lse[i] : col_lse[jj]))) : 0.f;
            float ds[4][4];
            dot_tile<D>(ds, sR2 + wrow * (D + 4), sT2 + cg * (D + 4));
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj)   // beyond the list P is zero and the streamed rows and statistics are any
                    ds[i][jj] = 8 * jj + cg < valid ? p[i][jj] * (ds[i][jj] - (MODE == 0 ? row_delta[i] : col_delta[jj])) : 0.f;
            if (MODE == 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) sP[(wrow + 4 * i) * PS + 8 * jj + cg] = p[i][jj];
                __syncwarp();
                acc_tile<D>(b, one, sP + wrow * PS, sT2, cg);   // dv += P dO
                __syncwarp();
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) sP[(wrow + 4 * i) * PS + 8 * jj + cg] = ds[i][jj];
            __syncwarp();
            acc_tile<D>(a, one, sP + wrow * PS, sT1, cg);       // dq += dS k  |  dk += dS q
        }
        __syncthreads();   // ... and free again; the other CTAs of the SM work while the next ones come
        if (j + 1 < j1) load(j + 1);
        cp_commit();
    }
    cp_wait<0>();
    if (share.parts == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = wrow + 4 * i;
            if (r >= it.q_rows) continue;
#pragma unroll
            for (int c = 0; c < C; ++c) a[i][c] *= scale;
            store_cols<D>(out_a + (long long)(it.q_start + r) * stride_s, cg, a[i]);
            if (MODE == 1) store_cols<D>(out_b + (long long)(it.q_start + r) * stride_s, cg, b[i]);
        }
        return;
    }
    // sum of the cluster's shares, in rank order; rank c writes rows [64 c / parts, 64 (c + 1) / parts)
    // (the resident tiles' space holds them)
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        store_cols<D>(sR1 + (wrow + 4 * i) * (D + 4), cg, a[i]);
        if (MODE == 1) store_cols<D>(sR2 + (wrow + 4 * i) * (D + 4), cg, b[i]);
    }
    cluster_sync();
    const int rows = BR / share.parts, r0 = rows * share.rank;
    for (int e = threadIdx.x; e < (MODE + 1) * rows * (D / 4); e += kThreads) {
        const bool second = e >= rows * (D / 4);
        const int f = second ? e - rows * (D / 4) : e;
        const int r = r0 + f / (D / 4), c4 = f % (D / 4);
        if (r >= it.q_rows) continue;
        const float *src = (second ? sR2 : sR1) + r * (D + 4) + 4 * c4;
        float4 y[8];
#pragma unroll
        for (int p = 0; p < 8; ++p)
            if (p < share.parts) y[p] = peer_ld4(peer_addr(src, p));
        float4 acc = y[0];
#pragma unroll
        for (int p = 1; p < 8; ++p)
            if (p < share.parts) {
                acc.x += y[p].x;
                acc.y += y[p].y;
                acc.z += y[p].z;
                acc.w += y[p].w;
            }
        const float f4 = second ? 1.f : scale;
        *reinterpret_cast<float4 *>((second ? out_b : out_a) + (long long)(it.q_start + r) * stride_s + 4 * c4) =
            make_float4(acc.x * f4, acc.y * f4, acc.z * f4, acc.w * f4);
    }
    cluster_sync();   // no CTA leaves while a peer may still read its shared memory
}

template <int D>
__global__ void __launch_bounds__(kThreads, D == 128 ? 2 : 3)
attn_fp32_bwd_kernel(const float *__restrict__ q, const float *__restrict__ k, const float *__restrict__ v,
                     const float *__restrict__ dout, const float *__restrict__ lse, const float *__restrict__ delta,
                     float *__restrict__ dq, float *__restrict__ dk, float *__restrict__ dv, long long stride_b,
                     long long stride_h, long long stride_s, int heads, int bhs, int S, const WorkItem *__restrict__ work,
                     int n_items, int n_split, int cluster, float scale) {
    const Share share(n_items, n_split, cluster, 2 * bhs);
    if (share.item < 0) return;
    const WorkItem it = work[share.item];
    allow_next();
    wait_for_previous();
    const bool keys = share.column < bhs;   // the direction with more work per pair first
    const int bh = keys ? share.column : share.column - bhs;
    const long long base = (long long)(bh / heads) * stride_b + (long long)(bh % heads) * stride_h;
    lse += (long long)bh * S;
    delta += (long long)bh * S;
    if (keys)
        bwd_tile<D, 1>(k + base, v + base, q + base, dout + base, lse, delta, dk + base, dv + base, stride_s, it, share, scale);
    else
        bwd_tile<D, 0>(q + base, dout + base, k + base, v + base, lse, delta, dq + base, nullptr, stride_s, it, share, scale);
}

// The rows of short lists, one mode for one warp: the row in registers, the streamed rows one after another.
template <int D, int MODE>
__device__ __forceinline__ void bwd_row(const float *r1, const float *r2, const float *t1, const float *t2, const float *lse,
                                        const float *delta, float *out_a, float *out_b, long long stride_s,
                                        const SingleRow &it, float scale) {
    constexpr int E = D / 32;
    const int lane = threadIdx.x & 31;
    const long long at = (long long)it.row * stride_s + lane;
    float a1[E], a2[E], acc_a[E], acc_b[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        a1[e] = r1[at + 32 * e];
        a2[e] = r2[at + 32 * e];
        acc_a[e] = acc_b[e] = 0.f;
    }
    const float row_lse = lse[it.row], row_delta = delta[it.row];
    for (int s = 0; s < 3; ++s) {
        const int end = it.start[s] + it.len[s];
        for (int j = it.start[s]; j < end; ++j) {
            const float *x1 = t1 + (long long)j * stride_s + lane, *x2 = t2 + (long long)j * stride_s + lane;
            float b1[E], b2[E], dot1 = 0.f, dot2 = 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                b1[e] = __ldg(x1 + 32 * e);
                b2[e] = __ldg(x2 + 32 * e);
                dot1 = fmaf(a1[e], b1[e], dot1);
                dot2 = fmaf(a2[e], b2[e], dot2);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                dot1 += __shfl_xor_sync(0xffffffffu, dot1, o);
                dot2 += __shfl_xor_sync(0xffffffffu, dot2, o);
            }
            // the statistics belong to the QUERY of the pair
            const float p = expf(fmaf(dot1, scale, -(MODE == 0 ? row_lse : __ldg(lse + j))));
            const float ds = p * (dot2 - (MODE == 0 ? row_delta : __ldg(delta + j)));
#pragma unroll
            for (int e = 0; e < E; ++e) {
                acc_a[e] = fmaf(ds, b1[e], acc_a[e]);                   // dq += dS k  |  dk += dS q
                if (MODE == 1) acc_b[e] = fmaf(p, b2[e], acc_b[e]);     //             |  dv += P dO
            }
        }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
        out_a[at + 32 * e] = acc_a[e] * scale;
        if (MODE == 1) out_b[at + 32 * e] = acc_b[e];
    }
}

// Bound by the shuffles and, with few keys a row, by how fast CTAs start, hence eight rows to a CTA, as few
// registers as let 64 warps run on an SM, and a row's ranges in its own record (48 x 48 tokens, tiles of 4, 48 heads
// of 64, with the row statistics: 139 us; four rows, 40 registers and a table lookup 173; 32: 120, 128). z: the direction,
// the one with more work per pair first.
constexpr int kBwdRows = 8;
template <int D>
__global__ void __launch_bounds__(kBwdRows * 32, D == 128 ? 5 : 8)
attn_fp32_bwd_rows_kernel(const float *__restrict__ q, const float *__restrict__ k, const float *__restrict__ v,
                          const float *__restrict__ dout, const float *__restrict__ lse, const float *__restrict__ delta,
                          float *__restrict__ dq, float *__restrict__ dk, float *__restrict__ dv, long long stride_b,
                          long long stride_h, long long stride_s, int heads, int S, int P,
                          const Fp32Row *__restrict__ rows, int n_rows, float scale) {
    const SingleRow it(rows, n_rows, P, (int)blockIdx.x * kBwdRows + (int)(threadIdx.x >> 5));
    allow_next();
    wait_for_previous();
    if (it.row < 0) return;
    const int bh = blockIdx.y;
    const long long base = (long long)(bh / heads) * stride_b + (long long)(bh % heads) * stride_h;
    lse += (long long)bh * S;
    delta += (long long)bh * S;
    if (blockIdx.z == 0) bwd_row<D, 1>(k + base, v + base, q + base, dout + base, lse, delta, dk + base, dv + base, stride_s, it, scale);
    else bwd_row<D, 0>(q + base, dout + base, k + base, v + base, lse, delta, dq + base, nullptr, stride_s, it, scale);
}

template <int D>
int launch(const hilberta_plan_t *p, const float *dout, const float *q, const float *k, const float *v,
           const float *out, const float *lse, float *dq, float *dk, float *dv, float *delta, cudaStream_t stream) {
    const Fp32Work &w = p->f32_bwd;
    const int bhs = p->batch * p->heads;
    const long long ctas = items_grid(w, 2 * bhs);
    if (ctas > 0x7fffffffll) return HILBERTA_ERR_INVALID;
    HB_CUDA(launch_overlapping(delta_fp32_kernel<D>, dim3((p->S + kDeltaRows - 1) / kDeltaRows, bhs), kDeltaRows * 32, 0, 1, stream,
                               true, dout, out, delta, p->stride_b, p->stride_h, p->stride_s, p->heads, p->S));
    HB_LAUNCHED();
    if (ctas > 0) {
        HB_CUDA(launch_overlapping(attn_fp32_bwd_kernel<D>, (unsigned)ctas, kThreads, bwd_smem<D>(), (unsigned)w.cluster, stream,
                                   may_overlap(p, ctas), q, k, v, dout, lse, delta, dq, dk, dv, p->stride_b, p->stride_h,
                                   p->stride_s, p->heads, bhs, p->S, w.items, w.n_items, w.n_split, w.cluster, p->scale));
        HB_LAUNCHED();
    }
    if (w.n_rows > 0) {
        HB_CUDA(launch_overlapping(attn_fp32_bwd_rows_kernel<D>, dim3((w.n_rows + kBwdRows - 1) / kBwdRows, bhs, 2), kBwdRows * 32, 0, 1,
                                   stream, true, q, k, v, dout, lse, delta, dq, dk, dv, p->stride_b, p->stride_h, p->stride_s,
                                   p->heads, p->S, p->P, w.rows, w.n_rows, p->scale));
        HB_LAUNCHED();
    }
    return HILBERTA_OK;
}

}  // namespace

int attn_fp32_bwd_opt_in() {
    HB_CUDA(cudaFuncSetAttribute(attn_fp32_bwd_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, bwd_smem<32>()));
    HB_CUDA(cudaFuncSetAttribute(attn_fp32_bwd_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, bwd_smem<64>()));
    HB_CUDA(cudaFuncSetAttribute(attn_fp32_bwd_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, bwd_smem<128>()));
    return HILBERTA_OK;
}

int launch_attn_fp32_bwd(const hilberta_plan_t *p, const void *dout, const void *q, const void *k, const void *v,
                         const void *out, const float *lse, void *dq, void *dk, void *dv, float *delta,
                         cudaStream_t stream) {
    if ((p->stride_b | p->stride_h | p->stride_s) & 3) return HILBERTA_ERR_INVALID;
    switch (p->head_dim) {
        case 32:
            return launch<32>(p, (const float *)dout, (const float *)q, (const float *)k, (const float *)v,
                              (const float *)out, lse, (float *)dq, (float *)dk, (float *)dv, delta, stream);
        case 64:
            return launch<64>(p, (const float *)dout, (const float *)q, (const float *)k, (const float *)v,
                              (const float *)out, lse, (float *)dq, (float *)dk, (float *)dv, delta, stream);
        case 128:
            return launch<128>(p, (const float *)dout, (const float *)q, (const float *)k, (const float *)v,
                               (const float *)out, lse, (float *)dq, (float *)dk, (float *)dv, delta, stream);
        default: return HILBERTA_ERR_UNSUPPORTED;
    }
}

}  // namespace hilberta
