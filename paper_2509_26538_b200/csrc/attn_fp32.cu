// fp32 forward for fp32 inputs: online softmax over register-tiled products on the FMA pipes
// (attn_fp32_tile.cuh).  A CTA owns 64 query rows that share a key list (Algorithm 1: the global prefix
// plus the rows' slid tile, or the whole sequence for prefix rows) and walks it in blocks of 32 keys; the
// next block's K and V tiles arrive (cp.async) while this block is worked on, and a block costs one barrier.
// Bound: the FMA pipes and, next to them, shared memory.  Measured (B200): 32 x 32 + 64 tokens, 8 heads of 64,
// forward + backward 1500 -> 179 us (17 TFLOP/s useful; one warp per query row with a key per lane before,
// every lane reading whole rows of its own); 16 x 16 tokens, 2 heads of 64, 26 -> 10 us a call.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "attn_fp32_tile.cuh"

namespace hilberta {

using namespace fp32t;

namespace {

template <int D>
constexpr int fwd_smem() { return (res_floats(D) + 4 * blk_floats(D) + BR * PS + 2 * BR) * (int)sizeof(float); }

template <int D>
__global__ void __launch_bounds__(kThreads, D == 128 ? 2 : 3)
attn_fp32_kernel(const float *__restrict__ q, const float *__restrict__ k, const float *__restrict__ v,
                 float *__restrict__ out, long long stride_b, long long stride_h, long long stride_s,
                 int heads, int bhs, int S, const WorkItem *__restrict__ work, int n_items, int n_split, int cluster,
                 const int *__restrict__ out_map, const int *__restrict__ in_map, float *__restrict__ lse, float scale) {
    extern __shared__ float4 smem4[];
    constexpr int C = D / 8;
    float *sQ = reinterpret_cast<float *>(smem4), *sKV = sQ + res_floats(D);
    float *sP = sKV + 4 * blk_floats(D), *sM = sP + BR * PS, *sL = sM + BR;
    const Share share(n_items, n_split, cluster, bhs);
    if (share.item < 0) return;
    const WorkItem it = work[share.item];
    const KeyList kl(it);
    const int bh = share.column;
    const long long base = (long long)(bh / heads) * stride_b + (long long)(bh % heads) * stride_h;
    const int nb = (kl.total + BC - 1) / BC;
    const int j0 = (int)((long long)nb * share.rank / share.parts), j1 = (int)((long long)nb * (share.rank + 1) / share.parts);
    const int lane = threadIdx.x & 31, rg = lane >> 3, cg = lane & 7;
    const int wrow = (threadIdx.x >> 5) * 16 + rg;   // this lane's rows: wrow + 2 i

    allow_next();
    wait_for_previous();
    // in_map: q, k, v are in original order and physical row p lives at row in_map[p]
    load_rows<D>(sQ, q + base, stride_s, it.q_start, it.q_rows, in_map);
    if (j0 < j1) {
        load_block<D>(sKV, k + base, stride_s, kl, j0, in_map);
        load_block<D>(sKV + blk_floats(D), v + base, stride_s, kl, j0, in_map);
    }
    cp_commit();

    const bool busy = (int)(threadIdx.x >> 5) * 16 < it.q_rows;   // a warp without rows only helps with the loads
    float m[4], l[4], o[4][C];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m[i] = -INFINITY;
        l[i] = 0.f;
#pragma unroll
        for (int c = 0; c < C; ++c) o[i][c] = 0.f;
    }
    for (int j = j0; j < j1; ++j) {
        const float *sK = sKV + ((j - j0) & 1) * 2 * blk_floats(D), *sV = sK + blk_floats(D);
        cp_wait<0>();
        __syncthreads();     // this block's tiles are in, and every warp is done with the other pair
        if (j + 1 < j1) {
            float *nK = sKV + ((j + 1 - j0) & 1) * 2 * blk_floats(D);
            load_block<D>(nK, k + base, stride_s, kl, j + 1, in_map);
            load_block<D>(nK + blk_floats(D), v + base, stride_s, kl, j + 1, in_map);
        }
        cp_commit();
        if (!busy) continue;
        float x[4][4];
        dot_tile<D>(x, sQ + wrow * (D + 4), sK + cg * (D + 4));
        const int valid = kl.total - j * BC;   // >= 1
        float corr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float mx = -INFINITY;
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                x[i][jj] = 8 * jj + cg < valid ? x[i][jj] * scale : -INFINITY;
                mx = fmaxf(mx, x[i][jj]);
            }
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float mn = fmaxf(m[i], mx);
            corr[i] = m[i] == mn ? 1.f : expf(m[i] - mn);   // exp(-inf) = 0 on the first block
            m[i] = mn;
            float sum = 0.f;
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                const float p = 8 * jj + cg < valid ? expf(x[i][jj] - mn) : 0.f;
                sP[(wrow + 4 * i) * PS + 8 * jj + cg] = p;
                sum += p;
            }
            l[i] = fmaf(l[i], corr[i], sum);   // this lane's share of the row sum
        }
        __syncwarp();        // a warp's weights stay within the warp
        acc_tile<D>(o, corr, sP + wrow * PS, sV, cg);
        __syncwarp();
    }
    cp_wait<0>();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);

    if (share.parts == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = wrow + 4 * i;
            if (r >= it.q_rows) continue;
            const int out_row = out_map ? out_map[it.q_start + r] : it.q_start + r;   // optional fused exit scatter
            const float inv = 1.f / l[i];
#pragma unroll
            for (int c = 0; c < C; ++c) o[i][c] *= inv;
            store_cols<D>(out + base + (long long)out_row * stride_s, cg, o[i]);
            if (lse && cg == 0) lse[(long long)bh * S + out_row] = m[i] + logf(l[i]);
        }
        return;
    }
    // Merge of the cluster's partial states: every CTA leaves (m, l, O) of its share in shared memory,
    // rank c writes rows [64 c / parts, 64 (c + 1) / parts).
    __syncthreads();
    float *sO = sKV;   // 64 rows take the space of two K / V tiles
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = wrow + 4 * i;
        store_cols<D>(sO + r * (D + 4), cg, o[i]);
        if (cg == 0) {
            sM[r] = m[i];
            sL[r] = l[i];
        }
    }
    cluster_sync();
    const int rows = BR / share.parts, r0 = rows * share.rank;
    for (int e = threadIdx.x; e < rows * (D / 4); e += kThreads) {
        const int r = r0 + e / (D / 4), c4 = e % (D / 4);
        if (r >= it.q_rows) continue;
        // all loads of a CTA pair's states are in flight together (parts <= 8)
        float mp[8], lp[8];
        float4 y[8];
        float m_all = -INFINITY;
#pragma unroll
        for (int p = 0; p < 8; ++p)
            if (p < share.parts) {
                mp[p] = peer_ld(peer_addr(sM + r, p));
                lp[p] = peer_ld(peer_addr(sL + r, p));
                y[p] = peer_ld4(peer_addr(sO + r * (D + 4) + 4 * c4, p));
            }
#pragma unroll
        for (int p = 0; p < 8; ++p)
            if (p < share.parts) m_all = fmaxf(m_all, mp[p]);
        float l_all = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int p = 0; p < 8; ++p)
            if (p < share.parts) {
                const float w = mp[p] == m_all ? 1.f : expf(mp[p] - m_all);   // a share of no blocks has m = -inf
                l_all = fmaf(lp[p], w, l_all);
                acc.x = fmaf(y[p].x, w, acc.x);
                acc.y = fmaf(y[p].y, w, acc.y);
                acc.z = fmaf(y[p].z, w, acc.z);
                acc.w = fmaf(y[p].w, w, acc.w);
            }
        const float inv = 1.f / l_all;
        const int out_row = out_map ? out_map[it.q_start + r] : it.q_start + r;
        *reinterpret_cast<float4 *>(out + base + (long long)out_row * stride_s + 4 * c4) =
            make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        if (lse && c4 == 0) lse[(long long)bh * S + out_row] = m_all + logf(l_all);
    }
    cluster_sync();   // no CTA leaves while a peer may still read its shared memory
}

}  // namespace

// Work list of the fp32 kernels: items of 64 rows, longest key lists first, all of more than two blocks
// cut over clusters of up to 8 CTAs as long as that leaves no SM more than a few CTAs.  Prefix rows see the
// whole sequence, and on the problems this path serves a handful of them would otherwise outlast everything
// else (and a small problem would leave most SMs idle); every cut costs each CTA its start and a merge.  The
// bound (CTAs per SM up to which cuts double) is the best of 1.5, 2, 3, 4.5, 6 and 8 over 42 problems on the
// B200; geometric means in us, forward: head dim 64 65.8 / 61.2 / 55.4 / 54.6 / 55.8 / 56.7, 128 128 / 128 / 118 /
// 104 / 103 / 102, 32 37.6 / 35.0 / 33.7 / 36.9 / 37.1 / 37.0; forward + backward: 64 219 / 177 / 167 / 160 / 168 /
// 180, 128 242 / 208 / 204 / 191 / 207 / 223, 32 134 / 125 / 120 / 133 / 133 / 137.
int attn_fp32_prepare(hilberta_plan_t *p, BindImage &image) {
    std::vector<WorkItem> items = build_work_items(p, BR, BC);
    const int rc = check_work_items(items.data(), (int)items.size(), p->S, BR, BC);
    if (rc != HILBERTA_OK) return rc;
    auto blocks = [](const WorkItem &it) {
        long long n = 0;
        for (int s = 0; s < it.n_seg; ++s) n += it.seg_len[s];
        return (n + BC - 1) / BC;   // the kernels read the ranges as one list
    };
    std::stable_sort(items.begin(), items.end(), [&](const WorkItem &a, const WorkItem &b) { return blocks(a) > blocks(b); });
    const long long instances = (long long)items.size() * p->batch * p->heads;
    const long long most = (long long)p->sm_count * (p->head_dim == 32 ? 6 : 9) / 2;
    p->f32_cluster = 1;
    while (p->f32_cluster < 8 && instances * p->f32_cluster * 2 <= most) p->f32_cluster *= 2;
    p->n_f32_split = 0;
    if (p->f32_cluster > 1)
        while (p->n_f32_split < (int)items.size() && blocks(items[p->n_f32_split]) > 2) ++p->n_f32_split;
    p->n_f32_work = (int)items.size();
    if (items.empty()) return HILBERTA_OK;
    image.add(items, &p->d_f32_work);
    // scratch of the backward pass (delta per row; sized like the bf16 path's)
    image.add_scratch(2 * (size_t)p->batch * p->heads * p->S, &p->d_delta);
    // the shared-memory opt-in is an attribute of the kernel on one device
    static std::mutex attr_mutex;
    static bool attr_done[64] = {};
    std::lock_guard<std::mutex> lock(attr_mutex);
    if (p->device < 0 || p->device >= 64) return HILBERTA_ERR_INVALID;
    if (!attr_done[p->device]) {
        HB_CUDA(cudaFuncSetAttribute(attn_fp32_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd_smem<32>()));
        HB_CUDA(cudaFuncSetAttribute(attn_fp32_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd_smem<64>()));
        HB_CUDA(cudaFuncSetAttribute(attn_fp32_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd_smem<128>()));
        const int rc_bwd = attn_fp32_bwd_opt_in();
        if (rc_bwd != HILBERTA_OK) return rc_bwd;
        attr_done[p->device] = true;
    }
    return HILBERTA_OK;
}

int launch_attn_fp32(const hilberta_plan_t *p, const void *q, const void *k, const void *v, void *out,
                     float *lse, const int *out_map, const int *in_map, cudaStream_t stream, int chunk) {
    const uintptr_t bits = (uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out;
    if ((bits & 15) || ((p->stride_b | p->stride_h | p->stride_s) & 3)) return HILBERTA_ERR_INVALID;
    if (chunk >= 0) return HILBERTA_ERR_INVALID;   // fp32 bindings have no slices of heads
    if (p->n_f32_work == 0) return HILBERTA_OK;
    const long long ctas = grid_of(p, 1);
    if (ctas > 0x7fffffffll) return HILBERTA_ERR_INVALID;
#define HB_FP32_CASE(DD)                                                                                              \
    case DD:                                                                                                          \
        HB_CUDA(launch_overlapping(attn_fp32_kernel<DD>, (unsigned)ctas, kThreads, fwd_smem<DD>(), (unsigned)p->f32_cluster, stream, may_overlap(p, ctas), \
                                   (const float *)q, (const float *)k, (const float *)v, (float *)out, p->stride_b,   \
                                   p->stride_h, p->stride_s, p->heads, p->batch * p->heads, p->S, p->d_f32_work,      \
                                   p->n_f32_work, p->n_f32_split, p->f32_cluster, out_map, in_map, lse, p->scale));   \
        break;
    switch (p->head_dim) {
        HB_FP32_CASE(32)
        HB_FP32_CASE(64)
        HB_FP32_CASE(128)
        default: return HILBERTA_ERR_UNSUPPORTED;
    }
#undef HB_FP32_CASE
    HB_LAUNCHED();
    return HILBERTA_OK;
}

}  // namespace hilberta
