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
    const int wrow = (threadIdx.x >> 5) * 16 + rg;   // this lane's rows: wrow + 4 i

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

// The rows of short lists: a warp per row, a key per lane, every lane with an online softmax of its own; the 32
// states are merged at the end, which is what a row of few keys takes its time for.  48 x 48 tokens, tiles of 1, 48
// heads: of 64 280 us, of 32 117, of 128 649 (as items of 64-row CTAs 1350, 963, 3006).
template <int D>
__global__ void __launch_bounds__(kThreads, D == 128 ? 3 : D == 64 ? 4 : 6)
attn_fp32_rows_kernel(const float *__restrict__ q, const float *__restrict__ k, const float *__restrict__ v,
                      float *__restrict__ out, long long stride_b, long long stride_h, long long stride_s, int heads, int S,
                      int P, const Fp32Row *__restrict__ rows, int n_rows, const int *__restrict__ out_map,
                      const int *__restrict__ in_map, float *__restrict__ lse, float scale) {
    __shared__ __align__(16) float sq[kRowsPerCta][D];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const SingleRow it(rows, n_rows, P, (int)blockIdx.x * kRowsPerCta + warp);
    allow_next();
    wait_for_previous();
    if (it.row < 0) return;   // the whole warp leaves; no CTA-wide barrier below
    const int bh = blockIdx.y;
    const long long base = (long long)(bh / heads) * stride_b + (long long)(bh % heads) * stride_h;
    // in_map: q, k, v are in original order and physical row p lives at row in_map[p]
    const float *qrow = q + base + (long long)(in_map ? in_map[it.row] : it.row) * stride_s;
    for (int d = lane; d < D; d += 32) sq[warp][d] = qrow[d];
    __syncwarp();

    float m = -INFINITY, l = 0.f;
    float acc[D];
#pragma unroll
    for (int d = 0; d < D; ++d) acc[d] = 0.f;
    for (int s = 0; s < 3; ++s) {
        const int end = it.start[s] + it.len[s];
        for (int j = it.start[s] + lane; j < end; j += 32) {
            const long long jrow = in_map ? in_map[j] : j;
            const float4 *kj = reinterpret_cast<const float4 *>(k + base + jrow * stride_s);
            float2 dot = make_float2(0.f, 0.f);   // even and odd apart, as in dot_tile
#pragma unroll
            for (int d4 = 0; d4 < D / 4; ++d4) {
                const float4 kk = __ldg(kj + d4), qq = *reinterpret_cast<const float4 *>(&sq[warp][4 * d4]);
                dot = __ffma2_rn(make_float2(qq.x, qq.y), make_float2(kk.x, kk.y), dot);
                dot = __ffma2_rn(make_float2(qq.z, qq.w), make_float2(kk.z, kk.w), dot);
            }
            const float x = (dot.x + dot.y) * scale;
            if (x > m) {
                const float corr = expf(m - x);   // exp(-inf) = 0 on the first key
                l *= corr;
#pragma unroll
                for (int d = 0; d < D; ++d) acc[d] *= corr;
                m = x;
            }
            const float p = expf(x - m);
            l += p;
            const float4 *vj = reinterpret_cast<const float4 *>(v + base + jrow * stride_s);
#pragma unroll
            for (int d4 = 0; d4 < D / 4; ++d4) {
                const float4 vv = __ldg(vj + d4);
                acc[4 * d4 + 0] = fmaf(p, vv.x, acc[4 * d4 + 0]);
                acc[4 * d4 + 1] = fmaf(p, vv.y, acc[4 * d4 + 1]);
                acc[4 * d4 + 2] = fmaf(p, vv.z, acc[4 * d4 + 2]);
                acc[4 * d4 + 3] = fmaf(p, vv.w, acc[4 * d4 + 3]);
            }
        }
    }
    float m_all = m;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m_all = fmaxf(m_all, __shfl_xor_sync(0xffffffffu, m_all, off));
    const float f = m == -INFINITY ? 0.f : expf(m - m_all);
    l *= f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    const float inv = 1.f / l;
    float mine[D / 32];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        float a = acc[d] * f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if ((d & 31) == lane) mine[d >> 5] = a * inv;
    }
    const int out_row = out_map ? out_map[it.row] : it.row;   // optional fused exit scatter
    float *orow = out + base + (long long)out_row * stride_s;
    if (lse && lane == 0) lse[(long long)bh * S + out_row] = m_all + logf(l);
#pragma unroll
    for (int i = 0; i < D / 32; ++i) orow[i * 32 + lane] = mine[i];
}

// Estimated times in ns, fitted to 15 problems with tiles of 1 ... 32 tokens on the B200, none of which
// takes more than 13 % longer than with either way for all of its rows.  On a full chip: an item (a CTA
// has 64 rows whatever the item has) and each of its blocks of 32 keys, a single row and each of its keys.  And by
// themselves: an item for each block, a row for each key.
struct Fp32Cost {
    float item, block, row, key, block_alone, key_alone;
};
Fp32Cost fp32_cost(int head_dim, bool backward) {
    if (backward)
        return head_dim == 32 ? Fp32Cost{7.f, 13.5f, 0.54f, 0.13f, 3700.f, 100.f}
             : head_dim == 64 ? Fp32Cost{11.f, 22.f, 0.66f, 0.16f, 7400.f, 100.f} : Fp32Cost{16.f, 62.f, 1.f, 0.21f, 10400.f, 100.f};
    return head_dim == 32 ? Fp32Cost{4.6f, 4.1f, 1.f, 0.05f, 2400.f, 17.f}
         : head_dim == 64 ? Fp32Cost{8.f, 4.7f, 2.4f, 0.094f, 3800.f, 17.f} : Fp32Cost{9.f, 18.f, 5.9f, 0.153f, 5800.f, 17.f};
}
constexpr double kSecondLaunch = 3000.;   // ns

int key_count(const WorkItem &it) {
    int n = 0;
    for (int s = 0; s < it.n_seg; ++s) n += it.seg_len[s];
    return n;
}
int block_count(const WorkItem &it) { return (key_count(it) + BC - 1) / BC; }   // the ranges are read as one list

// Cuts for `items` (by descending length): all of more than two blocks over clusters of up to 8 CTAs as long as
// that leaves no SM more than a few CTAs; `most`: CTAs up to which cuts double.
void cut_items(const std::vector<WorkItem> &items, long long bhs, long long most, Fp32Work &w) {
    const long long instances = (long long)items.size() * bhs;
    w.n_items = (int)items.size();
    w.cluster = 1;
    while (w.cluster < 8 && instances * w.cluster * 2 <= most) w.cluster *= 2;
    w.n_split = 0;
    if (w.cluster > 1)
        while (w.n_split < w.n_items && block_count(items[w.n_split]) > 2) ++w.n_split;
}

double items_time(const std::vector<WorkItem> &items, long long bhs, const Fp32Work &w, const Fp32Cost &c) {
    double sum = 0, longest = 0;
    for (size_t i = 0; i < items.size(); ++i) {
        const int n = block_count(items[i]), parts = (int)i < w.n_split ? w.cluster : 1;
        sum += c.item + c.block * n;
        longest = std::max(longest, (double)c.block_alone * ((n + parts - 1) / parts));
    }
    return std::max(sum * (double)bhs, longest);
}

// Splits `items` into those that stay items, with their cuts in `w`, and the rows, returned with their ranges,
// that are better off with a warp each: rows of windows with so few of them that they take less time than an item
// would, if all those together, with the second launch and what it does for the cuts of the others, make the
// whole shorter.  (Never prefix rows, which see everything.)
std::vector<Fp32Row> take_short_rows(const hilberta_plan_t *p, std::vector<WorkItem> &items, long long most, const Fp32Cost &c, Fp32Work &w) {
    const long long bhs = (long long)p->batch * p->heads;
    cut_items(items, bhs, most, w);
    std::vector<WorkItem> kept, few;
    double rows_time = 0;
    int keys = 0;
    for (const WorkItem &it : items) {
        const int n = key_count(it);
        const float alone = (float)it.q_rows * (c.row + c.key * (float)n);
        const bool is_short = it.q_start >= p->P && alone < c.item + c.block * (float)block_count(it);
        (is_short ? few : kept).push_back(it);
        if (is_short) {
            rows_time += alone;
            keys = std::max(keys, n);
        }
    }
    if (few.empty()) return {};
    Fp32Work without{};
    cut_items(kept, bhs, most, without);
    const double time = items_time(kept, bhs, without, c) + std::max(rows_time * (double)bhs, (double)c.key_alone * keys) +
                        (kept.empty() ? 0. : kSecondLaunch);
    if (time >= items_time(items, bhs, w, c)) return {};
    w = without;
    items.swap(kept);
    std::vector<Fp32Row> rows;
    for (const WorkItem &it : few) {
        const int g = p->P > 0 ? 1 : 0;   // the item's first range that is not the prefix
        Fp32Row r{0, it.seg_start[g], it.seg_len[g], it.seg_start[g + 1], it.n_seg > g + 1 ? it.seg_len[g + 1] : 0, {0, 0, 0}};
        for (r.row = it.q_start; r.row < it.q_start + it.q_rows; ++r.row) rows.push_back(r);
    }
    // neighbours in memory next to each other
    std::sort(rows.begin(), rows.end(), [](const Fp32Row &a, const Fp32Row &b) { return a.row < b.row; });
    return rows;
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
    std::stable_sort(items.begin(), items.end(), [](const WorkItem &a, const WorkItem &b) { return block_count(a) > block_count(b); });
    const long long most = (long long)p->sm_count * (p->head_dim == 32 ? 6 : 9) / 2;
    for (const bool backward : {false, true}) {
        std::vector<WorkItem> mine = items;
        Fp32Work &w = backward ? p->f32_bwd : p->f32_fwd;
        const std::vector<Fp32Row> rows = take_short_rows(p, mine, most, fp32_cost(p->head_dim, backward), w);
        w.n_rows = (int)rows.size();
        p->cuts[backward][0] = w.n_split > 0 ? w.cluster : 1;
        p->cuts[backward][1] = w.n_split;
        p->cuts[backward][2] = w.n_split > 0 ? 1 : 0;
        image.add(mine, &w.items);
        image.add(rows, &w.rows);
    }
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

template <int D>
static int launch_fwd(const hilberta_plan_t *p, const float *q, const float *k, const float *v, float *out, float *lse,
                      const int *out_map, const int *in_map, cudaStream_t stream) {
    const Fp32Work &w = p->f32_fwd;
    const int bhs = p->batch * p->heads;
    const long long ctas = items_grid(w, bhs);
    if (ctas > 0x7fffffffll) return HILBERTA_ERR_INVALID;
    if (ctas > 0) {
        HB_CUDA(launch_overlapping(attn_fp32_kernel<D>, (unsigned)ctas, kThreads, fwd_smem<D>(), (unsigned)w.cluster, stream,
                                   may_overlap(p, ctas), q, k, v, out, p->stride_b, p->stride_h, p->stride_s, p->heads, bhs, p->S,
                                   w.items, w.n_items, w.n_split, w.cluster, out_map, in_map, lse, p->scale));
        HB_LAUNCHED();
    }
    if (w.n_rows > 0) {
        HB_CUDA(launch_overlapping(attn_fp32_rows_kernel<D>, dim3((w.n_rows + kRowsPerCta - 1) / kRowsPerCta, bhs), kThreads, 0, 1,
                                   stream, true, q, k, v, out, p->stride_b, p->stride_h, p->stride_s, p->heads, p->S, p->P,
                                   w.rows, w.n_rows, out_map, in_map, lse, p->scale));
        HB_LAUNCHED();
    }
    return HILBERTA_OK;
}

int launch_attn_fp32(const hilberta_plan_t *p, const void *q, const void *k, const void *v, void *out,
                     float *lse, const int *out_map, const int *in_map, cudaStream_t stream, int slice) {
    const uintptr_t bits = (uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out;
    if ((bits & 15) || ((p->stride_b | p->stride_h | p->stride_s) & 3)) return HILBERTA_ERR_INVALID;
    if (slice >= 0) return HILBERTA_ERR_INVALID;   // fp32 bindings have no slices of heads
    switch (p->head_dim) {
        case 32: return launch_fwd<32>(p, (const float *)q, (const float *)k, (const float *)v, (float *)out, lse, out_map, in_map, stream);
        case 64: return launch_fwd<64>(p, (const float *)q, (const float *)k, (const float *)v, (float *)out, lse, out_map, in_map, stream);
        case 128: return launch_fwd<128>(p, (const float *)q, (const float *)k, (const float *)v, (float *)out, lse, out_map, in_map, stream);
        default: return HILBERTA_ERR_UNSUPPORTED;
    }
}

}  // namespace hilberta
