// Register-tiled fp32 products shared by the fp32 forward and backward kernels (plain FMA: the tensor
// cores' fp32 modes round operands to tf32 and could not meet a 1e-5 tolerance).
//
// A CTA of 4 warps owns 64 resident rows (16 per warp) and walks its key list in blocks of 32 rows.
// Lane L of a warp has rows {4 i + L / 8, i < 4} of the warp's sixteen and, of a 32-wide block, columns
// {8 j + L % 8, j < 4}: a row of scores belongs to 8 lanes of ONE warp, so row statistics are three
// shuffles and the weights go through shared memory without a CTA-wide barrier.  Shared memory is the
// pipe to watch: a 16-byte load of a warp takes at least two wavefronts however few addresses it has and
// four with 16 distinct ones, so lanes as 4 x 8 (two wavefronts each, 16 per 16 cycles of the SM's 128 FMA
// lanes in the scores, 24 per 32 in the accumulation) beat 2 x 16 (24 per 16 in both).
// Tiles are padded by 16 bytes a row: consecutive rows start in consecutive 16-byte banks.
#pragma once
#include "common.cuh"

namespace hilberta {
namespace fp32t {

constexpr int kThreads = 128;
constexpr int BR = 64;          // resident rows per CTA
constexpr int BC = 32;          // streamed rows per block
constexpr int PS = 40;          // floats per row of the weights' tile: four rows are 8 banks apart
__host__ __device__ constexpr int res_floats(int D) { return BR * (D + 4); }   // resident tile
__host__ __device__ constexpr int blk_floats(int D) { return BC * (D + 4); }   // streamed tile

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// every thread of every CTA of the cluster arrives and waits
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void *p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ float peer_ld(uint32_t a) {
    float x;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
    return x;
}
__device__ __forceinline__ float4 peer_ld4(uint32_t a) {
    float4 x;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(a) : "memory");
    return x;
}

// A work item's key list seen as one sequence: position f -> physical row.  Blocks of 32 may straddle
// the ranges, so only the last block of the list is ragged.
struct KeyList {
    int len[3], start[3], total;
    __device__ __forceinline__ explicit KeyList(const WorkItem &it) {
        total = 0;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            len[s] = s < it.n_seg ? it.seg_len[s] : 0;
            start[s] = it.seg_start[s];
            total += len[s];
        }
    }
    __device__ __forceinline__ int row(int f) const {
        if (f < len[0]) return start[0] + f;
        f -= len[0];
        return f < len[1] ? start[1] + f : start[2] + (f - len[1]);
    }
};

// What a CTA does: the first n_split items are cut over the `parts` CTAs of a cluster (contiguous shares
// of their blocks, merged through distributed shared memory), each of the others has a CTA of its own.
// `columns` instances of every item (batch * heads, times the directions of the backward pass) follow
// each other, so that the grid starts with the longest items of all of them: with the instances
// outermost the last one's prefix rows started when the rest of the chip was done, and half of it idled.
struct Share {
    int item, column, rank, parts;
    __device__ __forceinline__ Share(int n_items, int n_split, int cluster, int columns) {
        const unsigned x = blockIdx.x, split = (unsigned)n_split * columns * cluster;
        unsigned u;
        if (x < split) {
            u = x / cluster;
            rank = cluster > 1 ? (int)cluster_rank() : 0;
            parts = cluster;
        } else {
            u = (unsigned)n_split * columns + (x - split);
            rank = 0;
            parts = 1;
        }
        item = u / columns;
        column = u % columns;
        if (item >= n_items) item = -1;   // grid rounded up to whole clusters
    }
};

// acc[i][j] = rows i of A . rows j of B over the head dim; even and odd head-dim values accumulate
// apart (packed fp32x2 multiply-adds), which also halves the length of the rounding chains.
template <int D>
__device__ __forceinline__ void dot_tile(float (&x)[4][4], const float *a, const float *b) {
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int d = 0; d < D; d += 4) {
        float4 u[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) u[i] = *reinterpret_cast<const float4 *>(a + (4 * i) * (D + 4) + d);
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4 *>(b + (8 * j) * (D + 4) + d);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[i][j] = __ffma2_rn(make_float2(u[i].x, u[i].y), make_float2(w[j].x, w[j].y), acc[i][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[i][j] = __ffma2_rn(make_float2(u[i].z, u[i].w), make_float2(w[j].z, w[j].w), acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) x[i][j] = acc[i][j].x + acc[i][j].y;
}

// o[i][c] = o[i][c] * f[i] + sum over the block's 32 rows of w[row i][n] * t[n][column c], column
// 32 (c / 4) + 4 cg + c % 4 of the head dim.  The block's sum is taken on its own and added once, which
// keeps every rounding chain short; head dims above 64 go in two passes to bound the registers.
template <int D>
__device__ __forceinline__ void acc_tile(float (&o)[4][D / 8], const float (&f)[4], const float *w, const float *t, int cg) {
    constexpr int C = D / 8 < 8 ? D / 8 : 8;
#pragma unroll
    for (int c0 = 0; c0 < D / 8; c0 += C) {
        float acc[4][C];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < C; ++c) acc[i][c] = 0.f;
#pragma unroll 2
        for (int n = 0; n < BC; n += 4) {
            float4 p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4 *>(w + (4 * i) * PS + n);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float v[C];
#pragma unroll
                for (int g = 0; g < C / 4; ++g) {
                    const float4 y = *reinterpret_cast<const float4 *>(t + (n + e) * (D + 4) + 8 * c0 + 32 * g + 4 * cg);
                    v[4 * g] = y.x;
                    v[4 * g + 1] = y.y;
                    v[4 * g + 2] = y.z;
                    v[4 * g + 3] = y.w;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float pe = e == 0 ? p[i].x : e == 1 ? p[i].y : e == 2 ? p[i].z : p[i].w;
#pragma unroll
                    for (int c = 0; c < C; ++c) acc[i][c] = fmaf(pe, v[c], acc[i][c]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < C; ++c) o[i][c0 + c] = fmaf(o[i][c0 + c], f[i], acc[i][c]);
    }
}

// a lane's columns of one row (see acc_tile)
template <int D>
__device__ __forceinline__ void store_cols(float *row, int cg, const float (&v)[D / 8]) {
#pragma unroll
    for (int g = 0; g < D / 32; ++g)
        *reinterpret_cast<float4 *>(row + 32 * g + 4 * cg) = make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
}

// Resident rows [row0, row0 + rows) of a tensor into a padded tile; rows beyond are zero.
template <int D>
__device__ __forceinline__ void load_rows(float *tile, const float *base, long long stride_s, int row0, int rows, const int *map) {
    constexpr int V = D / 4;
    for (int e = threadIdx.x; e < BR * V; e += kThreads) {
        const int r = e / V, c = e % V;
        const bool in = r < rows;
        const int pr = in ? row0 + r : row0;
        cp_async16(tile + r * (D + 4) + 4 * c, base + (long long)(map ? map[pr] : pr) * stride_s + 4 * c, in);
    }
}

// Block j of a key list into a padded tile; rows beyond the list are zero.
template <int D>
__device__ __forceinline__ void load_block(float *tile, const float *base, long long stride_s, const KeyList &kl, int j, const int *map) {
    constexpr int V = D / 4;
#pragma unroll
    for (int i = 0; i < BC * V / kThreads; ++i) {
        const int e = threadIdx.x + i * kThreads;
        const int r = e / V, c = e % V;
        const int f = j * BC + r;
        const bool in = f < kl.total;
        const int pr = kl.row(in ? f : 0);
        cp_async16(tile + r * (D + 4) + 4 * c, base + (long long)(map ? map[pr] : pr) * stride_s + 4 * c, in);
    }
}

// Rows whose key lists are so short that a CTA of 64 is not worth while have a warp each, kRowsPerCta to a CTA.
constexpr int kRowsPerCta = kThreads / 32;
struct SingleRow {
    int row;   // < 0: none left
    int start[3], len[3];
    __device__ __forceinline__ SingleRow(const Fp32Row *rows, int n_rows, int P, int at) {
        const Fp32Row r = rows[min(at, n_rows - 1)];
        row = at < n_rows ? r.row : -1;
        start[0] = 0;
        len[0] = P;
        start[1] = r.seg0_start;
        len[1] = r.seg0_len;
        start[2] = r.seg1_start;
        len[2] = r.seg1_len;
    }
};

// CTAs of a launch over the items: `columns` instances of each, whole clusters.
inline long long items_grid(const Fp32Work &w, long long columns) {
    const long long c = w.cluster, single = (w.n_items - w.n_split) * columns;
    return w.n_split * columns * c + (single + c - 1) / c * c;
}

// Several CTAs of these kernels share an SM.  One that is set up while the kernel before it still runs goes
// where there is room and not where the load is even.  Four layers, overlapping / in turn (B200, us): 80 CTAs 46 /
// 49, 96 34.7 / 35.7, 112 of head dim 128 68 / 62, 200 of 128 83 / 86, 264 of 32 305 / 230, 352 98 / 80 and 86 / 75,
// 384 49.5 / 49.5, 410 1510 / 1243, 608 142 / 145 and 213 / 201: up to the line it gains, beyond it mostly loses.
inline bool may_overlap(const hilberta_plan_t *p, long long ctas) { return 5 * ctas <= 3 * p->sm_count; }

}  // namespace fp32t
}  // namespace hilberta
