// Entry / exit row gathers of Sec. 3.4: HBM-bound copies of whole token rows
// through an index table.  Both directions are written as gathers (reads are
// indirect, writes are sequential), with 16-byte accesses and four independent
// loads in flight per thread; the grid covers the tensor in one pass (a capped grid whose
// threads loop a second, partly filled time lost 20 % of the copy bandwidth).
#include "common.cuh"

namespace hilberta {

constexpr int kGatherThreads = 256;
constexpr int kGatherUnroll = 4;
// Gathers of up to this many bytes may overlap the kernel before them.  They run for a few microseconds each,
// and launch latency is part of that; large ones that run into one another leave the forward after them less of
// K and V in L2.  Three gathers and a forward, overlapping / plain, by the bytes of one gather (B200, us): 2 MB 21.6 /
// 27.8, 5 MB 31.3 / 32.9, 13 MB 89 / 97, 28 MB 158 / 160, 33 MB 182.6 / 182.3, 47 MB 257.8 / 257.2, 52 MB (e4m3) 438 / 441,
// 52 MB (head dim 64) 421 / 423, 70 MB 374 / 369, 104 MB 625 / 612, 415 MB 4190 / 4120.
constexpr size_t kOverlapBytes = 32u << 20;

// n / d for n < 2^31 by a multiplication (Granlund and Montgomery, 1994): with s = ceil(log2 d),
// q = (mulhi(n, floor(2^32 (2^s - d) / d) + 1) + n) >> s.
struct Divider {
    unsigned d, mul, shift;
    explicit Divider(int div)
        : d((unsigned)div), mul(0), shift(div > 1 ? 32 - __builtin_clz((unsigned)div - 1) : 0) {
        mul = (unsigned)(((((unsigned long long)1 << shift) - d) << 32) / d + 1);
    }
    __device__ __forceinline__ unsigned quotient(unsigned n) const { return (__umulhi(n, mul) + n) >> shift; }
};

// dst[b, r, :] = src[b, index[r], :]; a row is vecs.d 16-byte vectors, a batch item rows.d rows.  Bound by HBM, and below
// some 30 MB by its chain of launch, index load, vector load and store.  A block copies kGatherThreads * kGatherUnroll
// consecutive vectors of dst: where its first one lies takes 64-bit divisions, the others follow from it with two
// multiplications each, and everything before the vector loads precedes the wait for the kernel before.  Three
// gathers in a row (B200, us, with two 64-bit divisions a vector / now): 13 MB each 22.5 / 17.6, 28 MB 32.6 / 29.7, 52 MB in
// rows of 3 KB 68.1 / 61.5, 104 MB 104.7 / 104.9, 405 MB 382 / 370 (6.6 TB/s).
__global__ void __launch_bounds__(kGatherThreads)
row_gather_kernel(const uint4 *__restrict__ src, uint4 *__restrict__ dst, const int *__restrict__ index,
                  Divider rows, Divider vecs, long long total) {
    allow_next();
    const long long first = (long long)blockIdx.x * (kGatherThreads * kGatherUnroll);
    const long long row0 = first / vecs.d, b0 = row0 / rows.d;
    const unsigned c0 = (unsigned)(first - row0 * vecs.d), r0 = (unsigned)(row0 - b0 * rows.d);
    long long from[kGatherUnroll];
#pragma unroll
    for (int u = 0; u < kGatherUnroll; ++u) {
        const unsigned i = u * kGatherThreads + threadIdx.x, n = c0 + i;
        unsigned r = vecs.quotient(n);
        const unsigned c = n - r * vecs.d;
        r += r0;
        const unsigned b = rows.quotient(r);
        r -= b * rows.d;
        from[u] = first + i < total ? ((b0 + b) * rows.d + __ldg(index + r)) * vecs.d + c : -1;
    }
    wait_for_previous();
    uint4 val[kGatherUnroll];
#pragma unroll
    for (int u = 0; u < kGatherUnroll; ++u)
        if (from[u] >= 0) val[u] = __ldcs(src + from[u]);
    uint4 *out = dst + first + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kGatherUnroll; ++u)
        if (from[u] >= 0) __stcs(out + u * kGatherThreads, val[u]);
}

static int gather(const void *src, void *dst, const int *index, const hilberta_plan_t *p, int batch,
                  int row_elems, int dtype, cudaStream_t stream) {
    if (!p || !src || !dst || batch < 1 || row_elems < 1) return HILBERTA_ERR_INVALID;
    if (dtype != HILBERTA_BF16 && dtype != HILBERTA_FP32 && dtype != HILBERTA_FP8_E4M3) return HILBERTA_ERR_INVALID;
    int dev = -1;
    HB_CUDA(cudaGetDevice(&dev));
    if (dev != p->device) return HILBERTA_ERR_INVALID;  // the plan's tables live on another device
    const size_t esz = dtype == HILBERTA_BF16 ? 2 : dtype == HILBERTA_FP8_E4M3 ? 1 : 4;
    const size_t row_bytes = (size_t)row_elems * esz;
    if (row_bytes % 16 || ((uintptr_t)src & 15) || ((uintptr_t)dst & 15)) return HILBERTA_ERR_INVALID;
    const size_t bytes = row_bytes * (size_t)p->S * (size_t)batch;
    const char *a = (const char *)src, *b = (const char *)dst;
    if (a < b + bytes && b < a + bytes) return HILBERTA_ERR_INVALID;  // overlap
    const int vecs = (int)(row_bytes / 16);
    const long long total = (long long)batch * p->S * vecs;
    const long long blocks = (total + (long long)kGatherThreads * kGatherUnroll - 1) / ((long long)kGatherThreads * kGatherUnroll);
    if (blocks > 0x7fffffffll) return HILBERTA_ERR_INVALID;   // 35 TB
    HB_CUDA(launch_overlapping(row_gather_kernel, (unsigned)blocks, kGatherThreads, 0, 1, stream, bytes <= kOverlapBytes, (const uint4 *)src, (uint4 *)dst,
                               index, Divider(p->S), Divider(vecs), total));
    HB_LAUNCHED();
    return HILBERTA_OK;
}

}  // namespace hilberta

extern "C" int hilberta_permute(const void *src, void *dst, const hilberta_plan_t *plan, int batch,
                                int row_elems, int dtype, void *stream) {
    return hilberta::gather(src, dst, plan ? plan->d_phys2orig : nullptr, plan, batch, row_elems, dtype,
                            (cudaStream_t)stream);
}

extern "C" int hilberta_unpermute(const void *src, void *dst, const hilberta_plan_t *plan, int batch,
                                  int row_elems, int dtype, void *stream) {
    return hilberta::gather(src, dst, plan ? plan->d_orig2phys : nullptr, plan, batch, row_elems, dtype,
                            (cudaStream_t)stream);
}
