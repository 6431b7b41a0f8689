// Internal definitions shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <atomic>
#include <new>
#include <vector>

#include "hilberta.h"

namespace hilberta {

extern thread_local int g_last_cuda_error;
extern std::atomic<uint64_t> g_launches;

#define HB_CUDA(expr)                                  \
    do {                                               \
        cudaError_t e__ = (expr);                      \
        if (e__ != cudaSuccess) {                      \
            ::hilberta::g_last_cuda_error = (int)e__;  \
            return HILBERTA_ERR_CUDA;                  \
        }                                              \
    } while (0)

#define HB_LAUNCHED()                                  \
    do {                                               \
        ::hilberta::g_launches.fetch_add(1);           \
        HB_CUDA(cudaGetLastError());                   \
    } while (0)

// The body of a C entry point that builds tables on the host: no exception leaves the library (the containers throw
// when memory runs out or a size is beyond them, nothing else here does).
template <class F>
int guarded(F body) noexcept {
    try {
        return body();
    } catch (...) {
        return HILBERTA_ERR_NOMEM;
    }
}

// One slid tile of the partition (Sec. 3.2) in physical coordinates: the
// non-shared members of Hilbert interval [lo, lo + tile) mod HW occupy seg0
// (the part starting at lo) and, if the interval wraps, seg1.
struct Window {
    int lo;
    int seg0_start, seg0_len;
    int seg1_start, seg1_len;
};

// One unit of work of the tensor-core kernel: up to `rows` consecutive physical
// query rows that share one key list of up to three contiguous ranges
// (prefix, seg0, seg1; or the whole sequence for prefix rows).
struct WorkItem {
    int q_start;
    int q_rows;
    int n_seg;
    int seg_start[3];
    int seg_len[3];
    int kv_blocks;  // sum over ranges of ceil(len / 128)
};

// A work item applied to one (batch, head).  Units are assigned to CTAs on the
// host (longest-processing-time-first) and stored grouped by CTA.  bh2 >= 0 (forward kernel
// only, items of one query tile): the same item for a second (batch, head), which takes the
// CTA's other query-tile slot with a K/V stream of its own.  bh2 == -2 (forward kernel in clusters): a
// share of an item's keys, the other shares being the same unit of the cluster's other CTAs.
struct WorkUnit {
    int item;
    int bh;
    int bh2;
};

// What one direction of an fp32 binding works through: items of up to 64 rows by descending key count, of
// which the first n_split are cut over clusters of `cluster` CTAs; and single rows, those of windows too short
// for an item of their own, with a warp each.
struct __align__(16) Fp32Row {
    int row, seg0_start, seg0_len, seg1_start, seg1_len, unused[3];   // the window's ranges by value: one trip to memory
};
struct Fp32Work {
    WorkItem *items;
    int n_items, n_split, cluster;
    Fp32Row *rows;
    int n_rows;
};

// How a schedule cuts its longest items (the first n_items of the list) over clusters of `cluster` CTAs;
// shares: cluster entries per cut item, in rank order, appended to the uploaded work list.
struct SplitChoice {
    int cluster = 1, n_clusters = 0, n_items = 0;
    bool pair_heads = true;
    long long merge_extra = 0;   // of a share, on top of what a forward merge costs
    std::vector<WorkItem> shares;
};

// Tables of a binding, gathered on the host: one allocation and one copy for all of them (every
// cudaMalloc, cudaFree and pageable copy is tens of microseconds of a bind).  `where` receives the device
// address; scratch lies behind the tables, uninitialised.
struct BindImage {
    std::vector<char> bytes;
    size_t scratch = 0;
    struct Place {
        void **where;
        size_t at;
        bool in_scratch;
    };
    std::vector<Place> places;
    static size_t up(size_t n) { return (n + 255) & ~(size_t)255; }
    template <class T>
    void add(const std::vector<T> &table, T **where) {
        const size_t at = bytes.size(), n = sizeof(T) * table.size();
        bytes.resize(up(at + n));
        if (n) memcpy(bytes.data() + at, table.data(), n);
        places.push_back(Place{(void **)where, at, false});
    }
    template <class T>
    void add_scratch(size_t count, T **where) {
        places.push_back(Place{(void **)where, scratch, true});
        scratch = up(scratch + sizeof(T) * count);
    }
};

}  // namespace hilberta

struct hilberta_plan_s {
    int device;
    int H, W, HW, k_log2;   // image grid; padded side n = 2^k_log2 >= max(H, W); HW = number of grid cells
    int frames, shared_frames;  // video volume: frames x H x W cells on a 3-D curve (frames == 1: an image)
    int ka_log2, kb_log2;       // video: frame axis padded to 2^ka, image axes to 2^kb
    int NP;                 // n * n: length of the padded Hilbert curve the tiles are cut on
    bool compact;           // tiles are equal groups over the non-shared tokens (Algorithm 1) instead of curve intervals
    int tile, offset, shared_region, n_text, n_shared, T, S, P;
    uint64_t nnz;
    // device tables: two allocations, made by the plan and by its binding; the pointers below point into them
    void *d_plan, *d_bind;
    size_t plan_bytes, bind_bytes;
    int *d_hil_d2t, *d_hil_t2d;      // [HW]
    int *d_c;                        // [NP + 1] real non-shared cells with padded Hilbert index below d
    int *d_phys2orig, *d_orig2phys;  // [S]
    hilberta::Window *d_windows;     // [T]
    // host mirrors of the small tables
    std::vector<hilberta::Window> h_windows;
    std::vector<int> h_shared_runs;  // (start, len) pairs
    // binding
    bool bound;
    int batch, heads, head_dim, dtype;
    int64_t stride_b, stride_h, stride_s;
    float scale;
    hilberta::WorkItem *d_work;
    int n_work;
    hilberta::WorkUnit *d_units;  // grouped by CTA: an (item, batch * head), two heads of an item, or a share of one
    int *d_cta_begin;             // [n_cta + 1]
    int n_cta;
    // The host-buffer entry point pipelines copies and launches over n_slices slices of heads (of all batch items): the
    // first heads % n_slices of them have a head more than the others, and a schedule of their own.
    int n_slices;
    // first head of slice c of n
    int slice_begin(int c, int n) const { return c * (heads / n) + (c < heads % n ? c : heads % n); }
    // The slices' schedules are made by the first host-buffer call (most bindings see none), in its workspace, from:
    std::vector<long long> fwd_cost, fwd_cost_two;
    hilberta::SplitChoice fwd_split;
    size_t slice_bytes;   // the most that they take
    bool slices_made;
    int split_cluster;            // CTAs per cluster of the forward launches (1: no clusters, no split units)
    long long fwd_load;           // largest CTA load of the forward schedule, in twentieths of a key block (1.45 us)
    hilberta::WorkUnit *d_units_slice[2];   // [1]: of the slices with a head more
    int *d_cta_begin_slice[2];
    int n_cta_slice[2];
    // the pair kernel's work list and schedule (bf16, head dim 128): items of 256 rows, one per
    // pair of SMs; n_pair == 0: the shape is served by the single-CTA kernel
    hilberta::WorkItem *d_work_pair;
    hilberta::WorkUnit *d_units_pair;
    int *d_pair_begin;
    int n_pair;
    // the one-tile kernel's work list and schedule (bf16, head dim 128): items of 128 rows
    hilberta::WorkItem *d_work_solo;
    hilberta::WorkUnit *d_units_solo;
    int *d_solo_begin;
    int n_solo;
    cudaStream_t s_in, s_out;           // copy streams of hilberta_forward_host (created on first use)
    std::vector<cudaEvent_t> ev_in, ev_done;
    // backward pass: 128-row items over the same key lists, their schedule, and the
    // per-row scratch (lse * log2 e, then delta = rowsum(dO * O)) that the backward kernel reads
    hilberta::WorkItem *d_bwd_work;
    int n_bwd_work;
    hilberta::WorkUnit *d_bwd_units;
    int *d_bwd_cta_begin;
    int n_bwd_cta, bwd_cluster;
    float *d_delta;               // [2 * batch * heads * S]
    hilberta::Fp32Work f32_fwd, f32_bwd;   // fp32 bindings
    int cuts[2][3];               // forward, backward: CTAs per cluster, cut items, the most cut units of a CTA
    int *d_status;  // [4] error word + diagnostics written by bounded waits
    // workspace of hilberta_forward_host
    void *ws;
    size_t ws_bytes;
    int sm_count;
};

namespace hilberta {

// Programmatic dependent launch: the library's kernels allow the next one in the stream to be set up while
// they drain (allow_next: once every CTA has said so), and each reads and writes nothing that an earlier
// kernel could still touch before wait_for_previous has returned -- until then only its plan's tables, which
// no kernel writes after the plan and its binding are made.  Every kernel launched this way waits (some thread
// of it at least) and the others are launched plainly, so a kernel's end implies the end of all before it.
// Saves the launch latency and the prologue between kernels, 1 ... 2 us each (one fused launch after another,
// 512^2 and 8 heads: 18.7 -> 16.6 us).  overlap = false: an ordinary launch.
__device__ __forceinline__ void allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... Params, class... Args>
cudaError_t launch_overlapping(void (*kernel)(Params...), dim3 grid, unsigned block, size_t smem, unsigned cluster,
                               cudaStream_t stream, bool overlap, const Args &...args) {
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t config{};
    config.gridDim = grid;
    config.blockDim = dim3(block);
    config.dynamicSmemBytes = smem;
    config.stream = stream;
    config.attrs = attr;
    config.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&config, kernel, Params(args)...);
}

// out_map: nullptr = write rows in physical order; else out_map[p] is the row of `out`
// that physical row p goes to (the exit gather fused into the epilogue).
// lse: nullptr, or [batch * heads, S] fp32 receiving log-sum-exp of the scaled logits
// (natural log), indexed like `out` rows.
// in_map: nullptr = q, k, v are in physical order; else they are in ORIGINAL order and physical
// row p is read from row in_map[p] (the entry gather fused into the loads).
// slice: -1 = the whole bound problem; c >= 0 = slice c of n_slices > 1, its heads
// of every batch item only (lse must be null then).
int launch_attn_fp32(const hilberta_plan_t *p, const void *q, const void *k, const void *v, void *out,
                     float *lse, const int *out_map, const int *in_map, cudaStream_t stream, int slice = -1);
int launch_attn_bf16(const hilberta_plan_t *p, const void *q, const void *k, const void *v, void *out,
                     float *lse, const int *out_map, const int *in_map, cudaStream_t stream, int slice = -1);
// schedule.cu: work lists (runs of item_rows rows with their up to three key ranges, counted in
// blocks of `block` rows) and the static longest-first assignment of (item, batch * head) units to CTAs
std::vector<WorkItem> build_work_items(const hilberta_plan_t *p, int item_rows, int block);
// HILBERTA_OK iff the list is safe to hand to a kernel (ranges inside [0, S), rows covered exactly once)
int check_work_items(const WorkItem *items, int n, int S, int item_rows, int block);
int check_shares(const WorkItem *items, int n, const WorkItem *shares, int cluster, int block);
// clusters: how many clusters of 2, 4 and 8 CTAs run at once.  items sorted by descending cost.  Of
// `choice` only merge_extra is read.  Not HILBERTA_OK: the shares are not safe to hand to a kernel.
int choose_split(const std::vector<WorkItem> &items, const std::vector<long long> &cost,
                 const std::vector<long long> &cost_two_heads, int bh, int sm_count, const int *clusters, int block,
                 SplitChoice &choice);
// The schedule of such a choice (units null: none is written); returns the largest CTA load.
// cost_two_heads: empty, or per item the cost of running it for TWO (batch, head) indices in one unit
// (0: the item is not paired); such items become units of two consecutive indices.
long long build_schedule(const std::vector<long long> &cost, const std::vector<long long> &cost_two_heads, int bh, int sm_count,
                         const SplitChoice &choice, std::vector<WorkUnit> *units, std::vector<int> *cta_begin);
int add_schedule(BindImage &image, const std::vector<long long> &cost, const std::vector<long long> &cost_two_heads, int bh,
                 int sm_count, const SplitChoice &choice, WorkUnit **d_units, int **d_cta_begin, int *n_cta_out,
                 int (*cuts)[3] = nullptr, long long *largest_load = nullptr);
// The forward kernel that the environment variable HILBERTA_FORWARD_KERNEL selects, read once: 'p' (pairs
// of SMs), 's' (one query tile per CTA) or 0 (the default kernel).
char forward_kernel_choice();
int attn_bf16_prepare(hilberta_plan_t *p, BindImage &image);
// makes the slices' schedules in slice_bytes bytes at `where`, on `stream`
int attn_bf16_make_slices(hilberta_plan_t *p, char *where, cudaStream_t stream);
// attn_bf16_pair_sm100.cu: the forward kernel on pairs of SMs (bf16, head dim 128, inputs in physical order)
int attn_bf16_pair_prepare(hilberta_plan_t *p, BindImage &image);
int launch_attn_bf16_pair(const hilberta_plan_t *p, const void *q, const void *k, const void *v, void *out,
                          float *lse, const int *out_map, cudaStream_t stream);
// attn_bf16_solo_sm100.cu: the forward kernel with one query tile per CTA and double-buffered scores
// (bf16, head dim 128, inputs in physical order)
int attn_bf16_solo_prepare(hilberta_plan_t *p, BindImage &image);
int launch_attn_bf16_solo(const hilberta_plan_t *p, const void *q, const void *k, const void *v, void *out,
                          float *lse, const int *out_map, cudaStream_t stream);
int attn_bwd_prepare(hilberta_plan_t *p, BindImage &image);
// dq, dk, dv (bf16, physical order, the bound strides) from dout, q, k, v, out and the forward's lse.
int launch_attn_bwd(const hilberta_plan_t *p, const void *dout, const void *q, const void *k, const void *v,
                    const void *out, const float *lse, void *dq, void *dk, void *dv, float *delta,
                    cudaStream_t stream);
int launch_attn_fp32_bwd(const hilberta_plan_t *p, const void *dout, const void *q, const void *k, const void *v,
                         const void *out, const float *lse, void *dq, void *dk, void *dv, float *delta,
                         cudaStream_t stream);
int attn_fp32_prepare(hilberta_plan_t *p, BindImage &image);
int attn_fp32_bwd_opt_in();   // shared-memory opt-in of the fp32 backward kernels on the current device
int launch_timeout_probe(const hilberta_plan_t *p, cudaStream_t stream);
// plan.cu: does a written tensor share a byte with another tensor of the bound layout?
bool bound_tensors_overlap(const hilberta_plan_t *p, const void *out, size_t esz_out, const void *in, size_t esz_in);
}  // namespace hilberta
