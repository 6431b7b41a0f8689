// Host-side work lists and static schedules shared by the tensor-core kernels.
//
// A work item is a run of consecutive physical rows that share one list of up to three
// contiguous ranges (prefix, tile range, wrapped tile range -- or the whole sequence for
// prefix rows).  The forward kernel keeps the rows resident as queries and streams the
// ranges as keys; the backward kernels use the same lists in both directions, because the
// mask is symmetric (Sec. 3.2 / 3.3).  Every (item, batch * head) unit is assigned to a CTA on
// the host, longest units first onto the least-loaded CTA, and stored grouped by CTA.
#include <algorithm>
#include <functional>
#include <utility>

#include "common.cuh"

namespace hilberta {

static void add_items(std::vector<WorkItem> &items, int row0, int rows, int item_rows, int block, int n_seg,
                      const int *seg_start, const int *seg_len) {
    for (int r = 0; r < rows; r += item_rows) {
        WorkItem it{};
        it.q_start = row0 + r;
        it.q_rows = std::min(item_rows, rows - r);
        it.n_seg = 0;
        it.kv_blocks = 0;
        for (int s = 0; s < n_seg; ++s) {
            if (seg_len[s] <= 0) continue;
            it.seg_start[it.n_seg] = seg_start[s];
            it.seg_len[it.n_seg] = seg_len[s];
            it.kv_blocks += (seg_len[s] + block - 1) / block;
            ++it.n_seg;
        }
        items.push_back(it);
    }
}

// Prefix rows see the whole sequence; the rows of each slid tile see the prefix and the
// tile's own one or two ranges.  item_rows: resident rows per item; block: streamed rows per
// block (kv_blocks counts them).
std::vector<WorkItem> build_work_items(const hilberta_plan_t *p, int item_rows, int block) {
    std::vector<WorkItem> items;
    {
        const int st[1] = {0}, ln[1] = {p->S};
        add_items(items, 0, p->P, item_rows, block, 1, st, ln);
    }
    for (const Window &w : p->h_windows) {
        const int st[3] = {0, w.seg0_start, w.seg1_start};
        const int ln[3] = {p->P, w.seg0_len, w.seg1_len};
        if (w.seg0_len > 0) add_items(items, w.seg0_start, w.seg0_len, item_rows, block, 3, st, ln);
        if (w.seg1_len > 0) add_items(items, w.seg1_start, w.seg1_len, item_rows, block, 3, st, ln);
    }
    return items;
}

// Every kernel reads the key ranges and query rows of its work items without further checks, so the
// lists are validated on the host before anything is uploaded (the shares of cut items by check_shares): each item's rows and key ranges lie
// inside [0, S), its key ranges do not overlap, its block count matches them, and the items' query
// ranges cover [0, S) exactly once.
int check_work_items(const WorkItem *items, int n, int S, int item_rows, int block) {
    if (n < 0 || S < 0 || item_rows < 1 || block < 1 || (n > 0 && !items)) return HILBERTA_ERR_INVALID;
    std::vector<std::pair<int, int>> rows;   // (q_start, q_rows)
    rows.reserve((size_t)n);
    for (int i = 0; i < n; ++i) {
        const WorkItem &it = items[i];
        if (it.q_rows < 1 || it.q_rows > item_rows || it.q_start < 0 || it.q_start > S - it.q_rows)
            return HILBERTA_ERR_INVALID;
        if (it.n_seg < 1 || it.n_seg > 3) return HILBERTA_ERR_INVALID;
        long long blocks = 0;
        for (int a = 0; a < it.n_seg; ++a) {
            if (it.seg_len[a] < 1 || it.seg_start[a] < 0 || it.seg_start[a] > S - it.seg_len[a])
                return HILBERTA_ERR_INVALID;
            blocks += (it.seg_len[a] + block - 1) / block;
            for (int b = 0; b < a; ++b)
                if (it.seg_start[a] < it.seg_start[b] + it.seg_len[b] && it.seg_start[b] < it.seg_start[a] + it.seg_len[a])
                    return HILBERTA_ERR_INVALID;   // a key would be counted twice
        }
        if (blocks != it.kv_blocks) return HILBERTA_ERR_INVALID;
        rows.push_back(std::make_pair(it.q_start, it.q_rows));
    }
    std::sort(rows.begin(), rows.end());
    int next = 0;
    for (const std::pair<int, int> &r : rows) {
        if (r.first != next) return HILBERTA_ERR_INVALID;   // a gap or an overlap between items
        next = r.first + r.second;
    }
    return next == S ? HILBERTA_OK : HILBERTA_ERR_INVALID;
}

// The same for the shares of cut items (cluster entries per item, in rank order): the rows of the item, and
// key ranges that make up the item's when read one after another, a block at least in every share.
int check_shares(const WorkItem *items, int n, const WorkItem *shares, int cluster, int block) {
    if (n < 0 || cluster < 1 || block < 1 || (n > 0 && (!items || !shares))) return HILBERTA_ERR_INVALID;
    for (int i = 0; i < n; ++i) {
        const WorkItem &it = items[i];
        int seg = 0, done = 0;   // the keys before position `done` of the item's range `seg` have been taken
        for (int r = 0; r < cluster; ++r) {
            const WorkItem &s = shares[i * cluster + r];
            if (s.q_start != it.q_start || s.q_rows != it.q_rows || s.n_seg < 1 || s.n_seg > 3) return HILBERTA_ERR_INVALID;
            long long blocks = 0;
            for (int a = 0; a < s.n_seg; ++a) {
                if (seg >= it.n_seg || s.seg_len[a] < 1 || s.seg_len[a] > it.seg_len[seg] - done ||
                    s.seg_start[a] != it.seg_start[seg] + done)
                    return HILBERTA_ERR_INVALID;
                done += s.seg_len[a];
                if (done == it.seg_len[seg]) {
                    ++seg;
                    done = 0;
                }
                blocks += (s.seg_len[a] + block - 1) / block;
            }
            if (blocks != s.kv_blocks) return HILBERTA_ERR_INVALID;
        }
        if (seg != it.n_seg) return HILBERTA_ERR_INVALID;   // keys that no share has
    }
    return HILBERTA_OK;
}

// ---------------------------------------------------------------------------
// Items cut over clusters.  A prefix item's key list is the whole sequence; with few heads a handful of
// them outlasts everything else (3 heads at 2048^2: 9 units of 132 blocks against 26 blocks per SM of
// work in all).  Such items are cut into one share per CTA of a cluster.
// ---------------------------------------------------------------------------

// Cost of merging a share, in the cost model's twentieths of a key block (1.45 us): the partial sums' way
// through shared memory and the waits for the cluster.  From one problem of five ten-block items on the
// B200: 22.7 us uncut, 21.3 in shares of two and 20.8 in shares of four, i.e. 6 and 8 us a merge.
static long long merge_cost(int cluster) { return cluster == 2 ? 85 : cluster == 4 ? 110 : 135; }

// Greedy assignment to the least loaded of n machines (of equally loaded ones the lowest number).  While machines are
// idle the next of them is the least loaded one, so the heap is built when the last one gets its first unit (built for the
// first unit that finds none idle: 0.2 us less of 6 for 54 units, 0.5 more of 12 for 432).  Plan, bind, export and destroy on
// a B200's host, a heap from the first unit on / this: 44 x 47 tokens, 2 x 12 heads 165 / 122 us, 64 x 64 + 512, 24 heads
// 221 / 184, 128 x 128 + 512 621 / 580.
struct LeastLoaded {
    typedef std::pair<long long, int> Load;   // (load, machine)
    std::vector<Load> heap;
    size_t idle = 0;   // machines from this number on are idle, and the heap is not one yet; heap.size(): it is
    explicit LeastLoaded(const std::vector<long long> &load) {
        heap.reserve(load.size());
        bool any = false;
        for (size_t i = 0; i < load.size(); ++i) {
            heap.push_back(Load(load[i], (int)i));
            any = any || load[i] != 0;
        }
        if (any) build();
    }
    void build() {
        std::make_heap(heap.begin(), heap.end(), std::greater<Load>());
        idle = heap.size();
    }
    // adds `cost` to the least loaded machine; returns its new load and its number
    Load add(long long cost) {
        const size_t n = heap.size();
        if (idle < n && cost > 0) {
            heap[idle].first = cost;
            const Load at = heap[idle];
            if (++idle == n) build();
            return at;
        }
        if (idle < n) build();
        const Load top(heap[0].first + cost, heap[0].second);
        size_t i = 0;
        for (;;) {   // sift the grown top down
            size_t c = 2 * i + 1;
            if (c >= n) break;
            if (c + 1 < n && heap[c + 1] < heap[c]) ++c;
            if (!(heap[c] < top)) break;
            heap[i] = heap[c];
            i = c;
        }
        heap[i] = top;
        return top;
    }
};

// The static schedule on the host: every (item, batch * head) unit -- items with a two-head cost as units of
// two consecutive indices -- goes, longest first, to the CTA with the smallest load so far.  With cut items
// every rank's list starts with the cut units of its cluster, in the same order.  units: grouped by CTA;
// cta_begin: n_cta + 1 offsets; both null: only the largest CTA load is wanted, which is returned.
// Aligned because its inner loop runs 40 % longer at odd multiples of 16 bytes, where code before it in the library
// may happen to put it (1680 units: 62 us at multiples of 32, 88 at the others).
__attribute__((aligned(64)))
long long build_schedule(const std::vector<long long> &cost, const std::vector<long long> &cost_two_heads, int bh, int sm_count,
                         const SplitChoice &ch, std::vector<WorkUnit> *units, std::vector<int> *cta_begin) {
    const int C = ch.cluster, n_items = (int)cost.size();
    // runs of equal units: of item i, for two heads each or for one, from head `first` on
    struct Run {
        long long cost;
        int item, first, count, step;
    };
    std::vector<Run> runs;
    long long n_units = (long long)ch.n_items * bh * C;
    for (int i = ch.n_items; i < n_items; ++i) {
        const long long two = ch.pair_heads && !cost_two_heads.empty() ? cost_two_heads[i] : 0;
        int j = 0;
        if (two > 0 && bh > 1) {
            runs.push_back(Run{two, i, 0, bh / 2, 2});
            j = bh / 2 * 2;
        }
        if (j < bh) runs.push_back(Run{cost[i], i, j, bh - j, 1});
        n_units += bh / 2 * (j > 0 ? 1 : 0) + (bh - j);
    }
    std::stable_sort(runs.begin(), runs.end(), [](const Run &a, const Run &b) { return a.cost > b.cost; });
    const int most = C > 1 ? ch.n_clusters * C : sm_count;
    const int n_cta = C > 1 ? (int)std::min<long long>((n_units + C - 1) / C * C, most) : (int)std::min<long long>(n_units, most);
    std::vector<int> cta_of;   // of every unit, in the order of assignment
    std::vector<WorkUnit> order;
    if (units) {
        cta_of.reserve((size_t)n_units);
        order.reserve((size_t)n_units);
    }
    long long makespan = 0;
    std::vector<long long> load((size_t)n_cta, 0);
    if (ch.n_items > 0) {
        LeastLoaded clusters(std::vector<long long>((size_t)(n_cta / C), 0));
        for (int i = 0; i < ch.n_items; ++i)
            for (int j = 0; j < bh; ++j) {
                const LeastLoaded::Load at = clusters.add((cost[i] + C - 1) / C + merge_cost(C) + ch.merge_extra);
                makespan = std::max(makespan, at.first);
                for (int r = 0; r < C; ++r) {
                    load[(size_t)(at.second * C + r)] = at.first;
                    if (units) {
                        order.push_back(WorkUnit{n_items + i * C + r, j, -2});
                        cta_of.push_back(at.second * C + r);
                    }
                }
            }
    }
    LeastLoaded ctas(load);
    for (const Run &run : runs)
        for (int k = 0; k < run.count; ++k) {
            const LeastLoaded::Load at = ctas.add(run.cost);
            makespan = std::max(makespan, at.first);
            if (units) {
                const int j = run.first + k * run.step;
                order.push_back(WorkUnit{run.item, j, run.step == 2 ? j + 1 : -1});
                cta_of.push_back(at.second);
            }
        }
    if (units) {
        cta_begin->assign((size_t)n_cta + 1, 0);
        for (int c : cta_of) ++(*cta_begin)[(size_t)c + 1];
        for (int c = 0; c < n_cta; ++c) (*cta_begin)[(size_t)c + 1] += (*cta_begin)[(size_t)c];
        std::vector<int> next(cta_begin->begin(), cta_begin->end() - 1);
        units->resize(order.size());
        for (size_t u = 0; u < order.size(); ++u) (*units)[(size_t)next[(size_t)cta_of[u]]++] = order[u];
    }
    return makespan;
}

// Blocks [lo, hi) of an item's key list as an item of its own (the same rows, part of the keys).
static WorkItem share_of(const WorkItem &it, int lo, int hi, int block) {
    WorkItem s = it;
    s.n_seg = 0;
    s.kv_blocks = hi - lo;
    for (int g = 0, b0 = 0; g < it.n_seg; ++g) {
        const int nb = (it.seg_len[g] + block - 1) / block;
        const int a = std::max(lo - b0, 0), e = std::min(hi - b0, nb);
        if (a < e) {
            s.seg_start[s.n_seg] = it.seg_start[g] + a * block;
            s.seg_len[s.n_seg] = std::min(it.seg_len[g], e * block) - a * block;
            ++s.n_seg;
        }
        b0 += nb;
    }
    for (int g = s.n_seg; g < 3; ++g) s.seg_start[g] = s.seg_len[g] = 0;
    return s;
}

int choose_split(const std::vector<WorkItem> &items, const std::vector<long long> &cost,
                 const std::vector<long long> &cost_two_heads, int bh, int sm_count, const int *clusters, int block,
                 SplitChoice &choice) {
    const long long merge_extra = choice.merge_extra;
    choice = SplitChoice();
    choice.merge_extra = merge_extra;
    long long total = 0, total_single = 0, n_units = 0, largest = 0;   // as scheduled without cuts, and a unit per head
    for (size_t i = 0; i < items.size(); ++i) {
        const int pairs = cost_two_heads[i] > 0 ? bh / 2 : 0;
        total += cost_two_heads[i] * pairs + cost[i] * (bh - 2 * pairs);
        total_single += cost[i] * bh;
        n_units += bh - pairs;
        largest = std::max(largest, pairs > 0 ? std::max(cost[i], cost_two_heads[i]) : cost[i]);
    }
    // Within 3 % of a perfect balance nothing is to be gained.  List scheduling is off by less than the largest
    // unit, so most large problems need no trial.
    if (n_units >= sm_count && largest * sm_count <= total / 32) return HILBERTA_OK;
    auto load_of = [&](const SplitChoice &c) {
        return build_schedule(cost, cost_two_heads, bh, sm_count, c, nullptr, nullptr);
    };
    long long best = load_of(choice);
    if (best * sm_count <= total + total / 32) return HILBERTA_OK;
    // (units per head instead of per two only matter where there are CTAs to take them)
    const bool few = n_units < 2ll * sm_count;
    if (few) {
        SplitChoice c = choice;
        c.pair_heads = false;   // idle CTAs: a unit per head is shorter than one for two
        const long long m = load_of(c);
        if (m < best) {
            best = m;
            choice = c;
        }
    }
    for (int k = 0; k < 3; ++k) {
        const int C = 2 << k;
        if (clusters[k] < 1) continue;
        SplitChoice c;
        c.merge_extra = merge_extra;
        c.cluster = C;
        c.n_clusters = clusters[k];
        // cut the items of the longest, of the two longest, ... lengths; every share gets a block at least
        int levels = 0;
        long long longest_share = 0;
        long long rest = total, rest_single = total_single, cut = 0;   // of the uncut units; of all shares
        for (int n = 1; n <= (int)items.size() && levels < (n_units > 16ll * sm_count ? 1 : 4); ++n) {
            if (items[n - 1].kv_blocks < C) break;
            const int pairs = cost_two_heads[n - 1] > 0 ? bh / 2 : 0;
            const long long share = (cost[n - 1] + C - 1) / C + merge_cost(C) + c.merge_extra;
            rest -= cost_two_heads[n - 1] * pairs + cost[n - 1] * (bh - 2 * pairs);
            rest_single -= cost[n - 1] * bh;
            cut += share * C * bh;
            longest_share = std::max(longest_share, share);
            if (n < (int)items.size() && items[n].kv_blocks == items[n - 1].kv_blocks) continue;
            ++levels;
            c.n_items = n;
            for (int pair = 1; pair >= (few ? 0 : 1); --pair) {
                // No schedule is shorter than the perfect balance, a share, or the longest item left: 4 trials instead of
                // 24 (128 x 128 tokens, 3 heads, both directions: 223 -> 122 us of a bind).
                const long long ctas = (long long)c.n_clusters * C;
                const long long least = std::max({((pair ? rest : rest_single) + cut + ctas - 1) / ctas, longest_share,
                                                  n < (int)items.size() ? cost[(size_t)n] : 0});
                if (least + least / 32 >= best) continue;
                c.pair_heads = pair != 0;
                const long long m = load_of(c);
                // clusters start together and merging is not free: only for a clear gain
                if (m + m / 32 < best) {
                    best = m;
                    choice = c;
                }
            }
        }
    }
    for (int i = 0; i < choice.n_items; ++i) {
        const int n = items[i].kv_blocks;
        for (int r = 0; r < choice.cluster; ++r)
            choice.shares.push_back(share_of(items[i], (int)((long long)n * r / choice.cluster),
                                             (int)((long long)n * (r + 1) / choice.cluster), block));
    }
    return check_shares(items.data(), choice.n_items, choice.shares.data(), choice.cluster, block);
}

// Adds the units grouped by CTA and the n_cta + 1 offsets to the image.
int add_schedule(BindImage &image, const std::vector<long long> &cost, const std::vector<long long> &cost_two_heads, int bh,
                 int sm_count, const SplitChoice &choice, WorkUnit **d_units, int **d_cta_begin, int *n_cta_out, int (*cuts)[3],
                 long long *largest_load) {
    if ((long long)cost.size() * bh > (1ll << 30)) return HILBERTA_ERR_INVALID;
    std::vector<WorkUnit> units;
    std::vector<int> cta_begin;
    const long long load = build_schedule(cost, cost_two_heads, bh, sm_count, choice, &units, &cta_begin);
    if (largest_load) *largest_load = load;
    *n_cta_out = (int)cta_begin.size() - 1;
    if (cuts) {
        (*cuts)[0] = choice.cluster;
        (*cuts)[1] = choice.n_items;
        (*cuts)[2] = 0;
        for (int c = 0; c < *n_cta_out; ++c) {
            int n = cta_begin[c];
            while (n < cta_begin[c + 1] && units[n].bh2 == -2) ++n;
            (*cuts)[2] = std::max((*cuts)[2], n - cta_begin[c]);
        }
    }
    image.add(units, d_units);
    image.add(cta_begin, d_cta_begin);
    return HILBERTA_OK;
}

}  // namespace hilberta

static_assert(sizeof(hilberta::WorkItem) == 10 * sizeof(int32_t), "hilberta_check_work_list takes ten ints per item");

extern "C" int hilberta_check_work_list(const int32_t *items, int n_items, int S, int item_rows, int block) {
    return hilberta::guarded(
        [&] { return hilberta::check_work_items(reinterpret_cast<const hilberta::WorkItem *>(items), n_items, S, item_rows, block); });
}

static_assert(sizeof(hilberta::WorkUnit) == 3 * sizeof(int32_t), "hilberta_schedule_units writes three ints per unit");

extern "C" int hilberta_schedule_units(int n_items, const int64_t *cost, const int64_t *cost_two_heads, int bh, int n_cta,
                                       int32_t *units, int32_t *cta_begin, int64_t *largest_load) {
    if (n_items < 0 || bh < 1 || n_cta < 1 || (n_items > 0 && !cost) || !units || !cta_begin) return HILBERTA_ERR_INVALID;
    if ((long long)n_items * bh > (1ll << 30)) return HILBERTA_ERR_INVALID;
    return hilberta::guarded([&] {
        std::vector<long long> c1(cost, cost + n_items), c2;
        if (cost_two_heads) c2.assign(cost_two_heads, cost_two_heads + n_items);
        std::vector<hilberta::WorkUnit> u;
        std::vector<int> cb;
        const long long m = hilberta::build_schedule(c1, c2, bh, n_cta, hilberta::SplitChoice(), &u, &cb);
        for (size_t i = 0; i < u.size(); ++i) {
            units[3 * i] = u[i].item;
            units[3 * i + 1] = u[i].bh;
            units[3 * i + 2] = u[i].bh2;
        }
        for (int c = 0; c <= n_cta; ++c) cta_begin[c] = c < (int)cb.size() ? cb[c] : (int)u.size();
        if (largest_load) *largest_load = m;
        return HILBERTA_OK;
    });
}

extern "C" int hilberta_check_shares(const int32_t *items, int n_items, const int32_t *shares, int cluster, int block) {
    return hilberta::check_shares(reinterpret_cast<const hilberta::WorkItem *>(items), n_items,
                                  reinterpret_cast<const hilberta::WorkItem *>(shares), cluster, block);
}

extern "C" int hilberta_cut_schedule(const int32_t *items, int n_items, const int64_t *cost, const int64_t *cost_two_heads,
                                     int bh, int sm_count, const int32_t *clusters, int block, int64_t merge_extra,
                                     int32_t *chosen, int32_t *shares, int32_t *units, int max_units, int32_t *cta_begin,
                                     int64_t *largest_load) {
    if (n_items < 1 || bh < 1 || sm_count < 1 || block < 1 || !items || !cost || !clusters || !chosen || !shares || !units ||
        !cta_begin || (long long)n_items * bh > (1ll << 27))
        return HILBERTA_ERR_INVALID;
    for (int k = 0; k < 3; ++k)
        if ((long long)clusters[k] << (k + 1) > sm_count) return HILBERTA_ERR_INVALID;
    return hilberta::guarded([&] {
        const hilberta::WorkItem *list = reinterpret_cast<const hilberta::WorkItem *>(items);
        const std::vector<hilberta::WorkItem> its(list, list + n_items);
        std::vector<long long> c1(cost, cost + n_items), c2((size_t)n_items, 0);
        if (cost_two_heads) c2.assign(cost_two_heads, cost_two_heads + n_items);
        hilberta::SplitChoice choice;
        choice.merge_extra = merge_extra;
        const int rc = hilberta::choose_split(its, c1, c2, bh, sm_count, clusters, block, choice);
        if (rc != HILBERTA_OK) return rc;
        std::vector<hilberta::WorkUnit> u;
        std::vector<int> cb;
        const long long m = hilberta::build_schedule(c1, c2, bh, sm_count, choice, &u, &cb);
        if ((int)u.size() > max_units) return HILBERTA_ERR_BUFFER;
        memcpy(units, u.data(), sizeof(hilberta::WorkUnit) * u.size());
        if (!choice.shares.empty()) memcpy(shares, choice.shares.data(), sizeof(hilberta::WorkItem) * choice.shares.size());
        for (int c = 0; c <= sm_count; ++c) cta_begin[c] = c < (int)cb.size() ? cb[c] : (int)u.size();
        chosen[0] = choice.cluster;
        chosen[1] = choice.n_items;
        chosen[2] = (int)cb.size() - 1;
        if (largest_load) *largest_load = m;
        return HILBERTA_OK;
    });
}
