// Batched sampler: all trees of thousands of small graphs in one CUDA-graph
// launch.  Trees are pulled one by one from device counters by persistent
// kernels (no grid-wide barrier); a tree's words live in shared memory and a
// block of 32 to 256 threads runs it (lane_tree.cuh).  The graphs are sorted by size and cut into bins of about a
// factor of two, one kernel each, so that every bin gets the shared memory
// (and thus the occupancy) and the threads its own graphs need; the bins run
// on forked streams, and fork and join are captured into the call's CUDA
// graph, which is replayed.  The schedule sets the split between the classes of
// large and small graphs, the largest block of the large class and whether the
// small class runs one tree per warp; the autotuner times candidates.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "rwc_common.cuh"
#include "lane_tree.cuh"

namespace rwc {
namespace {

struct BGraph {
    int64_t voff;   // first vertex in the concatenated arrays
    int32_t n;
    int32_t root;
};

// Trees 0 .. npull - 1 of a bin, T of each of its graphs: pull i is tree i % T of
// graph order[i / T].  The blocks take them in turn, after their first from the
// counter `next` (NULL: every gridDim.x-th).  Every pull is a tree, so
// lane_tree's barriers lie between the reads of sh_next and its next write.
template <bool OFF64, bool W, int NT>
__global__ void __launch_bounds__(NT) l_batch(DevGraph base, const BGraph *__restrict__ graphs,
                                              const int32_t *__restrict__ order, int64_t npull, unsigned long long *next,
                                              int64_t T, uint32_t k0, uint32_t k1, int max_n, double *sums,
                                              uint32_t *spill, int *err, unsigned long long *ctr) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long sh_next;
    using Sh = LaneShared<NT, 1>;
    Sh &sh = *reinterpret_cast<Sh *>(smem);
    uint32_t *word = reinterpret_cast<uint32_t *>(smem + sizeof(Sh));
    uint32_t *sp = spill + (int64_t)blockIdx.x * max_n;
    unsigned long long draws = 0;
    uint32_t rounds = 0;
    int64_t i = blockIdx.x;
    while (i < npull) {
        const int32_t gid = order[i / T];
        const int64_t t = i % T;
        const BGraph bg = graphs[gid];
        DevGraph g = base;
        g.n = bg.n;
        g.root = bg.root;
        if (OFF64) g.rp64 = base.rp64 + bg.voff;
        else g.rp32 = base.rp32 + bg.voff;
        const int kb = lt_kbits<uint32_t>(bg.n, NT);
        for (int u = threadIdx.x; u < bg.n; u += NT) word[u] = u == bg.root ? lt_root_word<uint32_t>(kb, NT) : 0u;
        __syncthreads();
        const int bad = lane_tree<OFF64, W, 0, NT, 1, true, uint32_t>(g, word, kb, 65535u, sh, sp, (uint32_t)t,
                                                                      (uint32_t)gid, k0, k1, rounds);
        if (bad) { if (threadIdx.x == 0) atomicOr(err, bad); break; }
        const uint32_t kmask = (1u << kb) - 1u;
        double *out = sums + bg.voff;
        for (int u = threadIdx.x; u < bg.n; u += NT) {
            if (u == bg.root) continue;
            const uint32_t vis = (word[u] & kmask) + 1u;
            draws += vis;
            atomicAdd(out + u, (double)vis);
        }
        if (!next) { i += gridDim.x; continue; }
        if (threadIdx.x == 0) sh_next = atomicAdd(next, 1ull);
        __syncthreads();
        i = (int64_t)gridDim.x + (int64_t)sh_next;
    }
    for (int o = 16; o > 0; o >>= 1) draws += __shfl_xor_sync(0xffffffffu, draws, o);
    if ((threadIdx.x & 31) == 0 && draws) atomicAdd(ctr + 1, draws);
    if (threadIdx.x == 0 && rounds) atomicAdd(ctr, (unsigned long long)rounds);
}

// Threads per tree of graphs of up to n vertices: what keeps about 40 warps on
// an SM beside n words of shared memory per tree (21 blocks of 64 up to 2500
// vertices by registers, 10 of 128 up to 5000, 2 of 256 at 20000).  512 graphs
// of 50 to 20000 vertices, 64 trees each: 158 ms with whole-block popping
// rounds (11 bytes per vertex, one kernel for each of two classes), 18.8 ms so.
// Calls of at most one tree per SM take 256 threads for each, which nothing else would
// use (one tree: BA 5000 0.154 -> 0.116 ms a call; of each of 64 weighted BA graphs of
// 2000 vertices: 0.186 -> 0.132).  Up to 448 vertices more than a warp gains nothing.
bool few_trees(int64_t trees) { return trees <= num_sms(); }
int batch_threads(int n, bool few) { return few && n > 448 ? 256 : n <= 2500 ? 64 : n <= 5000 ? 128 : 256; }
// One launch per graph: one warp up to 448 vertices, whose rounds need no block barrier
// (30 paths of 60, 1 tree each: 18.7 ms, 23.8 with 64 threads).
int single_threads(int n, bool few) { return n <= 448 ? 32 : batch_threads(n, few); }

size_t batch_tree_smem(int n, int nt) {
    const size_t head = nt == 32 ? sizeof(LaneShared<32, 1>) : nt == 64 ? sizeof(LaneShared<64, 1>)
                      : nt == 128 ? sizeof(LaneShared<128, 1>) : sizeof(LaneShared<256, 1>);
    return head + (size_t)n * 4;
}

template <class F>
void dispatch(bool off64, bool weighted, F f) {
    if (off64) {
        if (weighted) f(std::true_type{}, std::true_type{});
        else f(std::true_type{}, std::false_type{});
    } else {
        if (weighted) f(std::false_type{}, std::true_type{});
        else f(std::false_type{}, std::false_type{});
    }
}

template <class F>
void dispatch_nt(bool off64, bool weighted, int nt, F f) {
    dispatch(off64, weighted, [&](auto o64, auto wt) {
        constexpr bool O = decltype(o64)::value, W = decltype(wt)::value;
        if (nt == 32) f(l_batch<O, W, 32>);
        else if (nt == 64) f(l_batch<O, W, 64>);
        else if (nt == 128) f(l_batch<O, W, 128>);
        else f(l_batch<O, W, 256>);
    });
}

constexpr int MAX_BINS = 12;

// Graphs of one kernel: a range of a class's list.
struct Bin {
    int cls;
    int64_t begin, count;   // graphs
    int max_n, nt;
    size_t smem;
    int64_t blocks;
    int64_t spill;          // its blocks' ends in global memory: offset in entries
};

}  // namespace
}  // namespace rwc

using namespace rwc;

struct rwc_batch {
    int32_t G = 0;
    int64_t N = 0, nnz = 0;
    bool off64 = false, weighted = false;
    std::vector<BGraph> hgraphs;
    std::vector<int32_t> roots;
    DevGraph base;                     // concatenated CSR (local column ids)
    BGraph *graphs = nullptr;
    // schedule: largest block of the large graphs, the largest n of the small
    // class (0: one class), small class warp-per-tree (1) or block-per-tree
    // (0); tile is kept for saved schedules, trees are pulled one by one
    int threads = 512;
    int split = 1024;
    int warp = 1;
    int tile = 4;
    int conc = 1;                      // 1: the classes run concurrently (forked streams)
    cudaStream_t side[MAX_BINS] = {};  // the bins' streams (forked from the call's), made with the bins
    cudaEvent_t fork = nullptr, join[MAX_BINS] = {};
    int32_t *items[2] = {nullptr, nullptr};   // each class's graphs, the largest first
    int max_n[2] = {0, 0};             // largest n of each class
    std::vector<Bin> bins;
    uint32_t *spill = nullptr;         // the bins' pending ends beyond shared memory
    // one launch per graph: graph ids 0 .. G - 1, each graph's resident blocks
    // (made on first use) and their pending ends beyond shared memory
    int32_t *single = nullptr;
    std::vector<int64_t> single_blocks;
    uint32_t *single_spill = nullptr;
    int64_t single_spill_n = 0;
    int64_t items_T = -1;              // T the bins were built for
    int64_t items_split = -1;
    void *scratch = nullptr;           // [0] err, [8] rounds, [16] draws, [64..160) the bins' counters
    std::vector<void *> allocs;
    // captured launches
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    uint64_t cap_seed = 0;
    int64_t cap_T = -1;
    double *cap_sums = nullptr;
    cudaStream_t cap_stream = nullptr;
    int64_t *host = nullptr;
};

namespace {

cudaError_t balloc(rwc_batch *b, void **p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes ? bytes : 16);
    if (e == cudaSuccess) b->allocs.push_back(*p);
    return e;
}

template <class T>
void bfree(rwc_batch *b, T *&p) {
    if (!p) return;
    cudaFree(p);
    b->allocs.erase(std::find(b->allocs.begin(), b->allocs.end(), (void *)p));
    p = nullptr;
}

void drop_graph(rwc_batch *b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    b->cap_T = -1;
}

void drop_streams(rwc_batch *b) {
    for (int i = 0; i < MAX_BINS; ++i) {
        if (b->join[i]) cudaEventDestroy(b->join[i]);
        if (b->side[i]) cudaStreamDestroy(b->side[i]);
    }
    if (b->fork) cudaEventDestroy(b->fork);
}

// The largest schedule a batch accepts: a tree counts 11 n + 64 bytes of shared
// memory, eight of them in a block where the small class runs warp-per-tree.
size_t tree_allowance(int64_t n) { return (size_t)n * 11 + 64; }
size_t schedule_allowance(int max_large, int max_small, int warp) {
    const size_t large = max_large ? tree_allowance(max_large) : 64;
    const size_t small = !max_small ? 64 : warp ? 8 * ((tree_allowance(max_small) + 15) & ~(size_t)15)
                                                : tree_allowance(max_small);
    return std::max(large, small);
}
size_t batch_smem(const rwc_batch *b) { return schedule_allowance(b->max_n[0], b->max_n[1], b->warp); }

// Blocks of nt threads and smem bytes that the device holds at once.
rwc_status resident_blocks(const rwc_batch *b, int nt, size_t smem, int64_t *out) {
    int per_sm = 0;
    cudaError_t e = cudaSuccess;
    dispatch_nt(b->off64, b->weighted, nt, [&](auto kern) {
        // one value for all batches: other threads launch the kernel too
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem);
    });
    RWC_CUDA_TRY(e);
    if (per_sm < 1) return set_error(RWC_ERR_UNSUPPORTED, "batch block does not fit on an SM");
    *out = (int64_t)num_sms() * per_sm;
    return RWC_OK;
}

// Resident blocks of each graph's own launch with many trees (with few there is a
// block for each tree; blocks of 256 threads whose words need more than the default 48
// KB are those of many trees too, so their kernels' limit is set here).
rwc_status plan_single(rwc_batch *b) {
    std::vector<int64_t> blocks(b->G);
    for (int32_t g = 0; g < b->G; ++g) {
        const int n = b->hgraphs[g].n, nt = single_threads(n, false);
        RWC_TRY(resident_blocks(b, nt, batch_tree_smem(n, nt), &blocks[g]));
    }
    b->single_blocks = std::move(blocks);
    return RWC_OK;
}

rwc_status build_bins(rwc_batch *b, const std::vector<int32_t> (&order)[2], int64_t T) {
    b->bins.clear();
    const bool few = few_trees(T * b->G);
    for (int c = 0; c < 2; ++c)
        for (size_t i = 0; i < order[c].size();) {
            const int top = b->hgraphs[order[c][i]].n;
            size_t j = i;
            while (j < order[c].size() && (top <= 640 || 2 * b->hgraphs[order[c][j]].n > top)) ++j;
            Bin q{};
            q.cls = c;
            q.begin = (int64_t)i;
            q.count = (int64_t)(j - i);
            q.max_n = top;
            q.nt = batch_threads(top, few);
            if (c == 1 && b->warp) q.nt = 32;
            while (c == 0 && q.nt > b->threads) q.nt /= 2;
            q.smem = batch_tree_smem(top, q.nt);
            b->bins.push_back(q);
            i = j;
        }
    if (b->bins.size() > (size_t)MAX_BINS) return set_error(RWC_ERR_UNSUPPORTED, "too many size bins");
    for (size_t i = 1; i < b->bins.size(); ++i) {
        if (!b->fork) RWC_CUDA_TRY(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming));
        if (!b->side[i]) RWC_CUDA_TRY(cudaStreamCreateWithFlags(&b->side[i], cudaStreamNonBlocking));
        if (!b->join[i]) RWC_CUDA_TRY(cudaEventCreateWithFlags(&b->join[i], cudaEventDisableTiming));
    }
    int64_t spill = 0;
    for (Bin &q : b->bins) {
        RWC_TRY(resident_blocks(b, q.nt, q.smem, &q.blocks));
        q.blocks = std::max<int64_t>(1, std::min<int64_t>(q.count * T, q.blocks));
        q.spill = spill;
        spill += q.blocks * q.max_n;
    }
    bfree(b, b->spill);
    RWC_CUDA_TRY(balloc(b, (void **)&b->spill, (size_t)spill * sizeof(uint32_t)));
    return RWC_OK;
}

// Bins for T trees per graph: list 0 holds graphs with more than `split`
// vertices, list 1 the others; each list runs its largest graphs first.
rwc_status build_items(rwc_batch *b, int64_t T) {
    if (b->items_T == T && b->items_split == b->split) return RWC_OK;
    // nothing built for another T or schedule is used again, whatever fails below
    b->items_T = -1;
    drop_graph(b);
    std::vector<int32_t> orders[2];
    for (int c = 0; c < 2; ++c) {
        std::vector<int32_t> &order = orders[c];
        for (int32_t g = 0; g < b->G; ++g) {
            const int cls = b->hgraphs[g].n <= b->split ? 1 : 0;
            if (cls == c) order.push_back(g);
        }
        std::stable_sort(order.begin(), order.end(),
                         [&](int32_t x, int32_t y) { return b->hgraphs[x].n > b->hgraphs[y].n; });
        bfree(b, b->items[c]);
        if (!order.empty()) {
            RWC_CUDA_TRY(balloc(b, (void **)&b->items[c], order.size() * sizeof(int32_t)));
            RWC_CUDA_TRY(cudaMemcpy(b->items[c], order.data(), order.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
        }
        b->max_n[c] = 0;
        for (int32_t g : order) b->max_n[c] = std::max(b->max_n[c], b->hgraphs[g].n);
    }
    RWC_TRY(build_bins(b, orders, T));
    b->items_T = T;
    b->items_split = b->split;
    return RWC_OK;
}

// Enqueue one call: the first bin on st, the others on the batch's side streams
// forked from st and joined back (conc = 0: all on st).
rwc_status enqueue(rwc_batch *b, uint64_t seed, int64_t T, double *sums, cudaStream_t st) {
    int *err = (int *)b->scratch;
    unsigned long long *ctr = (unsigned long long *)((char *)b->scratch + 8);
    unsigned long long *next = (unsigned long long *)((char *)b->scratch + 64);
    RWC_CUDA_TRY(cudaMemsetAsync(next, 0, MAX_BINS * sizeof(*next), st));
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    if (batch_smem(b) > 227 * 1024) return set_error(RWC_ERR_UNSUPPORTED, "batch schedule needs %zu bytes of shared memory", batch_smem(b));
    const bool fork = b->conc && b->bins.size() > 1;
    if (fork) RWC_CUDA_TRY(cudaEventRecord(b->fork, st));
    cudaError_t e = cudaSuccess;
    size_t forked = 0;
    for (size_t i = 0; i < b->bins.size() && e == cudaSuccess; ++i) {
        const Bin &q = b->bins[i];
        cudaStream_t s = st;
        if (fork && i > 0) {
            s = b->side[i];
            if ((e = cudaStreamWaitEvent(s, b->fork, 0)) != cudaSuccess) break;
            forked = i;
        }
        ::rwc::count_launches(1);
        dispatch_nt(b->off64, b->weighted, q.nt, [&](auto kern) {
            kern<<<(unsigned)q.blocks, q.nt, q.smem, s>>>(b->base, b->graphs, b->items[q.cls] + q.begin,
                                                          q.count * T, next + i, T, k0, k1, q.max_n, sums,
                                                          b->spill + q.spill, err, ctr);
        });
        e = cudaGetLastError();
    }
    // every forked stream joins st again, after an error too
    for (size_t i = 1; i <= forked; ++i) {
        const cudaError_t e1 = cudaEventRecord(b->join[i], b->side[i]);
        const cudaError_t e2 = cudaStreamWaitEvent(st, b->join[i], 0);
        if (e == cudaSuccess) e = e1 != cudaSuccess ? e1 : e2;
    }
    RWC_CUDA_TRY(e);
    return RWC_OK;
}

rwc_status finish(rwc_batch *b, rwc_stats_t *stats, int mode, int64_t T, cudaStream_t st) {
    RWC_CUDA_TRY(cudaMemcpyAsync(b->host, b->scratch, 24, cudaMemcpyDeviceToHost, st));
    RWC_CUDA_TRY(cudaStreamSynchronize(st));
    const int e = (int)(b->host[0] & 0xffffffff);
    if (e & LE_KOVF) return set_error(RWC_ERR_UNSUPPORTED, "a vertex was popped more than 65535 times");
    if (e) return set_error(RWC_ERR_CUDA, "sampler internal check failed");
    if (stats) {
        stats->trees = T * b->G;
        stats->rounds = b->host[1];
        stats->draws = b->host[2];
        stats->marked = b->host[2];
        stats->chunks = 1;
        stats->mode = mode;
        stats->block_threads = mode == 3 ? 0 : b->threads;   // the schedule's bound on the large class's blocks
    }
    return RWC_OK;
}

}  // namespace

extern "C" rwc_status rwc_batch_create(int32_t G, const int64_t *voff, const int64_t *rp,
                                       const int32_t *col, const float *w, rwc_batch_t **out) {
    clear_error();
    if (!out || G <= 0 || !voff || !rp || !col) return set_error(RWC_ERR_INVALID, "bad argument");
    *out = nullptr;
    if (voff[0] != 0) return set_error(RWC_ERR_INVALID, "graph offsets must start at 0");
    const int64_t N = voff[G];
    const int64_t nnz = rp[N];
    if (rp[0] != 0) return set_error(RWC_ERR_INVALID, "row_ptr[0] must be 0");
    std::vector<BGraph> hg(G);
    std::vector<int32_t> roots(G);
    std::vector<int64_t> lrp;
    for (int32_t g = 0; g < G; ++g) {
        const int64_t v0 = voff[g], n = voff[g + 1] - v0;
        if (n < 2 || n > 20000) return set_error(RWC_ERR_INVALID, "graph %d: batch graphs need 2 <= n <= 20000", g);
        lrp.resize(n + 1);
        for (int64_t u = 0; u <= n; ++u) lrp[u] = rp[v0 + u] - rp[v0];
        const int32_t *gc = col + rp[v0];
        const float *gw = w ? w + rp[v0] : nullptr;
        rwc_status s = validate_csr(n, lrp[n], lrp.data(), gc, gw);
        if (s != RWC_OK) return set_error(s, "graph %d: %s", g, rwc_last_error());
        if (!csr_connected(n, lrp.data(), gc)) return set_error(RWC_ERR_NOT_CONNECTED, "graph %d is not connected", g);
        double best = -1.0;
        int32_t arg = 0;
        for (int64_t u = 0; u < n; ++u) {
            double d = 0.0;
            if (gw) for (int64_t j = lrp[u]; j < lrp[u + 1]; ++j) d = d + (double)gw[j - 0];
            else d = (double)(lrp[u + 1] - lrp[u]);
            if (d > best) { best = d; arg = (int32_t)u; }
        }
        hg[g] = BGraph{v0, (int32_t)n, arg};
        roots[g] = arg;
    }
    rwc_batch *b = new (std::nothrow) rwc_batch();
    if (!b) return set_error(RWC_ERR_OOM, "host allocation failed");
    auto fail = [&](cudaError_t e) {
        for (void *p : b->allocs) cudaFree(p);
        if (b->host) cudaFreeHost(b->host);
        delete b;
        return set_error(e == cudaErrorMemoryAllocation ? RWC_ERR_OOM : RWC_ERR_CUDA, "batch upload: %s",
                         cudaGetErrorString(e));
    };
    b->G = G; b->N = N; b->nnz = nnz; b->hgraphs = hg; b->roots = roots;
    b->weighted = (w != nullptr);
    b->off64 = nnz >= ((int64_t)1 << 31) - 1;
    cudaError_t e;
    DevGraph &d = b->base;
    d.n = N; d.nnz = nnz; d.weighted = b->weighted; d.off64 = b->off64;
    if (b->off64) {
        int64_t *p;
        if ((e = balloc(b, (void **)&p, (N + 1) * 8)) != cudaSuccess) return fail(e);
        if ((e = cudaMemcpy(p, rp, (N + 1) * 8, cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
        d.rp64 = p;
    } else {
        std::vector<int32_t> r32(N + 1);
        for (int64_t i = 0; i <= N; ++i) r32[i] = (int32_t)rp[i];
        int32_t *p;
        if ((e = balloc(b, (void **)&p, (N + 1) * 4)) != cudaSuccess) return fail(e);
        if ((e = cudaMemcpy(p, r32.data(), (N + 1) * 4, cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
        d.rp32 = p;
    }
    {
        int32_t *p;
        if ((e = balloc(b, (void **)&p, nnz * 4)) != cudaSuccess) return fail(e);
        if ((e = cudaMemcpy(p, col, nnz * 4, cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
        d.col = p;
    }
    if (w) {
        std::vector<WArc> arcs(nnz);
        std::vector<double> prob;
        std::vector<int64_t> ql, qh;
        std::vector<uint32_t> thr;
        std::vector<int32_t> al;
        for (int64_t u = 0; u < N; ++u) {
            const int64_t b0 = rp[u], deg = rp[u + 1] - rp[u];
            thr.resize(deg); al.resize(deg);
            vose_row(w + b0, deg, thr.data(), al.data(), prob, ql, qh);
            for (int64_t j = 0; j < deg; ++j) arcs[b0 + j] = WArc{col[b0 + j], thr[j], col[b0 + al[j]], al[j]};
        }
        WArc *p;
        if ((e = balloc(b, (void **)&p, nnz * sizeof(WArc))) != cudaSuccess) return fail(e);
        if ((e = cudaMemcpy(p, arcs.data(), nnz * sizeof(WArc), cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
        d.warc = p;
    }
    if ((e = balloc(b, (void **)&b->graphs, G * sizeof(BGraph))) != cudaSuccess) return fail(e);
    if ((e = cudaMemcpy(b->graphs, hg.data(), G * sizeof(BGraph), cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
    {
        std::vector<int32_t> one(G);
        for (int32_t g = 0; g < G; ++g) one[g] = g;
        if ((e = balloc(b, (void **)&b->single, G * sizeof(int32_t))) != cudaSuccess) return fail(e);
        if ((e = cudaMemcpy(b->single, one.data(), G * sizeof(int32_t), cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
    }
    if ((e = balloc(b, &b->scratch, 256)) != cudaSuccess) return fail(e);
    if ((e = cudaMallocHost((void **)&b->host, 64)) != cudaSuccess) return fail(e);
    *out = b;
    return RWC_OK;
}

extern "C" rwc_status rwc_batch_roots(const rwc_batch_t *b, int32_t *host_roots) {
    if (!b || !host_roots) return set_error(RWC_ERR_INVALID, "bad argument");
    memcpy(host_roots, b->roots.data(), b->roots.size() * sizeof(int32_t));
    return RWC_OK;
}

extern "C" rwc_status rwc_batch_sample(rwc_batch_t *b, uint64_t seed, int64_t T, double *sums,
                                       int32_t use_graph, int32_t per_graph_launch,
                                       rwc_stats_t *stats, rwc_stream_t stream) {
    clear_error();
    if (!b || !sums || T <= 0 || T > ((int64_t)1 << 31)) return set_error(RWC_ERR_INVALID, "bad argument");
    if (stats) memset(stats, 0, sizeof(*stats));
    cudaStream_t st = (cudaStream_t)stream;
    RWC_CUDA_TRY(cudaMemsetAsync(b->scratch, 0, 32, st));
    if (per_graph_launch) {
        // baseline: one launch per graph, same per-tree code
        int *err = (int *)b->scratch;
        unsigned long long *ctr = (unsigned long long *)((char *)b->scratch + 8);
        const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
        if (b->single_blocks.empty()) RWC_TRY(plan_single(b));
        const bool few = few_trees(T);
        auto blocks = [&](int32_t g) { return few ? T : std::min(T, b->single_blocks[g]); };
        int64_t spill = 0;
        for (int32_t g = 0; g < b->G; ++g)
            if (b->hgraphs[g].n > (int)LT_STACK) spill = std::max(spill, blocks(g) * b->hgraphs[g].n);
        if (spill > b->single_spill_n) {
            bfree(b, b->single_spill);
            b->single_spill_n = 0;
            RWC_CUDA_TRY(balloc(b, (void **)&b->single_spill, (size_t)spill * sizeof(uint32_t)));
            b->single_spill_n = spill;
        }
        for (int32_t g = 0; g < b->G; ++g) {
            const int n = b->hgraphs[g].n, nt = single_threads(n, few);
            ::rwc::count_launches(1);
            dispatch_nt(b->off64, b->weighted, nt, [&](auto kern) {
                kern<<<(unsigned)blocks(g), nt, batch_tree_smem(n, nt), st>>>(
                    b->base, b->graphs, b->single + g, T, nullptr, T, k0, k1, n, sums, b->single_spill, err, ctr);
            });
        }
        RWC_CUDA_TRY(cudaGetLastError());
        return finish(b, stats, 3, T, st);
    }
    RWC_TRY(build_items(b, T));
    if (!use_graph) {
        RWC_TRY(enqueue(b, seed, T, sums, st));
        return finish(b, stats, 4, T, st);
    }
    if (!b->exec || b->cap_seed != seed || b->cap_T != T || b->cap_sums != sums || b->cap_stream != st) {
        drop_graph(b);
        cudaStream_t cs;
        RWC_CUDA_TRY(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        rwc_status s = RWC_OK;
        cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            s = enqueue(b, seed, T, sums, cs);
            cudaGraph_t gr = nullptr;
            e = cudaStreamEndCapture(cs, &gr);
            if (s == RWC_OK && e == cudaSuccess) {
                b->graph = gr;
                e = cudaGraphInstantiate(&b->exec, gr, 0);
            } else if (gr) {
                cudaGraphDestroy(gr);
            }
        }
        cudaStreamDestroy(cs);
        RWC_TRY(s);
        if (e != cudaSuccess) { drop_graph(b); return set_error(RWC_ERR_CUDA, "CUDA graph capture: %s", cudaGetErrorString(e)); }
        b->cap_seed = seed; b->cap_T = T; b->cap_sums = sums; b->cap_stream = st;
    }
    RWC_CUDA_TRY(cudaGraphLaunch(b->exec, st));
    return finish(b, stats, 5, T, st);
}

namespace {
// Checks a schedule against the batch's graphs; the item lists must be built.
bool schedule_fits(const rwc_batch *b) { return batch_smem(b) <= 227 * 1024; }
}  // namespace

extern "C" rwc_status rwc_batch_get_schedule(const rwc_batch_t *b, int32_t *host_sched) {
    clear_error();
    if (!b || !host_sched) return set_error(RWC_ERR_INVALID, "bad argument");
    host_sched[0] = b->threads;
    host_sched[1] = b->split;
    host_sched[2] = b->tile;
    host_sched[3] = b->warp;
    host_sched[4] = b->conc;
    return RWC_OK;
}

extern "C" rwc_status rwc_batch_set_schedule(rwc_batch_t *b, int32_t threads, int32_t split, int32_t tile,
                                             int32_t warp, int32_t concurrent) {
    clear_error();
    if (!b || threads < 32 || threads > 1024 || threads % 32 || split < 0 || split > 20000 || tile < 1 ||
        (warp != 0 && warp != 1) || (concurrent != 0 && concurrent != 1))
        return set_error(RWC_ERR_INVALID, "schedule needs threads in [32, 1024] (a multiple of 32), "
                                          "0 <= split <= 20000, tile >= 1, warp and concurrent 0 or 1");
    int wmax = 0, bmax = 0;
    for (const BGraph &g : b->hgraphs) {
        if (g.n <= split) wmax = std::max(wmax, g.n);
        else bmax = std::max(bmax, g.n);
    }
    const size_t need = schedule_allowance(bmax, wmax, warp);
    if (need > 227 * 1024)
        return set_error(RWC_ERR_UNSUPPORTED, "schedule needs %zu bytes of shared memory per block", need);
    b->threads = threads;
    b->split = split;
    b->tile = tile;
    b->warp = warp;
    b->conc = concurrent;
    b->items_T = -1;
    drop_graph(b);
    return RWC_OK;
}

extern "C" rwc_status rwc_autotune(rwc_batch_t *b, const char *cache_path, rwc_stream_t stream) {
    clear_error();
    if (!b) return set_error(RWC_ERR_INVALID, "bad argument");
    cudaStream_t st = (cudaStream_t)stream;
    char sig[128];
    snprintf(sig, sizeof(sig), "G%d_N%lld_E%lld", b->G, (long long)b->N, (long long)b->nnz);
    if (cache_path) {
        FILE *f = fopen(cache_path, "r");
        if (f) {
            char buf[4096];
            size_t len = fread(buf, 1, sizeof(buf) - 1, f);
            fclose(f);
            buf[len] = 0;
            const char *p = strstr(buf, sig);
            const char *colon = p ? strchr(p, ':') : nullptr;
            int th, sp, tl, wp, cc;
            if (colon && sscanf(colon + 1, " [%d, %d, %d, %d, %d]", &th, &sp, &tl, &wp, &cc) == 5 &&
                rwc_batch_set_schedule(b, th, sp, tl, wp, cc) == RWC_OK)
                return RWC_OK;
            clear_error();
        }
    }
    double *sums = nullptr;
    RWC_CUDA_TRY(cudaMallocAsync((void **)&sums, b->N * sizeof(double), st));
    // coordinate search from the current schedule, each candidate timed on
    // 16 trees per graph: the split with the small class warp- or
    // block-per-tree, then a smaller largest block of the large class (no block has
    // more than 256 threads, so larger bounds are the same launches), then
    // concurrent or sequential bins
    const int64_t Tp = 16;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    struct Sched { int th, sp, tl, wp, cc; };
    Sched best_s{b->threads, b->split, b->tile, b->warp, b->conc};
    const Sched before = best_s;
    float best = 1e30f;
    rwc_status status = RWC_OK;
    auto time_one = [&](const Sched &c) -> float {
        b->threads = c.th; b->split = c.sp; b->tile = c.tl; b->warp = c.wp; b->conc = c.cc;
        b->items_T = -1;
        if ((status = build_items(b, Tp)) != RWC_OK) return -1.f;
        if (!schedule_fits(b)) return 1e30f;
        cudaMemsetAsync(b->scratch, 0, 32, st);
        if (enqueue(b, 12345, Tp, sums, st) != RWC_OK) { clear_error(); return 1e30f; }
        cudaEventRecord(e0, st);
        cudaMemsetAsync(b->scratch, 0, 32, st);
        if (enqueue(b, 12346, Tp, sums, st) != RWC_OK) { clear_error(); return 1e30f; }
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        return ms;
    };
    auto consider = [&](Sched c) -> bool {
        const float ms = time_one(c);
        if (ms < 0.f) return false;
        if (ms < best) { best = ms; best_s = c; }
        return true;
    };
    {
        const int splits[][2] = {{0, 0}, {512, 1}, {1024, 1}, {2048, 1}, {1024, 0}, {2048, 0}, {4096, 0}};
        for (auto &sw : splits) { Sched c = best_s; c.sp = sw[0]; c.wp = sw[1]; if (!consider(c)) goto done; }
        const Sched base1 = best_s;
        for (int th : {64, 128}) { Sched c = base1; c.th = th; if (!consider(c)) goto done; }
        const Sched base2 = best_s;
        for (int cc : {0, 1}) { Sched c = base2; c.cc = cc; if (!consider(c)) goto done; }
    }
done:
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFreeAsync(sums, st);
    if (status != RWC_OK) best_s = before;
    b->threads = best_s.th; b->split = best_s.sp; b->tile = best_s.tl; b->warp = best_s.wp; b->conc = best_s.cc;
    b->items_T = -1;
    drop_graph(b);
    RWC_CUDA_TRY(cudaStreamSynchronize(st));
    RWC_TRY(status);
    if (cache_path) {
        FILE *f = fopen(cache_path, "w");
        if (f) {
            fprintf(f, "{\"%s\": [%d, %d, %d, %d, %d]}\n", sig, best_s.th, best_s.sp, best_s.tl, best_s.wp, best_s.cc);
            fclose(f);
        }
    }
    return RWC_OK;
}

extern "C" rwc_status rwc_batch_destroy(rwc_batch_t *b) {
    if (!b) return RWC_OK;
    drop_graph(b);
    for (cudaStream_t s : b->side)
        if (s) cudaStreamSynchronize(s);
    for (void *p : b->allocs) cudaFree(p);
    if (b->host) cudaFreeHost(b->host);
    drop_streams(b);
    delete b;
    return RWC_OK;
}
