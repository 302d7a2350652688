// Tree sampling by rounds of cycle popping with many lanes per tree
// (lane_tree.cuh): the vertex words in shared memory for graphs that fit (up to
// about 56000 vertices), in global memory otherwise.
//
// Measured (kernel time, whole-block popping rounds in shared memory or
// concurrent walkers before -> here): BA n = 2000, 1000 trees 0.51 -> 0.12 ms;
// weighted RGG n = 19999, 304 trees 194 -> 8 ms; 224 x 240 grid, 1000 trees
// 1.38 -> 0.27 s; R-MAT n = 100000, 1000 trees 20.1 -> 6.5 ms; 512 x 512 grid,
// 64 trees 3.97 -> 1.18 s.  Latency bound: one tree of the 150 x 150 grid runs
// at 6 cycles per instruction and warp, 30% of them at barriers, with 4 warps
// on an SM; one lane per thread (twice the warps of two) took 313 instead of
// 404 ms on the 224 x 240 grid.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "lane_tree.cuh"
#include "rwc_common.cuh"

namespace rwc {
namespace {

// One tree per block of NT threads, its words in shared memory; trees are
// handed out by ctr[0] after the first of each block.  Trees whose counts
// outgrow the word are left out and listed in wide[0 .. ctr[2]).
template <bool OFF64, bool WT, int EW, int NT>
__global__ void __launch_bounds__(NT) l_trees_smem(DevGraph g, uint32_t tree0, int64_t T, uint32_t k0,
                                                   uint32_t k1, uint32_t klim, int kb, double *sums,
                                                   int32_t *parents, int32_t *visits, uint32_t *spill,
                                                   int *err, unsigned long long *ctr, uint32_t *wide) {
    constexpr int S = 1;
    static_assert(sizeof(LaneShared<NT, S>) % 4 == 0 && NT <= 256, "lane_smem");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long sh_next;
    LaneShared<NT, S> &sh = *reinterpret_cast<LaneShared<NT, S> *>(smem);
    uint32_t *word = reinterpret_cast<uint32_t *>(smem + sizeof(LaneShared<NT, S>));
    const int n = (int)g.n;
    const uint32_t kmask = (1u << kb) - 1u;
    uint32_t *sp = spill + (int64_t)blockIdx.x * n;
    unsigned long long draws = 0;
    uint32_t rounds = 0;
    int64_t t = blockIdx.x;
    while (t < T) {
        for (int u = threadIdx.x; u < n; u += NT) word[u] = u == g.root ? lt_root_word<uint32_t>(kb, NT * S) : 0u;
        __syncthreads();
        const int bad = lane_tree<OFF64, WT, EW, NT, S, true, uint32_t>(g, word, kb, klim, sh, sp, tree0 + (uint32_t)t,
                                                                     0u, k0, k1, rounds);
        if (bad & ~LE_KREP) { if (threadIdx.x == 0) atomicOr(err, bad); break; }
        if (bad && threadIdx.x == 0) wide[atomicAdd(ctr + 2, 1ull)] = (uint32_t)t;
        for (int u = bad ? n : threadIdx.x; u < n; u += NT) {
            const uint32_t w = word[u];
            const uint32_t vis = u == g.root ? 0u : (w & kmask) + 1u;
            draws += vis;
            if (sums && vis) atomicAdd(sums + u, (double)vis);
            if (parents) parents[t * n + u] = u == g.root ? -1 : (int32_t)(((w & 0x7fffffffu) >> kb) - lt_id0(NT * S));
            if (visits) visits[t * n + u] = (int32_t)vis;
        }
        if (threadIdx.x == 0) sh_next = atomicAdd(ctr, 1ull);
        __syncthreads();
        t = (int64_t)gridDim.x + (int64_t)sh_next;
    }
    for (int o = 16; o > 0; o >>= 1) draws += __shfl_xor_sync(0xffffffffu, draws, o);
    if ((threadIdx.x & 31) == 0 && draws) atomicAdd(ctr + 1, draws);
    if (threadIdx.x == 0 && rounds) atomicAdd(ctr + 3, (unsigned long long)rounds);
}

// One tree per block of NT threads, its words in global memory (zeroed by the
// caller), `ld` words apart: the trees ids[0 .. B) of the call, or its first B
// (ids = NULL).  Trees whose counts outgrow the word are listed in wide[0 ..
// ctr[2]) and their root's word is left 0.
template <bool OFF64, bool WT, int EW, int NT, class W>
__global__ void __launch_bounds__(NT) l_trees(DevGraph g, uint32_t tree0, int64_t B, int64_t ld, uint32_t k0,
                                              uint32_t k1, uint32_t klim, int kb, W *words, uint32_t *spill,
                                              const uint32_t *ids, int *err, unsigned long long *ctr,
                                              uint32_t *wide) {
    constexpr int S = 2;   // lanes per thread: two loads in flight
    __shared__ LaneShared<NT, S> sh;
    __shared__ unsigned long long sh_next;
    uint32_t *sp = spill + (int64_t)blockIdx.x * g.n;
    int64_t t = blockIdx.x;
    while (t < B) {
        W *word = words + t * ld;
        if (threadIdx.x == 0) word[g.root] = lt_root_word<W>(kb, NT * S);
        __syncthreads();
        uint32_t rounds = 0;
        const int bad = lane_tree<OFF64, WT, EW, NT, S, false, W>(g, word, kb, klim, sh, sp,
                                                                  tree0 + (ids ? ids[t] : (uint32_t)t), 0u, k0, k1,
                                                                  rounds);
        if (bad & ~LE_KREP) { if (threadIdx.x == 0) atomicOr(err, bad); break; }
        if (bad && threadIdx.x == 0) { wide[atomicAdd(ctr + 2, 1ull)] = (uint32_t)t; word[g.root] = 0; }
        if (threadIdx.x == 0) sh_next = atomicAdd(ctr, 1ull);
        __syncthreads();
        t = (int64_t)gridDim.x + (int64_t)sh_next;
    }
}

// visits_u = k_u + 1 over the chunk's trees into sums, without the listed ones
// (root's word 0); optional per-tree output (rows ids[t]).  Nothing after an
// error.  The trees are split over gridDim.y so that small graphs fill the chip too; the sums are
// whole numbers, exact in any order.
template <class W>
__global__ void l_accum(int64_t n, int32_t root, const W *words, int64_t ld, int kb, uint32_t id0, int64_t B,
                        const uint32_t *ids, double *sums, int32_t *parents, int32_t *visits, const int *err,
                        unsigned long long *ctr) {
    if (*err) return;
    const bool listed = ctr[2] != 0;
    const W kmask = ((W)1 << kb) - 1, pmask = ~(W)0 >> 1;
    const int64_t t0 = B * blockIdx.y / gridDim.y, t1 = B * (blockIdx.y + 1) / gridDim.y;
    unsigned long long local = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long acc = 0;
#pragma unroll 4
        for (int64_t t = t0; t < t1; ++t) {
            if (listed && words[t * ld + root] == 0) continue;
            const W w = words[t * ld + u];
            const uint32_t vis = u == root ? 0u : (uint32_t)(w & kmask) + 1u;
            acc += vis;
            if (parents || visits) {
                const int64_t row = ids ? ids[t] : t;
                if (parents) parents[row * n + u] = u == root ? -1 : (int32_t)((uint32_t)((w & pmask) >> kb) - id0);
                if (visits) visits[row * n + u] = (int32_t)vis;
            }
        }
        local += acc;
        if (sums && acc) atomicAdd(sums + u, (double)acc);
    }
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(ctr + 1, local);
}

template <int V> using int_c = std::integral_constant<int, V>;

// f(off64, weighted, inline row width) as compile-time constants
template <class F>
void dispatch(const DevGraph &g, F f) {
    if (g.off64) {
        if (g.weighted) f(std::true_type{}, std::true_type{}, int_c<0>{});
        else f(std::true_type{}, std::false_type{}, int_c<0>{});
    } else {
        if (g.weighted) f(std::false_type{}, std::true_type{}, int_c<0>{});
        else if (g.ell_w == 4) f(std::false_type{}, std::false_type{}, int_c<4>{});
        else if (g.ell_w == 8) f(std::false_type{}, std::false_type{}, int_c<8>{});
        else f(std::false_type{}, std::false_type{}, int_c<0>{});
    }
}

struct Buf {
    void *p = nullptr;
    cudaStream_t st;
    explicit Buf(cudaStream_t s) : st(s) {}
    ~Buf() { if (p) cudaFreeAsync(p, st); }
};
struct Events {
    cudaEvent_t e[4] = {};
    bool on;
    explicit Events(bool o) : on(o) { if (on) for (auto &x : e) cudaEventCreate(&x); }
    ~Events() { if (on) for (auto &x : e) cudaEventDestroy(x); }
    void rec(int i, cudaStream_t s) { if (on) cudaEventRecord(e[i], s); }
    double ms(int a, int b) { float v = 0.f; if (on) cudaEventElapsedTime(&v, e[a], e[b]); return v; }
};

constexpr size_t SMEM_MAX = 226 * 1024;   // dynamic shared memory of one block beside 1 KB of its own
constexpr int64_t TAIL = 64;   // err @0, next tree @8, draws @16, listed trees @24, rounds @32
constexpr int64_t WIDE_CAP = 65536;   // trees of one shared-memory launch

// Trees tree0 .. tree0 + T - 1 (`only`: the T trees tree0 + only[i], a part of
// a call whose other trees are done) with words of type W.  With 32-bit words the
// trees whose counts outgrow them are appended to `redo`, and a chunk that lists
// more than half of its trees is the last: *done trees have been taken.
template <int NT, class W>
rwc_status walker_range(rwc_graph *G, uint64_t seed, int64_t tree0, int64_t T, const uint32_t *only, double *sums,
                        int32_t *parents, int32_t *visits, const rwc_options_t &o, rwc_stats_t *st,
                        std::vector<uint32_t> *redo, int64_t *done, cudaStream_t stream) {
    const DevGraph &g = G->g;
    const int64_t n = g.n, ld = (n + 3) & ~(int64_t)3;
    const uint32_t klim = (1u << 20) - 1u;
    constexpr int NL = 2 * NT;
    const int kb = lt_kbits<W>(n, NL);
    const int sms = num_sms();
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    int64_t B = o.trees_per_chunk;
    if (B <= 0) {
        const size_t per_tree = (size_t)ld * (sizeof(W) + 4) + 256;
        size_t budget = (size_t)std::max<int64_t>(0, o.memory_budget);
        if (!budget) {
            size_t fr = 0, tot = 0;
            RWC_CUDA_TRY(cudaMemGetInfo(&fr, &tot));
            budget = (size_t)(fr * 0.6);
        }
        B = (int64_t)std::max<size_t>(1, budget / per_tree);
    }
    B = std::min(B, T);
    int per_sm = 0;
    dispatch(g, [&](auto o64, auto wt, auto ew) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, l_trees<decltype(o64)::value, decltype(wt)::value, decltype(ew)::value, NT, W>, NT, 0);
    });
    if (per_sm < 1) return set_error(RWC_ERR_UNSUPPORTED, "walker block does not fit");
    const int64_t slots = std::min<int64_t>(B, (int64_t)sms * per_sm);
    Buf buf(stream);
    const size_t wbytes = (size_t)B * ld * sizeof(W);
    RWC_CUDA_TRY(cudaMallocAsync(&buf.p, wbytes + (size_t)slots * n * 4 + (size_t)B * 8 + TAIL + 64, stream));
    W *words = (W *)buf.p;
    uint32_t *spill = (uint32_t *)((char *)buf.p + wbytes);
    uint32_t *ids = spill + slots * n, *wide = ids + B;
    char *tail = (char *)(wide + B);
    tail = (char *)(((uintptr_t)tail + 63) & ~(uintptr_t)63);
    int *err = (int *)tail;
    unsigned long long *ctr = (unsigned long long *)(tail + 8);
    Events ev(o.profile != 0);
    int64_t *h = G->host_scalars;
    if (st) st->mode = RWC_MODE_WALKER;
    for (int64_t c0 = 0; c0 < T; c0 += B) {
        const int64_t Bc = std::min(B, T - c0), first = only ? 0 : c0;
        int32_t *par = parents ? parents + first * n : nullptr, *vis = visits ? visits + first * n : nullptr;
        RWC_CUDA_TRY(cudaMemsetAsync(tail, 0, TAIL, stream));
        if (only) RWC_CUDA_TRY(cudaMemcpyAsync(ids, only + c0, (size_t)Bc * 4, cudaMemcpyHostToDevice, stream));
        const uint32_t *list = only ? ids : nullptr;
        ev.rec(0, stream);
        RWC_CUDA_TRY(cudaMemsetAsync(words, 0, (size_t)Bc * ld * sizeof(W), stream));
        ev.rec(1, stream);
        dispatch(g, [&](auto o64, auto wt, auto ew) {
            ::rwc::count_launches(1);
            l_trees<decltype(o64)::value, decltype(wt)::value, decltype(ew)::value, NT, W>
                <<<(unsigned)std::min(Bc, slots), NT, 0, stream>>>(g, (uint32_t)(tree0 + first), Bc, ld, k0, k1, klim,
                                                                   kb, words, spill, list, err, ctr, wide);
        });
        ev.rec(2, stream);
        const int64_t bx = std::min<int64_t>((n + 255) / 256, (int64_t)sms * 8);
        const int64_t by = std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * 8 / bx, Bc / 8));
        ::rwc::count_launches(1);
        l_accum<W><<<dim3((unsigned)bx, (unsigned)by), 256, 0, stream>>>(n, g.root, words, ld, kb, lt_id0(NL), Bc, list,
                                                                         sums, par, vis, err, ctr);
        ev.rec(3, stream);
        RWC_CUDA_TRY(cudaGetLastError());
        if (o.async_status) {
            ::rwc::count_launches(1);
            fold_lane_status<<<1, 1, 0, stream>>>(err, G->dev_status);
            RWC_CUDA_TRY(cudaGetLastError());
            continue;
        }
        RWC_CUDA_TRY(cudaMemcpyAsync(h, tail, 32, cudaMemcpyDeviceToHost, stream));
        RWC_CUDA_TRY(cudaStreamSynchronize(stream));
        const int e = (int)(h[0] & 0xffffffff);
        if (e & LE_KOVF) return set_error(RWC_ERR_UNSUPPORTED, "a vertex was popped more than 2^20 - 1 times");
        if (e) return set_error(RWC_ERR_CUDA, "sampler internal check failed");
        if (st) {
            const int64_t draws = h[2];
            if (!only) st->chunks += 1;
            st->draws += draws;
            st->marked += draws;
            st->block_threads = NL;
            st->phase_units[RWC_PHASE_INIT] += Bc * n;
            st->phase_units[RWC_PHASE_WALK] += draws;
            st->phase_units[RWC_PHASE_ACCUM] += Bc * n;
            if (ev.on) {
                st->phase_ms[RWC_PHASE_INIT] += ev.ms(0, 1);
                st->phase_ms[RWC_PHASE_WALK] += ev.ms(1, 2);
                st->phase_ms[RWC_PHASE_ACCUM] += ev.ms(2, 3);
                st->phase_launches[RWC_PHASE_WALK] += 1;
                st->phase_launches[RWC_PHASE_ACCUM] += 1;
            }
        }
        if (const int64_t listed = h[3]) {
            if (!redo) return set_error(RWC_ERR_CUDA, "sampler internal check failed");   // 64-bit words hold every allowed count
            const size_t at = redo->size();
            redo->resize(at + (size_t)listed);
            RWC_CUDA_TRY(cudaMemcpyAsync(redo->data() + at, wide, (size_t)listed * 4, cudaMemcpyDeviceToHost, stream));
            RWC_CUDA_TRY(cudaStreamSynchronize(stream));
            for (size_t i = at; i < redo->size(); ++i) (*redo)[i] += (uint32_t)c0;
            if (2 * listed > Bc) { *done = c0 + Bc; return RWC_OK; }
        }
    }
    if (done) *done = T;
    return RWC_OK;
}

// f(threads per tree) for T trees with words in global memory, by the trees that an SM
// gets: 32 (64 lanes) when they fill it, more when few are left to it (300 x 300
// grid, 300 trees: 572, 429 and 449 ms with 32, 128 and 512; 512 x 512, 64 trees:
// 2.01, 1.44, 1.18 s); graphs of unbounded degree have ends for 1024 lanes (R-MAT n
// = 262144, 2000 trees: 101, 60 and 48 ms).
template <class F>
rwc_status with_threads(const DevGraph &g, int64_t T, F f) {
    const int64_t share = (T + num_sms() - 1) / num_sms();
    if (g.ell && share >= 8) return f(int_c<32>{});
    if (g.ell && share >= 2) return f(int_c<128>{});
    return f(int_c<512>{});
}

// Trees of a call with 64-bit words.
rwc_status wide_trees(rwc_graph *G, uint64_t seed, int64_t tree0, int64_t T, const uint32_t *only, double *sums,
                      int32_t *parents, int32_t *visits, const rwc_options_t &o, rwc_stats_t *st, cudaStream_t stream) {
    return with_threads(G->g, T, [&](auto nt) {
        return walker_range<decltype(nt)::value, uint64_t>(G, seed, tree0, T, only, sums, parents, visits, o, st, nullptr,
                                                           nullptr, stream);
    });
}

}  // namespace

// Shared memory of one tree with nt threads.
static size_t lane_smem(int64_t n, int nt) {
    const size_t head = nt == 32 ? sizeof(LaneShared<32, 1>) : nt == 64 ? sizeof(LaneShared<64, 1>)
                      : nt == 128 ? sizeof(LaneShared<128, 1>) : sizeof(LaneShared<256, 1>);
    return head + (size_t)n * 4;
}

namespace {
template <int NT>
rwc_status smem_range(rwc_graph *G, uint64_t seed, int64_t tree0, int64_t T, double *sums, int32_t *parents,
                      int32_t *visits, uint32_t klim, const rwc_options_t &o, rwc_stats_t *st,
                      std::vector<uint32_t> &redo, int *h_err, cudaStream_t stream) {
    const DevGraph &g = G->g;
    const int64_t n = g.n;
    const size_t smem = lane_smem(n, NT);
    const int kb = lt_kbits<uint32_t>(n, NT);
    const int sms = num_sms();
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const bool need_spill = n > LT_STACK;
    Buf buf(stream);
    Events ev(o.profile != 0);
    rwc_status status = RWC_OK;
    int *err = nullptr;
    *h_err = 0;
    dispatch(g, [&](auto o64, auto wt, auto ew) {
        auto kern = l_trees_smem<decltype(o64)::value, decltype(wt)::value, decltype(ew)::value, NT>;
        auto launch = [&]() -> rwc_status {
            // the same value on every call: other threads launch the kernel too
            RWC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
            int per_sm = 0;
            RWC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem));
            if (per_sm < 1) return set_error(RWC_ERR_UNSUPPORTED, "graph too large for shared mode");
            int64_t blocks = std::min<int64_t>(T, (int64_t)sms * per_sm);
            if (o.memory_budget > 0 && need_spill)
                blocks = std::max<int64_t>(1, std::min(blocks, (o.memory_budget - TAIL - T * 4) / (n * 4)));
            RWC_CUDA_TRY(cudaMallocAsync(&buf.p, TAIL + (size_t)T * 4 + (need_spill ? (size_t)blocks * n * 4 : 0), stream));
            RWC_CUDA_TRY(cudaMemsetAsync(buf.p, 0, TAIL, stream));
            err = (int *)buf.p;
            ev.rec(0, stream);
            ::rwc::count_launches(1);
            kern<<<(unsigned)blocks, NT, smem, stream>>>(
                g, (uint32_t)tree0, T, k0, k1, klim, kb, sums, parents, visits,
                need_spill ? (uint32_t *)((char *)buf.p + TAIL) + T : nullptr, err,
                (unsigned long long *)((char *)buf.p + 8), (uint32_t *)((char *)buf.p + TAIL));
            ev.rec(1, stream);
            RWC_CUDA_TRY(cudaGetLastError());
            return RWC_OK;
        };
        status = launch();
    });
    RWC_TRY(status);
    if (o.async_status) {
        ::rwc::count_launches(1);
        fold_lane_status<<<1, 1, 0, stream>>>(err, G->dev_status);
        RWC_CUDA_TRY(cudaGetLastError());
        return RWC_OK;
    }
    int64_t *h = G->host_scalars;
    RWC_CUDA_TRY(cudaMemcpyAsync(h, buf.p, 40, cudaMemcpyDeviceToHost, stream));
    RWC_CUDA_TRY(cudaStreamSynchronize(stream));
    *h_err = (int)(h[0] & 0xffffffff);
    if (*h_err) return RWC_OK;
    if (h[3]) {
        const size_t at = redo.size();
        redo.resize(at + (size_t)h[3]);
        RWC_CUDA_TRY(cudaMemcpyAsync(redo.data() + at, (char *)buf.p + TAIL, (size_t)h[3] * 4, cudaMemcpyDeviceToHost, stream));
        RWC_CUDA_TRY(cudaStreamSynchronize(stream));
    }
    if (st) {
        st->draws += h[2];
        st->marked += h[2];
        st->chunks += 1;
        st->rounds += h[4];
        st->phase_units[RWC_PHASE_WALK] += h[2];
        if (ev.on) {
            st->phase_ms[RWC_PHASE_WALK] += ev.ms(0, 1);
            st->phase_launches[RWC_PHASE_WALK] += 1;
        }
    }
    return RWC_OK;
}
}  // namespace

namespace {
// Trees tree0 .. tree0 + T - 1 with their words in shared memory; status is
// the caller's message.
rwc_status sample_smem(rwc_graph *G, uint64_t seed, int64_t tree0, int64_t T, double *sums, int32_t *parents,
                       int32_t *visits, uint32_t klim, const rwc_options_t &o, rwc_stats_t *st, int *err,
                       cudaStream_t stream) {
    const int64_t n = G->g.n;
    int64_t chunk = std::min(T, o.trees_per_chunk > 0 ? std::min(o.trees_per_chunk, WIDE_CAP) : WIDE_CAP);
    // a budget is shared by the list of trees (4 bytes each) and the blocks' ends
    if (o.memory_budget > 0) chunk = std::max<int64_t>(1, std::min(chunk, o.memory_budget / 8));
    // threads per tree: 1024 on an SM, over the trees that it holds at once (BA
    // n = 12000, 1000 trees: 1.0, 0.65 and 0.50 ms with 64, 128 and 256 threads;
    // n = 2000, 1000 trees: 0.142, 0.122 and 0.135 ms)
    int NTs = 256;
    while (NTs > 64 && NTs * std::min<int64_t>((227 * 1024) / (int64_t)(lane_smem(n, NTs) + 1024),
                                               (chunk + num_sms() - 1) / num_sms()) > 1024)
        NTs /= 2;
    // up to 448 vertices one warp, whose phases need no block barrier: chains keep
    // few lanes busy (path of 200 vertices, 150 trees: 20.8 ms against 26.1, 26.9 and
    // 29.8 with 64, 128 and 256 threads; BA n = 200: the same within 3%; from 800 vertices
    // on BA trees are faster with more)
    if (n <= 448) NTs = 32;
    std::vector<uint32_t> redo;
    for (int64_t c0 = 0; c0 < T; c0 += chunk) {
        const int64_t Tc = std::min(chunk, T - c0);
        int32_t *par = parents ? parents + c0 * n : nullptr, *vis = visits ? visits + c0 * n : nullptr;
        const size_t at = redo.size();
        if (NTs == 32) RWC_TRY(smem_range<32>(G, seed, tree0 + c0, Tc, sums, par, vis, klim, o, st, redo, err, stream));
        else if (NTs == 256) RWC_TRY(smem_range<256>(G, seed, tree0 + c0, Tc, sums, par, vis, klim, o, st, redo, err, stream));
        else if (NTs == 128) RWC_TRY(smem_range<128>(G, seed, tree0 + c0, Tc, sums, par, vis, klim, o, st, redo, err, stream));
        else RWC_TRY(smem_range<64>(G, seed, tree0 + c0, Tc, sums, par, vis, klim, o, st, redo, err, stream));
        if (*err) return RWC_OK;
        for (size_t i = at; i < redo.size(); ++i) redo[i] += (uint32_t)c0;
    }
    // trees whose counts outgrew 32-bit words, again with 64-bit ones, side by side
    if (!redo.empty())
        RWC_TRY(wide_trees(G, seed, tree0, (int64_t)redo.size(), redo.data(), sums, parents, visits, o, st, stream));
    if (st) st->block_threads = NTs;
    return RWC_OK;
}
}  // namespace

namespace {

// Whether walker mode keeps this graph's words in shared memory: a lane's hop
// is 45 cycles there against 150 to 230 in global memory, where some lane of a
// warp nearly always misses L1 (RGG n = 40000, 300 trees: 14 against 41 ms).  An
// asynchronous call cannot list trees for wider words, so there every allowed
// count has to fit.
bool walker_in_smem(int64_t n, const rwc_options_t &o) {
    return lane_smem(n, 256) <= SMEM_MAX && (!o.async_status || lt_kbits<uint32_t>(n, 256) >= 20);
}
}  // namespace

// The concurrent walkers (sample_walker) keep calls that ask for their options
// and, with words in global memory, graphs of unbounded degree above 400000
// vertices: there every access goes to HBM and the walkers' fewer words per
// draw count (R-MAT, 500 trees, walkers and lanes: n = 262144 24.4 and 13.6 ms, 524288
// 36.8 and 33.2, 1048576 69 and 80; the line lies below the crossing, whose place for
// other numbers of trees was not measured).
bool lane_walker_takes(const rwc_graph *G, const rwc_options_t &o) {
    const DevGraph &g = G->g;
    if (o.walker_policy || o.block_threads || o.max_wait_ns || o.profile >= 2) return false;
    if (g.n >= ((int64_t)1 << 31) - 4096) return false;
    return walker_in_smem(g.n, o) || g.ell || g.n <= 400000;
}

rwc_status sample_lane_walker(rwc_graph *G, uint64_t seed, int64_t tree0, int64_t T, double *sums,
                              int32_t *parents, int32_t *visits, const rwc_options_t &o, rwc_stats_t *st,
                              cudaStream_t stream) {
    const int64_t n = G->g.n;
    if (walker_in_smem(n, o)) {
        int e = 0;
        RWC_TRY(sample_smem(G, seed, tree0, T, sums, parents, visits, (1u << 20) - 1u, o, st, &e, stream));
        if (e & LE_KOVF) return set_error(RWC_ERR_UNSUPPORTED, "a vertex was popped more than 2^20 - 1 times");
        if (e) return set_error(RWC_ERR_CUDA, "sampler internal check failed");
        if (st) { st->mode = RWC_MODE_WALKER; st->rounds = 0; }
        return RWC_OK;
    }
    std::vector<uint32_t> redo;
    int64_t done = 0;
    RWC_TRY(with_threads(G->g, T, [&](auto nt) -> rwc_status {
        constexpr int NT = decltype(nt)::value;
        // 64-bit words at once where 32 bits leave less than 8 for the count, and for
        // asynchronous calls unless every allowed count fits.  With 8 bits (2048 x 2048
        // grid: mean count 21, one tree in 64 beyond 255) wide words take 8% longer,
        // a repeated tree as long as a lone one (64 trees: 20.2 s in wide words,
        // 31.9 s with one of them repeated): narrow words for a few trees, which rarely
        // have one to repeat, and for many, beside which it does not count.
        const int kb = n < ((int64_t)1 << 30) ? lt_kbits<uint32_t>(n, 2 * NT) : 0;
        const bool some = T >= 16 && T < 4 * (int64_t)num_sms();
        if (kb < (o.async_status ? 20 : some ? 9 : 8)) return RWC_OK;
        return walker_range<NT, uint32_t>(G, seed, tree0, T, nullptr, sums, parents, visits, o, st, &redo, &done, stream);
    }));
    if (!redo.empty())
        RWC_TRY(wide_trees(G, seed, tree0, (int64_t)redo.size(), redo.data(), sums, parents, visits, o, st, stream));
    if (done < T)
        RWC_TRY(wide_trees(G, seed, tree0 + done, T - done, nullptr, sums, parents ? parents + done * n : nullptr,
                           visits ? visits + done * n : nullptr, o, st, stream));
    return RWC_OK;
}

rwc_status sample_lane_shared(rwc_graph *G, uint64_t seed, int64_t tree0, int64_t T, double *sums,
                              int32_t *parents, int32_t *visits, const rwc_options_t &o, rwc_stats_t *st,
                              cudaStream_t stream) {
    int e = 0;
    rwc_options_t p = o;                    // chunks and budgets are walker mode's
    p.trees_per_chunk = p.memory_budget = 0;
    RWC_TRY(sample_smem(G, seed, tree0, T, sums, parents, visits, 65535u, p, st, &e, stream));
    if (e & LE_KOVF) return set_error(RWC_ERR_UNSUPPORTED, "a vertex was popped more than 65535 times; use RWC_MODE_GLOBAL");
    if (e) return set_error(RWC_ERR_CUDA, "sampler internal check failed");
    if (st) st->mode = RWC_MODE_SHARED;
    return RWC_OK;
}

}  // namespace rwc
