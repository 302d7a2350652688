// Host driver of the batched sampler and of the one-column solve on a stand-in for
// the CUDA runtime.  Batch: it keeps track of device allocations, fails one on
// request and checks that no launch (direct, or replayed from a captured graph) is
// given freed memory and that every launch has as many pulls as trees.  Solve: it
// refuses cooperative launches of more blocks than a limit.
#include <cstdio>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <utility>
#include <vector>

#include <cuda_runtime_api.h>

#include "rwc.h"

static std::map<char *, std::pair<size_t, bool>> blocks;   // address -> size, live
static int fail_in = -1;                                    // allocations until one fails
static int stale = 0, launches = 0;
static int64_t pulls = 0;                                   // pulls launched
static unsigned coop_limit = 0, coop_blocks = 0;            // solve: the limit (0: batch), blocks launched
static unsigned last_grid = 0, last_block = 0;              // the last launch
static bool capturing = false;
static std::vector<char *> captured;                        // pointers of the captured launches

static void check(char *p) {
    auto it = blocks.upper_bound(p);
    if (it == blocks.begin()) { ++stale; return; }
    --it;
    if (p >= it->first + it->second.first || !it->second.second) ++stale;
}

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
    if (fail_in >= 0 && fail_in-- == 0) return cudaErrorMemoryAllocation;
    *p = calloc(1, n);
    blocks[(char *)*p] = {n, true};
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) { if (p) blocks[(char *)p].second = false; return cudaSuccess; }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { capturing = true; captured.clear(); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { capturing = false; *g = (cudaGraph_t)&captured; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)&captured; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { ++launches; for (char *p : captured) check(p); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// what nvcc's host code calls to register and launch kernels
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t, struct CUstream_st *) {
    last_grid = grid.x;
    last_block = block.x;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t cudaLaunchCooperativeKernel(const void *, dim3 grid, dim3, void **, size_t, cudaStream_t) {
    if (grid.x > coop_limit) return cudaErrorCooperativeLaunchTooLarge;
    coop_blocks = grid.x;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *, dim3 grid, dim3, void **, size_t, cudaStream_t) { coop_blocks = grid.x; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *, void **) { coop_blocks = c->gridDim.x; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **args, size_t, cudaStream_t) {
    if (coop_limit) return cudaSuccess;
    // kernel arguments 1, 2 and 10: the graphs' records, the bin's graphs, the
    // pending ends beyond shared memory; 3: pulls
    pulls += *(int64_t *)args[3];
    for (int i : {1, 2, 10}) {
        char *p = *(char **)args[i];
        if (capturing) captured.push_back(p);
        else { ++launches; check(p); }
    }
    return cudaSuccess;
}
}

#define EXPECT(c) do { if (!(c)) { printf("line %d: %s (stale %d, %s)\n", __LINE__, #c, stale, rwc_last_error()); return 1; } } while (0)

// A cycle with unit weights of its own (general rows, many blocks).
static int solve() {
    const int n = 200000;
    std::vector<int64_t> rp{0};
    std::vector<int32_t> col;
    for (int u = 0; u < n; ++u) {
        const int a = (u + n - 1) % n, b = (u + 1) % n;
        col.push_back(a < b ? a : b);
        col.push_back(a < b ? b : a);
        rp.push_back((int64_t)col.size());
    }
    std::vector<float> w(col.size(), 1.f);
    std::vector<double> b(n), x(n);
    for (unsigned limit : {1000u, 60u, 20u, 9u, 8u}) {
        rwc_graph_t *g = nullptr;
        coop_limit = limit;
        EXPECT(rwc_graph_create(n, (int64_t)col.size(), rp.data(), col.data(), w.data(), -1, 0, &g) == RWC_OK);
        EXPECT(rwc_solve(g, 1, b.data(), x.data(), 1e-10, nullptr, nullptr) == RWC_OK);
        EXPECT(coop_blocks <= limit && coop_blocks >= (limit < 100 ? limit / 2 : 100));
        EXPECT(rwc_graph_destroy(g) == RWC_OK);
    }
    printf("ok\n");
    return 0;
}

// Complete graphs: few rows, on a cluster of blocks only while their arcs are few too.
static int dense() {
    for (int n : {250, 400, 900}) {
        std::vector<int64_t> rp{0};
        std::vector<int32_t> col;
        for (int u = 0; u < n; ++u) {
            for (int v = 0; v < n; ++v)
                if (v != u) col.push_back(v);
            rp.push_back((int64_t)col.size());
        }
        std::vector<double> b(n), x(n);
        rwc_graph_t *g = nullptr;
        coop_limit = 1000;
        EXPECT(rwc_graph_create(n, (int64_t)col.size(), rp.data(), col.data(), nullptr, -1, 0, &g) == RWC_OK);
        EXPECT(rwc_solve(g, 1, b.data(), x.data(), 1e-10, nullptr, nullptr) == RWC_OK);
        EXPECT(n == 250 ? coop_blocks <= 8 : (int64_t)coop_blocks >= (int64_t)col.size() / 4096);
        EXPECT(rwc_graph_destroy(g) == RWC_OK);
    }
    printf("ok\n");
    return 0;
}

// One cycle of n vertices, T trees: threads and blocks of the launch.
static int few() {
    const struct { int n, T, per_graph; unsigned threads, blocks; } want[] = {
        {40, 1, 0, 32, 1}, {40, 1, 1, 32, 1}, {40, 9000, 1, 32, 152}, {448, 5, 1, 32, 5}, {449, 5, 1, 256, 5},
        {1500, 1, 0, 256, 1}, {1500, 152, 0, 256, 152}, {1500, 153, 0, 64, 152}, {1500, 152, 1, 256, 152},
        {1500, 153, 1, 64, 152}, {20000, 1, 1, 256, 1}, {20000, 1000, 1, 256, 152}};
    for (const auto &q : want) {
        std::vector<int64_t> voff{0, q.n}, rp{0};
        std::vector<int32_t> col;
        for (int u = 0; u < q.n; ++u) {
            const int a = (u + q.n - 1) % q.n, b = (u + 1) % q.n;
            col.push_back(a < b ? a : b);
            col.push_back(a < b ? b : a);
            rp.push_back((int64_t)col.size());
        }
        std::vector<double> sums(q.n);
        rwc_batch_t *b = nullptr;
        EXPECT(rwc_batch_create(1, voff.data(), rp.data(), col.data(), nullptr, &b) == RWC_OK);
        EXPECT(rwc_batch_sample(b, 1, q.T, sums.data(), 0, q.per_graph, nullptr, nullptr) == RWC_OK);
        EXPECT(last_block == q.threads && last_grid == q.blocks);
        EXPECT(rwc_batch_destroy(b) == RWC_OK);
    }
    printf("ok\n");
    return 0;
}

int main(int argc, char **argv) {
    if (argc > 1 && !strcmp(argv[1], "few")) return few();
    if (argc > 1 && !strcmp(argv[1], "dense")) return dense();
    if (argc > 1 && !strcmp(argv[1], "solve")) return solve();
    const int nth = argc > 1 ? atoi(argv[1]) : -1, use_graph = argc > 2 ? atoi(argv[2]) : 0;
    // two cycles, one for each size class
    const int ns[2] = {40, 1500};
    std::vector<int64_t> voff{0}, rp{0};
    std::vector<int32_t> col;
    for (int n : ns) {
        for (int u = 0; u < n; ++u) {
            const int a = (u + n - 1) % n, b = (u + 1) % n;
            col.push_back(a < b ? a : b);
            col.push_back(a < b ? b : a);
            rp.push_back((int64_t)col.size());
        }
        voff.push_back(voff.back() + n);
    }
    rwc_batch_t *b = nullptr;
    EXPECT(rwc_batch_create(2, voff.data(), rp.data(), col.data(), nullptr, &b) == RWC_OK);
    std::vector<double> sums((size_t)voff[2]);
    for (int T : {1, 5, 6, 7, 4}) {
        pulls = 0;
        EXPECT(rwc_batch_sample(b, 1, T, sums.data(), use_graph, 0, nullptr, nullptr) == RWC_OK);
        EXPECT(pulls == 2 * T);
    }
    fail_in = nth;
    const rwc_status s = rwc_batch_sample(b, 1, 8, sums.data(), use_graph, 0, nullptr, nullptr);
    EXPECT(nth < 0 || fail_in >= 0 ? s == RWC_OK : s == RWC_ERR_OOM);
    fail_in = -1;
    const int before = launches;
    EXPECT(rwc_batch_sample(b, 1, 4, sums.data(), use_graph, 0, nullptr, nullptr) == RWC_OK);
    EXPECT(launches > before && stale == 0);
    EXPECT(rwc_batch_destroy(b) == RWC_OK);
    printf("ok\n");
    return 0;
}
