// Evaluation measures of Section 6: the mean relative error of an estimate
// and the Kendall distance of two rankings, on the device.
//
// MRE = (1/n) sum_u |H_u - H~_u| / H_u: block partial sums in a fixed order,
// then one block adds the partials in a fixed order (deterministic).
//
// K(L1, L2) = 2 (alpha - beta) / (n (n - 1)) with alpha / beta the concordant
// / discordant pairs (tied pairs count neither way).  Each double becomes an
// order-preserving 64-bit key (-0.0 merged into +0.0 so that the two compare
// equal, as they do as doubles).
//   Few elements: every pair i < j is compared once.  A block keeps 4 rows per
// thread in registers and streams a tile of 2048 keys through shared memory;
// O(n^2) comparisons, ALU bound.
//   Else by sorting: in order of (a, b) the discordant pairs are the inversions
// of b, so alpha - beta = n (n - 1) / 2 - T_a - T_b + T_ab - 2 inversions, T the
// pairs tied in a, in b and in both.  A merge sort orders the pairs, a second
// one the b keys with the inversions counted in its merges; ties are counted in
// the sorted arrays.  Latency bound: 2 log2(n / 2048) passes over 16 and 8 bytes
// per element with a binary search in L2 at the start of each.
// All counts are 64-bit integers added by atomics: exact, order independent.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "rwc_common.cuh"

namespace rwc {
namespace {

constexpr int MRE_THREADS = 256;
constexpr int MRE_BLOCKS = 1024;

__global__ void mre_partial(int64_t n, const double *H, const double *He, double *part) {
    __shared__ double sh[MRE_THREADS];
    double acc = 0.0;
    for (int64_t u = blockIdx.x * (int64_t)MRE_THREADS + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * MRE_THREADS)
        acc += fabs(H[u] - He[u]) / H[u];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = MRE_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void mre_final(int nb, int64_t n, const double *part, double *out) {
    __shared__ double sh[MRE_THREADS];
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += MRE_THREADS) acc += part[i];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = MRE_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0] / (double)n;
}

// Predicted MRE (variance law of the visit counts): block partial sums of
// sqrt(t (t - 1) / T) / (pi_u |H_u|) over u != v, t = sums_u / T.
__global__ void pmre_partial(int64_t n, const double *d, double vol, int32_t v, const double *sums,
                             double invT, const double *H, double *part) {
    __shared__ double sh[MRE_THREADS];
    double acc = 0.0;
    for (int64_t u = blockIdx.x * (int64_t)MRE_THREADS + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * MRE_THREADS) {
        if (u == v) continue;
        const double t = sums[u] * invT;
        const double se = sqrt(fmax(t * (t - 1.0), 0.0) * invT) / (d[u] / vol);
        acc += se / fabs(H[u]);
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = MRE_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

constexpr int KT_THREADS = 256;
constexpr int KT_ROWS = 4;                          // rows per thread
constexpr int KT_BI = KT_THREADS * KT_ROWS;         // rows per block
constexpr int KT_BJ = 2048;                         // columns per shared tile

// Order-preserving key of a double: a > b  <=>  key(a) > key(b) (no NaN).
__device__ __forceinline__ uint64_t okey(double x) {
    uint64_t b = (uint64_t)__double_as_longlong(x);
    if (b == 0x8000000000000000ull) b = 0;          // -0.0 == +0.0
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__device__ __forceinline__ int sgn_cmp(uint64_t p, uint64_t q) { return (int)(p > q) - (int)(p < q); }

__global__ void __launch_bounds__(KT_THREADS) kendall_tiles(int64_t n, const double *a, const double *b,
                                                           unsigned long long *out) {
    __shared__ uint64_t ka[KT_BJ], kb[KT_BJ];
    __shared__ long long red[KT_THREADS / 32];
    const int64_t i0 = (int64_t)blockIdx.x * KT_BI;
    const int64_t j0 = (int64_t)blockIdx.y * KT_BJ;
    // pairs i < j only: a tile wholly at or below the diagonal has none
    if (j0 + KT_BJ - 1 <= i0) return;
    const int64_t jn = min((int64_t)KT_BJ, n - j0);
    for (int t = threadIdx.x; t < jn; t += KT_THREADS) {
        ka[t] = okey(a[j0 + t]);
        kb[t] = okey(b[j0 + t]);
    }
    uint64_t ra[KT_ROWS], rb[KT_ROWS];
    int64_t ri[KT_ROWS];
#pragma unroll
    for (int r = 0; r < KT_ROWS; ++r) {
        ri[r] = i0 + threadIdx.x + (int64_t)r * KT_THREADS;
        ra[r] = ri[r] < n ? okey(a[ri[r]]) : 0;
        rb[r] = ri[r] < n ? okey(b[ri[r]]) : 0;
    }
    __syncthreads();
    int cnt = 0;
    const bool above = j0 > i0 + KT_BI - 1;     // every j of the tile exceeds every i
    if (above) {
        // rows past n contribute nothing only if masked: keep them out
        bool live[KT_ROWS];
#pragma unroll
        for (int r = 0; r < KT_ROWS; ++r) live[r] = ri[r] < n;
        for (int t = 0; t < jn; ++t) {
            const uint64_t xa = ka[t], xb = kb[t];
#pragma unroll
            for (int r = 0; r < KT_ROWS; ++r)
                if (live[r]) cnt += sgn_cmp(ra[r], xa) * sgn_cmp(rb[r], xb);
        }
    } else {
        for (int t = 0; t < jn; ++t) {
            const uint64_t xa = ka[t], xb = kb[t];
            const int64_t j = j0 + t;
#pragma unroll
            for (int r = 0; r < KT_ROWS; ++r)
                if (ri[r] < j) cnt += sgn_cmp(ra[r], xa) * sgn_cmp(rb[r], xb);
        }
    }
    long long v = cnt;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long s = 0;
        for (int w = 0; w < KT_THREADS / 32; ++w) s += red[w];
        if (s) atomicAdd(out, (unsigned long long)s);
    }
}

// ------------------------------------------------------- sorting and inversions
constexpr int MS_THREADS = 256, MS_ITEMS = 8, MS_TILE = MS_THREADS * MS_ITEMS;

struct KeyPair { uint64_t a, b; };
__device__ __forceinline__ bool after(const KeyPair &x, const KeyPair &y) { return x.a > y.a || (x.a == y.a && x.b > y.b); }
__device__ __forceinline__ bool after(uint64_t x, uint64_t y) { return x > y; }
__device__ __forceinline__ KeyPair last_key(KeyPair) { return {~0ull, ~0ull}; }
__device__ __forceinline__ uint64_t last_key(uint64_t) { return ~0ull; }

// Elements of L among the first d of the stable merge of L (nl) and R (nr): the
// diagonal search of merge path (Odeh, Green, Mwassi, Shmueli, Birk 2012).
template <class K, class I>
__device__ __forceinline__ I merge_split(const K *L, I nl, const K *R, I nr, I d) {
    I lo = d > nr ? d - nr : 0, hi = d < nl ? d : nl;
    while (lo < hi) {
        const I m = (lo + hi) >> 1;
        if (!after(L[m], R[d - 1 - m])) lo = m + 1;
        else hi = m;
    }
    return lo;
}

// MS_ITEMS outputs of the merge from (i, j) on; COUNT: the elements of L that
// come after each element taken from R (inversions), with `rest` more of them
// behind L.
template <bool COUNT, class K>
__device__ __forceinline__ void merge_items(const K *L, int nl, const K *R, int nr, int i, int j, int64_t rest,
                                            K (&out)[MS_ITEMS], unsigned long long &inv) {
#pragma unroll
    for (int q = 0; q < MS_ITEMS; ++q) {
        const bool left = j >= nr || (i < nl && !after(L[i], R[j]));
        if (i >= nl && j >= nr) { out[q] = last_key(K{}); continue; }
        out[q] = left ? L[i] : R[j];
        if (COUNT && !left) inv += (unsigned long long)(nl - i + rest);
        i += left;
        j += !left;
    }
}

__device__ __forceinline__ void add_count(unsigned long long v, unsigned long long *out, unsigned long long factor) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(out, v * factor);
}

// Sorts each tile of MS_TILE keys in shared memory: eight keys per thread by
// insertion, then merges of neighbouring runs.  load(i): key i.  COUNT adds
// `factor` per inversion to *out.
template <bool COUNT, class K, class Load>
__device__ void sort_tile(int64_t n, Load load, K *dst, unsigned long long *out, unsigned long long factor) {
    __shared__ K sh[MS_TILE];
    const int64_t t0 = (int64_t)blockIdx.x * MS_TILE;
    const int m = (int)min((int64_t)MS_TILE, n - t0);
    const int tid = threadIdx.x;
    K k[MS_ITEMS];
    unsigned long long inv = 0;
    for (int i = tid; i < MS_TILE; i += MS_THREADS) sh[i] = i < m ? load(t0 + i) : last_key(K{});
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MS_ITEMS; ++q) k[q] = sh[tid * MS_ITEMS + q];
    // odd-even transposition: a swap of neighbours removes one inversion
#pragma unroll
    for (int r = 0; r < MS_ITEMS; ++r)
#pragma unroll
        for (int q = r & 1; q + 1 < MS_ITEMS; q += 2)
            if (after(k[q], k[q + 1])) {
                const K x = k[q];
                k[q] = k[q + 1];
                k[q + 1] = x;
                if (COUNT) ++inv;
            }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MS_ITEMS; ++q) sh[tid * MS_ITEMS + q] = k[q];
    for (int len = MS_ITEMS; len < MS_TILE; len *= 2) {
        __syncthreads();
        const int p = tid * MS_ITEMS, base = p & ~(2 * len - 1), d = p - base;
        const K *L = sh + base, *R = L + len;
        const int i = merge_split(L, len, R, len, d);
        merge_items<COUNT>(L, len, R, len, i, d - i, 0, k, inv);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < MS_ITEMS; ++q) sh[p + q] = k[q];
    }
    __syncthreads();
    for (int i = tid; i < m; i += MS_THREADS) dst[t0 + i] = sh[i];
    if (COUNT) add_count(inv, out, factor);
}
__global__ void __launch_bounds__(MS_THREADS) sort_pairs(int64_t n, const double *a, const double *b, KeyPair *dst) {
    sort_tile<false, KeyPair>(n, [&](int64_t i) { return KeyPair{okey(a[i]), okey(b[i])}; }, dst, nullptr, 0);
}
__global__ void __launch_bounds__(MS_THREADS) sort_keys(int64_t n, const KeyPair *src, uint64_t *dst,
                                                       unsigned long long *out) {
    // every inversion takes two off alpha - beta
    sort_tile<true, uint64_t>(n, [&](int64_t i) { return src[i].b; }, dst, out, ~0ull - 1);
}

// Merges neighbouring runs of len keys (a multiple of MS_TILE), one tile of the
// output per block.
template <bool COUNT, class K>
__global__ void __launch_bounds__(MS_THREADS) merge_runs(int64_t n, int64_t len, const K *src, K *dst,
                                                        unsigned long long *out, unsigned long long factor) {
    __shared__ K sh[MS_TILE];
    __shared__ int64_t split[2];
    const int tid = threadIdx.x;
    const int64_t p0 = (int64_t)blockIdx.x * MS_TILE;
    const int64_t base = p0 / (2 * len) * (2 * len);
    const int64_t nl = min(len, n - base), nr = max((int64_t)0, min(len, n - base - len));
    const int64_t d0 = p0 - base, d1 = min(d0 + MS_TILE, nl + nr);
    const K *L = src + base, *R = L + len;
    if (tid < 2) split[tid] = merge_split<K, int64_t>(L, nl, R, nr, tid ? d1 : d0);
    __syncthreads();
    const int64_t i0 = split[0], i1 = split[1], j0 = d0 - i0;
    const int ml = (int)(i1 - i0), m = (int)(d1 - d0), mr = m - ml;
    for (int i = tid; i < m; i += MS_THREADS) sh[i] = i < ml ? L[i0 + i] : R[j0 + i - ml];
    __syncthreads();
    K k[MS_ITEMS];
    unsigned long long inv = 0;
    const int d = min(tid * MS_ITEMS, m);
    const int i = merge_split<K, int>(sh, ml, sh + ml, mr, d);
    merge_items<COUNT>(sh, ml, sh + ml, mr, i, d - i, nl - i1, k, inv);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MS_ITEMS; ++q)
        if (tid * MS_ITEMS + q < m) sh[tid * MS_ITEMS + q] = k[q];
    __syncthreads();
    for (int q = tid; q < m; q += MS_THREADS) dst[p0 + q] = sh[q];
    if (COUNT) add_count(inv, out, factor);
}

// Pairs of equal keys in a sorted array: every key that equals the one before
// it finds the start of its run.
template <class Same>
__device__ unsigned long long tied_before(int64_t i, Same same) {
    if (i == 0 || !same(i - 1)) return 0;
    int64_t lo = 0, hi = i - 1;            // the first index whose key is the same
    while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        if (same(m)) hi = m;
        else lo = m + 1;
    }
    return (unsigned long long)(i - lo);
}
// *out += n (n - 1) / 2 - T_a - T_b + T_ab.
__global__ void __launch_bounds__(256) kendall_ties(int64_t n, const KeyPair *s, const uint64_t *b, unsigned long long *out) {
    unsigned long long v = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const KeyPair x = s[i];
        const uint64_t y = b[i];
        v += (unsigned long long)i;        // adds up to n (n - 1) / 2
        v -= tied_before(i, [&](int64_t j) { return s[j].a == x.a; });
        v += tied_before(i, [&](int64_t j) { return s[j].a == x.a && s[j].b == x.b; });
        v -= tied_before(i, [&](int64_t j) { return b[j] == y; });
    }
    add_count(v, out, 1ull);
}

// alpha - beta by sorting; scratch: 2 n KeyPairs.
void kendall_sorted(int64_t n, const double *a, const double *b, KeyPair *scratch, unsigned long long *out, cudaStream_t st) {
    const unsigned tiles = (unsigned)((n + MS_TILE - 1) / MS_TILE);
    KeyPair *src = scratch, *dst = scratch + n;
    count_launches(3);
    sort_pairs<<<tiles, MS_THREADS, 0, st>>>(n, a, b, src);
    for (int64_t len = MS_TILE; len < n; len *= 2) {
        count_launches(1);
        merge_runs<false, KeyPair><<<tiles, MS_THREADS, 0, st>>>(n, len, src, dst, nullptr, 0);
        std::swap(src, dst);
    }
    uint64_t *k0 = reinterpret_cast<uint64_t *>(dst), *k1 = k0 + n;   // the other half holds two key arrays
    sort_keys<<<tiles, MS_THREADS, 0, st>>>(n, src, k0, out);
    for (int64_t len = MS_TILE; len < n; len *= 2) {
        count_launches(1);
        merge_runs<true, uint64_t><<<tiles, MS_THREADS, 0, st>>>(n, len, k0, k1, out, ~0ull - 1);
        std::swap(k0, k1);
    }
    kendall_ties<<<(unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 8), 256, 0, st>>>(n, src, k0, out);
}

// Up to this many elements all pairs are compared: one launch in place of 9 to 11
// passes of about 10 us (whole calls, all pairs and by sorting: n = 8300 0.353 and 0.380
// ms, 16000 0.358 and 0.384, 20000 0.540 and 0.405, 32000 0.86 and 0.40): 16384 elements
// are the last whose tiles are one wave of blocks.
constexpr int64_t KENDALL_PAIRS_MAX = 16384;

}  // namespace
}  // namespace rwc

extern "C" rwc_status rwc_mre(int64_t n, const double *H, const double *H_est, double *out,
                              rwc_stream_t stream_) {
    using namespace rwc;
    clear_error();
    if (n < 1 || !H || !H_est || !out) return set_error(RWC_ERR_INVALID, "rwc_mre: n >= 1 and non-NULL pointers required");
    cudaStream_t stream = (cudaStream_t)stream_;
    const int nb = (int)std::min<int64_t>(MRE_BLOCKS, (n + MRE_THREADS - 1) / MRE_THREADS);
    double *part = nullptr;
    RWC_CUDA_TRY(cudaMallocAsync(&part, sizeof(double) * nb, stream));
    count_launches(2);
    mre_partial<<<nb, MRE_THREADS, 0, stream>>>(n, H, H_est, part);
    mre_final<<<1, MRE_THREADS, 0, stream>>>(nb, n, part, out);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(part, stream);
    RWC_CUDA_TRY(e);
    return RWC_OK;
}

extern "C" rwc_status rwc_kendall(int64_t n, const double *a, const double *b, int64_t *out_diff,
                                  double *host_tau, rwc_stream_t stream_) {
    using namespace rwc;
    clear_error();
    if (n < 0 || !out_diff || (n > 0 && (!a || !b)))
        return set_error(RWC_ERR_INVALID, "rwc_kendall: n >= 0 and non-NULL pointers required");
    if (n > ((int64_t)1 << 26))
        return set_error(RWC_ERR_INVALID, "rwc_kendall: n must be at most 2^26");
    cudaStream_t stream = (cudaStream_t)stream_;
    RWC_CUDA_TRY(cudaMemsetAsync(out_diff, 0, sizeof(int64_t), stream));
    KeyPair *scratch = nullptr;
    if (n > KENDALL_PAIRS_MAX && cudaMallocAsync((void **)&scratch, (size_t)n * 2 * sizeof(KeyPair), stream) != cudaSuccess) {
        (void)cudaGetLastError();          // no room to sort: compare all pairs
        scratch = nullptr;
    }
    if (scratch) {
        kendall_sorted(n, a, b, scratch, (unsigned long long *)out_diff, stream);
        const cudaError_t e = cudaGetLastError();
        cudaFreeAsync(scratch, stream);
        RWC_CUDA_TRY(e);
    } else if (n >= 2) {
        const dim3 grid((unsigned)((n + KT_BI - 1) / KT_BI), (unsigned)((n + KT_BJ - 1) / KT_BJ));
        count_launches(1);
        kendall_tiles<<<grid, KT_THREADS, 0, stream>>>(n, a, b, (unsigned long long *)out_diff);
        RWC_CUDA_TRY(cudaGetLastError());
    }
    if (host_tau) {
        int64_t s = 0;
        RWC_CUDA_TRY(cudaMemcpyAsync(&s, out_diff, sizeof(s), cudaMemcpyDeviceToHost, stream));
        RWC_CUDA_TRY(cudaStreamSynchronize(stream));
        *host_tau = n >= 2 ? 2.0 * (double)s / ((double)n * (double)(n - 1)) : 0.0;
    }
    return RWC_OK;
}

extern "C" rwc_status rwc_predict_mre(rwc_graph_t *G, const double *sums, int64_t num_trees,
                                      const double *H, double target, double *host_mre,
                                      int64_t *host_trees, rwc_stream_t stream_) {
    using namespace rwc;
    clear_error();
    if (!G || !sums || !H || !host_mre || num_trees <= 0)
        return set_error(RWC_ERR_INVALID, "rwc_predict_mre: graph, sums, H, host_mre and num_trees > 0 required");
    const DevGraph &g = G->g;
    const int64_t n = g.n;
    cudaStream_t stream = (cudaStream_t)stream_;
    const int nb = (int)std::min<int64_t>(MRE_BLOCKS, (n + MRE_THREADS - 1) / MRE_THREADS);
    double *part = nullptr;
    RWC_CUDA_TRY(cudaMallocAsync(&part, sizeof(double) * (nb + 1), stream));
    count_launches(2);
    pmre_partial<<<nb, MRE_THREADS, 0, stream>>>(n, g.d, g.vol, g.root, sums, 1.0 / (double)num_trees, H, part);
    mre_final<<<1, MRE_THREADS, 0, stream>>>(nb, n, part, part + nb);
    cudaError_t e = cudaGetLastError();
    double m = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&m, part + nb, sizeof(double), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    cudaFreeAsync(part, stream);
    RWC_CUDA_TRY(e);
    *host_mre = std::sqrt(2.0 / M_PI) * m;
    if (host_trees && target > 0.0)
        *host_trees = (int64_t)std::ceil((double)num_trees * (*host_mre / target) * (*host_mre / target));
    return RWC_OK;
}
