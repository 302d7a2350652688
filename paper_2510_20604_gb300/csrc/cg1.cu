// LapSolve for one right-hand side, x = L^+ b, in one launch: FP64 residual
// refinement around Jacobi-preconditioned conjugate gradients in FP32, all of it
// in a cooperative kernel (the host reads one status at the end).
//
// What bounds it: FP64 arithmetic (2 FMA per cycle and SM), grid barriers and
// L2 latency, in that order for the earlier kernel.  So
//   - the iteration's sums are taken in pairs of floats (exact products and
//     sums by FMA and two-sum, about 48 bits) up to one value per warp;
//   - the direction p = z + beta p is formed where the sparse product gathers
//     it, from (z, p) pairs in two buffers used in turn, so an iteration has
//     two grid barriers (<p,q>; <r,z> and <r,r>) and no pass for p;
//   - graphs of bounded degree keep a thread's rows of e, r, p, q in registers
//     and their inline neighbour rows in shared memory.
// Measured (pivot solve and recovery, one kernel per inner solve with FP64 dots
// and three grid barriers -> here): 1024 x 1024 grid 369 -> 122 ms (45 -> 14.8 us
// per iteration), R-MAT 20 21.4 -> 12.7 ms, BA 2000 0.67 -> 0.37 ms, ER 100 0.54
// -> 0.18 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include <cooperative_groups.h>

#include "pair_sum.cuh"
#include "rwc_common.cuh"

namespace cg = cooperative_groups;

namespace rwc {
namespace {

constexpr int CSR_TPB = 512;
constexpr int ELL_TPB = 1024;
constexpr int ELL_RMAX = 7;             // rows per thread held in registers
constexpr int64_t CG_FUSED_MAX = 8000000;
constexpr int CG_WINDOW = 1024;         // iterations without a halved residual: stagnation
constexpr double CG_INNER_TOL = 1e-5;

struct CgArgs {
    DevGraph g;
    const double *B;
    double *X, *R;
    const float *d32;                   // [n] degrees
    float *e, *r, *q;                   // [n] (not used by the register kernel)
    float2 *zp[2];                      // [n] (z, p) of the last iteration, in turn
    float *hsum;                        // heavy chunks' sums, FP32 and FP64
    double *hsumd;
    double *parts;                      // [2][2][gridDim] block sums, in turn
    double tol;
    double scale;                       // |r| of an inner solve's start (inner_scale)
    int max_outer, max_inner;
    int use_smem;                       // inline rows fit shared memory
    bool clustered;                     // the blocks are one cluster
    double *out;                        // iterations, relative residual, status
};
enum : int { CG_OK = 0, CG_NAN = 1, CG_STALLED = 2, CG_MAX_OUTER = 3 };

// All blocks: one cluster (its barrier is a few hundred cycles) or the grid.
__device__ __forceinline__ void blocks_sync(bool clustered) {
    if (clustered) cg::this_cluster().sync();
    else cg::this_grid().sync();
}
__device__ __forceinline__ void all_sync(bool clustered) {
    if (gridDim.x > 1) blocks_sync(clustered);
    else __syncthreads();
}

// a + b over the lanes of a warp by a shuffle tree, the same bits in every lane.
__device__ __forceinline__ double warp_tree(double a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}
template <int K>
__device__ __forceinline__ void warp_tree(Pair (&v)[K]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float s2 = __shfl_xor_sync(0xffffffffu, v[k].s, o), c2 = __shfl_xor_sync(0xffffffffu, v[k].c, o);
            // both partners add the same pair in the same order
            Pair lo = (lane & o) ? Pair{s2, c2} : v[k];
            const Pair hi = (lane & o) ? v[k] : Pair{s2, c2};
            pair_add(lo, hi.s, hi.c);
            v[k] = lo;
        }
}
template <int K>
__device__ __forceinline__ void warp_tree(double (&v)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = warp_tree(v[k]);
}
__device__ __forceinline__ Pair load_part(const Pair *p) {
    const float2 v = __ldcg(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ double load_part(const double *p) { return __ldcg(p); }
__device__ __forceinline__ void add_part(Pair &a, const Pair &b) { pair_add(a, b.s, b.c); }
__device__ __forceinline__ void add_part(double &a, double b) { a += b; }

// Fixed-order sums over the grid of K values per thread (FP64, or pairs of
// floats on the iteration's path: an FP64 addition costs ten times a pair's
// there): a shuffle tree in every warp, the warps of a block, then the blocks.
// Thread 0 of every block passes them to post(sums), which gets the same bits in
// every block and returns what all threads get.  `flip` alternates the blocks'
// slots, so that a block can write its next sums while another still reads
// these.
template <int K, class Out, class T, class Post>
__device__ Out grid_sums(T (&v)[K], double *parts, int &flip, bool clustered, Post post) {
    static_assert(sizeof(T) == 8, "a slot");
    __shared__ T ws[K][32];
    __shared__ Out bc;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nb = gridDim.x;
    T *slot = reinterpret_cast<T *>(parts) + (size_t)flip * 2 * nb;
    flip ^= 1;
    warp_tree(v);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) ws[k][wid] = v[k];
    __syncthreads();
    T t[K];
    if (wid == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) t[k] = lane < nw ? ws[k][lane] : T{};
        warp_tree(t);
        if (nb > 1 && lane == 0)
#pragma unroll
            for (int k = 0; k < K; ++k) slot[(size_t)k * nb + blockIdx.x] = t[k];
    }
    if (nb > 1) {
        blocks_sync(clustered);
        if (wid == 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) t[k] = T{};
            for (int i = lane; i < nb; i += 32)
#pragma unroll
                for (int k = 0; k < K; ++k) add_part(t[k], load_part(slot + (size_t)k * nb + i));
            warp_tree(t);
        }
    }
    if (threadIdx.x == 0) bc = post(t);
    __syncthreads();
    return bc;
}

template <bool OFF64>
__device__ __forceinline__ void row_of(const DevGraph &g, int64_t u, int64_t &b, int64_t &e) {
    if (OFF64) { b = g.rp64[u]; e = g.rp64[u + 1]; }
    else { b = g.rp32[u]; e = g.rp32[u + 1]; }
}

// ------------------------------------------------------- general sparse rows
// f(u, sum) for the rows of a degree bin, VW lanes per row (rows of at most VW
// arcs, or more than 16 for VW = 32), term(arc) summed in type T.  Several rows
// per group of lanes (arcs per lane for VW = 32) are in flight, since a row is
// a chain of four dependent loads.
template <int VW, bool OFF64, class T, class Term, class F>
__device__ __forceinline__ void bin_rows(const DevGraph &g, int bin, Term term, F f) {
    constexpr int NR = VW == 32 ? 1 : 4;
    const int32_t *rows = g.bin_rows + g.bin_off[bin];
    const int64_t nrows = g.bin_off[bin + 1] - g.bin_off[bin];
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t ngroups = (int64_t)gridDim.x * blockDim.x / VW;
    const int sub = threadIdx.x & (VW - 1);
    const int64_t mine = tid / VW, first = mine - mine % (32 / VW);
    for (int64_t i0 = first; i0 < nrows; i0 += NR * ngroups) {
        int32_t u[NR];
        int64_t b[NR], e[NR];
        T s[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const int64_t i = i0 + (mine - first) + k * ngroups;
            u[k] = i < nrows ? rows[i] : -1;
        }
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            b[k] = e[k] = 0;
            if (u[k] >= 0) row_of<OFF64>(g, u[k], b[k], e[k]);
        }
        if (VW == 32) {
            T s4[4] = {};
            for (int64_t j = b[0] + sub; j < e[0]; j += 128) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (j + 32 * k < e[0]) s4[k] += term(j + 32 * k);
            }
            s[0] = (s4[0] + s4[1]) + (s4[2] + s4[3]);
        } else {
#pragma unroll
            for (int k = 0; k < NR; ++k) s[k] = b[k] + sub < e[k] ? term(b[k] + sub) : (T)0;
        }
#pragma unroll
        for (int k = 0; k < NR; ++k) {
#pragma unroll
            for (int o = VW / 2; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o, VW);
            if (sub == 0 && u[k] >= 0) f(u[k], s[k]);
        }
    }
}
// The same rows where there are few: a warp takes units of 32 / VW rows of any
// bin in turn, so that the bins' chains of loads run side by side.
template <int VW, bool OFF64, class T, class Term, class F>
__device__ __forceinline__ void one_unit(const DevGraph &g, int bin, int64_t unit, Term term, F f) {
    const int lane = threadIdx.x & 31, sub = lane & (VW - 1);
    const int64_t i = unit * (32 / VW) + lane / VW;
    const int64_t nrows = g.bin_off[bin + 1] - g.bin_off[bin];
    int32_t u = -1;
    int64_t b = 0, e = 0;
    if (i < nrows) { u = g.bin_rows[g.bin_off[bin] + i]; row_of<OFF64>(g, u, b, e); }
    T s = 0;
    if (VW == 32) {
        T s4[4] = {};
        for (int64_t j = b + sub; j < e; j += 128) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (j + 32 * k < e) s4[k] += term(j + 32 * k);
        }
        s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
    } else if (b + sub < e) {
        s = term(b + sub);
    }
#pragma unroll
    for (int o = VW / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, VW);
    if (sub == 0 && u >= 0) f(u, s);
}
template <bool OFF64, class T, class Term, class F>
__device__ __forceinline__ bool few_rows(const DevGraph &g, Term term, F f) {
    const int64_t warps = (int64_t)gridDim.x * blockDim.x / 32;
    int64_t end[5], total = 0;
#pragma unroll
    for (int b = 0; b < 5; ++b) {
        const int rows = 16 >> b;
        total += (g.bin_off[b + 1] - g.bin_off[b] + rows - 1) / rows;
        end[b] = total;
    }
    if (total > 8 * warps) return false;
    for (int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; w < total; w += warps) {
        if (w < end[0]) one_unit<2, OFF64, T>(g, 0, w, term, f);
        else if (w < end[1]) one_unit<4, OFF64, T>(g, 1, w - end[0], term, f);
        else if (w < end[2]) one_unit<8, OFF64, T>(g, 2, w - end[1], term, f);
        else if (w < end[3]) one_unit<16, OFF64, T>(g, 3, w - end[2], term, f);
        else one_unit<32, OFF64, T>(g, 4, w - end[3], term, f);
    }
    return true;
}
// A warp's units of rows held in registers for the whole solve (small systems):
// row, first arc and weight of every lane.  An iteration then waits for one
// gather instead of a chain of four loads per unit, which the barrier's acquire
// sends to L2 each time (BA 2000: 13500 -> 4700 cycles per product).
constexpr int RES_UNITS = 4, RES_TPB = 1024;
constexpr int64_t RES_ARCS = 80000;
template <bool OFF64, bool W>
struct ResidentRows {
    int32_t u[RES_UNITS], c[RES_UNITS];
    float w[RES_UNITS];
    int32_t more[RES_UNITS];               // arcs of the lane beyond the first, 32 apart
    int vw[RES_UNITS];
    __device__ void load(const DevGraph &g) {
        const int64_t warps = (int64_t)gridDim.x * blockDim.x / 32;
        const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32;
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int q = 0; q < RES_UNITS; ++q) {
            int64_t unit = w0 + q * warps;
            u[q] = c[q] = -1;
            w[q] = 0.f;
            more[q] = 0;
            vw[q] = 0;
            for (int b = 0; b < 5; ++b) {
                const int rows = 16 >> b, v = 2 << b;
                const int64_t nrows = g.bin_off[b + 1] - g.bin_off[b], nu = (nrows + rows - 1) / rows;
                if (unit < nu) {
                    vw[q] = v;
                    const int64_t i = unit * rows + lane / v;
                    if (i < nrows) {
                        u[q] = g.bin_rows[g.bin_off[b] + i];
                        int64_t rb, re;
                        row_of<OFF64>(g, u[q], rb, re);
                        const int64_t j = rb + (lane & (v - 1));
                        if (j < re) {
                            c[q] = g.col[j];
                            w[q] = W ? g.w[j] : 1.f;
                            more[q] = (int32_t)((re - 1 - j) / 32);
                        }
                    }
                    break;
                }
                unit -= nu;
            }
        }
    }
    // f(row, sum over its arcs of weight times dir(head))
    template <class Dir, class F>
    __device__ __forceinline__ void rows(const DevGraph &g, Dir dir, F f) const {
        const int lane = threadIdx.x & 31;
        float s[RES_UNITS];
#pragma unroll
        for (int q = 0; q < RES_UNITS; ++q) s[q] = c[q] >= 0 ? w[q] * dir(c[q]) : 0.f;
#pragma unroll
        for (int q = 0; q < RES_UNITS; ++q) {
            if (vw[q] == 32) {
                int64_t rb = 0, re;
                if (more[q]) row_of<OFF64>(g, u[q], rb, re);
                for (int k = 1; k <= more[q]; ++k) {
                    const int64_t j = rb + lane + 32 * (int64_t)k;
                    s[q] += (W ? g.w[j] : 1.f) * dir(g.col[j]);
                }
                __syncwarp();
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (o < vw[q]) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
            if (u[q] >= 0 && (lane & (vw[q] - 1)) == 0) f(u[q], s[q]);
        }
    }
};
// Units of a graph's rows, a heavy row's chunks among them.
inline int64_t row_units(const DevGraph &g) {
    int64_t t = g.hc_n;
    for (int b = 0; b < 5; ++b) t += (g.bin_off[b + 1] - g.bin_off[b] + (16 >> b) - 1) / (16 >> b);
    return t;
}
// all rows of at most HEAVY_DEG arcs through f, the heavy rows' chunks through
// h(chunk, row, first chunk of its row, sum)
template <bool OFF64, class T, class Term, class F, class H>
__device__ __forceinline__ void all_rows(const DevGraph &g, Term term, F f, H h) {
    if (!few_rows<OFF64, T>(g, term, f)) {
        bin_rows<2, OFF64, T>(g, 0, term, f);
        bin_rows<4, OFF64, T>(g, 1, term, f);
        bin_rows<8, OFF64, T>(g, 2, term, f);
        bin_rows<16, OFF64, T>(g, 3, term, f);
        bin_rows<32, OFF64, T>(g, 4, term, f);
    }
    const int lane = threadIdx.x & 31;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nthr = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = tid / 32; c < g.hc_n; c += nthr / 32) {
        const int32_t u = g.hc_row[c];
        int64_t rb, re;
        row_of<OFF64>(g, u, rb, re);
        const int64_t b = g.hc_beg[c], e = min(b + HEAVY_CHUNK, re);
        T s4[4] = {};
        for (int64_t j = b + lane; j < e; j += 128) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (j + 32 * k < e) s4[k] += term(j + 32 * k);
        }
        T s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) h(c, u, b == rb, s);
    }
}
// all rows of a graph of bounded degree by their inline neighbours, one thread
// per row, several rows in flight: f(row, sum of get(neighbour))
template <int EW, class T, class Get, class F>
__device__ __forceinline__ void inline_rows(const DevGraph &g, Get get, F f) {
    constexpr int NR = EW == 4 ? 4 : 2, E4 = EW / 4;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nthr = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = tid; i < g.n; i += NR * nthr) {
        int4 c[NR][E4];
        T s[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k)
#pragma unroll
            for (int j = 0; j < E4; ++j)
                c[k][j] = i + k * nthr < g.n ? __ldg(g.ell + (i + k * nthr) * E4 + j) : make_int4(-1, -1, -1, -1);
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            s[k] = 0;
#pragma unroll
            for (int j = 0; j < E4; ++j) {
                const int4 q = c[k][j];
                const T v0 = q.x >= 0 ? get(q.x) : (T)0, v1 = q.y >= 0 ? get(q.y) : (T)0;
                const T v2 = q.z >= 0 ? get(q.z) : (T)0, v3 = q.w >= 0 ? get(q.w) : (T)0;
                s[k] += v0; s[k] += v1; s[k] += v2; s[k] += v3;
            }
        }
#pragma unroll
        for (int k = 0; k < NR; ++k)
            if (i + k * nthr < g.n) f((int32_t)(i + k * nthr), s[k]);
    }
}
// sum of a heavy row's chunks in chunk order
template <bool OFF64, class T>
__device__ __forceinline__ T heavy_sum(const DevGraph &g, int64_t u, const T *hsum) {
    int64_t rb, re;
    row_of<OFF64>(g, u, rb, re);
    const int64_t nc = (re - rb + HEAVY_CHUNK - 1) / HEAVY_CHUNK;
    T s = 0;
    for (int64_t c = 0; c < nc; ++c) s += hsum[g.hfirst[u] + c];
    return s;
}

// Outer loop shared by both kernels: INNER runs the conjugate gradients on R /
// |R| times the scale and adds the correction to X; RESID fills R = B - L X and returns this
// thread's share of its sum; EACH visits the thread's rows.
template <class Resid, class Each, class Inner>
__device__ void refine(const CgArgs &a, int &flip, Resid resid, Each each, Inner inner) {
    const double n = (double)a.g.n;
    double bn = 0.0, prev = INFINITY, worst = 0.0;
    int total = 0, slow = 0, status = CG_MAX_OUTER;
    for (int outer = 0; outer <= a.max_outer; ++outer) {
        double sum[1] = {resid()};
        const double mean = grid_sums<1, double>(sum, a.parts, flip, a.clustered, [&](const double *t) { return t[0] / n; });
        sum[0] = 0.0;
        each([&](int64_t i) {
            const double v = a.R[i] - mean;
            a.R[i] = v;
            sum[0] += v * v;
        });
        const double rn = grid_sums<1, double>(sum, a.parts, flip, a.clustered, [&](const double *t) { return sqrt(t[0]); });
        if (outer == 0) bn = rn;
        worst = bn > 0 ? rn / bn : 0.0;
        if (!(worst == worst)) { status = CG_NAN; break; }
        if (worst <= a.tol) { status = CG_OK; break; }
        if (worst < 0.5 * prev) { prev = worst; slow = 0; }
        else if (++slow >= 4) { status = CG_STALLED; break; }
        if (outer == a.max_outer) break;
        total += inner(rn);
    }
    // X onto 1-perp
    double sum[1] = {0.0};
    each([&](int64_t i) { sum[0] += a.X[i]; });
    const double mean = grid_sums<1, double>(sum, a.parts, flip, a.clustered, [&](const double *t) { return t[0] / n; });
    each([&](int64_t i) { a.X[i] -= mean; });
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.out[0] = (double)total;
        a.out[1] = worst;
        a.out[2] = (double)status;
    }
}

// num / den to float precision: a float quotient corrected by its residual.
__device__ __forceinline__ float quotient(Pair num, Pair den) {
    const float q = __fdiv_rn(num.s, den.s);
    const float r = __fadd_rn(__fmaf_rn(-q, den.s, num.s), __fmaf_rn(-q, den.c, num.c));
    return __fadd_rn(q, __fdividef(r, den.s));
}
// the pair's value as its leading float, the rest in c
__device__ __forceinline__ Pair normal(Pair a) {
    const float t = __fadd_rn(a.s, a.c);
    return {t, __fsub_rn(a.c, __fsub_rn(t, a.s))};
}

// Step length and direction factor with their guards, and the exit test of the
// inner iteration: thread 0's, the same in every block.
struct Inner {
    Pair rz = {0.f, 0.f};
    float stop;                             // <r, r> that ends the iteration
    float best = INFINITY;
    int since = 0;
    __device__ explicit Inner(double scale) : stop((float)(CG_INNER_TOL * scale * (CG_INNER_TOL * scale))) {}
    __device__ float step(Pair den) const {
        den = normal(den);
        return den.s > 0.f && rz.s > 0.f ? quotient(rz, den) : 0.f;
    }
    // the direction factor, and whether the iteration ends
    __device__ float2 next(Pair rz1, Pair rr2) {
        rz1 = normal(rz1);
        const float rr = normal(rr2).s;
        if (!(rr == rr) || rr <= stop) return make_float2(0.f, 1.f);
        if (rr < 0.25f * best) { best = rr; since = 0; }
        else if (++since >= CG_WINDOW) return make_float2(0.f, 1.f);
        const float beta = rz.s > 0.f ? quotient(rz1, rz) : 0.f;
        rz = rz1;
        return make_float2(beta, 0.f);
    }
};

// FUSED: the direction is formed from (z, p) pairs as it is gathered; else it is
// an array of its own with a pass and a barrier per iteration, for systems whose
// pairs do not stay in L2 while the directions do.  EW: inline rows of EW slots,
// for graphs of bounded degree with more rows than cg1_ell holds (0: CSR).
template <bool OFF64, bool W, bool RES, bool FUSED, int EW = 0>
__global__ void __launch_bounds__(RES ? RES_TPB : CSR_TPB, RES ? 1 : 2) cg1_csr(CgArgs a) {
    const DevGraph &g = a.g;
    const int64_t n = g.n;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nthr = (int64_t)gridDim.x * blockDim.x;
    int flip = 0;
    auto each = [&](auto f) { for (int64_t i = tid; i < n; i += nthr) f(i); };
    auto resid = [&]() -> double {
        double s = 0.0;
        auto row = [&](int32_t u, double t) { a.R[u] = a.B[u] - (g.d[u] * a.X[u] - t); };
        if constexpr (EW > 0)
            inline_rows<EW, double>(g, [&](int32_t v) { return a.X[v]; }, row);
        else
            all_rows<OFF64, double>(g, [&](int64_t j) { return (W ? (double)g.w[j] : 1.0) * a.X[g.col[j]]; }, row,
                                    [&](int64_t c, int32_t, bool, double t) { a.hsumd[c] = t; });
        all_sync(a.clustered);
        each([&](int64_t i) {
            if (g.hc_n && g.hfirst[i] >= 0)
                a.R[i] = a.B[i] - (g.d[i] * a.X[i] - heavy_sum<OFF64, double>(g, i, a.hsumd));
            s += a.R[i];
        });
        return s;
    };
    float *p1 = reinterpret_cast<float *>(a.zp[0]), *z1 = reinterpret_cast<float *>(a.zp[1]);   // !FUSED
    ResidentRows<OFF64, W> held;
    if constexpr (RES) held.load(g);
    auto inner = [&](double rn) -> int {
        const double rs = rn / a.scale;
        Pair acc[1] = {{0.f, 0.f}};
        each([&](int64_t i) {
            const float rv = (float)(a.R[i] / rs), zv = g.dinv32[i] * rv;
            a.r[i] = rv;
            a.e[i] = 0.f;
            if (FUSED) a.zp[0][i] = make_float2(zv, 0.f);
            else p1[i] = zv;
            pair_fma(acc[0], rv, zv);
        });
        Inner s(a.scale);
        float beta = grid_sums<1, float>(acc, a.parts, flip, a.clustered, [&](const Pair *t) { s.rz = normal(t[0]); return 0.f; });
        int it = 0;
        while (it < a.max_inner) {
            const float2 *zi = a.zp[it & 1];
            float2 *zo = a.zp[(it & 1) ^ 1];
            // q = L p, <p, q>; a heavy row's share of <p, q> comes from its chunks
            Pair pq[1] = {{0.f, 0.f}};
            auto dir = [&](int64_t v) -> float {
                if (!FUSED) return p1[v];
                const float2 t = zi[v];
                return fmaf(beta, t.y, t.x);
            };
            auto row = [&](int32_t u, float t) {
                const float pu = dir(u), qu = a.d32[u] * pu - t;
                a.q[u] = qu;
                pair_fma(pq[0], pu, qu);
            };
            auto chunk = [&](int64_t c, int32_t u, bool start, float t) {
                a.hsum[c] = t;
                const float pu = dir(u);
                if (start) pair_fma(pq[0], pu, a.d32[u] * pu);
                pair_fma(pq[0], -pu, t);
            };
            auto term = [&](int64_t j) { return (W ? g.w[j] : 1.f) * dir(g.col[j]); };
            if constexpr (RES) held.rows(g, dir, row);
            else if constexpr (EW > 0) inline_rows<EW, float>(g, dir, row);
            else all_rows<OFF64, float>(g, term, row, chunk);
            const float al = grid_sums<1, float>(pq, a.parts, flip, a.clustered, [&](const Pair *t) { return s.step(t[0]); });
            Pair z2[2] = {{0.f, 0.f}, {0.f, 0.f}};
            each([&](int64_t i) {
                const float pi = dir(i);
                const float qi = g.hc_n && g.hfirst[i] >= 0 ? a.d32[i] * pi - heavy_sum<OFF64, float>(g, i, a.hsum) : a.q[i];
                a.e[i] += al * pi;
                const float rv = a.r[i] - al * qi;
                a.r[i] = rv;
                const float zv = g.dinv32[i] * rv;
                if (FUSED) zo[i] = make_float2(zv, pi);
                else z1[i] = zv;
                pair_fma(z2[0], rv, zv);
                pair_fma(z2[1], rv, rv);
            });
            const float2 nx = grid_sums<2, float2>(z2, a.parts, flip, a.clustered, [&](const Pair *t) { return s.next(t[0], t[1]); });
            ++it;
            beta = nx.x;
            if (nx.y != 0.f) break;
            if (!FUSED) {
                each([&](int64_t i) { p1[i] = z1[i] + beta * p1[i]; });
                all_sync(a.clustered);
            }
        }
        each([&](int64_t i) { a.X[i] += rs * (double)a.e[i]; });
        all_sync(a.clustered);
        return it;
    };
    refine(a, flip, resid, each, inner);
}

// Bounded degree: block b owns consecutive rows, thread t of it the rows t, t +
// ELL_TPB, ... (RT of them), whose e, r, p and q stay in registers.
template <int EW, int RT>
__global__ void __launch_bounds__(ELL_TPB, 1) cg1_ell(CgArgs a) {
    extern __shared__ int4 rows_s[];
    const DevGraph &g = a.g;
    const int n = (int)g.n;
    const int rpb = (n + gridDim.x - 1) / gridDim.x;
    const int row0 = blockIdx.x * rpb, nrow = max(0, min(rpb, n - row0));
    int flip = 0;
    constexpr int E4 = EW / 4;
    if (a.use_smem) {
        for (int i = threadIdx.x; i < nrow * E4; i += ELL_TPB) rows_s[i] = g.ell[(int64_t)row0 * E4 + i];
        __syncthreads();
    }
    // sum over the row's neighbours of get(v)
    auto row_sum = [&](int l, auto zero, auto get) {
        auto s = zero;
#pragma unroll
        for (int k = 0; k < E4; ++k) {
            const int4 c = a.use_smem ? rows_s[l * E4 + k] : __ldg(g.ell + (int64_t)(row0 + l) * E4 + k);
            const auto v0 = c.x >= 0 ? get(c.x) : zero, v1 = c.y >= 0 ? get(c.y) : zero;
            const auto v2 = c.z >= 0 ? get(c.z) : zero, v3 = c.w >= 0 ? get(c.w) : zero;
            s += v0; s += v1; s += v2; s += v3;
        }
        return s;
    };
    auto each = [&](auto f) { for (int l = threadIdx.x; l < nrow; l += ELL_TPB) f((int64_t)(row0 + l)); };
    auto resid = [&]() -> double {
        double s = 0.0;
        for (int l = threadIdx.x; l < nrow; l += ELL_TPB) {
            const int64_t u = row0 + l;
            const double v = a.B[u] - (g.d[u] * a.X[u] - row_sum(l, 0.0, [&](int c) { return a.X[c]; }));
            a.R[u] = v;
            s += v;
        }
        return s;
    };
    auto inner = [&](double rn) -> int {
        const double rs = rn / a.scale;
        float e[RT], r[RT], p[RT], q[RT], d[RT];
        Pair acc[1] = {{0.f, 0.f}};
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const int l = threadIdx.x + i * ELL_TPB;
            e[i] = r[i] = p[i] = q[i] = 0.f;
            d[i] = 1.f;
            if (l < nrow) {
                const int64_t u = row0 + l;
                d[i] = a.d32[u];
                r[i] = (float)(a.R[u] / rs);
                const float zv = r[i] * __fdividef(1.f, d[i]);
                a.zp[0][u] = make_float2(zv, 0.f);
                pair_fma(acc[0], r[i], zv);
            }
        }
        Inner s(a.scale);
        float beta = grid_sums<1, float>(acc, a.parts, flip, a.clustered, [&](const Pair *t) { s.rz = normal(t[0]); return 0.f; });
        int it = 0;
        while (it < a.max_inner) {
            const float2 *zi = a.zp[it & 1];
            float2 *zo = a.zp[(it & 1) ^ 1];
            Pair pq[1] = {{0.f, 0.f}};
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const int l = threadIdx.x + i * ELL_TPB;
                if (l < nrow) {
                    p[i] = fmaf(beta, p[i], r[i] * __fdividef(1.f, d[i]));
                    const float t = row_sum(l, 0.f, [&](int c) { const float2 v = zi[c]; return fmaf(beta, v.y, v.x); });
                    q[i] = d[i] * p[i] - t;
                    pair_fma(pq[0], p[i], q[i]);
                }
            }
            const float al = grid_sums<1, float>(pq, a.parts, flip, a.clustered, [&](const Pair *t) { return s.step(t[0]); });
            Pair z2[2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const int l = threadIdx.x + i * ELL_TPB;
                if (l < nrow) {
                    e[i] += al * p[i];
                    r[i] -= al * q[i];
                    const float zv = r[i] * __fdividef(1.f, d[i]);
                    zo[row0 + l] = make_float2(zv, p[i]);
                    pair_fma(z2[0], r[i], zv);
                    pair_fma(z2[1], r[i], r[i]);
                }
            }
            const float2 nx = grid_sums<2, float2>(z2, a.parts, flip, a.clustered, [&](const Pair *t) { return s.next(t[0], t[1]); });
            ++it;
            beta = nx.x;
            if (nx.y != 0.f) break;
        }
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const int l = threadIdx.x + i * ELL_TPB;
            if (l < nrow) a.X[row0 + l] += rs * (double)e[i];
        }
        all_sync(a.clustered);
        return it;
    };
    refine(a, flip, resid, each, inner);
}

__global__ void degrees32(int64_t n, const double *d, float *d32, double *X) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        d32[i] = (float)d[i];
        X[i] = 0.0;
    }
}

struct Buf {
    void *p = nullptr;
    cudaStream_t st;
    explicit Buf(cudaStream_t s) : st(s) {}
    ~Buf() { if (p) cudaFreeAsync(p, st); }
};

}  // namespace

rwc_status solve_one(rwc_graph *G, const double *B, double *X, double tol, int *iters_out, cudaStream_t st) {
    const DevGraph &g = G->g;
    const int64_t n = g.n;
    const int sms = num_sms();
    // the grid: rows in registers where they fit, else blocks for about four
    // arcs a thread (small graphs in one block need no grid barrier)
    const bool ell = g.ell && n <= (int64_t)sms * ELL_TPB * ELL_RMAX;
    int rt = 1;
    while (ell && (n + (int64_t)ELL_TPB * rt - 1) / ((int64_t)ELL_TPB * rt) > sms) rt = rt == 1 ? 2 : rt == 2 ? 4 : ELL_RMAX;
    // small systems: rows in registers, up to a cluster of blocks (the smallest
    // take one block of half the threads: ER 100 178 against 215 us).  Registers hold
    // one arc per lane, so beyond about 10000 arcs a block the rest streams through too
    // few SMs (complete graphs of 400, 700 and 1000 vertices, weighted: 492, 582 and 736
    // us so, 453, 504 and 526 on up to 304 blocks; ER 1000 of mean degree 40 and 80: 541 and
    // 524 against 559 and 501).
    const int64_t units = row_units(g);
    const bool held = !ell && g.hc_n == 0 && units > 64 && units <= 8 * (RES_TPB / 32) * RES_UNITS && g.nnz <= RES_ARCS;
    int64_t blocks = ell ? (n + (int64_t)ELL_TPB * rt - 1) / ((int64_t)ELL_TPB * rt)
                         : held ? (units <= RES_TPB / 32 * RES_UNITS ? 1 : std::min<int64_t>(8, (units + 63) / 64))
                         : units <= 64 ? 1
                         : std::min<int64_t>(2 * sms, g.nnz / (4 * CSR_TPB));
    const size_t rows_b = ell ? (size_t)((n + blocks - 1) / blocks) * g.ell_w * 4 : 0;
    const size_t smem = rows_b <= 200 * 1024 ? rows_b : 0;
    Buf buf(st);
    const size_t np = (size_t)(n + 31) & ~(size_t)31;
    const size_t parts_b = (size_t)4 * std::max<int64_t>(2 * sms, blocks) * 8;
    const size_t bytes = np * (8 + 4 + 3 * 4 + 2 * 8) + (size_t)(g.hc_n + 1) * 12 + parts_b + 16 * 256;
    RWC_CUDA_TRY(cudaMallocAsync(&buf.p, bytes, st));
    CgArgs a{};
    char *q = (char *)buf.p;
    auto take = [&](size_t b) { char *r = q; q += (b + 255) & ~(size_t)255; return r; };
    a.out = (double *)take(256);
    a.R = (double *)take(np * 8);
    a.zp[0] = (float2 *)take(np * 8);
    a.zp[1] = (float2 *)take(np * 8);
    float *d32 = (float *)take(np * 4);
    a.e = (float *)take(np * 4);
    a.r = (float *)take(np * 4);
    a.q = (float *)take(np * 4);
    a.hsumd = (double *)take((size_t)(g.hc_n + 1) * 8);
    a.hsum = (float *)take((size_t)(g.hc_n + 1) * 4);
    a.parts = (double *)take(parts_b);
    a.g = g;
    a.B = B;
    a.X = X;
    a.d32 = d32;
    a.tol = tol;
    a.scale = inner_scale(g);
    a.max_outer = 30;
    a.max_inner = (int)std::min<int64_t>(200000, std::max<int64_t>(1000, 4 * n));
    a.use_smem = smem > 0;
    ::rwc::count_launches(2);
    degrees32<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(4 * sms, (n + 255) / 256)), 256, 0, st>>>(n, g.d, d32, X);
    RWC_CUDA_TRY(cudaGetLastError());
    void *args[] = {&a};
    // up to eight blocks are one cluster
    a.clustered = blocks > 1 && blocks <= 8;
    auto launch = [&](auto kern, int tpb, size_t sm, int64_t nb) -> cudaError_t {
        if (sm > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(200 * 1024));
            if (e != cudaSuccess) return e;
        }
        if (nb == 1) return cudaLaunchKernel((const void *)kern, dim3(1), dim3(tpb), args, sm, st);
        if (nb <= 8) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)nb);
            cfg.blockDim = dim3(tpb);
            cfg.dynamicSmemBytes = sm;
            cfg.stream = st;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)nb;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            return cudaLaunchKernelExC(&cfg, (const void *)kern, args);
        }
        return cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)nb), dim3(tpb), args, sm, st);
    };
    // pairs of 8 bytes in half of the 126 MB L2 or not
    const bool fused = n <= CG_FUSED_MAX;
    auto csr_of = [&](auto res, auto fu, int tpb, int64_t nb) -> cudaError_t {
        constexpr bool RES = decltype(res)::value, FU = decltype(fu)::value;
        if (g.off64)
            return g.weighted ? launch(cg1_csr<true, true, RES, FU>, tpb, 0, nb) : launch(cg1_csr<true, false, RES, FU>, tpb, 0, nb);
        return g.weighted ? launch(cg1_csr<false, true, RES, FU>, tpb, 0, nb) : launch(cg1_csr<false, false, RES, FU>, tpb, 0, nb);
    };
    auto csr = [&](int64_t nb) -> cudaError_t {
        if (g.ell) {
            // more rows than cg1_ell's registers hold
            if (fused) return g.ell_w == 4 ? launch(cg1_csr<false, false, false, true, 4>, CSR_TPB, 0, nb)
                                           : launch(cg1_csr<false, false, false, true, 8>, CSR_TPB, 0, nb);
            return g.ell_w == 4 ? launch(cg1_csr<false, false, false, false, 4>, CSR_TPB, 0, nb)
                                : launch(cg1_csr<false, false, false, false, 8>, CSR_TPB, 0, nb);
        }
        if (held && nb == blocks) return csr_of(std::true_type{}, std::true_type{}, RES_TPB, nb);
        if (fused) return csr_of(std::false_type{}, std::true_type{}, CSR_TPB, nb);
        return csr_of(std::false_type{}, std::false_type{}, CSR_TPB, nb);
    };
    auto inl = [&](auto ew) -> cudaError_t {
        constexpr int EW = decltype(ew)::value;
        return rt == 1 ? launch(cg1_ell<EW, 1>, ELL_TPB, smem, blocks) : rt == 2 ? launch(cg1_ell<EW, 2>, ELL_TPB, smem, blocks)
             : rt == 4 ? launch(cg1_ell<EW, 4>, ELL_TPB, smem, blocks) : launch(cg1_ell<EW, ELL_RMAX>, ELL_TPB, smem, blocks);
    };
    cudaError_t e = !ell ? csr(blocks) : g.ell_w == 4 ? inl(std::integral_constant<int, 4>{}) : inl(std::integral_constant<int, 8>{});
    // a device or context that does not hold that many blocks at once: as many as it does
    for (int64_t nb = blocks / 2; e != cudaSuccess && nb >= 1; nb /= 2) {
        (void)cudaGetLastError();
        a.clustered = nb > 1 && nb <= 8;
        e = csr(nb);
    }
    RWC_CUDA_TRY(e);
    double h[3];
    RWC_CUDA_TRY(cudaMemcpyAsync(h, a.out, sizeof(h), cudaMemcpyDeviceToHost, st));
    RWC_CUDA_TRY(cudaStreamSynchronize(st));
    if (iters_out) *iters_out = (int)h[0];
    switch ((int)h[2]) {
        case CG_OK: return RWC_OK;
        case CG_NAN: return set_error(RWC_ERR_NOT_CONVERGED, "solver produced NaN");
        case CG_STALLED:
            return set_error(RWC_ERR_NOT_CONVERGED, "Laplacian solve stalled at relative residual %.3g (tol %.3g)", h[1], tol);
        default:
            return set_error(RWC_ERR_NOT_CONVERGED, "Laplacian solve reached %d refinements at relative residual %.3g (tol %.3g)",
                             a.max_outer, h[1], tol);
    }
}

}  // namespace rwc
