// Laplacian solves with several right-hand sides (the gradient, rwc_solve).
//
// X = L^+ B for k columns.  Outer loop in FP64: R = B - L X (FP64 sparse product
// over the FP32 weights), columns projected onto 1-perp; inner loop:
// Jacobi-preconditioned conjugate gradients on the k columns together (one
// shared FP32 sparse product per iteration, per-column step sizes), X +=
// correction.  One right-hand side goes to cg1.cu.
//
// Layout: node-major [n][k], the FP32 arrays padded to quads of columns.  A
// thread owns one quad of columns and a slot of rows, so a neighbour row is
// read as consecutive 16-byte loads, the weight and the column index are shared
// by its threads, and the dot products stay in the thread until the end of the
// kernel: four pairs of floats (exact products and sums by FMA and two-sum,
// about 48 bits; FP64 runs at 2 FMA per cycle and SM).  The iteration is three
// passes (product and <p,q>; r and its sums; e and p), whose working set of four
// arrays stays in L2 for 66 columns of 100000 rows.
// Measured (whole gradient calls, a warp per row with FP64 dots -> here): RGG
// 100000, 64 sketch columns 39.7 -> 13.7 ms; BA 100000, 64 columns 42.3 -> 15.1;
// BA 8792, 16 columns 4.7 -> 3.4; RGG 1500, 8 columns 3.1 -> 2.5.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "pair_sum.cuh"
#include "rwc_common.cuh"

namespace rwc {
namespace {

constexpr int TPB = 256;

struct Buf {
    void *p = nullptr;
    cudaStream_t st;
    explicit Buf(cudaStream_t s) : st(s) {}
    ~Buf() { if (p) cudaFreeAsync(p, st); }
};

template <bool OFF64>
__device__ __forceinline__ void rowb(const DevGraph &g, int64_t u, int64_t &b, int64_t &e) {
    if (OFF64) { b = g.rp64[u]; e = g.rp64[u + 1]; }
    else { b = g.rp32[u]; e = g.rp32[u + 1]; }
}

// The threads of a block as quads of columns x rows: quad q (of this block's
// tile) and row slot rs; the slots of all blocks take rows u0, u0 + step, ... in
// turn, so that neighbouring ids, which often are the hubs, fall to different
// blocks.
struct Tile {
    int q, rs, slots;
    int64_t u0, step;
    bool on;
    __device__ Tile(int k4, int qt)
        : q(blockIdx.y * qt + threadIdx.x % qt), rs(threadIdx.x / qt), slots(blockDim.x / qt) {
        u0 = (int64_t)blockIdx.x * slots + rs;
        step = (int64_t)gridDim.x * slots;
        on = q < k4;
    }
};

// parts[column][block] = the sums over the block's row slots by a fixed tree, in
// pairs (a serial FP64 sum of 85 slots took longer than the rest of a small
// system's pass).
__device__ __forceinline__ void quad_parts(const Tile &t, const Pair (&a)[4], int qt, double *parts) {
    __shared__ Pair sh[4][TPB];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) sh[i][threadIdx.x] = a[i];
    int h = 1;
    while (h < t.slots) h *= 2;
    for (h /= 2; h > 0; h /= 2) {
        __syncthreads();
        if (t.rs < h && t.rs + h < t.slots)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                Pair x = sh[i][threadIdx.x];
                const Pair y = sh[i][threadIdx.x + h * qt];
                pair_add(x, y.s, y.c);
                sh[i][threadIdx.x] = x;
            }
    }
    __syncthreads();
    if (t.rs == 0 && t.on)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const Pair x = sh[i][threadIdx.x];
            parts[(int64_t)(4 * t.q + i) * gridDim.x + blockIdx.x] = (double)x.s + (double)x.c;
        }
}

__device__ __forceinline__ void fma4(float4 &s, float w, const float4 &v) {
    s.x = fmaf(w, v.x, s.x); s.y = fmaf(w, v.y, s.y); s.z = fmaf(w, v.z, s.z); s.w = fmaf(w, v.w, s.w);
}
__device__ __forceinline__ void dot4(Pair (&a)[4], const float4 &x, const float4 &y) {
    pair_fma(a[0], x.x, y.x); pair_fma(a[1], x.y, y.y); pair_fma(a[2], x.z, y.z); pair_fma(a[3], x.w, y.w);
}

// Rows of more arcs are shared by a block's slots: one slot takes about 150 cycles
// per arc, so the hub of a BA graph of 9000 vertices alone took longer than the
// rest of the product (gradients with 64 columns, rows of more than 128 and of more than
// 1024 arcs shared: BA 8792 4.84 and 5.82 ms, BA 60000 9.42 and 9.55, BA 100000 15.1 and
// 14.7, R-MAT 65536 54 and 58).
constexpr int WIDE_ROW = 128;

// Q = L P and the parts of <P, Q>.  Four neighbour rows are in flight.
template <bool OFF64, bool W>
__global__ void __launch_bounds__(TPB) bcg_product(DevGraph g, int k4, int qt, const float4 *__restrict__ P,
                                                   float4 *__restrict__ Q, double *parts) {
    const Tile t(k4, qt);
    Pair a[4] = {};
    if (t.on)
        for (int64_t u = t.u0; u < g.n; u += t.step) {
            int64_t b, e;
            rowb<OFF64>(g, u, b, e);
            if (e - b > WIDE_ROW) continue;
            float4 s0 = {}, s1 = {};
            int64_t j = b;
            for (; j + 4 <= e; j += 4) {
                int32_t c[4];
                float w[4];
                float4 v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) { c[i] = g.col[j + i]; w[i] = W ? g.w[j + i] : 1.f; }
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = P[(int64_t)c[i] * k4 + t.q];
                fma4(s0, w[0], v[0]); fma4(s1, w[1], v[1]); fma4(s0, w[2], v[2]); fma4(s1, w[3], v[3]);
            }
            for (; j < e; ++j) fma4(s0, W ? g.w[j] : 1.f, P[(int64_t)g.col[j] * k4 + t.q]);
            const float d = (float)g.d[u];
            const float4 p = P[u * k4 + t.q];
            const float4 q = {d * p.x - (s0.x + s1.x), d * p.y - (s0.y + s1.y), d * p.z - (s0.z + s1.z),
                              d * p.w - (s0.w + s1.w)};
            Q[u * k4 + t.q] = q;
            dot4(a, p, q);
        }
    // longer rows: the block's slots share the arcs of one
    __shared__ float4 hs[TPB];
    for (int64_t base = (int64_t)blockIdx.x * t.slots; base < g.n; base += t.step) {
        int64_t b = 0, e = 0;
        if (base + t.rs < g.n) rowb<OFF64>(g, base + t.rs, b, e);
        if (!__syncthreads_or(e - b > WIDE_ROW)) continue;
        for (int r = 0; r < t.slots && base + r < g.n; ++r) {
            const int64_t u = base + r;
            rowb<OFF64>(g, u, b, e);
            if (e - b <= WIDE_ROW) continue;
            float4 s = {};
            if (t.on)
#pragma unroll 4
                for (int64_t j = b + t.rs; j < e; j += t.slots) fma4(s, W ? g.w[j] : 1.f, P[(int64_t)g.col[j] * k4 + t.q]);
            hs[threadIdx.x] = s;
            int h = 1;
            while (h < t.slots) h *= 2;
            for (h /= 2; h > 0; h /= 2) {
                __syncthreads();
                if (t.rs < h && t.rs + h < t.slots) fma4(hs[threadIdx.x], 1.f, hs[threadIdx.x + h * qt]);
            }
            __syncthreads();
            if (t.rs == 0 && t.on) {
                s = hs[threadIdx.x];
                const float d = (float)g.d[u];
                const float4 p = P[u * k4 + t.q];
                const float4 q = {d * p.x - s.x, d * p.y - s.y, d * p.z - s.z, d * p.w - s.w};
                Q[u * k4 + t.q] = q;
                dot4(a, p, q);
            }
            __syncthreads();
        }
    }
    quad_parts(t, a, qt, parts);
}

// Few columns (at most SHARE_QUADS quads): a block has up to 256 slots, so that a slot's
// serial chain of arcs bounds the product from short rows on.  The lanes of a warp hold
// several arcs of a quad side by side instead: a warp takes each row of 17 to 1024 arcs
// (the last degree bin) by itself, a block's slots share each heavy row.  (Two columns:
// dense n = 1000 7.5 -> 1.15 ms, BA 100000 7.3 -> 2.95, BA 10^6 18.5 -> 6.2; gradient of BA
// 60000 with 34 columns 7.5 -> 5.7.)  Blocks of TPB threads; those beyond the slots
// only help in the warps.
constexpr int SHARE_QUADS = 16, SHARE_ROW = 16;

template <bool OFF64, bool W>
__global__ void __launch_bounds__(TPB) bcg_product_few(DevGraph g, int k4, int qt, const float4 *__restrict__ P,
                                                       float4 *__restrict__ Q, double *parts) {
    const Tile t(k4, qt);
    const bool slot = t.on && t.rs < t.slots;
    Pair a[4] = {};
    auto finish = [&](int64_t u, const float4 &s) {
        const float d = (float)g.d[u];
        const float4 p = P[u * k4 + t.q];
        const float4 q = {d * p.x - s.x, d * p.y - s.y, d * p.z - s.z, d * p.w - s.w};
        Q[u * k4 + t.q] = q;
        dot4(a, p, q);
    };
    if (slot)
        for (int64_t u = t.u0; u < g.n; u += t.step) {
            int64_t b, e;
            rowb<OFF64>(g, u, b, e);
            if (e - b > SHARE_ROW) continue;
            float4 s0 = {}, s1 = {};
            int64_t j = b;
            for (; j + 4 <= e; j += 4) {
                int32_t c[4];
                float w[4];
                float4 v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) { c[i] = g.col[j + i]; w[i] = W ? g.w[j + i] : 1.f; }
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = P[(int64_t)c[i] * k4 + t.q];
                fma4(s0, w[0], v[0]); fma4(s1, w[1], v[1]); fma4(s0, w[2], v[2]); fma4(s1, w[3], v[3]);
            }
            for (; j < e; ++j) fma4(s0, W ? g.w[j] : 1.f, P[(int64_t)g.col[j] * k4 + t.q]);
            fma4(s0, 1.f, s1);
            finish(u, s0);
        }
    {
        // lanes of a warp as arcs x quads (rotated where qt does not divide 32)
        const int lane = threadIdx.x & 31, na = 32 / qt, al = lane / qt;
        const bool on = al < na && t.on;
        int top = 1;
        while (top < na) top *= 2;
        const int32_t *rows = g.bin_rows + g.bin_off[4];
        const int64_t nrows = g.bin_off[5] - g.bin_off[4], nw = (int64_t)gridDim.x * (TPB / 32);
        for (int64_t i = (int64_t)blockIdx.x * (TPB / 32) + (threadIdx.x >> 5); i < nrows; i += nw) {
            const int64_t u = rows[i];
            int64_t b, e;
            rowb<OFF64>(g, u, b, e);
            float4 s = {};
            if (on)
#pragma unroll 4
                for (int64_t j = b + al; j < e; j += na) fma4(s, W ? g.w[j] : 1.f, P[(int64_t)g.col[j] * k4 + t.q]);
            for (int h = top / 2; h > 0; h /= 2) {
                const float4 o = {__shfl_down_sync(0xffffffffu, s.x, h * qt), __shfl_down_sync(0xffffffffu, s.y, h * qt),
                                  __shfl_down_sync(0xffffffffu, s.z, h * qt), __shfl_down_sync(0xffffffffu, s.w, h * qt)};
                if (al < h && al + h < na) fma4(s, 1.f, o);
            }
            if (on && al == 0) finish(u, s);
        }
    }
    __shared__ float4 hs[TPB];
    for (int64_t c = blockIdx.x; c < g.hc_n; c += gridDim.x) {
        const int64_t u = g.hc_row[c];
        int64_t b, e;
        rowb<OFF64>(g, u, b, e);
        if (g.hc_beg[c] != b) continue;          // not the row's first chunk
        float4 s = {};
        if (slot)
#pragma unroll 4
            for (int64_t j = b + t.rs; j < e; j += t.slots) fma4(s, W ? g.w[j] : 1.f, P[(int64_t)g.col[j] * k4 + t.q]);
        hs[threadIdx.x] = s;
        int h = 1;
        while (h < t.slots) h *= 2;
        for (h /= 2; h > 0; h /= 2) {
            __syncthreads();
            if (t.rs < h && t.rs + h < t.slots) fma4(hs[threadIdx.x], 1.f, hs[threadIdx.x + h * qt]);
        }
        __syncthreads();
        if (t.rs == 0 && t.on) finish(u, hs[threadIdx.x]);
        __syncthreads();
    }
    quad_parts(t, a, qt, parts);
}

__device__ __forceinline__ float step_of(double num, double den) {
    return den > 0.0 && num > 0.0 ? (float)(num / den) : 0.f;
}

// r -= alpha q; parts of <r, z> (z = D^-1 r) and <r, r>.  Every parts array is
// [4 k4][gridDim.x].
__global__ void __launch_bounds__(TPB) bcg_residual(int64_t n, int k4, int qt, const double *rz, const double *pq,
                                                    const float *dinv, const float4 *__restrict__ Q,
                                                    float4 *__restrict__ r, double *parts, double *parts2) {
    const Tile t(k4, qt);
    Pair a[4] = {}, b[4] = {};
    if (t.on) {
        const double *z = rz + 4 * t.q, *d = pq + 4 * t.q;
        const float4 al = {step_of(z[0], d[0]), step_of(z[1], d[1]), step_of(z[2], d[2]), step_of(z[3], d[3])};
        for (int64_t u = t.u0; u < n; u += t.step) {
            const int64_t i = u * k4 + t.q;
            const float4 q = Q[i];
            float4 v = r[i];
            v.x -= al.x * q.x; v.y -= al.y * q.y; v.z -= al.z * q.z; v.w -= al.w * q.w;
            r[i] = v;
            const float di = dinv[u];
            dot4(a, v, float4{di * v.x, di * v.y, di * v.z, di * v.w});
            dot4(b, v, v);
        }
    }
    quad_parts(t, a, qt, parts);
    quad_parts(t, b, qt, parts2);
}

// e += alpha p; p = D^-1 r + beta p.
__global__ void __launch_bounds__(TPB) bcg_direction(int64_t n, int k4, int qt, const double *rz0, const double *pq,
                                                     const double *rz1, const float *dinv,
                                                     const float4 *__restrict__ r, float4 *__restrict__ e,
                                                     float4 *__restrict__ p) {
    const Tile t(k4, qt);
    if (!t.on) return;
    const double *z = rz0 + 4 * t.q, *d = pq + 4 * t.q, *z1 = rz1 + 4 * t.q;
    float al[4], be[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        al[i] = step_of(z[i], d[i]);
        be[i] = z[i] > 0.0 ? (float)(z1[i] / z[i]) : 0.f;
    }
    for (int64_t u = t.u0; u < n; u += t.step) {
        const int64_t i = u * k4 + t.q;
        const float di = dinv[u];
        const float4 v = r[i];
        float4 pv = p[i], ev = e[i];
        ev.x += al[0] * pv.x; ev.y += al[1] * pv.y; ev.z += al[2] * pv.z; ev.w += al[3] * pv.w;
        pv.x = di * v.x + be[0] * pv.x; pv.y = di * v.y + be[1] * pv.y;
        pv.z = di * v.z + be[2] * pv.z; pv.w = di * v.w + be[3] * pv.w;
        e[i] = ev;
        p[i] = pv;
    }
}

// Start of an inner solve: r = scale R / |R_c|, e = 0, p = z = D^-1 r, parts of
// <r, z>; columns beyond k are 0.
__global__ void __launch_bounds__(TPB) bcg_start(int64_t n, int k, int k4, int qt, double scale, const double *__restrict__ R,
                                                 const double *rnrm2, const float *dinv, float4 *__restrict__ r,
                                                 float4 *__restrict__ e, float4 *__restrict__ p, double *parts) {
    const Tile t(k4, qt);
    Pair a[4] = {};
    if (t.on) {
        double nr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) nr[i] = 4 * t.q + i < k ? sqrt(rnrm2[4 * t.q + i]) / scale : 0.0;
        for (int64_t u = t.u0; u < n; u += t.step) {
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = nr[i] > 0.0 ? (float)(R[u * k + 4 * t.q + i] / nr[i]) : 0.f;
            const float di = dinv[u];
            const float4 rv = {v[0], v[1], v[2], v[3]}, zv = {di * v[0], di * v[1], di * v[2], di * v[3]};
            const int64_t i = u * k4 + t.q;
            r[i] = rv;
            e[i] = float4{0.f, 0.f, 0.f, 0.f};
            p[i] = zv;
            dot4(a, rv, zv);
        }
    }
    quad_parts(t, a, qt, parts);
}

// X += |R_c| e times unscale, 1 / scale.
__global__ void __launch_bounds__(TPB) bcg_add(int64_t n, int k, int k4, double unscale, const double *rnrm2, const float *e, double *X) {
    const int64_t tot = n * k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tot; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = i / k;
        const int c = (int)(i - u * k);
        X[i] += sqrt(rnrm2[c]) * unscale * (double)e[u * 4 * k4 + c];
    }
}

// R = B - L X in FP64, one thread per (row, column), ct columns per block.
template <bool OFF64, bool W>
__global__ void __launch_bounds__(TPB) resid64(DevGraph g, int k, int ct, const double *__restrict__ B,
                                               const double *__restrict__ X, double *__restrict__ R) {
    const int c = blockIdx.y * ct + threadIdx.x % ct, rs = threadIdx.x / ct, slots = blockDim.x / ct;
    if (c >= k || rs >= slots) return;
    for (int64_t u = blockIdx.x * (int64_t)slots + rs; u < g.n; u += (int64_t)gridDim.x * slots) {
        int64_t b, e;
        rowb<OFF64>(g, u, b, e);
        double s = 0.0;
        int64_t j = b;
        for (; j + 4 <= e; j += 4) {
            double v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = X[(int64_t)g.col[j + i] * k + c];
#pragma unroll
            for (int i = 0; i < 4; ++i) s += (W ? (double)g.w[j + i] : 1.0) * v[i];
        }
        for (; j < e; ++j) s += (W ? (double)g.w[j] : 1.0) * X[(int64_t)g.col[j] * k + c];
        R[u * k + c] = B[u * k + c] - (g.d[u] * X[u * k + c] - s);
    }
}

// Per-column sums of X or X^2 over the rows of a node-major FP64 [n][k] array,
// in a fixed order: block b adds the rows [b rpb, (b + 1) rpb).  With k <
// blockDim, thread t takes column t % k of the rows t / k, t / k + P, ... and
// the phases' sums are added in phase order; otherwise thread t takes the
// columns t, t + blockDim, ... over all the block's rows.  parts[c * gridDim +
// b]; sum_cols adds them in block order.
template <bool SQUARE>
__global__ void __launch_bounds__(TPB) col_parts(int64_t n, int k, const double *__restrict__ A, double *parts) {
    __shared__ double s1[TPB];
    const int nb = gridDim.x, bk = blockIdx.x, t = threadIdx.x;
    const int64_t rpb = (n + nb - 1) / nb;
    const int64_t u0 = bk * rpb, u1 = u0 + rpb < n ? u0 + rpb : n;
    if (k < (int)blockDim.x) {
        const int P = (int)blockDim.x / k, c = t % k, ph = t / k;
        double a = 0.0;
        if (ph < P)
            for (int64_t u = u0 + ph; u < u1; u += P) { const double v = A[u * k + c]; a += SQUARE ? v * v : v; }
        s1[t] = a;
        __syncthreads();
        if (t < k) {
            double r = 0.0;
            for (int q = 0; q < P; ++q) r += s1[q * k + t];
            parts[(int64_t)t * nb + bk] = r;
        }
    } else {
        for (int c = t; c < k; c += blockDim.x) {
            double a = 0.0;
            for (int64_t u = u0; u < u1; ++u) { const double v = A[u * k + c]; a += SQUARE ? v * v : v; }
            parts[(int64_t)c * nb + bk] = a;
        }
    }
}

// A column whose residual is a tenth of the inner tolerance stands still while the
// others go on.  Iterated further its residual is soon the rounding errors along the
// constant vector, on which L is 0: <p, q> is noise, the step is huge and the column
// diverges, and all of them go on for hundreds or thousands of iterations (weighted
// complete graph of 1500 vertices, 7 columns 254 -> 2.7 ms; star of 300, 16 columns 43
// -> 1.05; gradient of the 100 x 100 grid, 64 columns 169 -> 56; a hundredth of the
// tolerance is too late for that grid).
// The step is 0 because sum_cols gives it a <p, q> of 0: the passes over the rows,
// whose FP64 quotients count, know nothing of it.
constexpr double STILL = 0.01;   // (1/10)^2: of squares

// out[c] = sum over b of parts[c * nb + b] in order of b, or 0 for a column whose rr[c]
// is at most `still` (rr = NULL: none); one block per column (blockIdx.y = 1: the
// second set of parts, into out2).
__global__ void __launch_bounds__(128) sum_cols(const double *parts, const double *parts2, int nb, double *out,
                                                double *out2, const double *rr = nullptr, double still = 0.0) {
    const int c = blockIdx.x;
    const double *p = (blockIdx.y ? parts2 : parts) + (int64_t)c * nb;
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s += p[b];
    s = block_sum_fixed(s);
    if (threadIdx.x == 0) (blockIdx.y ? out2 : out)[c] = rr && rr[c] <= still ? 0.0 : s;
}

// V[u][c] -= colsum[c] / n (FP64).
__global__ void center64(int64_t n, int k, double *V, const double *colsum) {
    const int64_t tot = n * k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tot;
         i += (int64_t)gridDim.x * blockDim.x)
        V[i] -= colsum[(int)(i % k)] / (double)n;
}

template <class F>
void dispatch(const DevGraph &g, F f) {
    if (g.off64) {
        if (g.weighted) f(std::true_type{}, std::true_type{});
        else f(std::true_type{}, std::false_type{});
    } else {
        if (g.weighted) f(std::false_type{}, std::true_type{});
        else f(std::false_type{}, std::false_type{});
    }
}

unsigned grid_for(int64_t work) {
    const int64_t cap = (int64_t)num_sms() * 8;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(cap, (work + TPB - 1) / TPB));
}

}  // namespace

// X = L^+ B for node-major FP64 B, X ([n][k]).  Internal entry.
rwc_status solve_nodemajor(rwc_graph *G, int k, const double *B, double *X, double tol,
                           int *iters_out, cudaStream_t st) {
    const DevGraph &g = G->g;
    const int64_t n = g.n;
    if (k <= 0) return set_error(RWC_ERR_INVALID, "k must be positive");
    if (tol <= 0) tol = 1e-10;
    if (k == 1) return solve_one(G, B, X, tol, iters_out, st);
    const int64_t nk = n * k;
    const int max_inner = (int)std::min<int64_t>(200000, std::max<int64_t>(1000, 4 * n));
    const int max_outer = 30;
    const double inner_tol = 1e-5, scale = inner_scale(g);
    const double still = STILL * (inner_tol * scale) * (inner_tol * scale);
    const int k4 = (k + 3) / 4, kp = 4 * k4;
    // blocks: qt quads of columns x TPB / qt row slots; nb row ranges, fewer for
    // many column tiles (the parts are [kp][nb])
    const int qt = std::min(k4, 64), threads = qt * (TPB / qt), tiles = (k4 + qt - 1) / qt;
    const int64_t rows_nb = (n + threads / qt - 1) / (threads / qt);
    // a warp for each row that is not one slot's, a block for each heavy row
    const int64_t wide_nb =
        qt <= SHARE_QUADS ? std::max((g.bin_off[5] - g.bin_off[4] + TPB / 32 - 1) / (TPB / 32), g.hc_n) : 0;
    const unsigned nb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(((int64_t)num_sms() * 6 + tiles - 1) / tiles,
                                                                         std::max(rows_nb, wide_nb)));
    const dim3 grid(nb, (unsigned)tiles);
    const int ct = std::min(k, 128), rthreads = ct * (TPB / ct);
    const dim3 rgrid((unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms() * 8, (n * ct + rthreads - 1) / rthreads)),
                     (unsigned)((k + ct - 1) / ct));
    const unsigned nbc = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms() * 4, (n + 63) / 64));
    Buf buf(st);
    const size_t fbytes = (size_t)n * kp * sizeof(float);
    const size_t nparts = (size_t)kp * std::max(nb, nbc);
    const size_t bytes = (size_t)nk * 8 + 4 * fbytes + 2 * nparts * 8 + (size_t)8 * kp * 8 + 16 * 256;
    RWC_CUDA_TRY(cudaMallocAsync(&buf.p, bytes, st));
    char *at = (char *)buf.p;
    auto take = [&](size_t b) { char *r = at; at += (b + 255) & ~(size_t)255; return r; };
    double *R = (double *)take((size_t)nk * 8);
    float4 *r = (float4 *)take(fbytes), *e = (float4 *)take(fbytes), *p = (float4 *)take(fbytes), *q = (float4 *)take(fbytes);
    double *pa = (double *)take(nparts * 8), *pb = (double *)take(nparts * 8);
    double *colsum = (double *)take((size_t)kp * 8), *rn2 = (double *)take((size_t)kp * 8);
    double *pq = (double *)take((size_t)kp * 8), *rr = (double *)take((size_t)kp * 8);
    double *rz[2] = {(double *)take((size_t)kp * 8), (double *)take((size_t)kp * 8)};
    const unsigned gs = grid_for(nk);
    auto col_sum = [&](auto square, const double *A, double *out) {
        ::rwc::count_launches(2);
        col_parts<decltype(square)::value><<<nbc, TPB, 0, st>>>(n, k, A, pa);
        sum_cols<<<dim3((unsigned)k, 1), 128, 0, st>>>(pa, nullptr, (int)nbc, out, nullptr);
    };
    RWC_CUDA_TRY(cudaMemsetAsync(X, 0, (size_t)nk * sizeof(double), st));
    std::vector<double> h(kp), bn(k);
    int total_iters = 0;
    double prev_worst = INFINITY;
    int slow = 0;
    for (int outer = 0; outer <= max_outer; ++outer) {
        dispatch(g, [&](auto o64, auto wt) {
            ::rwc::count_launches(1);
            resid64<decltype(o64)::value, decltype(wt)::value><<<rgrid, rthreads, 0, st>>>(g, k, ct, B, X, R);
        });
        col_sum(std::false_type{}, R, colsum);
        ::rwc::count_launches(1);
        center64<<<gs, TPB, 0, st>>>(n, k, R, colsum);
        col_sum(std::true_type{}, R, rn2);
        RWC_CUDA_TRY(cudaGetLastError());
        RWC_CUDA_TRY(cudaMemcpyAsync(h.data(), rn2, (size_t)k * 8, cudaMemcpyDeviceToHost, st));
        RWC_CUDA_TRY(cudaStreamSynchronize(st));
        if (outer == 0)
            for (int c = 0; c < k; ++c) bn[c] = std::sqrt(h[c]);
        double worst = 0.0;
        for (int c = 0; c < k; ++c) {
            const double rel = bn[c] > 0 ? std::sqrt(h[c]) / bn[c] : 0.0;
            if (!(rel == rel)) return set_error(RWC_ERR_NOT_CONVERGED, "solver produced NaN");
            worst = std::max(worst, rel);
        }
        if (worst <= tol) break;
        if (worst < 0.5 * prev_worst) { prev_worst = worst; slow = 0; }
        else if (++slow >= 4)
            return set_error(RWC_ERR_NOT_CONVERGED, "Laplacian solve stalled at relative residual %.3g (tol %.3g)", worst, tol);
        if (outer == max_outer)
            return set_error(RWC_ERR_NOT_CONVERGED, "Laplacian solve reached %d refinements at relative residual %.3g (tol %.3g)", max_outer, worst, tol);
        // inner FP32 PCG on the normalised residual
        ::rwc::count_launches(2);
        bcg_start<<<grid, threads, 0, st>>>(n, k, k4, qt, scale, R, rn2, g.dinv32, r, e, p, pa);
        sum_cols<<<dim3((unsigned)kp, 1), 128, 0, st>>>(pa, nullptr, (int)nb, rz[0], nullptr);
        RWC_CUDA_TRY(cudaMemsetAsync(rr, 0x7f, (size_t)kp * 8, st));   // 1e306: every column starts
        int it = 0;
        // iterations between looks at the residual (a host round trip each)
        const int check = (int64_t)n * kp >= 1000000 ? 4 : 8;
        bool inner_done = false;
        double best = INFINITY;
        int since_best = 0;
        while (!inner_done && it < max_inner) {
            for (int j = 0; j < check && it < max_inner; ++j, ++it) {
                double *z0 = rz[it & 1], *z1 = rz[(it & 1) ^ 1];
                ::rwc::count_launches(5);
                dispatch(g, [&](auto o64, auto wt) {
                    constexpr bool O = decltype(o64)::value, W = decltype(wt)::value;
                    if (qt <= SHARE_QUADS) bcg_product_few<O, W><<<grid, TPB, 0, st>>>(g, k4, qt, p, q, pa);
                    else bcg_product<O, W><<<grid, threads, 0, st>>>(g, k4, qt, p, q, pa);
                });
                sum_cols<<<dim3((unsigned)kp, 1), 128, 0, st>>>(pa, nullptr, (int)nb, pq, nullptr, rr, still);
                bcg_residual<<<grid, threads, 0, st>>>(n, k4, qt, z0, pq, g.dinv32, q, r, pa, pb);
                sum_cols<<<dim3((unsigned)kp, 2), 128, 0, st>>>(pa, pb, (int)nb, z1, rr);
                bcg_direction<<<grid, threads, 0, st>>>(n, k4, qt, z0, pq, z1, g.dinv32, r, e, p);
            }
            RWC_CUDA_TRY(cudaGetLastError());
            RWC_CUDA_TRY(cudaMemcpyAsync(h.data(), rr, (size_t)k * 8, cudaMemcpyDeviceToHost, st));
            RWC_CUDA_TRY(cudaStreamSynchronize(st));
            double w2 = 0.0;
            bool bad = false;
            for (int c = 0; c < k; ++c) {
                bad = bad || !(h[c] == h[c]);
                w2 = std::max(w2, h[c]);
            }
            if (std::sqrt(w2) <= inner_tol * scale || bad) inner_done = true;
            // FP32 stagnation: the residual norm has not halved for 1024
            // iterations; CG residuals are not monotone, so the window is long
            if (w2 < 0.25 * best) { best = w2; since_best = 0; }
            else if (++since_best >= 1024 / check) inner_done = true;
        }
        total_iters += it;
        ::rwc::count_launches(1);
        bcg_add<<<gs, TPB, 0, st>>>(n, k, k4, 1.0 / scale, rn2, (const float *)e, X);
        RWC_CUDA_TRY(cudaGetLastError());
    }
    // final projection of X onto 1-perp
    col_sum(std::false_type{}, X, colsum);
    ::rwc::count_launches(1);
    center64<<<gs, TPB, 0, st>>>(n, k, X, colsum);
    RWC_CUDA_TRY(cudaGetLastError());
    if (iters_out) *iters_out = total_iters;
    return RWC_OK;
}

}  // namespace rwc
