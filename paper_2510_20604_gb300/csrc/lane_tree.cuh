// One rooted spanning tree per group of threads (a warp or a block): cycle
// popping by many lanes at once, in rounds.
//
// Every vertex has one word [ go | p' | k ]: k its pop count, p' = 0 while its
// current successor succ(u, k) has not been drawn (a pending end), 1 + id while
// lane id works on it (an active end), else id0 + its successor; go = 1 on
// chain vertices, 0 on ends and on settled ones (id0 <= p').  The words form a
// forest of successor chains that lead to ends or to the tree.
// A round has three phases with a group barrier after each:
//   draw   idle lanes take pending ends (popped ones first, last in first out,
//          then vertices that were never an end, in order of id); every lane
//          with a new end e draws succ(e, k) and makes e active;
//   chase  lanes follow the chain from succ(e, k).  Nothing is written.  A lane
//          stops at a settled vertex, at another end, or at its own;
//   act    settled: e's chain belongs to the tree and is marked settled.
//          Another end: no cycle can close through e before that end has
//          moved, so e becomes an ordinary chain vertex (it parks).  Its own
//          end: a cycle of the top graph, which is popped: k + 1 on each of its
//          vertices, which become pending ends; the lane draws again for e.
// Every pop is a genuine cycle of the top graph, so by Wilson's cycle-popping
// theorem the tree and the counts are the sequential algorithm's.  When no end
// is left every chain leads to the root.  Why no lock is needed:
//   - a cycle holds exactly one active end, so one lane pops it; cycles,
//     settled chains and the lanes' own ends are disjoint sets of words;
//   - lanes whose ends meet in one round: of lane i stopped at j's end with j
//     itself stopped at a foreign end, only i > j parks, so no ring of parked
//     ends is left without an active one;
//   - a chase that goes on over several rounds can lose the part behind it
//     only to a pop of the cycle it is in, whose vertices are then ends, and
//     one that runs into the end of a cycle still being popped may have lost
//     it: both start again from their own end.
//
// What bounds it: the dependent word load of a hop (shared memory or L1 about
// 40 cycles, L2 300, HBM 800) and, with one warp per scheduler, the latency of
// the instructions between two loads; so a hop is a load, a shift and a sign
// test, with the go bit left in the successor's number (base is moved by it).
#pragma once

#include "rwc_common.cuh"

namespace rwc {

constexpr int LE_KOVF = 1;   // a pop count exceeded the caller's limit
constexpr int LE_KREP = 2;   // a pop count exceeded the word's field
constexpr int LE_LOOP = 4;   // internal: steps without a draw exceeded their bound

constexpr uint32_t LT_STACK = 192;       // pending ends kept in shared memory, per warp
constexpr int LT_HOPS = 32;              // hops of a chase per round
constexpr int LT_ACT = 16;               // steps of marking and popping per round

// dst |= the status bits of a sampler's LE_* error word.  One thread.
static __global__ void fold_lane_status(const int *err, int *dst) {
    const int e = *err;
    if (e)
        atomicOr(dst, ((e & LE_KOVF) ? STATUS_KOVF : 0) | ((e & (LE_LOOP | LE_KREP)) ? STATUS_INTERNAL : 0));
}

// p' of successor v is v + lt_id0(lanes per tree).  Inside lane_tree a
// vertex's number includes the go bit above p' ("raw": word >> kb of a chain
// vertex that points to it).
__host__ __device__ constexpr uint32_t lt_id0(int nl) { return (uint32_t)nl + 2u; }
// Bits of p' for graphs of n vertices and nl lanes per tree.
__host__ __device__ inline int lt_pbits(int64_t n, int nl) {
    int b = 7;
    while (((int64_t)1 << b) < n + (int64_t)lt_id0(nl)) ++b;
    return b;
}
// Bits of k in a word of type W.
template <class W>
__host__ __device__ inline int lt_kbits(int64_t n, int nl) { return sizeof(W) == 8 ? 32 : 31 - lt_pbits(n, nl); }

// The row of a vertex that is drawn: its CSR bounds (EW = 0), or, for graphs
// whose degrees are at most EW (4 or 8), its inline neighbour list (heads in
// arc order, -1 after the last), read with one or two 16-byte loads.
template <bool OFF64, int EW>
struct DrawRow {
    int4 e[EW / 4];
    __device__ __forceinline__ void load(const DevGraph &g, int32_t u) {
#pragma unroll
        for (int i = 0; i < EW / 4; ++i) e[i] = __ldg(g.ell + (int64_t)u * (EW / 4) + i);
    }
    // head of the arc picked by the 32-bit uniform x: arc floor(x deg / 2^32)
    __device__ __forceinline__ int32_t pick(uint32_t x) const {
        uint32_t deg = 0;
#pragma unroll
        for (int i = 0; i < EW / 4; ++i)
            deg += (e[i].x >= 0) + (e[i].y >= 0) + (e[i].z >= 0) + (e[i].w >= 0);
        const uint32_t j = __umulhi(x, deg);
        const int4 q = (EW == 4 || j < 4) ? e[0] : e[EW / 4 - 1];
        const uint32_t jj = j & 3u;
        return jj < 2 ? (jj == 0 ? q.x : q.y) : (jj == 2 ? q.z : q.w);
    }
};
template <bool OFF64>
struct DrawRow<OFF64, 0> {
    int64_t rb;
    uint32_t deg;
    __device__ __forceinline__ void load(const DevGraph &g, int32_t u) { row_bounds<OFF64>(g, u, rb, deg); }
    template <bool WT>
    __device__ __forceinline__ int32_t pick_csr(const DevGraph &g, uint32_t x, uint32_t y) const {
        const uint32_t j = __umulhi(x, deg);
        if (WT) {
            const WArc arc = g.warc[rb + j];
            return (y < arc.thr) ? arc.col : arc.alias_col;
        }
        return __ldg(g.col + rb + j);
    }
};

// A tree's words by raw vertex number, in shared (SM) or global memory, with
// predicated accesses: no branch, and nothing moves for lanes that sit out.
template <class W, bool SM>
struct Words;
template <>
struct Words<uint32_t, true> {
    uint32_t base;
    __device__ __forceinline__ Words(uint32_t *word, uint32_t off)
        : base((uint32_t)__cvta_generic_to_shared(word) - 4u * off) {}
    __device__ __forceinline__ void ld(uint32_t &w, uint32_t x, bool on) const {
        asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q ld.shared.u32 %0, [%1];}"
                     : "+r"(w) : "r"(base + 4u * x), "r"((int)on) : "memory");
    }
    __device__ __forceinline__ void st(uint32_t x, uint32_t v, bool on) const {
        asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q st.shared.u32 [%0], %1;}"
                     :: "r"(base + 4u * x), "r"(v), "r"((int)on) : "memory");
    }
    // if w is a chain vertex's: x = its successor, w = the successor's word
    __device__ __forceinline__ void hop(uint32_t &w, uint32_t &x, int kb) const {
        asm volatile("{.reg .pred q; .reg .u32 p, a; setp.lt.s32 q, %0, 0; shr.u32 p, %0, %2; "
                     "mad.lo.u32 a, p, 4, %3; @q mov.u32 %1, p; @q ld.shared.u32 %0, [a];}"
                     : "+r"(w), "+r"(x) : "r"(kb), "r"(base) : "memory");
    }
};
template <>
struct Words<uint32_t, false> {
    uint32_t *base;
    __device__ __forceinline__ Words(uint32_t *word, uint32_t off) : base(word - off) {}
    __device__ __forceinline__ void ld(uint32_t &w, uint32_t x, bool on) const {
        asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q ld.global.u32 %0, [%1];}"
                     : "+r"(w) : "l"(base + x), "r"((int)on) : "memory");
    }
    __device__ __forceinline__ void st(uint32_t x, uint32_t v, bool on) const {
        asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q st.global.u32 [%0], %1;}"
                     :: "l"(base + x), "r"(v), "r"((int)on) : "memory");
    }
    __device__ __forceinline__ void hop(uint32_t &w, uint32_t &x, int kb) const {
        asm volatile("{.reg .pred q; .reg .u32 p; .reg .u64 a; setp.lt.s32 q, %0, 0; shr.u32 p, %0, %2; "
                     "mad.wide.u32 a, p, 4, %3; @q mov.u32 %1, p; @q ld.global.u32 %0, [a];}"
                     : "+r"(w), "+r"(x) : "r"(kb), "l"(base) : "memory");
    }
};
template <>
struct Words<uint64_t, false> {
    uint64_t *base;
    __device__ __forceinline__ Words(uint64_t *word, uint32_t off) : base(word - off) {}
    __device__ __forceinline__ void ld(uint64_t &w, uint32_t x, bool on) const {
        asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q ld.global.u64 %0, [%1];}"
                     : "+l"(w) : "l"(base + x), "r"((int)on) : "memory");
    }
    __device__ __forceinline__ void st(uint32_t x, uint64_t v, bool on) const {
        asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q st.global.u64 [%0], %1;}"
                     :: "l"(base + x), "l"(v), "r"((int)on) : "memory");
    }
    __device__ __forceinline__ void hop(uint64_t &w, uint32_t &x, int kb) const {
        const bool go = (int64_t)w < 0;
        x = go ? (uint32_t)(w >> kb) : x;
        ld(w, x, go);
    }
};

enum : int { LM_NEED = 0, LM_REDRAW, LM_CHASE, LM_SETTLE, LM_POP };

// What the threads of one tree share.
template <int NT, int S>
struct LaneShared {
    // pending ends (raw numbers) pushed by each warp, with room for two steps
    uint32_t stack[NT / 32][LT_STACK + 64 * S];
    uint32_t top[NT / 32];                      // heights of the warps' stacks
    uint32_t hit[NT / 32 * S];           // per lane: stopped at a foreign active end
    uint32_t pop[NT / 32 * S];           // per lane: in a pop that began in an earlier round
    uint32_t gsp, taken;                        // ends in global memory, ends asked for this round
    int err;
};

// The word of the root before a tree starts: settled.
template <class W>
__host__ __device__ inline W lt_root_word(int kb, int nl) { return (W)lt_id0(nl) << kb; }

// Runs one tree with the NT threads of the calling group (NT = 32: a warp, else
// the whole block), S lanes per thread.  word: [n] state, zero but for the root's lt_root_word
// (made visible to the group), in shared memory if SM; spill: [n] entries of global memory for the
// stack's overflow.  kb: bits of k; klim: largest pop count allowed.  Returns
// a group-uniform error mask and adds the tree's rounds to `rounds`; on success
// every word holds its vertex's successor and count.
template <bool OFF64, bool WT, int EW, int NT, int S, bool SM, class W>
__device__ __forceinline__ int lane_tree(const DevGraph &g, W *word, int kb, uint32_t klim, LaneShared<NT, S> &sh,
                                         uint32_t *spill, uint32_t tree, uint32_t gid, uint32_t k0,
                                         uint32_t k1, uint32_t &rounds) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr bool WARP = NT == 32;
    constexpr int NW = NT / 32;
    constexpr uint32_t ID0 = lt_id0(NT * S);
    const int lane = threadIdx.x & 31, wid = WARP ? 0 : (int)(threadIdx.x >> 5);
    const unsigned below = (1u << lane) - 1u;
    const uint32_t nstart = (uint32_t)g.n - 1u, root = (uint32_t)g.root;
    const W kmask = ((W)1 << kb) - 1, gobit = (W)1 << (8 * sizeof(W) - 1);
    const uint32_t kcap = kmask < (W)klim ? (uint32_t)kmask : klim;
    const uint32_t OFF = ID0 + (sizeof(W) == 8 ? 0x80000000u : 1u << (31 - kb));   // raw = v + OFF
    const Words<W, SM> wv(word, OFF);
    int mode[S];
    uint32_t e[S], x[S], first[S], ke[S];
    bool carry[S];
#pragma unroll
    for (int s = 0; s < S; ++s) { mode[s] = LM_NEED; e[s] = x[s] = first[s] = OFF; ke[s] = 0; carry[s] = false; }
    if (!WARP) __syncthreads();
    if (threadIdx.x % NT == 0) { sh.gsp = sh.taken = 0; sh.err = 0; }
    if (WARP) __syncwarp(); else __syncthreads();
    // this round's values: the warp's stack height, the ends in all stacks and
    // in the stacks of earlier warps, those in global memory, the next
    // untouched vertex
    uint32_t top = 0, total = 0, before[NW], gsp = 0, scan = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) before[w] = 0;
    uint32_t round = 0;
    bool drew = false;
    int err = 0;
    for (;;) {
        // ---- draw
        if (total == 0 && gsp) {
            // the other warps may still be adding up the heights written below
            // (one that saw the new height would skip this branch and its barrier)
            if (WARP) __syncwarp(); else __syncthreads();
            const uint32_t c = gsp < LT_STACK / 2 ? gsp : LT_STACK / 2;
            for (uint32_t i = threadIdx.x % NT; i < c; i += NT) sh.stack[0][i] = spill[gsp - c + i];
            gsp -= c;
            total = c;
            if (wid == 0) top = c;
            if (threadIdx.x % NT == 0) sh.top[0] = c;
#pragma unroll
            for (int w = 1; w < NW; ++w) before[w] = c;
            if (WARP) __syncwarp(); else __syncthreads();
        }
        bool draw[S];
        uint32_t want, rank[S];
        {
            unsigned m[S];
            uint32_t c = 0;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                m[s] = __ballot_sync(FULL, mode[s] == LM_NEED);
                rank[s] = c + __popc(m[s] & below);
                c += __popc(m[s]);
            }
            want = c;
            if (!WARP && c) {
                uint32_t b = 0;
                if (lane == 0) b = atomicAdd(&sh.taken, c);
                b = __shfl_sync(FULL, b, 0);
#pragma unroll
                for (int s = 0; s < S; ++s) rank[s] += b;
            }
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const bool need = mode[s] == LM_NEED;
            const bool old = need && rank[s] < total;
            const uint32_t i = scan + (rank[s] - total);
            const bool fresh = need && !old && rank[s] - total < nstart - scan;
            if (__any_sync(FULL, old)) {
                uint32_t w = 0, b = 0;
#pragma unroll
                for (int q = 1; q < NW; ++q)
                    if (rank[s] >= before[q]) { w = q; b = before[q]; }
                // the top of a stack goes first
                const uint32_t h = old ? sh.top[w] - 1u - (rank[s] - b) : 0u;
                W ew = 0;
                if (old) e[s] = sh.stack[w][h];
                wv.ld(ew, e[s], old);
                ke[s] = old ? (uint32_t)(ew & kmask) : ke[s];
            }
            e[s] = fresh ? i + (i >= root ? 1u : 0u) + OFF : e[s];
            ke[s] = fresh ? 0u : ke[s];
            draw[s] = mode[s] == LM_REDRAW || old || fresh;
        }
        int32_t px[S];
        {
            DrawRow<OFF64, EW> row[S];
#pragma unroll
            for (int s = 0; s < S; ++s) row[s].load(g, (int32_t)((draw[s] ? e[s] : root + OFF) - OFF));
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const Ctr4 o = philox4x32_10(Ctr4{ke[s], e[s] - OFF, tree, gid}, k0, k1);
                if constexpr (EW > 0) px[s] = row[s].pick(o.x);
                else px[s] = row[s].template pick_csr<WT>(g, o.x, o.y);
            }
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            first[s] = draw[s] ? (uint32_t)px[s] + OFF : first[s];
            x[s] = draw[s] ? first[s] : x[s];
            mode[s] = draw[s] ? LM_CHASE : mode[s];
            carry[s] = carry[s] && !draw[s];
            drew = drew || draw[s];
            wv.st(e[s], ((W)(1 + ((wid * S + s) * 32 + lane)) << kb) | (W)ke[s], draw[s]);
        }
        if (WARP) __syncwarp();
        else {
            __syncthreads();
            want = sh.taken;
        }
        // every lane asked and there was nothing to give: the tree is done
        if (want == NT * S && total == 0 && scan == nstart) break;
        ++rounds;
        {
            const uint32_t fresh = want > total ? want - total : 0u, used = want < total ? want : total;
            scan = nstart - scan < fresh ? nstart : scan + fresh;
            uint32_t mine = 0;
#pragma unroll
            for (int q = 0; q < NW; ++q)
                if (q == wid) mine = before[q];
            const uint32_t gone = used > mine ? used - mine : 0u;
            top = gone < top ? top - gone : 0u;
            if (threadIdx.x % NT == 0) sh.gsp = gsp;
        }
        // ---- chase: reads only
        unsigned hitm[S], popm[S];
        {
            bool run[S];
            W w[S];
#pragma unroll
            for (int s = 0; s < S; ++s) {
                popm[s] = __ballot_sync(FULL, mode[s] == LM_POP);
                run[s] = mode[s] == LM_CHASE;
                w[s] = 0;
                wv.ld(w[s], x[s], run[s]);
            }
            // a chase taken up again that finds an end at once starts over
            {
                bool again[S], any = false;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    again[s] = run[s] && carry[s] && (uint32_t)(w[s] >> kb) < ID0;
                    any = any || again[s];
                }
                if (__any_sync(FULL, any)) {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        x[s] = again[s] ? first[s] : x[s];
                        wv.ld(w[s], x[s], again[s]);
                    }
                }
            }
            int running = 0;
#pragma unroll
            for (int s = 0; s < S; ++s) running += __popc(__ballot_sync(FULL, run[s]));
            // four hops between looks at who still goes; a warp leaves when half
            // of its lanes have stopped, the others go on next round
            for (int h = 0; h < LT_HOPS; h += 4) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
#pragma unroll
                    for (int s = 0; s < S; ++s) wv.hop(w[s], x[s], kb);
                }
                int going = 0;
#pragma unroll
                for (int s = 0; s < S; ++s) going += __popc(__ballot_sync(FULL, (w[s] & gobit) != 0));
                if (going == 0 || 2 * going < running) break;
            }
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const uint32_t p = (uint32_t)(w[s] >> kb);
                carry[s] = (w[s] & gobit) != 0;  // not at its stop yet
                hitm[s] = __ballot_sync(FULL, run[s] && p - 1u < ID0 - 2u && x[s] != e[s]);
            }
            if (!WARP) {
                if (lane == 0) {
#pragma unroll
                    for (int s = 0; s < S; ++s) { sh.hit[wid * S + s] = hitm[s]; sh.pop[wid * S + s] = popm[s]; }
                }
                __syncthreads();
                if (threadIdx.x == 0) sh.taken = 0;
            }
            // ---- act
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const uint32_t p = (uint32_t)(w[s] >> kb);
                const bool stopped = run[s] && !carry[s];
                const bool tree_ = stopped && p >= ID0, own = stopped && !tree_ && x[s] == e[s];
                const bool act = (hitm[s] >> lane) & 1;
                bool park = stopped && p == 0, again = false;
                if (hitm[s]) {
                    const uint32_t j = act ? p - 1u : 0u;
                    const unsigned jb = 1u << (j & 31);
                    const unsigned hj = WARP ? (j < 32 ? hitm[0] : hitm[S - 1]) : sh.hit[j >> 5];
                    const unsigned pj = WARP ? (j < 32 ? popm[0] : popm[S - 1]) : sh.pop[j >> 5];
                    again = act && (pj & jb);
                    park = park || (act && !again && (!(hj & jb) || (uint32_t)((wid * S + s) * 32 + lane) > j));
                    carry[s] = carry[s] || (act && !again && !park);
                }
                const W chain = ((W)first[s] << kb) | (W)ke[s];
                wv.st(e[s], tree_ ? chain & ~gobit : chain, tree_ || park);
                x[s] = tree_ || own || again ? first[s] : x[s];
                mode[s] = tree_ ? LM_SETTLE : own ? LM_POP : park ? LM_NEED : mode[s];
            }
        }
        // marking and popping, one vertex a step up to the chain's stop (the
        // tree, or the popped cycle's end); long ones go on next round
        {
            W w[S], keep[S];
            bool on[S], any = false;
            uint32_t kseen = 0;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                on[s] = mode[s] >= LM_SETTLE;
                keep[s] = mode[s] == LM_POP ? kmask : ~gobit;
                any = any || on[s];
                w[s] = 0;
                wv.ld(w[s], x[s], on[s]);
            }
            for (int h = 0; h < LT_ACT && __any_sync(FULL, any); h += 2) {
                uint32_t y[2 * S];
                bool push[2 * S];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        const int i = q * S + s;
                        const bool step = (w[s] & gobit) != 0;
                        push[i] = step && mode[s] == LM_POP;
                        y[i] = x[s];
                        const W v = (w[s] & keep[s]) + (push[i] ? 1 : 0);
                        kseen = push[i] && v > (W)kseen ? (uint32_t)(sizeof(W) == 8 && v > (W)0xffffffffu ? (W)0xffffffffu : v) : kseen;
                        wv.hop(w[s], x[s], kb);
                        wv.st(y[i], v, step);
                    }
                }
#pragma unroll
                for (int i = 0; i < 2 * S; ++i) {
                    const unsigned m = __ballot_sync(FULL, push[i]);
                    if (push[i]) sh.stack[wid][top + __popc(m & below)] = y[i];
                    top += __popc(m);
                }
                if (top > LT_STACK) {            // the overflow goes to global memory
                    __syncwarp();
                    uint32_t b = 0;
                    if (lane == 0) b = atomicAdd(&sh.gsp, top - LT_STACK);
                    b = __shfl_sync(FULL, b, 0);
                    for (uint32_t i = LT_STACK + lane; i < top; i += 32) spill[b + i - LT_STACK] = sh.stack[wid][i];
                    top = LT_STACK;
                    __syncwarp();
                }
                any = false;
#pragma unroll
                for (int s = 0; s < S; ++s) any = any || (w[s] & gobit);
            }
            if (kseen > kcap) err |= kseen > klim ? LE_KOVF : LE_KREP;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                if (on[s] && !(w[s] & gobit)) {
                    if (mode[s] == LM_POP) {
                        if (x[s] != e[s]) err |= LE_LOOP;
                        if (++ke[s] > kcap) err |= ke[s] > klim ? LE_KOVF : LE_KREP;
                        mode[s] = LM_REDRAW;
                    } else {
                        if ((uint32_t)(w[s] >> kb) < ID0) err |= LE_LOOP;
                        mode[s] = LM_NEED;
                    }
                }
            }
        }
        if (lane == 0) sh.top[wid] = top;
        if (err) sh.err = err;
        if (WARP) __syncwarp(); else __syncthreads();
        if (sh.err) break;
        // rounds without a draw are bounded: the longest chain is walked,
        // marked or popped in far fewer
        if (++round == nstart / 8 + 8192u) {
            if (!(WARP ? __any_sync(FULL, drew) : __syncthreads_or(drew))) { err = LE_LOOP; break; }
            round = 0;
            drew = false;
        }
        total = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) { before[w] = total; total += sh.top[w]; }
        gsp = sh.gsp;
    }
    // any error of the group, in every thread
    int mask = 0;
#pragma unroll
    for (int bit = LE_KOVF; bit <= LE_LOOP; bit <<= 1)
        if (WARP ? __any_sync(FULL, err & bit) : __syncthreads_or(err & bit)) mask |= bit;
    return mask;
}

}  // namespace rwc
