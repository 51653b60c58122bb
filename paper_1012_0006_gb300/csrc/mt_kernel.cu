// Multi-try FM after the pairwise improvements of a matching (Sanders & Schulz,
// Section 4.2, run from active block scheduling as Section 4.3 describes): every
// boundary vertex of a pair goes on the pair's todo list, the list is taken in a
// random order, and each vertex that no earlier search of the pass touched and that
// still lies on the boundary starts a k-way local search from itself and its boundary
// neighbours; no search touches a vertex an earlier search of the pass touched.
//
// The k-way search is the one of Section 2.2: a single queue keyed by the max gain
// g(v) = max_P omega(v, P) - omega(v, own block) over the blocks P next to v; the
// best vertex moves to its best block unless that block would exceed L_max; each
// vertex moves at most once; the search stops when the queue is empty or by the
// KaSPar rule (over the p moves since the last new minimum, with mean mu and variance
// sigma^2 of their gains: p mu^2 > alpha sigma^2 + beta, beta = ln n) and rolls back
// to the first lowest cut.  Readings, as in the CPU oracle: keys order by gain, then
// by the time of the vertex's last keying (later first): the start set in its order,
// then after each move the moved vertex's neighbours in CSR order; target ties go to
// the smaller splitmix64(tseed ^ u << 32 ^ P); a vertex that may not move leaves the
// queue; after a move every unmoved neighbour the search may touch is keyed again if
// it is a boundary vertex and leaves the queue if not; the pairs' todo lists are
// visited round-robin (entry j of every pair in pair order, then entry j + 1).
//
// GPU form.  The searches of a pass are sequential by definition: each sees the
// partition and the touched marks the earlier ones left.  So one warp runs the whole
// pass, and what bounds it is the chain of dependent loads per move.  Every vertex has a
// 64-byte record (built by the grid before the searches) that holds its row range, block,
// marks and its connection weight to each block around it; a move of x from block P to
// block Q changes the weights of x's neighbours by omega(x, u) at P and Q, so their gains
// follow from their records alone: a move is the popped entry, x's arcs, the neighbours'
// records.  Summing every neighbour's arcs again instead, as first built, read two more
// dependent levels (arcs, their blocks) for every neighbour: the global rounds of a 3D
// rgg of 524,288 vertices and 64 blocks (29,191 moves) took 90 ms so and take 48.7 ms now,
// about 3,300 cycles a move, half of it loads that miss L1 (300 cycles near in L2, some 700
// when first touched) and half the warp's own instructions.  The queue is an array of gain buckets, each a stack of 16-byte entries in global memory with
// its top and a non-empty bitmap in shared memory; an entry carries what the move needs
// (vertex, target, block, adjacency range) and is live while that word is not zero: keying
// pushes a new entry (so each stack stays ordered by keying time) and zeroes the word in the
// vertex's previous entry of the same search; pops skip dead entries.  The last kMtRing
// entries are also in shared memory, where most pops find theirs.  The block weights live
// in shared memory for the pass.  Grid-wide kernels before it build the records, sum the
// block weights, fill the todo lists and sort each (one CTA per pair, bitonic by key).
//
// The same search, without the touched rule and started from the whole boundary (or
// its corner vertices), makes one round of the global k-way refinement (end of file).
#include <climits>

#include "mt_kernel.cuh"

namespace fr {

constexpr int kMtTPB = 256;
constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------- records ----
// Record of vertex v: four int4 at m.rec + 4 v.
//   [0] {row begin, row end, block, 1 if more than eight blocks lie around v}
//   [1] {latest entry, search that queued v (0: none), search that moved v, -}
//   [2], [3] eight slots block << 16 | connection weight, 0 empty (weights are at most
//   the weighted degree, <= kMtGmax; k <= kMtMaxK).  With more than eight blocks the
//   slots mean nothing and the gain is summed over the row (mt_gain_row).
struct MtSlots {
    int s[8];
};

__device__ __forceinline__ MtSlots mt_slots(const int4 &c, const int4 &d) {
    return {{c.x, c.y, c.z, c.w, d.x, d.y, d.z, d.w}};
}

// Slot s holds block P: s - (P << 16) is its weight.
__device__ __forceinline__ bool mt_is(int s, int P) { return (unsigned)(s - (P << 16) - 1) < 0xffffu; }

// Adds w to block P's slot (or the first empty one) among the first N; false if there is
// no room.
template <int N>
__device__ __forceinline__ bool mt_slot_add(MtSlots &q, int P, int w) {
    unsigned at = 0, hole = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        at |= mt_is(q.s[i], P) ? 1u << i : 0u;
        hole |= q.s[i] == 0 ? 1u << i : 0u;
    }
    const int add = at ? w : (P << 16) | w;
    at = at ? at : hole & (0u - hole);
#pragma unroll
    for (int i = 0; i < N; ++i) q.s[i] += (at >> i) & 1u ? add : 0;
    return at != 0;
}

// Takes w from block P's slot; a slot that comes to nothing is empty again.
template <int N>
__device__ __forceinline__ void mt_slot_sub(MtSlots &q, int P, int w) {
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (mt_is(q.s[i], P)) q.s[i] = q.s[i] - (P << 16) > w ? q.s[i] - w : 0;
}

// Max gain of u (block pu) and its target over the first N slots: the adjacent block
// other than pu with the largest connection weight, ties to the smaller
// splitmix64(tseed ^ u << 32 ^ P), then the smaller P.  False if u has no neighbour
// outside its block.
template <int N>
__device__ __forceinline__ bool mt_gain(const MtSlots &q, int u, int pu, unsigned long long tseed, int &gain,
                                        int &to) {
    int own = 0, bw = 0, w[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const bool mine = mt_is(q.s[i], pu);
        w[i] = mine ? 0 : q.s[i] & 0xffff;
        own = mine ? q.s[i] & 0xffff : own;
        bw = max(bw, w[i]);
    }
    if (bw == 0) return false;
    unsigned ties = 0;
    int best = -1;
#pragma unroll
    for (int i = N - 1; i >= 0; --i)
        if (w[i] == bw) {
            ties |= 1u << i;
            best = q.s[i] >> 16;
        }
    if (ties & (ties - 1)) {   // a target's hash only when its weight ties the best
        const unsigned long long hu = tseed ^ ((unsigned long long)(unsigned)u << 32);
        unsigned long long bh = ~0ull;
        best = INT_MAX;
#pragma unroll
        for (int i = 0; i < N; ++i)
            if ((ties >> i) & 1u) {
                const int P = q.s[i] >> 16;
                const unsigned long long h = splitmix64(hu ^ (unsigned)P);
                if (h < bh || (h == bh && P < best)) {
                    bh = h;
                    best = P;
                }
            }
    }
    gain = bw - own;
    to = best;
    return true;
}

// True (for the whole warp) if every lane's blocks lie in its first four slots with room
// for one more: the common case, at half the work.
__device__ __forceinline__ bool mt_narrow(const MtSlots &q) {
    return __all_sync(kFull, (q.s[4] | q.s[5] | q.s[6] | q.s[7]) == 0 &&
                                 (q.s[0] == 0 || q.s[1] == 0 || q.s[2] == 0 || q.s[3] == 0));
}

// The same for a vertex with more than eight blocks around it, by one whole warp: its
// row's weights summed per block in hist ([k] words of shared memory, zero before and
// after), then the best block over the row.  All lanes return the same values.
__device__ bool mt_gain_row(const GraphDev &G, int *hist, int u, int pu, int j0, int j1, unsigned long long tseed,
                            int &gain, int &to) {
    const int lane = threadIdx.x & 31;
    for (int j = j0 + lane; j < j1; j += 32) atomicAdd(hist + G.part[__ldg(G.adjncy + j)], __ldg(G.adjwgt + j));
    __syncwarp();
    const unsigned long long hu = tseed ^ ((unsigned long long)(unsigned)u << 32);
    const int own = hist[pu];
    int bw = 0, best = INT_MAX;
    unsigned long long bh = ~0ull;
    for (int j = j0 + lane; j < j1; j += 32) {
        const int P = G.part[__ldg(G.adjncy + j)];
        if (P == pu) continue;
        const int w = hist[P];
        if (w < bw) continue;
        const unsigned long long h = splitmix64(hu ^ (unsigned)P);
        if (w > bw || h < bh || (h == bh && P < best)) {
            bw = w;
            bh = h;
            best = P;
        }
    }
    __syncwarp();
    for (int j = j0 + lane; j < j1; j += 32) hist[G.part[__ldg(G.adjncy + j)]] = 0;
    for (int d = 16; d > 0; d >>= 1) {
        const int w2 = __shfl_xor_sync(kFull, bw, d), b2 = __shfl_xor_sync(kFull, best, d);
        const unsigned long long h2 = __shfl_xor_sync(kFull, bh, d);
        if (w2 > bw || (w2 == bw && (h2 < bh || (h2 == bh && b2 < best)))) {
            bw = w2;
            bh = h2;
            best = b2;
        }
    }
    __syncwarp();
    gain = bw - own;
    to = best;
    return bw > 0;
}

// Gains of the lanes' vertices (ask: the lane has one; over: it needs its row summed).
// The whole warp calls it; returns whether the lane's vertex has a block to move to.
__device__ __forceinline__ bool mt_gain_lanes(const GraphDev &G, int *hist, bool ask, bool over, const MtSlots &q,
                                              int u, int pu, int j0, int j1, unsigned long long tseed, int &gain,
                                              int &to) {
    bool has = false;
    if (__all_sync(kFull, (q.s[4] | q.s[5] | q.s[6] | q.s[7]) == 0)) {
        if (ask && !over) has = mt_gain<4>(q, u, pu, tseed, gain, to);
    } else {
        if (ask && !over) has = mt_gain<8>(q, u, pu, tseed, gain, to);
    }
    for (unsigned ov = __ballot_sync(kFull, ask && over); ov; ov &= ov - 1) {
        const int l = __ffs(ov) - 1;
        int g, t;
        const bool h = mt_gain_row(G, hist, __shfl_sync(kFull, u, l), __shfl_sync(kFull, pu, l),
                                   __shfl_sync(kFull, j0, l), __shfl_sync(kFull, j1, l), tseed, g, t);
        if ((threadIdx.x & 31) == l) {
            has = h;
            gain = g;
            to = t;
        }
    }
    return has;
}

// Builds v's record from the partition; its slots and block are left in q and pv.
__device__ __forceinline__ bool mt_build(const GraphDev &G, const MtDev &m, int v, MtSlots &q, int &pv) {
    const int j0 = __ldg(G.xadj + v), j1 = __ldg(G.xadj + v + 1);
    pv = G.part[v];
    q = {};
    bool over = false;
    for (int j = j0; j < j1; j += 4) {   // four arcs at a time, their loads issued together
        int w[4], P[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int x = min(j + t, j1 - 1);
            P[t] = __ldg(G.adjncy + x);
            w[t] = __ldg(G.adjwgt + x);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) P[t] = G.part[P[t]];
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (j + t < j1 && !mt_slot_add<8>(q, P[t], w[t])) over = true;
    }
    int4 *r = m.rec + 4LL * v;
    r[0] = make_int4(j0, j1, pv, over ? 1 : 0);
    r[1] = make_int4(-1, 0, 0, 0);
    r[2] = make_int4(q.s[0], q.s[1], q.s[2], q.s[3]);
    r[3] = make_int4(q.s[4], q.s[5], q.s[6], q.s[7]);
    return over;
}

// Distinct blocks other than pv around v.
__device__ __forceinline__ int mt_foreign(const MtSlots &q, int pv) {
    int c = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) c += q.s[i] != 0 && (q.s[i] >> 16) != pv;
    return c;
}

// Pair of the pass that v's block x belongs to (and the partner block), if v has a
// neighbour in the partner block; else -1.
__device__ __forceinline__ int mt_pair_of(const GraphDev &G, const MtDev &m, int v, int x, bool over,
                                          const MtSlots &q) {
    const int p = m.bpair[x];
    if (p < 0) return -1;
    const int other = m.pa[p] == x ? m.pb[p] : m.pa[p];
    bool next = false;
    if (!over) {
#pragma unroll
        for (int i = 0; i < 8; ++i) next |= q.s[i] != 0 && (q.s[i] >> 16) == other;
    } else {
        const int j1 = __ldg(G.xadj + v + 1);
        for (int j = __ldg(G.xadj + v); j < j1 && !next; ++j) next = G.part[__ldg(G.adjncy + j)] == other;
    }
    return next ? p : -1;
}

__device__ __forceinline__ unsigned long long mt_list_seed(unsigned long long seed, int a, int b) {
    return splitmix64(splitmix64(seed ^ ((unsigned long long)(unsigned)a << 32) ^ (unsigned)b) + 1);
}

// Records, block weights and the todo list length of every pair.
__global__ void __launch_bounds__(kMtTPB) mt_count_kernel(GraphDev G, MtDev m) {
    extern __shared__ long long s_bw[];   // [k]
    for (int i = threadIdx.x; i < G.k; i += blockDim.x) s_bw[i] = 0;
    __syncthreads();
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < G.n; v += gridDim.x * blockDim.x) {
        const int c = __ldg(G.vwgt + v);
        if (c) atomicAdd(reinterpret_cast<unsigned long long *>(s_bw + G.part[v]), (unsigned long long)c);
        MtSlots q;
        int pv;
        const bool over = mt_build(G, m, v, q, pv);
        const int p = mt_pair_of(G, m, v, pv, over, q);
        if (p >= 0) atomicAdd(m.cnt + p, 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G.k; i += blockDim.x)
        if (s_bw[i]) atomicAdd(reinterpret_cast<unsigned long long *>(m.bw + i), (unsigned long long)s_bw[i]);
}

// Todo list offsets, each list padded to a power of two for its sort.
__global__ void mt_offsets_kernel(MtDev m, Ctl *ctl) {
    if (threadIdx.x != 0) return;
    long long o = 0;
    for (int p = 0; p < m.np; ++p) {
        m.off[p] = o;
        long long q = 1;
        while (q < m.cnt[p]) q <<= 1;
        o += q;
        m.fil[p] = 0;
    }
    m.off[m.np] = o;
    if (o > m.scap) fail(ctl, E_INTERNAL, 801);
}

__global__ void __launch_bounds__(kMtTPB) mt_fill_kernel(GraphDev G, MtDev m, Ctl *ctl) {
    if (__ldcg(&ctl->error)) return;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < G.n; v += gridDim.x * blockDim.x) {
        const int4 *r = m.rec + 4LL * v;
        const int4 a = r[0];
        const int p = mt_pair_of(G, m, v, a.z, a.w != 0, mt_slots(r[2], r[3]));
        if (p < 0) continue;
        const int pos = atomicAdd(m.fil + p, 1);
        if (pos >= m.cnt[p]) {   // cannot happen: the count pass saw the same partition
            fail(ctl, E_INTERNAL, 802);
            return;
        }
        const long long i = m.off[p] + pos;
        m.tv[i] = v;
        m.tkey[i] = splitmix64(mt_list_seed(m.seed, m.pa[p], m.pb[p]) ^ (unsigned long long)(unsigned)v);
    }
}

// One CTA per pair: its todo list ascending by (key, vertex), bitonic in global memory.
__global__ void __launch_bounds__(kMtTPB) mt_sort_kernel(MtDev m, Ctl *ctl) {
    if (__ldcg(&ctl->error)) return;
    const int p = blockIdx.x;
    const long long o = m.off[p], len = m.off[p + 1] - o;
    const int c = m.cnt[p];
    unsigned long long *K = m.tkey + o;
    int *V = m.tv + o;
    for (long long i = c + threadIdx.x; i < len; i += blockDim.x) {
        K[i] = ~0ull;
        V[i] = INT_MAX;
    }
    __syncthreads();
    for (long long kk = 2; kk <= len; kk <<= 1)
        for (long long j = kk >> 1; j > 0; j >>= 1) {
            for (long long i = threadIdx.x; i < len; i += blockDim.x) {
                const long long l = i ^ j;
                if (l <= i) continue;
                const unsigned long long ki = K[i], kl = K[l];
                const int vi = V[i], vl = V[l];
                const bool l_less = kl < ki || (kl == ki && vl < vi);
                const bool i_less = ki < kl || (ki == kl && vi < vl);
                if ((i & kk) == 0 ? l_less : i_less) {
                    K[i] = kl; K[l] = ki;
                    V[i] = vl; V[l] = vi;
                }
            }
            __syncthreads();
        }
}

// ---------------------------------------------------------------- the pass ----

// KaSPar rule p mu^2 > alpha sigma^2 + beta (mu, sigma^2: mean and variance of the p
// gains since the last new minimum; S1, S2: their sum and sum of squares), decided as the
// oracle's rounded double operations in its order decide it.  Times p^2 the rule reads
// D = p S1^2 - alpha (p S2 - S1^2) - beta p^2 > 0.  D is first estimated in single
// precision; with M the sum of the four terms' magnitudes, that estimate is within about
// 1.1e-6 M of the exact D (18 roundings of 2^-24), and the double expression within
// about 1e-15 M, so whenever the estimate exceeds 1e-5 M in magnitude all three have the
// same sign.  Only the rest take the double path (FP64 is slow on this part).
__device__ __forceinline__ bool kaspar_stop(int p, long long S1, long long S2, int alpha, double beta) {
    {
        const float pf = (float)p, s1 = (float)S1, s2 = (float)S2, af = (float)alpha, bf = (float)beta;
        const float s11 = s1 * s1;
        const float t1 = pf * s11, t2 = af * (pf * s2), t3 = af * s11, t4 = bf * (pf * pf);
        const float D = ((t1 - t2) + t3) - t4;
        const float M = ((t1 + t2) + t3) + t4;
        if (fabsf(D) > 1e-5f * M) return D > 0.f;
    }
    const double pd = (double)p;
    const double mu = __ddiv_rn((double)S1, pd);
    const double var = __dsub_rn(__ddiv_rn((double)S2, pd), __dmul_rn(mu, mu));
    const double lhs = __dmul_rn(__dmul_rn(pd, mu), mu);
    const double rhs = __dadd_rn(__dmul_rn((double)alpha, var), beta);
    return lhs > rhs;
}

__device__ __forceinline__ unsigned mt_lanemask_lt() {
    unsigned r;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(r));
    return r;
}

struct MtShared {
    int top[kMtBuckets];               // top entry of each gain bucket with its bit set
    unsigned bits[kMtBuckets / 32];    // non-empty buckets (possibly holding only dead entries)
    long long bw[kMtMaxK];             // block weights during the pass
    int hist[kMtMaxK];                 // mt_gain_row's sums, zero between uses
    int4 ring[kMtRing];                // the last kMtRing entries pushed (entry e at e % kMtRing)
    long long prog;                    // what the searching warp is at: todo position or start entry
    int4 last[kMtLast];                // its last moves: {vertex, source << 10 | target, row}
    int done;                          // 1: it has finished
    unsigned sink;                     // (the prefetching warps' loads end here)
};

// The searching warp has its SM to itself, and each of a move's loads that misses L1 costs
// it several hundred cycles.  So kMtAhead more warps of its CTA read what it will need next
// into L1: they follow S.prog, a few todo entries (or start entries) ahead.  They write
// nothing, and what they miss costs time only.  Without them those rounds take 58 ms; four
// warps or a longer lead gain nothing, nor do warps that read around the moved vertex.
constexpr int kMtAhead = 2;            // warps that run ahead
constexpr int kMtWarps = 1 + kMtAhead;
constexpr int kMtSeedsAhead = 8;       // todo entries they run ahead of a pass
constexpr int kKwEntsAhead = 16;       // start entries they run ahead of a global round
constexpr int kMtIdle = 1 << 22;       // polls without work before such a warp gives up

// Reads the records of a row's neighbours (two sectors each).
__device__ __forceinline__ unsigned mt_warm_row(const GraphDev &G, const MtDev &m, int y0, int y1) {
    const int lane = threadIdx.x & 31;
    unsigned acc = 0;
    for (int j = y0 + lane; j < y1; j += 32) {
        const int u = __ldg(G.adjncy + j);
        acc ^= (unsigned)__ldg(G.adjwgt + j) ^ (unsigned)m.rec[4LL * u].x ^ (unsigned)m.rec[4LL * u + 2].x;
    }
    return acc;
}

// Waits (a limited number of polls) until item i is at most `ahead` items in front of the
// searching warp; items it has passed are skipped.  False: finished, or idle too long.
__device__ __forceinline__ bool mt_follow(MtShared &S, long long &i, int ahead) {
    for (int polls = 0; polls < kMtIdle; ++polls) {
        if (*(volatile int *)&S.done) return false;
        const long long prog = *(volatile long long *)&S.prog;
        if (i <= prog) i += (prog - i) / kMtAhead * kMtAhead + kMtAhead;
        if (i <= prog + ahead) return true;
        __nanosleep(200);
    }
    return false;
}

// A queue entry: {vertex, entry below it in its bucket, word, row begin}, the word 0 once
// the entry is dead, else live bit | degree << 20 | block << 10 | target (a degree is at
// most the weighted degree, <= kMtGmax).
__device__ __forceinline__ int mt_word(int deg, int block, int to) {
    return (int)(0x80000000u | ((unsigned)(deg & 1023) << 20) | ((unsigned)block << 10) | (unsigned)to);
}
__device__ __forceinline__ int mt_word_deg(int word) { return (word >> 20) & 1023; }

// Entry e of the current search, nxt of them pushed, those from rbase on by its warp.
__device__ __forceinline__ bool mt_in_ring(int e, int nxt, int rbase) { return e >= rbase && e >= nxt - kMtRing; }
__device__ __forceinline__ int4 mt_entry(const MtShared &S, const MtDev &m, int e, int nxt, int rbase) {
    return mt_in_ring(e, nxt, rbase) ? S.ring[e & (kMtRing - 1)] : m.ent[e];
}
__device__ __forceinline__ void mt_kill(MtShared &S, const MtDev &m, bool kill, int e, int nxt, int rbase) {
    if (kill) m.ent[e].z = 0;
    if (kill && mt_in_ring(e, nxt, rbase)) S.ring[e & (kMtRing - 1)].z = 0;
}

// Pushes the lanes' entries (in lane order) onto their buckets: entries go to
// [nxt, nxt + popc(pm)); a lower lane's entry lies below a higher lane's in one bucket.
// Returns the lane's entry.
__device__ __forceinline__ int mt_push(MtShared &S, const MtDev &m, unsigned pm, bool push, int bk, int u, int word,
                                       int u0, int nxt, int lane) {
    const int pos = nxt + __popc(pm & mt_lanemask_lt());
    const unsigned grp = __match_any_sync(kFull, push ? bk : -1);   // (its time grows with the distinct values)
    const unsigned lower = grp & mt_lanemask_lt();
    const int pos_lower = __shfl_sync(kFull, pos, lower ? 31 - __clz(lower) : lane);
    const unsigned word_b = S.bits[bk >> 5];
    const int top_b = S.top[bk];
    const int below = lower ? pos_lower : (word_b >> (bk & 31)) & 1u ? top_b : -1;
    __syncwarp();
    if (push) {
        const int4 e = make_int4(u, below, word, u0);
        m.ent[pos] = e;
        S.ring[pos & (kMtRing - 1)] = e;
        if ((grp & ~lower & ~(1u << lane)) == 0) {   // highest lane of its bucket
            S.top[bk] = pos;
            atomicOr(&S.bits[bk >> 5], 1u << (bk & 31));
        }
    }
    __syncwarp();
    return pos;
}

// The neighbours of a vertex that moves from block `from` to block `to` (omega w each):
// their slots, in the lane's copy of the record.  over: no room was left for `to`.
template <int N>
__device__ __forceinline__ void mt_shift(MtSlots &q, int from, int to, int w, bool &over) {
    mt_slot_sub<N>(q, from, w);
    if (!mt_slot_add<N>(q, to, w)) over = true;
}

// One k-way search (one warp) from the entries already pushed, nxt of them (those before
// rbase by the grid): pop the highest live entry, move its vertex unless the target would
// exceed L_max, key its unmoved neighbours again (CSR order), stop by the KaSPar rule or
// an empty queue.  sid: the search's number in its pass, in the records' marks.  touch:
// the multi-try pass's rule (a vertex another search of the pass queued is neither queued
// nor moved); false: no such rule (the global k-way rounds).  Returns the best prefix
// (best < 0 is the largest cut decrease), the moves made and kept, and whether the KaSPar
// rule stopped it; bad on an error.
__device__ __forceinline__ void mt_search(const GraphDev &G, const MtDev &m, MtShared &S, Ctl *ctl, int sid,
                                          bool touch, int nxt, int rbase, long long Lmax, unsigned long long tseed,
                                          int lane, bool &bad, long long &best, int &nm, int &best_len,
                                          bool &stopped) {
    long long delta = 0, S1 = 0, S2 = 0;
    int pc = 0;
    best = 0;
    nm = 0;
    best_len = 0;
    stopped = false;
    bool off = false;
    while (!bad) {
        // pop the highest live entry (every lane reads it)
        int4 e = make_int4(-1, 0, 0, 0);
        int b;
        for (;;) {
            const uint2 w2 = reinterpret_cast<const uint2 *>(S.bits)[lane];
            const unsigned has = __ballot_sync(kFull, (w2.x | w2.y) != 0);
            if (!has) {
                e.x = -1;
                break;
            }
            const int own = 31 - __clz(has);   // the lane whose words hold the highest bit
            b = __shfl_sync(kFull, w2.y ? lane * 64 + 63 - __clz(w2.y) : lane * 64 + 31 - __clz(w2.x), own);
            int at = S.top[b];
            e = mt_entry(S, m, at, nxt, rbase);
            while (!e.z && e.y >= 0) {   // dead ones on one another: no new look at the bits
                // (three global rounds of rgg3d 524,288, k = 64: 51.4 -> 49.1 ms)
                at = e.y;
                e = mt_entry(S, m, at, nxt, rbase);
            }
            __syncwarp();
            if (lane == own) {
                S.top[b] = e.y;
                if (e.y < 0) S.bits[b >> 5] = ((b >> 5) & 1 ? w2.y : w2.x) & ~(1u << (b & 31));
                if (at < rbase) *(volatile long long *)&S.prog = at;
            }
            __syncwarp();
            if (e.z) break;   // live: the vertex leaves the queue
        }
        const int x = e.x;
        if (x < 0) break;   // the queue is empty
        const int g = b - kMtGmax;
        const int to = e.z & 1023, from = (e.z >> 10) & 1023;
        // the weight and the first 32 arcs, then those neighbours' records, are on their
        // way while the move is booked
        const int y0 = e.w, y1 = y0 + mt_word_deg(e.z);
        const int cw = __ldg(G.vwgt + x);
        int u = -1, wu = 0;
        if (y0 + lane < y1) {
            u = __ldg(G.adjncy + y0 + lane);
            wu = __ldg(G.adjwgt + y0 + lane);
        }
        int4 *r = m.rec + 4LL * (u < 0 ? 0 : u);
        int4 A = make_int4(0, 0, 0, 0), B = A, C = A, D = A;
        if (u >= 0) {
            A = r[0];
            B = r[1];
            C = r[2];
            D = r[3];
        }
        const long long cx = cw, bw_from = S.bw[from], bw_to = S.bw[to];
        if (bw_to + cx > Lmax) continue;   // would overload the target: not moved
        __syncwarp();
        if (lane == 0) {
            G.part[x] = to;
            m.rec[4LL * x].z = to;
            m.rec[4LL * x + 1].z = sid;
            S.bw[from] = bw_from - cx;
            S.bw[to] = bw_to + cx;
            const int4 mv = make_int4(x, (from << 10) | to, y0, y1);
            S.last[nm & (kMtLast - 1)] = mv;
            m.lmv[nm] = make_int2(mv.x, mv.y);
        }
        ++nm;
        delta -= g;
        __syncwarp();
        // key the neighbours again, 32 at a time in CSR order
        for (int jb = y0; jb < y1; jb += 32) {
            if (jb > y0) {
                u = -1;
                A = B = C = D = make_int4(0, 0, 0, 0);
                if (jb + lane < y1) {
                    u = __ldg(G.adjncy + jb + lane);
                    wu = __ldg(G.adjwgt + jb + lane);
                    r = m.rec + 4LL * u;
                    A = r[0];
                    B = r[1];
                    C = r[2];
                    D = r[3];
                }
            }
            MtSlots q = mt_slots(C, D);
            bool over = A.w != 0;
            const bool elig = u >= 0 && B.z != sid && (!touch || B.y == 0 || B.y == sid);
            const bool fits = u >= 0 && !over;   // (its slots are kept)
            if (mt_narrow(q)) {
                if (fits) {
                    mt_shift<4>(q, from, to, wu, over);
                    r[2] = make_int4(q.s[0], q.s[1], q.s[2], q.s[3]);
                }
            } else if (fits) {
                mt_shift<8>(q, from, to, wu, over);
                r[2] = make_int4(q.s[0], q.s[1], q.s[2], q.s[3]);
                r[3] = make_int4(q.s[4], q.s[5], q.s[6], q.s[7]);
                if (over) r[0].w = 1;
            }
            int gu = 0, tu = -1;
            const bool push = mt_gain_lanes(G, S.hist, elig, over, q, u, A.z, A.x, A.y, tseed, gu, tu);
            // (a gain or target out of range: only if the rows' weights are not symmetric;
            // kept in bounds here, and the search fails when it ends)
            off |= push && ((unsigned)(gu + kMtGmax) > 2u * kMtGmax || tu >= G.k);
            const unsigned pm = __ballot_sync(kFull, push);
            if ((long long)nxt + __popc(pm) > m.ecap) {
                if (lane == 0) fail(ctl, E_TOO_LARGE, 805);
                bad = true;
                break;
            }
            mt_kill(S, m, elig && B.y == sid && B.x >= 0, B.x, nxt, rbase);   // its old entry is dead from here on
            const int bk = min(max(gu + kMtGmax, 0), 2 * kMtGmax);
            const int pos = mt_push(S, m, pm, push, bk, u, mt_word(A.y - A.x, A.z, tu), A.x, nxt, lane);
            if (push) r[1] = make_int4(pos, sid, B.z, 0);
            nxt += __popc(pm);
        }
        if (bad) break;
        if (delta < best) {
            best = delta; best_len = nm; pc = 0; S1 = 0; S2 = 0;
        } else {
            ++pc;
            S1 += g;
            S2 += (long long)g * g;
            if (kaspar_stop(pc, S1, S2, m.alpha, m.beta)) {
                stopped = true;
                break;
            }
        }
    }
    if (__any_sync(kFull, off)) {
        if (lane == 0) fail(ctl, E_INTERNAL, 807);
        bad = true;
    }
    __syncwarp();
}

// After a search: roll back to the first lowest cut, last move first (so a record never
// needs more slots than it held at that point of the search).  With bookkeeping (the
// multi-try pass), mark the blocks the kept moves left and entered and list the kept
// movers (kbase: the pass's count so far) for the boundary list, which mt_bl_kernel
// fills after the pass.
__device__ __forceinline__ void mt_finish(const GraphDev &G, const MtDev &m, MtShared &S, int nm, int best_len,
                                          int lane, bool keep, int &kbase) {
    for (int i = nm - 1; i >= best_len; --i) {
        int4 mv;
        if (i >= nm - kMtLast) {
            mv = S.last[i & (kMtLast - 1)];
        } else {
            const int2 h = m.lmv[i];
            mv = make_int4(h.x, h.y, __ldg(G.xadj + h.x), __ldg(G.xadj + h.x + 1));
        }
        const int x = mv.x, to = mv.y & 1023, from = mv.y >> 10;
        const long long cx = __ldg(G.vwgt + x);
        if (lane == 0) {
            G.part[x] = from;
            m.rec[4LL * x].z = from;
            S.bw[to] -= cx;
            S.bw[from] += cx;
        }
        for (int jb = mv.z; jb < mv.w; jb += 32) {
            const int j = jb + lane;
            MtSlots q = {};
            bool over = true;
            int wu = 0;
            int4 *r = m.rec;
            if (j < mv.w) {
                r = m.rec + 4LL * __ldg(G.adjncy + j);
                wu = __ldg(G.adjwgt + j);
                over = r[0].w != 0;
                q = mt_slots(r[2], r[3]);
            }
            const bool fits = !over;
            if (mt_narrow(q)) {
                if (fits) {
                    mt_shift<4>(q, to, from, wu, over);
                    r[2] = make_int4(q.s[0], q.s[1], q.s[2], q.s[3]);
                }
            } else if (fits) {
                mt_shift<8>(q, to, from, wu, over);
                r[2] = make_int4(q.s[0], q.s[1], q.s[2], q.s[3]);
                r[3] = make_int4(q.s[4], q.s[5], q.s[6], q.s[7]);
                if (over) r[0].w = 1;
            }
        }
        __syncwarp();
    }
    if (keep) {
        for (int i = lane; i < best_len; i += 32) {
            const int2 mv = m.lmv[i];
            m.chg[mv.y & 1023] = 1;
            m.chg[mv.y >> 10] = 1;
            m.kept[kbase + i] = mv.x;
        }
        kbase += best_len;
    }
    __syncwarp();
}

// The whole pass: one searching warp, and the warps that prefetch for it.
__global__ void __launch_bounds__(32 * kMtWarps, 1) mt_pass_kernel(GraphDev G, MtDev m, Ctl *ctl) {
    extern __shared__ __align__(16) char mt_smem[];
    MtShared &S = *reinterpret_cast<MtShared *>(mt_smem);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (__ldcg(&ctl->error)) return;
    if (G.k > kMtMaxK) {
        if (threadIdx.x == 0) fail(ctl, E_TOO_LARGE, 803);
        return;
    }
    int maxlen = 0;
    for (int p = 0; p < m.np; ++p) maxlen = max(maxlen, m.cnt[p]);
    const long long total = (long long)maxlen * m.np;
    if (threadIdx.x == 0) {
        S.prog = -1;
        S.done = 0;
    }
    __syncthreads();
    if (wid > 0) {
        unsigned acc = 0;
        for (long long i = wid - 1; i < total && mt_follow(S, i, kMtSeedsAhead); i += kMtAhead) {
            if (i >= total) break;
            const int j = (int)(i / m.np), p = (int)(i - (long long)j * m.np);
            if (j >= m.cnt[p]) continue;
            const int v = m.tv[m.off[p] + j];
            const int4 *r = m.rec + 4LL * v;
            const int4 A = r[0];
            if (r[1].y != 0) continue;
            acc ^= (unsigned)r[2].x ^ (unsigned)__ldg(G.vwgt + v) ^ mt_warm_row(G, m, A.x, A.y);
        }
        if (acc == 0x9e3779b9u) S.sink = acc;
        return;
    }
    for (int i = lane; i < G.k; i += 32) S.bw[i] = m.bw[i];
    for (int i = lane; i < kMtMaxK; i += 32) S.hist[i] = 0;
    const unsigned long long tseed = splitmix64(~m.seed);
    const long long Lmax = G.Lmax;
    long long gain_tot = 0;
    int searches = 0, tried_tot = 0, kept_tot = 0, sid = 0;
    int kbase = 0;   // kept movers listed so far (the list is kept_tot long at the end)
    bool bad = false;
    __syncwarp();
    // the todo entries in pass order (entry j of every pair, then j + 1), 32 at a time:
    // the lanes fetch them and their touched marks together; marks only ever go from 0
    // to set during a pass, so an entry seen touched is skipped at once and the others
    // are checked again when their turn comes
    for (long long pos = 0; pos < total && !bad; pos += 32) {
        if (lane == 0) *(volatile long long *)&S.prog = pos - 1;
        const long long q0 = pos + lane;
        int cv = -1;
        bool fresh = false;
        if (q0 < total) {
            const int j = (int)(q0 / m.np), p = (int)(q0 - (long long)j * m.np);
            if (j < m.cnt[p]) {
                cv = m.tv[m.off[p] + j];
                fresh = m.rec[4LL * cv + 1].y == 0;
            }
        }
        unsigned live = __ballot_sync(kFull, fresh);
        while (live && !bad) {
            const int v = __shfl_sync(kFull, cv, __ffs(live) - 1);
            if (lane == 0) *(volatile long long *)&S.prog = pos + __ffs(live) - 1;
            live &= live - 1;
            const int4 *rv = m.rec + 4LL * v;
            const int4 VA = rv[0], VB = rv[1], VC = rv[2], VD = rv[3];
            if (VB.y != 0) continue;
            if (!VA.w && mt_foreign(mt_slots(VC, VD), VA.z) == 0) continue;
            const int x0 = VA.x, x1 = VA.y;
            if (VA.w) {   // its slots mean nothing: is a neighbour outside its block?
                bool bnd = false;
                for (int jb = x0; jb < x1 && !bnd; jb += 32) {
                    const int jj = jb + lane;
                    bnd = __any_sync(kFull, jj < x1 && G.part[__ldg(G.adjncy + jj)] != VA.z);
                }
                if (!bnd) continue;
            }
            ++sid;
            // ---- one k-way search ----
            for (int i = lane; i < kMtBuckets / 32; i += 32) S.bits[i] = 0;
            __syncwarp();
            int nxt = 0;
            // start set: v, then its neighbours in CSR order that no search of the pass
            // queued and that are boundary vertices (all chosen before any is queued)
            const int deg = x1 - x0;
            for (int base = -1; base < deg && !bad; base += 32) {
                const int i = base + lane;
                int u = -1;
                if (i < 0) u = v;
                else if (i < deg) u = __ldg(G.adjncy + x0 + i);
                int4 A = make_int4(0, 0, 0, 0), B = A;
                MtSlots q = {};
                int4 *r = m.rec + 4LL * (u < 0 ? 0 : u);
                if (u >= 0) {
                    A = r[0];
                    B = r[1];
                    q = mt_slots(r[2], r[3]);
                }
                int g = 0, t = -1;
                const bool push = mt_gain_lanes(G, S.hist, u >= 0 && (u == v || B.y == 0), A.w != 0, q, u, A.z, A.x,
                                                A.y, tseed, g, t);
                const bool range = __all_sync(kFull, !push || (g >= -kMtGmax && g <= kMtGmax && t < G.k));
                const unsigned pm = __ballot_sync(kFull, push);
                if (!range || (long long)nxt + __popc(pm) > m.ecap) {
                    if (lane == 0) fail(ctl, range ? E_INTERNAL : E_TOO_LARGE, 804);
                    bad = true;
                    break;
                }
                const int at = mt_push(S, m, pm, push, push ? g + kMtGmax : 0, u, mt_word(A.y - A.x, A.z, t), A.x, nxt, lane);
                if (push) r[1] = make_int4(at, sid, B.z, 0);
                nxt += __popc(pm);
            }
            __syncwarp();
            long long best;
            int nm, best_len;
            bool stopped;
            mt_search(G, m, S, ctl, sid, true, nxt, 0, Lmax, tseed, lane, bad, best, nm, best_len, stopped);
            mt_finish(G, m, S, nm, best_len, lane, true, kbase);
            gain_tot -= best;
            tried_tot += nm;
            kept_tot += best_len;
            ++searches;
        }
    }
    __syncwarp();
    for (int i = lane; i < G.k; i += 32) {
        m.bw[i] = S.bw[i];
        G.blockw[i] = S.bw[i];
    }
    if (lane == 0) {
        *(volatile int *)&S.done = 1;
        m.res->gain = gain_tot;
        m.res->searches = searches;
        m.res->tried = tried_tot;
        m.res->kept = kept_tot;
    }
}

// The boundary candidates of the pass's kept moves, as a flow's commit lists them: each
// mover and its neighbours outside its block (one warp per mover).  Taken on the
// partition the pass leaves: a vertex that is a boundary vertex after the pass is a
// mover, a neighbour of one in another block, or was one before the pass (and listed).
__global__ void __launch_bounds__(kMtTPB) mt_bl_kernel(GraphDev G, MtDev m, Ctl *ctl) {
    if (__ldcg(&ctl->error)) return;
    const int nk = m.res->kept;
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nk; i += nw) {
        const int y = m.kept[i], t = G.part[y];
        const int a0 = __ldg(G.xadj + y), a1 = __ldg(G.xadj + y + 1);
        // slot a0 - 1 stands for the mover itself
        for (int q = a0 - 1 + lane; q < a1; q += 32) {
            const int z = q < a0 ? y : __ldg(G.adjncy + q);
            if ((q < a0 || G.part[z] != t) && !__ldcg(G.inb + z) && atomicExch(G.inb + z, 1) == 0)
                G.bl[atomicAdd(G.blc, 1)] = z;
        }
    }
}

// The search kernels' shared memory is above the default limit, and the rest of the SM's
// memory is to be L1: the prefetched rows and records live there.
static cudaError_t mt_shared_size(const void *kernel) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MtShared));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)((sizeof(MtShared) + 2048) * 100 / (228 * 1024)) + 1);
    return e;
}

cudaError_t launch_mt(const GraphDev &G, const MtDev &md, Ctl *ctl, int sms, cudaStream_t st, int *nl) {
    if (md.np <= 0) return cudaSuccess;
    cudaError_t e;
    if ((e = cudaMemsetAsync(md.cnt, 0, sizeof(int) * (size_t)md.np, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(md.bw, 0, sizeof(long long) * (size_t)G.k, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(md.chg, 0, (size_t)G.k, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(md.res, 0, sizeof(MtRes), st)) != cudaSuccess) return e;
    const int grid = 4 * (sms > 0 ? sms : 1);
    mt_count_kernel<<<grid, kMtTPB, sizeof(long long) * (size_t)G.k, st>>>(G, md);
    mt_offsets_kernel<<<1, 32, 0, st>>>(md, ctl);
    mt_fill_kernel<<<grid, kMtTPB, 0, st>>>(G, md, ctl);
    mt_sort_kernel<<<md.np, kMtTPB, 0, st>>>(md, ctl);
    if ((e = mt_shared_size(reinterpret_cast<const void *>(mt_pass_kernel))) != cudaSuccess) return e;
    mt_pass_kernel<<<1, 32 * kMtWarps, sizeof(MtShared), st>>>(G, md, ctl);
    *nl += 5;
    if (G.bl) {
        mt_bl_kernel<<<grid, kMtTPB, 0, st>>>(G, md, ctl);
        *nl += 1;
    }
    return cudaGetLastError();
}

// ------------------------------------------------- global k-way rounds ----
// One round of Section 2.2 with the setup of Section 6: a single k-way search started
// from every vertex with at least `need` blocks other than its own around it (1: the
// whole boundary; 2: the corner vertices), in ascending splitmix64(rs ^ v) order.
// Grid-wide: the start set is bucketed by the top bits of its keys (the keys are
// hashes, so the buckets hold a few entries each), each bucket is sorted by one
// thread, and the start vertices' gains and targets are computed side by side; then
// one warp queues them in order and runs the search.  Bucket scratch, in the entry
// array (free until the search): counts, fill cursors and offsets of the nb buckets
// (kw_scratch); the sorted start set: tv, with its packed gains and targets in tkey.

// counts, fill cursors, offsets (nb + 1 each) of the start set's buckets
struct KwScratch {
    int *cnt, *fil, *off;
};
__device__ __forceinline__ KwScratch kw_scratch(const MtDev &m, int nb) {
    int *b = reinterpret_cast<int *>(m.ent);
    return {b, b + (nb + 1), b + 2 * (nb + 1)};
}

__global__ void __launch_bounds__(kMtTPB) kw_count_kernel(GraphDev G, MtDev m, int need, unsigned long long rs,
                                                          int bbits) {
    const KwScratch K = kw_scratch(m, 1 << bbits);
    extern __shared__ long long s_bw[];   // [k]
    for (int i = threadIdx.x; i < G.k; i += blockDim.x) s_bw[i] = 0;
    __syncthreads();
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < G.n; v += gridDim.x * blockDim.x) {
        const int c = __ldg(G.vwgt + v);
        if (c) atomicAdd(reinterpret_cast<unsigned long long *>(s_bw + G.part[v]), (unsigned long long)c);
        MtSlots q;
        int pv;
        const bool over = mt_build(G, m, v, q, pv);
        if (!over && mt_foreign(q, pv) < need) continue;   // (over: at least eight blocks are not its own)
        const unsigned long long key = splitmix64(rs ^ (unsigned long long)(unsigned)v);
        atomicAdd(K.cnt + (int)(key >> (64 - bbits)), 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G.k; i += blockDim.x)
        if (s_bw[i]) atomicAdd(reinterpret_cast<unsigned long long *>(m.bw + i), (unsigned long long)s_bw[i]);
}

// Exclusive scan of the bucket counts (one CTA of 1,024 threads, 4,096 counts a step, read
// and written side by side: a contiguous range per thread took 167 us for 65,536
// buckets); the start set's size goes to cnt[0].
__global__ void __launch_bounds__(1024) kw_offsets_kernel(MtDev m, int nb) {
    __shared__ int wsum[32];
    __shared__ int s_carry;
    const KwScratch K = kw_scratch(m, nb);
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    if (t == 0) s_carry = 0;
    __syncthreads();
    for (int b0 = 0; b0 < nb; b0 += 4096) {
        int c[4], s = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int b = b0 + 4 * t + i;
            c[i] = b < nb ? K.cnt[b] : 0;
            s += c[i];
        }
        int incl = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            int x = wsum[lane];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(kFull, x, d);
                if (lane >= d) x += y;
            }
            wsum[lane] = x;
        }
        __syncthreads();
        int o = s_carry + (wid ? wsum[wid - 1] : 0) + incl - s;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int b = b0 + 4 * t + i;
            if (b < nb) {
                K.off[b] = o;
                K.fil[b] = 0;
                o += c[i];
            }
        }
        __syncthreads();
        if (t == 0) s_carry += wsum[31];
        __syncthreads();
    }
    if (t == 0) {
        K.off[nb] = s_carry;
        m.cnt[0] = s_carry;
    }
}

__global__ void __launch_bounds__(kMtTPB) kw_place_kernel(GraphDev G, MtDev m, int need, unsigned long long rs,
                                                          int bbits) {
    const KwScratch K = kw_scratch(m, 1 << bbits);
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < G.n; v += gridDim.x * blockDim.x) {
        const int4 *r = m.rec + 4LL * v;
        const int4 a = r[0];
        if (!a.w && mt_foreign(mt_slots(r[2], r[3]), a.z) < need) continue;
        const unsigned long long key = splitmix64(rs ^ (unsigned long long)(unsigned)v);
        const int b = (int)(key >> (64 - bbits));
        const int pos = K.off[b] + atomicAdd(K.fil + b, 1);
        m.tkey[pos] = key;
        m.tv[pos] = v;
    }
}

// Each bucket ascending by (key, vertex), one thread per bucket (insertion sort).
__global__ void __launch_bounds__(kMtTPB) kw_bsort_kernel(MtDev m, int nb) {
    const KwScratch K = kw_scratch(m, nb);
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
        const int o0 = K.off[b], o1 = K.off[b + 1];
        for (int i = o0 + 1; i < o1; ++i) {
            const unsigned long long ki = m.tkey[i];
            const int vi = m.tv[i];
            int j = i - 1;
            while (j >= o0 && (m.tkey[j] > ki || (m.tkey[j] == ki && m.tv[j] > vi))) {
                m.tkey[j + 1] = m.tkey[j];
                m.tv[j + 1] = m.tv[j];
                --j;
            }
            m.tkey[j + 1] = ki;
            m.tv[j + 1] = vi;
        }
    }
}

// Gain and target of every start vertex on the round's starting partition, packed as
// (gain + kMtGmax) << 32 | target into tkey; a gain out of range fails the round.
__global__ void __launch_bounds__(kMtTPB) kw_gain_kernel(GraphDev G, MtDev m, Ctl *ctl) {
    __shared__ int s_hist[kMtTPB / 32][kMtMaxK];
    int *hist = s_hist[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < kMtMaxK; i += 32) hist[i] = 0;
    __syncwarp();
    const int ns = m.cnt[0];
    const unsigned long long tseed = splitmix64(~m.seed);
    for (int b = blockIdx.x * blockDim.x + threadIdx.x - lane; b < ns; b += gridDim.x * blockDim.x) {
        const int i = b + lane;
        int u = 0, g = 0, t = -1;
        int4 A = make_int4(0, 0, 0, 0);
        MtSlots q = {};
        if (i < ns) {
            u = m.tv[i];
            const int4 *r = m.rec + 4LL * u;
            A = r[0];
            q = mt_slots(r[2], r[3]);
        }
        const bool has = mt_gain_lanes(G, hist, i < ns, A.w != 0, q, u, A.z, A.x, A.y, tseed, g, t);
        if (i >= ns) continue;
        if (!has || g < -kMtGmax || g > kMtGmax) {
            fail(ctl, E_INTERNAL, 806);
            continue;
        }
        m.tkey[i] = ((unsigned long long)(unsigned)(g + kMtGmax) << 32) | (unsigned)t;
    }
}

// The round's queue, built on the grid: the start set pushed in its order makes bucket
// stacks whose entries leave the highest bucket first and, within a bucket, last pushed
// first.  The entries are laid out in that order (a counting sort by bucket), each on the
// one after it, so that the search pops neighbouring words and the warps that prefetch for
// it know what comes next.  Each warp of kw_hist_kernel ranks a chunk of kKwChunk entries
// within the chunk's buckets (32 at a time, a shared-memory count of each bucket),
// kw_stitch_kernel turns the chunks' counts into offsets, kw_fix_kernel writes the entries.
constexpr int kKwWarps = 4;       // warps per CTA of kw_hist_kernel (2,048 counts each)
constexpr int kKwRankShift = 48;  // tkey: rank in its chunk and bucket << 48 | bucket << 32 | target

__global__ void __launch_bounds__(32 * kKwWarps) kw_hist_kernel(MtDev m, Ctl *ctl) {
    __shared__ int s_cnt[kKwWarps][kMtBuckets];
    if (__ldcg(&ctl->error)) return;   // (a gain out of range left the packed keys unwritten)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int ns = m.cnt[0];
    const int nch = (ns + kKwChunk - 1) / kKwChunk;
    const int chunk = blockIdx.x * kKwWarps + wid;
    if (chunk >= nch || chunk >= m.kwchunks) return;   // (the whole warp leaves together)
    int *cnt = s_cnt[wid];
    for (int b = lane; b < kMtBuckets; b += 32) cnt[b] = 0;
    __syncwarp();
    const int c0 = chunk * kKwChunk, c1 = min(ns, c0 + kKwChunk);
    for (int base = c0; base < c1; base += 32) {
        const int i = base + lane;
        const bool valid = i < c1;
        unsigned long long pk = 0;
        int b = 0;
        if (valid) {
            pk = m.tkey[i];
            b = min((int)(pk >> 32), kMtBuckets - 1);   // (always in range: the gains were checked)
        }
        const unsigned grp = __match_any_sync(kFull, valid ? b : -1);
        const unsigned lower = grp & mt_lanemask_lt();
        int had = 0;
        if (valid) had = cnt[b];
        __syncwarp();
        if (valid) {
            m.tkey[i] = pk | (unsigned long long)(had + __popc(lower)) << kKwRankShift;
            if (lower == 0) cnt[b] = had + __popc(grp);   // (the bucket's lowest lane)
        }
        __syncwarp();
    }
    int *cl = m.kwtab + (long long)chunk * kMtBuckets;
    for (int b = lane; b < kMtBuckets; b += 32) cl[b] = cnt[b];
}

// One thread per bucket: over the chunks in order, the bucket's entries before each
// chunk, and all of them.
__global__ void __launch_bounds__(256) kw_stitch_kernel(MtDev m) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= kMtBuckets) return;
    const int ns = m.cnt[0];
    const int nch = min((ns + kKwChunk - 1) / kKwChunk, m.kwchunks);
    int carry = 0;
    for (int k = 0; k < nch; k += 8) {
        int c[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) c[t] = k + t < nch ? m.kwtab[(long long)(k + t) * kMtBuckets + b] : 0;
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (k + t < nch) {
                m.kwtab[(long long)(k + t) * kMtBuckets + b] = carry;
                carry += c[t];
            }
    }
    m.kwtab[(long long)m.kwchunks * kMtBuckets + b] = carry;
}

// First entry of each bucket (base, in shared memory; kMtBuckets of them): the entries
// of all higher buckets come before it.  Every thread of a CTA of kMtTPB calls it.
__device__ __forceinline__ void kw_bases(const MtDev &m, int *base) {
    __shared__ int wsum[kMtTPB / 32];
    constexpr int E = kMtBuckets / kMtTPB;
    const int *tot = m.kwtab + (long long)m.kwchunks * kMtBuckets;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    int c[E], s = 0;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        c[i] = tot[kMtBuckets - 1 - (t * E + i)];
        s += c[i];
    }
    int incl = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    int o = incl - s;
    for (int i = 0; i < wid; ++i) o += wsum[i];
#pragma unroll
    for (int i = 0; i < E; ++i) {
        base[kMtBuckets - 1 - (t * E + i)] = o;
        o += c[i];
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kMtTPB) kw_fix_kernel(MtDev m, Ctl *ctl) {
    __shared__ int base[kMtBuckets];
    if (__ldcg(&ctl->error)) return;
    kw_bases(m, base);
    const int ns = m.cnt[0];
    const int *tot = m.kwtab + (long long)m.kwchunks * kMtBuckets;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ns; i += gridDim.x * blockDim.x) {
        const unsigned long long pk = m.tkey[i];
        const int u = m.tv[i], b = min((int)(pk >> 32) & 0xffff, kMtBuckets - 1);
        const int rank = m.kwtab[(long long)(i / kKwChunk) * kMtBuckets + b] + (int)(pk >> kKwRankShift);
        const int pos = base[b] + tot[b] - 1 - rank;
        const int4 A = m.rec[4LL * u];
        m.ent[pos] = make_int4(u, rank > 0 ? pos + 1 : -1, mt_word(A.y - A.x, A.z, (int)(unsigned)pk), A.x);
        m.rec[4LL * u + 1] = make_int4(pos, 1, 0, 0);   // (queued by search 1, the round's only one)
    }
}

// The round's search: one warp takes the queue the grid built and searches.
// res: gain kept, tried, kept; stopped = 1 if the KaSPar rule stopped the search.
__global__ void __launch_bounds__(32 * kMtWarps, 1) kw_search_kernel(GraphDev G, MtDev m, Ctl *ctl) {
    extern __shared__ __align__(16) char mt_smem[];
    MtShared &S = *reinterpret_cast<MtShared *>(mt_smem);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (__ldcg(&ctl->error)) return;
    const int ns = m.cnt[0];
    for (int i = threadIdx.x; i < G.k; i += blockDim.x) S.bw[i] = m.bw[i];
    for (int i = threadIdx.x; i < kMtMaxK; i += blockDim.x) S.hist[i] = 0;
    if (threadIdx.x == 0) {
        S.prog = -1;
        S.done = 0;
    }
    const int *tot = m.kwtab + (long long)m.kwchunks * kMtBuckets;
    for (int w = threadIdx.x; w < kMtBuckets / 32; w += blockDim.x) {
        unsigned word = 0;
        for (int j = 0; j < 32; ++j) word |= (tot[w * 32 + j] > 0 ? 1u : 0u) << j;
        S.bits[w] = word;
    }
    __syncthreads();
    if (wid == 0) {
        // each bucket's first entry: the entries of all higher buckets come before it
        int o = 0;   // 32 buckets at a time, from the highest
        for (int b0 = 0; b0 < kMtBuckets; b0 += 32) {
            const int b = kMtBuckets - 1 - (b0 + lane), c = tot[b];
            int incl = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += y;
            }
            S.top[b] = o + incl - c;
            o += __shfl_sync(kFull, incl, 31);
        }
    } else {
        unsigned acc = 0;
        for (long long i = wid - 1; i < ns && mt_follow(S, i, kKwEntsAhead); i += kMtAhead) {
            if (i >= ns) break;
            const int4 e = m.ent[i];
            if (e.z == 0) continue;
            acc ^= (unsigned)__ldg(G.vwgt + e.x) ^ mt_warm_row(G, m, e.w, e.w + mt_word_deg(e.z));
        }
        if (acc == 0x9e3779b9u) S.sink = acc;
        return;
    }
    __syncwarp();
    const unsigned long long tseed = splitmix64(~m.seed);
    bool bad = false;
    long long best = 0;
    int nm = 0, best_len = 0, kbase = 0;
    bool stopped = false;
    mt_search(G, m, S, ctl, 1, false, ns, ns, G.Lmax, tseed, lane, bad, best, nm, best_len, stopped);
    mt_finish(G, m, S, nm, best_len, lane, false, kbase);
    for (int i = lane; i < G.k; i += 32) m.bw[i] = S.bw[i];
    if (lane == 0) {
        *(volatile int *)&S.done = 1;
        m.res->gain = -best;
        m.res->searches = 1;
        m.res->tried = nm;
        m.res->kept = best_len;
        m.res->stopped = stopped ? 1 : 0;
    }
}

cudaError_t launch_kway_round(const GraphDev &G, const MtDev &md, Ctl *ctl, int need, unsigned long long rs,
                              int sms, cudaStream_t st, int *nl) {
    int bbits = 1;
    while (bbits < 16 && (2ll << (bbits + 3)) <= G.n) ++bbits;   // about 8 vertices per bucket
    const int nb = 1 << bbits;
    cudaError_t e;
    if ((e = cudaMemsetAsync(md.ent, 0, sizeof(int) * (size_t)nb, st)) != cudaSuccess) return e;   // bucket counts
    if ((e = cudaMemsetAsync(md.bw, 0, sizeof(long long) * (size_t)G.k, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(md.res, 0, sizeof(MtRes), st)) != cudaSuccess) return e;
    const int grid = 4 * (sms > 0 ? sms : 1);
    kw_count_kernel<<<grid, kMtTPB, sizeof(long long) * (size_t)G.k, st>>>(G, md, need, rs, bbits);
    kw_offsets_kernel<<<1, 1024, 0, st>>>(md, nb);
    kw_place_kernel<<<grid, kMtTPB, 0, st>>>(G, md, need, rs, bbits);
    kw_bsort_kernel<<<(nb + kMtTPB - 1) / kMtTPB, kMtTPB, 0, st>>>(md, nb);
    kw_gain_kernel<<<grid, kMtTPB, 0, st>>>(G, md, ctl);
    // the queue: chunks of the start set ranked by warps, stitched per bucket, written
    const int chunks = (G.n + kKwChunk - 1) / kKwChunk;   // >= the start set's chunks
    kw_hist_kernel<<<(chunks + kKwWarps - 1) / kKwWarps, 32 * kKwWarps, 0, st>>>(md, ctl);
    kw_stitch_kernel<<<(kMtBuckets + 255) / 256, 256, 0, st>>>(md);
    kw_fix_kernel<<<grid, kMtTPB, 0, st>>>(md, ctl);
    if ((e = mt_shared_size(reinterpret_cast<const void *>(kw_search_kernel))) != cudaSuccess) return e;
    kw_search_kernel<<<1, 32 * kMtWarps, sizeof(MtShared), st>>>(G, md, ctl);
    *nl += 9;
    return cudaGetLastError();
}

}  // namespace fr
