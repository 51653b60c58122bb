// Two-way FM local search with TopGain on each pair of a round, before the pair's flow
// (Sanders & Schulz, Section 2.2: one priority queue of movable vertices per block,
// keyed by the gain -- the decrease of the pair cut when the vertex changes blocks --,
// every vertex moves at most once, the queues start with the boundary in random order,
// TopGain takes the block whose best vertex has the larger gain and the heavier block
// while one is overloaded, and the moves are rolled back to the best cut found within
// the balance constraint; the setup of Section 6 stops a search once more than a given
// fraction of the pair's vertices moved without an improvement, and runs the FM search
// first and the flow after it).
//
// The keys follow the readings of the CPU oracle: gains and the boundary within
// G[A u B]; order by gain, then by stamp, larger first, where the initial stamps are
// random 63-bit values (splitmix64 of the pair's seed and the vertex id, the random
// initial order) and every later insertion or gain change takes a larger stamp than
// any before, in the adjacency order of the moved vertex; ties of the two top gains
// go by a seeded bit; the best state is the smallest (overload, cut, max block weight).
//
// GPU form.  Pairs of a round are block-disjoint, so one CTA searches one pair on
// 16-byte vertex records shared by the round, one load for all that a move needs of a
// neighbour.  Each block's queue is an array of gain buckets, each bucket a stack of
// entries in global memory with its top in shared memory: a gain change pushes a new
// entry (its stamp is larger than every earlier one, so a stack stays ordered by stamp)
// and marks the vertex's old one dead; pops skip dead entries.  The latest 4,096 entries
// are in shared memory too, with their vertices' rows, so that most tops are found there.
// The initial stacks come from a sort of the boundary by (block, gain, stamp).
// One warp runs the moves: the top of each block's highest non-empty bucket (16 lanes a
// block look at 16 buckets; flags tell which groups of 16 may hold an entry), the TopGain
// choice, then the moved vertex's arcs 32 at a time -- gain updates and the pushes, placed
// in arc order so that every bucket stays ordered.  The other warps read the rows of the
// entries that are pushed, and the records of the rows' neighbours, into L1 before they are
// popped.  The kept moves, the block weights and the boundary candidate list are written by
// the whole CTA afterwards.  Bound by the one warp's chain, about 2,100 cycles a move (shared
// memory and L1 round trips, and five cycles an instruction).  One round of rgg3d 262,144
// vertices, k = 64 with its flows: 35.5 ms with separate arrays, entries told stale by the
// vertex's version and a lookahead of one entry; 32.1 with dead entries and the ring; 25.0
// with records, the warps that read ahead (2.1 ms of it) and the search by groups.
#include <climits>

#include "fm_kernel.cuh"

namespace fr {

constexpr int kFmTPB = 256;

// ---------------------------------------------------------------- counts ----
// Vertex and arc counts of every paired block.
__global__ void __launch_bounds__(kFmTPB) fm_count_kernel(Work w, FmDev f) {
    const GraphDev G = w.graphs[0];
    extern __shared__ int s_cnt[];   // [2k]
    for (int i = threadIdx.x; i < 2 * G.k; i += blockDim.x) s_cnt[i] = 0;
    __syncthreads();
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < G.n; v += gridDim.x * blockDim.x) {
        const int b = G.part[v];
        if (side_of(G, b) < 0) continue;
        atomicAdd(&s_cnt[b], 1);
        atomicAdd(&s_cnt[G.k + b], __ldg(G.xadj + v + 1) - __ldg(G.xadj + v));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G.k; i += blockDim.x) {
        if (s_cnt[i]) atomicAdd(f.blockn + i, s_cnt[i]);
        if (s_cnt[G.k + i]) atomicAdd(f.blockarcs + i, s_cnt[G.k + i]);
    }
}

// Region offsets of the pairs (one CTA): vertices (vlist, mlog) by pair vertex counts,
// stack entries by vertex + arc counts (every push is a boundary vertex at the start or
// the update of one arc of a moved vertex).  Clears the block counts for the next round.
__global__ void __launch_bounds__(1024) fm_offsets_kernel(Work w, FmDev f) {
    const GraphDev G = w.graphs[0];
    if (threadIdx.x == 0) {
        long long vo = 0, eo = 0;
        for (int p = 0; p < w.npairs; ++p) {
            const PairDev P = w.pairs[p];
            const int n_p = f.blockn[P.a] + f.blockn[P.b];
            const long long a_p = (long long)f.blockarcs[P.a] + f.blockarcs[P.b];
            f.voff[p] = vo;
            f.eoff[p] = eo;
            f.np[p] = n_p;
            f.bcnt[p] = 0;
            vo += n_p;
            eo += n_p + a_p;
        }
        f.eoff[w.npairs] = eo;
        if (vo > G.n || eo > f.ecap) fail(w.ctl, E_INTERNAL, 700);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G.k; i += blockDim.x) f.blockn[i] = f.blockarcs[i] = 0;
}

// The records of all vertices: the weights of a paired vertex to its own block and to the
// partner block within G[A u B] (so that the moves never scan an adjacency for them) and
// its row; vertices with an edge to the partner are the boundary and enter their pair's list.
__global__ void __launch_bounds__(kFmTPB) fm_gather_kernel(Work w, FmDev f) {
    if ((w.prev_err && __ldcg(w.prev_err)) || __ldcg(&w.ctl->error)) return;
    const GraphDev G = w.graphs[0];
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < G.n; v += gridDim.x * blockDim.x) {
        const int b = G.part[v];
        const int s = side_of(G, b);
        if (s < 0) {
            f.rec[v].z = -1;
            continue;
        }
        const PairDev P = w.pairs[s >> 1];
        const int partner = (s & 1) ? P.a : P.b;
        int in = 0, ex = 0;
        const int j0 = __ldg(G.xadj + v), j1 = __ldg(G.xadj + v + 1);
        for (int j = j0; j < j1; ++j) {
            const int pu = G.part[__ldg(G.adjncy + j)];
            const int wt = __ldg(G.adjwgt + j);
            if (pu == b) in += wt;
            else if (pu == partner) ex += wt;
        }
        // (a weight beyond ten bits ends the search before it reads the record)
        f.rec[v] = make_int4((in & 1023) | (ex & 1023) << 10 | (int)((unsigned)(j1 - j0) << 20), 0, b, j0);
        if (ex == 0) continue;
        const int pos = atomicAdd(f.bcnt + (s >> 1), 1);
        f.vlist[f.voff[s >> 1] + pos] = v;
    }
}

// --------------------------------------------------------------- search ----

struct SortRef {   // one sort element: (bucket key, stamp, vertex), ascending by (bk, st, -v)
    unsigned long long *st;
    int *bk, *v;
    __device__ bool less(int i, int j) const {
        if (bk[i] != bk[j]) return bk[i] < bk[j];
        if (st[i] != st[j]) return st[i] < st[j];
        return v[i] > v[j];
    }
    __device__ void swap(int i, int j) const {
        const unsigned long long t = st[i]; st[i] = st[j]; st[j] = t;
        const int b = bk[i]; bk[i] = bk[j]; bk[j] = b;
        const int x = v[i]; v[i] = v[j]; v[j] = x;
    }
};

// Bitonic sort of m (a power of two) elements by the whole CTA.
__device__ void bitonic(const SortRef &r, int m) {
    for (int k = 2; k <= m; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < m; i += blockDim.x) {
                const int l = i ^ j;
                if (l <= i) continue;
                const bool up = (i & k) == 0;
                if (up ? r.less(l, i) : r.less(i, l)) r.swap(i, l);
            }
            __syncthreads();
        }
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

constexpr int kFmGroup = 16, kFmGroups = kFmMaxBuckets / kFmGroup;   // buckets of a group, groups of a block

constexpr int kFmAhead = kFmTPB / 32 - 1;   // warps that read ahead of the moves
constexpr int kFmFresh = 64;                // pushed entries older than this are left
constexpr int kFmSeedsAhead = 16;           // entries of each block's start they are ahead
constexpr int kFmIdle = 1 << 22;            // polls without work before such a warp gives up
constexpr int kFmRing = kFmSortSmem;   // latest entries kept where the boundary was sorted (16 bytes each)

struct __align__(16) FmShared {
    int top[2 * kFmMaxBuckets];          // top entry of each (block, bucket) stack, -1 empty
    unsigned char group[2 * kFmGroups];  // groups of stacks that may hold an entry
    long long red[kFmTPB / 32];
    int best_len, tried;
    int pushes, moves, done;             // progress, for the warps that read ahead
    unsigned sink;                       // (their loads end here)
    long long best_cut, best_wA, best_wB;
};

// What the warps behind the moving one do: they read the rows, and the records of the rows'
// neighbours, that it will need next into L1, so that a move finds them there.  The start's
// entries come first, from the top of each block down and two a move; then the pushed
// entries, while they are new.
__device__ __forceinline__ void fm_ahead(const GraphDev &G, const FmDev &f, FmShared &S, const int4 *ring,
                                         long long E, int n0, int B) {
    const int lane = threadIdx.x & 31, me = (threadIdx.x >> 5) - 1;
    const int nnz = __ldg(G.xadj + G.n);
    unsigned acc = 0;
    auto warm = [&](int v, int j0, int j1) {
        acc ^= (unsigned)__ldg(G.vwgt + v);
        for (int j = j0 + lane, end = fm_row_end(j0, j1, nnz); j < end; j += 32)
            acc ^= (unsigned)__ldg(G.adjwgt + j) ^ (unsigned)f.rec[__ldg(G.adjncy + j)].x;
    };
    int seed = me, push = me;
    for (int polls = 0; polls < kFmIdle; ++polls) {
        if (*(volatile int *)&S.done) break;
        const int pushes = *(volatile int *)&S.pushes, moves = *(volatile int *)&S.moves;
        if (push < pushes) {
            if (push < pushes - kFmFresh) push += (pushes - kFmFresh - push + kFmAhead - 1) / kFmAhead * kFmAhead;
            if (push >= pushes) continue;
            const int4 t = ring[(int)((E + B + push) & (kFmRing - 1))];
            push += kFmAhead;
            if (t.x >= 0) warm(t.x, t.z, t.w);
            polls = 0;
        } else if (seed < 2 * max(n0, B - n0) && seed < 2 * (moves + kFmSeedsAhead)) {
            const int lo = (seed & 1) ? n0 : 0, i = ((seed & 1) ? B : n0) - 1 - (seed >> 1);
            seed += kFmAhead;
            const int v = i >= lo ? f.ent[E + i].x : -1;
            if (v >= 0) {
                const int4 r = f.rec[v];
                warm(v, r.w, r.w + fm_deg(r.x));
            }
            polls = 0;
        } else {
            __nanosleep(100);
        }
    }
    if (acc == 0x9e3779b9u) S.sink = acc;
}

__global__ void __launch_bounds__(kFmTPB, 1) fm_pair_kernel(Work w, FmDev f) {
    extern __shared__ __align__(16) char fm_smem[];
    FmShared &S = *reinterpret_cast<FmShared *>(fm_smem);
    const GraphDev G = w.graphs[0];
    const int p = blockIdx.x;
    const PairDev P = w.pairs[p];
    const int a = P.a, b = P.b;
    const int n_p = f.np[p];
    if ((w.prev_err && __ldcg(w.prev_err)) || __ldcg(&w.ctl->error)) return;   // (the gather may not have run)
    const int B = f.bcnt[p];
    int *vl = f.vlist + f.voff[p];
    int *ml = f.mlog + f.voff[p];
    FmRes *R = f.res + p;
    const long long wA0 = G.blockw[a], wB0 = G.blockw[b];
    if (n_p == 0 || f.permille <= 0) {
        if (threadIdx.x == 0) *R = FmRes{0, wA0, wB0, 0, wA0, wB0, 0, 0};
        return;
    }
    const int gmax = __ldcg(f.maxwdeg);   // |gain| <= max weighted degree
    if (2 * gmax + 1 > kFmMaxBuckets) {
        if (threadIdx.x == 0) fail(w.ctl, E_TOO_LARGE, 701);
        return;
    }
    const unsigned long long fs = splitmix64(w.seed ^ ((unsigned long long)(unsigned)a << 32) ^ (unsigned)b);
    const long long E = f.eoff[p];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    unsigned long long t_mark = globaltimer();
    auto mark = [&](int idx) {
        const unsigned long long now = globaltimer();
        if (threadIdx.x == 0) atomicAddLL(&w.ctl->timers[idx], (long long)(now - t_mark));
        t_mark = now;
    };
    // 1. sort the boundary by (block, bucket, stamp)
    int m = 1;
    while (m < B) m <<= 1;
    SortRef sr;
    char *sm_sort = fm_smem + sizeof(FmShared);
    if (m <= kFmSortSmem) {
        sr.st = reinterpret_cast<unsigned long long *>(sm_sort);
        sr.bk = reinterpret_cast<int *>(sm_sort + 8ull * kFmSortSmem);
        sr.v = sr.bk + kFmSortSmem;
    } else {
        long long so = 0;   // this pair's scratch: after the larger boundaries of earlier pairs
        for (int q = 0; q < p; ++q) {
            const int bq = f.bcnt[q];
            int mq = 1;
            while (mq < bq) mq <<= 1;
            if (mq > kFmSortSmem) so += mq;
        }
        if (so + m > f.scap) {
            if (threadIdx.x == 0) fail(w.ctl, E_INTERNAL, 702);
            return;
        }
        sr.st = f.skey + so;
        sr.bk = f.sbkt + so;
        sr.v = f.sv + so;
    }
    long long c0 = 0;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        if (i < B) {
            const int v = vl[i];
            const int4 r = f.rec[v];
            const int side = r.z == a ? 0 : 1;
            const int g = fm_ext(r.x) - fm_in(r.x);
            sr.bk[i] = side * kFmMaxBuckets + g + gmax;
            sr.st[i] = splitmix64(fs ^ (unsigned long long)(unsigned)v) >> 1;
            sr.v[i] = v;
            if (side == 0) c0 += fm_ext(r.x);
        } else {
            sr.bk[i] = INT_MAX;
            sr.st[i] = ~0ull;
            sr.v[i] = -1;
        }
    }
    for (int i = threadIdx.x; i < 2 * kFmMaxBuckets; i += blockDim.x) S.top[i] = -1;
    for (int i = threadIdx.x; i < 2 * kFmGroups; i += blockDim.x) S.group[i] = 0;
    for (int o = 16; o > 0; o >>= 1) c0 += __shfl_down_sync(0xffffffffu, c0, o);
    if (lane == 0) S.red[warp] = c0;
    __syncthreads();
    bitonic(sr, m);
    long long cut0 = 0;
    for (int i = 0; i < kFmTPB / 32; ++i) cut0 += S.red[i];
    // 2. initial stacks: entries in sorted order, each below its predecessor in the bucket
    for (int i = threadIdx.x; i < B; i += blockDim.x) {
        const int bk = sr.bk[i], v = sr.v[i];
        const int below = (i > 0 && sr.bk[i - 1] == bk) ? (int)(E + i - 1) : -1;
        f.ent[E + i] = make_int2(v, below);
        f.rec[v].y = (int)(E + i) + 1;
        if (i + 1 == B || sr.bk[i + 1] != bk) {
            S.top[bk] = (int)(E + i);
            S.group[bk / kFmGroup] = 1;
        }
    }
    int n0 = 0;   // boundary vertices of block a: the first n0 entries
    for (int h = B; n0 < h;) {
        const int mid = (n0 + h) >> 1;
        if (sr.bk[mid] < kFmMaxBuckets) n0 = mid + 1;
        else h = mid;
    }
    if (threadIdx.x == 0) S.pushes = S.moves = S.done = 0;
    __syncthreads();   // (the sort's shared memory is free from here: the ring)
    int4 *ring = reinterpret_cast<int4 *>(fm_smem + sizeof(FmShared));   // {vertex or -1, entry below, row}
    for (int i = threadIdx.x; i < kFmRing; i += blockDim.x) ring[i] = make_int4(-1, -1, 0, 0);
    __syncthreads();

    mark(T_FM_SORT);
    // 3. the moves (warp 0)
    if (warp > 0) {
        fm_ahead(G, f, S, ring, E, n0, B);
    } else {
        const long long Lmax = G.Lmax;
        const int limit = (int)min((long long)f.permille * n_p / 1000, (long long)INT_MAX - 1);
        long long cut = cut0, wA = wA0, wB = wB0;
        long long bcut = cut, bwA = wA, bwB = wB;
        long long bmx = wA > wB ? wA : wB, bov = bmx > Lmax ? bmx - Lmax : 0;
        int nm = 0, best_len = 0;
        int idle = 0;
        int nxt = (int)E + B;
        const int eend = (int)f.eoff[p + 1];   // entries of this pair: [E, eend)
        const int ring0 = nxt;                 // first entry pushed by a move
        unsigned ties = 0;                     // bits of moves nm & ~31 on
        bool over = bov > 0;                   // a block is overloaded
        const int hl = lane & 15, side = lane >> 4;
        int hg0 = kFmGroups - 1, hg1 = kFmGroups - 1;   // no group above these holds an entry
        bool bad = false;
        for (;;) {
            // top of each block: the highest bucket with a live entry (lanes 0 to 15 look at
            // the buckets of block a's highest group, 16 to 31 at those of block b's); dead
            // entries above it go
            int tb[2], hb;
            int4 t;
            const int ring_lo = max(ring0, nxt - kFmRing);   // entries from here on are in the ring
            int hg = lane < 16 ? hg0 : hg1, key0 = side * kFmMaxBuckets + hg * kFmGroup;
            int mine = hg >= 0 ? S.top[key0 + hl] : -1;      // this lane's stack
            for (;;) {
                const unsigned has = (__ballot_sync(0xffffffffu, mine >= 0) >> (lane & 16)) & 0xffffu;
                const int w16 = has ? 31 - __clz(has) : 0;
                int e = __shfl_sync(0xffffffffu, mine, (lane & 16) + w16);
                hb = has ? hg * kFmGroup + w16 : -1;
                t = make_int4(-1, -1, 0, 0);
                if (e >= ring_lo) t = ring[e & (kFmRing - 1)];
                if (!__any_sync(0xffffffffu, hg >= 0 && t.x < 0)) break;
                if (e >= 0 && t.x < 0) {   // an entry from before the ring, or a dead one (uniform within a half)
                    const bool dead = e >= ring_lo;
                    if (dead) e = t.y;
                    while (e >= 0) {
                        if (e >= ring_lo) {
                            t = ring[e & (kFmRing - 1)];
                        } else {
                            const int2 h = f.ent[e];
                            t = make_int4(h.x, h.y, 0, 0);
                            if (h.x >= 0) {
                                const int4 r = f.rec[h.x];
                                t.z = r.w;
                                t.w = r.w + fm_deg(r.x);
                            }
                        }
                        if (t.x >= 0) break;
                        e = t.y;
                    }
                    if (hl == w16 && e != mine) S.top[key0 + hl] = mine = e;
                }
                if (__any_sync(0xffffffffu, hg >= 0 && !has)) {   // a group without entries: the next one
                    if (hg >= 0 && !has && hl == 0) S.group[side * kFmGroups + hg] = 0;
                    __syncwarp();
                    const uint2 fl = reinterpret_cast<const uint2 *>(S.group)[lane];
                    const int g8 = fl.y ? 7 - (__clz(fl.y) >> 3) : 3 - (__clz(fl.x) >> 3);
                    const int g = fl.x | fl.y ? hl * 8 + g8 : -1;
                    hg0 = __reduce_max_sync(0xffffffffu, lane < 16 ? g : -1);
                    hg1 = __reduce_max_sync(0xffffffffu, lane < 16 ? -1 : g);
                    hg = lane < 16 ? hg0 : hg1;
                    key0 = side * kFmMaxBuckets + hg * kFmGroup;
                    mine = hg >= 0 ? S.top[key0 + hl] : -1;
                } else if (!__any_sync(0xffffffffu, has && t.x < 0)) {
                    break;
                }
            }
            tb[0] = __shfl_sync(0xffffffffu, hb, 0);
            tb[1] = __shfl_sync(0xffffffffu, hb, 16);
            if (tb[0] < 0 && tb[1] < 0) break;
            if ((nm & 31) == 0) ties = __ballot_sync(0xffffffffu, splitmix64(~fs ^ (unsigned long long)(nm + lane)) & 1);
            int s = tb[0] == tb[1] ? (int)(ties >> (nm & 31)) & 1 : tb[0] < tb[1];
            if (over) {
                s = wA >= wB ? 0 : 1;
                if ((s ? tb[1] : tb[0]) < 0) s = 1 - s;
            }
            const int ts = s ? tb[1] : tb[0], key = s * kFmMaxBuckets + ts;
            const int v = __shfl_sync(0xffffffffu, t.x, s * 16), j0 = __shfl_sync(0xffffffffu, t.z, s * 16);
            const int j1 = __shfl_sync(0xffffffffu, t.w, s * 16);
            const int g = ts - gmax;
            const int from = s ? b : a;
            const long long cv = __ldg(G.vwgt + v);
            // pop
            if (lane == s * 16) {
                S.top[key] = t.y;
                f.rec[v].z = -1;
                ml[nm] = v;
            }
            ++nm;
            cut -= g;
            __syncwarp();
            // the moved vertex's arcs, 32 at a time in adjacency order
            for (int jb = j0; jb < j1; jb += 32) {
                const int j = jb + lane;
                int u = -1, wt = 0;
                if (j < j1) { u = __ldg(G.adjncy + j); wt = __ldg(G.adjwgt + j); }
                bool act = false;
                int nex = 0, ukey = -1, old = 0;
                int4 r = make_int4(0, 0, -1, 0);
                if (u >= 0) {
                    r = f.rec[u];
                    act = r.z == a || r.z == b;
                    if (act) {
                        const int gk = (r.z == a ? 0 : kFmMaxBuckets) + gmax;
                        old = r.y;
                        r.x += r.z == from ? wt * 1023 : -wt * 1023;   // wt from in to ext, or back
                        nex = fm_ext(r.x);
                        ukey = gk + nex - fm_in(r.x);
                    }
                }
                if (old > 0) {   // u's old entry is dead now
                    f.ent[old - 1].x = -1;
                    if (old > max(ring0, nxt - kFmRing)) ring[(old - 1) & (kFmRing - 1)].x = -1;
                }
                const bool push = act && nex > 0;
                const unsigned pm = __ballot_sync(0xffffffffu, push);
                if (nxt + __popc(pm) > eend) {   // cannot happen: pushes <= boundary + arcs
                    if (lane == 0) fail(w.ctl, E_INTERNAL, 703);
                    bad = true;
                    break;
                }
                const int pos = nxt + __popc(pm & lanemask_lt());
                // lanes pushing onto the same stack: the lower lane's entry goes below
                const unsigned grp = __match_any_sync(0xffffffffu, push ? ukey : -1);   // (its time grows with the distinct values)
                const unsigned lower = grp & lanemask_lt();
                const int pos_lower = __shfl_sync(0xffffffffu, pos, lower ? 31 - __clz(lower) : lane);
                int ubelow = -1;
                if (push) ubelow = lower ? pos_lower : S.top[ukey];
                __syncwarp();
                if (act) {
                    *reinterpret_cast<int2 *>(f.rec + u) = make_int2(r.x, push ? pos + 1 : 0);
                    if (push) {
                        f.ent[pos] = make_int2(u, ubelow);
                        ring[pos & (kFmRing - 1)] = make_int4(u, ubelow, r.w, r.w + fm_deg(r.x));
                        if ((grp & ~lower & ~(1u << lane)) == 0) {   // highest lane of the group
                            S.top[ukey] = pos;
                            S.group[ukey / kFmGroup] = 1;
                        }
                    }
                }
                nxt += __popc(pm);
                hg0 = max(hg0, __reduce_max_sync(0xffffffffu, push && ukey < kFmMaxBuckets ? ukey / kFmGroup : -1));
                hg1 = max(hg1, __reduce_max_sync(0xffffffffu, push ? ukey / kFmGroup - kFmGroups : -1));
                __syncwarp();
                if (lane == 0) *(volatile int *)&S.pushes = nxt - ring0;
            }
            if (bad) break;
            if (lane == 0) *(volatile int *)&S.moves = nm;
            if (s == 0) { wA -= cv; wB += cv; } else { wB -= cv; wA += cv; }   // (its load overlapped the arcs)
            // best state: smallest (overload, cut, max block weight)
            const long long mx = wA > wB ? wA : wB, ov = mx > Lmax ? mx - Lmax : 0;
            over = ov > 0;
            if (ov < bov || (ov == bov && (cut < bcut || (cut == bcut && mx < bmx)))) {
                bcut = cut; bwA = wA; bwB = wB; bov = ov; bmx = mx; best_len = nm; idle = 0;
            } else if (++idle > limit) {
                break;
            }
        }
        if (lane == 0) {
            S.best_len = best_len;
            S.tried = nm;
            S.best_cut = bcut;
            S.best_wA = bwA;
            S.best_wB = bwB;
            *(volatile int *)&S.done = 1;
        }
    }
    __syncthreads();
    mark(T_FM_MOVES);
    const int best_len = S.best_len, nm = S.tried;
    // 4. the moves up to the best prefix
    for (int i = threadIdx.x; i < best_len; i += blockDim.x) {
        const int v = ml[i];
        G.part[v] = G.part[v] == a ? b : a;
    }
    __syncthreads();
    // 5. block weights and boundary candidates of the kept moves (the moved vertex and
    // its neighbours in its old block, as the commit of a flow does)
    if (threadIdx.x == 0) {
        G.blockw[a] = S.best_wA;
        G.blockw[b] = S.best_wB;
        *R = FmRes{cut0, wA0, wB0, S.best_cut, S.best_wA, S.best_wB, best_len, nm};
    }
    if (G.bl) {
        for (int i = threadIdx.x; i < best_len; i += blockDim.x) {
            const int v = ml[i];
            const int ob = G.part[v] == a ? b : a;
            if (!__ldcg(G.inb + v) && atomicExch(G.inb + v, 1) == 0) G.bl[atomicAdd(G.blc, 1)] = v;
            const int j1 = __ldg(G.xadj + v + 1);
            for (int j = __ldg(G.xadj + v); j < j1; ++j) {
                const int x = __ldg(G.adjncy + j);
                if (__ldcg(G.inb + x)) continue;
                if (G.part[x] == ob && atomicExch(G.inb + x, 1) == 0) G.bl[atomicAdd(G.blc, 1)] = x;
            }
        }
    }
    __syncthreads();
    mark(T_FM_FINISH);
}

size_t fm_pair_smem() {
    return sizeof(FmShared) + (8ull + 4 + 4) * kFmSortSmem;
}

static bool g_fm_setup = false;

cudaError_t launch_fm(const Work &w, const FmDev &f, int k, int sms, cudaStream_t st, int *nl) {
    if (!g_fm_setup) {
        cudaError_t e = cudaFuncSetAttribute(fm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)fm_pair_smem());
        if (e != cudaSuccess) return e;
        g_fm_setup = true;
    }
    if (w.npairs <= 0) return cudaSuccess;
    const int grid = 4 * (sms > 0 ? sms : 1);
    fm_count_kernel<<<grid, kFmTPB, 2 * sizeof(int) * (size_t)k, st>>>(w, f);
    fm_offsets_kernel<<<1, 1024, 0, st>>>(w, f);
    fm_gather_kernel<<<grid, kFmTPB, 0, st>>>(w, f);
    fm_pair_kernel<<<w.npairs, kFmTPB, fm_pair_smem(), st>>>(w, f);
    *nl += 4;
    return cudaGetLastError();
}

}  // namespace fr
