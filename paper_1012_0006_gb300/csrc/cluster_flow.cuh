// ClusterFlow: max flow, residual sets and SCCs of one pair inside one thread-block
// cluster, on distributed shared memory (Sanders & Schulz, Section 4.1 and 4.1.1).
// Used by the round's cluster kernel (cluster_flow.cu) and by the queue sweep
// (queue_sweep.cu).
#pragma once

#include <cooperative_groups.h>

#include <climits>

#include "fr_internal.cuh"

namespace fr {

namespace cg = cooperative_groups;

#ifndef FULL
#define FULL 0xffffffffu
#endif

constexpr int kClusterMax = 16;
constexpr int kHdrBytes = 1024;
// A network of up to this many vertices stays in one CTA of its cluster: fewer vertices than
// the CTA has threads are not worth the updates that cross CTAs.  Split, 128 and 384: the pair
// of the 64 x 64 grid 308, 293, 285 us; a V-cycle of rgg3d 1,000,003 vertices, k = 64, 69.1,
// 67.4, 67.0 ms; a W-cycle of rgg3d 65,536, k = 64, 97.3, 93.6, 93.5 ms.
constexpr int kWhole = 384;

struct ClusterHdr {
    int klo[kClusterMax + 1];   // member ranges of the CTAs (identical in every CTA)
    int cab[kClusterMax + 1];   // first arc (pair-local prefix) of each CTA's range
    int cnt[3];                 // rotating counters (CTA 0's copy is the cluster's)
    int err;                    // cluster error (CTA 0's copy)
    int nvcap, nacap;           // common capacities (identical in every CTA)
    int nv, na;                 // this CTA's vertices and arcs
    int counts[kClusterMax];    // scratch for the member scan (CTA 0's copy)
    int counts2[kClusterMax];   // second scratch (byte prefix of the split)
    int kloc[3][kClusterMax + 1];   // candidate splits (by arcs, by bytes, by vertices; CTA 0's copy)
    int cabc[3][kClusterMax + 1];
    int grab[2];                // slot of the size order taken (CTA 0's copy, by parity)
    int nrem;                   // remote arcs of this CTA
    int qn[3];                  // entries of the outgoing queue, rotating
    int wn[2];                  // entries of the worklist, by parity
    int any[3];                 // rotating votes (each CTA's copy holds the cluster's)
    long long flow;
};
static_assert(sizeof(ClusterHdr) <= kHdrBytes, "the header leads the dynamic shared memory");

// Bytes of a vertex and of an arc (packed residuals; 4 more otherwise) in a CTA's shared memory,
// of an arc into another CTA in the remote tables, and the widths of the places of vertices
// and arcs.  A launch asks for no more shared memory than these widths can address, whatever
// the device offers (227 KB on sm_103a).
constexpr int kVtxBytes = 31, kArcBytes = 8, kRemoteBytes = 10;
constexpr int kVtxBits = 13, kArcBits = 15;
constexpr int kClusterSmemMax = 227 * 1024;
static_assert((kClusterSmemMax - kHdrBytes) / kVtxBytes <= 1 << kVtxBits, "a vertex's place");
static_assert((kClusterSmemMax - kHdrBytes) / kArcBytes <= 1 << kArcBits, "an arc's place");
static_assert((kClusterSmemMax - kHdrBytes) / kRemoteBytes <= 1 << 16, "a remote slot in 16 bits");
static_assert(kClusterMax <= 1 << (32 - kVtxBits - kArcBits), "a rank above both places");

// Distributed shared memory by explicit address: a shared::cluster address (32 bits) of an
// element of some CTA's shared memory, and plain loads / relaxed reductions at it.  Every
// CTA carves its arrays at the same offsets, so the address of array X at the same index
// is the address of array Y plus a fixed byte offset.
__device__ __forceinline__ unsigned cta_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned map_rank(unsigned a, int rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ int dsm_ld(unsigned a) {
    int v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void dsm_st(unsigned a, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_add(unsigned a, int v) {
    asm volatile("red.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_min(unsigned a, int v) {
    asm volatile("red.shared::cluster.min.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_max(unsigned a, int v) {
    asm volatile("red.shared::cluster.max.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_or(unsigned a, int v) {
    asm volatile("red.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// An array in the dynamic shared memory, by its byte offset there: the compiler sees that
// every access is to shared memory (through a pointer kept in a struct it may not).
template <class T>
struct ShArr {
    unsigned o;
    __device__ __forceinline__ T *ptr() const {
        extern __shared__ __align__(16) char csmem[];
        return reinterpret_cast<T *>(csmem + o);
    }
    __device__ __forceinline__ T &operator[](int i) const { return ptr()[i]; }
};

template <int N>
struct Int {
    __device__ constexpr int operator()() const { return N; }
};

template <int TPB>
struct ClusterFlow {
    const Work &w;
    cg::cluster_group cl;
    const int rank, C;
    ClusterHdr *hdr;
    ClusterHdr *hdr0;          // CTA 0's header
    static __device__ __forceinline__ ClusterHdr *H() {   // this CTA's
        extern __shared__ __align__(16) char csmem[];
        return reinterpret_cast<ClusterHdr *>(csmem);
    }
    // local arrays
    ShArr<int> lab, ex, fx, cofs, gidx, rfl, cla, res, csum;
    // narrow: every capacity sum csum(a) = c(a) + c(reverse a) is below 2^16, and
    // res[a] holds res(a) | csum(a) << 16 (csum unused); additions to the residual
    // never carry into the upper half because res(a) <= csum(a)
    bool narrow;
    __device__ __forceinline__ int rs(int a) const {
        const int x = *(volatile int *)&res[a];
        return narrow ? (x & 0xFFFF) : x;
    }
    __device__ __forceinline__ int cs(int a) const { return narrow ? (int)((unsigned)res[a] >> 16) : csum[a]; }
    __device__ __forceinline__ void set_rs(int a, int v) { res[a] = narrow ? ((res[a] & ~0xFFFF) | v) : v; }
    // Per arc, one word.  An arc whose head this CTA holds: its rank, the head's index and
    // the index of the reverse arc.  An arc into another CTA: another rank, and a slot of the
    // remote tables, which hold the same three for it (rw), a copy of the head's label (rg)
    // and the slot of the reverse arc in the head's CTA (rslot).  With the residual an arc is
    // 8 bytes, 18 if remote: cluster-wide addresses of both and a copy of every head's label
    // took 16, and the widest pair of a 65,536-vertex 2D rgg (31,456 vertices, 248 K arcs)
    // then fitted no cluster.
    ShArr<unsigned> adr, rw;
    ShArr<int> rg;
    ShArr<unsigned short> rslot;
    ShArr<unsigned short> wl;  // worklist: the vertices a pass or scan works on
    unsigned lab0, res0, rg0, adr0;   // shared::cta addresses of lab, res, rg, adr
    unsigned o_ex, o_rfl, o_cla;      // byte offsets: ex/rfl/cla from lab
    ShArr<unsigned char> bord;
    int rot, arot;             // rotating counter and vote indexes (identical in every CTA)

    static __device__ __forceinline__ unsigned pack_adr(int rk, int v, int a) {
        return ((unsigned)rk << (kVtxBits + kArcBits)) | ((unsigned)v << kArcBits) | (unsigned)a;
    }
    static __device__ __forceinline__ int adr_rank(unsigned w) { return (int)(w >> (kVtxBits + kArcBits)); }
    static __device__ __forceinline__ int adr_vtx(unsigned w) { return (int)(w >> kArcBits) & ((1 << kVtxBits) - 1); }
    static __device__ __forceinline__ int adr_arc(unsigned w) { return (int)(w & ((1u << kArcBits) - 1)); }
    static __device__ __forceinline__ int adr_slot(unsigned w) { return (int)(w & ((1u << (kVtxBits + kArcBits)) - 1)); }
    __device__ __forceinline__ bool local(unsigned w) const { return adr_rank(w) == rank; }
    // of a remote table word: the head in the array `off` bytes after lab, the reverse
    // arc's residual
    __device__ __forceinline__ unsigned head_at(unsigned w, unsigned off = 0) const {
        return map_rank(lab0 + off + 4 * adr_vtx(w), adr_rank(w));
    }
    __device__ __forceinline__ unsigned rev_at(unsigned w) const {
        return map_rank(res0 + 4 * adr_arc(w), adr_rank(w));
    }
    // label of an arc's head: exact in this CTA, the copy elsewhere
    __device__ __forceinline__ int head_label(unsigned w) const {
        return *(volatile int *)(local(w) ? &lab[adr_vtx(w)] : &rg[adr_slot(w)]);
    }

    // Updates of other CTAs' memory go through a queue in shared memory, sent 32 entries an
    // instruction after a block barrier: an instruction that reaches another CTA holds its
    // warp 200-370 cycles, however few lanes take part.  Sent arc by arc as they arise (one
    // in seven, in nearly every instruction) they made up most of the flow's time.  Two
    // halves and three counters rotate, so a barrier before the sending is all it needs; an
    // entry that finds its half full is sent at once.
    enum { Q_PUSH = 0, Q_LABEL = 1, Q_MIN = 2, Q_OR = 3, Q_MAX = 4 };
    static constexpr int kQueue = 512;   // entries of a half
    ShArr<int2> queue;
    int qrot;                            // block barriers passed by the queue (the same in every thread)

    __device__ __forceinline__ void send(int op, int slot, int val) const {
        const unsigned w = rw[slot];
        if (op == Q_PUSH) {
            dsm_add(rev_at(w), val);
            dsm_add(head_at(w, o_ex), val);
        } else if (op == Q_LABEL) {
            dsm_st(map_rank(rg0 + 4 * rslot[slot], adr_rank(w)), val);
        } else if (op == Q_MIN) {
            dsm_min(head_at(w), val);
        } else if (op == Q_OR) {
            dsm_or(head_at(w, o_rfl), val);
        } else {
            dsm_max(head_at(w, o_cla), val);
        }
    }
    __device__ __forceinline__ void enqueue(int op, int slot, int val) {
        const int at = atomicAdd(&H()->qn[qrot % 3], 1);
        if (at < kQueue) queue[(qrot & 1) * kQueue + at] = make_int2(op << 28 | slot, val);
        else send(op, slot, val);
    }
    // Every thread of the CTA: ends a pass or scan, with a block barrier, and sends.
    __device__ __forceinline__ void flush() {
        if (threadIdx.x == 0) H()->qn[(qrot + 1) % 3] = 0;   // (last read before the previous barrier)
        __syncthreads();
        const int n = min(*(volatile int *)&H()->qn[qrot % 3], kQueue);
        for (int i = threadIdx.x; i < n; i += TPB) {
            const int2 q = queue[(qrot & 1) * kQueue + i];
            send((int)((unsigned)q.x >> 28), q.x & 0xfffffff, q.y);
        }
        ++qrot;
    }

    // The vertices of this CTA that pred holds for go on the worklist (one reservation per
    // warp); returns their number, the same in every thread, behind a block barrier.  The
    // work on them is then shared evenly over the warps (each): the vertices with
    // something to do lie together, and the warp that holds most of them made a pass over the
    // CTA's own strips last several times the average.
    int wrot;
    template <class Pred>
    __device__ __forceinline__ int collect(int nv, Pred pred) {
        const int lane = threadIdx.x & 31;
        int *wn = &H()->wn[wrot & 1];
        for (int base = threadIdx.x - lane; base < nv; base += TPB) {
            const int lv = base + lane;
            const bool f = lv < nv && pred(lv);
            const unsigned m = __ballot_sync(FULL, f);
            if (!m) continue;
            int at = 0;
            if (lane == 0) at = atomicAdd(wn, __popc(m));
            at = __shfl_sync(FULL, at, 0);
            if (f) wl[at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)lv;
        }
        __syncthreads();
        const int n = *(volatile int *)wn;
        ++wrot;
        if (threadIdx.x == 0) H()->wn[wrot & 1] = 0;   // (last read before the previous flush's barrier)
        return n;
    }
    // f(u, gl) for every vertex u of the worklist (n of them), G lanes each (gl of G); on
    // all lanes of a warp together, u = -1 where a group has none.
    template <int G, class Fn>
    __device__ __forceinline__ void each(int n, Fn f) {
        const int lane = threadIdx.x & 31;
        for (int b = (int)(threadIdx.x >> 5) * (32 / G); b < n; b += TPB / G) {
            const int i = b + lane / G;
            f(i < n ? (int)wl[i] : -1, lane % G);
        }
    }

    static constexpr int U = 8;   // arcs whose loads are issued together

    // Calls f(word, res, csum) for arcs gl, gl + G, ... of vertex u's row, four at a time with
    // their loads issued together (one arc after the other is a chain of shared
    // memory loads and branches: a relabel of a 3D rgg pair took 80 K cycles so).
    template <int G, class Fn>
    __device__ __forceinline__ void walk(int u, int gl, Fn f) const {
        const int a1 = cofs[u + 1];
        for (int a = cofs[u] + gl; a < a1; a += 4 * G) {
            unsigned w4[4];
            int r[4], c[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int x = a + i * G;
                w4[i] = x < a1 ? adr[x] : 0u;
                const int v = x < a1 ? *(volatile int *)&res[x] : 0;
                r[i] = narrow ? v & 0xFFFF : v;
                c[i] = narrow ? (int)((unsigned)v >> 16) : x < a1 ? csum[x] : 0;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) f(w4[i], r[i], c[i]);   // (past the row: res = csum = 0)
        }
    }

    __device__ ClusterFlow(const Work &w_, char *smem)
        : w(w_), cl(cg::this_cluster()), rank((int)cg::this_cluster().block_rank()),
          C((int)cg::this_cluster().num_blocks()) {
        hdr = reinterpret_cast<ClusterHdr *>(smem);
        hdr0 = cl.map_shared_rank(hdr, 0);
        rot = arot = 0;
        qrot = wrot = 0;
    }

    long long nsync = 0;       // cluster barriers of the current pair (CTA 0, thread 0)

    __device__ void sync() {
        ++nsync;
        cl.sync();
    }

    // True if x holds for any thread of the cluster: a block vote, then one instruction sets
    // every CTA's copy, so that after the one cluster barrier each reads its own.  (A copy's
    // next slot was last read before the previous barrier, so its CTA may clear it now.)
    __device__ bool cluster_any(bool x) {
        const int s = __syncthreads_or(x);
        if (s && threadIdx.x < C) dsm_or(map_rank(cta_addr(&H()->any[arot]), (int)threadIdx.x), 1);
        if (threadIdx.x == 0) H()->any[(arot + 1) % 3] = 0;
        sync();
        const bool r = *(volatile int *)&H()->any[arot] != 0;
        arot = (arot + 1) % 3;
        return r;
    }

    // Cluster-wide sum of x (one value per thread); every thread gets the total.
    // Each warp adds its sum straight into CTA 0's counter, so one cluster barrier
    // is the only synchronisation.  The counters rotate over three slots: slot
    // rot + 1 was last read before the previous barrier, so CTA 0 may clear it now.
    __device__ int cluster_sum(int x) { return cluster_reduce(x, false); }
    // cluster-wide maximum of non-negative x
    __device__ int cluster_max(int x) { return cluster_reduce(x, true); }

    __device__ int cluster_reduce(int x, bool is_max) {
        x = is_max ? (int)__reduce_max_sync(FULL, (unsigned)x) : (int)__reduce_add_sync(FULL, (unsigned)x);
        int *c = &hdr0->cnt[rot];
        if ((threadIdx.x & 31) == 0 && x) {
            if (is_max) atomicMax(c, x); else atomicAdd(c, x);
        }
        if (rank == 0 && threadIdx.x == 0) H()->cnt[(rot + 1) % 3] = 0;
        sync();
        const int tot = *(volatile int *)c;
        rot = (rot + 1) % 3;
        return tot;
    }

    int nrcap;                 // remote arcs the tables have room for (the same in every CTA)
    __device__ void carve(size_t smem_bytes, int nvcap, int nacap, bool narrow_) {
        narrow = narrow_;
        unsigned p = kHdrBytes;
        auto take = [&](unsigned bytes) {
            const unsigned r = p;
            p += (bytes + 15) / 16 * 16;
            return r;
        };
        lab.o = take(4u * nvcap);
        ex.o = take(4u * nvcap);
        fx.o = take(4u * nvcap);
        cofs.o = take(4u * (nvcap + 1));
        gidx.o = take(4u * nvcap);
        rfl.o = take(4u * nvcap);
        cla.o = take(4u * nvcap);
        bord.o = take(nvcap);
        wl.o = take(2u * nvcap);
        adr.o = take(4u * nacap);
        res.o = take(4u * nacap);
        csum.o = narrow ? 0u : take(4u * nacap);
        queue.o = take(2 * kQueue * sizeof(int2));
        // the rest: the remote tables
        nrcap = (int)(smem_bytes - p - 48) / kRemoteBytes;
        rw.o = take(4u * nrcap);
        rg.o = take(4u * nrcap);
        rslot.o = p;
        lab0 = cta_addr(lab.ptr());
        res0 = cta_addr(res.ptr());
        rg0 = cta_addr(rg.ptr());
        adr0 = cta_addr(adr.ptr());
        o_ex = ex.o - lab.o;
        o_rfl = rfl.o - lab.o;
        o_cla = cla.o - lab.o;
    }

    // (4 bytes a vertex more than carve takes: what is left is room for the remote tables)
    static __host__ __device__ size_t bytes_for(int nvcap, int nacap, bool narrow) {
        auto a = [](size_t b) { return (b + 15) / 16 * 16; };
        return kHdrBytes + 7 * a(4ull * nvcap) + a(4ull * (nvcap + 1)) + a(nvcap) + a(2ull * nvcap) + (narrow ? 2 : 3) * a(4ull * nacap) +
               2 * kQueue * sizeof(int2) + 64;
    }

    __device__ int owner(int k) const {   // CTA whose range holds member k
        int r = 0;
        while (r + 1 < C && H()->klo[r + 1] <= k) ++r;
        return r;
    }

    // ------------------------------------------------------------ one pair --
    // Returns false when the pair does not fit (left to the grid-wide path).
    // adds the time since t to timer slot idx (one thread per cluster; sums over clusters)
    __device__ bool mark(unsigned long long &t, int idx) {
        const unsigned long long now = globaltimer();
        if (rank == 0 && threadIdx.x == 0) atomicAddLL(&w.ctl->timers[idx], (long long)(now - t));
        t = now;
        return true;
    }

    __device__ bool solve(int p, char *smem, size_t smem_bytes) {
        unsigned long long t_in = globaltimer();
        nsync = 0;
        const int nu = __ldcg(&w.ctl->nu);
        const int V = __ldcg(&w.pacc[p].nc), A = __ldcg(&w.pacc[p].m);
        if (V == 0) return true;
        // members of pair p in local-id order: pmem = cid, their arc prefix = outoff, plocal = color
        int pbase = 0;
        for (int q = 0; q < p; ++q) pbase += __ldcg(&w.pacc[q].nc);
        int *pmem = w.cid + pbase, *pacs = w.outoff + pbase, *plocal = w.color;
        {
            // every warp takes a contiguous chunk of the CTA's share of the union and
            // reads it 32 entries at a time (coalesced), counting and then placing the
            // pair's members with ballots; one block scan over the warps' counts and one
            // cluster prefix give the positions, so the list stays in local-id order
            const long long per = (nu + C - 1) / C;
            const long long c0 = per * rank, c1 = min((long long)nu, c0 + per);
            const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
            const long long wper = ((max(0LL, c1 - c0) + TPB / 32 - 1) / (TPB / 32) + 31) / 32 * 32;
            const long long w0 = min(c1, c0 + wper * wid), w1 = min(c1, w0 + wper);
            int mine = 0;
            for (long long b = w0; b < w1; b += 32) {
                const long long i = b + lane;
                mine += __popc(__ballot_sync(FULL, i < w1 && (__ldcg(&w.sid[i]) >> 1) == p));
            }
            int tot;
            const int ex0 = block_exclusive_scan<TPB>(lane == 0 ? mine : 0, &tot);
            if (threadIdx.x == 0) hdr0->counts[rank] = tot;
            sync();
            int pos = __shfl_sync(FULL, ex0, 0);
            for (int r = 0; r < rank; ++r) pos += *(volatile int *)&hdr0->counts[r];
            sync();   // counts read before they are reused
            for (long long b = w0; b < w1; b += 32) {
                const long long i = b + lane;
                const bool m = i < w1 && (__ldcg(&w.sid[i]) >> 1) == p;
                const unsigned bal = __ballot_sync(FULL, m);
                if (m) {
                    const int at = pos + __popc(bal & ((1u << lane) - 1u));
                    pmem[at] = (int)i;
                    plocal[i] = at;
                }
                pos += __popc(bal);
            }
        }
        __threadfence();
        sync();
        // arc and shared-memory byte prefixes over members (each CTA a slice of the
        // member list, each thread a contiguous part of it), and three candidate splits
        // into C contiguous ranges: equal arcs (the work of the flow), equal bytes (31
        // per vertex, 8 or 12 per arc) and equal vertices.  Every CTA carves its arrays
        // for the largest range's vertices and arcs, so the first candidate that fits
        // shared memory is taken: the arc split where it fits, the others where the
        // order of the vertices puts many light vertices together.
        const int ab = w.narrow ? kArcBytes : kArcBytes + 4;
        {
            const long long Btot = (long long)kVtxBytes * V + (long long)ab * A;
            const long long tot3[3] = {(long long)A, Btot, (long long)V};
            const int per = (V + C - 1) / C;
            const int k0 = min(V, per * rank), k1 = min(V, k0 + per);
            const int tper = (k1 - k0 + TPB - 1) / TPB;
            const int s0 = min(k1, k0 + tper * (int)threadIdx.x), s1 = min(k1, s0 + tper);
            int mine = 0;
            for (int k = s0; k < s1; ++k) {
                const int i = __ldcg(&pmem[k]);
                mine += w.off[i + 1] - w.off[i];
            }
            int tot, btot;
            const int e0 = block_exclusive_scan<TPB>(mine, &tot);
            const int b0 = block_exclusive_scan<TPB>(kVtxBytes * (s1 - s0) + ab * mine, &btot);
            if (threadIdx.x == 0) {
                hdr0->counts[rank] = tot;
                hdr0->counts2[rank] = btot;
            }
            sync();
            int run = e0;
            long long brun = b0;
            for (int r = 0; r < rank; ++r) {
                run += *(volatile int *)&hdr0->counts[r];
                brun += *(volatile int *)&hdr0->counts2[r];
            }
            sync();
            // split points of candidate c: kloc[c][r] = the first member whose prefix
            // reaches tot3[c] * r / C, so the member whose share (prefix, prefix + size]
            // holds that target is the one before it; its thread writes the split and
            // the range's first arc into CTA 0
            if (rank == 0 && threadIdx.x == 0) {
                for (int c = 0; c < 3; ++c) {
                    H()->kloc[c][0] = 0;
                    H()->cabc[c][0] = 0;
                    H()->kloc[c][C] = V;
                    H()->cabc[c][C] = A;
                    for (int r = 1; r < C; ++r)
                        if (tot3[c] * r / C <= 0) { H()->kloc[c][r] = 0; H()->cabc[c][r] = 0; }
                }
            }
            for (int k = s0; k < s1; ++k) {
                const int i = __ldcg(&pmem[k]);
                const int d = w.off[i + 1] - w.off[i];
                const int b = kVtxBytes + ab * d;
                pacs[k] = run;
                const long long lo3[3] = {(long long)run, brun, (long long)k};
                const long long sz3[3] = {(long long)d, (long long)b, 1};
                for (int c = 0; c < 3; ++c)
                    for (int r = 1; r < C; ++r) {
                        const long long target = tot3[c] * r / C;
                        if (target > lo3[c] && target <= lo3[c] + sz3[c]) {
                            hdr0->kloc[c][r] = k + 1;
                            hdr0->cabc[c][r] = run + d;
                        }
                    }
                run += d;
                brun += b;
            }
        }
        __threadfence();
        sync();
        if (rank == 0 && threadIdx.x == 0) {
            int pick = 0;
            for (int c = 0; c < 3; ++c) {
                int nvc = 0, nac = 0;
                for (int r = 0; r < C; ++r) {
                    nvc = max(nvc, H()->kloc[c][r + 1] - H()->kloc[c][r]);
                    nac = max(nac, H()->cabc[c][r + 1] - H()->cabc[c][r]);
                }
                pick = c;
                if (bytes_for(nvc, nac, w.narrow != 0) <= smem_bytes) break;
            }
            const bool whole = V <= kWhole && bytes_for(V, A, w.narrow != 0) <= smem_bytes;
            for (int r = 0; r <= C; ++r) {
                H()->klo[r] = whole && r > 0 ? V : H()->kloc[pick][r];
                H()->cab[r] = whole && r > 0 ? A : H()->cabc[pick][r];
            }
        }
        sync();
        // the C ranges, copied from CTA 0 (same in every CTA)
        if (threadIdx.x <= C && rank != 0) {
            H()->klo[threadIdx.x] = *(volatile int *)&hdr0->klo[threadIdx.x];
            H()->cab[threadIdx.x] = *(volatile int *)&hdr0->cab[threadIdx.x];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int nvcap = 0, nacap = 0;
            for (int r = 0; r < C; ++r) {
                nvcap = max(nvcap, H()->klo[r + 1] - H()->klo[r]);
                nacap = max(nacap, H()->cab[r + 1] - H()->cab[r]);
            }
            H()->nvcap = nvcap;
            H()->nacap = nacap;
        }
        __syncthreads();
        const int nvcap = H()->nvcap, nacap = H()->nacap;
        const bool nar = w.narrow != 0;
        unsigned long long t1 = t_in;
        mark(t1, T_CL_MEMBERS);
        if (bytes_for(nvcap, nacap, nar) > smem_bytes) return false;   // same decision in every CTA
        carve(smem_bytes, nvcap, nacap, nar);
        if (threadIdx.x == 0) {
            H()->nrem = 0;
            H()->qn[0] = H()->qn[1] = H()->qn[2] = 0;
            H()->any[0] = H()->any[1] = H()->any[2] = 0;
            H()->wn[0] = H()->wn[1] = 0;
        }
        qrot = wrot = 0;
        __syncthreads();
        const int klo = H()->klo[rank], khi = H()->klo[rank + 1];
        const int nv = khi - klo;
        const int abase = H()->cab[rank];
        // load this CTA's vertices and arcs
        for (int lv = threadIdx.x; lv < nv; lv += TPB) {
            const int i = __ldcg(&pmem[klo + lv]);
            gidx[lv] = i;
            ex[lv] = (int)__ldcg(&w.ex[i]);
            fx[lv] = __ldcg(&w.fx[i]);
            bord[lv] = w.border[i];
            const int a0 = __ldcg(&pacs[klo + lv]) - abase;
            cofs[lv] = a0;
            const int j0 = w.off[i], j1 = w.off[i + 1];
            // four arcs at a time, their loads issued together (each arc is a chain
            // head -> head's member index -> its arc prefix)
            for (int jb = j0; jb < j1; jb += 4) {
                int h[4], rv[4], r0[4], cj[4], kh[4], oh[4], cr[4], ph[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = min(jb + u, j1 - 1);
                    h[u] = w.head[j];
                    rv[u] = w.rev[j];
                    r0[u] = __ldcg(&w.res[j]);
                    cj[u] = w.cap[j];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    kh[u] = __ldcg(&plocal[h[u]]);
                    oh[u] = w.off[h[u]];
                    cr[u] = w.cap[rv[u]];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) ph[u] = __ldcg(&pacs[kh[u]]);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (jb + u >= j1) break;
                    const int la = a0 + (jb + u - j0);
                    const int rh = owner(kh[u]);
                    const unsigned wd = pack_adr(rh, kh[u] - H()->klo[rh], ph[u] - H()->cab[rh] + (rv[u] - oh[u]));
                    if (rh == rank) {
                        adr[la] = wd;
                    } else {
                        const int sl = atomicAdd(&H()->nrem, 1);
                        adr[la] = pack_adr((rank + 1) & (kClusterMax - 1), 0, 0) | (unsigned)sl;
                        if (sl < nrcap) rw[sl] = wd;
                    }
                    const int c0 = cj[u] + cr[u];   // res(a) + res(reverse of a), fixed
                    if (nar) {
                        res[la] = r0[u] | (c0 << 16);
                    } else {
                        res[la] = r0[u];
                        csum[la] = c0;
                    }
                }
            }
        }
        if (threadIdx.x == 0) {
            H()->nv = nv;
            const int a1 = khi < V ? __ldcg(&pacs[khi]) : A;
            cofs[nv] = a1 - abase;
            H()->na = a1 - abase;
            if (rank == 0) { H()->cnt[0] = H()->cnt[1] = H()->cnt[2] = 0; H()->err = 0; }
        }
        rot = arot = 0;
        sync();
        const int nrem = H()->nrem;
        if (cluster_any(nrem > nrcap)) return false;   // no room for the remote tables
        if (threadIdx.x == 0 && nrem) atomicAddLL(&w.ctl->cl_remote, (long long)nrem);
        for (int i = threadIdx.x; i < nrem; i += TPB)
            rslot[i] = (unsigned short)adr_slot((unsigned)dsm_ld(map_rank(adr0 + 4 * adr_arc(rw[i]), adr_rank(rw[i]))));
        sync();   // (no CTA sends into another's tables before it has read its slots)
        const int hmax = V + 2;
        mark(t1, T_CL_LOAD);
        // a maximum preflow is enough for the cut (see the grid-wide maxflow); the
        // excess goes back to s only when the flow itself is handed out
        // The pulse phase stops when no excess can move by its labels; whether the
        // preflow is maximum is then read off the residual sets: no vertex reached
        // from s -- the s-border or one holding excess -- may reach t.  If one does
        // (lagging label copies), the phase resumes from exact labels.
        bool ok = true;
        for (int attempt = 0;; ++attempt) {
            ok = w.flow_sched == 1 ? phase_wave(0, nv, hmax, 0)
                                   : phase_pulse(0, nv, hmax, false, w.wave_votes != nullptr && attempt == 0);
            mark(t1, T_CL_FLOW);
            if (ok && w.full_flow) ok = w.flow_sched == 1 ? phase_wave(1, nv, hmax, 0) : phase_pulse(1, nv, hmax, true, false);
            mark(t1, T_CL_RETURN);
            if (!ok) break;
            reach(nv);
            mark(t1, T_CL_REACH);
            int open = 0;
            for (int lv = threadIdx.x; lv < nv; lv += TPB) open += rfl[lv] == 3;
            if (!cluster_any(open)) break;
            if (attempt >= 16) {   // the same count in every CTA
                if (rank == 0 && threadIdx.x == 0) fail(w.ctl, E_INTERNAL, 304);
                break;
            }
        }
        if (!ok) {
            // cap reached: report, leave the pair's arrays as they were
            if (rank == 0 && threadIdx.x == 0) fail(w.ctl, E_ITER, 300);
            sync();
            return true;
        }
        // write back: residuals, s/t flows, zero excess, reachability and plain sides
        for (int lv = threadIdx.x; lv < nv; lv += TPB) {
            const int i = gidx[lv];
            const int j0 = w.off[i];
            const int a0 = cofs[lv], a1 = cofs[lv + 1];
            for (int a = a0; a < a1; ++a) w.res[j0 + (a - a0)] = rs(a);
            w.fx[i] = fx[lv];
            w.ex[i] = ex[lv];
            w.rflag[i] = rfl[lv];
            w.side_out[i] = (rfl[lv] & 1) ? 0 : 1;
            if (w.full_flow && ex[lv] != 0) fail(w.ctl, E_INTERNAL, 301);
            if (rfl[lv] == 3) fail(w.ctl, E_INTERNAL, 302);
        }
        sync();
        // most balanced cut: SCCs of the residual graph on the vertices reached from
        // neither s nor t (lab, ex, fx are free now)
        const ShArr<int> sc = fx;
        if (w.pairs[p].mb) {
            scc_local(nv, V, sc);
        } else {
            for (int lv = threadIdx.x; lv < nv; lv += TPB) sc[lv] = -2;
        }
        for (int lv = threadIdx.x; lv < nv; lv += TPB) w.scc[gidx[lv]] = sc[lv];
        mark(t1, T_CL_SCC);
        sync();
        if (rank == 0 && threadIdx.x == 0) atomicAddLL(&w.ctl->cl_syncs, nsync);
        return true;
    }

    // SCCs of the residual graph on X = the vertices with rfl == 0, labelled by
    // their smallest union id (the same labels as the grid-wide colouring): in
    // rounds, every unassigned vertex takes the smallest union id that reaches it
    // over unassigned vertices (colour; label correction pushed along residual arcs
    // with an atomic min), a vertex whose colour is its own id is a root, and the
    // vertices of its colour that reach it join it: members claim the tails of
    // their residual in-arcs with an atomic max of their colour, and a vertex
    // joins when the largest claim it received is its own colour (claims from
    // other classes are smaller: whatever reaches a vertex reaches its
    // successors).  sc: -2 outside X, else the root's union id.
    // V, the pair's vertex count, bounds the rounds: the same bound in every CTA, so
    // that every CTA leaves the loop after the same barrier.
    __device__ void scc_local(int nv, int V, const ShArr<int> sc) {
        const ShArr<int> col = lab, done = ex;
        for (int lv = threadIdx.x; lv < nv; lv += TPB) sc[lv] = rfl[lv] == 0 ? -1 : -2;
        sync();
        long long rounds = 0;
        for (;;) {
            int rem = 0;
            for (int lv = threadIdx.x; lv < nv; lv += TPB) {
                const bool un = sc[lv] == -1;
                col[lv] = un ? gidx[lv] : INT_MAX;
                done[lv] = un ? INT_MAX : 0;   // colour last passed on
                cla[lv] = -1;
                rem += un;
            }
            if (!cluster_any(rem)) break;
            if (++rounds > (long long)V + 1) {
                if (rank == 0 && threadIdx.x == 0) fail(w.ctl, E_ITER, 303);
                break;
            }
            // colours
            for (;;) {
                bool any = false;
                for (int k = 0; k < kScans; ++k) {
                    const int n = collect(nv, [&](int lv) {
                        return sc[lv] == -1 && *(volatile int *)&col[lv] < done[lv];
                    });
                    if (n == 0) break;
                    any = true;
                    each<4>(n, [&](int u, int gl) {
                        // (one value for the vertex's lanes: it may drop meanwhile)
                        const int cu = __shfl_sync(FULL, u >= 0 ? *(volatile int *)&col[u] : 0, 0, 4);
                        if (u < 0) return;
                        if (gl == 0) done[u] = cu;
                        walk<4>(u, gl, [&](unsigned wd, int r, int) {
                            if (r <= 0) return;
                            if (local(wd)) atomicMin(&col[adr_vtx(wd)], cu);
                            else enqueue(Q_MIN, adr_slot(wd), cu);   // (col is lab)
                        });
                    });
                    flush();
                }
                if (!cluster_any(any)) break;
            }
            // roots, then members claim the vertices of their colour that reach them
            for (int lv = threadIdx.x; lv < nv; lv += TPB) {
                done[lv] = sc[lv] == -1 ? 0 : 1;   // 1: nothing to pass on
                if (sc[lv] == -1 && col[lv] == gidx[lv]) sc[lv] = gidx[lv];
            }
            sync();
            for (;;) {
                bool any = false;
                for (int k = 0; k < kScans; ++k) {
                    const int n = collect(nv, [&](int lv) {
                        return !done[lv] && (sc[lv] >= 0 || *(volatile int *)&cla[lv] == col[lv]);
                    });
                    if (n == 0) break;
                    any = true;
                    each<4>(n, [&](int u, int gl) {
                        if (u < 0) return;
                        const int su = sc[u] >= 0 ? sc[u] : col[u];   // (the same before and after the next line)
                        if (gl == 0) {
                            sc[u] = su;
                            done[u] = 1;
                        }
                        walk<4>(u, gl, [&](unsigned wd, int r, int c) {
                            if (c <= r) return;
                            if (local(wd)) atomicMax(&cla[adr_vtx(wd)], su);
                            else enqueue(Q_MAX, adr_slot(wd), su);
                        });
                    });
                    flush();
                }
                if (!cluster_any(any)) break;
            }
        }
        if (rank == 0 && threadIdx.x == 0) atomicAdd(&w.ctl->scc_rounds, (int)rounds);
    }

    static constexpr int kScans = 8;   // local scans between cluster barriers, at most (relabel, reach, SCCs)
    static constexpr int kMaxSweeps = 1024;   // sweeps of one wave (a bound; a wave ends when one moves nothing)
    static constexpr int kMaxLocalRounds = 4096;   // local rounds of one sweep (a bound)

    // Exact labels: distances over residual arcs to the level-1 vertices, found by
    // label correction pushed outward.  A vertex whose label dropped since it last
    // passed it on lowers the label of each v with a residual arc v -> u to its own
    // + 1 (an atomic min into v's CTA; the residual of v -> u is csum - res of
    // u -> v).  Every CTA rescans its own
    // vertices kScans times between cluster barriers, without waiting for the
    // others; a barrier window in which no CTA had a vertex to pass on ends it
    // (every update sent before the window's barrier was seen in it), and the
    // fixed point is the breadth-first distance.  rfl, free during the flow, holds
    // the label each vertex last passed on.  phase 0: distance to t; phase 1:
    // distance to s.  Returns the highest label below hmax if want_top.
    __device__ int relabel(int ph, int nv, int hmax, bool want_top = false) {
        const unsigned long long t_rel = globaltimer();
        for (int lv = threadIdx.x; lv < nv; lv += TPB) {
            const bool src = ph ? (bord[lv] == 1 && fx[lv] > 0) : (bord[lv] == 2);
            lab[lv] = src ? 1 : hmax;
            rfl[lv] = hmax;
        }
        sync();
        long long arcs = 0;   // arcs this thread's vertices passed their labels along
        const int lane = threadIdx.x & 31;
        for (;;) {
            bool any = false;
            for (int k = 0; k < kScans; ++k) {
                const int n = collect(nv, [&](int lv) { return *(volatile int *)&lab[lv] < rfl[lv]; });
                if (n == 0) break;
                any = true;
                auto pass_on = [&](auto G, int u, int gl) {
                    // (one value for the vertex's lanes: it may drop meanwhile)
                    const int Lu = __shfl_sync(FULL, u >= 0 ? *(volatile int *)&lab[u] : 0, 0, G());
                    if (u < 0) return;
                    if (gl == 0) {
                        rfl[u] = Lu;
                        arcs += cofs[u + 1] - cofs[u];
                    }
                    walk<G()>(u, gl, [&](unsigned wd, int r, int c) {
                        if (c <= r) return;
                        if (local(wd)) atomicMin(&lab[adr_vtx(wd)], Lu + 1);
                        else enqueue(Q_MIN, adr_slot(wd), Lu + 1);
                    });
                };
                if (n <= TPB / 8) each<8>(n, [&](int u, int gl) { pass_on(Int<8>(), u, gl); });
                else each<4>(n, [&](int u, int gl) { pass_on(Int<4>(), u, gl); });
                flush();
            }
            if (!cluster_any(any)) break;
        }
        for (int o = 16; o > 0; o >>= 1) arcs += __shfl_xor_sync(FULL, arcs, o);
        if (lane == 0 && arcs) atomicAddLL(&w.ctl->gr_arcs, arcs);
        // the copies of remote labels (the barrier: none is read after its owner lifts it)
        const int nrem = H()->nrem;
        for (int i = threadIdx.x; i < nrem; i += TPB) rg[i] = dsm_ld(head_at(rw[i]));
        sync();
        int top = 0;
        if (want_top) {
            top = 1;
            for (int lv = threadIdx.x; lv < nv; lv += TPB)
                if (lab[lv] < hmax && lab[lv] > top) top = lab[lv];
            top = cluster_max(top);
        }
        if (rank == 0 && threadIdx.x == 0) atomicAddLL(&w.ctl->timers[T_CL_RELABEL], (long long)(globaltimer() - t_rel));
        return top;
    }

    // d along an arc in a wave: its reverse residual and its head's excess grow
    __device__ __forceinline__ void give(unsigned wd, int d) {
        if (local(wd)) {
            atomicAdd(&res[adr_arc(wd)], d);
            atomicAdd(&ex[adr_vtx(wd)], d);
        } else {
            send(Q_PUSH, adr_slot(wd), d);
        }
    }

    // One level-synchronous wave (the waves before the pulses): the levels from the
    // top down, each level pushing only along admissible arcs into the level below
    // (level 1 into the target), one cluster barrier per level.  Within a level step
    // a vertex is the only writer of its own excess and of the residuals of its arcs
    // and their reverses, so only the excess of the receiving vertex needs an atomic.
    __device__ void wave_levels_sync(int ph, int nv, int top) {
        for (int L = top; L >= 1; --L) {
            for (int lv = threadIdx.x; lv < nv; lv += TPB) {
                if (lab[lv] != L) continue;
                int e = ex[lv];
                if (e <= 0) continue;
                if (L == 1) {
                    if (!ph) { fx[lv] += e; e = 0; }
                    else if (bord[lv] == 1) { const int d = e < fx[lv] ? e : fx[lv]; fx[lv] -= d; e -= d; }
                } else {
                    const int a1 = cofs[lv + 1];
                    for (int a = cofs[lv]; a < a1 && e > 0; a += U) {
                        int r[U], l[U];
                        unsigned hr[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            r[u] = a + u < a1 ? rs(a + u) : 0;
                            hr[u] = a + u < a1 ? adr[a + u] : 0u;
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) l[u] = r[u] > 0 ? head_label(hr[u]) : -1;
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            if (e > 0 && l[u] == L - 1) {
                                const int d = e < r[u] ? e : r[u];
                                set_rs(a + u, r[u] - d);
                                give(hr[u], d);
                                e -= d;
                            }
                        }
                    }
                }
                ex[lv] = e;
            }
            sync();
        }
    }

    // One wave with fixed labels (the waves schedule).  Every vertex holding excess
    // at a level L in [1, top] pushes along its admissible arcs into level L - 1
    // (level 1 into the target).  Each CTA repeats local rounds -- one pass over its vertices, then a
    // CTA barrier -- while a push lands on one of its own vertices; excess sent to
    // another CTA lands there as an atomic addition whenever it lands.  One cluster
    // barrier then ends a sweep, and sweeps repeat until one moves nothing: no
    // excess has an admissible arc with residual capacity any more, and only new
    // labels can move it.  With labels fixed, no two vertices push along an arc and
    // its reverse at once (one of the two pushes would go uphill), so the owner of
    // an arc is the only writer of its residual besides the atomic additions of
    // pushes along the reverse, and every change of an excess is atomic (a vertex
    // pushes at most what it read; others only add).  Every push lowers the sum of
    // excess times label, so the rounds and the sweeps end.
    __device__ void wave_levels(int ph, int nv, int top) {
        for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
            int moved = 0;
            for (int round = 0; round < kMaxLocalRounds; ++round) {
                int landed = 0;
                for (int lv = threadIdx.x; lv < nv; lv += TPB) {
                    const int L = lab[lv];
                    if (L < 1 || L > top) continue;
                    int e = *(volatile int *)&ex[lv];
                    if (e <= 0) continue;
                    int sent = 0;
                    if (L == 1) {
                        if (!ph) { sent = e; fx[lv] += e; }
                        else if (bord[lv] == 1) { sent = e < fx[lv] ? e : fx[lv]; fx[lv] -= sent; }
                    } else {
                        const int a1 = cofs[lv + 1];
                        for (int a = cofs[lv]; a < a1 && e > 0; a += U) {
                            int r[U], l[U];
                            unsigned hr[U];
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                r[u] = a + u < a1 ? rs(a + u) : 0;
                                hr[u] = a + u < a1 ? adr[a + u] : 0u;
                            }
#pragma unroll
                            for (int u = 0; u < U; ++u) l[u] = r[u] > 0 ? head_label(hr[u]) : -1;
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                if (e > 0 && l[u] == L - 1) {
                                    const int d = e < r[u] ? e : r[u];
                                    set_rs(a + u, r[u] - d);
                                    give(hr[u], d);
                                    e -= d;
                                    sent += d;
                                    landed |= local(hr[u]);
                                }
                            }
                        }
                    }
                    if (sent) {
                        atomicSub(&ex[lv], sent);
                        ++moved;
                    }
                }
                if (!__syncthreads_or(landed)) break;
            }
            if (!cluster_any(moved)) break;
        }
    }

    // Push-relabel in waves: exact labels, then one wave; repeat until no vertex
    // with excess can reach the target.  Phase 0 sends excess to t, phase 1 returns
    // what is left to s.
    // (done: waves before this call)
    __device__ bool phase_wave(int ph, int nv, int hmax, long long done) {
        long long waves = done;
        for (;;) {
            const int top = relabel(ph, nv, hmax, true);
            int act = 0;
            for (int lv = threadIdx.x; lv < nv; lv += TPB) act += ex[lv] > 0 && lab[lv] < hmax;
            if (!cluster_any(act)) break;
            if (++waves > w.pulse_cap) return false;
            wave_levels(ph, nv, top);
        }
        if (rank == 0 && threadIdx.x == 0) {
            atomicAddLL(&w.ctl->pulses, waves);
            atomicAddLL(&w.ctl->relabels, waves + 1);   // (each wave starts from one, and the last finds nothing)
        }
        return true;
    }

    // One vertex holding excess, G lanes: lift it just above its lowest residual neighbour if
    // it is not, push along the arc to that neighbour, up to `iters` times or until the excess
    // is gone.  Copies of remote labels may lag; they never run ahead of the label, and
    // labels only rise between exact relabels, so a lagging copy only makes a push look
    // admissible that is not -- capacities and excesses stay exact, and a phase ends only once
    // exact labels (phase 1) or the residual sets (phase 0) show that no excess can still
    // reach its target.  Returns (on the vertices' first lanes) whether the vertex pushed along
    // an arc or still holds excess that may move.  All lanes of a warp call it (u < 0: none).
    // The passes are bound by the instructions of a visit (four warps a scheduler, each some
    // hundreds): pushing along all arcs to the lowest label at once, their shares by a prefix
    // sum, took three times as many an iteration.
    template <int G>
    __device__ __forceinline__ bool discharge(int ph, int u, int gl, int hmax, int iters) {
        int e = 0, f = 0, h = hmax, sent = 0, a0 = 0, deg = 0;
        bool border = false, pushed = false;
        if (u >= 0) {
            e = *(volatile int *)&ex[u];
            f = fx[u];
            h = lab[u];
            a0 = cofs[u];
            deg = cofs[u + 1] - a0;
            border = bord[u] == (ph ? 1 : 2);
        }
        e = __shfl_sync(FULL, e, 0, G);   // (it may grow meanwhile)
        __syncwarp();
        if (border) {   // the arc to the target
            sent = ph ? min(e, f) : e;
            if (gl == 0) fx[u] = ph ? f - sent : f + sent;
            e -= sent;
        }
        const int longest = (int)__reduce_max_sync(FULL, (unsigned)(e > 0 ? deg : 0));
        if (longest <= 16) discharge_row<G, 16 / G>(a0, deg, u, gl, hmax, iters, h, e, sent, pushed);
        else if (longest <= 32) discharge_row<G, 32 / G>(a0, deg, u, gl, hmax, iters, h, e, sent, pushed);
        else discharge_long<G>(a0, deg, u, gl, hmax, iters, h, e, sent, pushed);
        if (gl != 0 || u < 0) return false;
        if (sent) atomicSub(&ex[u], sent);
        return pushed || (e > 0 && h < hmax);
    }

    // the lowest of a vertex's G lanes
    template <int G>
    __device__ __forceinline__ int lowest(int x) const {
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1) x = min(x, __shfl_xor_sync(FULL, x, d));
        return x;
    }
    __device__ __forceinline__ void push_arc(int a, unsigned wd, int d) {
        atomicSub(&res[a], d);
        if (local(wd)) {
            atomicAdd(&res[adr_arc(wd)], d);
            atomicAdd(&ex[adr_vtx(wd)], d);
        } else {
            enqueue(Q_PUSH, adr_slot(wd), d);
        }
    }
    __device__ __forceinline__ void publish(int a0, int na, int gl, int G, int h) {
#pragma unroll 1
        for (int a = gl; a < na; a += G) {
            const unsigned wd = adr[a0 + a];
            if (!local(wd)) enqueue(Q_LABEL, adr_slot(wd), h);
        }
    }

    // rows of up to G R <= 32 arcs: the lanes keep label << 5 | place for their residual arcs
    template <int G, int R>
    __device__ __forceinline__ void discharge_row(int a0, int deg, int u, int gl, int hmax, int iters, int &h, int &e,
                                                  int &sent, bool &pushed) {
        int key[R];
        unsigned wd[R];
        const int h0 = h, na = e > 0 ? deg : 0;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const bool v = gl + G * i < na;
            wd[i] = v ? adr[a0 + gl + G * i] : 0u;
            key[i] = v ? rs(a0 + gl + G * i) : 0;
        }
#pragma unroll
        for (int i = 0; i < R; ++i) key[i] = key[i] > 0 ? head_label(wd[i]) << 5 | (gl + G * i) : INT_MAX;
        for (int it = 0; it < iters; ++it) {
            const bool go = e > 0 && h < hmax;
            if (!__any_sync(FULL, go)) break;
            int k = INT_MAX;
#pragma unroll
            for (int i = 0; i < R; ++i) k = min(k, key[i]);
            k = lowest<G>(k);
            const int hm = k >> 5, at = k & 31;
            if (go && h <= hm) h = hm >= hmax - 1 ? hmax : hm + 1;
            const bool push = go && h < hmax;
            int d = 0, r = 0;
            if (push) {
                r = rs(a0 + at);
                d = min(e, r);
            }
            d = __shfl_sync(FULL, d, 0, G);   // (a residual may grow meanwhile)
            if (push) {
                if (gl == 0) push_arc(a0 + at, adr[a0 + at], d);
#pragma unroll
                for (int i = 0; i < R; ++i) key[i] = key[i] == k && d < e ? INT_MAX : key[i];   // saturated
                pushed = true;
                sent += d;
                e -= d;
            }
        }
        if (h != h0) {
            if (gl == 0) lab[u] = h;
            publish(a0, na, gl, G, h);
        }
    }

    // longer rows: the same, an iteration reading its arcs again
    template <int G>
    __device__ __forceinline__ void discharge_long(int a0, int deg, int u, int gl, int hmax, int iters, int &h, int &e,
                                                   int &sent, bool &pushed) {
        const int h0 = h, na = e > 0 ? deg : 0;
        for (int it = 0; it < iters; ++it) {
            const bool go = e > 0 && h < hmax;
            if (!__any_sync(FULL, go)) break;
            int hm = INT_MAX, at = INT_MAX;
            if (go)
                for (int a = gl; a < deg; a += G) {
                    const int l = rs(a0 + a) > 0 ? head_label(adr[a0 + a]) : INT_MAX;
                    if (l < hm) {
                        hm = l;
                        at = a;
                    }
                }
            const int mine = hm;
            hm = lowest<G>(hm);
            at = lowest<G>(mine == hm ? at : INT_MAX);
            if (go && h <= hm) h = hm >= hmax - 1 ? hmax : hm + 1;
            const bool push = go && h < hmax;
            int d = 0;
            if (push) d = min(e, rs(a0 + at));
            d = __shfl_sync(FULL, d, 0, G);
            if (push) {
                if (gl == 0) push_arc(a0 + at, adr[a0 + at], d);
                pushed = true;
                sent += d;
                e -= d;
            }
        }
        if (h != h0) {
            if (gl == 0) lab[u] = h;
            publish(a0, na, gl, G, h);
        }
    }

    // Lock-free pulses (every vertex holding excess is discharged) until no
    // vertex with excess has a label below hmax; phase 1 returns excess to s.
    // certify: end only after an exact relabel confirms that no excess can move
    // (phase 1; phase 0 is checked by the residual sets instead).
    // may_wave: the first step is a wave, and if it brings three quarters of the excess to the
    // target the rest is left to waves too.  On the 128^3 grid a wave does (4,457 units, then
    // 436, 72, 0 are left) and the sweep takes 8 ms against 14.0 with pulses; on 2D and 3D
    // rggs two thirds of the excess are left after it, every wave is short of the next, and
    // pulses are the faster (waves alone: 34.4 ms against 23.0 on 4.2 M vertices, 64 blocks;
    // the one wave costs a pair 4-9 %).  So a queue sweep tries it on some pairs and then
    // on all while it pays (wave_votes).
    __device__ bool phase_pulse(int ph, int nv, int hmax, bool certify, bool may_wave) {
        long long pulses = 0;
        if (may_wave && w.pre_waves == 0) {
            const int top = relabel(ph, nv, hmax, true);
            int live = 0;   // (each vertex's share bounded, so that the sum stays an int)
            for (int lv = threadIdx.x; lv < nv; lv += TPB) live += lab[lv] < hmax ? min(ex[lv], 4096) : 0;
            live = cluster_sum(live);
            wave_levels(ph, nv, top);
            int left = 0;
            for (int lv = threadIdx.x; lv < nv; lv += TPB) left += lab[lv] < hmax ? min(ex[lv], 4096) : 0;
            left = cluster_sum(left);
            const bool pays = left <= live / 4;
            if (rank == 0 && threadIdx.x == 0) atomicAdd(w.wave_votes, pays ? 1 : -1);
            if (pays) return phase_wave(ph, nv, hmax, 1);
            pulses = 1;
        } else {
            // w.pre_waves waves first move the bulk of the excess along shortest paths
            // (labels stay valid: pushes go one level down); the pulses finish
            const int top = relabel(ph, nv, hmax, w.pre_waves > 0);
            for (int k = 0; k < w.pre_waves; ++k) {
                wave_levels_sync(ph, nv, top);
                if (k + 1 < w.pre_waves) relabel(ph, nv, hmax);
            }
        }
        long long relabels = 1;
        int since = 0;
        for (;;) {
            int act = 0;
            for (int pass = 0; pass < w.passes; ++pass) {
                const bool last = pass + 1 == w.passes;
                const int n = collect(nv, [&](int lv) { return lab[lv] < hmax && *(volatile int *)&ex[lv] > 0; });
                auto visit = [&](auto G, int u, int gl) {
                    const bool on = discharge<G()>(ph, u, gl, hmax, w.inner);
                    if (last) act += on;
                };
                if (n <= TPB / 8) each<8>(n, [&](int u, int gl) { visit(Int<8>(), u, gl); });
                else each<4>(n, [&](int u, int gl) { visit(Int<4>(), u, gl); });
                flush();
            }
            ++pulses;
            ++since;
            const bool a = cluster_any(act);
            if (pulses > w.pulse_cap) return false;
            if (!a) {
                // pushes of earlier passes may land after their target was scanned
                int left = 0;
                for (int lv = threadIdx.x; lv < nv; lv += TPB)
                    left += ex[lv] > 0 && lab[lv] < hmax;
                if (!cluster_any(left)) {
                    if (!certify) break;
                    // Nothing can move by the current labels.  Exact labels decide:
                    // the phase ends only if no vertex with excess can reach its
                    // target (the preflow of phase 0 is then maximum; phase 1 has
                    // returned every excess); otherwise they start the next pulse.
                    relabel(ph, nv, hmax);
                    since = 0;
                    ++relabels;
                    left = 0;
                    for (int lv = threadIdx.x; lv < nv; lv += TPB)
                        left += ex[lv] > 0 && lab[lv] < hmax;
                    if (!cluster_any(left)) break;
                    continue;
                }
            }
            if (since >= w.gr_interval) {
                relabel(ph, nv, hmax);
                since = 0;
                ++relabels;
            } else if (w.gap_interval > 0 && since % w.gap_interval == 0) {
                gap(nv, hmax);
            }
        }
        if (rank == 0 && threadIdx.x == 0) {
            atomicAddLL(&w.ctl->pulses, pulses);
            atomicAddLL(&w.ctl->relabels, relabels);
        }
        return true;
    }

    // Gap heuristic (the paper's max-flow solver, HIPR, uses it): between barriers no
    // label moves, and a valid labelling never lets a residual arc drop more than one
    // label, so if no vertex holds some label h below the largest label held (below
    // hmax), no vertex above h can reach the target: all of them go to hmax at once
    // instead of climbing one push at a time until the next exact relabel.  The held
    // labels are marked in a bitmap in CTA 0's claim array (free during the flow).
    // Returns the vertices lifted (cluster-wide).
    __device__ int gap(int nv, int hmax) {
        const int nwords = (hmax + 31) >> 5;
        if (nwords > H()->nvcap) return 0;   // (tiny ranges: the bitmap does not fit; the same in every CTA)
        const ShArr<unsigned> bm{cla.o};
        if (rank == 0)
            for (int i = threadIdx.x; i < nwords; i += TPB) bm[i] = 0u;
        sync();
        const unsigned bm0 = map_rank(cta_addr(bm.ptr()), 0);
        int top = 0;
        for (int lv = threadIdx.x; lv < nv; lv += TPB) {
            const int h = lab[lv];
            if (h >= 1 && h < hmax) {
                dsm_or(bm0 + 4u * (unsigned)(h >> 5), (int)(1u << (h & 31)));
                top = max(top, h);
            }
        }
        top = cluster_max(top);   // (its barrier also completes the marks)
        // the smallest label in [1, top) that no vertex holds (CTA 0 reads its bitmap)
        int pos = INT_MAX;
        if (rank == 0)
            for (int i = threadIdx.x; i <= (top >> 5); i += TPB) {
                unsigned empty = ~bm[i];
                if (i == 0) empty &= ~1u;                                     // label 0: the target
                if (i == (top >> 5)) empty &= (top & 31) ? ((1u << (top & 31)) - 1u) : 0u;   // below top
                if (empty) pos = min(pos, (i << 5) + __ffs(empty) - 1);
            }
        pos = __reduce_min_sync(FULL, pos);
        const int found = cluster_max(pos == INT_MAX ? 0 : (1 << 30) - pos);
        if (found == 0) return 0;
        const int h0 = (1 << 30) - found;
        int lifted = 0;
        for (int lv = threadIdx.x; lv < nv; lv += TPB) {
            const int h = lab[lv];
            if (h > h0 && h < hmax) {
                lab[lv] = hmax;
                const int a1 = cofs[lv + 1];
                for (int a = cofs[lv]; a < a1; ++a)
                    if (!local(adr[a])) enqueue(Q_LABEL, adr_slot(adr[a]), hmax);
                ++lifted;
            }
        }
        flush();
        lifted = cluster_sum(lifted);
        if (rank == 0 && threadIdx.x == 0) {
            atomicAddLL(&w.ctl->gaps, 1);
            atomicAddLL(&w.ctl->gap_lifted, lifted);
        }
        return lifted;
    }

    // bit 1: reachable from s, seeded with the s-border and with every vertex
    // holding excess (the flow that carries each excess back over a new arc v -> s
    // leaves the residual arc s -> v); bit 2: reaches t.  Frontier pushes: a vertex
    // with a bit not yet passed on sets bit 1 at the heads of its residual arcs and
    // bit 2 at the tails of residual arcs into it (atomic or into the owner's CTA),
    // kScans local scans per cluster barrier as in relabel.  lab, free after the
    // flow, holds the bits already passed on.
    __device__ void reach(int nv) {
        for (int lv = threadIdx.x; lv < nv; lv += TPB) {
            rfl[lv] = (bord[lv] == 1 || ex[lv] > 0 ? 1 : 0) | (bord[lv] == 2 ? 2 : 0);
            lab[lv] = 0;
        }
        sync();
        for (;;) {
            bool any = false;
            for (int k = 0; k < kScans; ++k) {
                const int n = collect(nv, [&](int lv) { return (*(volatile int *)&rfl[lv] & ~lab[lv]) != 0; });
                if (n == 0) break;
                any = true;
                each<4>(n, [&](int u, int gl) {
                    int nw = 0, f = 0;
                    if (u >= 0) {
                        f = *(volatile int *)&rfl[u];
                        nw = f & ~lab[u];
                    }
                    // (the vertex's lanes may have read different bits: all pass on all of them)
                    nw |= __shfl_xor_sync(FULL, nw, 1);
                    nw |= __shfl_xor_sync(FULL, nw, 2);
                    if (u < 0) return;
                    if (gl == 0) lab[u] |= nw;
                    walk<4>(u, gl, [&](unsigned wd, int r, int c) {
                        const int bits = ((nw & 1) && r > 0 ? 1 : 0) | ((nw & 2) && c > r ? 2 : 0);
                        if (!bits) return;
                        if (local(wd)) atomicOr(&rfl[adr_vtx(wd)], bits);
                        else enqueue(Q_OR, adr_slot(wd), bits);
                    });
                });
                flush();
            }
            if (!cluster_any(any)) break;
        }
    }
};

}  // namespace fr
