// C ABI, host side of the queue sweep (queue_sweep.cu): per-cluster workspaces, the
// choice of cluster size, the launch (captured as a CUDA graph like the round-by-round
// sweep) and the fallback to the round-by-round sweep when a pair outgrows a cluster.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "api_internal.h"

using namespace fr;

#define CK(call)                                                 \
    do {                                                         \
        cudaError_t e_ = (call);                                 \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, #call); \
    } while (0)

namespace {

// relative time of one pair on clusters of 4, 6, 8, 12, 16 CTAs (measured on 3D rgg and
// grid pairs; the same table as the round-by-round cluster launches)
constexpr double kRelTime[fr_ctx::kNumClusterSizes] = {1.25, 1.05, 1.0, 0.85, 0.74};
// The time of a sweep on clusters of one size: a vertex of the quotient graph is in up to nr
// pairs that wait for one another, and the clusters have turns = pairs / clusters to take;
// sqrt(nr^2 + turns^2) times the time of one pair fits both ends.  Corridors of fewer
// vertices than a cluster of 8 has threads gain little from more CTAs, of fewer than one CTA
// has nothing (rgg2d 20,011, k = 7: the kernel 1.47 ms on 4, 1.49, 1.52, 1.57, 1.66 on 16).  Taking the most pairs in flight over a pair's time alone (the chain left out)
// chose 4 CTAs for rgg3d 524,287 vertices, k = 32 (18 rounds, 155 pairs, 1,316 vertices):
// 8.2 ms, against 7.5 on 6 and 7.4 on 8; 8 for rgg2d 20,011, k = 7 (346 vertices): 1.83 ms
// for the call against 1.70 on 4; 16 for rgg3d 77,488, k = 5 (930 vertices): 2.69 against
// 2.53 on 8; and what this rule chooses, too, for 1,000,003, k = 64 (4: 9.7 ms, 6: 9.9, 8:
// 12.2) and 4M, k = 64 (6: 23.0, 8: 26.1).
constexpr long long kTiny = 512, kSmall = 4096;
constexpr double kRelSmall[fr_ctx::kNumClusterSizes] = {1.17, 1.05, 1.0, 1.0, 1.0};
constexpr double kRelTiny[fr_ctx::kNumClusterSizes] = {1.0, 1.01, 1.02, 1.06, 1.13};
// host staging offsets (the first megabytes of h_stage belong to the other paths)
constexpr size_t kStageGraphs = 4u << 20;
constexpr size_t kStagePrev = (4u << 20) + (64u << 10);
// a round on the queue kernel (enqueue_round_queue): descriptors, read-back
constexpr size_t kStageRound = 6u << 20, kStageRoundCtl = (6u << 20) + (512u << 10);
constexpr unsigned long long kWaitNs = 10ull * 1000 * 1000 * 1000;   // one dependency wait, at most 10 s

size_t al256(size_t b) { return (b + 255) / 256 * 256; }

struct QCaps {
    long long nu, mu, vq, words, swords;
};

// Per-pair capacities of a cluster of `ctas` CTAs: dyn / 28 vertices per CTA, more than its
// shared memory holds (31 bytes a vertex, see ClusterFlow::carve); arcs have room for dyn / 16
// (8 bytes each would fit, but a pair that large is better off on a larger cluster, and the
// HBM arrays of every slot would double).
QCaps caps_for(int ctas, int n) {
    const long long dyn = (long long)queue_smem();
    QCaps c;
    c.nu = (long long)ctas * dyn / 28 + 64;
    c.mu = (long long)ctas * dyn / 16 + 64;
    c.vq = std::min<long long>(n, std::max<long long>(4 * c.nu, 1 << 16));
    // the ids are numbered a group of 1,024 at a time, so the last group's words are read to
    // its end: they exist, and are cleared with the others
    c.words = 32LL * (n / 1024 + 1);
    c.swords = n / 32768 + 2;
    return c;
}

size_t slot_bytes(const QCaps &c, int ctas, int k, int reps) {
    size_t b = 0;
    auto add = [&](size_t elem, long long cnt) { b += al256(elem * (size_t)cnt); };
    add(4, k);                                      // sob
    add(8, 3LL * 2 * kHistBins);                    // hist
    add(4, ctas + 1);                               // cta_cnt
    add(4, c.words);                                // cbits
    add(4, c.words);                                // sdbits
    add(4, c.swords);                               // sbits
    add(4, c.vq); add(4, c.vq);                     // vq_v vq_s
    for (int i = 0; i < 21; ++i) add(4, c.nu + 1);  // gid .. sinkc, pcur
    add(8, c.nu); add(8, c.nu);                     // ex cw
    add(1, c.nu); add(1, c.nu);                     // border side_out
    for (int i = 0; i < 5; ++i) add(4, c.mu);       // head rev res cap outs
    for (int i = 0; i < 3; ++i) add(4, (long long)reps * c.nu);   // indeg_r order hcomp
    add(8, (long long)reps * c.nu);                 // hkey
    add(8, reps); add(4, reps);                     // sw_absd sw_j
    return b;
}

template <class T>
T *take(char *&p, long long count) {
    T *r = reinterpret_cast<T *>(p);
    p += al256(sizeof(T) * (size_t)count);
    return r;
}

// Ticket, votes, scan length, abort word, control blocks and counters of a launch on
// `clusters` clusters.
size_t queue_state_bytes(const QueueMem &Q, int clusters) {
    return 2 * al256(sizeof(int)) + al256(sizeof(QueueMem::QCtl) * (size_t)Q.clusters) +
           4 * sizeof(long long) * (size_t)clusters;
}

// Entries of a block's region for the commits' appends (a sweep that fills one runs again
// round by round).
long long qb_cap_for(int n, int k) { return std::max<long long>(4096, 8LL * ((n + k - 1) / k)); }

// lists: a sweep's predecessors and per-block candidate lists (24 to 40 bytes a vertex), which
// a single round does not read.
size_t queue_bytes(int ctas, int clusters, int n, int nnz, int k, int reps, int np, bool lists) {
    size_t b = 2 * al256(4) + al256(4ull * nnz) + al256(sizeof(QSlot) * clusters) + al256(sizeof(GraphDev) * clusters) +
               al256(sizeof(QueueMem::QCtl) * clusters) + al256(32ull * clusters) +
               slot_bytes(caps_for(ctas, n), ctas, k, reps) * clusters;
    if (!lists) b += al256(8ull * k);   // blockw0
    if (lists)
        b += al256(8ull * np) + 2 * al256(4ull * n) + al256(4ull * (k + 1)) + 2 * al256(4ull * k) +
             al256(4ull * k * qb_cap_for(n, k));
    return b;
}

// Lays Q out for launches on up to `clusters` clusters of `ctas` CTAs.  Sweeps and rounds have
// a workspace each: a program that calls both would lay a shared one out again at every change
// of cluster size, and drop its captured sweeps with it (a sweep of rgg2d 20,011, k = 7, in turn
// with a pair of 65,536 vertices: 1.97 ms, 1.90 with two), and a sweep under an arena bound
// could be refused for the sizes that a pair call before it had asked for.
fr_status ensure_queue(fr_ctx *ctx, QueueMem &Q, int ctas, int clusters, int n, int nnz, int k, int reps, int np) {
    if (Q.mem && ctas == Q.ctas && clusters <= Q.clusters && n <= Q.n && nnz <= Q.nnz && k <= Q.k && reps <= Q.reps &&
        np <= Q.np)
        return FR_OK;
    const bool sweep = &Q == &ctx->sweep_q;
    int nn = n, mm = nnz, kk = k, rr = std::max(reps, 1), pp = np, cc = clusters;
    if (Q.ctas == ctas) {   // as large as the calls before asked for
        nn = std::max(nn, Q.n); mm = std::max(mm, Q.nnz); kk = std::max(kk, Q.k);
        rr = std::max(rr, Q.reps); pp = std::max(pp, Q.np); cc = std::max(cc, Q.clusters);
    }
    // A round's workspace is taken where it fits beside everything held (its launches have
    // another form); the sweeps' is needed, and others make room for it.
    const size_t others = sweep ? ctx->base_bytes + ctx->pair_bytes + ctx->reps_bytes : held_bytes(ctx) - Q.bytes;
    auto fits = [&](size_t b) { return ctx->arena_limit == 0 || b + others <= ctx->arena_limit; };
    size_t bytes = queue_bytes(ctas, cc, nn, mm, kk, rr, pp, sweep);
    if (!fits(bytes)) {   // what this call asks for alone
        nn = n; mm = nnz; kk = k; rr = std::max(reps, 1); pp = np; cc = clusters;
        bytes = queue_bytes(ctas, cc, nn, mm, kk, rr, pp, sweep);
    }
    if (!fits(bytes)) {
        ctx_error(ctx, "queue sweep workspace exceeds the arena bound");
        return FR_ERR_OOM;
    }
    // Another cluster size lays the same memory out again where it is large enough: a V-cycle
    // and the rounds of active scheduling change sizes often, and a cudaFree and cudaMalloc
    // pair takes longer than a small round.
    if (!Q.mem || bytes > Q.bytes) {
        free_queue(Q);
        if ((sweep ? alloc_workspace(ctx, &Q.mem, bytes) : cudaMalloc(&Q.mem, bytes)) != cudaSuccess) {
            cudaGetLastError();
            Q.mem = nullptr;
            ctx_error(ctx, "cudaMalloc(%zu) for the queue sweep failed", bytes);
            return FR_ERR_OOM;
        }
        Q.bytes = bytes;
    }
    const QCaps c = caps_for(ctas, nn);
    Q.ctas = ctas; Q.clusters = cc; Q.n = nn; Q.nnz = mm; Q.k = kk; Q.reps = rr; Q.np = pp;
    Q.nu = c.nu; Q.mu = c.mu; Q.vq = c.vq;
    char *p = reinterpret_cast<char *>(Q.mem);
    Q.ticket = take<int>(p, 3);   // ticket, votes, scan length
    Q.gabort = take<int>(p, 1);
    Q.ctls = take<QueueMem::QCtl>(p, cc);   // (cleared with the words before them, and the
    Q.stats = take<long long>(p, 4LL * cc);   // abort word read back with them: queue_state_bytes)
    Q.crank = take<int>(p, mm);
    Q.slots = take<QSlot>(p, cc);
    if (sweep) {
        Q.prev = take<int>(p, 2LL * pp);
        Q.qb_sorted = take<int>(p, nn);
        Q.qb_start = take<int>(p, kk + 1);
        Q.qb_cnt = take<int>(p, kk);
        Q.qb_app = take<int>(p, kk);
        Q.qb_cap = (int)qb_cap_for(nn, kk);
        Q.qb_pool = take<int>(p, (long long)kk * Q.qb_cap);
        Q.qb_lst = take<int>(p, nn);
    } else {
        Q.blockw0 = take<long long>(p, kk);
    }
    Q.graphs = take<GraphDev>(p, cc);
    Q.host.assign(cc, QSlot());
    // what is idle between launches lies together over the slots, to be cleared in two calls
    char *const idle = p;
    for (QSlot &S : Q.host) S.sob = take<int>(p, kk);
    char *const bits = p;
    for (QSlot &S : Q.host) {
        S.cbits = take<unsigned int>(p, c.words);
        S.sdbits = take<unsigned int>(p, c.words);
        S.sbits = take<unsigned int>(p, c.swords);
    }
    char *const slots = p;
    for (int i = 0; i < cc; ++i) {
        QSlot &S = Q.host[i];
        S.graph = Q.graphs + i;
        S.ctl = &Q.ctls[i].c;
        S.hist = take<long long>(p, 3LL * 2 * kHistBins);
        S.cta_cnt = take<int>(p, ctas + 1);
        S.vq_v = take<int>(p, c.vq); S.vq_s = take<int>(p, c.vq);
        int **v21[21] = {&S.gid, &S.sid, &S.off, &S.infc, &S.fx, &S.lab, &S.rflag, &S.color, &S.scc, &S.vc,
                         &S.fq0, &S.fq1, &S.cid, &S.cpair, &S.cmin, &S.indeg, &S.outoff, &S.ocur, &S.plist,
                         &S.sinkc, &S.pcur};
        for (auto a : v21) *a = take<int>(p, c.nu + 1);
        S.ex = take<long long>(p, c.nu); S.cw = take<long long>(p, c.nu);
        S.border = take<unsigned char>(p, c.nu); S.side_out = take<unsigned char>(p, c.nu);
        S.head = take<int>(p, c.mu); S.rev = take<int>(p, c.mu); S.res = take<int>(p, c.mu);
        S.cap = take<int>(p, c.mu); S.outs = take<int>(p, c.mu);
        S.indeg_r = take<int>(p, (long long)rr * c.nu); S.order = take<int>(p, (long long)rr * c.nu);
        S.hcomp = take<int>(p, (long long)rr * c.nu);
        S.hkey = take<unsigned long long>(p, (long long)rr * c.nu);
        S.sw_absd = take<long long>(p, rr); S.sw_j = take<int>(p, rr);
        S.stat = Q.stats + 4LL * i;
    }
    // idle state: no block paired, no corridor bit set
    CK(cudaMemsetAsync(idle, 0xFF, (size_t)(bits - idle), ctx->stream));
    CK(cudaMemsetAsync(bits, 0, (size_t)(slots - bits), ctx->stream));
    CK(cudaMemcpyAsync(Q.slots, Q.host.data(), sizeof(QSlot) * cc, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    if (sweep) destroy_graph_cache(ctx);   // captured sweeps hold pointers into the old workspace
    return FR_OK;
}

// After a failed or abandoned launch: BFS marks, corridor bits and block sides idle.
fr_status reset_queue_idle(fr_ctx *ctx, QueueMem &Q) {
    fr_status st = reset_idle(ctx);
    if (st != FR_OK) return st;
    const QCaps c = caps_for(Q.ctas, Q.n);
    for (const QSlot &S : Q.host) {
        CK(cudaMemsetAsync(S.sob, 0xFF, sizeof(int) * (size_t)Q.k, ctx->stream));
        CK(cudaMemsetAsync(S.cbits, 0, sizeof(unsigned int) * (size_t)c.words, ctx->stream));
        CK(cudaMemsetAsync(S.sdbits, 0, sizeof(unsigned int) * (size_t)c.words, ctx->stream));
        CK(cudaMemsetAsync(S.sbits, 0, sizeof(unsigned int) * (size_t)c.swords, ctx->stream));
    }
    CK(cudaStreamSynchronize(ctx->stream));
    return FR_OK;
}

}  // namespace

void free_queue(QueueMem &Q) {
    if (Q.mem) cudaFree(Q.mem);
    Q = QueueMem();
}

int queue_size_for(fr_ctx *ctx, const BatchPlan &pl, const fr_options *opt) {
    if (opt->fm_permille > 0 || opt->sweep_sched == 1 || pl.np == 0) return -1;
    if (2LL * pl.np * (long long)sizeof(int) > (long long)(kHostStage - kStagePrev)) return -1;
    const size_t dyn = queue_smem();
    if (dyn == 0) return -1;
    long long est = 0;
    for (long long e : pl.est_max) est = std::max(est, e);
    // The workspace depends on the size, and with it which calls an arena bound admits: under a
    // bound the size is the one with the most pairs in flight over a pair's time, whatever is
    // fastest, so that no call is refused for speed.
    const bool bounded = ctx->arena_limit != 0;
    // (an estimate: 31 bytes a vertex rounded down, and 16 an arc, the arcs a slot has room for,
    // see caps_for)
    const double need = 1.05 * (double)est * (29.0 + (bounded && !ctx->narrow_ok ? 20.0 : 16.0) * pl.avg_degree);
    const double per_cta = 0.95 * (double)dyn;
    const int force = opt->cluster_ctas ? opt->cluster_ctas : ctx->tune_ctas;
    int best = -1, kept = -1;
    double bestv = 0, keptv = 0;
    for (int t = 0; t < fr_ctx::kNumClusterSizes; ++t) {
        if (ctx->q_cap[t] <= 0) continue;
        const int c = fr_ctx::kClusterSizes[t];
        if (force) {
            if (force == c) return t;
            continue;
        }
        if (need > per_cta * c) continue;
        const double chain = pl.nr, turns = (double)pl.np / std::min(ctx->q_cap[t], pl.np);
        const double v = bounded ? -(double)std::min(ctx->q_cap[t], pl.np) / kRelTime[t] :
                         std::sqrt(chain * chain + turns * turns) *
                             (est <= kTiny ? kRelTiny : est <= kSmall ? kRelSmall : kRelTime)[t];
        if (best < 0 || v < bestv) { best = t; bestv = v; }
        if (ctx->sweep_q.mem && ctx->sweep_q.ctas == c) { kept = t; keptv = v; }
    }
    // The size laid out already, unless another is clearly better: laying out again takes a few
    // tenths of a millisecond and drops the captured sweeps (a V-cycle of grid3d 108,570
    // vertices, k = 14, that went between 4 and 8 CTAs: 25.4 ms, 23.8 on 4 throughout).
    if (!bounded && kept >= 0 && keptv <= 1.07 * bestv) return kept;
    return best;
}

fr_status run_queue_sweep(fr_ctx *ctx, const fr_graph *g, int32_t *part, const BatchPlan &pl, const fr_options *opt,
                          int t, float *ms, bool *ran, std::vector<Ctl> *ctls) {
    *ran = false;
    const int ctas = fr_ctx::kClusterSizes[t];
    // resident clusters, or fewer when opt->grid_blocks bounds the CTAs
    int clusters = std::max(1, std::min(ctx->q_cap[t], pl.np));
    if (opt->grid_blocks > 0) clusters = std::max(1, std::min(clusters, opt->grid_blocks / ctas));
    const int reps = opt->mb_reps > 0 ? opt->mb_reps : 1;
    QueueMem &Q = ctx->sweep_q;
    fr_status st = ensure_queue(ctx, Q, ctas, clusters, g->n, g->nnz, pl.k, reps, pl.np);
    if (st != FR_OK) return st;
    // per-cluster graph descriptors (each with its own sob) and each pair's predecessors
    GraphDev *hg = reinterpret_cast<GraphDev *>(ctx->h_stage + kStageGraphs);
    for (int i = 0; i < clusters; ++i) {
        GraphDev &gd = hg[i];
        memset(&gd, 0, sizeof(gd));
        gd.xadj = g->xadj; gd.adjncy = g->adjncy; gd.adjwgt = g->adjwgt; gd.vwgt = g->vwgt;
        gd.part = part; gd.dist = ctx->dist; gd.lid = ctx->lid;
        gd.sob = Q.host[i].sob;
        gd.blockw = ctx->blockw;
        gd.n = g->n; gd.nnz = g->nnz; gd.k = pl.k; gd.base = 0; gd.Lmax = pl.Lmax;
        gd.bl = ctx->bl; gd.blc = ctx->blc; gd.inb = ctx->inb;
    }
    int *hp = reinterpret_cast<int *>(ctx->h_stage + kStagePrev);
    {
        std::vector<int> last(pl.k, -1);
        for (int j = 0; j < pl.np; ++j) {
            hp[2 * j] = last[pl.pa[j]];
            hp[2 * j + 1] = last[pl.pb[j]];
            last[pl.pa[j]] = last[pl.pb[j]] = j;
        }
    }
    CK(cudaMemcpyAsync(Q.graphs, hg, sizeof(GraphDev) * (size_t)clusters, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(Q.prev, hp, sizeof(int) * 2 * (size_t)pl.np, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(ctx->part_backup, part, sizeof(int) * (size_t)g->n, cudaMemcpyDeviceToDevice, ctx->stream));

    QueueArgs q;
    memset(&q, 0, sizeof(q));
    q.wt = make_work(ctx, 0, 0, pl.np, g->n, opt);
    q.wt.vq_cap = (int)Q.vq;
    q.wt.nu_cap = (int)Q.nu;
    q.wt.mu_cap = (int)Q.mu;
    q.wt.crank = Q.crank;
    q.wt.total_n = g->n;
    q.wt.qb_sorted = Q.qb_sorted;
    q.wt.qb_start = Q.qb_start;
    q.wt.qb_app = Q.qb_app;
    q.wt.qb_pool = Q.qb_pool;
    q.wt.qb_lst = Q.qb_lst;
    q.wt.qb_cap = Q.qb_cap;
    q.slots = Q.slots;
    q.np = pl.np;
    q.ticket = Q.ticket;
    q.votes = q.wt.flow_sched == 0 ? Q.ticket + 1 : nullptr;
    q.prev = Q.prev;
    q.gabort = Q.gabort;
    q.wait_ns = kWaitNs;

    auto enqueue = [&]() -> fr_status {
        CK(launch_fill_pairs(ctx->pairs, ctx->pair_a, ctx->pair_b, pl.np, 0, opt->mb ? 1 : 0, pl.Ubase, ctx->stream));
        CK(cudaMemsetAsync(ctx->sides, 0, sizeof(SideDev) * 2 * (size_t)pl.np, ctx->stream));
        CK(cudaMemsetAsync(ctx->pacc, 0, sizeof(PairAcc) * (size_t)pl.np, ctx->stream));
        CK(cudaMemsetAsync(Q.ticket, 0, queue_state_bytes(Q, clusters), ctx->stream));
        CK(cudaMemsetAsync(Q.qb_lst, 0xFF, sizeof(int) * (size_t)g->n, ctx->stream));
        CK(cudaMemsetAsync(Q.qb_cnt, 0, sizeof(int) * (size_t)pl.k, ctx->stream));
        CK(launch_qb_build(ctx->bl, ctx->blc, part, pl.k, Q.qb_cnt, Q.qb_start, Q.qb_app, Q.qb_lst,
                           Q.qb_sorted, ctx->stream));
        if (ctx->profiling) CK(cudaEventRecord(ctx->pev[0], ctx->stream));
        CK(launch_queue_sweep(q, ctas, clusters, ctx->stream));
        if (ctx->profiling) CK(cudaEventRecord(ctx->pev[1], ctx->stream));
        return FR_OK;
    };
    while (ctx->profiling && ctx->pev.size() < 2) {
        cudaEvent_t e;
        CK(cudaEventCreate(&e));
        ctx->pev.push_back(e);
    }
    // launches of the sweep: prep, compaction, colouring, pair fill, the three list
    // kernels, the queue kernel
    const long long launches = 8;
    std::vector<long long> key = {-7, (long long)(uintptr_t)g->xadj, (long long)(uintptr_t)part, g->n, g->nnz,
                                  pl.np, pl.Ubase, opt->mb, reps, (long long)opt->seed, opt->gr_interval,
                                  opt->inner_ops, opt->pulse_cap, (long long)(uintptr_t)ctx->base_mem,
                                  (long long)(uintptr_t)ctx->pair_mem, (long long)(uintptr_t)Q.mem,
                                  ctx->tune_gr, ctx->tune_inner, opt->pulse_passes, ctx->tune_passes,
                                  q.wt.flow_sched, ctx->tune_sched, ctx->narrow_ok, opt->pre_waves,
                                  ctx->tune_prewaves, ctas, clusters, pl.Lmax, opt->gap_interval};
    ctx->prof.scan_ms = ctx->prof.step_ms = ctx->prof.cluster_ms = 0;
    ctx->round_ms.clear();
    ctx->pair_ms.clear();
    cudaGraphExec_t exec = nullptr;
    if (ctx->use_graphs && !ctx->profiling) {
        for (auto &e : ctx->gcache)
            if (e.key == key) { exec = e.exec; break; }
        if (!exec) {
            cudaGraph_t graph = nullptr;
            CK(cudaStreamSynchronize(ctx->stream));
            cudaError_t e = cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal);
            fr_status est = FR_OK;
            if (e == cudaSuccess) {
                est = enqueue();
                cudaError_t e2 = cudaStreamEndCapture(ctx->stream, &graph);
                if (est == FR_OK && e2 == cudaSuccess && graph) {
                    e2 = cudaGraphInstantiate(&exec, graph, 0);
                    cudaGraphDestroy(graph);
                    if (e2 != cudaSuccess) exec = nullptr;
                } else if (graph) {
                    cudaGraphDestroy(graph);
                }
            }
            cudaGetLastError();
            if (exec) {
                if (ctx->gcache.size() >= 16) {
                    cudaGraphExecDestroy(ctx->gcache.front().exec);
                    ctx->gcache.erase(ctx->gcache.begin());
                }
                ctx->gcache.push_back({key, exec, launches});
            } else {
                ctx->use_graphs = false;
            }
        }
    }
    CK(cudaEventRecord(ctx->ev0, ctx->stream));
    if (exec) {
        CK(cudaGraphLaunch(exec, ctx->stream));
    } else {
        if ((st = enqueue()) != FR_OK) return st;
    }
    CK(cudaEventRecord(ctx->ev1, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    CK(cudaEventElapsedTime(ms, ctx->ev0, ctx->ev1));
    ctx->sweep_launches = launches;
    ctx->last_launches = launches;
    int gab = 0;
    CK(cudaMemcpyAsync(&gab, Q.gabort, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    std::vector<QueueMem::QCtl> qc(clusters);
    CK(cudaMemcpyAsync(qc.data(), Q.ctls, sizeof(QueueMem::QCtl) * (size_t)clusters, cudaMemcpyDeviceToHost,
                       ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    ctls->resize(clusters);
    for (int i = 0; i < clusters; ++i) (*ctls)[i] = qc[i].c;
    ctx->last_queue_ctas = ctas;
    ctx->last_queue_clusters = clusters;
    if (gab != 0) {
        // leave part exactly as it was, and the workspace idle
        CK(cudaMemcpyAsync(part, ctx->part_backup, sizeof(int) * (size_t)g->n, cudaMemcpyDeviceToDevice, ctx->stream));
        if ((st = reset_queue_idle(ctx, Q)) != FR_OK) return st;
        if (gab == E_MISFIT) {
            ++ctx->queue_fallbacks;
            int where = 0;
            for (const Ctl &x : *ctls)
                if (x.error == E_MISFIT) { where = x.error_where; break; }
            ctx_error(ctx, "queue sweep: a pair outgrew its cluster's workspace (check %d); ran round by round",
                      where);
            return FR_OK;   // *ran = false: the caller runs the sweep round by round
        }
        Ctl c;
        memset(&c, 0, sizeof(c));
        c.error = gab;
        for (const Ctl &x : *ctls)
            if (x.error) { c = x; break; }
        return status_from_ctl(ctx, c, "fr_refine_batch (queue sweep)");
    }
    if (ctx->profiling) {
        // the queue kernel alone; the setup launches before it (pair fill, clears, lists)
        float qk = 0.f, pre = 0.f;
        CK(cudaEventElapsedTime(&pre, ctx->ev0, ctx->pev[0]));
        CK(cudaEventElapsedTime(&qk, ctx->pev[0], ctx->pev[1]));
        ctx->prof.cluster_ms = qk;
        ctx->prof.scan_ms = pre;
        std::vector<PairAcc> A(pl.np);
        CK(cudaMemcpyAsync(A.data(), ctx->pacc, sizeof(PairAcc) * pl.np, cudaMemcpyDeviceToHost, ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
        unsigned long long first = ~0ull;
        for (int i = 0; i < pl.np; ++i)
            if (A[i].t1 && A[i].t0 < first) first = A[i].t0;
        ctx->pair_ms.assign(3 * (size_t)pl.np, 0.f);
        int r = 0;
        for (int i = 0; i < pl.np; ++i) {
            while (r + 1 < pl.nr && i >= pl.off[r + 1]) ++r;
            float *pm = &ctx->pair_ms[3 * (size_t)i];
            pm[0] = (float)r;
            pm[1] = A[i].t1 ? (float)((A[i].t0 - first) * 1e-6) : -1.f;
            pm[2] = A[i].t1 ? (float)((A[i].t1 - first) * 1e-6) : -1.f;
        }
    }
    *ran = true;
    return FR_OK;
}

// ------------------------------------------------- one round, one launch ----
// The pairs of one round (block-disjoint, so none waits for another) through the queue
// kernel, a cluster for each pair, instead of the sequence boundary scan, step, cluster flow,
// step.  Those two steps are cooperative launches over the whole grid, some 140 us each for a
// corridor of a few thousand vertices whatever its size: about forty grid barriers of 2-3 us
// and dependent loads between them.  A cluster barrier is 0.25 us.

int queue_round_size(fr_ctx *ctx, int P, long long est, double avg_degree, const fr_options *opt) {
    if (P <= 0 || opt->sweep_sched == 1 || ctx->max_clusters <= 0 || queue_smem() == 0) return -1;
    const double need = 1.05 * (double)est * (29.0 + 16.0 * avg_degree);   // (as for a sweep)
    const double per_cta = 0.95 * (double)queue_smem();
    const int force = opt->cluster_ctas ? opt->cluster_ctas : ctx->tune_ctas;
    int best = -1, kept = -1;
    double bestc = 0, keptc = 0;
    for (int t = 0; t < fr_ctx::kNumClusterSizes; ++t) {
        if (ctx->q_cap[t] <= 0) continue;
        const int c = fr_ctx::kClusterSizes[t];
        if (force) {
            if (force == c) return t;
            continue;
        }
        if (need > per_cta * c) continue;
        // turns of resident clusters times the time of one pair; a corridor of fewer vertices
        // than one CTA has threads only loses by being spread (122 vertices: 288 us on 4 CTAs,
        // 308 on 16, the whole call)
        const double v = est <= kTiny ? (double)c :
                                        (double)((P + ctx->q_cap[t] - 1) / ctx->q_cap[t]) * kRelTime[t];
        if (best < 0 || v < bestc) { best = t; bestc = v; }
        if (ctx->round_q.mem && ctx->round_q.ctas == c) { kept = t; keptc = v; }
    }
    // the size laid out already, unless another is clearly better
    return kept >= 0 && keptc <= 1.25 * bestc ? kept : best;
}

fr_status enqueue_round_queue(fr_ctx *ctx, const fr_graph *g, int32_t *part, int k, int P, long long Lmax,
                              const fr_options *opt, int t, RoundQueue *rq) {
    *rq = RoundQueue();
    const int ctas = fr_ctx::kClusterSizes[t];
    int clusters = std::max(1, std::min(ctx->q_cap[t], P));
    if (opt->grid_blocks > 0) clusters = std::max(1, std::min(clusters, opt->grid_blocks / ctas));
    const int reps = opt->mb_reps > 0 ? opt->mb_reps : 1;
    QueueMem &Q = ctx->round_q;
    const fr_status st = ensure_queue(ctx, Q, ctas, clusters, g->n, g->nnz, k, reps, P);
    if (st == FR_ERR_OOM) return FR_OK;   // no room under the arena bound: the round's own launches
    if (st != FR_OK) return st;
    GraphDev *hg = reinterpret_cast<GraphDev *>(ctx->h_stage + kStageRound);
    static_assert(kStageRound + 64 * sizeof(GraphDev) <= kStageRoundCtl, "descriptors of every resident cluster");
    if (clusters > 64) clusters = 64;
    for (int i = 0; i < clusters; ++i) {
        GraphDev &gd = hg[i];
        memset(&gd, 0, sizeof(gd));
        gd.xadj = g->xadj; gd.adjncy = g->adjncy; gd.adjwgt = g->adjwgt; gd.vwgt = g->vwgt;
        gd.part = part; gd.dist = ctx->dist; gd.lid = ctx->lid;
        gd.sob = Q.host[i].sob;
        gd.blockw = ctx->blockw;
        gd.n = g->n; gd.nnz = g->nnz; gd.k = k; gd.base = 0; gd.Lmax = Lmax;
        gd.bl = ctx->bl; gd.blc = ctx->blc; gd.inb = ctx->inb;
    }
    CK(cudaMemcpyAsync(Q.graphs, hg, sizeof(GraphDev) * (size_t)clusters, cudaMemcpyHostToDevice, ctx->stream));
    QueueArgs q;
    memset(&q, 0, sizeof(q));
    q.wt = make_work(ctx, 0, 0, P, g->n, opt);
    q.wt.vq_cap = (int)Q.vq;
    q.wt.nu_cap = (int)Q.nu;
    q.wt.mu_cap = (int)Q.mu;
    q.wt.crank = Q.crank;
    q.wt.total_n = g->n;
    q.slots = Q.slots;
    q.np = P;
    q.ticket = Q.ticket;
    q.votes = q.wt.flow_sched == 0 && low_degree(ctx, kTryDeg) ? Q.ticket + 1 : nullptr;
    q.prev = nullptr;   // no pair waits for another
    q.gabort = Q.gabort;
    q.wait_ns = kWaitNs;
    q.wt.scan_len = Q.ticket + 2;   // pairs commit to the list while others scan it: they scan what is on it now
    RoundBegin rb;
    rb.part = part; rb.part0 = ctx->spare; rb.n = g->n;
    rb.blockw = ctx->blockw; rb.blockw0 = Q.blockw0; rb.k = k;
    rb.clear[0] = reinterpret_cast<int *>(ctx->sides); rb.words[0] = (int)(sizeof(SideDev) / 4 * 2 * (size_t)P);
    rb.clear[1] = reinterpret_cast<int *>(ctx->pacc); rb.words[1] = (int)(sizeof(PairAcc) / 4 * (size_t)P);
    rb.clear[2] = Q.ticket; rb.words[2] = (int)(queue_state_bytes(Q, clusters) / 4);
    rb.blc = ctx->blc; rb.scan_len = Q.ticket + 2;
    CK(launch_round_begin(rb, ctx->sms, ctx->stream));
    CK(launch_queue_sweep(q, ctas, clusters, ctx->stream));
    char *h = ctx->h_stage + kStageRoundCtl;
    CK(cudaMemcpyAsync(h, Q.gabort, 256 + sizeof(QueueMem::QCtl) * (size_t)clusters, cudaMemcpyDeviceToHost,
                       ctx->stream));
    rq->queued = true;
    rq->clusters = clusters;
    return FR_OK;
}

fr_status finish_round_queue(fr_ctx *ctx, const fr_graph *g, int32_t *part, int k, const char *where, RoundQueue *rq) {
    const char *h = ctx->h_stage + kStageRoundCtl;
    const int gab = *reinterpret_cast<const int *>(h);
    const QueueMem::QCtl *qc = reinterpret_cast<const QueueMem::QCtl *>(h + 256);
    memset(&rq->ctl, 0, sizeof(rq->ctl));
    for (int i = 0; i < rq->clusters; ++i) {
        const Ctl &c = qc[i].c;
        rq->ctl.pulses += c.pulses;
        rq->ctl.relabels += c.relabels;
        rq->ctl.levels = std::max(rq->ctl.levels, c.levels);
        rq->ctl.scc_rounds += c.scc_rounds;
        if (gab != 0 && c.error && !rq->ctl.error) {
            rq->ctl.error = c.error;
            rq->ctl.error_where = c.error_where;
        }
    }
    if (gab == 0) return FR_OK;
    fr_status st = reset_queue_idle(ctx, ctx->round_q);
    if (st != FR_OK) return st;
    if (gab == E_MISFIT) {
        rq->queued = false;
        ++ctx->queue_fallbacks;
        CK(cudaMemcpyAsync(part, ctx->spare, sizeof(int) * (size_t)g->n, cudaMemcpyDeviceToDevice, ctx->stream));
        CK(cudaMemcpyAsync(ctx->blockw, ctx->round_q.blockw0, sizeof(long long) * (size_t)k, cudaMemcpyDeviceToDevice,
                           ctx->stream));
        return FR_OK;
    }
    if (!rq->ctl.error) rq->ctl.error = gab;
    return status_from_ctl(ctx, rq->ctl, where);
}
