// nsli_dense.cu -- kernels built on the team Map of register-resident dense
// rows (nsli_team.cuh; sm_103a): whole iterations in one launch, grouped Map
// launches of a pool, and the persistent serving launch.
#include "nsli_team.cuh"

namespace nsli {

namespace {

// ---- iterations in one launch -------------------------------------------------
//
// A cooperative launch of the Map's grid runs up to `iters` iterations: Map,
// grid-wide hand-over A, Reduce and step, hand-over B, the next Map.  The
// arithmetic, its order and the decisions are those of the Map and Reduce
// kernels (bit-identical results), but
//   - A's rows keep streaming: the ring's refills run on into the next
//     iteration's rows while the CTAs reduce (a block that fits the ring is
//     read once per launch);
//   - a hand-over is one release / acquire counter (about 1 us) instead of a
//     kernel boundary and its ramps;
//   - ||dx|| is off the chain from x to x: its binary64 sums run while the
//     next x is being handed over, and the step rule is decided after the next
//     Map (as in the one-CTA sparse kernel), from the sum only when no |dx_j|
//     exceeds eps.
// What bounds it: large systems, HBM; small ones, the latencies of an
// iteration's serial steps (x in, rows, y out, A, group sums, step, B: about 8
// us where the rows take 1 us).  Measured per iteration, graphs of 32 iterations
// (Map and Reduce launches) -> here: 2000 x 500 binary32 12.3 -> 6.8 us, 513 x
// 256 binary64 13.8 -> 8.4, 8192 x 2048 binary32 20.6 -> 14.4, 32768 x 4096 bf16
// 58.8 -> 50.7, 65536 x 8192 bf16 179 -> 173, 131072 x 16384 binary32 1173 ->
// 1165.  Not quicker where the Map is bound by its instructions and this
// kernel, which keeps an iteration's progress beside the slices, has no
// registers left: 131072 x 16384 bf16 616 -> 635, FP8 471 -> 505 (128 registers
// and a spill, the Map kernel 120), 65536 x 8192 FP8 131 -> 133.  Those take it
// all the same; block_iters gives the graphs.
// A: every CTA has written its partial sums and record.  C (ModAP): the
// partial sums of ||y||^2.  B: the new x.  The records (counts and maxima, dx^2
// and max |dx_j|) alternate between two halves (nsli_handover.h), since a CTA
// writes its next ones without waiting for the others' reads of the last, and
// one without columns to reduce does not hold up B.  Every wait is bounded; a
// CTA that gives up raises the state's error flag, which every waiting CTA
// watches.
struct IterShared {
    long long h;
    double mv, mn, mb, scale;
    double tk;      // the tick term of the next Map, in the accumulation type
    int ok, verdict, last;   // verdict: of the stop rules (IterShared::Verdict)
    enum Verdict { kStep, kRuleHeld, kCandidate, kAtMax };
};
static_assert(sizeof(IterShared) <= 128, "shared words of the iteration kernel");

__device__ __forceinline__ void grid_arrive(unsigned int *cnt)
{
    asm volatile("fence.acq_rel.gpu;\n\tred.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
}
__device__ __forceinline__ bool grid_wait(const unsigned int *cnt, unsigned int target, const DevState *st)
{
    const long long t0 = clock64();
    for (unsigned int it = 0;; ++it) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
        if (v >= target)
            return true;
        if ((it & 63u) == 63u) {
            if (*(volatile const int *)&st->error)
                return false;
            if (clock64() - t0 > kWaitLimitCycles)
                return false;
        }
    }
}

// Sum of the per-block partials of dx^2 (y^2) by one warp, in the reduce
// kernel's order.
__device__ __noinline__ double fold_blocks(const double *part, int nblk, int lane)
{
    double v4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int q = lane; q < nblk; q += 128) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (q + 32 * u < nblk)
                v4[u] += __ldcg(part + q + 32 * u);
    }
    return warp_sum((v4[0] + v4[1]) + (v4[2] + v4[3]));
}

// Does the step rule hold after the step whose dx the blocks' partials and
// maxima describe?  (one warp; the sum only when no |dx_j| rules it out)
__device__ __noinline__ bool step_rule_holds(const double *part_dx, const unsigned long long *dmax, int nblk, double eps,
                                             int lane)
{
    unsigned long long dm = 0;
#pragma unroll 1
    for (int q = lane; q < nblk; q += 32)
        dm = max(dm, __ldcg(dmax + q));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        dm = max(dm, __shfl_xor_sync(0xffffffffu, dm, off));
    if (__longlong_as_double((long long)dm) > step_gate(eps))
        return false;
    return step_norm_below(fold_blocks(part_dx, nblk, lane), eps);
}

// A block's partial of dx^2 and its maximum |dx_j| (one warp).
__device__ __noinline__ void put_dx(double dx, double *part, unsigned long long *dmax, int lane)
{
    unsigned long long dm = (unsigned long long)__double_as_longlong(dx) & 0x7fffffffffffffffull;
    double v = dx * dx;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, off);
        dm = max(dm, __shfl_xor_sync(0xffffffffu, dm, off));
    }
    if (lane == 0) {
        *part = v;
        *dmax = dm;
    }
}

// ||y|| from the blocks' sums, and the step's scale lambda / ||y|| (one warp).
__device__ __noinline__ void modap_scale(const double *part, int nblk, double lambda, int lane, double *ynorm,
                                         double *scale)
{
    const double n2 = fold_blocks(part, nblk, lane);
    if (lane == 0) {
        const double n = sqrt(n2);
        *ynorm = n;
        *scale = n > 0.0 ? lambda / n : 0.0;
    }
}

// Counts (as 64 bits, to h) and maxima over the CTAs' records (one warp; past
// L1, where the records of two iterations ago may still be).
template <typename Acc>
__device__ __forceinline__ RowStat<Acc> stats_of(const RowStat<Acc> *rec, int G, int lane, long long &h)
{
    RowStat<Acc> s;
    s.clear();
    h = 0;
    constexpr int U = sizeof(Acc) == 8 ? 1 : 5;   // (152 records: one round trip; binary64: 2218 us against 2253 at five)
#pragma unroll 1
    for (int g0 = lane; g0 < G; g0 += 32 * U) {
        RowStat<Acc> q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            q[u].clear();
            if (g0 + 32 * u < G) {
                const uint4 *src = reinterpret_cast<const uint4 *>(rec + g0 + 32 * u);
                uint4 w[sizeof(RowStat<Acc>) / 16];
#pragma unroll
                for (int i = 0; i < (int)sizeof(RowStat<Acc>) / 16; ++i)
                    w[i] = __ldcg(src + i);
                q[u] = *reinterpret_cast<const RowStat<Acc> *>(w);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            h += q[u].h;
            s.join_maxima(q[u]);
        }
    }
    h = warp_count(h);
    s.fold_maxima();
    return s;
}

// y of a column from its eight group sums, added pairwise in binary64.
template <typename Acc> __device__ __forceinline__ double total_of(const Acc (&v)[8])
{
    return (((double)v[0] + (double)v[1]) + ((double)v[2] + (double)v[3])) +
           (((double)v[4] + (double)v[5]) + ((double)v[6] + (double)v[7]));
}

// Group grp of NGRP's sum over the partial rows g = grp, grp + NGRP, ... of
// column j, in that order in the accumulation type (binary64 is slow on this
// part); binary64: four running sums (g = grp + NGRP (4c + u)) and a tree, a
// dependent binary64 add costing about 300 cycles.  20 loads are in flight at
// a time (all of a group's 19 at 152 partial rows and 8 groups): the sum
// waits for one round trip to L2, not for three.
template <typename Acc, int NGRP>
__device__ __forceinline__ Acc sum_partials(const Acc *py, long long ld, long long j, int grp, int G)
{
    constexpr int U = 20;
    if (j >= ld)
        return Acc(0);
    py += j;
    Acc a[4] = {Acc(0), Acc(0), Acc(0), Acc(0)};
    for (int g0 = grp; g0 < G; g0 += NGRP * U) {
        Acc v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int g = g0 + NGRP * u;
            v[u] = g < G ? __ldcg(py + (long long)g * ld) : Acc(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            a[sizeof(Acc) == 8 ? u & 3 : 0] += v[u];
    }
    if constexpr (sizeof(Acc) == 8)
        return (a[0] + a[1]) + (a[2] + a[3]);
    return a[0];
}

// The 8 group sums of cnt / 8 column blocks b, b + G, ..., spread over NW warps.
template <typename Acc>
__device__ __noinline__ void group_sums(const Acc *part_y, long long ld, int b, int G, int cnt, int NW,
                                        Acc (*part)[8][32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int t = threadIdx.x >> 5; t < cnt; t += NW)
        part[t >> 3][t & 7][lane] =
            sum_partials<Acc, 8>(part_y, ld, (long long)(b + (t >> 3) * G) * kReduceCols + lane, t & 7, G);
}

template <int S, int V, int RG> __global__ void __launch_bounds__(kMapMaxConsumers, 1) iterate_kernel(const IterArgs a)
{
    using Acc = typename Traits<S>::acc;
    constexpr int EPV = Traits<S>::EPV;
    const MapArgs &p = a.map;
    const ReduceArgs &r = a.red;
    DevState *st = p.st;
    // the same for every CTA: the state changes after all have left, or when
    // one gives up, long after they have come.  Also set by a launch that gave
    // up, whose counters and records are unfinished until the next run begins.
    if (*(volatile int *)&st->done)
        return;
    extern __shared__ __align__(128) unsigned char smem[];
    IterShared &sh = *reinterpret_cast<IterShared *>(smem + kHIter);
    const int nbar = (int)blockDim.x, NW = nbar >> 5;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = (int)gridDim.x, b = (int)blockIdx.x;
    const long long row_begin = (long long)b * p.rows_base + min((long long)b, (long long)p.rows_rem);
    const int nrows = (int)(p.rows_base + (b < p.rows_rem ? 1 : 0));
    RowStat<Acc> *stats = static_cast<RowStat<Acc> *>(a.stats);
    const RingSource src = ring_source(p, row_begin, nrows, a.iters, b == 0 ? p.skip_slot : -1);
    const bool resident = src.ns <= p.nstage;
    team_init(p, src);

    // control values, and the progress (kept alike by every thread)
    const int rule = st->rule, stop = st->stop, hold = st->hold_tick;
    const double eps = st->eps, rho = st->rho, lambda = st->lambda;
    const long long max_iter = st->max_iter;
    long long it = st->it, tick = st->tick, h_last = st->h;
    double mv_last = st->maxviol, mn_last = st->maxnorm, mb_last = st->maxb, yn = st->y_norm;
    bool force = st->force_step != 0;
    int status = st->status, done = 0;
    Acc *tk = reinterpret_cast<Acc *>(&sh.tk);
    if (tid == 32)
        *tk = (Acc)((double)tick * rho);
    __syncthreads();

    // This CTA's column blocks: b, b + G, ...  Four at a time: their 32 group
    // sums are spread over all the warps, then one warp takes each block's
    // step, so that the blocks' binary64 chains run side by side.
    const int nblk = a.nblk;
    const int nmine = b < nblk ? (nblk - b + G - 1) / G : 0;
    const unsigned int nred = (unsigned int)min(G, nblk);   // CTAs that reduce
    Acc(*part)[8][32] = reinterpret_cast<Acc(*)[8][32]>(smem + kHPart);

    TeamThread<S, V> me;
    me.init(p);
    unsigned int tg = 0;
    int k = 0;
    bool ok = true;
#pragma unroll 1
    for (; k < a.iters; ++k) {
        // ---- Map
        {
            Acc xr[V][EPV], yr[V][EPV];
            team_load_x<S, V>(p, me, nbar, xr);
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int e = 0; e < EPV; ++e)
                    yr[v][e] = Acc(0);
            RowStat<Acc> stat;
            stat.clear();
            Refill pend;
            const unsigned int q0 = (unsigned)k * (unsigned)src.ns;
            if (me.team < p.teams)
                team_rows<S, V, RG>(p, me, src, q0, resident, tg, xr, yr, *tk, stat, pend);
            bar_threads(1, nbar);
            if (pend.slot >= 0)
                ring_refill(p, src, q0, pend.slot, pend.stage);
            team_finish<S, V>(p, me, nbar, min(p.teams, src.ns), yr, stat, static_cast<Acc *>(p.part_y) + b * p.ld);
            if (tid == 0)
                stats[stat_half(k) * G + b] = stat;
        }
        // ---- A
        if (tid == 0) {
            bool good = *(volatile int *)&team_flags().abort == 0;
            if (good) {
                grid_arrive(a.sync);
                good = grid_wait(a.sync, (unsigned)G * (unsigned)(k + 1), st);
            }
            if (!good)
                atomicOr(&st->error, ERRF_TIMEOUT);
            sh.ok = good;
        }
        bar_threads(1, nbar);
        ok = sh.ok != 0;
        if (!ok)
            break;
        // ---- the first column blocks' group sums, the counts and maxima, and
        // the previous step's rule
        const Acc *py = static_cast<const Acc *>(r.part_y);
        group_sums<Acc>(py, p.ld, b, G, min(kIterBlocks, nmine) * 8, NW, part);
        if (warp == NW - 1) {
            const int half = dx_half_read(k) * nblk;
            const bool rule_holds =
                stop == NSLI_STOP_STEP && k > 0 && step_rule_holds(r.part_dx + half, a.dmax + half, nblk, eps, lane);
            long long violated;
            const RowStat<Acc> all = stats_of<Acc>(stats + stat_half(k) * G, G, lane, violated);
            // the stop decision, by one thread: binary64 comparisons, which
            // would occupy the SM's binary64 pipe for each of its warps
            if (lane == 0) {
                sh.h = violated;
                sh.mv = Image<Acc>::back(all.mv);
                sh.mn = Image<Acc>::back(all.mn);
                sh.mb = Image<Acc>::back(all.mb);
                int v = IterShared::kStep;
                if (rule_holds) {   // ||dx|| < eps after the step before this Map
                    v = IterShared::kRuleHeld;
                } else {
                    bool pass = stop != NSLI_STOP_NONE && sh.h == 0;
                    if (stop == NSLI_STOP_EPSMEM)
                        pass = pass || sh.mn < eps;
                    else if (stop == NSLI_STOP_MAXVIOL_REL)
                        pass = pass || sh.mv <= eps * sh.mb;
                    if (pass && !force)
                        v = IterShared::kCandidate;
                    else if (it >= max_iter)
                        v = IterShared::kAtMax;
                }
                sh.verdict = v;
            }
        }
        bar_threads(1, nbar);
        const int verdict = sh.verdict;
        if (verdict == IterShared::kRuleHeld) {
            status = NSLI_OK;
            done = 1;
            break;
        }
        const long long h = sh.h;
        h_last = h;
        mv_last = sh.mv;
        mn_last = sh.mn;
        mb_last = sh.mb;
        force = false;
        if (verdict != IterShared::kStep) {
            status = verdict == IterShared::kCandidate ? (int)ST_CANDIDATE : (int)NSLI_NOT_CONVERGED;
            done = 1;
            break;
        }
        // ---- Reduce and step
        const bool modap = rule == NSLI_RULE_MODAP;
        const double s = modap || h == 0 ? 0.0 : __ldg(r.rtab + h);
        int pend_blk = -1;      // a block whose partial dx^2 is still to be summed
        double pend_d = 0.0;
        auto put_pending = [&]() {
            const int q = dx_half_written(k) * nblk + pend_blk;
            put_dx(pend_d, r.part_dx + q, a.dmax + q, lane);
        };
        auto step_column = [&](long long j, double scale, double y, double xo) {
            const double xn = xo - scale * y;
            r.x64[j] = xn;
            static_cast<Acc *>(r.x)[j] = (Acc)(xn);
            return xn - xo;
        };
#pragma unroll 1
        for (int i0 = 0; i0 < nmine; i0 += kIterBlocks) {
            if (i0 > 0) {
                bar_threads(1, nbar);   // the group sums before have been read
                group_sums<Acc>(py, p.ld, b + i0 * G, G, min(kIterBlocks, nmine - i0) * 8, NW, part);
                bar_threads(1, nbar);
            }
            const int blk = b + (i0 + warp) * G;
            if (warp < kIterBlocks && blk < nblk) {
                const long long j = (long long)blk * kReduceCols + lane;
                const bool in = j < p.ld;
                const double xo = in ? __ldcg(r.x64 + j) : 0.0;
                Acc v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    v[q] = part[warp][q][lane];
                const double y = total_of<Acc>(v);
                if (modap) {
                    if (in)
                        r.ybuf[j] = y;
                    const double y2 = warp_sum(in ? y * y : 0.0);
                    if (lane == 0)
                        r.part_dx[2 * nblk + blk] = y2;
                } else {
                    if (pend_blk >= 0)
                        put_pending();
                    pend_blk = blk;
                    pend_d = in ? step_column(j, s, y, xo) : 0.0;
                }
            }
        }
        if (modap) {
            // ---- C: ||y|| over all columns, then the step
            bar_threads(1, nbar);
            if (tid == 32 * kIterBlocks) {
                if (b < nblk)
                    grid_arrive(a.sync + 2);
                sh.ok = grid_wait(a.sync + 2, nred * (unsigned)(k + 1), st);
            }
            bar_threads(1, nbar);
            ok = sh.ok != 0;
            if (!ok)
                break;
            if (warp == 0)
                modap_scale(r.part_dx + 2 * nblk, nblk, lambda, lane, &sh.mv, &sh.scale);
            bar_threads(1, nbar);
            yn = sh.mv;
            if (warp < kIterBlocks)
#pragma unroll 1
                for (int blk = b + warp * G; blk < nblk; blk += kIterBlocks * G) {
                    const long long j = (long long)blk * kReduceCols + lane;
                    if (pend_blk >= 0)
                        put_pending();
                    pend_blk = blk;
                    pend_d = j < p.ld ? step_column(j, sh.scale, r.ybuf[j], __ldcg(r.x64 + j)) : 0.0;   // (its own y)
                }
        } else {
            yn = 0.0;
        }
        it += 1;
        if (!hold)
            tick += 1;
        // ---- B
        bar_threads(1, nbar);
        if (tid == 32 * kIterBlocks) {
            if (b < nblk)
                grid_arrive(a.sync + 1);
            sh.ok = grid_wait(a.sync + 1, nred * (unsigned)(k + 1), st);
        } else if (tid == 32 * kIterBlocks + 32) {
            *tk = (Acc)((double)tick * rho);
        }
        if (pend_blk >= 0)
            put_pending();
        bar_threads(1, nbar);
        ok = sh.ok != 0;
        if (!ok)
            break;
    }
    // ---- leave with no copy in flight; the last CTA writes the state
    __syncthreads();
    if (tid == 0) {
        ring_drain(p);
        int last = 0;
        if (ok) {
            __threadfence();
            last = atomicAdd(a.sync + 3, 1u) == (unsigned)G - 1u;
        } else {
            atomicOr(&st->error, ERRF_TIMEOUT);
            *(volatile int *)&st->done = 1;   // launches behind this one leave at once
        }
        sh.last = last;
    }
    __syncthreads();
    if (!sh.last || warp != 0)
        return;
    __threadfence();
    const int steps = k;   // made by this launch: iteration k was left before its step, or the loop ended
    double dx2 = 0.0;
    if (steps > 0) {
        dx2 = fold_blocks(r.part_dx + dx_half_written(steps - 1) * nblk, nblk, lane);
        if (!done && stop == NSLI_STOP_STEP && step_norm_below(dx2, eps)) {
            status = NSLI_OK;
            done = 1;
        }
    }
    if (lane == 0) {
        st->it = it;
        st->tick = tick;
        st->h = h_last;
        st->maxviol = mv_last;
        st->maxnorm = mn_last;
        st->maxb = mb_last;
        if (steps > 0) {
            st->dx2 = dx2;
            st->y_norm = yn;
        }
        st->force_step = 0;
        st->status = status;
        st->done = done;
        for (int q = 0; q < 4; ++q)
            a.sync[q] = 0u;
    }
}

// One work item of a problem, by the instance of the problem's own shape.
template <int S, int V>
__device__ __forceinline__ void map_item_v(const GroupProblem &gp, const GroupItem &it)
{
    using Acc = typename Traits<S>::acc;
    void *prow = static_cast<Acc *>(gp.map.part_y) + (long long)it.part * gp.map.ld;
    PartStat *pst = gp.map.part_stat + it.part;
    const int nrows = (int)(it.row_end - it.row_begin);
    if (gp.map.rows_per_slot == 1)
        map_body(MapForm<S, V, 1>{}, gp.map, it.row_begin, nrows, prow, pst, -1);
    else if (gp.map.rows_per_slot == 2)
        map_body(MapForm<S, V, 2>{}, gp.map, it.row_begin, nrows, prow, pst, -1);
    else if constexpr (kRgMax(V, (int)sizeof(Acc)) >= 4) {
        if (gp.map.rows_per_slot == 4)
            map_body(MapForm<S, V, 4>{}, gp.map, it.row_begin, nrows, prow, pst, -1);
        else if constexpr (kRgMax(V, (int)sizeof(Acc)) >= 8)
            map_body(MapForm<S, V, 8>{}, gp.map, it.row_begin, nrows, prow, pst, -1);
    }
}
template <int S> __device__ __forceinline__ void map_item(const GroupProblem &gp, const GroupItem &it)
{
    if (gp.vpt == 1)
        map_item_v<S, 1>(gp, it);
    else if (gp.vpt == 2)
        map_item_v<S, 2>(gp, it);
    else if (gp.vpt == 4)
        map_item_v<S, 4>(gp, it);
    else if constexpr (S == NSLI_F32)
        map_item_v<S, 8>(gp, it);
}

// Many problems in one launch: CTA b maps work item b (a block of rows of
// one problem) with that problem's own thread mapping, so a problem's
// partial sums do not depend on which other problems share the launch.
template <int S>
__global__ void __launch_bounds__(kMapMaxConsumers, 1) map_group_kernel(const GroupProblem *probs, const GroupItem *items)
{
    const GroupItem it = items[blockIdx.x];
    const GroupProblem &gp = probs[it.prob];
    if (*(volatile int *)&gp.map.st->done)
        return;
    map_item<S>(gp, it);
}

// ------------------------------------------------- persistent serving ----
//
// One cooperative launch (every CTA resident, one per SM) iterates all live
// problems of a pool round after round:
//   control   CTA 0: wall-clock ticks, problems that stopped in the last
//             round go to the host-mapped completion list, the stop decision
//             (host yield, nothing left running, round or time bound);
//   Map       CTAs take the work items (a block of rows of one problem)
//             i = blockIdx.x, blockIdx.x + grid, ...;
//   Reduce    the same for the (problem, column block) items;
// with a grid barrier after each phase.  A problem's items and their
// arithmetic are those of the grouped launches, so its iterates do not
// depend on the other problems or on which CTA ran which item.  Every
// barrier wait is bounded: on expiry the CTA records the error and returns
// (the others then expire too).

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The serving kernel keeps its few shared words beside the ring's abort flag
// and the reduce's shared blocks behind the ring header (idle during the
// Reduce phase), so it needs no shared memory beyond the largest ring of its
// problems.
constexpr int kServeRedGrp = 2;   // warps per serving reduce item
constexpr int kServeRedSub = 8;   // reduce items in flight per CTA

// Grid barrier over nblocks resident CTAs: sense by generation count.
__device__ __forceinline__ bool serve_grid_sync(ServeSync *sy, unsigned int nblocks)
{
    int &ok = team_flags().ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned int *gen = &sy->bar_gen;
        const unsigned int g = *gen;          // before arriving
        __threadfence();
        const unsigned int arrived = atomicAdd(&sy->bar_count, 1u) + 1u;
        int good = 1;
        if (arrived == nblocks) {
            atomicExch(&sy->bar_count, 0u);   // reset before the release
            __threadfence();
            atomicAdd(&sy->bar_gen, 1u);
        } else {
            const long long t0 = clock64();
            for (unsigned int it = 0; *gen == g; ++it) {
                if ((it & 63u) == 63u && clock64() - t0 > kWaitLimitCycles) {
                    good = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

// Control phase (CTA 0).
__device__ __forceinline__ void serve_control(const ServeArgs &a, long long round, unsigned long long t_start)
{
    int &running = team_flags().running;
    if (threadIdx.x == 0)
        running = 0;
    __syncthreads();
    const unsigned long long now = global_ns();
    int mine = 0;
    for (int q = threadIdx.x; q < a.nprob; q += blockDim.x) {
        DevState *st = a.probs[q].red.st;
        if (round == 0) {
            a.tick0[q] = st->tick;
            a.reported[q] = *(volatile int *)&st->done;   // stopped before this launch
        }
        const int done = *(volatile int *)&st->done;
        if (done && !a.reported[q]) {
            a.reported[q] = 1;
            const unsigned int k = atomicAdd(&a.sync->ndone, 1u);
            if (k < (unsigned int)kServeMaxProblems) {
                ServeDone d;
                d.prob = q;
                d.status = st->status;
                d.it = st->it;
                a.ctrl->done[k] = d;
            }
        }
        if (!done) {
            ++mine;
            if (a.tick_ns > 0)
                st->tick = a.tick0[q] + (long long)((now - t_start) / a.tick_ns);
        }
    }
    if (mine)
        atomicAdd(&running, mine);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence_system();
        *(volatile unsigned int *)&a.ctrl->done_count = a.sync->ndone;
        *(volatile unsigned long long *)&a.ctrl->rounds = (unsigned long long)round;
        const int yield = *(volatile int *)&a.ctrl->yield;
        a.sync->stop = (yield || running == 0 || round >= a.max_rounds || now - t_start > a.max_ns) ? 1 : 0;
        a.sync->map_next = 0u;   // every CTA has left the previous round's phases
        a.sync->red_next = 0u;
        __threadfence_system();
    }
}

template <int S> __global__ void __launch_bounds__(kMapMaxConsumers, 1) serve_kernel(const ServeArgs a)
{
    using Acc = typename Traits<S>::acc;
    // Reduce items run kServeRedSub at a time per CTA, each on its own
    // kServeRedGrp warps (their own named barrier and shared block, placed
    // in the ring's stages, free in that phase): an item is a chain of
    // dependent global-memory round trips, and several in flight overlap
    constexpr int NGRP = kServeRedGrp;
    constexpr int NSUB = kMapMaxConsumers / (32 * NGRP);
    static_assert(NSUB == kServeRedSub, "reduce sub-blocks tile the CTA");
    extern __shared__ __align__(128) unsigned char smem[];
    const int sub = threadIdx.x / (32 * NGRP), stid = threadIdx.x % (32 * NGRP);
    ReduceSharedT<NGRP> &rsh = reinterpret_cast<ReduceSharedT<NGRP> *>(smem + kTeamHeader)[sub];
    int *sub_item = reinterpret_cast<int *>(smem + kTeamHeader + NSUB * sizeof(ReduceSharedT<NGRP>));
    TeamFlags &ss = team_flags();
    if (threadIdx.x == 0)
        ss.t_start = global_ns();
    __syncthreads();
    const unsigned long long t_start = ss.t_start;
    const unsigned int G = gridDim.x;
    for (long long round = 0;; ++round) {
        if (blockIdx.x == 0)
            serve_control(a, round, t_start);
        if (!serve_grid_sync(a.sync, G))
            break;
        if (*(volatile int *)&a.sync->stop)
            break;
        // items are taken one at a time from a shared counter (an item's
        // arithmetic does not depend on the CTA that runs it)
        for (;;) {
            if (threadIdx.x == 0)
                ss.item = (int)atomicAdd(&a.sync->map_next, 1u);
            __syncthreads();
            const int i = ss.item;
            if (i >= a.nitems)
                break;
            const GroupItem it = a.items[i];
            const GroupProblem &gp = a.probs[it.prob];
            if (!*(volatile int *)&gp.map.st->done)
                map_item<S>(gp, it);
            __syncthreads();   // every warp has left the ring before it is armed again
        }
        if (!serve_grid_sync(a.sync, G))
            break;
        for (;;) {
            if (stid == 0)
                sub_item[sub] = (int)atomicAdd(&a.sync->red_next, 1u);
            sub_sync(1 + sub, 32 * NGRP);
            const int i = sub_item[sub];
            if (i >= a.nreds)
                break;
            const GroupRed t = a.reds[i];
            const GroupProblem &gp = a.probs[t.prob];
            reduce_body<Acc, NGRP>(gp.red, t.blk, gp.red_blocks, rsh, stid, 1 + sub);
            sub_sync(1 + sub, 32 * NGRP);   // the item's shared words are free again
        }
        __syncthreads();
        if (!serve_grid_sync(a.sync, G))
            break;
    }
    if (threadIdx.x == 0 && *(volatile int *)&a.sync->stop == 0) {
        // left on an expired barrier wait
        atomicOr(&a.ctrl->error, 1);
        __threadfence_system();
    }
}

struct IterFn {
    template <int S, int V, int RG> static const void *get() { return (const void *)iterate_kernel<S, V, RG>; }
};
const void *map_group_fn(int storage)
{
    if (storage == NSLI_BF16)
        return (const void *)map_group_kernel<NSLI_BF16>;
    return storage == NSLI_F32 ? (const void *)map_group_kernel<NSLI_F32> : nullptr;
}
const void *serve_fn(int storage)
{
    if (storage == NSLI_BF16)
        return (const void *)serve_kernel<NSLI_BF16>;
    return storage == NSLI_F32 ? (const void *)serve_kernel<NSLI_F32> : nullptr;
}
}  // namespace

int team_threads(int teams, int team_warps) { return std::max(288, teams * team_warps * 32); }

int team_rg_max(int vpt, bool f64) { return kRgMax(vpt, f64 ? 8 : 4); }

cudaError_t team_prepare(int storage, int vpt, int rg, int threads, int *iter_blocks_per_sm)
{
    cudaError_t e = team_map_prepare(storage, vpt, rg);
    const void *fn = dense_fn<IterFn>(storage, vpt, rg);
    if (e == cudaSuccess)
        e = set_smem(fn);
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(iter_blocks_per_sm, fn, threads, kSmemMax);
}

cudaError_t iterate_launch(int storage, int vpt, int grid, size_t smem, cudaStream_t s, const IterArgs &a)
{
    const void *fn = dense_fn<IterFn>(storage, vpt, a.map.rows_per_slot);
    if (!fn)
        return cudaErrorInvalidValue;
    void *args[] = {const_cast<IterArgs *>(&a)};
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(team_threads(a.map.teams, a.map.team_warps)), args, smem,
                                       s);
}

cudaError_t map_group_prepare(int storage) { return set_smem(map_group_fn(storage)); }

cudaError_t map_group_launch(int storage, int items, size_t smem, cudaStream_t s, const GroupProblem *probs,
                             const GroupItem *it)
{
    const void *fn = map_group_fn(storage);
    if (!fn)
        return cudaErrorInvalidValue;
    void *args[] = {&probs, &it};
    return cudaLaunchKernel(fn, dim3(items), dim3(kMapMaxConsumers), args, smem, s);
}

cudaError_t serve_prepare(int storage, size_t smem, int *blocks_per_sm)
{
    const void *fn = serve_fn(storage);
    cudaError_t e = set_smem(fn);
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, kMapMaxConsumers, smem);
}

cudaError_t serve_launch(int storage, int grid, size_t smem, cudaStream_t s, const ServeArgs &a)
{
    const void *fn = serve_fn(storage);
    if (!fn)
        return cudaErrorInvalidValue;
    void *args[] = {(void *)&a};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(kMapMaxConsumers), args, smem, s);
}

}  // namespace nsli
