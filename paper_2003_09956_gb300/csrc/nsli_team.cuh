// nsli_team.cuh -- the Map of register-resident dense rows (sm_103a): one
// block of rows by a CTA, for the Map's own kernel (nsli_kernels.cu), whole
// iterations in one launch, grouped Map launches of a pool and the persistent
// serving launch (nsli_dense.cu).
//
// Team Map.  Every mapping thread keeps a fixed column slice of the iterate
// x and of the partial sum y in registers (at most 32 binary32 entries of
// each), so a row of n entries needs W = ceil(n / 1024) warps (binary64:
// ceil(n / 512)).  Such W warps are a team; a CTA holds T = floor(16 / W)
// teams, and team t maps row groups t, t + T, ... of the CTA's rows.  Only the
// warps of a team meet (an mbarrier per row group), so while one team waits
// for its warps' dot products the others stream.  The shared-memory ring's
// stage is one row group (R rows and their records), filled by one bulk copy
// each with completion on the stage's "full" barrier.  Small teams: the last
// warp to finish with a stage refills it.  Teams of eight warps or more are
// bound by their own chain of steps, which the last warp's detour would
// lengthen: their first warp refills the stage of the group before, once the
// next barrier shows that all have finished it (Map of 131072 x 16384
// binary32: 1.17 ms against 1.35 ms).  No producer warp: a seventeenth warp
// would leave 96 registers a thread instead of 128, and the slices of x and y
// would spill.
//
// What bounds it: HBM, or for systems that fit there L2, as long as a row
// group's chain (dot, fold, barrier, coefficient, slice: about 0.9 us whatever
// its bytes) is shared by enough rows or covered by other teams.
#pragma once

#include "nsli_handover.h"
#include "nsli_map.cuh"

#include <algorithm>
#include <type_traits>

namespace nsli {

namespace {

// ---- shared-memory layout (bytes) -------------------------------------------
constexpr int kTeamWarps = kMapMaxConsumers / 32;         // mapping warps at most
constexpr int kHFull = 0;                                 // full barriers
constexpr int kHIssued = kHFull + kMapMaxStages * 8;      // copies issued per stage
constexpr int kHFreed = kHIssued + kMapMaxStages * 4;     // warps that have finished with the stage
constexpr int kHTeam = kHFreed + kMapMaxStages * 4;       // 4 barriers per team
constexpr int kHFlags = kHTeam + kTeamWarps * 4 * 8;      // abort flag and a few words
constexpr int kHRed = kHFlags + 128;                      // [team][4][RG][W] warp sums (16 x 4 x 8 binary32)
constexpr int kHStat = kHRed + kTeamWarps * 4 * 4 * 8;    // one RowStat per team
constexpr int kHEnd = kHStat + kTeamWarps * 32;
constexpr int kHPart = kHEnd;                             // iterations in one launch: the reduce's group sums
constexpr int kIterBlocks = 4;                            // column blocks a CTA reduces at a time
constexpr int kHIter = kHPart + kIterBlocks * 8 * 32 * 8; // ... and its shared words
static_assert(kHIter + 128 <= kTeamHeader, "team Map header fits");

struct TeamFlags {
    int abort;                   // a bounded wait expired in this CTA: everyone leaves
    int item;                    // serving: the work item the CTA took
    int ok, running;             // serving: barrier outcome, problems still running
    unsigned long long t_start;  // serving: start of the launch
};
__device__ __forceinline__ TeamFlags &team_flags()
{
    extern __shared__ __align__(128) unsigned char smem[];
    return *reinterpret_cast<TeamFlags *>(smem + kHFlags);
}

// (Code size matters here: what runs once per pass or per iteration comes from
// the instruction caches, and a kernel of 120 KB spent more time fetching its
// instructions than on a small system's rows.  So: one copy of each piece,
// rolled loops outside the row loop, cold parts in functions of their own.)

// Has a bounded wait that began at t0 to end?  (asked once in 64 polls)
__device__ __forceinline__ bool give_up(unsigned int polls, long long t0)
{
    if ((polls & 63u) != 63u)
        return false;
    volatile int *abort = &team_flags().abort;
    if (clock64() - t0 > kWaitLimitCycles)
        *abort = 1;
    return *abort != 0;
}

// Wait for a phase, polling; gives up (and makes every role give up) after
// kWaitLimitCycles or when another role has.
__device__ __forceinline__ bool team_wait(unsigned int bar, unsigned int parity)
{
    if (mbar_test(bar, parity))
        return true;
    const long long t0 = clock64();
    for (unsigned int it = 0; !mbar_test(bar, parity); ++it)
        if (give_up(it, t0))
            return false;
    return true;
}

// Named barrier of n threads.  The warp converges first: bar.sync is an
// aligned instruction, and lanes that leave a polling loop or one lane's refill
// late would otherwise arrive apart.
__device__ __forceinline__ void bar_threads(int id, int n)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Counts and maxima of some rows of one CTA (an int holds their number; over
// the grid the counts are added as 64 bits: warp_count, stats_of).  Binary64
// maxima are kept as order-preserving integers: exact, and quicker than
// binary64 comparisons.
template <typename Acc> struct Image;
template <> struct Image<float> {
    using type = float;
    static __device__ __forceinline__ float of(float v) { return v; }
    static __device__ __forceinline__ double back(float v) { return (double)v; }
    static __device__ __forceinline__ float lowest() { return -INFINITY; }
};
template <> struct Image<double> {
    using type = unsigned long long;
    static __device__ __forceinline__ unsigned long long of(double v) { return red_ord_enc(v); }
    static __device__ __forceinline__ double back(unsigned long long v) { return red_ord_dec(v); }
    static __device__ __forceinline__ unsigned long long lowest() { return 0x000fffffffffffffull; }   // of -infinity
};
__device__ __forceinline__ long long warp_count(long long h)
{
    const CountParts c = count_parts(h);
    const unsigned int lo = __reduce_add_sync(0xffffffffu, c.lo), hi = __reduce_add_sync(0xffffffffu, c.hi);
    return count_join(lo, hi);
}
template <typename Acc> struct alignas(4 * sizeof(Acc)) RowStat {
    using I = typename Image<Acc>::type;
    typename std::conditional<sizeof(Acc) == 8, long long, int>::type h;
    I mv, mn, mb;
    __device__ __forceinline__ void clear()
    {
        h = 0;
        mv = mn = mb = Image<Acc>::lowest();
    }
    __device__ __forceinline__ void add(Acc ri, Acc rn, Acc ab, bool viol)
    {
        h += viol ? 1 : 0;
        mv = up(mv, Image<Acc>::of(ri));
        mn = up(mn, Image<Acc>::of(rn));
        mb = up(mb, Image<Acc>::of(ab));
    }
    __device__ __forceinline__ void join_maxima(const RowStat &o)
    {
        mv = up(mv, o.mv);
        mn = up(mn, o.mn);
        mb = up(mb, o.mb);
    }
    // over the warp, in every lane: integer reductions of one instruction
    // instead of five shuffles and maxima each (exact; no value is a NaN: up()
    // never takes one)
    __device__ __forceinline__ void fold()
    {
        if constexpr (sizeof(Acc) == 8)
            h = warp_count(h);
        else
            h = __reduce_add_sync(0xffffffffu, h);
        fold_maxima();
    }
    __device__ __forceinline__ void fold_maxima()
    {
        mv = top(mv);
        mn = top(mn);
        mb = top(mb);
    }
    static __device__ __forceinline__ float top(float v)
    {
        // binary32 values order like their bits as signed integers, the
        // negative ones reversed
        const int b = __float_as_int(v), k = __reduce_max_sync(0xffffffffu, b < 0 ? b ^ 0x7fffffff : b);
        return __int_as_float(k < 0 ? k ^ 0x7fffffff : k);
    }
    static __device__ __forceinline__ unsigned long long top(unsigned long long v)
    {
        const unsigned int hi = __reduce_max_sync(0xffffffffu, (unsigned int)(v >> 32));
        const unsigned int lo =
            __reduce_max_sync(0xffffffffu, (unsigned int)(v >> 32) == hi ? (unsigned int)v : 0u);
        return ((unsigned long long)hi << 32) | lo;
    }
    __device__ __forceinline__ PartStat record() const
    {
        return PartStat{(long long)h, Image<Acc>::back(mv), Image<Acc>::back(mn), Image<Acc>::back(mb)};
    }
    static __device__ __forceinline__ I up(I a, I b) { return b > a ? b : a; }
};
static_assert(sizeof(RowStat<float>) == 16 && sizeof(RowStat<double>) == 32, "one or two 16-byte loads");

// One thread's place: its team, its warp within the team, its vectors.
template <int S, int V> struct TeamThread {
    int team, wt, lane;
    int voff[V];   // byte offset of each owned vector in a row (0 when beyond the row)
    bool vok[V];   // the vector lies inside the row
    __device__ __forceinline__ void init(const MapArgs &p)
    {
        const int warp = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
        team = warp / p.team_warps;
        wt = warp - team * p.team_warps;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int j = wt * 32 + lane + v * p.team_warps * 32;
            vok[v] = j < p.nv;
            // vectors beyond the row read its first one against x = 0
            voff[v] = vok[v] ? j * 16 : 0;
        }
    }
};

// What a CTA streams: its block of rows, in `total` slots from first to last
// (a whole number of passes over the block's ns slots).
struct RingSource {
    const unsigned char *A, *meta;   // the block's first row and record
    int nrows, ns;
    unsigned int total;              // (below 2^32: iterations_of)
    int skip;                        // failure injection: this slot never arrives (-1: none)
};
__device__ __forceinline__ RingSource ring_source(const MapArgs &p, long long row_begin, int nrows, int passes, int skip)
{
    RingSource r;
    r.A = static_cast<const unsigned char *>(p.A) + row_begin * (long long)p.row_bytes;
    r.meta = static_cast<const unsigned char *>(p.meta) + row_begin * 32;
    r.nrows = nrows;
    r.ns = (nrows + p.rows_per_slot - 1) / p.rows_per_slot;
    r.total = (unsigned)r.ns * (unsigned)passes;
    r.skip = skip;
    return r;
}

// Issue the copies of slot s into a stage (one thread; the stage is free).
__device__ __forceinline__ void ring_issue(const MapArgs &p, const RingSource &src, int s, int stage)
{
    extern __shared__ __align__(128) unsigned char smem[];
    if (s == src.skip)
        return;
    const int R = p.rows_per_slot;
    const unsigned int rows = (unsigned int)min(R, src.nrows - s * R);
    const unsigned int bytesA = rows * (unsigned int)p.row_bytes, bytesM = rows * 32u;
    const unsigned int dst = smem_u32(smem + p.ring_offset) + (unsigned int)stage * (unsigned int)p.stage_stride;
    const unsigned int fb = smem_u32(smem + kHFull) + 8u * stage;
    const long long r0 = (long long)s * R;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_expect_tx(fb, bytesA + bytesM);
    bulk_g2s(dst, src.A + r0 * p.row_bytes, bytesA, fb);
    bulk_g2s(dst + (unsigned int)R * (unsigned int)p.row_bytes, src.meta + r0 * 32, bytesM, fb);
    // the fill's barrier phase is open: teams may wait for it (slot_wait)
    if (p.teams > 1)
        __threadfence_block();
    reinterpret_cast<volatile int *>(smem + kHIssued)[stage] += 1;
}

// Wait (bounded) until no copy into the ring is in flight (one thread, after
// the block has synchronised).
__device__ __noinline__ void ring_drain(const MapArgs &p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const volatile int *issued = reinterpret_cast<const volatile int *>(smem + kHIssued);
#pragma unroll 1
    for (int q = 0; q < p.nstage; ++q)
        if (issued[q] > 0)
            mbar_wait_bounded(smem_u32(smem + kHFull) + 8u * q, (unsigned int)(issued[q] - 1) & 1u);
}

// Wait for fill number `fill` (from 0) of a stage.  A parity wait alone tells
// only whether the phase before the current one was even or odd, so it must
// not begin before fill - 1 has been consumed: one team knows (it consumed
// it), several do not (another team may lag behind), and look at the stage's
// count of fills issued first (a fill is issued only once the one before has
// been consumed).
__device__ __forceinline__ bool slot_wait(const MapArgs &p, int stage, unsigned int fill)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const volatile int *issued = reinterpret_cast<const volatile int *>(smem + kHIssued) + stage;
    const unsigned int bar = smem_u32(smem + kHFull) + 8u * stage;
    const bool several = p.teams > 1;
    if (!several && mbar_test(bar, fill & 1u))
        return true;
    const long long t0 = clock64();
    for (unsigned int it = 0; (several && (unsigned)*issued <= fill) || !mbar_test(bar, fill & 1u); ++it)
        if (give_up(it, t0))
            return false;
    return true;
}

// Refill the stage that held slot `slot` of the pass that begins at ring
// index q0 (one thread; every warp of the team has finished with it).
__device__ __forceinline__ void ring_refill(const MapArgs &p, const RingSource &src, unsigned int q0, int slot,
                                            int stage)
{
    if (q0 + (unsigned)(slot + p.nstage) >= src.total)
        return;
    int s = slot + p.nstage;
    if (s >= src.ns)
        s -= src.ns;   // the next pass (a ring with refills is shorter than the block)
    ring_issue(p, src, s, stage);
}

// The calling warp (one thread of it) has finished with a stage: is it the
// team's last to do so?
__device__ __forceinline__ bool ring_release(const MapArgs &p, int stage)
{
    extern __shared__ __align__(128) unsigned char smem[];
    if (p.team_warps == 1)
        return true;
    int *freed = reinterpret_cast<int *>(smem + kHFreed) + stage;
    __threadfence_block();
    if (atomicAdd(freed, 1) != p.team_warps - 1)
        return false;
    *freed = 0;   // (seen by the stage's next warps through its full barrier)
    __threadfence_block();
    return true;
}

// A slot whose stage a large team's first thread has yet to refill.
struct Refill {
    int slot = -1, stage = 0;
};

// The rows of one pass over the block mapped by the calling warp's team: dots,
// residuals, statistics and positive slices.  `q0` is the ring index of the
// pass's first slot, `tg` the number of row groups this team has mapped since
// its barriers were initialised.  `resident`: the ring holds the whole block
// and is filled once.  pend: the slot that the team's first thread has to
// refill once every mapping thread has finished the pass (large teams).
template <int S, int V, int RG>
__device__ __forceinline__ bool team_rows(const MapArgs &p, const TeamThread<S, V> &me, const RingSource &src,
                                          const unsigned int q0, const bool resident, unsigned int &tg,
                                          const typename Traits<S>::acc (&xr)[V][Traits<S>::EPV],
                                          typename Traits<S>::acc (&yr)[V][Traits<S>::EPV],
                                          const typename Traits<S>::acc tk, RowStat<typename Traits<S>::acc> &stat,
                                          Refill &pend)
{
    using Tr = Traits<S>;
    using Acc = typename Tr::acc;
    using Meta = typename Tr::meta;
    constexpr int EPV = Tr::EPV;
    constexpr int WL = 32 / RG;   // lanes per row in the folded reductions
    // independent chains per row.  More of them do not pay in binary64 either:
    // its pipe is the limit with many warps on the SM, and every chain is one
    // more addition per thread and row (16385 x 8192 binary64, per iteration:
    // a chain per vector 926 us, two chains 716 us)
    constexpr int NCH = (V >= 4 && RG <= 2) ? 2 : 1;
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int R = RG;   // a slot is one row group
    const int W = p.team_warps, T = p.teams, lane = me.lane;
    const int ng = me.team < src.ns ? (src.ns - me.team + T - 1) / T : 0;
    const bool large = W >= kLargeTeam, refiller = large && !resident && me.wt == 0 && lane == 0;
    const unsigned int tbar = smem_u32(smem + kHTeam) + (unsigned int)me.team * 32u;
    Acc *red = reinterpret_cast<Acc *>(smem + kHRed) + (size_t)me.team * W * (4 * RG);
    const unsigned char *stages = smem + p.ring_offset;
    const unsigned int qt = (resident ? 0u : q0) + (unsigned)me.team;
    int stage = (int)(qt % (unsigned)p.nstage);
    unsigned int fill = (unsigned int)(qt / (unsigned)p.nstage);   // which fill of the stage
    int slot = me.team;
    // butterfly width that covers the team's warps
    int fold0 = 1;
    while (fold0 < W && fold0 < WL)
        fold0 <<= 1;
    fold0 >>= 1;
    const int fq = lane / WL, fi = lane % WL;

#pragma unroll 1
    for (int i = 0; i < ng; ++i) {
        const int rows = min(R, src.nrows - slot * R);
        if (!slot_wait(p, stage, fill))
            return false;
        const unsigned char *sb = stages + stage * p.stage_stride;
        Acc acc[RG];
#pragma unroll
        for (int rr = 0; rr < RG; ++rr) {
            // (a short last group repeats its last row, masked below, so
            // that the rows' loads and sums interleave without branches)
            const unsigned char *row = sb + min(rr, rows - 1) * p.row_bytes;
            Acc pe[NCH], po[NCH];
#pragma unroll
            for (int q = 0; q < NCH; ++q) {
                pe[q] = Acc(0);
                po[q] = Acc(0);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                Acc a[EPV];
                decode<S>(*reinterpret_cast<const uint4 *>(row + me.voff[v]), a);
#pragma unroll
                for (int e = 0; e < EPV; e += 2)
                    fma2(pe[v % NCH], po[v % NCH], a[e], a[e + 1], xr[v][e], xr[v][e + 1]);
            }
#pragma unroll
            for (int q = 0; q < NCH; ++q)
                pe[q] += po[q];
#pragma unroll
            for (int w = NCH / 2; w > 0; w >>= 1)
#pragma unroll
                for (int q = 0; q < w; ++q)
                    pe[q] += pe[q + w];
            acc[rr] = pe[0];
        }
        const Acc ws = warp_fold_rows<RG>(acc, lane);
        const unsigned int g = tg + (unsigned)i, buf = g & 3u;
        if (fi == 0)
            red[(buf * RG + fq) * W + me.wt] = ws;
        __syncwarp();
        if (W > 1) {
            if (lane == 0)
                mbar_arrive(tbar + 8u * buf);
            if (!team_wait(tbar + 8u * buf, (g >> 2) & 1u))
                return false;
        }
        if (refiller) {
            // every warp arrived, i.e. has finished the group before
            if (pend.slot >= 0)
                ring_refill(p, src, q0, pend.slot, pend.stage);
            pend.slot = slot;
            pend.stage = stage;
        }
        // team totals, lane (fq, fi): row fq; then r, the coefficient and
        // the statistics of the row in the lanes of its group
        Acc dot = Acc(0);
#pragma unroll 1
        for (int w = fi; w < W; w += WL)
            dot += red[(buf * RG + fq) * W + w];
#pragma unroll 1
        for (int off = fold0; off > 0; off >>= 1)
            dot += __shfl_xor_sync(0xffffffffu, dot, off);
        const bool valid = fq < rows;
        const Meta md = *reinterpret_cast<const Meta *>(sb + R * p.row_bytes + (valid ? fq : 0) * 32);
        const Acc sc = (Acc)meta_scale(md);
        const Acc bi = fma(tk, (Acc)md.av, (Acc)md.b0);
        const Acc ri = (S == NSLI_FP8E4M3) ? dot * sc - bi : dot - bi;
        const bool viol = valid && ri > Acc(0);
        const Acc cl = viol ? ((S == NSLI_FP8E4M3) ? ri * (Acc)md.inv_n2 * sc : ri * (Acc)md.inv_n2) : Acc(0);
        if (me.wt == 0 && fi == 0 && valid)
            stat.add(ri, ri * (Acc)md.inv_n, bi < Acc(0) ? -bi : bi, viol);
#pragma unroll
        for (int rr = 0; rr < RG; ++rr) {
            const Acc c = __shfl_sync(0xffffffffu, cl, rr * WL);
            if (c != Acc(0)) {
                const unsigned char *row = sb + rr * p.row_bytes;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    Acc a[EPV];
                    decode<S>(*reinterpret_cast<const uint4 *>(row + me.voff[v]), a);
#pragma unroll
                    for (int e = 0; e < EPV; e += 2)
                        fma2(yr[v][e], yr[v][e + 1], c, c, a[e], a[e + 1]);
                }
            }
        }
        if (!resident && !large) {
            __syncwarp();
            if (lane == 0 && ring_release(p, stage))
                ring_refill(p, src, q0, slot, stage);
        }
        slot += T;
        stage += T;
#pragma unroll 1
        while (stage >= p.nstage) {
            stage -= p.nstage;
            ++fill;
        }
    }
    tg += (unsigned)ng;
    return true;
}

// Initialise the ring's and the teams' barriers and fill the ring, spread over
// the block's threads.  Every thread calls it; the barriers are ready when it
// returns.
__device__ __forceinline__ void team_init(const MapArgs &p, const RingSource &src)
{
    extern __shared__ __align__(128) unsigned char smem[];
    static_assert(kMapMaxStages <= 32 * 8 && 4 * kTeamWarps <= 32 * 8, "a thread per barrier (eight warps at least)");
    const int t = threadIdx.x;
    if (t < p.nstage) {
        mbar_init(smem_u32(smem + kHFull) + 8u * t, 1u);
        reinterpret_cast<volatile int *>(smem + kHIssued)[t] = 0;
        reinterpret_cast<volatile int *>(smem + kHFreed)[t] = 0;
    }
    if (t < 4 * p.teams)
        mbar_init(smem_u32(smem + kHTeam) + 8u * t, (unsigned int)p.team_warps);
    if (t == 0)
        team_flags().abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    if (t < min(p.nstage, src.ns))
        ring_issue(p, src, t, t);
    __syncwarp();
}

// The barriers' memory is free for others again (nothing waits on them, and
// no copy is in flight); the caller synchronises before it is reused.
__device__ __forceinline__ void team_retire(const MapArgs &p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int t = threadIdx.x;
    if (t < p.nstage)
        asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(smem + kHFull) + 8u * t) : "memory");
    if (t < 4 * p.teams)
        asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(smem + kHTeam) + 8u * t) : "memory");
}

// x into this thread's slices (0 beyond the row).  With several teams every
// one needs all of x: the CTA stages it in shared memory once (the exchange
// area), 16 bytes per load, instead of reading it from L2 once per team.
template <int S, int V>
__device__ __forceinline__ void team_load_x(const MapArgs &p, const TeamThread<S, V> &me, const int nbar,
                                            typename Traits<S>::acc (&xr)[V][Traits<S>::EPV])
{
    using Acc = typename Traits<S>::acc;
    constexpr int EPV = Traits<S>::EPV;
    constexpr int NQ = EPV * (int)sizeof(Acc) / 16;   // 16-byte pieces of x per vector of A
    extern __shared__ __align__(128) unsigned char smem[];
    const uint4 *xg = static_cast<const uint4 *>(p.x);
    uint4 *xs = reinterpret_cast<uint4 *>(smem + kTeamHeader);
    if (p.teams > 1) {
        const int nq = p.nv * NQ;
#pragma unroll 1
        for (int q = threadIdx.x; q < nq; q += nbar)
            xs[q] = __ldcg(xg + q);
        bar_threads(1, nbar);
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int j = me.voff[v] >> 4;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            uint4 w = make_uint4(0u, 0u, 0u, 0u);
            if (me.vok[v] && me.team < p.teams)
                w = p.teams > 1 ? xs[j * NQ + q] : __ldcg(xg + (size_t)j * NQ + q);
            const Acc *a = reinterpret_cast<const Acc *>(&w);
#pragma unroll
            for (int e = 0; e < 16 / (int)sizeof(Acc); ++e)
                xr[v][q * (16 / (int)sizeof(Acc)) + e] = a[e];
        }
    }
}

// The CTA's sum of its teams' y (pairwise, a fixed order), written to
// part_row by team 0, and the CTA's statistics (in warp 0's `stat`).  The nbar
// mapping threads have met since the last row.  `nt`: teams that mapped rows.
template <int S, int V>
__device__ __forceinline__ void team_finish(const MapArgs &p, const TeamThread<S, V> &me, const int nbar, const int nt,
                                            typename Traits<S>::acc (&yr)[V][Traits<S>::EPV],
                                            RowStat<typename Traits<S>::acc> &stat, void *part_row)
{
    using Acc = typename Traits<S>::acc;
    constexpr int EPV = Traits<S>::EPV;
    constexpr int NQ = EPV * (int)sizeof(Acc) / 16;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tthr = p.team_warps * 32, tt = me.wt * 32 + me.lane;
    uint4 *xb = reinterpret_cast<uint4 *>(smem + kTeamHeader);
    RowStat<Acc> *ts = reinterpret_cast<RowStat<Acc> *>(smem + kHStat);
    if (me.wt == 0 && me.team < nt) {
        stat.fold();
        if (me.lane == 0)
            ts[me.team] = stat;
    }
#pragma unroll 1
    for (int t = nt; t > 1;) {
        const int h = (t + 1) / 2;
        if (t != nt)
            bar_threads(1, nbar);   // the exchange area is free
        if (me.team >= h && me.team < t) {
            uint4 *dst = xb + (size_t)(me.team - h) * (V * NQ) * tthr;
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    uint4 w;
                    Acc *a = reinterpret_cast<Acc *>(&w);
#pragma unroll
                    for (int e = 0; e < 16 / (int)sizeof(Acc); ++e)
                        a[e] = yr[v][q * (16 / (int)sizeof(Acc)) + e];
                    dst[(v * NQ + q) * tthr + tt] = w;
                }
        }
        bar_threads(1, nbar);
        if (me.team < t - h) {
            const uint4 *src = xb + (size_t)me.team * (V * NQ) * tthr;
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const uint4 w = src[(v * NQ + q) * tthr + tt];
                    const Acc *a = reinterpret_cast<const Acc *>(&w);
#pragma unroll
                    for (int e = 0; e < 16 / (int)sizeof(Acc); ++e)
                        yr[v][q * (16 / (int)sizeof(Acc)) + e] += a[e];
                }
        }
        t = h;
    }
    if (me.team == 0) {
        uint4 *py = static_cast<uint4 *>(part_row);
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (me.vok[v]) {
                const int j = me.voff[v] >> 4;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    uint4 w;
                    Acc *a = reinterpret_cast<Acc *>(&w);
#pragma unroll
                    for (int e = 0; e < 16 / (int)sizeof(Acc); ++e)
                        a[e] = yr[v][q * (16 / (int)sizeof(Acc)) + e];
                    py[(size_t)j * NQ + q] = w;
                }
            }
    }
    bar_threads(1, nbar);   // (also orders the team statistics)
    if (threadIdx.x < 32 && nt > 1) {   // (one team: warp 0 has them already)
        stat.clear();
        if ((int)threadIdx.x < nt)
            stat = ts[threadIdx.x];
        stat.fold();
    }
}

// An instance: storage, vectors per thread, rows per group.
template <int S, int V, int RG> struct MapForm {};

// One block of rows [row_begin, row_begin + nrows) by the whole CTA, the ring
// set up for it: the sum of its positive slices to part_row, its statistics
// to *stat_out.  Every thread of the block calls it; ends synchronised.
template <int S, int V, int RG>
__device__ __forceinline__ void map_body(MapForm<S, V, RG>, const MapArgs &p, const long long row_begin,
                                         const int nrows, void *part_row, PartStat *stat_out, const int skip)
{
    using Acc = typename Traits<S>::acc;
    constexpr int EPV = Traits<S>::EPV;
    const int nbar = (int)blockDim.x;
    const RingSource src = ring_source(p, row_begin, nrows, 1, skip);
    team_init(p, src);
    TeamThread<S, V> me;
    me.init(p);
    Acc xr[V][EPV], yr[V][EPV];
    team_load_x<S, V>(p, me, nbar, xr);
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int e = 0; e < EPV; ++e)
            yr[v][e] = Acc(0);
    RowStat<Acc> stat;
    stat.clear();
    const Acc tk = (Acc)((double)p.st->tick * p.st->rho);
    unsigned int tg = 0;
    Refill pend;
    if (me.team < p.teams)
        team_rows<S, V, RG>(p, me, src, 0u, false, tg, xr, yr, tk, stat, pend);
    bar_threads(1, nbar);
    team_finish<S, V>(p, me, nbar, min(p.teams, src.ns), yr, stat, part_row);
    if (threadIdx.x == 0)
        *stat_out = stat.record();
    __syncthreads();
    if (*(volatile int *)&team_flags().abort) {
        // a wait expired: record it, and leave with no copy in flight
        if (threadIdx.x == 0) {
            atomicOr(&p.st->error, ERRF_TIMEOUT);
            ring_drain(p);
        }
        __syncthreads();
    }
    team_retire(p);
}

// most rows per group of the instances with V vectors per thread (the fixed
// cost of a group's fold and barrier is shared by its rows): eight for one
// vector with binary32 sums (short rows on one team), fewer where the sums of
// more rows would not fit the registers beside the slices of x and y
__host__ __device__ constexpr int kRgMax(int v, int acc_bytes)
{
    return v >= 4 ? 2 : (v >= 2 || acc_bytes > 4 ? 4 : 8);
}

// instances of a kernel (F::get): S x vectors per thread x rows per group
template <int S, int V, typename F> const void *dense_fn_v(int rg)
{
    if (rg == 1)
        return F::template get<S, V, 1>();
    if (rg == 2)
        return F::template get<S, V, 2>();
    constexpr int most = kRgMax(V, (int)sizeof(typename Traits<S>::acc));
    if constexpr (most >= 4) {
        if (rg == 4)
            return F::template get<S, V, 4>();
    }
    if constexpr (most >= 8) {
        if (rg == 8)
            return F::template get<S, V, 8>();
    }
    return nullptr;
}
template <int S, typename F> const void *dense_fn_s(int vpt, int rg)
{
    switch (vpt) {
    case 1: return dense_fn_v<S, 1, F>(rg);
    case 2: return dense_fn_v<S, 2, F>(rg);
    case 4:
        if constexpr (S != NSLI_FP8E4M3)
            return dense_fn_v<S, 4, F>(rg);
        return nullptr;
    case 8:
        if constexpr (S == NSLI_F64 || S == NSLI_F32)
            return dense_fn_v<S, 8, F>(rg);
        return nullptr;
    default: return nullptr;
    }
}
template <typename F> const void *dense_fn(int storage, int vpt, int rg)
{
    switch (storage) {
    case NSLI_F64: return dense_fn_s<NSLI_F64, F>(vpt, rg);
    case NSLI_F32: return dense_fn_s<NSLI_F32, F>(vpt, rg);
    case NSLI_BF16: return dense_fn_s<NSLI_BF16, F>(vpt, rg);
    case NSLI_FP8E4M3: return dense_fn_s<NSLI_FP8E4M3, F>(vpt, rg);
    default: return nullptr;
    }
}
// the limit belongs to the kernel, not to a handle: always the largest, so a
// handle with a small ring does not lower it under another's
inline cudaError_t set_smem(const void *fn)
{
    if (!fn)
        return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
}

}  // namespace

}  // namespace nsli
