// nsli_kernels.cu -- device code of the pseudo-projection solver (sm_103a).
//
// Kernels of one iteration (Sokolinsky & Sokolinskaya 2020):
//   Map            Map of Eq. 13 fused with the CTA-level Reduce(+): streams
//                  the CTA's contiguous block of rows of A once through a
//                  shared-memory ring filled by the bulk-copy (TMA) engine,
//                  forms r_i = <a_i, x> - b_i(k) with b_i(k) = b0_i + k rho Av_i
//                  (Section 5 tick, never materialised), and while the row is
//                  still on chip adds the positive slice (Eq. 7)
//                  r_i / ||a_i||^2 * a_i into register-resident partial sums
//                  (rows up to the register-resident limit: nsli_team.cuh;
//                  longer rows: below).
//   reduce_update  deterministic fixed-order sum of the per-CTA partials,
//                  the stopping test (Eq. 10 and the step rule), and the step
//                  x <- x - lambda y / h (Eq. 8) or x <- x - lambda y / ||y||
//                  (Eq. 12), with ||dx|| in binary64.
// Plus the set-up kernels (quantisation of A, binary64 row norms, per-row
// records) and the binary64 feasibility check (Eq. 10 on the stored A).
#include "nsli_team.cuh"
#include "nsli_sumsq.cuh"

namespace nsli {

namespace {

// One problem: CTA b maps its contiguous balanced block of rows.
template <int S, int V, int RG> __global__ void __launch_bounds__(kMapMaxConsumers, 1) map_kernel(const MapArgs p)
{
    using Acc = typename Traits<S>::acc;
    if (!p.ignore_done && *(volatile int *)&p.st->done)
        return;
    const long long b = blockIdx.x;
    const long long row_begin = b * p.rows_base + (b < p.rows_rem ? b : (long long)p.rows_rem);
    const int nrows = (int)(p.rows_base + (b < p.rows_rem ? 1 : 0));
    map_body(MapForm<S, V, RG>{}, p, row_begin, nrows, static_cast<Acc *>(p.part_y) + b * p.ld,
             p.part_stat + b, b == 0 ? p.skip_slot : -1);
}

struct MapFn {
    template <int S, int V, int RG> static const void *get() { return (const void *)map_kernel<S, V, RG>; }
};

}  // namespace

// --------------------------------------------------- Map, long rows --------
//
// Rows longer than the register-resident limit (n > 16384 for 4-, 2- and
// 1-byte storage, n > 8192 for binary64).  The CTA takes its rows RG at a
// time and walks them in column chunks of 512 * 8 / RG 16-byte vectors:
// thread t owns vectors t, t + 512, ... of every chunk.  Pass 1 streams the chunk of
// the RG rows from HBM with 16-byte loads and accumulates the dots against
// the chunk of x (loaded once per group, 16 bytes at a time); one block
// reduction gives the RG residuals.  A thread owns 8 / RG vectors per chunk,
// so every thread has 8 row vectors in flight whatever RG is.  Pass 2 re-reads the chunks of the violated rows and adds
// r_i / ||a_i||^2 * a_i into the CTA's row of partial sums, each thread its
// own columns (no atomics, a fixed order).  The host picks RG (4, 2 or 1) so
// that the rows of a group, over all CTAs, stay within a budget of L2 until
// pass 2 re-reads them, and keeps the partial sums in shared memory (SY)
// when a row of them fits there; otherwise they live in global memory.
constexpr int kLongThreads = 512;

// x entries of one 16-byte vector of A, loaded 16 bytes at a time
template <typename Acc, int EPV> __device__ __forceinline__ void load_x_vec(const Acc *xg, long long j, Acc (&xv)[EPV])
{
    const uint4 *src = reinterpret_cast<const uint4 *>(xg + j * EPV);
    constexpr int NQ = EPV * (int)sizeof(Acc) / 16;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const uint4 w = __ldg(src + q);
        const Acc *a = reinterpret_cast<const Acc *>(&w);
#pragma unroll
        for (int e = 0; e < 16 / (int)sizeof(Acc); ++e)
            xv[q * (16 / (int)sizeof(Acc)) + e] = a[e];
    }
}

template <int S, int RG, bool SY>
__global__ void __launch_bounds__(kLongThreads, 1) map_long_kernel(const MapArgs p)
{
    using Tr = Traits<S>;
    using Acc = typename Tr::acc;
    using Meta = typename Tr::meta;
    constexpr int EPV = Tr::EPV;
    constexpr int W = 32 / RG;
    // vectors per thread per chunk: 8 row vectors in flight per thread
    // whatever the group size
    constexpr int kLongVPT = 8 / RG;

    DevState *st = p.st;
    if (!p.ignore_done && *(volatile int *)&st->done)
        return;
    __shared__ Acc red[2][RG][32];
    extern __shared__ __align__(16) unsigned char long_smem[];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nwarps = kLongThreads / 32;
    const long long b = blockIdx.x;
    const long long row_begin = b * p.rows_base + (b < p.rows_rem ? b : (long long)p.rows_rem);
    const long long row_end = row_begin + p.rows_base + (b < p.rows_rem ? 1 : 0);
    const long long nv = p.nv;
    const long long chunk = (long long)kLongThreads * kLongVPT;
    const int nchunks = (int)((nv + chunk - 1) / chunk);
    const unsigned char *Ab = static_cast<const unsigned char *>(p.A);
    const Meta *meta = static_cast<const Meta *>(p.meta);
    const Acc *xg = static_cast<const Acc *>(p.x);
    Acc *py_g = static_cast<Acc *>(p.part_y) + b * p.ld;
    Acc *py = SY ? reinterpret_cast<Acc *>(long_smem) : py_g;
    for (long long e = tid; e < p.ld; e += kLongThreads)
        py[e] = Acc(0);
    const Acc tk = (Acc)((double)st->tick * st->rho);

    long long h_loc = 0;
    Acc mv = neg_inf<Acc>(), mn = neg_inf<Acc>(), mb = Acc(0);
    int grp_counter = 0;
    for (long long r0 = row_begin; r0 < row_end; r0 += RG) {
        const int gr = (int)((row_end - r0) < RG ? (row_end - r0) : RG);
        Acc pe[RG], po[RG];
#pragma unroll
        for (int rr = 0; rr < RG; ++rr) {
            pe[rr] = Acc(0);
            po[rr] = Acc(0);
        }
        // ---- pass 1: dots of the group's rows, chunk by chunk
        for (int c = 0; c < nchunks; ++c) {
            long long j[kLongVPT];
            bool ok[kLongVPT];
            Acc xv[kLongVPT][EPV];
            uint4 q[RG][kLongVPT];
#pragma unroll
            for (int v = 0; v < kLongVPT; ++v) {
                j[v] = (long long)c * chunk + tid + v * kLongThreads;
                ok[v] = j[v] < nv;
#pragma unroll
                for (int rr = 0; rr < RG; ++rr)
                    q[rr][v] = (ok[v] && rr < gr)
                                   ? __ldg(reinterpret_cast<const uint4 *>(Ab + (r0 + rr) * (long long)p.row_bytes) + j[v])
                                   : make_uint4(0u, 0u, 0u, 0u);
                if (ok[v]) {
                    load_x_vec<Acc, EPV>(xg, j[v], xv[v]);
                } else {
#pragma unroll
                    for (int e = 0; e < EPV; ++e)
                        xv[v][e] = Acc(0);
                }
            }
#pragma unroll
            for (int rr = 0; rr < RG; ++rr) {
#pragma unroll
                for (int v = 0; v < kLongVPT; ++v) {
                    Acc a[EPV];
                    decode<S>(q[rr][v], a);
#pragma unroll
                    for (int e = 0; e < EPV; e += 2)
                        fma2(pe[rr], po[rr], a[e], a[e + 1], xv[v][e], xv[v][e + 1]);
                }
            }
        }
        Acc acc[RG];
#pragma unroll
        for (int rr = 0; rr < RG; ++rr)
            acc[rr] = pe[rr] + po[rr];
        Acc *rb = &red[grp_counter & 1][0][0];
        const Acc wsum = warp_fold_rows<RG>(acc, lane);
        if ((lane & (W - 1)) == 0)
            rb[(lane / W) * 32 + warp] = wsum;
        __syncthreads();
        Acc tsum = Acc(0);
        {
            const int qq = lane / W, i = lane % W;
            for (int w = i; w < nwarps; w += W)
                tsum += rb[qq * 32 + w];
#pragma unroll
            for (int off = W / 2; off > 0; off >>= 1)
                tsum += __shfl_xor_sync(0xffffffffu, tsum, off);
        }
        Acc cr[RG];
        bool any = false;
#pragma unroll
        for (int rr = 0; rr < RG; ++rr) {
            const Acc dot = __shfl_sync(0xffffffffu, tsum, rr * W);
            const bool valid = rr < gr;
            const Meta md = meta[r0 + (valid ? rr : 0)];
            const Acc sc = (Acc)meta_scale(md);
            const Acc bi = fma(tk, (Acc)md.av, (Acc)md.b0);
            const Acc ri = (S == NSLI_FP8E4M3) ? dot * sc - bi : dot - bi;
            const bool viol = valid && ri > Acc(0);
            cr[rr] = viol ? ((S == NSLI_FP8E4M3) ? ri * (Acc)md.inv_n2 * sc : ri * (Acc)md.inv_n2) : Acc(0);
            any = any || viol;
            if (warp == 0 && valid) {
                h_loc += viol ? 1 : 0;
                mv = ri > mv ? ri : mv;
                const Acc rn = ri * (Acc)md.inv_n;
                mn = rn > mn ? rn : mn;
                const Acc ab = bi < Acc(0) ? -bi : bi;
                mb = ab > mb ? ab : mb;
            }
        }
        // ---- pass 2: add the violated rows' slices (rows re-read from L2)
        if (any) {
            for (int c = 0; c < nchunks; ++c) {
#pragma unroll
                for (int v = 0; v < kLongVPT; ++v) {
                    const long long jj = (long long)c * chunk + tid + v * kLongThreads;
                    if (jj >= nv)
                        continue;
                    Acc y[EPV];
#pragma unroll
                    for (int e = 0; e < EPV; ++e)
                        y[e] = py[jj * EPV + e];
#pragma unroll
                    for (int rr = 0; rr < RG; ++rr) {
                        if (cr[rr] != Acc(0)) {
                            Acc a[EPV];
                            decode<S>(__ldg(reinterpret_cast<const uint4 *>(Ab + (r0 + rr) * (long long)p.row_bytes) + jj), a);
#pragma unroll
                            for (int e = 0; e < EPV; e += 2)
                                fma2(y[e], y[e + 1], cr[rr], cr[rr], a[e], a[e + 1]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < EPV; ++e)
                        py[jj * EPV + e] = y[e];
                }
            }
        }
        ++grp_counter;
    }
    if (SY) {
        // each thread wrote only its own columns; the copy-out mixes them
        __syncthreads();
        for (long long e = tid; e < p.ld; e += kLongThreads)
            py_g[e] = py[e];
    }
    if (tid == 0) {
        PartStat ps;
        ps.h = h_loc;
        ps.maxviol = (double)mv;
        ps.maxnorm = (double)mn;
        ps.maxb = (double)mb;
        p.part_stat[b] = ps;
    }
}

// ------------------------------------------ Map, long rows on a cluster ----
//
// A thread-block cluster of C CTAs (C = 2, 4 or 8, one per SM) maps a block
// of rows whose columns it splits: CTA q of the cluster owns the vectors
// [q S, (q + 1) S) of every row (S = slice_nv), keeps the matching slices of
// x and of the cluster's partial y in registers, and streams its slice of
// each row through its own ring of bulk copies (one row slice and the row's
// record per stage).  Per row every CTA forms its partial dot (thread
// chains, warp butterfly, the warps' sums in order), writes it into slot q
// of the row's exchange buffer in EVERY CTA of the cluster (distributed
// shared memory) and arrives on that CTA's exchange barrier; each CTA then
// adds the C partials in rank order, so all of them hold the same r_i, and
// adds the violated row's slice from its own shared-memory copy.  A is read
// from HBM once, with no second pass.  The exchange of row k is waited for
// D rows later (D = cluster_lag, 1..3), while the dots of rows k+1 .. k+D
// run, so the exchange latency is not on the critical path.  Eight exchange
// buffers suffice: a CTA sends row k only after every CTA sent row k - D,
// i.e. after every CTA finished reading rows up to k - 2D - 1, and
// 8 >= 2D + 1.  A row's stage is refilled as soon as every mapping warp has
// finished the row (an "empty" barrier per stage that the warps arrive on
// and the exchange warp waits for), so the ring holds the D + 1 rows in use
// and the rest of its stages are in flight.  Every wait is bounded; all CTAs
// of a cluster meet at a cluster barrier before they exit, so no CTA's
// shared memory is written after it has gone.
__device__ __forceinline__ unsigned int cluster_rank()
{
    unsigned int r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned int map_to_rank(unsigned int addr, unsigned int rank)
{
    unsigned int r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_remote(unsigned int raddr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(raddr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_remote(unsigned int raddr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(raddr), "d"(v) : "memory");
}
__device__ __forceinline__ void arrive_remote(unsigned int rbar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(rbar) : "memory");
}
__device__ __forceinline__ bool mbar_test_cluster(unsigned int bar, unsigned int parity)
{
    unsigned int ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster_bounded(unsigned int bar, unsigned int parity)
{
    const long long t0 = clock64();
    for (unsigned int it = 0;; ++it) {
        if (mbar_test_cluster(bar, parity))
            return true;
        if ((it & 255u) == 255u && clock64() - t0 > kWaitLimitCycles)
            return false;
    }
}

// shared-memory header of the cluster Map (within kSmemHeader)
constexpr int kClXB = 8;          // exchange buffers (group k uses k % 8)
constexpr int kClMaxStages = 16;  // ring stages (one row slice each)
constexpr int kClFull = 0;        // 16 full barriers (stages)
constexpr int kClXbar = 128;      // 8 exchange barriers
constexpr int kClEmpty = 192;     // 16 empty barriers (stages)
constexpr int kClRed = 512;       // [2][RG][16] warp sums (at most 512 bytes)
constexpr int kClXch = 1024;      // [8][RG][8] exchanged partial dots (at most 1024 bytes)
static_assert(kClEmpty + kClMaxStages * 8 <= kClRed, "cluster Map barriers fit");
static_assert(kClXch + 1024 <= kSmemHeader, "cluster Map header fits");

// 512 threads map; a 17th warp (the exchange warp) issues the bulk copies,
// waits for the exchanges, adds the warps' sums and sends the partial dots,
// so the latency of the remote stores and releases is off the mapping
// warps' path (they only meet it at the per-group block barrier).
constexpr int kClusterCompute = 512;
constexpr int kClusterThreads = kClusterCompute + 32;

// RG = rows per group (1, 2 or 4): the rows of a group share one block
// barrier and one exchange message, and their dependent chains interleave.  The
// arithmetic of every row is the same for all (the warp fold of two rows
// adds the same operands in the same tree as one warp butterfly per row,
// and rows enter y in row order).
// Bound: HBM for binary32; for bf16 and FP8 the mapping warps' instructions
// per group.  A group's dots have no branch between its rows, its residuals
// are taken once per row (a lane group each) instead of once per lane, and
// ring positions are counted along: six remainders by a run-time stage count
// had taken a third of the instructions.  Map of 27000 x 54000, before ->
// with these: binary32 1.069 -> 1.036 ms, bf16 0.800 -> 0.668 ms (4.4 TB/s), FP8
// 0.700 -> 0.550 ms.
template <int S, int VPT, int RG>
__global__ void __launch_bounds__(kClusterThreads, 1) map_cluster_kernel(const MapArgs p)
{
    static_assert(RG == 1 || RG == 2 || RG == 4, "one, two or four rows per group");
    static_assert(2 * RG * 16 * sizeof(typename Traits<S>::acc) <= kClXch - kClRed, "warp sums fit");
    static_assert(kClXB * RG * 8 * sizeof(typename Traits<S>::acc) <= 1024, "exchange buffers fit");
    using Tr = Traits<S>;
    using Acc = typename Tr::acc;
    using Meta = typename Tr::meta;
    constexpr int EPV = Tr::EPV;
    constexpr int NCW = kClusterCompute / 32;   // mapping warps

    DevState *st = p.st;
    if (!p.ignore_done && *(volatile int *)&st->done)
        return;   // the same for every CTA of the grid
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned long long *full = reinterpret_cast<unsigned long long *>(smem + kClFull);
    unsigned long long *xbar = reinterpret_cast<unsigned long long *>(smem + kClXbar);
    unsigned long long *empty = reinterpret_cast<unsigned long long *>(smem + kClEmpty);
    Acc *xch = reinterpret_cast<Acc *>(smem + kClXch);   // [group % 8][row][rank]
    Acc *red = reinterpret_cast<Acc *>(smem + kClRed);   // [group & 1][row][warp]
    unsigned char *stages = smem + kSmemHeader;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool xw = warp == NCW;                 // the exchange warp
    const bool leader = xw && lane == 0;
    const int C = p.cluster;
    const unsigned int rank = cluster_rank();
    const long long cl = blockIdx.x / C;
    const long long row_begin = cl * p.rows_base + (cl < p.rows_rem ? cl : (long long)p.rows_rem);
    const long long row_end = row_begin + p.rows_base + (cl < p.rows_rem ? 1 : 0);
    const int nrows = (int)(row_end - row_begin);
    const int ngroups = (nrows + RG - 1) / RG;
    const long long v0 = (long long)rank * p.slice_nv;
    const int my_nv = (int)max(0ll, min((long long)p.slice_nv, (long long)p.nv - v0));
    const unsigned int slice_bytes = (unsigned int)my_nv * 16u;
    const unsigned int meta_off = (unsigned int)p.slice_nv * 16u;   // record after the largest slice
    const unsigned char *Ab = static_cast<const unsigned char *>(p.A);
    const unsigned char *Mb = static_cast<const unsigned char *>(p.meta);

    // ring positions are counted along (a remainder by the stage count, which
    // the compiler does not know, costs some twenty instructions)
    auto wrap = [&](int stage) { return stage >= p.nstage ? stage - p.nstage : stage; };
    int istage = 0;             // the issuing thread: the next stage to fill
    auto issue = [&](int s) {   // row s of the block into its stage
        const int stage = istage;
        istage = wrap(istage + 1);
        const long long row = row_begin + s;
        unsigned char *dst = stages + (size_t)stage * p.stage_stride;
        const unsigned int fb = smem_u32(&full[stage]);
        mbar_expect_tx(fb, slice_bytes + 32u);
        if (slice_bytes)
            bulk_g2s(smem_u32(dst), Ab + row * (long long)p.row_bytes + v0 * 16, slice_bytes, fb);
        bulk_g2s(smem_u32(dst + meta_off), Mb + row * 32, 32u, fb);
    };

    if (tid == 0) {
        for (int q = 0; q < p.nstage; ++q) {
            mbar_init(smem_u32(&full[q]), 1u);
            mbar_init(smem_u32(&empty[q]), (unsigned int)NCW);
        }
        for (int q = 0; q < kClXB; ++q)
            mbar_init(smem_u32(&xbar[q]), (unsigned int)C);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    cluster_sync_all();   // every exchange barrier of the cluster is initialised
    int issued = 0;
    if (leader) {
        const int first = nrows < p.nstage ? nrows : p.nstage;
        for (int q = 0; q < first; ++q)
            issue(q);
        issued = first;
    }

    int voff[VPT];
    bool vok[VPT];
    Acc xr[VPT][EPV], yr[VPT][EPV];
    {
        const Acc *xg = static_cast<const Acc *>(p.x);
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const int j = tid + v * kClusterCompute;
            vok[v] = !xw && j < my_nv;
            voff[v] = vok[v] ? j * 16 : 0;   // beyond the slice: its first vector against x = 0
#pragma unroll
            for (int e = 0; e < EPV; ++e) {
                xr[v][e] = vok[v] ? xg[(v0 + j) * EPV + e] : Acc(0);
                yr[v][e] = Acc(0);
            }
        }
    }
    const Acc tk = (Acc)((double)st->tick * st->rho);
    long long h_loc = 0;
    Acc mv = neg_inf<Acc>(), mn = neg_inf<Acc>(), mb = Acc(0);
    int aborted = 0, at = 0, stalled = 0;

    const int D = p.cluster_lag;
    int dstage = 0, sstage = 0;     // stages of the group being dotted, and being finished
    unsigned int dph = 0, sph = 0;  // fills of those stages
    for (int g = 0; g < ngroups + D; ++g) {
        int flag = 0;
        if (g < ngroups && !xw) {
            // partial dots of the group's rows: side by side, without
            // branches between them (a short last group repeats its last row,
            // masked below), two chains of FMAs per row where a thread has
            // four vectors or more
            const int last = min(RG, nrows - g * RG) - 1;
            const unsigned char *row[RG];
#pragma unroll
            for (int rr = 0; rr < RG; ++rr) {
                const int at_rr = dstage + min(rr, last);
                const int stage = wrap(at_rr);
                if (!mbar_wait_bounded(smem_u32(&full[stage]), (dph + (at_rr >= p.nstage ? 1u : 0u)) & 1u))
                    flag = 1;
                row[rr] = stages + (size_t)stage * p.stage_stride;
            }
            constexpr int NCH = VPT == 4 ? 2 : 1;
            Acc acc[RG];
#pragma unroll
            for (int rr = 0; rr < RG; ++rr) {
                Acc pe[NCH], po[NCH];
#pragma unroll
                for (int q = 0; q < NCH; ++q) {
                    pe[q] = Acc(0);
                    po[q] = Acc(0);
                }
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    Acc a[EPV];
                    decode<S>(*reinterpret_cast<const uint4 *>(row[rr] + voff[v]), a);
#pragma unroll
                    for (int e = 0; e < EPV; e += 2)
                        fma2(pe[v % NCH], po[v % NCH], a[e], a[e + 1], xr[v][e], xr[v][e + 1]);
                }
                acc[rr] = pe[0] + po[0];
#pragma unroll
                for (int q = 1; q < NCH; ++q)
                    acc[rr] += pe[q] + po[q];
            }
            const Acc ws = warp_fold_rows<RG>(acc, lane);   // lanes [16q, 16q + 16) end with row q
            if ((lane & (32 / RG - 1)) == 0)
                red[(g & 1) * (RG * 16) + (lane / (32 / RG)) * 16 + warp] = ws;
            dstage += RG;
            if (dstage >= p.nstage) {
                dstage -= p.nstage;
                ++dph;
            }
        }
        if (leader && g >= D) {
            const int t = g - D;
            if (stalled || !mbar_wait_cluster_bounded(smem_u32(&xbar[t % kClXB]), (unsigned int)((t / kClXB) & 1)))
                flag = 1;
        }
        aborted = bar_all_or((int)blockDim.x, flag);
        at = g;
        if (aborted)
            break;
        if (xw) {
            if (g < ngroups) {
                // the mapping warps' sums in a fixed butterfly, 32 at a time
                // (rows 2h and 2h + 1 in lanes [0, 16) and [16, 32) of
                // chunk h); lane q sends this CTA's partial dots of the
                // group to CTA q
                constexpr int NCHK = RG >= 2 ? RG / 2 : 1;
                Acc rowv[RG];
#pragma unroll
                for (int h = 0; h < NCHK; ++h) {
                    Acc tot = (RG >= 2 || lane < NCW) ? red[(g & 1) * (RG * 16) + h * 32 + lane] : Acc(0);
#pragma unroll
                    for (int off = 8; off > 0; off >>= 1)
                        tot += __shfl_xor_sync(0xffffffffu, tot, off);
                    rowv[(2 * h) % RG] = __shfl_sync(0xffffffffu, tot, 0);
                    if constexpr (RG >= 2)
                        rowv[2 * h + 1] = __shfl_sync(0xffffffffu, tot, 16);
                }
                if (lane < C) {
                    const unsigned int la = smem_u32(&xch[(g % kClXB) * (RG * 8) + rank]);
                    const unsigned int lb = smem_u32(&xbar[g % kClXB]);
#pragma unroll
                    for (int r = 0; r < RG; ++r)
                        st_remote(map_to_rank(la + (unsigned int)(r * 8 * sizeof(Acc)), (unsigned int)lane), rowv[r]);
                    arrive_remote(map_to_rank(lb, (unsigned int)lane));
                }
            }
            if (lane == 0 && g >= D) {
                // refill the stages of group g - D once every mapping warp
                // has finished it (in this iteration, below)
                const int t = g - D;
                for (int rr = 0; rr < RG && !stalled; ++rr) {
                    const int r = t * RG + rr, at_rr = sstage + rr;
                    if (r >= nrows || issued >= nrows)
                        break;
                    if (mbar_wait_bounded(smem_u32(&empty[wrap(at_rr)]),
                                          (sph + (at_rr >= p.nstage ? 1u : 0u)) & 1u)) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        issue(issued);
                        ++issued;
                    } else {
                        atomicOr(&st->error, ERRF_TIMEOUT);   // the next barrier ends the loop
                        stalled = 1;
                    }
                }
            }
        } else if (g >= D) {
            // the group's residuals and coefficients, row fq in the lanes of
            // group fq, then the slices row after row
            const int t = g - D;
            constexpr int WL = 32 / RG;
            const int fq = lane / WL;
            const int cnt = min(RG, nrows - t * RG);
            const bool valid = fq < cnt;
            const Acc *xc = xch + (t % kClXB) * (RG * 8) + fq * 8;
            Acc dot = Acc(0);
            for (int q = 0; q < C; ++q)
                dot += xc[q];
            const int mine = wrap(sstage + (valid ? fq : 0));
            const Meta md = *reinterpret_cast<const Meta *>(stages + (size_t)mine * p.stage_stride + meta_off);
            const Acc sc = (Acc)meta_scale(md);
            const Acc bi = fma(tk, (Acc)md.av, (Acc)md.b0);
            const Acc ri = (S == NSLI_FP8E4M3) ? dot * sc - bi : dot - bi;
            const bool viol = valid && ri > Acc(0);
            const Acc cl = viol ? ((S == NSLI_FP8E4M3) ? ri * (Acc)md.inv_n2 * sc : ri * (Acc)md.inv_n2) : Acc(0);
            if (warp == 0 && valid) {   // (the lanes of a row alike; one of each is counted at the end)
                h_loc += viol ? 1 : 0;
                mv = ri > mv ? ri : mv;
                const Acc rn = ri * (Acc)md.inv_n;
                mn = rn > mn ? rn : mn;
                const Acc ab = bi < Acc(0) ? -bi : bi;
                mb = ab > mb ? ab : mb;
            }
#pragma unroll
            for (int rr = 0; rr < RG; ++rr) {
                const Acc c = __shfl_sync(0xffffffffu, cl, rr * WL);
                if (c != Acc(0)) {
                    const unsigned char *row = stages + (size_t)wrap(sstage + rr) * p.stage_stride;
#pragma unroll
                    for (int v = 0; v < VPT; ++v) {
                        Acc a[EPV];
                        decode<S>(*reinterpret_cast<const uint4 *>(row + voff[v]), a);
#pragma unroll
                        for (int e = 0; e < EPV; e += 2)
                            fma2(yr[v][e], yr[v][e + 1], c, c, a[e], a[e + 1]);
                    }
                }
            }
            __syncwarp();
            if (lane < cnt)
                mbar_arrive(smem_u32(&empty[wrap(sstage + lane)]));   // these rows' stages are free
        }
        if (g >= D) {
            sstage += RG;
            if (sstage >= p.nstage) {
                sstage -= p.nstage;
                ++sph;
            }
        }
    }

    if (aborted) {
        // record the error; wait (bounded) for this CTA's copies in flight
        // (rows before the aborted group were waited for already)
        if (leader) {
            atomicOr(&st->error, ERRF_TIMEOUT);
            const int first = at * RG < nrows ? at * RG : nrows;
            for (int q = first; q < issued; ++q)
                mbar_wait_bounded(smem_u32(&full[q % p.nstage]), (unsigned int)((q / p.nstage) & 1));
        }
    } else {
        Acc *py = static_cast<Acc *>(p.part_y) + cl * p.ld + v0 * EPV;
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            if (vok[v]) {
                const long long j = tid + v * (long long)kClusterCompute;
#pragma unroll
                for (int e = 0; e < EPV; ++e)
                    py[j * EPV + e] = yr[v][e];
            }
        }
        if (warp == 0) {
            // one lane of each row group (0, 32 / RG, ...)
#pragma unroll 1
            for (int off = 32 / RG; off < 32; off <<= 1) {
                h_loc += __shfl_xor_sync(0xffffffffu, h_loc, off);
                const Acc a = __shfl_xor_sync(0xffffffffu, mv, off), b = __shfl_xor_sync(0xffffffffu, mn, off),
                          c = __shfl_xor_sync(0xffffffffu, mb, off);
                mv = a > mv ? a : mv;
                mn = b > mn ? b : mn;
                mb = c > mb ? c : mb;
            }
        }
        if (tid == 0 && rank == 0) {
            PartStat ps;
            ps.h = h_loc;
            ps.maxviol = (double)mv;
            ps.maxnorm = (double)mn;
            ps.maxb = (double)mb;
            p.part_stat[cl] = ps;
        }
    }
    __syncthreads();
    cluster_sync_all();   // no CTA leaves while a peer may still write to it
}

// instances up to the register-resident limit of the storage type (8, 8,
// 4, 2 vectors per thread for binary64, binary32, bf16, fp8)
template <int S> constexpr int cluster_vpt_max() { return S == NSLI_BF16 ? 4 : (S == NSLI_FP8E4M3 ? 2 : 8); }
// rows per group: up to four for FP8 and two for bf16 (short row slices,
// whose fixed cost per group would otherwise dominate); binary64 and
// binary32 take one
template <int S> constexpr int cluster_rg_max() { return S == NSLI_FP8E4M3 ? 4 : (S == NSLI_BF16 ? 2 : 1); }
template <int S, int RG> const void *cluster_fn_v(int vpt)
{
    if (vpt == 1)
        return (const void *)map_cluster_kernel<S, 1, RG>;
    if (vpt == 2)
        return (const void *)map_cluster_kernel<S, 2, RG>;
    if constexpr (cluster_vpt_max<S>() >= 4) {
        if (vpt == 4)
            return (const void *)map_cluster_kernel<S, 4, RG>;
    }
    if constexpr (cluster_vpt_max<S>() >= 8) {
        if (vpt == 8)
            return (const void *)map_cluster_kernel<S, 8, RG>;
    }
    return nullptr;
}
template <int S> const void *cluster_fn_s(int vpt, int rg)
{
    if (rg == 1)
        return cluster_fn_v<S, 1>(vpt);
    if constexpr (cluster_rg_max<S>() >= 4) {
        if (rg == 4)
            return cluster_fn_v<S, 4>(vpt);
    }
    if constexpr (cluster_rg_max<S>() >= 2) {
        if (rg == 2)
            return cluster_fn_v<S, 2>(vpt);
    }
    return nullptr;
}
const void *cluster_fn(int storage, int vpt, int rg)
{
    if (vpt > map_vpt_limit(storage))
        return nullptr;
    switch (storage) {
    case NSLI_F64: return cluster_fn_s<NSLI_F64>(vpt, rg);
    case NSLI_F32: return cluster_fn_s<NSLI_F32>(vpt, rg);
    case NSLI_BF16: return cluster_fn_s<NSLI_BF16>(vpt, rg);
    case NSLI_FP8E4M3: return cluster_fn_s<NSLI_FP8E4M3>(vpt, rg);
    default: return nullptr;
    }
}

template <int S, int RG, bool SY> const void *long_fn_rg() { return (const void *)map_long_kernel<S, RG, SY>; }
template <int S> const void *long_fn_s(int rg, bool sy)
{
    if (sy)
        return rg == 4 ? long_fn_rg<S, 4, true>() : (rg == 2 ? long_fn_rg<S, 2, true>() : long_fn_rg<S, 1, true>());
    return rg == 4 ? long_fn_rg<S, 4, false>() : (rg == 2 ? long_fn_rg<S, 2, false>() : long_fn_rg<S, 1, false>());
}
// the long-row instance for a storage type, rows per group and y placement
const void *long_fn(int storage, int rg, bool sy)
{
    if (rg != 1 && rg != 2 && rg != 4)
        return nullptr;
    switch (storage) {
    case NSLI_F64: return long_fn_s<NSLI_F64>(rg, sy);
    case NSLI_F32: return long_fn_s<NSLI_F32>(rg, sy);
    case NSLI_BF16: return long_fn_s<NSLI_BF16>(rg, sy);
    case NSLI_FP8E4M3: return long_fn_s<NSLI_FP8E4M3>(rg, sy);
    default: return nullptr;
    }
}

// ---------------------------------------------------- reduce and update ----

template <typename Acc>
__global__ void __launch_bounds__(256) reduce_update_kernel(const ReduceArgs p)
{
    __shared__ ReduceShared sh;
    reduce_body<Acc>(p, blockIdx.x, gridDim.x, sh, threadIdx.x, -1);
}

// Many problems in one launch: block b serves (problem, column block) tab[b].
template <typename Acc>
__global__ void __launch_bounds__(256) reduce_group_kernel(const GroupProblem *probs, const GroupRed *tab)
{
    __shared__ ReduceShared sh;
    const GroupRed t = tab[blockIdx.x];
    const GroupProblem &gp = probs[t.prob];
    reduce_body<Acc>(gp.red, t.blk, gp.red_blocks, sh, threadIdx.x, -1);
}

// Map + Reduce without a step (diagnostics and parity): y in binary64.
template <typename Acc>
__global__ void __launch_bounds__(256) reduce_only_kernel(const ReduceArgs p, double *y_out)
{
    __shared__ ReduceShared sh;
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const long long j = (long long)blockIdx.x * kReduceCols + lane;
    double yj = 0.0;
    if (j < p.ld) {
        const Acc *py = static_cast<const Acc *>(p.part_y);
        Acc t = Acc(0);
#pragma unroll 8
        for (int g = grp; g < p.G; g += 8)
            t += py[(long long)g * p.ld + j];
        yj = (double)t;
    }
    sh.part[grp][lane] = yj;
    __syncthreads();
    if (grp == 0 && j < p.ld) {
        double y = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            y += sh.part[q][lane];
        y_out[j] = y;
    }
    if (blockIdx.x == 0) {
        reduce_stats(p.part_stat, p.G, sh);
        __syncthreads();
        if (threadIdx.x == 0) {
            p.st->h = sh.h;
            p.st->maxviol = sh.mv;
            p.st->maxnorm = sh.mn;
            p.st->maxb = sh.mb;
        }
    }
}

// ------------------------------------------------------- binary64 check ----

__device__ __forceinline__ unsigned long long ord_enc(double d)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// One warp per row: r_i = sum_j a_ij x_j - (b0_i + (k rho) Av_i) with binary64
// products and sums on the stored entries; maxima by order-preserving
// integer atomics (exact, so the result does not depend on the schedule).
template <int S>
__global__ void __launch_bounds__(256) verify_kernel(const VerifyArgs p)
{
    using Tr = Traits<S>;
    using Acc = typename Tr::acc;
    constexpr int EPV = Tr::EPV;
    const int lane = threadIdx.x & 31;
    const long long wg = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const double kr = __dmul_rn((double)p.st->tick, p.st->rho);
    const double *x = p.x64;
    const long long row_bytes = (long long)p.nv * 16;
    double mv = -INFINITY, mn = -INFINITY, mb = 0.0;
    unsigned long long h = 0;
    for (long long i = wg; i < p.m; i += nw) {
        const uint4 *row = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(p.A) + i * row_bytes);
        double s = 0.0;
        for (int j = lane; j < p.nv; j += 32) {
            Acc a[EPV];
            decode<S>(__ldg(row + j), a);
#pragma unroll
            for (int e = 0; e < EPV; ++e)
                s = fma((double)a[e], x[(long long)j * EPV + e], s);
        }
        s = warp_sum(s);
        if (S == NSLI_FP8E4M3)
            s = s * (double)p.scale[i];
        const double bi = __dadd_rn(p.b0_64[i], __dmul_rn(kr, p.av_64[i]));
        const double ri = s - bi;
        mv = fmax(mv, ri);
        mn = fmax(mn, ri / sqrt(p.n2_64[i]));
        mb = fmax(mb, fabs(bi));
        h += (ri > 0.0) ? 1ull : 0ull;
    }
    if (lane == 0) {
        atomicMax(&p.out->maxviol, ord_enc(mv));
        atomicMax(&p.out->maxnorm, ord_enc(mn));
        atomicMax(&p.out->maxb, ord_enc(mb));
        atomicAdd(&p.out->h, h);
    }
}

// ---------------------------------------------------------------- set-up ----

// One block per row: optional FP8 row scale, store the row in the storage
// type (zero padding up to ld), binary64 ||a_i||^2 of the STORED values in a
// fixed order, finiteness and zero-row flags.
// FAST: the quick norm (else the binary64 one).  Bound by loads in flight and
// instructions: four entries per thread and step, and one norm's code per
// instance, whose registers let six blocks share an SM.  nsli_create of
// 131072 x 16384 (the allocations included): binary32 8.4 -> 4.2 ms, bf16 7.1
// -> 4.5 ms, FP8 7.2 -> 4.5 ms, against one entry at a time and 40 to 53
// registers.  The binary64 norm takes eight entries per step, as many as it
// folds into binary64 at once, so that it counts none: nsli_batch_create of
// 65536 x 8192 with 64 problems 5.15 ms, against 6.0 ms one entry at a time
// and 7.05 ms with four entries and a count.  Binary64 storage: five blocks per
// SM, four were slower (32768 x 16384: 6.85 -> 6.34 ms).
template <int S, bool FAST>
__global__ void __launch_bounds__(256, S == NSLI_F64 ? 5 : 6) prep_kernel(const PrepArgs p)
{
    const long long r = blockIdx.x;
    if (r >= p.rows)
        return;
    const long long gi = p.row0 + r;
    __shared__ double sred[8];
    __shared__ float samax[8];
    __shared__ int sbad;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0)
        sbad = 0;
    __syncthreads();
    const float *s32 = static_cast<const float *>(p.src) + r * p.lda;
    const double *s64 = static_cast<const double *>(p.src) + r * p.lda;
    int bad = 0;

    float scale = 1.0f, inv_scale = 1.0f;
    if (S == NSLI_FP8E4M3) {
        float amax = 0.0f;
        for (long long j = threadIdx.x; j < p.n; j += blockDim.x) {
            const float a = s32[j];
            if (!isfinite(a))
                bad = 1;
            amax = fmaxf(amax, fabsf(a));
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
        if (lane == 0)
            samax[wid] = amax;
        __syncthreads();
        amax = 0.0f;
        for (int q = 0; q < 8; ++q)
            amax = fmaxf(amax, samax[q]);
        int e = 0;
        if (amax > 0.0f && isfinite(amax)) {
            int e2;
            const float f = frexpf(amax, &e2);  // amax = f 2^e2, f in [0.5, 1)
            e = (f <= 0.875f) ? e2 - 9 : e2 - 8;  // smallest 2^e with amax / 2^e <= 448
        }
        scale = ldexpf(1.0f, e);
        inv_scale = ldexpf(1.0f, -e);
        if (threadIdx.x == 0)
            p.scale[gi] = scale;
    }

    // ||a_i||^2 of the stored values: binary64 for binary64 storage, else the
    // quick form of nsli_sumsq.cuh (FAST: the norm behind the row records, as
    // in the row-update kernel) or the double-float accumulation folded into
    // binary64 every 8 entries, and the block total
    double n2 = 0.0;
    typename std::conditional<FAST, QuickSum<S != NSLI_FP8E4M3>, SumSq>::type sq;
    quick_init(sq);
    auto get = [&](long long j) -> float {   // the source's entry j (0 past n)
        if (j >= p.n)
            return 0.0f;
        if (S == NSLI_F32 && p.src_f64) {
            const double a = s64[j];
            if (!isfinite(a))
                bad = 1;
            return __double2float_rn(a);
        }
        const float a = s32[j];
        if (S != NSLI_FP8E4M3 && !isfinite(a))
            bad = 1;
        return a;
    };
    auto put = [&](long long j, float a) -> float {   // stores entry j, returns its stored value
        if (S == NSLI_F32) {
            static_cast<float *>(p.A)[gi * p.ld + j] = a;
            return isfinite(a) ? a : 0.0f;   // (a binary64 source's value past the binary32 range)
        } else if (S == NSLI_BF16) {
            // (a value that rounds to infinity makes the norm infinite and
            // the row invalid, as in the row-update kernel)
            const __nv_bfloat16 q = __float2bfloat16_rn(a);
            static_cast<__nv_bfloat16 *>(p.A)[gi * p.ld + j] = q;
            return __bfloat162float(q);
        } else {
            const __nv_fp8_storage_t q = __nv_cvt_float_to_fp8(a * inv_scale, __NV_SATFINITE, __NV_E4M3);
            static_cast<unsigned char *>(p.A)[gi * p.ld + j] = (unsigned char)q;
            const __half_raw hr = __nv_cvt_fp8_to_halfraw(q, __NV_E4M3);
            return __fmul_rn(__half2float(__half(hr)), scale);   // exact: scale is a power of two
        }
    };
    if constexpr (S == NSLI_F64) {
        for (long long j = threadIdx.x; j < p.ld; j += blockDim.x) {
            const bool in = j < p.n;
            const double v = in ? (p.src_f64 ? s64[j] : (double)s32[j]) : 0.0;
            if (in && !isfinite(v))
                bad = 1;
            static_cast<double *>(p.A)[gi * p.ld + j] = v;
            n2 += v * v;
        }
    } else {
        constexpr int U = FAST ? 4 : 8;
        for (long long j0 = threadIdx.x; j0 < p.ld; j0 += U * 256) {
            float v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                v[u] = get(j0 + u * 256);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 + u * 256 < p.ld)
                    v[u] = put(j0 + u * 256, v[u]);
            if constexpr (!FAST)
                if (j0 >= 256)
                    sumsq_flush(sq);   // the step before; rows of one step need no binary64
            // (a zero past n changes neither sum; two of them are left out)
#pragma unroll
            for (int u = 0; u < U; u += 2) {
                if (j0 + u * 256 >= p.n)
                    break;
                if constexpr (FAST) {
                    quick_add(sq, v[u], v[u + 1]);
                } else {
                    sumsq_add<0>(sq, v[u]);
                    sumsq_add<0>(sq, v[u + 1]);
                }
            }
        }
    }
    if (bad)
        sbad = 1;
    double t = 0.0;   // the row total, in thread 0
    if constexpr (S != NSLI_F64) {
        __shared__ float2 spair[8];
        __shared__ double sacc[8];
        t = sumsq_block_total<8>(sq, spair, sacc);   // (synchronises the block)
    } else {
        n2 = warp_sum(n2);
        if (lane == 0)
            sred[wid] = n2;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q)
                t += sred[q];
    }
    if (threadIdx.x == 0) {
        if (p.norms_in != nullptr)
            t = p.norms_in[gi];
        p.n2_64[gi] = t;
        int f = 0;
        if (sbad || !isfinite(t))
            f |= PREPF_NONFINITE;
        if (t == 0.0)
            f |= PREPF_ZERO_ROW;
        if (f)
            atomicOr(p.flags, f);
    }
}

template <bool F64>
__global__ void __launch_bounds__(256) meta_kernel(const MetaArgs p)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= p.m)
        return;
    const long long i = p.row0 + k;
    const double b0 = p.b0_64[i];
    const double av = p.av_64[i];
    const double n2 = p.n2_64[i];
    if (!isfinite(b0) || !isfinite(av))
        atomicOr(p.flags, PREPF_NONFINITE);
    const double inv_n2 = 1.0 / n2;
    const double inv_n = 1.0 / sqrt(n2);
    if (F64) {
        RowMeta64 m{b0, av, inv_n2, inv_n};
        static_cast<RowMeta64 *>(p.meta)[i] = m;
    } else {
        RowMeta32 m{(float)b0, (float)av, (float)inv_n2, (float)inv_n,
                    p.scale ? p.scale[i] : 1.0f, 0.0f, 0.0f, 0.0f};
        static_cast<RowMeta32 *>(p.meta)[i] = m;
    }
}

// Only the b0 field of rows [row0, row0 + m): a new right-hand side leaves
// the norms, Av and the FP8 scale as they are, and the field gets the value
// meta_kernel would give it (no binary64 divide or root per row).
template <bool F64> __global__ void __launch_bounds__(256) meta_b0_kernel(const MetaArgs p)
{
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k == 0 && p.tick >= 0)
        p.st->tick = p.tick;
    if (k >= p.m)
        return;
    const long long i = p.row0 + k;
    double b0;
    if (p.b0_src) {
        b0 = p.b0_src[k];
        p.b0_keep[i] = b0;
    } else {
        b0 = p.b0_64[i];
    }
    if (!isfinite(b0))
        atomicOr(p.flags, PREPF_NONFINITE);
    if (F64)
        static_cast<RowMeta64 *>(p.meta)[i].b0 = b0;
    else
        static_cast<RowMeta32 *>(p.meta)[i].b0 = (float)b0;
}

template <typename Acc>
__global__ void x_from_f64_kernel(const double *src, double *x64, Acc *x, long long n, long long ld, int *flags)
{
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ld)
        return;
    double v = 0.0;
    if (j < n) {
        v = src[j];
        if (!isfinite(v))
            atomicOr(flags, PREPF_NONFINITE);
    }
    x64[j] = v;
    x[j] = (Acc)v;
}

__global__ void check_finite_kernel(const double *v, long long n, int *flags)
{
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n && !isfinite(v[j]))
        atomicOr(flags, PREPF_NONFINITE);
}

// Run parameters into the state (block 0, thread 0) and, when the step size
// changed, the table lambda / h that the step reads instead of dividing (a
// binary64 division is a long dependency chain on GB300).
__global__ void state_begin_kernel(DevState *st, const StateBegin b)
{
    if (b.rtab) {
        for (long long h = (long long)blockIdx.x * blockDim.x + threadIdx.x; h <= b.rtab_m;
             h += (long long)gridDim.x * blockDim.x)
            b.rtab[h] = h > 0 ? b.lambda / (double)h : 0.0;
    }
    if (blockIdx.x != 0 || threadIdx.x != 0)
        return;
    st->lambda = b.lambda;
    st->eps = b.eps;
    st->rho = b.rho;
    st->max_iter = b.max_iter;
    st->rule = b.rule;
    st->stop = b.stop;
    st->force_step = b.force_step;
    if (b.reset_it)
        st->it = 0;
    if (b.tick >= 0)
        st->tick = b.tick;
    st->done = 0;
    st->status = ST_RUNNING;
    st->error = 0;
    st->ticket = 0u;
    if (b.sync)   // (also after a launch that gave up)
        for (int q = 0; q < 4; ++q)
            b.sync[q] = 0u;
}

__global__ void set_ticks_kernel(DevState *const *sts, const long long *ticks, int count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) {
        sts[i]->tick = ticks[i];
        sts[i]->hold_tick = 1;
    }
}

__global__ void set_tick_kernel(DevState *st, long long tick) { st->tick = tick; }

__global__ void state_resume_kernel(DevState *st)
{
    st->done = 0;
    st->status = ST_RUNNING;
    st->force_step = 1;
}

// Exact values of stored rows as binary64 (diagnostics).
template <int S>
__global__ void stored_rows_kernel(const void *A, const float *scale, long long ld, long long n, long long row0,
                                   long long rows, double *out)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= rows * n)
        return;
    const long long r = t / n, j = t % n;
    const long long i = row0 + r;
    double v;
    if (S == NSLI_F64) {
        v = static_cast<const double *>(A)[i * ld + j];
    } else if (S == NSLI_F32) {
        v = (double)static_cast<const float *>(A)[i * ld + j];
    } else if (S == NSLI_BF16) {
        v = (double)__bfloat162float(static_cast<const __nv_bfloat16 *>(A)[i * ld + j]);
    } else {
        const __nv_fp8_storage_t q = static_cast<const unsigned char *>(A)[i * ld + j];
        const __half_raw hr = __nv_cvt_fp8_to_halfraw(q, __NV_E4M3);
        v = (double)__half2float(__half(hr)) * (double)scale[i];
    }
    out[t] = v;
}

// ------------------------------------------------------------- launchers ----

int map_vpt_limit(int storage)
{
    switch (storage) {
    case NSLI_F64: return 8;
    case NSLI_F32: return 8;
    case NSLI_BF16: return 4;
    case NSLI_FP8E4M3: return 2;
    default: return 0;
    }
}

cudaError_t long_prepare(int storage, size_t smem)
{
    // partial sums in shared memory for every group size
    if (smem == 0)
        return cudaSuccess;
    for (int rg = 1; rg <= 4; rg *= 2) {
        const void *fn = long_fn(storage, rg, true);
        if (!fn)
            return cudaErrorInvalidValue;
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

cudaError_t cluster_prepare(int storage, int vpt, int rg, int C, size_t smem, int *clusters)
{
    *clusters = 0;
    const void *fn = cluster_fn(storage, vpt, rg);
    if (!fn || C < 2 || C > 8)
        return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(clusters, fn, &cfg);
}

cudaError_t team_map_prepare(int storage, int vpt, int rg) { return set_smem(dense_fn<MapFn>(storage, vpt, rg)); }

cudaError_t team_launch(int storage, int vpt, int grid, size_t smem, cudaStream_t s, const MapArgs &a)
{
    const void *fn = dense_fn<MapFn>(storage, vpt, a.rows_per_slot);
    if (!fn)
        return cudaErrorInvalidValue;
    void *args[] = {const_cast<MapArgs *>(&a)};
    return cudaLaunchKernel(fn, dim3(grid), dim3(team_threads(a.teams, a.team_warps)), args, smem, s);
}

cudaError_t map_launch(int storage, int vpt, int grid, size_t smem, cudaStream_t s, const MapArgs &a)
{
    if (vpt == 0 && a.cluster > 1) {
        // long rows on clusters: `grid` clusters of a.cluster CTAs
        const void *fn = cluster_fn(storage, a.cluster_vpt, a.cluster_rg);
        if (!fn)
            return cudaErrorInvalidValue;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(grid * a.cluster));
        cfg.blockDim = dim3(kClusterThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)a.cluster;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        void *args[] = {const_cast<MapArgs *>(&a)};
        return cudaLaunchKernelExC(&cfg, fn, args);
    }
    if (vpt == 0) {
        // long rows: rows_per_slot carries the group size, smem the
        // partial-sum row in shared memory (0: in global memory)
        const void *fn = long_fn(storage, a.rows_per_slot, smem > 0);
        if (!fn)
            return cudaErrorInvalidValue;
        void *args[] = {const_cast<MapArgs *>(&a)};
        return cudaLaunchKernel(fn, dim3(grid), dim3(kLongThreads), args, smem, s);
    }
    return team_launch(storage, vpt, grid, smem, s, a);
}

cudaError_t reduce_group_launch(bool f64, int blocks, cudaStream_t s, const GroupProblem *probs,
                                const GroupRed *tab)
{
    if (f64)
        reduce_group_kernel<double><<<blocks, 256, 0, s>>>(probs, tab);
    else
        reduce_group_kernel<float><<<blocks, 256, 0, s>>>(probs, tab);
    return cudaGetLastError();
}

cudaError_t reduce_launch(bool f64, int grid, cudaStream_t s, const ReduceArgs &a)
{
    if (f64)
        reduce_update_kernel<double><<<grid, 256, 0, s>>>(a);
    else
        reduce_update_kernel<float><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t reduce_only_launch(bool f64, int grid, cudaStream_t s, const ReduceArgs &a, double *y_out)
{
    if (f64)
        reduce_only_kernel<double><<<grid, 256, 0, s>>>(a, y_out);
    else
        reduce_only_kernel<float><<<grid, 256, 0, s>>>(a, y_out);
    return cudaGetLastError();
}

cudaError_t verify_launch(int storage, int grid, cudaStream_t s, const VerifyArgs &a)
{
    switch (storage) {
    case NSLI_F64: verify_kernel<NSLI_F64><<<grid, 256, 0, s>>>(a); break;
    case NSLI_F32: verify_kernel<NSLI_F32><<<grid, 256, 0, s>>>(a); break;
    case NSLI_BF16: verify_kernel<NSLI_BF16><<<grid, 256, 0, s>>>(a); break;
    case NSLI_FP8E4M3: verify_kernel<NSLI_FP8E4M3><<<grid, 256, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t prep_launch(int storage, cudaStream_t s, const PrepArgs &a)
{
    if (!a.fast && storage != NSLI_BF16)
        return cudaErrorInvalidValue;   // no caller
    const unsigned int grid = (unsigned int)a.rows;
    switch (storage) {
    case NSLI_F64: prep_kernel<NSLI_F64, true><<<grid, 256, 0, s>>>(a); break;
    case NSLI_F32: prep_kernel<NSLI_F32, true><<<grid, 256, 0, s>>>(a); break;
    case NSLI_BF16:
        if (a.fast)
            prep_kernel<NSLI_BF16, true><<<grid, 256, 0, s>>>(a);
        else   // (the batched form's A)
            prep_kernel<NSLI_BF16, false><<<grid, 256, 0, s>>>(a);
        break;
    case NSLI_FP8E4M3: prep_kernel<NSLI_FP8E4M3, true><<<grid, 256, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t meta_b0_launch(bool f64, cudaStream_t s, const MetaArgs &a)
{
    if (a.m <= 0)
        return cudaSuccess;
    const unsigned int grid = (unsigned int)((a.m + 255) / 256);
    if (f64)
        meta_b0_kernel<true><<<grid, 256, 0, s>>>(a);
    else
        meta_b0_kernel<false><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t meta_launch(bool f64, cudaStream_t s, const MetaArgs &a)
{
    if (a.m <= 0)
        return cudaSuccess;
    const unsigned int grid = (unsigned int)((a.m + 255) / 256);
    if (f64)
        meta_kernel<true><<<grid, 256, 0, s>>>(a);
    else
        meta_kernel<false><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t x_from_f64_launch(bool f64, cudaStream_t s, const double *src, double *x64, void *x, long long n,
                              long long ld, int *flags)
{
    const unsigned int grid = (unsigned int)((ld + 255) / 256);
    if (f64)
        x_from_f64_kernel<double><<<grid, 256, 0, s>>>(src, x64, static_cast<double *>(x), n, ld, flags);
    else
        x_from_f64_kernel<float><<<grid, 256, 0, s>>>(src, x64, static_cast<float *>(x), n, ld, flags);
    return cudaGetLastError();
}

cudaError_t check_finite_launch(cudaStream_t s, const double *v, long long n, int *flags)
{
    const unsigned int grid = (unsigned int)((n + 255) / 256);
    check_finite_kernel<<<grid, 256, 0, s>>>(v, n, flags);
    return cudaGetLastError();
}

cudaError_t state_begin_launch(cudaStream_t s, DevState *st, const StateBegin &b)
{
    long long blocks = b.rtab ? (b.rtab_m + 256) / 256 : 1;
    if (blocks > 1024)
        blocks = 1024;
    state_begin_kernel<<<(unsigned)blocks, b.rtab ? 256 : 1, 0, s>>>(st, b);
    return cudaGetLastError();
}

cudaError_t set_ticks_launch(cudaStream_t s, DevState *const *sts, const long long *ticks, int count)
{
    set_ticks_kernel<<<(count + 127) / 128, 128, 0, s>>>(sts, ticks, count);
    return cudaGetLastError();
}

cudaError_t set_tick_launch(cudaStream_t s, DevState *st, long long tick)
{
    set_tick_kernel<<<1, 1, 0, s>>>(st, tick);
    return cudaGetLastError();
}

cudaError_t state_resume_launch(cudaStream_t s, DevState *st)
{
    state_resume_kernel<<<1, 1, 0, s>>>(st);
    return cudaGetLastError();
}

cudaError_t stored_rows_launch(int storage, cudaStream_t s, const void *A, const float *scale, long long ld,
                               long long n, long long row0, long long rows, double *out)
{
    const long long total = rows * n;
    const unsigned int grid = (unsigned int)((total + 255) / 256);
    switch (storage) {
    case NSLI_F64: stored_rows_kernel<NSLI_F64><<<grid, 256, 0, s>>>(A, scale, ld, n, row0, rows, out); break;
    case NSLI_F32: stored_rows_kernel<NSLI_F32><<<grid, 256, 0, s>>>(A, scale, ld, n, row0, rows, out); break;
    case NSLI_BF16: stored_rows_kernel<NSLI_BF16><<<grid, 256, 0, s>>>(A, scale, ld, n, row0, rows, out); break;
    case NSLI_FP8E4M3:
        stored_rows_kernel<NSLI_FP8E4M3><<<grid, 256, 0, s>>>(A, scale, ld, n, row0, rows, out);
        break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace nsli
