// cg_resident.cu -- the conjugate gradient iterations of one solve in one
// launch, for lattices whose thread blocks are all resident on the GPU at once.
//
// Kernel by kernel, an iteration is five launches, each of which waits for the
// last block of the one before, starts its blocks and drains; on a lattice of
// one wave or less that costs more than the work.  Here the blocks stay: a
// cooperative launch (so that all of them run at the same time) in which block
// b owns the DS_BLOCK sites of block b of the kernel-by-kernel path, the four
// hopping terms of an iteration are separated by barriers over the grid, and
// every block forms the CG scalars itself from the block partials behind the
// barrier.  Site arithmetic, block partials, their summation order and the
// scalar steps are those of dslash.cu and dslash.cuh, so the iterates and the
// iteration count are bitwise those of the kernel-by-kernel path and of the
// multi-system engine.
//
// An iteration's five barriers take about 4,000 cycles each and a block sum
// with its FP64 scalar step 3,000 (14^4; the hops 4,000 each), so whatever
// needs no other block's data lies between a barrier's two halves: the pAp
// step and alpha in the wait behind the next hop, the update of x in the wait
// for |r|^2, the links and neighbours of the next hop beside the epilogue.
//
// Measured, solves of about 30 iterations, kernel by kernel and resident:
// FP16+norm (3 reliable updates) 4^4 924 and 762 us, 8^4 997 and 803, 12^4 1074
// and 965, 14^4 1147 and 1022, 16^4 1351 and 1203, 16^3x32 (512 blocks) 1851 and
// 1763; BF16 (7 updates) 8^4 1138 and 991, 16^3x32 2398 and 2307; FP32 (4) 8^4
// 1297 and 1002, 16^3x32 2190 and 2020; FP64 8^4 1806 and 1517, 14^4 (601 blocks)
// 4604 and 4394.  Of that the overlap above is 4% on 8^4 and 8% on 16^3x32.  Up
// to 16 blocks the grid is one cluster, whose hardware barrier makes an
// iteration of 8^4 4 us shorter than the barrier through L2.  The blocks have to
// be resident together, so the path ends at 608 of them; there the kernel
// boundaries cost 5% (FP32 8%) and fall with the number of waves, while more
// sites per block would leave SMs unevenly filled.
// Four threads per site on lattices of up to 152 blocks were no faster: an SM's
// instructions are the same, and exchanging the hops adds shared-memory traffic.
#include "cg.cuh"
#include "dslash_f64.cuh"
#include "dslash_packed.cuh"
#include "dslash_site.cuh"

#include <algorithm>
#include <climits>

namespace lqcd {

// iterations after which a launch returns to the host in any case, polls of a
// barrier before a block gives up (about a second), and the blocks that are
// taken to run at the same time (0: what the device says), of the solves that
// the calling thread makes (lqcd_solver_limits)
struct ResidentLimits {
    int iters = 512;
    int polls = 1 << 21;
    int blocks = 0;
};
static thread_local ResidentLimits t_limits;

// Barrier over the grid's blocks, in two halves: what any block wrote before its
// grid_arrive is visible to every block after its grid_wait; between the two a
// block does work that needs no other block's.  CLUSTER: the grid is one
// thread-block cluster, whose hardware barrier does it, in the form that each
// thread executes for itself: both halves follow branches that a warp need not
// take as a whole (the sites of a ragged last block, lane 0 of a block sum), and
// the .aligned form asks for converged warps.  Otherwise sc->bar
// counts arrivals (0 at the launch) and thread 0, which keeps the next target,
// waits for it: one release-add that nobody waits for and a polled acquire
// load.  Bounded: a block that waits too long sets sc->bar_abort, and every
// block's grid_wait then returns false.
template <bool CLUSTER>
__device__ __forceinline__ void grid_arrive(CgScalars *sc, unsigned &target)
{
    if constexpr (CLUSTER) {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    } else {
        __syncthreads();
        if (threadIdx.x == 0) {
            target += gridDim.x;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&sc->bar) : "memory");
        }
    }
}
template <bool CLUSTER>
__device__ __forceinline__ bool grid_wait(CgScalars *sc, unsigned target, int polls)
{
    if constexpr (CLUSTER) {
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        return true;
    } else {
        __shared__ int good;
        if (threadIdx.x == 0) {
            int ok = 1;
            for (int k = 0;; k++) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&sc->bar) : "memory");
                if (v >= target) break;
                if (k >= polls) atomicExch(&sc->bar_abort, 1u);
                if ((k & 63) == 63 || k >= polls) {
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&sc->bar_abort) : "memory");
                    if (v) {
                        ok = 0;
                        break;
                    }
                }
            }
            good = ok;
        }
        __syncthreads();
        return good != 0;
    }
}
template <bool CLUSTER>
__device__ __forceinline__ bool grid_barrier(CgScalars *sc, unsigned &target, int polls)
{
    grid_arrive<CLUSTER>(sc, target);
    return grid_wait<CLUSTER>(sc, target, polls);
}

// blocks per SM the register budget is cut for: they set the largest lattice
// that one launch holds (152 SMs x 4 x 128 sites = 77,824 even sites; FP64, 32
// sites a block, 19,456)
constexpr int RESIDENT_PER_SM = 4;

// the outcome of a launch, by one thread of the grid
__device__ __forceinline__ void resident_result(CgScalars *sc, CgScalars &s, bool ok)
{
    if (!ok) {
        s.pause = 1;
        s.reason = PAUSE_TIMEOUT;
    }
    sc->rr = s.rr, sc->pAp = s.pAp, sc->alpha = s.alpha, sc->beta = s.beta, sc->rr_new = s.rr_new;
    sc->maxrr2 = s.maxrr2, sc->pause = s.pause, sc->reason = s.reason, sc->iter = s.iter;
}

// the scalar step behind a reducing hopping term, by every block on its own copy
template <int BLOCK>
__device__ __forceinline__ void resident_scalars(CgScalars &s, const double *partials, int nb, bool rr)
{
    const double total = block_final_sum<BLOCK>(partials, nb);
    if (threadIdx.x == 0) {
        if (rr)
            cg_rr_step(&s, total);
        else
            cg_pap_step(&s, total);
    }
    __syncthreads();
}

// What the packed 16-bit hops of a block keep over the launch: the neighbours
// of its sites' two parities, and the links of the hop to come, whose copies
// (LinkPrefetchT) start as soon as the hop before has read its own: index
// arithmetic and link latency then lie beside the epilogue and the barrier
template <lqcd_prec SP>
struct ResidentHops {
    LinkPrefetchT<DS_BLOCK> lp;
    int nb[2][8][DS_BLOCK]; // [output on the even sites]; the time neighbours' top bit: the boundary sign flips
};
template <>
struct ResidentHops<LQCD_F32> {};

template <lqcd_prec SP>
__device__ __forceinline__ void resident_neighbours(ResidentHops<SP> &sh, const Geo &g, int cb)
{
    for (int odd = 0; odd < 2; odd++) {
        int c[4], n[8];
        bool tf, tb;
        cb_coords(g, cb, 1 - odd, c);
        cb_neighbours(g, cb, c, n, tf, tb);
        if (g.t_bc < 0) {
            n[6] |= tf ? INT_MIN : 0;
            n[7] |= tb ? INT_MIN : 0;
        }
#pragma unroll
        for (int k = 0; k < 8; k++) sh.nb[odd][k][threadIdx.x] = n[k];
    }
}

template <lqcd_prec SP>
__device__ __forceinline__ void resident_links(ResidentHops<SP> &sh, const GaugeRef<SP> &U, int cb, int odd)
{
    const int i = threadIdx.x;
    const auto &n = sh.nb[odd];
    packed_prefetch<DS_BLOCK, SP>(sh.lp, U, cb, 1 - odd, {n[1][i], n[3][i], n[5][i], n[7][i] & INT_MAX});
}

// D or D^dag at one site in the form the kernel-by-kernel path takes by default
template <typename R, lqcd_prec SP, bool DAG>
__device__ __forceinline__ Sp<R> resident_site(ResidentHops<SP> &sh, const SpinorRef<SP> &in,
                                               const GaugeRef<SP> &U, const Geo &g, int cb, int odd)
{
    if constexpr (SP == LQCD_F16N || SP == LQCD_BF16) {
        const int i = threadIdx.x;
        int n[8];
#pragma unroll
        for (int k = 0; k < 8; k++) n[k] = sh.nb[odd][k][i];
        const bool ff = n[6] < 0, fb = n[7] < 0;
        n[6] &= INT_MAX;
        n[7] &= INT_MAX;
        return packed_values(packed_hops<DAG, DS_BLOCK, true, SP>(sh.lp, in, U, g, n, ff, fb));
    } else {
        return dslash_site<R, SP, SP, DAG, true>(in, U, g, cb, 1 - odd);
    }
}

template <lqcd_prec SP, bool CLUSTER>
__global__ void __launch_bounds__(DS_BLOCK, RESIDENT_PER_SM)
    cg_resident_kernel(SpinorRef<SP> p, SpinorRef<SP> r, SpinorRef<SP> t, SpinorRef<SP> tmp, SpinorRef<LQCD_F32> xs,
                       GaugeRef<SP> U, Geo g, float b, double *partials, int nb, CgScalars *sc, ResidentLimits lim)
{
    using R = float;
    constexpr bool PACKED = SP == LQCD_F16N || SP == LQCD_BF16;
    __shared__ ResidentHops<SP> hops;
    __shared__ CgScalars s; // this block's copy: every block takes the same steps
    if (threadIdx.x == 0) s = *sc;
    __syncthreads();
    if (s.pause) return;
    const int cb = blockIdx.x * DS_BLOCK + threadIdx.x;
    unsigned target = 0;
    const bool live = cb < g.Vh;
    bool ok = true;
    if constexpr (PACKED)
        if (live) {
            resident_neighbours<SP>(hops, g, cb);
            resident_links<SP>(hops, U, cb, 0);
        }
    for (int it = 0; it < lim.iters; it++) {
        // tmp = D p;  t = p + b D tmp, |t|^2;  tmp = D^dag t;  A p = t + b D^dag tmp, r -= alpha A p, |r|^2, x += alpha p
#pragma unroll 1
        for (int ph = 0; ph < 4; ph++) {
            const int odd = ph & 1; // output on the even sites
            R n2 = R(0);
            if (live) {
                const SpinorRef<SP> in = odd ? tmp : ph == 0 ? p : t;
                Sp<R> d = ph < 2 ? resident_site<R, SP, false>(hops, in, U, g, cb, odd)
                                 : resident_site<R, SP, true>(hops, in, U, g, cb, odd);
                if constexpr (PACKED) resident_links<SP>(hops, U, cb, 1 - odd);
                if (!odd) {
                    tmp.store(cb, d);
                } else {
                    const Sp<R> x = (ph == 1 ? p : t).template load_rw<R>(cb);
#pragma unroll
                    for (int a = 0; a < 4; a++)
#pragma unroll
                        for (int k = 0; k < 3; k++) d.c[a][k] = x.c[a][k] + b * d.c[a][k];
                    if (ph == 1) {
                        t.store(cb, d);
                        n2 = sp_norm2(d);
                    } else {
                        const R alpha = (R)s.alpha;
                        Sp<R> rv = r.template load_rw<R>(cb);
#pragma unroll
                        for (int a = 0; a < 4; a++)
#pragma unroll
                            for (int k = 0; k < 3; k++) rv.c[a][k] = rv.c[a][k] - alpha * d.c[a][k];
                        r.store(cb, rv);
                        n2 = sp_norm2(rv);
                    }
                }
            }
            // |t|^2 and |r|^2 of an iteration in two places: the first is read while others store the second
            if (odd) block_sum_store_wp<DS_BLOCK>(n2, partials + (ph == 3 ? gridDim.x : 0));
            grid_arrive<CLUSTER>(sc, target);
            if (ph == 2) { // alpha, which nothing needs before the next hop's epilogue
                resident_scalars<DS_BLOCK>(s, partials, nb, false);
            } else if (ph == 3 && live) {
                const R alpha = (R)s.alpha;
                const Sp<R> pv = p.template load_rw<R>(cb);
                Sp<R> xv = xs.template load_rw<R>(cb);
#pragma unroll
                for (int a = 0; a < 4; a++)
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        xv.c[a][k].re += alpha * pv.c[a][k].re;
                        xv.c[a][k].im += alpha * pv.c[a][k].im;
                    }
                xs.store(cb, xv);
            }
            if (!(ok = grid_wait<CLUSTER>(sc, target, lim.polls))) break;
            if (ph == 3) resident_scalars<DS_BLOCK>(s, partials + gridDim.x, nb, true);
            if (ph >= 2 && s.pause) break;
        }
        if (!ok || s.pause) break;
        if (live) { // p = r + beta p: each thread its own site
            const R beta = (R)s.beta;
            Sp<R> pv = p.template load_rw<R>(cb);
            const Sp<R> rv = r.template load_rw<R>(cb);
#pragma unroll
            for (int a = 0; a < 4; a++)
#pragma unroll
                for (int k = 0; k < 3; k++) pv.c[a][k] = rv.c[a][k] + beta * pv.c[a][k];
            p.store(cb, pv);
        }
        if (!(ok = grid_barrier<CLUSTER>(sc, target, lim.polls))) break;
    }
    if constexpr (PACKED) cp_async_wait<0>();
    if (blockIdx.x == 0 && threadIdx.x == 0) resident_result(sc, s, ok);
}

// The plain FP64 solve: blocks of 32 sites, a thread per site and spin row
// (dslash_f64.cuh), the accurate solution updated in place
template <bool CLUSTER>
__global__ void __launch_bounds__(QUAD_BLOCK, RESIDENT_PER_SM)
    cg_resident_f64_kernel(SpinorRef<LQCD_F64> p, SpinorRef<LQCD_F64> r, SpinorRef<LQCD_F64> t, SpinorRef<LQCD_F64> tmp,
                           SpinorRef<LQCD_F64> xs, GaugeRef<LQCD_F64> U, Geo g, double b, double *partials, int nb,
                           CgScalars *sc, ResidentLimits lim)
{
    __shared__ QuadF64 sh;
    __shared__ CgScalars s;
    if (threadIdx.x == 0) s = *sc;
    __syncthreads();
    if (s.pause) return;
    const int cb = blockIdx.x * QUAD_SITES + (threadIdx.x & 31);
    const bool live = cb < g.Vh;
    unsigned target = 0;
    bool ok = true;
    for (int it = 0; it < lim.iters; it++) {
#pragma unroll 1
        for (int ph = 0; ph < 4; ph++) {
            const bool odd = ph & 1;
            const SpinorRef<LQCD_F64> in = odd ? tmp : ph == 0 ? p : t;
            RowF64 d = ph < 2 ? quad_row<false, true>(sh, in, U, g, cb, odd ? 0 : 1, live)
                              : quad_row<true, true>(sh, in, U, g, cb, odd ? 0 : 1, live);
            double n2 = 0.0;
            if (live) {
                if (!odd) {
                    store_row(tmp, cb, d);
                } else if (ph == 1) {
                    d = row_xpay(load_row(p, cb), b, d);
                    store_row(t, cb, d);
                    n2 = row_norm2(d);
                } else {
                    d = row_xpay(load_row(t, cb), b, d);
                    const RowF64 rv = row_xpay(load_row(r, cb), -s.alpha, d);
                    store_row(r, cb, rv);
                    n2 = row_norm2(rv);
                }
            }
            if (odd) block_sum_store_wp<QUAD_BLOCK>(n2, partials + (ph == 3 ? gridDim.x : 0));
            grid_arrive<CLUSTER>(sc, target);
            if (ph == 2)
                resident_scalars<QUAD_BLOCK>(s, partials, nb, false);
            else if (ph == 3 && live)
                store_row(xs, cb, row_xpay(load_row(xs, cb), s.alpha, load_row(p, cb)));
            if (!(ok = grid_wait<CLUSTER>(sc, target, lim.polls))) break;
            if (ph == 3) resident_scalars<QUAD_BLOCK>(s, partials + gridDim.x, nb, true);
            if (ph >= 2 && s.pause) break;
        }
        if (!ok || s.pause) break;
        if (live) store_row(p, cb, row_xpay(load_row(r, cb), s.beta, load_row(p, cb)));
        if (!(ok = grid_barrier<CLUSTER>(sc, target, lim.polls))) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) resident_result(sc, s, ok);
}

// the kernels' addresses, types and sites per block by storage precision
template <lqcd_prec SP>
struct Resident {
    using R = float;
    static constexpr lqcd_prec XP = LQCD_F32;
    static constexpr int SITES = DS_BLOCK, BLOCK = DS_BLOCK;
    static const void *kernel(bool cluster)
    {
        return cluster ? (const void *)cg_resident_kernel<SP, true> : (const void *)cg_resident_kernel<SP, false>;
    }
};
template <>
struct Resident<LQCD_F64> {
    using R = double;
    static constexpr lqcd_prec XP = LQCD_F64;
    static constexpr int SITES = QUAD_SITES, BLOCK = QUAD_BLOCK;
    static const void *kernel(bool cluster)
    {
        return cluster ? (const void *)cg_resident_f64_kernel<true> : (const void *)cg_resident_f64_kernel<false>;
    }
};

// what the current device holds of the kernel at once, asked once per device:
// blocks of a cooperative launch, and whether a cluster of 16 blocks fits
struct ResidentCapacity {
    int blocks = 0;
    bool cluster16 = false;
};

constexpr int CLUSTER_MAX = 16;

static cudaLaunchConfig_t cluster_config(int nb, int block, cudaLaunchAttribute *attr, cudaStream_t s)
{
    int n = 1; // a power of two: blocks past the lattice have no sites
    while (n < nb) n *= 2;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = n;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <lqcd_prec SP>
static ResidentCapacity resident_capacity()
{
    constexpr int MAX_DEV = 64;
    static std::atomic<int> known[MAX_DEV]; // 1 + 2 blocks + cluster16
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) {
        cudaGetLastError();
        return {};
    }
    int c = known[dev].load(std::memory_order_relaxed);
    if (c == 0) {
        int coop = 0, sms = 0, per = 0, clusters = 0;
        if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, Resident<SP>::kernel(false), Resident<SP>::BLOCK, 0) !=
                cudaSuccess)
            coop = 0;
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = cluster_config(CLUSTER_MAX, Resident<SP>::BLOCK, &attr, nullptr);
        const void *f = Resident<SP>::kernel(true);
        if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&clusters, f, &cfg) != cudaSuccess)
            clusters = 0;
        cudaGetLastError();
        c = 1 + 2 * (coop ? sms * per : 0) + (clusters > 0 ? 1 : 0);
        known[dev].store(c, std::memory_order_relaxed);
    }
    return {(c - 1) / 2, ((c - 1) & 1) != 0};
}

template <lqcd_prec SP>
static lqcd_status launch_resident(CgRun &run, cudaStream_t s, bool *launched)
{
    using R = typename Resident<SP>::R;
    constexpr lqcd_prec XP = Resident<SP>::XP;
    constexpr int BLOCK = Resident<SP>::BLOCK;
    int nb = nblocks_for(run.Vh, Resident<SP>::SITES);
    const ResidentCapacity cap = resident_capacity<SP>();
    const bool cluster = cap.cluster16 && nb <= CLUSTER_MAX;
    if (!cluster && nb > (t_limits.blocks ? t_limits.blocks : cap.blocks)) return LQCD_OK;
    if (2 * (size_t)std::max(nb, CLUSTER_MAX) * sizeof(double) > run.ws->partials.bytes) return LQCD_OK;
    SpinorRef<SP> p = spinor_ref<SP>(run.P), r = spinor_ref<SP>(run.R), t = spinor_ref<SP>(run.T),
                  tmp = spinor_ref<SP>(run.TMP);
    SpinorRef<XP> xs = spinor_ref<XP>(run.XS);
    GaugeRef<SP> U = gauge_ref<SP>(run.UU);
    Geo g = make_geo(run.x->lat);
    R b = (R)(-run.k2);
    double *partials = (double *)run.ws->partials.p;
    CgScalars *sc = run.sc;
    ResidentLimits lim = t_limits;
    void *args[] = {&p, &r, &t, &tmp, &xs, &U, &g, &b, &partials, &nb, &sc, &lim};
    cudaError_t refused;
    if (cluster) {
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = cluster_config(nb, BLOCK, &attr, s);
        refused = cudaLaunchKernelExC(&cfg, Resident<SP>::kernel(true), args);
    } else {
        LQCD_CUDA(cudaMemsetAsync(&sc->bar, 0, 2 * sizeof(unsigned int), s)); // bar and bar_abort
        refused = cudaLaunchCooperativeKernel(Resident<SP>::kernel(false), dim3(nb), dim3(BLOCK), args, 0, s);
    }
    // A launch that the runtime refuses (the process may have fewer SMs than the
    // device's attributes say) leaves the solve as it was: it goes on kernel by
    // kernel.  An error of the context itself comes back from those launches.
    if (refused != cudaSuccess) {
        cudaGetLastError();
        run.resident_refused = true;
        return LQCD_OK;
    }
    LQCD_LAUNCHED();
    *launched = true;
    return LQCD_OK;
}

lqcd_status CgRun::iterate_resident(cudaStream_t s, bool *launched)
{
    *launched = false;
    if (resident_refused) return LQCD_OK;
    const lqcd_prec sp = mixed ? prm.sloppy : LQCD_F64;
    // timed hopping-term classes count and time single launches; the resident
    // kernel has the default form of the FP16+norm hopping term
    if (kernel_class_timed(dslash_class(sp))) return LQCD_OK;
    switch (sp) {
    case LQCD_F64: return launch_resident<LQCD_F64>(*this, s, launched);
    case LQCD_F32: return launch_resident<LQCD_F32>(*this, s, launched);
    case LQCD_F16N:
        if (kernel_class_timed(K_DSLASH_F16N_PLAIN) || plan.form != 2) return LQCD_OK;
        return launch_resident<LQCD_F16N>(*this, s, launched);
    case LQCD_BF16: return launch_resident<LQCD_BF16>(*this, s, launched);
    default: return LQCD_OK;
    }
}

} // namespace lqcd

extern "C" lqcd_status lqcd_solver_limits(int iterations, int polls, int blocks)
{
    using namespace lqcd;
    LQCD_REQUIRE(iterations >= 0 && polls >= 0 && blocks >= 0, "solver_limits: a limit is negative");
    const ResidentLimits dflt;
    t_limits.iters = iterations ? iterations : dflt.iters;
    t_limits.polls = polls ? polls : dflt.polls;
    t_limits.blocks = blocks;
    return LQCD_OK;
}
