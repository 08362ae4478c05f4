// dslash.cuh -- internal interface of the Wilson hopping kernels and the CG
// scalar block shared by dslash.cu and cg.cu.
#pragma once

#include "lqcd_internal.cuh"

namespace lqcd {

// Device-resident scalars of one CG solve.  The reduction kernels update them
// and set `pause` when the host must act (convergence of the iterated
// residual, a reliable update, maxiter, a non-finite value); every iteration
// kernel returns immediately while `pause` is set.
struct CgScalars {
    double rr;      // |r|^2 of the current residual
    double pAp;     // <p, A p> = |Mhat p|^2
    double alpha;   // rr / pAp
    double beta;    // rr_new / rr
    double rr_new;  // |r|^2 after the update
    double stop2;   // tol^2 |b|^2
    double delta2;  // reliable-update threshold factor delta^2 (0: none)
    double maxrr2;  // max |r|^2 since the last reliable update
    int pause;
    int reason;     // 1 iterated residual converged, 2 reliable update due, 3 maxiter, 4 non-finite
    int iter;
    int maxiter;
    unsigned int arrive; // blocks of the current reduction that have stored their partial (0 between kernels)
    unsigned int bar, bar_abort; // the resident solver's grid barrier: arrivals, and a wait that gave up
};

enum {
    PAUSE_NONE = 0,
    PAUSE_CONVERGED = 1,
    PAUSE_RELIABLE = 2,
    PAUSE_MAXITER = 3,
    PAUSE_NONFINITE = 4,
    PAUSE_TIMEOUT = 5 // a wait of the resident solver's grid barrier gave up
};

// alpha = rr / pAp from the summed pAp (a non-positive or non-finite pAp pauses)
__device__ __forceinline__ void cg_pap_step(CgScalars *sc, double pAp)
{
    sc->pAp = pAp;
    if (!(pAp > 0.0) || !isfinite(pAp)) {
        sc->alpha = 0.0;
        sc->pause = 1;
        sc->reason = PAUSE_NONFINITE;
    } else {
        sc->alpha = sc->rr / pAp;
    }
}

// the new |r|^2: the pause decision (non-finite, converged, reliable update
// due, maxiter -- in that order) or beta = rr_new / rr
__device__ __forceinline__ void cg_rr_step(CgScalars *sc, double rr_new)
{
    sc->rr_new = rr_new;
    sc->iter += 1;
    int reason = PAUSE_NONE;
    if (!isfinite(rr_new))
        reason = PAUSE_NONFINITE;
    else if (rr_new <= sc->stop2)
        reason = PAUSE_CONVERGED;
    else if (sc->delta2 > 0.0 && rr_new < sc->delta2 * sc->maxrr2)
        reason = PAUSE_RELIABLE;
    else if (sc->iter >= sc->maxiter)
        reason = PAUSE_MAXITER;
    if (reason != PAUSE_NONE) {
        sc->pause = 1;
        sc->reason = reason;
    } else {
        sc->beta = rr_new / sc->rr;
        sc->rr = rr_new;
        sc->maxrr2 = fmax(sc->maxrr2, rr_new);
    }
}

// Fixed-order sum of partials[0..n) by one block of BLOCK threads: thread i
// adds partials[i], partials[i + BLOCK], ... in that order (sixteen loads in
// flight, read from L2 since other blocks wrote them), then the warps reduce
// by shuffles and warp 0 adds the warp totals in warp order.  The result,
// valid in thread 0, does not depend on which block computes it.  Warps past
// the n partials have nothing to add and leave the FP64 pipe to the others.
template <int BLOCK>
__device__ __forceinline__ double block_final_sum(const double *partials, int n)
{
    __shared__ double wsum[BLOCK / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp * 32 < n) {
        double s = 0.0;
        int i = threadIdx.x;
        for (; i + 15 * BLOCK < n; i += 16 * BLOCK) {
            double v[16];
#pragma unroll
            for (int k = 0; k < 16; k++) v[k] = __ldcg(partials + i + k * BLOCK);
#pragma unroll
            for (int k = 0; k < 16; k++) s += v[k];
        }
        for (; i < n; i += BLOCK) s += __ldcg(partials + i);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0) wsum[warp] = s;
    }
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < BLOCK / 32 && w * 32 < n; w++) t += wsum[w];
    return t;
}

// The scalar step of a CG reduction, done by the grid that produced the block
// partial sums: every block calls it after its thread 0 stored the block's
// partial; thread 0 publishes that store and counts the block in sc->arrive;
// the block that arrives last sums all nblocks partials in a fixed order,
// applies the pAp step (RR false) or the rr step (RR true) and resets the
// count.  No block waits for another.
template <int BLOCK, bool RR>
__device__ __forceinline__ void cg_finish(CgScalars *sc, const double *partials, int nblocks)
{
    __shared__ int last;
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned int prev = atomicAdd(&sc->arrive, 1u);
        last = prev == (unsigned int)(nblocks - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const double total = block_final_sum<BLOCK>(partials, nblocks);
    if (threadIdx.x == 0) {
        sc->arrive = 0;
        if (RR)
            cg_rr_step(sc, total);
        else
            cg_pap_step(sc, total);
    }
}

#ifndef LQCD_DS_BLOCK
#define LQCD_DS_BLOCK 128
#endif
// threads per block of the hopping-term kernels (one output site each)
constexpr int DS_BLOCK = LQCD_DS_BLOCK;
// FP64 (dslash_f64.cuh): four threads per site
constexpr int QUAD_SITES = 32, QUAD_BLOCK = 4 * QUAD_SITES;

inline int dslash_blocks(int Vh) { return nblocks_for(Vh, DS_BLOCK); }

// The pAp step that the block partials of an earlier launch wait for, done by
// the first block of a plain 16-bit hop, which the CG runs between the reducing
// hop that stores them and the one that needs alpha.  The reducing hop's blocks
// then end with their stores; with the step in its last block (cg_finish) each
// of them waits for a fence and an atomic.  FP16+norm axpy hop on 32^3x64 about
// 9 us shorter (77 -> 68 us), sixteen batched chains 30.4 -> 29.6 ms.
// A step that pauses the solve (a pAp that is not positive) sets the flag that
// this hop's other blocks read when they start: some of them may do their sites
// and some not, and nothing reads the hop's output, since the CG-update hop
// behind it sees the pause.
struct PapStep {
    CgScalars *sc = nullptr; // NULL: none
    const double *partials = nullptr;
    int n = 0;
};
template <int BLOCK>
__device__ __forceinline__ void pap_step(const PapStep &f)
{
    const double total = block_final_sum<BLOCK>(f.partials, f.n);
    if (threadIdx.x == 0) cg_pap_step(f.sc, total);
}

// The process-wide settings of the FP16+norm hopping term (dslash_form_set and
// the autotuner's table), read once for all launches that have to agree: the
// form decides whether a plain hop takes a PapStep, the block size how many
// partials a reducing hop stores.  A solve keeps the one it started with, so
// that a change by another thread meanwhile does not reach it.
struct HopPlan {
    int form = 2;
    int block = DS_BLOCK; // threads per block of the packed FP16+norm kernels
};
HopPlan hop_plan(const lqcd_field *in);
// whether the plain hop of this storage takes a PapStep (the 16-bit packed forms)
inline bool hop_takes_pap_step(lqcd_prec p, const HopPlan &plan)
{
    return p == LQCD_BF16 || (p == LQCD_F16N && plan.form == 2);
}
// block partials that a reducing hop on this lattice stores
inline int hop_partials(const lqcd_field *in, const HopPlan &plan)
{
    const int sites = in->prec == LQCD_F64                       ? QUAD_SITES
                      : in->prec == LQCD_F16N && plan.form == 2 ? plan.block
                                                                 : DS_BLOCK;
    return nblocks_for(in->Vh, sites);
}

// out = D_{out<-in} in (dagger: D^dag).  Parities from the field kinds.
// pap (optional, hop_takes_pap_step): applied beside the hop.  plan (here and
// below): NULL takes the settings of the moment.
lqcd_status dslash_plain(lqcd_field *out, const lqcd_field *U, const lqcd_field *in, int dagger, const int *skip,
                         cudaStream_t s, PapStep pap = {}, const HopPlan *plan = nullptr);

// out = x + b D in; if partials != NULL also the per-block partial sums of
// |out|^2 (hop_partials of them), and if fin != NULL the last block then
// sums them and applies the CG pAp step to fin (cg_finish).
lqcd_status dslash_xpay(lqcd_field *out, const lqcd_field *U, const lqcd_field *in, int dagger, const lqcd_field *x,
                        double b, double *partials, const int *skip, cudaStream_t s, CgScalars *fin = nullptr,
                        const HopPlan *plan = nullptr);

// CG update fused into the last half of Mhat^dag Mhat:
//   Ap = t + b D in;  xs += alpha p;  r -= alpha Ap;  partials of |r|^2,
// whose last block applies the CG rr step to sc (alpha from sc).  t, r, p in
// the sloppy precision of in; xs F64 (plain FP64 solve) or F32 (mixed solve).
lqcd_status dslash_cg(const lqcd_field *U, const lqcd_field *in, int dagger, const lqcd_field *t, double b,
                      lqcd_field *xs, lqcd_field *r, const lqcd_field *p, double *partials, CgScalars *sc,
                      cudaStream_t s, const HopPlan *plan = nullptr);

// the FP16+norm hopping-term form: 2 prefetched links with packed FP32x2
// arithmetic (default), 1 prefetched links, 0 gathered; returns the previous
// form (form < 0: query; -1 and an error for an unknown form)
int dslash_form_set(int form);

// out = D in, or x + b D in if x is given, with float-float fields and links
// (precision code 4; dslash_df.cu)
lqcd_status dslash_df_launch(lqcd_field *out, const lqcd_field *U, const lqcd_field *in, int dagger,
                             const lqcd_field *x, double b, const int *skip, cudaStream_t s);

// the accurate residual's last float-float term: r = bsrc - (x + b D^dag in),
// with one partial of |r|^2 per block of DF_SITES sites in partials[0 ..
// nblocks_for(Vh, DF_SITES)) (dslash_df.cu)
lqcd_status dslash_df_residual(lqcd_field *r, const lqcd_field *U, const lqcd_field *in, const lqcd_field *x,
                               double b, const lqcd_field *bsrc, double *partials, cudaStream_t s);

} // namespace lqcd
