// dslash_f64.cuh -- the FP64 hopping term with four threads per output site,
// shared by the kernels of dslash.cu, the resident solver (cg_resident.cu) and
// the sparse set-up of the solve service (service.cu).
//
// FP64 runs at two lanes a clock and SM, so the kernel is bound by the number
// of FP64 instructions and by how evenly they are dealt to the SMs.  With one
// thread per site a warp carries 32 sites' worth of them (about 900 x 16
// clocks), a lattice of a few thousand sites leaves most SMs without any, and
// all warps of an SM load, then compute, in step.  Here a block of 128 threads
// has 32 sites: warp mu forms the forward and the backward hop of direction mu
// (f and b: the spin rows 0, 1 get f + b, the rows 2, 3 are the fixed multiples
// of f - b, since the two projectors differ in sign), leaves its 24 reals in
// shared memory, and after one block barrier warp q adds the four directions'
// spin row q and takes it through the epilogue.  865 FP64 instructions per site
// (counted) instead of 980, the pipe 89% active on 16^3x32 (plain hop 108 us).
// FP64 solves of 32 iterations, one and four threads per site: 4^4 4.33 and
// 1.49 ms, 8^4 4.64 and 1.70 ms, 12^4 4.76 and 3.73 ms, 16^3x32 18.5 and 16.5
// ms, 24^4 39.9 and 39.1 ms; at 14^4, where one thread per site gave each SM one
// full block, 4.79 and 4.90 ms.
#pragma once

#include "dslash.cuh"
#include "spin.cuh"

namespace lqcd {

constexpr int QUAD_PER_SM = 4; // blocks the register budget is cut for

struct QuadF64 {
    double v[4][24][QUAD_SITES]; // [direction][real][site]: 24 KiB
};

struct RowF64 { // one spin row
    Cx<double> c[3];
};

template <int MU, bool DAG, bool COH>
__device__ __forceinline__ void quad_direction(QuadF64 &sh, const SpinorRef<LQCD_F64> &in,
                                               const GaugeRef<LQCD_F64> &U, int lane, int cb, int out_par, int nf,
                                               int nbk, bool flip_f, bool flip_b)
{
    constexpr int FS = DAG ? +1 : -1; // (1 + FS gamma) forward, (1 - FS gamma) backward
    Hs<double> f = mul_link(U.load<double>(MU, out_par, cb), project<MU, FS>(in.load<double, COH>(nf)));
    Hs<double> b = mul_link_dag(U.load<double>(MU, 1 - out_par, nbk), project<MU, -FS>(in.load<double, COH>(nbk)));
    if (MU == 3) {
        if (flip_f) negate(f);
        if (flip_b) negate(b);
    }
    // rows 2, 3 as sums of f and b with the signs taken in (a sign change of a
    // stored double would be one more FP64 instruction): P - Q in the order
    // that S = FS asks for, i (x + i y) = -y + i x
    const auto diff = [](double x, double y) { return FS > 0 ? x - y : y - x; };
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const Cx<double> f0 = f.c[0][c], f1 = f.c[1][c], b0 = b.c[0][c], b1 = b.c[1][c];
        Cx<double> r2, r3;
        if (MU == 0) { // -S i d1, -S i d0
            r2 = cx<double>(diff(f1.im, b1.im), diff(b1.re, f1.re));
            r3 = cx<double>(diff(f0.im, b0.im), diff(b0.re, f0.re));
        } else if (MU == 1) { // S d1, -S d0
            r2 = cx<double>(diff(f1.re, b1.re), diff(f1.im, b1.im));
            r3 = cx<double>(diff(b0.re, f0.re), diff(b0.im, f0.im));
        } else if (MU == 2) { // -S i d0, S i d1
            r2 = cx<double>(diff(f0.im, b0.im), diff(b0.re, f0.re));
            r3 = cx<double>(diff(b1.im, f1.im), diff(f1.re, b1.re));
        } else { // S d0, S d1
            r2 = cx<double>(diff(f0.re, b0.re), diff(f0.im, b0.im));
            r3 = cx<double>(diff(f1.re, b1.re), diff(f1.im, b1.im));
        }
        const Cx<double> r[4] = {f0 + b0, f1 + b1, r2, r3};
#pragma unroll
        for (int s = 0; s < 4; s++) {
            sh.v[MU][2 * (3 * s + c)][lane] = r[s].re;
            sh.v[MU][2 * (3 * s + c) + 1][lane] = r[s].im;
        }
    }
}

// Spin row `warp` of D in (DAG: D^dag) at site cb, the caller's block having
// its sites in lane order.  Every thread of the block calls it (live false: a
// lane without a site).  A second call needs a block barrier in between.
template <bool DAG, bool COH = false>
__device__ __forceinline__ RowF64 quad_row(QuadF64 &sh, const SpinorRef<LQCD_F64> &in, const GaugeRef<LQCD_F64> &U,
                                           const Geo &g, int cb, int out_par, bool live)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (live) {
        int c[4], nb[8];
        bool tf, tb;
        cb_coords(g, cb, out_par, c);
        cb_neighbours(g, cb, c, nb, tf, tb);
        const bool antip = g.t_bc < 0;
        switch (warp) {
        case 0: quad_direction<0, DAG, COH>(sh, in, U, lane, cb, out_par, nb[0], nb[1], false, false); break;
        case 1: quad_direction<1, DAG, COH>(sh, in, U, lane, cb, out_par, nb[2], nb[3], false, false); break;
        case 2: quad_direction<2, DAG, COH>(sh, in, U, lane, cb, out_par, nb[4], nb[5], false, false); break;
        default:
            quad_direction<3, DAG, COH>(sh, in, U, lane, cb, out_par, nb[6], nb[7], antip && tf, antip && tb);
            break;
        }
    }
    __syncthreads();
    RowF64 d;
    if (live) {
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const int i = 6 * warp + k;
            double v = sh.v[0][i][lane] + sh.v[1][i][lane] + sh.v[2][i][lane];
            if (g.aniso) v *= g.cs; // the spatial hops' weight (a uniform branch)
            v += sh.v[3][i][lane];
            (k & 1 ? d.c[k >> 1].im : d.c[k >> 1].re) = v;
        }
    }
    return d;
}

// spin row `warp` of a field at site cb
__device__ __forceinline__ RowF64 load_row(const SpinorRef<LQCD_F64> &f, int cb)
{
    RowF64 d;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const double2 v = f.d[(size_t)(3 * (threadIdx.x >> 5) + a) * f.Vh + cb];
        d.c[a] = cx<double>(v.x, v.y);
    }
    return d;
}
__device__ __forceinline__ void store_row(const SpinorRef<LQCD_F64> &f, int cb, const RowF64 &d)
{
#pragma unroll
    for (int a = 0; a < 3; a++)
        f.d[(size_t)(3 * (threadIdx.x >> 5) + a) * f.Vh + cb] = make_double2(d.c[a].re, d.c[a].im);
}
// x + b y, and |x|^2
__device__ __forceinline__ RowF64 row_xpay(const RowF64 &x, double b, const RowF64 &y)
{
    RowF64 d;
#pragma unroll
    for (int a = 0; a < 3; a++) d.c[a] = cx<double>(fma(b, y.c[a].re, x.c[a].re), fma(b, y.c[a].im, x.c[a].im));
    return d;
}
__device__ __forceinline__ double row_norm2(const RowF64 &x)
{
    double n = 0.0;
#pragma unroll
    for (int a = 0; a < 3; a++) n = fma(x.c[a].re, x.c[a].re, fma(x.c[a].im, x.c[a].im, n));
    return n;
}

} // namespace lqcd
