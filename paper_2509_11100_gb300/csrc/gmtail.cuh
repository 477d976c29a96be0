// gmtail.cuh -- the small dense part of an Arnoldi iteration on one warp.
#pragma once

#include "launch.cuh"

namespace relsim {

// where the cycle's Hessenberg factor, rotations and right-hand side live
struct GmTail {
    double *H, *cs, *sn, *gv, *rinv, *y;
    int m;
};

// |w - V h|^2 = <w,w> - |h|^2 of iteration j's sums [h_0 .. h_j, <w,w>] (two
// chains: every FP64 operation waits for the last)
__device__ __forceinline__ double gm_rest2(const double* sums, int j)
{
    double a = sums[j + 1], b = 0.0;
    for (int c = 0; c + 1 <= j; c += 2) {
        a -= sums[c] * sums[c];
        b -= sums[c + 1] * sums[c + 1];
    }
    if (j % 2 == 0) a -= sums[j] * sums[j];
    return a + b;
}

// The tail of iteration j: Hessenberg column, Givens rotations, residual
// estimate, stop test, and at a cycle's end the back substitution. Every lane
// of the warp calls it. The lanes form the products of the earlier rotations
// with the column together; only the chain through them is serial (one
// multiply-add a rotation: an FP64 operation takes a warp about 64 cycles, on
// one thread the tail took 5000). hn2 = gm_rest2, rhn its reciprocal root (0
// if hn2 <= 0), stop the residual to reach, total the iterations so far. go: 1
// for another iteration; kd: the columns to use when the cycle ends.
__device__ __forceinline__ void gm_tail_warp(const GmTail& t, const double* sums, int j, double hn2, double rhn,
                                             double stop, int total, int maxit, int lane, int& go, int& kd,
                                             int& status)
{
    const int m = t.m;
    go = 0;
    kd = 0;
    status = kGmOk;
    if (!isfinite(hn2)) {
        status = kGmNonfinite;
    } else if (j > 0 && hn2 < 1e-4 * sums[j + 1]) {
        kd = j;   // end the cycle without column j; restart from the true residual
    } else {
        const double hn = hn2 > 0.0 ? hn2 * rhn : 0.0;
        double v = sums[0];
        if (j == 0) v += 1.0;   // A = I + B
        for (int i0 = 0; i0 < j; i0 += 32) {
            const int i = i0 + lane, kc = min(32, j - i0);
            double p = 0.0, q = 0.0, c = 0.0, vm = 0.0;
            if (i < j) {
                double nxt = sums[i + 1];
                if (i + 1 == j) nxt += 1.0;
                c = t.cs[i];
                p = c * nxt;
                q = t.sn[i] * nxt;
            }
            for (int k = 0; k < kc; ++k) {
                if (lane == k) vm = v;
                v = -t.sn[i0 + k] * v + __shfl_sync(0xffffffffu, p, k);
            }
            if (i < j) t.H[i * m + j] = c * vm + q;
        }
        // one reciprocal square root for the rotation; where the squares
        // would leave the range, hypot and divisions
        const double r2 = v * v + hn * hn;
        double r, ri, c1, s1;
        if (r2 > 1e-200 && r2 < 1e200) {
            ri = rsqrt(r2);
            r = r2 * ri;
            c1 = v * ri;
            s1 = hn * ri;
        } else {
            r = hypot(v, hn);
            ri = r == 0.0 ? 0.0 : 1.0 / r;
            c1 = r == 0.0 ? 1.0 : v / r;
            s1 = r == 0.0 ? 0.0 : hn / r;
        }
        const double g0 = t.gv[j], g1 = -s1 * g0;
        __syncwarp();
        if (lane == 0) {
            t.cs[j] = c1;
            t.sn[j] = s1;
            t.rinv[j] = ri;
            t.H[j * m + j] = r;
            t.gv[j + 1] = g1;
            t.gv[j] = c1 * g0;
        }
        kd = j + 1;
        go = !(fabs(g1) <= stop || total >= maxit || hn == 0.0 || j + 1 >= m);
    }
    __syncwarp();
    if (!go)   // R y = g over the finished cycle's columns: y_i, then its column off the others
        for (int i = kd - 1; i >= 0; --i) {
            const double y = t.gv[i] * t.rinv[i];
            __syncwarp();
            for (int k = lane; k < i; k += 32) t.gv[k] -= t.H[k * m + i] * y;
            if (lane == 0) t.y[i] = y;
            __syncwarp();
        }
}

}  // namespace relsim
