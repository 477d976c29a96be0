// gmres.cu -- the control of the restarted GMRES solve (Sec. 2: the field
// solver is the implicit part of the method) decided on the device.
//
// The Arnoldi process runs on B = A - I with an FP64 Krylov basis (double-
// float pairs in the FP32 form of the 2D scheme with linear shapes). Its
// heavy kernels (operator with fused dot products, their reduction, the
// fused basis update) are in fields.cu; the small dense part stays on the
// device too: the Hessenberg column, the Givens rotations, the residual
// estimate, the stop tests and the triangular solve (gmtail.cuh) run on one
// warp of an extra block of the basis update, hidden behind it (as a launch
// of its own on one thread the tail took 7 us an iteration), and leave the
// launch arguments of the next iteration (GmDyn).
// With nothing left for the host to decide between iterations, the whole
// solve can run as a CUDA graph whose loops are conditional while nodes
// (the kernels set the loop conditions), or be driven from the host.
//
// When the norm of w - V h loses most of its digits (|w - V h|^2 < 1e-4
// |w|^2, so the new basis vector would not be orthogonal to the others), the
// cycle ends without that column and GMRES restarts from the true residual
// (at j = 0 the column is kept: the Krylov space is then nearly invariant).
#include "launch.cuh"

namespace relsim {
namespace {

__global__ void k_gm_begin(GmState* st, const double* __restrict__ sums)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const double bn = sqrt(sums[0]);
    st->bnorm = bn;
    st->beta = 0.0;
    st->relres = 0.0;
    st->total = 0;
    st->restarts = 0;
    st->kdim = 0;
    st->run = 0;
    st->inner = 0;
    st->status = isfinite(bn) ? kGmOk : kGmNonfinite;
    st->zero = bn == 0.0 ? 1 : 0;
    st->dyn.live = 0;
}

__global__ void k_gm_zero_x(const GmState* __restrict__ st, double* __restrict__ x, int64_t n)
{
    if (!st->zero) return;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        x[e] = 0.0;
}

__global__ void k_gm_cycle(GmState* st, const double* __restrict__ sums, GmPtrs p, GmParams q,
                           cudaGraphConditionalHandle cond, int has_cond)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int run = 0;
    if (st->run) st->restarts += 1;   // a cycle has ended
    if (st->status == kGmOk) {
        const double beta = sqrt(sums[0]);
        if (!isfinite(beta)) {
            st->status = kGmNonfinite;
        } else {
            st->beta = beta;
            const double rr = st->zero ? 0.0 : beta / st->bnorm;
            st->relres = rr;
            if (st->zero || rr <= q.tol) {
                // converged
            } else if (st->total >= q.maxit || st->restarts > q.maxit) {
                // (every cycle runs at least one iteration, so the second
                // bound only backs up the first: the loop always ends)
                st->status = kGmNotConverged;
            } else {
                run = 1;
                st->gv[0] = beta;
                st->kdim = 0;
                GmDyn& d = st->dyn;
                d.in = p.r;      // v_0 = r / beta, written to V_0 by iteration 0
                d.vj = p.V;
                d.out = p.w0;
                d.ds = p.ds0;
                d.s = 1.0 / beta;
                d.nv = 0;
            }
        }
    }
    st->run = run;
    st->inner = run;
    st->dyn.live = run;
    if (has_cond) cudaGraphSetConditional(cond, run);
}

__global__ void k_gm_arm(const GmState* __restrict__ st, cudaGraphConditionalHandle cond, int has_cond)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    if (has_cond) cudaGraphSetConditional(cond, st->run);
}

}  // namespace

cudaError_t gm_begin(GmState* st, const double* sums, cudaStream_t s)
{
    count_launches(1);
    k_gm_begin<<<1, 32, 0, s>>>(st, sums);
    return cudaGetLastError();
}

cudaError_t gm_zero_x(const GmState* st, double* x, int64_t n, cudaStream_t s)
{
    count_launches(1);
    const int64_t b = (n + 255) / 256;
    k_gm_zero_x<<<(int)(b < 152 * 4 ? (b < 1 ? 1 : b) : 152 * 4), 256, 0, s>>>(st, x, n);
    return cudaGetLastError();
}

cudaError_t gm_cycle(GmState* st, const double* sums, GmPtrs p, GmParams q, GmCond cond, cudaStream_t s)
{
    count_launches(1);
    k_gm_cycle<<<1, 32, 0, s>>>(st, sums, p, q, (cudaGraphConditionalHandle)cond.h, cond.has);
    return cudaGetLastError();
}

cudaError_t gm_arm(const GmState* st, GmCond cond, cudaStream_t s)
{
    count_launches(1);
    k_gm_arm<<<1, 32, 0, s>>>(st, (cudaGraphConditionalHandle)cond.h, cond.has);
    return cudaGetLastError();
}

}  // namespace relsim
