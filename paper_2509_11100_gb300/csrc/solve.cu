// solve.cu -- the whole restarted GMRES solve of the 2D implicit field
// equation (linear shapes) in one cooperative launch, for grids whose tiles
// all fit on the GPU at once.
//
// On such grids an Arnoldi iteration is a few microseconds of arithmetic, and
// the iteration as separate launches (operator, reduction, basis update, the
// control's Givens rotations on one thread, the loop's condition) is bound by
// the launches and by each kernel's own start: at 128x64 (FP32 form, 5
// iterations) the solve took 261 us of launches, here 66; at 251x99 324 and
// 95; in FP64 at 64x32 (8 iterations) 440 and 104, at 256x128 (13) 820 and
// 352. What is left is the FP64 pipe (FP64 form), the two grid barriers (about
// 1.2 us each) and the serial control. A block keeps one tile of 32 x Y nodes
// for the whole solve: its mass-matrix rows are brought into shared memory
// once, w and v_j stay in registers, and two grid barriers per iteration
// separate what the tiles exchange (the partial dot products, and v_{j+1} for
// the halos). Every block adds up all partial sums itself, in one fixed
// order, so all take the same decisions without a further exchange; the
// Hessenberg column, its Givens rotations and the stop test (gmtail.cuh) run
// on one warp of block 0 while the others update the basis. Same
// iteration, stop tests, restart rule and arithmetic per vector element as
// the launches it replaces; only the order of the dot products' partial
// sums differs.
#include "gmtail.cuh"
#include "launch.cuh"
#include "opcore.cuh"

namespace relsim {
namespace {

constexpr int kSX = 32;                       // tile width
constexpr int kSVW = kSX + 2;                 // staged input row
constexpr int kSCW = kSX + 1;                  // its centres
constexpr int kSU = 5;                         // staged values per thread at most: 3 (Y + 2) 34 / threads
constexpr long long kGridPolls = 1ll << 24;   // bounded wait at a grid barrier

template <typename T>
struct SolveArgs {
    const T* M;
    const double* b;
    double* x;
    double* r;
    double* V;
    int64_t ldv;
    GridP g;
    int Y, tma, m, maxit;
    double tol;
    double* partial;   // [sum][block]
    GmState* st;
    int* err;
};

// an element of a GMRES vector
template <bool DF>
struct Vec;
template <>
struct Vec<true> {
    using E = dfl;
    static __device__ __forceinline__ E zero() { return dfl{0.f, 0.f}; }
    static __device__ __forceinline__ E load(const double* v, int64_t k)
    {
        const float2 a = __ldcg(reinterpret_cast<const float2*>(v) + k);
        return dfl{a.x, a.y};
    }
    // a value that this thread wrote itself: L1 may keep it
    static __device__ __forceinline__ E load_own(const double* v, int64_t k) { return reinterpret_cast<const dfl*>(v)[k]; }
    static __device__ __forceinline__ void store(double* v, int64_t k, E a) { reinterpret_cast<dfl*>(v)[k] = a; }
    static __device__ __forceinline__ E from(double a) { return df_from_double(a); }
    static __device__ __forceinline__ E mul(E a, E b) { return df_mul(a, b); }
    static __device__ __forceinline__ double to_double(E a) { return df_to_double(a); }
    static __device__ __forceinline__ E add(E a, E b) { return df_add(a, b); }
    static __device__ __forceinline__ E warp_total(E a) { return df_warp_sum(a); }
};
template <>
struct Vec<false> {
    using E = double;
    static __device__ __forceinline__ E zero() { return 0.0; }
    static __device__ __forceinline__ E load(const double* v, int64_t k) { return __ldcg(v + k); }
    static __device__ __forceinline__ E load_own(const double* v, int64_t k) { return v[k]; }
    static __device__ __forceinline__ void store(double* v, int64_t k, E a) { v[k] = a; }
    static __device__ __forceinline__ E from(double a) { return a; }
    static __device__ __forceinline__ E mul(E a, E b) { return a * b; }
    static __device__ __forceinline__ double to_double(E a) { return a; }
    static __device__ __forceinline__ E add(E a, E b) { return a + b; }
    static __device__ __forceinline__ E warp_total(E a) { return warp_sum(a); }
};
// a running sum of products of vector elements
template <bool DF>
struct Sum;
template <>
struct Sum<true> : Dot2 {
    __device__ __forceinline__ Sum() {}
    __device__ __forceinline__ explicit Sum(dfl a)
    {
        s = a.hi;
        e = a.lo;
    }
};
template <>
struct Sum<false> {
    double s = 0.0;
    __device__ __forceinline__ Sum() {}
    __device__ __forceinline__ explicit Sum(double a) : s(a) {}
    __device__ __forceinline__ void add(double a, double b) { s += a * b; }
    __device__ __forceinline__ void sub(double a, double b) { s -= a * b; }
    __device__ __forceinline__ double value() const { return s; }
};

// Threads of a block. FP32: a thread a node, at least four warps. FP64: up to
// tiles of two rows four threads a node, three of which apply the mass matrix
// to a component each and one the curl: the FP64 pipes of an SM's four
// quarters each take a warp's operation in about 64 cycles, and one row of
// nodes would use a single quarter.
template <typename T>
__host__ __device__ constexpr int solve_parts(int Y)
{
    return sizeof(T) == 8 && Y <= 2 ? 4 : 1;
}
template <typename T>
__host__ __device__ constexpr int solve_threads(int Y)
{
    return 32 * Y * solve_parts<T>(Y) < 128 ? 128 : 32 * Y * solve_parts<T>(Y);
}
template <typename T>
__host__ __device__ constexpr size_t solve_smem(int Y)
{
    // mass-matrix rows, halo columns, the staged input and its curl in T (rounded up to 16
    // bytes), the dot products of kOpChunk sums
    const size_t t = ((size_t)(Y + 1) * kSX * kMBlock + (size_t)(Y + 1) * 2 * kMBlock + 3 * (size_t)(Y + 2) * kSVW +
                      3 * (size_t)(Y + 1) * kSCW) *
                     sizeof(T);
    return (t + 15) / 16 * 16 + (size_t)kOpChunk * solve_threads<T>(Y) * 8;
}

template <typename T, bool DF, bool TR>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1)
k_gm_solve(const __grid_constant__ SolveArgs<T> a)
{
    using W = Vec<DF>;
    using E = typename W::E;
    extern __shared__ __align__(128) unsigned char solve_dyn[];
    __shared__ uint64_t mbar;
    __shared__ double sums[kMaxRestart + 2];
    __shared__ E hs[kMaxRestart + 2];
    __shared__ E scale;          // 1/|w - V h|
    __shared__ double shn2, srn;   // |w - V h|^2, 1/|w - V h|
    __shared__ double cs[kMaxRestart], sn[kMaxRestart], gv[kMaxRestart + 1],
        rinv[kMaxRestart];   // block 0's
    __shared__ double sbeta, sbn;
    __shared__ int srun, sstatus, szero;
    __shared__ unsigned sctl;    // the tail's decision: inner | status << 8 | kdim << 16
    __shared__ int sok;
    const int nx = a.g.nx, ny = a.g.ny, nc = a.g.ncell, Y = a.Y;
    const int NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = NT >> 5;
    const int nblk = gridDim.x, blk = blockIdx.x;
    T* const Mm = reinterpret_cast<T*>(solve_dyn);         // [Y + 1][32 * 45]: rows j0-1 ..
    T* const Mh = Mm + (Y + 1) * kSX * kMBlock;            // [Y + 1][2][45]: columns i0-1 and i0+tw
    T* const sv = Mh + (Y + 1) * 2 * kMBlock;              // [3][Y + 2][34]
    T* const sc = sv + 3 * (Y + 2) * kSVW;                 // [3][Y + 1][33]: curl_c v on the centres
    E* const buf = reinterpret_cast<E*>(solve_dyn + solve_smem<T>(Y) - (size_t)kOpChunk * NT * 8);   // [kOpChunk][NT]
    const int tilesx = (nx + kSX - 1) / kSX;
    const int i0 = (blk % tilesx) * kSX, j0 = (blk / tilesx) * Y;
    const int tw = min(kSX, nx - i0), th = min(Y, ny - j0);
    const int tx = lane, ty = wid % Y, part = wid / Y;   // part 0 owns the node
    const bool there = tx < tw && ty < th, active = there && part == 0;
    const bool split = solve_parts<T>(Y) > 1;
    const int64_t gidx = there ? (int64_t)(j0 + ty) * nx + i0 + tx : 0;
    // the residual's sums apart from the iteration's: a block writes the first
    // iteration's while another may still read the residual's
    double* const rpart = a.partial + (int64_t)(a.m + 2) * nblk;
    unsigned target = 0;

    // a barrier over the grid (every wait bounded, and left early once a
    // block raised the error flag); thread 0 then reads the tail's decision
    auto grid_sync = [&]() -> bool {
        __syncthreads();
        target += (unsigned)nblk;
        if (tid == 0) {
            __threadfence();
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&a.st->bar) : "memory");
            int ok = 0;
            for (long long it = 0; it < kGridPolls; ++it) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&a.st->bar) : "memory");
                if (v >= target) {
                    ok = 1;
                    break;
                }
                if ((it & 255) == 255 && (*(volatile int*)a.err & 2)) break;
            }
            if (!ok) atomicOr(a.err, 2);
            sctl = *(volatile unsigned*)&a.st->ctl;
            sok = ok;
        }
        __syncthreads();
        return sok != 0;
    };
    // the totals of nq sums over all blocks' partials, the same order in every
    // block: 16 lanes a sum, eight loads in flight a lane
    auto grid_sums = [&](const double* part, int nq) {
        for (int q0 = 0; q0 < nq; q0 += NT / 16) {
            const int q = q0 + tid / 16;
            if (__all_sync(0xffffffffu, q >= nq)) break;   // the warp has no sum left
            const double* p = part + (int64_t)(q < nq ? q : 0) * nblk;
            double t = 0.0;
            for (int ib = 0; ib < nblk; ib += 128) {
                double u[8];
                const int i = ib + tid % 16;
#pragma unroll
                for (int h = 0; h < 8; ++h) u[h] = i + 16 * h < nblk ? __ldcg(p + i + 16 * h) : 0.0;
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    if (ib + 16 * h >= nblk) break;   // a branch: no FP64 work for nothing
                    t += u[h];
                }
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (tid % 16 == 0 && q < nq) sums[q] = t;
        }
        __syncthreads();
    };
    // the block's partials of the sums q0 .. q0 + kc - 1, whose thread values lie in buf
    auto block_partials = [&](double* part, int q0, int kc) {
        __syncthreads();
        for (int c = wid; c < kc; c += nw) {
            E t = W::zero();
            for (int m = 0; m < nw && m < Y; ++m) t = W::add(t, buf[c * NT + m * 32 + lane]);
            t = W::warp_total(t);
            if (lane == 0) part[(int64_t)(q0 + c) * nblk + blk] = W::to_double(t);
        }
        __syncthreads();
    };
    // this thread's share of the tile with its 1-node halo: where its values
    // lie in a vector and in shared memory (the same for every vector)
    int gat[kSU], sat[kSU];
    {
        const int vw = tw + 2, vh = th + 2;
#pragma unroll
        for (int u = 0; u < kSU; ++u) {
            const int q = tid + u * NT;
            const int k = q / (vh * vw), rem = q - k * (vh * vw), r = rem / vw, cc = rem - r * vw;
            const bool in = q < 3 * vh * vw;
            gat[u] = in ? k * nc + wrap1(j0 - 1 + r, ny) * nx + wrap1(i0 - 1 + cc, nx) : 0;
            sat[u] = in ? (k * (Y + 2) + r) * kSVW + cc : -1;
        }
    }
    // the input on the tile and its halo, in T (double-float: the leading
    // part), times s; all of a thread's loads in flight together
    auto stage = [&](const double* in, bool scaled, T s) {
        E t[kSU];
#pragma unroll
        for (int u = 0; u < kSU; ++u) t[u] = sat[u] >= 0 ? W::load(in, gat[u]) : W::zero();
#pragma unroll
        for (int u = 0; u < kSU; ++u) {
            T val;
            if constexpr (DF) val = (T)t[u].hi;
            else val = (T)t[u];
            if (scaled) val *= s;
            if (sat[u] >= 0) sv[sat[u]] = val;
        }
        __syncthreads();
    };
    auto blockrow = [&](int c, int r) -> const T* {
        return c < 0 ? Mh + ((r + 1) * 2) * kMBlock
                     : (c >= tw ? Mh + ((r + 1) * 2 + 1) * kMBlock : Mm + (r + 1) * kSX * kMBlock + c * kMBlock);
    };
    // curl_c v on the tile's centres, each formed once (all threads; v staged)
    auto centres = [&]() {
        for (int q = tid; q < (th + 1) * (tw + 1); q += NT) {
            const int r = q / (tw + 1), c = q - r * (tw + 1);
            T C[3];
            op_curl_c<T>([&](int k, int p, int o) { return sv[(k * (Y + 2) + r + o) * kSVW + c + p]; },
                         gc<T>(a.g).hdx, gc<T>(a.g).hdy, C);
#pragma unroll
            for (int k = 0; k < 3; ++k) sc[(k * (Y + 1) + r) * kSCW + c] = C[k];
        }
        __syncthreads();
    };
    // B v of the node (v staged, its curl on the centres formed), left with
    // the node's owner; every thread of the block calls it
    auto apply = [&](T (&bv)[3]) {
        const T td = gc<T>(a.g).td;
        auto cen = [&](int k, int ca, int cb) { return sc[(k * (Y + 1) + ty + cb) * kSCW + tx + ca]; };
        auto stencil = [&](T (&f)[3][3][3], const T* (&Mn)[4]) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int p = 0; p < 3; ++p)
#pragma unroll
                    for (int q = 0; q < 3; ++q) f[k][p][q] = sv[(k * (Y + 2) + ty + q) * kSVW + tx + p];
            Mn[0] = blockrow(tx - 1, ty) + 9;
            Mn[1] = blockrow(tx + 1, ty - 1) + 18;
            Mn[2] = blockrow(tx, ty - 1) + 27;
            Mn[3] = blockrow(tx - 1, ty - 1) + 36;
        };
        T cc[3], mv[3];
        if (sizeof(T) == 8 && split) {
            T* const pb = reinterpret_cast<T*>(buf);   // [4][32 Y]: M v by component, then curl curl v apart
            const int at = ty * 32 + tx, n = 32 * Y;
            if (there && part < 3) {
                T f[3][3][3];
                const T* Mn[4];
                stencil(f, Mn);
                pb[part * n + at] = op_mass_row<T, const T*, TR>(f, blockrow(tx, ty), Mn, part);
            } else if (there) {
                op_curl_n<T>(cen, gc<T>(a.g).hdx, gc<T>(a.g).hdy, cc);
#pragma unroll
                for (int k = 0; k < 3; ++k) pb[(3 + k) * n + at] = td * td * cc[k];
            }
            __syncthreads();
            if (active)
#pragma unroll
                for (int k = 0; k < 3; ++k) bv[k] = pb[(3 + k) * n + at] + td * pb[k * n + at];
            __syncthreads();
        } else if (active) {
            T f[3][3][3];
            const T* Mn[4];
            stencil(f, Mn);
            op_curl_n<T>(cen, gc<T>(a.g).hdx, gc<T>(a.g).hdy, cc);
            op_mass<T, const T*, TR>(f, blockrow(tx, ty), Mn, mv);
#pragma unroll
            for (int k = 0; k < 3; ++k) bv[k] = td * td * cc[k] + td * mv[k];
        }
    };
    // r = b - A x of the node; stores r, leaves the products for the sums
    E own[3] = {W::zero(), W::zero(), W::zero()};
    auto residual = [&](const E (&xo)[3], bool with_b) {
        Sum<DF> rr, bb;
        T bv[3] = {T(0), T(0), T(0)};
        centres();
        apply(bv);
        if (active) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int64_t at = (int64_t)k * nc + gidx;
                const E bk = W::load(a.b, at);
                if constexpr (DF) own[k] = df_sub(bk, df_add_f(xo[k], (float)bv[k]));
                else own[k] = bk - (xo[k] + (double)bv[k]);
                W::store(a.r, at, own[k]);
                rr.add(own[k], own[k]);
                if (with_b) bb.add(bk, bk);
            }
        }
        buf[tid] = rr.value();
        if (with_b) buf[NT + tid] = bb.value();
        block_partials(rpart, 0, with_b ? 2 : 1);
    };

    int total = 0, restarts = 0, status = kGmOk, kdim = 0;   // the same in every thread of every block
    double bn = 0.0;
    // the tail of iteration j, by one warp of block 0
    auto tail = [&](int j) {
        int go, kd, stt;
        gm_tail_warp(GmTail{a.st->H, cs, sn, gv, rinv, a.st->y, a.m}, sums, j, shn2, srn, a.tol * bn, total, a.maxit,
                     lane, go, kd, stt);
        if (lane == 0)
            *(volatile unsigned*)&a.st->ctl = (unsigned)go | (unsigned)stt << 8 | (unsigned)kd << 16;
    };

    // ---- the tile's mass matrix, for the whole solve
    bool ok = true;
    if (a.tma) {
        if (tid == 0) {
            mbar_init(&mbar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            const unsigned bytes = (unsigned)(tw * kMBlock * sizeof(T));
            mbar_expect_tx_arrive(&mbar, bytes * (unsigned)(th + 1));
            for (int r = 0; r <= th; ++r) {
                const int jr = wrap1(j0 - 1 + r, ny);
                bulk_g2s(Mm + r * kSX * kMBlock, a.M + ((int64_t)jr * nx + i0) * kMBlock, bytes, &mbar);
            }
        }
    } else {
        for (int r = 0; r <= th; ++r) {
            const T* src = a.M + ((int64_t)wrap1(j0 - 1 + r, ny) * nx + i0) * kMBlock;
            for (int q = tid; q < tw * kMBlock; q += NT) Mm[r * kSX * kMBlock + q] = ld(src + q);
        }
    }
    for (int q = tid; q < (th + 1) * 2 * kMBlock; q += NT) {
        const int r = q / (2 * kMBlock), side = (q / kMBlock) % 2, e = q % kMBlock;
        const int ic = side == 0 ? wrap1(i0 - 1, nx) : wrap1(i0 + tw, nx);
        Mh[q] = ld(a.M + ((int64_t)wrap1(j0 - 1 + r, ny) * nx + ic) * kMBlock + e);
    }
    E xo[3] = {W::zero(), W::zero(), W::zero()};
    if (active)
#pragma unroll
        for (int k = 0; k < 3; ++k) xo[k] = W::load(a.x, (int64_t)k * nc + gidx);
    stage(a.x, false, T(1));   // its barrier also publishes the mbarrier
    if (a.tma) ok = mbar_wait(&mbar, 0, kOpMaxPolls);
    if (!ok) atomicOr(a.err, 2);

    double relres = 0.0;
    if (__syncthreads_and(ok)) {
        residual(xo, true);
        ok = grid_sync();
        for (bool first = true; ok; first = false) {
            // ---- the start of a cycle: converged, out of iterations, or run
            grid_sums(rpart, first ? 2 : 1);
            if (tid == 0) {
                if (first) {
                    sbn = sqrt(sums[1]);
                    szero = sbn == 0.0;
                }
                const double beta = sqrt(sums[0]);
                const int st0 = first && !isfinite(sbn) ? kGmNonfinite : kGmOk;
                sbeta = beta;
                sstatus = st0;
                srun = 0;
                if (st0 == kGmOk) {
                    if (szero) {
                    } else if (!isfinite(beta)) sstatus = kGmNonfinite;
                    else if (beta / sbn <= a.tol) {
                    } else if (total >= a.maxit || restarts > a.maxit) sstatus = kGmNotConverged;
                    else srun = 1;
                }
                gv[0] = beta;
            }
            __syncthreads();
            bn = sbn;
            status = sstatus;
            if (status != kGmNonfinite) relres = szero ? 0.0 : sbeta / sbn;
            if (szero && active)
#pragma unroll
                for (int k = 0; k < 3; ++k) W::store(a.x, (int64_t)k * nc + gidx, W::zero());
            if (!srun) break;
            const double s0 = 1.0 / sbeta;
            bool inner = true;
            for (int j = 0; inner; ++j) {
                if (j == 0) {
                    const E se = W::from(s0);
                    if (active)
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            own[k] = W::mul(own[k], se);
                            W::store(a.V, (int64_t)k * nc + gidx, own[k]);
                        }
                    stage(a.r, true, (T)s0);
                } else {
                    stage(a.V + (int64_t)j * a.ldv, false, T(1));
                }
                centres();
                T bv[3] = {T(0), T(0), T(0)};
                apply(bv);
                E w[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    if constexpr (DF) w[k] = df_from_f((float)bv[k]);
                    else w[k] = (double)bv[k];
                }
                // <w, V_0> .. <w, V_{j-1}>, <w, v_j>, <w, w>
                const int nq = j + 2;
                for (int q0 = 0; q0 < nq; q0 += kOpChunk) {
                    const int kc = min(kOpChunk, nq - q0);
                    E vq[kOpChunk][3];
#pragma unroll
                    for (int c = 0; c < kOpChunk; ++c)
#pragma unroll
                        for (int k = 0; k < 3; ++k)
                            vq[c][k] = active && q0 + c < j
                                           ? W::load_own(a.V + (int64_t)(q0 + c) * a.ldv, (int64_t)k * nc + gidx) : W::zero();
#pragma unroll
                    for (int c = 0; c < kOpChunk; ++c) {
                        if (c >= kc) break;
                        const int q = q0 + c;
                        Sum<DF> d;
                        if (active) {
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                const E o = q == j + 1 ? w[k] : (q == j ? own[k] : vq[c][k]);
                                if constexpr (DF) d.add(o, (float)bv[k]);
                                else d.add(o, w[k]);
                            }
                        }
                        buf[c * NT + tid] = d.value();
                    }
                    block_partials(a.partial, q0, kc);
                }
                if (!(ok = grid_sync())) break;
                grid_sums(a.partial, nq);
                if (tid < nq) hs[tid] = W::from(sums[tid]);
                if (tid == 0) {
                    const double h2 = gm_rest2(sums, j);
                    shn2 = h2;
                    srn = h2 > 0.0 ? rsqrt(h2) : 0.0;
                    scale = W::from(srn);
                }
                __syncthreads();
                ++total;
                if (blk == 0 && wid == nw - 1) tail(j);
                // v_{j+1} = (w - V h)/|w - V h|
                if (active) {
                    Sum<DF> d[3] = {Sum<DF>(w[0]), Sum<DF>(w[1]), Sum<DF>(w[2])};
                    for (int c0 = 0; c0 < j; c0 += 4) {
                        E vv[4][3];
#pragma unroll
                        for (int c = 0; c < 4; ++c)
#pragma unroll
                            for (int k = 0; k < 3; ++k)
                                vv[c][k] = c0 + c < j
                                               ? W::load_own(a.V + (int64_t)(c0 + c) * a.ldv, (int64_t)k * nc + gidx)
                                               : W::zero();
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            if (c0 + c >= j) break;
#pragma unroll
                            for (int k = 0; k < 3; ++k) d[k].sub(hs[c0 + c], vv[c][k]);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        d[k].sub(hs[j], own[k]);
                        own[k] = W::mul(d[k].value(), scale);
                        W::store(a.V + (int64_t)(j + 1) * a.ldv, (int64_t)k * nc + gidx, own[k]);
                    }
                }
                if (!(ok = grid_sync())) break;
                inner = (sctl & 255u) != 0;
                status = (int)(sctl >> 8 & 255u);
                kdim = (int)(sctl >> 16);
            }
            if (!ok || status == kGmNonfinite) break;
            // ---- the end of a cycle: x += V y, the true residual
            ++restarts;
            if (tid < kdim) hs[tid] = W::from(__ldcg(&a.st->y[tid]));
            __syncthreads();
            if (active) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    Sum<DF> d(xo[k]);
                    for (int c = 0; c < kdim; ++c)
                        d.add(hs[c], W::load_own(a.V + (int64_t)c * a.ldv, (int64_t)k * nc + gidx));
                    xo[k] = d.value();
                    W::store(a.x, (int64_t)k * nc + gidx, xo[k]);
                }
            }
            if (!(ok = grid_sync())) break;
            stage(a.x, false, T(1));
            residual(xo, false);
            if (!(ok = grid_sync())) break;
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (blk == 0) {
            GmState* st = a.st;
            st->bnorm = bn;
            st->relres = relres;
            st->total = total;
            st->restarts = restarts;
            st->kdim = kdim;
            st->run = 0;
            st->inner = 0;
            st->status = status;
            st->zero = szero;
            st->dyn.live = 0;
        }
        // the last block out resets the barrier for the next launch
        __threadfence();
        if (atomicAdd(&a.st->bar_out, 1u) == (unsigned)nblk - 1u) {
            a.st->bar = 0u;
            a.st->bar_out = 0u;
        }
    }
}

template <typename T, bool DF, bool TR>
cudaError_t launch_solve(const SolveArgs<T>& a, int blocks, cudaStream_t st)
{
    const size_t smem = solve_smem<T>(a.Y);
    void* args[] = {const_cast<SolveArgs<T>*>(&a)};
    count_launches(1);
    return cudaLaunchCooperativeKernel((const void*)k_gm_solve<T, DF, TR>, dim3(blocks), dim3(solve_threads<T>(a.Y)), args,
                                       smem, st);
}

int solve_tiles(GridP g, int Y) { return ((g.nx + kSX - 1) / kSX) * ((g.ny + Y - 1) / Y); }

// blocks of one of the kernel's variants that can be resident at once
template <typename T, bool DF, bool TR>
cudaError_t solve_resident(int Y, int nsm, int* blocks)
{
    int per = 0;
    cudaError_t e = cudaFuncSetAttribute(k_gm_solve<T, DF, TR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)solve_smem<T>(sizeof(T) == 4 ? 8 : 4));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_gm_solve<T, DF, TR>, solve_threads<T>(Y),
                                                          solve_smem<T>(Y));
    const int b = per * nsm;
    if (e == cudaSuccess && b < *blocks) *blocks = b;
    return e;
}

}  // namespace

// The tile height of the one-launch solve: the smallest (most blocks in
// flight) that leaves at most one block per SM, else the form's largest if
// its blocks are all resident together, else 0 (the launches of gmres.cu).
template <typename T>
cudaError_t gm_solve_rows(GridP g, int* rows, double* share)
{
    *rows = 0;
    *share = 0.0;
    if (g.dim != 2 || g.shape != 1) return cudaSuccess;
    int dev = 0, nsm = 0, coop = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e != cudaSuccess || !coop) return e;
    constexpr int top = sizeof(T) == 4 ? 8 : 4;
    int Y = 1;
    while (Y < top && solve_tiles(g, Y) > nsm) Y *= 2;
    int most = 1 << 30;
    if constexpr (sizeof(T) == 4) {
        if (g.df) {
            e = solve_resident<T, true, false>(Y, nsm, &most);
            if (e == cudaSuccess) e = solve_resident<T, true, true>(Y, nsm, &most);
        }
    }
    if (e == cudaSuccess && !g.df) {
        e = solve_resident<T, false, false>(Y, nsm, &most);
        if (e == cudaSuccess) e = solve_resident<T, false, true>(Y, nsm, &most);
    }
    if (e == cudaSuccess && solve_tiles(g, Y) <= most) {
        *rows = Y;
        *share = (double)solve_tiles(g, Y) / (double)most;
    }
    return e;
}

int64_t gm_solve_partials(GridP g, int rows, int m) { return (int64_t)solve_tiles(g, rows) * (m + 4); }

template <typename T>
cudaError_t gm_solve(const T* M, const double* b, double* x, const GmPtrs& p, const GmParams& q, GridP g, int rows,
                     double* partial, GmState* st, int* err, bool tr, cudaStream_t s)
{
    SolveArgs<T> a;
    a.M = M;
    a.b = b;
    a.x = x;
    a.r = p.r;
    a.V = p.V;
    a.ldv = p.ldv;
    a.g = g;
    a.Y = rows;
    a.tma = ((int64_t)g.nx * kMBlock * sizeof(T)) % 16 == 0 ? 1 : 0;
    a.m = q.m;
    a.maxit = q.maxit;
    a.tol = q.tol;
    a.partial = partial;
    a.st = st;
    a.err = err;
    const int blocks = solve_tiles(g, rows);
    if constexpr (sizeof(T) == 4)
        if (g.df) return tr ? launch_solve<T, true, true>(a, blocks, s) : launch_solve<T, true, false>(a, blocks, s);
    return tr ? launch_solve<T, false, true>(a, blocks, s) : launch_solve<T, false, false>(a, blocks, s);
}

template cudaError_t gm_solve_rows<float>(GridP, int*, double*);
template cudaError_t gm_solve_rows<double>(GridP, int*, double*);
template cudaError_t gm_solve<float>(const float*, const double*, double*, const GmPtrs&, const GmParams&, GridP, int,
                                     double*, GmState*, int*, bool, cudaStream_t);
template cudaError_t gm_solve<double>(const double*, const double*, double*, const GmPtrs&, const GmParams&, GridP, int,
                                      double*, GmState*, int*, bool, cudaStream_t);

}  // namespace relsim
