// opcore.cuh -- device pieces shared by the kernels that apply the 2D implicit
// operator (linear shapes): loads and stores of GMRES vectors, the operator's
// stencil at a node, and compensated dot products.
#pragma once

#include "dfloat.cuh"
#include "launch.cuh"

namespace relsim {

constexpr long long kOpMaxPolls = 1ll << 26;   // bounded mbarrier wait
constexpr int kOpChunk = 8;                    // dot products reduced per shared-memory pass

// store v (formed in T) in a GMRES vector slot
template <bool DF, typename T>
__device__ __forceinline__ void vst(double* v, int64_t k, T val)
{
    if constexpr (DF) reinterpret_cast<dfl*>(v)[k] = df_from_f((float)val);
    else v[k] = (double)val;
}

// Node-local loads of a GMRES vector as T
template <typename T, bool DF = false>
__device__ __forceinline__ T vld(const double* v, int64_t k)
{
    if constexpr (DF) {
        const float2 a = __ldg(reinterpret_cast<const float2*>(v) + k);
        return (T)df_to_f(dfl{a.x, a.y});
    } else {
        return (T)__ldg(v + k);
    }
}
__device__ __forceinline__ dfl dld(const double* v, int64_t k)
{
    const float2 a = __ldg(reinterpret_cast<const float2*>(v) + k);
    return dfl{a.x, a.y};
}

// curl_c at a centre from its four nodes f(k, a, b), a, b = 0, 1 along x, y
template <typename T, class F>
__device__ __forceinline__ void op_curl_c(F f, T idx2, T idy2, T (&C)[3])
{
    T dx[3], dy[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        dx[k] = (f(k, 1, 0) - f(k, 0, 0) + f(k, 1, 1) - f(k, 0, 1)) * idx2;
        dy[k] = (f(k, 0, 1) - f(k, 0, 0) + f(k, 1, 1) - f(k, 1, 0)) * idy2;
    }
    C[0] = dy[2];
    C[1] = -dx[2];
    C[2] = dx[1] - dy[0];
}

// curl_n at a node from its four centres C(k, a, b)
template <typename T, class F>
__device__ __forceinline__ void op_curl_n(F C, T idx2, T idy2, T (&cc)[3])
{
    T dx[3], dy[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        dx[k] = (C(k, 1, 1) - C(k, 0, 1) + C(k, 1, 0) - C(k, 0, 0)) * idx2;
        dy[k] = (C(k, 1, 1) - C(k, 1, 0) + C(k, 0, 1) - C(k, 0, 0)) * idy2;
    }
    cc[0] = dy[2];
    cc[1] = -dx[2];
    cc[2] = dx[1] - dy[0];
}

// M v at a node from its 3x3 stencil of v, f[k][a][b] = component k at node
// (i-1+a, j-1+b), and its mass-matrix blocks: Mg = the node's own five blocks
// M[g][0..4], Mn[o] = the block M[g-o][o+1] of the neighbour g - o for the
// half offsets o = (1,0), (-1,1), (0,1), (1,1) (M_{g,g-o} = M_{g-o,g}). With
// TR every 3x3 block is applied transposed (M^T v: the stored block of the
// pair (g, g') serves both orders, M_{g'g} = M_{gg'}).
template <typename T, typename P, bool TR>
__device__ __forceinline__ void op_mass(const T (&f)[3][3][3], P Mg, const P (&Mn)[4], T (&mv)[3])
{
    constexpr int pa[4] = {2, 0, 1, 2}, pb[4] = {1, 2, 2, 2};   // g + o in the stencil
    constexpr int ma[4] = {0, 2, 1, 0}, mb[4] = {1, 0, 0, 0};   // g - o
    T r[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int rr = 0; rr < 3; ++rr)
#pragma unroll
        for (int s = 0; s < 3; ++s) r[rr] += T(Mg[TR ? s * 3 + rr : rr * 3 + s]) * f[s][1][1];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        P Mo = Mg + (o + 1) * 9;
#pragma unroll
        for (int rr = 0; rr < 3; ++rr)
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                // (two statements: two fused multiply-adds instead of three operations)
                r[rr] += T(Mo[TR ? s * 3 + rr : rr * 3 + s]) * f[s][pa[o]][pb[o]];
                r[rr] += T(Mn[o][TR ? s * 3 + rr : rr * 3 + s]) * f[s][ma[o]][mb[o]];
            }
    }
    mv[0] = r[0];
    mv[1] = r[1];
    mv[2] = r[2];
}

// one component (rr, the same across the warp) of the same
template <typename T, typename P, bool TR>
__device__ __forceinline__ T op_mass_row(const T (&f)[3][3][3], P Mg, const P (&Mn)[4], int rr)
{
    constexpr int pa[4] = {2, 0, 1, 2}, pb[4] = {1, 2, 2, 2};
    constexpr int ma[4] = {0, 2, 1, 0}, mb[4] = {1, 0, 0, 0};
    const int at = TR ? rr : rr * 3;
    constexpr int step = TR ? 3 : 1;
    T r = T(0);
#pragma unroll
    for (int s = 0; s < 3; ++s) r += T(Mg[at + step * s]) * f[s][1][1];
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            r += T(Mg[(o + 1) * 9 + at + step * s]) * f[s][pa[o]][pb[o]];
            r += T(Mn[o][at + step * s]) * f[s][ma[o]][mb[o]];
        }
    return r;
}

// (curl_n curl_c v) and (M v) at a node from its 3x3 stencil of v
template <typename T, typename P, bool TR>
__device__ __forceinline__ void op_stencil_t(const T (&f)[3][3][3], P Mg, const P (&Mn)[4], T idx2, T idy2,
                                             T (&cc)[3], T (&mv)[3])
{
    T C[2][2][3];
#pragma unroll
    for (int ca = 0; ca < 2; ++ca)
#pragma unroll
        for (int cb = 0; cb < 2; ++cb)
            op_curl_c<T>([&](int k, int p, int q) { return f[k][ca + p][cb + q]; }, idx2, idy2, C[ca][cb]);
    op_curl_n<T>([&](int k, int ca, int cb) { return C[ca][cb][k]; }, idx2, idy2, cc);
    op_mass<T, P, TR>(f, Mg, Mn, mv);
}

template <typename T, typename P>
__device__ __forceinline__ void op_stencil(const T (&f)[3][3][3], P Mg, const P (&Mn)[4], T idx2, T idy2,
                                           T (&cc)[3], T (&mv)[3])
{
    op_stencil_t<T, P, false>(f, Mg, Mn, idx2, idy2, cc, mv);
}

// Dot2 (Ogita, Rump and Oishi, "Accurate sum and dot product", SIAM J. Sci.
// Comput. 26, 2005) on the FP32 pipe: a running sum s with its error e,
// each term's product split exactly by TwoProduct and added by TwoSum.
struct Dot2 {
    float s = 0.0f, e = 0.0f;
    // += a b, a double-float, b FP32
    __device__ __forceinline__ void add(dfl a, float b)
    {
        const dfl p = df_two_prod(a.hi, b);
        const dfl t = df_two_sum(s, p.hi);
        s = t.hi;
        e = __fadd_rn(e, __fadd_rn(t.lo, __fmaf_rn(a.lo, b, p.lo)));
    }
    // += a b, both double-float
    __device__ __forceinline__ void add(dfl a, dfl b)
    {
        const dfl p = df_two_prod(a.hi, b.hi);
        const float pe = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
        const dfl t = df_two_sum(s, p.hi);
        s = t.hi;
        e = __fadd_rn(e, __fadd_rn(t.lo, pe));
    }
    // -= a b, both double-float
    __device__ __forceinline__ void sub(dfl a, dfl b)
    {
        const dfl p = df_two_prod(a.hi, b.hi);
        const float pe = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
        const dfl t = df_two_sum(s, -p.hi);
        s = t.hi;
        e = __fadd_rn(e, __fsub_rn(t.lo, pe));
    }
    __device__ __forceinline__ dfl value() const { return df_fast_two_sum(s, e); }
};

}  // namespace relsim
