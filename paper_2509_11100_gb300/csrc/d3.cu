// d3.cu -- the 3D form of the step: periodic nx x ny x nz grid, trilinear
// (CIC) shape functions, so a particle touches the 8 nodes of its cell and
// its mass-matrix contributions couple node pairs up to one cell apart in
// each direction (the 27-node stencil), of which 14 offsets are stored (the
// stored block of a pair serves both orders). The scheme is that of the 2D
// kernels (Sec. 2: explicit pusher, implicit field solve through the mass
// matrices); node and cell (i,j,k) have linear index (k ny + j) nx + i,
// centres sit at (i+1/2, j+1/2, k+1/2), and a particle is stored as its cell
// (implicit in the cell-sorted order) plus FP32 offsets fx, fy, fz.
//
// Kernels:
//   k_load3, k_gather3, k_export3   load, re-sort gather, read-back
//   k_deposit3   warp per row segment of cells; for each cell the lanes stage
//                their particles' weights, c alpha and c alpha u / gbar in
//                shared memory, then each lane accumulates the node pairs it
//                owns over the cell's particles in registers and flushes them
//                once per cell (FP32 or FP64 atomics)
//   k_op3        the operator A = I + (theta dt)^2 curl_n curl_c + theta dt M,
//                one thread per node, in the three modes of the 2D operator
//   k_rhs3, k_field_update3   the right-hand side, the field update with the
//                field ledger terms
//   k_push3      warp per row segment, the push with the cell change of the
//                general path (any move length), followed by the radix sort
#include "launch.cuh"

namespace relsim {
namespace {

unsigned grid3(int64_t n, int threads, int64_t cap)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > cap) b = cap;
    return (unsigned)(b > 0 ? b : 1);
}

__host__ __device__ __forceinline__ int64_t node3(int i, int j, int k, const GridP& g)
{
    return ((int64_t)k * g.ny + j) * g.nx + i;
}

// the half-stored offset index of d = (di, dj, dk), or -1 when -d is the
// stored one
__host__ __device__ __forceinline__ int half3(int di, int dj, int dk)
{
    if (dk == 1) return 5 + (dj + 1) * 3 + (di + 1);
    if (dk == 0 && dj == 1) return 2 + (di + 1);
    if (dk == 0 && dj == 0 && di >= 0) return di;
    return -1;
}

// ---------------------------------------------------------------------------
// load, gather, export

template <typename T>
__global__ void k_load3(const double* __restrict__ x, const double* __restrict__ u, const double* __restrict__ w,
                        int64_t n, GridP g, PArrays<T> out, T* __restrict__ ofz, int32_t* __restrict__ key,
                        int32_t* __restrict__ val, int* bad)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        double s[3] = {x[3 * p] / g.dx, x[3 * p + 1] / g.dy, x[3 * p + 2] / g.dz};
        const double ux = u[3 * p], uy = u[3 * p + 1], uz = u[3 * p + 2], ww = w[p];
        if (!isfinite(s[0]) || !isfinite(s[1]) || !isfinite(s[2]) || !isfinite(ux) || !isfinite(uy) ||
            !isfinite(uz) || !isfinite(ww)) {
            atomicOr(bad, 1);
            s[0] = s[1] = s[2] = 0.0;
        }
        const int nn[3] = {g.nx, g.ny, g.nz};
        int c[3];
        T f[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (s[a] < 0.0 || s[a] >= (double)nn[a]) s[a] -= nn[a] * floor(s[a] / nn[a]);
            const double fl = floor(s[a]);
            int ci = (int)fl;
            if (ci >= nn[a]) ci -= nn[a];
            if (ci < 0) ci = 0;
            c[a] = ci;
            f[a] = from_double_rz<T>(s[a] - fl);
        }
        out.fx[p] = f[0];
        out.fy[p] = f[1];
        ofz[p] = f[2];
        out.ux[p] = (T)ux;
        out.uy[p] = (T)uy;
        out.uz[p] = (T)uz;
        out.w[p] = (T)ww;
        key[p] = (int32_t)node3(c[0], c[1], c[2], g);
        val[p] = (int32_t)p;
    }
}

template <typename T>
__global__ void k_gather3(const int32_t* __restrict__ perm, PArrays<T> src, const T* __restrict__ sfz, PArrays<T> dst,
                          T* __restrict__ dfz, int64_t n, bool ids_from_perm)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t s = perm[p];
        dst.fx[p] = src.fx[s];
        dst.fy[p] = src.fy[s];
        dfz[p] = sfz[s];
        dst.ux[p] = src.ux[s];
        dst.uy[p] = src.uy[s];
        dst.uz[p] = src.uz[s];
        dst.w[p] = src.w[s];
        if (dst.id) dst.id[p] = ids_from_perm ? s : src.id[s];
    }
}

// one warp per cell: absolute positions back to FP64 (x, y, z interleaved)
template <typename T>
__global__ void k_export3(PArrays<T> pa, const T* __restrict__ fz, const int32_t* __restrict__ start, GridP g,
                          double* x, double* u, double* w, int32_t* id)
{
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int c = warp; c < g.ncell; c += nwarps) {
        const int i = c % g.nx, j = (c / g.nx) % g.ny, k = c / (g.nx * g.ny);
        const int p1 = start[c + 1];
        for (int p = start[c] + lane; p < p1; p += 32) {
            if (x) {
                x[3 * (int64_t)p] = ((double)i + (double)pa.fx[p]) * g.dx;
                x[3 * (int64_t)p + 1] = ((double)j + (double)pa.fy[p]) * g.dy;
                x[3 * (int64_t)p + 2] = ((double)k + (double)fz[p]) * g.dz;
            }
            if (u) {
                u[3 * (int64_t)p] = (double)pa.ux[p];
                u[3 * (int64_t)p + 1] = (double)pa.uy[p];
                u[3 * (int64_t)p + 2] = (double)pa.uz[p];
            }
            if (w) w[p] = (double)pa.w[p];
            if (id && pa.id) id[p] = pa.id[p];
        }
    }
}

// ---------------------------------------------------------------------------
// per-particle arithmetic shared by the deposit and the push

// trilinear weights of the 8 corners a = (a&1, (a>>1)&1, (a>>2)&1)
template <typename T>
__device__ __forceinline__ void corner_weights(T fx, T fy, T fz, T (&W)[8])
{
    const T X[2] = {T(1) - fx, fx}, Y[2] = {T(1) - fy, fy}, Z[2] = {T(1) - fz, fz};
#pragma unroll
    for (int a = 0; a < 8; ++a) W[a] = X[a & 1] * Y[(a >> 1) & 1] * Z[(a >> 2) & 1];
}

// alpha = (I - [a]x + a a^T)/(1 + |a|^2), a = bg B, bg = beta/gbar (row-major)
template <typename T>
__device__ __forceinline__ void alpha3(const T (&Bp)[3], T bg, T (&al)[9])
{
    const T ax = bg * Bp[0], ay = bg * Bp[1], az = bg * Bp[2];
    const T ia = T(1) / (T(1) + ax * ax + ay * ay + az * az);
    al[0] = (T(1) + ax * ax) * ia; al[1] = (ax * ay + az) * ia; al[2] = (ax * az - ay) * ia;
    al[3] = (ax * ay - az) * ia; al[4] = (T(1) + ay * ay) * ia; al[5] = (ay * az + ax) * ia;
    al[6] = (ax * az + ay) * ia; al[7] = (ay * az - ax) * ia; al[8] = (T(1) + az * az) * ia;
}

// ---------------------------------------------------------------------------
// field tiles of a row segment (cells i0 .. i0+cn-1 of row (j, k)), staged in
// shared memory once per segment instead of 24 gathers per particle per field

template <typename T>
struct Tile3B {
    T B[3][3][3][34];   // [comp][dy][dz][c]: centre (i0 - 1 + c, j - 1 + dy, k - 1 + dz)
};
template <typename T>
__device__ __forceinline__ void load_tile3B(Tile3B<T>& tl, const T* __restrict__ B, int i0, int cn, int j, int k,
                                            const GridP& g, int lane)
{
    const int64_t nc = g.ncell;
    for (int q = lane; q < 3 * 3 * 3 * 34; q += 32) {
        const int c = q % 34, dz = (q / 34) % 3, dy = (q / 102) % 3, comp = q / 306;
        if (c <= cn + 1)
            tl.B[comp][dy][dz][c] =
                ld(B + comp * nc + node3(wrap1(i0 - 1 + c, g.nx), wrap1(j - 1 + dy, g.ny), wrap1(k - 1 + dz, g.nz), g));
    }
    __syncwarp();
}

// B^n at a particle of local cell cl with offsets f, from the tile
template <typename T>
__device__ __forceinline__ void tile_B3(const T (&B)[3][3][3][34], int cl, T fx, T fy, T fz, T (&Bp)[3])
{
    const bool lx = fx < T(0.5), ly = fy < T(0.5), lz = fz < T(0.5);
    const T tx = lx ? fx + T(0.5) : fx - T(0.5);
    const T ty = ly ? fy + T(0.5) : fy - T(0.5);
    const T tz = lz ? fz + T(0.5) : fz - T(0.5);
    const int c0 = lx ? cl : cl + 1, y0 = ly ? 0 : 1, z0 = lz ? 0 : 1;
    T W[8];
    corner_weights(tx, ty, tz, W);
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
        T b = T(0);
#pragma unroll
        for (int a = 0; a < 8; ++a) b += W[a] * B[comp][y0 + ((a >> 1) & 1)][z0 + ((a >> 2) & 1)][c0 + (a & 1)];
        Bp[comp] = b;
    }
}

// The push's tiles hold every value with its right neighbour, so that the two
// columns of a gather come in one load: 24 shared loads a particle instead
// of 48
template <typename T>
struct Pair3 {
    T a, b;
};
template <>
struct __align__(8) Pair3<float> {
    float a, b;
};
template <>
struct __align__(16) Pair3<double> {
    double a, b;
};
template <typename T>
struct PairTile3 {
    Pair3<T> E[3][2][2][32];   // [comp][dy][dz][c]: nodes (i0 + c, j + dy, k + dz) and (i0 + c + 1, ..)
    Pair3<T> B[3][3][3][33];   // [comp][dy][dz][c]: centres (i0 - 1 + c, j - 1 + dy, k - 1 + dz) and (i0 + c, ..)
    __device__ __forceinline__ void gather_E(int cl, T fx, T fy, T fz, T (&E3)[3]) const
    {
        T W[8];
        corner_weights(fx, fy, fz, W);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            T e = T(0);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const Pair3<T> q = E[c][a & 1][a >> 1][cl];
                e += W[2 * a] * q.a;
                e += W[2 * a + 1] * q.b;
            }
            E3[c] = e;
        }
    }
    __device__ __forceinline__ void gather_B(int cl, T fx, T fy, T fz, T (&Bp)[3]) const
    {
        const bool lx = fx < T(0.5), ly = fy < T(0.5), lz = fz < T(0.5);
        const T tx = lx ? fx + T(0.5) : fx - T(0.5);
        const T ty = ly ? fy + T(0.5) : fy - T(0.5);
        const T tz = lz ? fz + T(0.5) : fz - T(0.5);
        const int c0 = lx ? cl : cl + 1, y0 = ly ? 0 : 1, z0 = lz ? 0 : 1;
        T W[8];
        corner_weights(tx, ty, tz, W);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            T e = T(0);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const Pair3<T> q = B[c][y0 + (a & 1)][z0 + (a >> 1)][c0];
                e += W[2 * a] * q.a;
                e += W[2 * a + 1] * q.b;
            }
            Bp[c] = e;
        }
    }
};

template <typename T>
__device__ __forceinline__ void load_pairs3(PairTile3<T>& tl, const T* __restrict__ E, const T* __restrict__ B, int i0,
                                            int cn, int j, int k, const GridP& g, int lane)
{
    const int64_t nc = g.ncell;
    // a lane a column, the rows in turn (a column's right neighbour is the
    // next lane's value but for the last)
    const int ca = wrap1(i0 + min(lane, cn - 1), g.nx), cb = wrap1(i0 + min(lane, cn - 1) + 1, g.nx);
    const int cz = wrap1(i0 - 1, g.nx);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t row = node3(0, wrap1(j + (r & 1), g.ny), wrap1(k + (r >> 1), g.nz), g);
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (lane < cn) tl.E[c][r & 1][r >> 1][lane] = Pair3<T>{ld(E + c * nc + row + ca), ld(E + c * nc + row + cb)};
    }
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const int64_t row = node3(0, wrap1(j - 1 + r % 3, g.ny), wrap1(k - 1 + r / 3, g.nz), g);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (lane < cn)
                tl.B[c][r % 3][r / 3][lane + 1] = Pair3<T>{ld(B + c * nc + row + ca), ld(B + c * nc + row + cb)};
            if (lane == 0) tl.B[c][r % 3][r / 3][0] = Pair3<T>{ld(B + c * nc + row + cz), ld(B + c * nc + row + ca)};
        }
    }
    __syncwarp();
}

// ---------------------------------------------------------------------------
// deposit

// A warp takes a row segment of cells and, batch after batch, 32 particles of
// it whatever cell and species they belong to: each lane forms one particle's
// weights, c alpha and current and stages them in shared memory (the lanes are
// full whatever the cells hold); then the warp runs over the staged particles,
// and lane k adds to the 9 sums of one of the cell's 27 moments
//   S[xx][yy][zz][e] = sum_p XX YY ZZ c_p alpha_e,   XX in (X0^2, X0 X1, X1^2), ..
// (the 36 corner pairs take 27 distinct weight products), two particles per
// paired FP32 FMA. When a cell is done, its 36 blocks go to M from shared
// memory in address order, so that a warp's additions fall in few sectors, and
// the moments of the cell's upper x face start the next cell's lower face
// instead of being added to memory twice.
//
// Bound by issue. Before, each lane owned one or two of the 36 pairs, a cell's
// own batches were often half empty, and each lane added its blocks by itself:
// 61 warp instructions a particle, 11.5 ms on 256x128x128 with 32 particles a
// cell (FP32 form), 0.23 ms on 64x32x32.
template <typename T>
struct DepCfg3 {
    static constexpr int warps = sizeof(T) == 4 ? 4 : 2;   // static shared memory < 48 KB
};
constexpr int kMom3 = 27;
constexpr int kItems3 = 36 * 9;        // a cell's additions to M
constexpr int kFace3 = 26 * 9;         // those not on the upper x face
// staged values of a particle: c alpha, XX YY, ZZ, corner weights, current
enum { kS3E = 0, kS3XY = 9, kS3Z = 18, kS3W = 21, kS3V = 29, kS3N = 32 };

// the staged particles of a warp: FP32 two by two, (value of particle 2r,
// value of particle 2r + 1), rows 16-byte aligned
template <typename T>
struct Stage3 {
    T v[32][kS3N + 1];
    __device__ __forceinline__ void put(int t, int k, T a) { v[t][k] = a; }
};
template <>
struct Stage3<float> {
    static constexpr int row = 2 * kS3N + 4;
    float v[16][row];
    __device__ __forceinline__ void put(int t, int k, float a) { v[t >> 1][2 * k + (t & 1)] = a; }
    __device__ __forceinline__ float2 get2(int r, int k) const { return *reinterpret_cast<const float2*>(&v[r][2 * k]); }
};

// a lane's sums of one moment and one current value over a cell
template <typename T>
struct Acc3 {
    T m[9], j;
    __device__ __forceinline__ void start(const T (&v)[9], T vj)
    {
#pragma unroll
        for (int e = 0; e < 9; ++e) m[e] = v[e];
        j = vj;
    }
    __device__ __forceinline__ void add(const Stage3<T>& st, int t0, int t1, int k1, int k2, int ja, int jc)
    {
        for (int t = t0; t < t1; ++t) {
            const T w = st.v[t][kS3XY + k1] * st.v[t][kS3Z + k2];
#pragma unroll
            for (int e = 0; e < 9; ++e) m[e] += w * st.v[t][kS3E + e];
            j += st.v[t][kS3W + ja] * st.v[t][kS3V + jc];
        }
    }
    __device__ __forceinline__ void get(T (&v)[9], T& vj) const
    {
#pragma unroll
        for (int e = 0; e < 9; ++e) v[e] = m[e];
        vj = j;
    }
};
template <>
struct Acc3<float> {
    float2 m[9], j;   // even and odd staged particles apart
    __device__ __forceinline__ void start(const float (&v)[9], float vj)
    {
#pragma unroll
        for (int e = 0; e < 9; ++e) m[e] = make_float2(v[e], 0.f);
        j = make_float2(vj, 0.f);
    }
    // EDGE: the row holds a particle of another cell (its weights are left out)
    template <bool EDGE>
    __device__ __forceinline__ void row(const Stage3<float>& st, int r, int t0, int t1, int k1, int k2, int ja, int jc)
    {
        const float2 xy = st.get2(r, kS3XY + k1), z = st.get2(r, kS3Z + k2);
        float2 w = make_float2(xy.x * z.x, xy.y * z.y), wj = st.get2(r, kS3W + ja);
        if (EDGE) {
            if (2 * r < t0) w.x = wj.x = 0.f;
            if (2 * r + 1 >= t1) w.y = wj.y = 0.f;
        }
        const float4* e4 = reinterpret_cast<const float4*>(&st.v[r][0]);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float4 q = e4[h];
            m[2 * h] = __ffma2_rn(w, make_float2(q.x, q.y), m[2 * h]);
            m[2 * h + 1] = __ffma2_rn(w, make_float2(q.z, q.w), m[2 * h + 1]);
        }
        m[8] = __ffma2_rn(w, st.get2(r, kS3E + 8), m[8]);
        j = __ffma2_rn(wj, st.get2(r, kS3V + jc), j);
    }
    __device__ __forceinline__ void add(const Stage3<float>& st, int t0, int t1, int k1, int k2, int ja, int jc)
    {
        int r = t0 >> 1;
        const int r1 = t1 >> 1;   // rows r0 .. r1-1 are whole but for the first
        if (t0 & 1) {
            row<true>(st, r, t0, t1, k1, k2, ja, jc);
            ++r;
        }
#pragma unroll 2
        for (; r < r1; ++r) row<false>(st, r, t0, t1, k1, k2, ja, jc);
        if ((t1 & 1) && r == r1) row<true>(st, r, t0, t1, k1, k2, ja, jc);
    }
    __device__ __forceinline__ void get(float (&v)[9], float& vj) const
    {
#pragma unroll
        for (int e = 0; e < 9; ++e) v[e] = m[e].x + m[e].y;
        vj = j.x + j.y;
    }
};

// the 36 unordered corner pairs (a <= b) of a cell, pair q
__device__ __forceinline__ void pair_of(int q, int& a, int& b)
{
    int r = q;
    a = 0;
    while (r >= 8 - a) {
        r -= 8 - a;
        ++a;
    }
    b = a + r;
}
// where pair q's block is stored (corner at, offset index hs: at corner a
// with the offset b - a when that is in the stored half, else at b with
// a - b), its moment, and its place in the order (upper x face last, then by
// corner and offset)
__device__ __forceinline__ void pair_block(int q, int& at, int& hs, int& mom, int& place)
{
    int a, b;
    pair_of(q, a, b);
    const int di = (b & 1) - (a & 1), dj = ((b >> 1) & 1) - ((a >> 1) & 1), dk = ((b >> 2) & 1) - ((a >> 2) & 1);
    hs = half3(di, dj, dk);
    at = a;
    if (hs < 0) {
        hs = half3(-di, -dj, -dk);
        at = b;
    }
    mom = ((a >> 2 & 1) + (b >> 2 & 1)) * 9 + ((a & 1) + (b & 1)) * 3 + (a >> 1 & 1) + (b >> 1 & 1);
    place = ((a & b & 1) * 8 + at) * kHalf3 + hs;
}

template <typename T>
__global__ void __launch_bounds__(32 * DepCfg3<T>::warps)
k_deposit3(const __grid_constant__ DepositSpecies<T> ds, const __grid_constant__ FzArrays<T> fz,
           const T* __restrict__ B, T* __restrict__ M, T* __restrict__ J,
           GridP g, int uw)
{
    constexpr int kW = DepCfg3<T>::warps;
    __shared__ __align__(16) Stage3<T> sst[kW];
    __shared__ Tile3B<T> stl[kW];
    __shared__ T smom[kW][kMom3 * 9];   // a cell's moments, for the additions
    __shared__ int64_t snode[kW][8];    // its corners' nodes
    __shared__ unsigned item[kItems3];  // an addition: corner << 16 | place in the node's blocks << 8 | moment value
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < 36; q += blockDim.x) {
        int at, hs, mom, place, rank = 0;
        pair_block(q, at, hs, mom, place);
        for (int o = 0; o < 36; ++o) {
            int at2, hs2, mom2, place2;
            pair_block(o, at2, hs2, mom2, place2);
            rank += place2 < place ? 1 : 0;
        }
        for (int e = 0; e < 9; ++e)
            item[rank * 9 + e] = (unsigned)at << 16 | (unsigned)(hs * 9 + e) << 8 | (unsigned)(mom * 9 + e);
    }
    __syncthreads();
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int nseg = (g.nx + uw - 1) / uw;
    const int64_t nunits = (int64_t)nseg * g.ny * g.nz;
    const int nsp = ds.nsp, gcells = 32 / nsp;   // cells whose (cell, species) ranges fit the lanes
    Stage3<T>& st = sst[wib];
    // the moment this lane sums (lanes 0 .. 26: ZZ, XX, YY) and the current
    // value (lanes 0 .. 23: corner, component)
    const int k1 = lane < kMom3 ? lane % 9 : 0, k2 = lane < kMom3 ? lane / 9 : 0;
    const int ja = lane < 24 ? lane / 3 : 0, jc = lane < 24 ? lane % 3 : 0;
    const bool low = lane < kMom3 && k1 < 3;   // a moment of the lower x face
    for (int64_t u = warp; u < nunits; u += nwarps) {
        const int i0 = (int)(u % nseg) * uw;
        const int jk = (int)(u / nseg);
        const int j = jk % g.ny, k = jk / g.ny;
        const int cn = min(uw, g.nx - i0);
        __syncwarp();
        load_tile3B<T>(stl[wib], B, i0, cn, j, k, g, lane);
        Acc3<T> acc;
        {
            const T zero[9] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
            acc.start(zero, T(0));
        }
        bool carry = false;   // the previous cell left sums on this cell's lower face
        for (int cg = 0; cg < cn; cg += gcells) {
            // the particles of up to gcells cells as one list: lane l holds
            // the range of cell l / nsp, species l % nsp
            const int gc0 = min(gcells, cn - cg);
            int first = 0, cnt = 0;
            if (lane < gc0 * nsp) {
                const int64_t c = node3(i0 + cg + lane / nsp, j, k, g);
                const int32_t* sp = ds.start[lane % nsp];
                first = sp[c];
                cnt = sp[c + 1] - first;
            }
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += up;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            const int base = first - (incl - cnt);   // particle = base + list index
            int cl = 0;                              // the cell the warp is adding up
            int cend = __shfl_sync(0xffffffffu, incl, nsp - 1);
            for (int w0 = 0; cl < gc0; w0 += 32) {   // (every pass ends cells or takes 32 particles)
                const int t = w0 + lane;
                // the range the lane's particle lies in (all lanes search)
                int seg = 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    if (__shfl_sync(0xffffffffu, incl, seg + o - 1) <= t) seg += o;
                const int p = __shfl_sync(0xffffffffu, base, seg) + t;
                if (t < total) {
                    const int s = seg % nsp, pc = cg + seg / nsp;
                    const T fx = ld(ds.fx[s] + p), fy = ld(ds.fy[s] + p), fzz = ld(fz.fz[s] + p);
                    const T ux = ld(ds.ux[s] + p), uy = ld(ds.uy[s] + p), uz = ld(ds.uz[s] + p);
                    const T wt = ld(ds.w[s] + p);
                    T W[8], Bp[3], al[9];
                    corner_weights(fx, fy, fzz, W);
                    tile_B3(stl[wib].B, pc, fx, fy, fzz, Bp);
                    const T ig = T(1) / sqrt(T(1) + ux * ux + uy * uy + uz * uz);
                    alpha3(Bp, ds.beta[s] * ig, al);
                    const T cM = wt * ds.cM[s] * ig, cJ = wt * ds.cJ[s] * ig;
                    const T X[3] = {(T(1) - fx) * (T(1) - fx), (T(1) - fx) * fx, fx * fx};
                    const T Y[3] = {(T(1) - fy) * (T(1) - fy), (T(1) - fy) * fy, fy * fy};
#pragma unroll
                    for (int e = 0; e < 9; ++e) st.put(lane, kS3E + e, cM * al[e]);
#pragma unroll
                    for (int e = 0; e < 9; ++e) st.put(lane, kS3XY + e, X[e / 3] * Y[e % 3]);
                    st.put(lane, kS3Z, (T(1) - fzz) * (T(1) - fzz));
                    st.put(lane, kS3Z + 1, (T(1) - fzz) * fzz);
                    st.put(lane, kS3Z + 2, fzz * fzz);
#pragma unroll
                    for (int a = 0; a < 8; ++a) st.put(lane, kS3W + a, W[a]);
#pragma unroll
                    for (int r = 0; r < 3; ++r)
                        st.put(lane, kS3V + r, cJ * (al[3 * r] * ux + al[3 * r + 1] * uy + al[3 * r + 2] * uz));
                } else {
#pragma unroll
                    for (int q = 0; q < kS3N; ++q) st.put(lane, q, T(0));
                }
                __syncwarp();
                const int wend = min(w0 + 32, total);
                int pos = w0;
                while (cl < gc0) {
                    const int upto = min(cend, wend);
                    if (upto > pos) acc.add(st, pos - w0, upto - w0, k1, k2, ja, jc);
                    pos = max(pos, upto);
                    if (cend > wend) break;   // the cell goes on in the next batch
                    // the cell is done
                    const int before = cl == 0 ? 0 : __shfl_sync(0xffffffffu, incl, cl * nsp - 1);
                    const bool last = cg + cl == cn - 1;
                    T v[9], vj;
                    acc.get(v, vj);
                    if (carry || cend > before) {
                        if (lane < kMom3)
#pragma unroll
                            for (int e = 0; e < 9; ++e) smom[wib][lane * 9 + e] = v[e];
                        const int i = i0 + cg + cl;
                        const int64_t nd = node3(wrap1(i + (lane & 1), g.nx), wrap1(j + ((lane >> 1) & 1), g.ny),
                                                 wrap1(k + ((lane >> 2) & 1), g.nz), g);
                        if (lane < 8) snode[wib][lane] = nd;
                        __syncwarp();
                        const int nit = last ? kItems3 : kFace3;
                        for (int it = lane; it < nit; it += 32) {
                            const unsigned q = item[it];
                            atomicAdd(M + snode[wib][q >> 16] * kMBlock3 + ((q >> 8) & 255u), smom[wib][q & 255u]);
                        }
                        if (lane < 24 && (last || (ja & 1) == 0))
                            atomicAdd(J + (int64_t)jc * g.ncell + snode[wib][ja], vj);
                        __syncwarp();
                        carry = !last;
                    }
                    // the upper x face's sums start the next cell's lower face
                    T n9[9];
#pragma unroll
                    for (int e = 0; e < 9; ++e) {
                        const T up = __shfl_down_sync(0xffffffffu, v[e], 6);
                        n9[e] = low && !last ? up : T(0);
                    }
                    const T upj = __shfl_down_sync(0xffffffffu, vj, 3);
                    acc.start(n9, lane < 24 && (ja & 1) == 0 && !last ? upj : T(0));
                    ++cl;
                    if (cl < gc0) cend = __shfl_sync(0xffffffffu, incl, cl * nsp + nsp - 1);
                }
                __syncwarp();
            }
        }
    }
}

// ---------------------------------------------------------------------------
// the implicit operator, the right-hand side and the field update

enum { k3A = 0, k3Residual = 1, k3Arnoldi = 2 };
constexpr int kOpX3 = 32, kOpY3 = 4, kOpZ3 = 2;
constexpr int kOpT3 = kOpX3 * kOpY3 * kOpZ3;
constexpr int kOpChunk3 = 8;

// the offset of stored block h (0..13)
__device__ __forceinline__ void half_offset3(int h, int& di, int& dj, int& dk)
{
    if (h < 2) { di = h; dj = 0; dk = 0; }
    else if (h < 5) { di = h - 3; dj = 1; dk = 0; }
    else { di = (h - 5) % 3 - 1; dj = (h - 5) / 3 - 1; dk = 1; }
}

// (curl_n curl_c v) at a node from v on its 3x3x3 neighbourhood,
// f(comp, a, b, c) = component comp at node (i-1+a, j-1+b, k-1+c)
template <typename T, typename F>
__device__ __forceinline__ void curlcurl3(F f, T rdx4, T rdy4, T rdz4, T (&out)[3])
{
    // curl_c at the 8 cells around the node: cell (ci, cj, ck) spans local
    // nodes ci..ci+1, cj..cj+1, ck..ck+1 (ci = 0: the cell i-1)
    T C[3][2][2][2];
#pragma unroll
    for (int ci = 0; ci < 2; ++ci)
#pragma unroll
        for (int cj = 0; cj < 2; ++cj)
#pragma unroll
            for (int ck = 0; ck < 2; ++ck) {
                T d[3][3];   // d[axis][comp]
#pragma unroll
                for (int comp = 0; comp < 3; ++comp) {
                    T sx = T(0), sy = T(0), sz = T(0);
#pragma unroll
                    for (int e1 = 0; e1 < 2; ++e1)
#pragma unroll
                        for (int e2 = 0; e2 < 2; ++e2) {
                            sx += f(comp, ci + 1, cj + e1, ck + e2) - f(comp, ci, cj + e1, ck + e2);
                            sy += f(comp, ci + e1, cj + 1, ck + e2) - f(comp, ci + e1, cj, ck + e2);
                            sz += f(comp, ci + e1, cj + e2, ck + 1) - f(comp, ci + e1, cj + e2, ck);
                        }
                    d[0][comp] = sx * rdx4;
                    d[1][comp] = sy * rdy4;
                    d[2][comp] = sz * rdz4;
                }
                C[0][ci][cj][ck] = d[1][2] - d[2][1];
                C[1][ci][cj][ck] = d[2][0] - d[0][2];
                C[2][ci][cj][ck] = d[0][1] - d[1][0];
            }
    // curl_n at the node from the 8 cells
    T d[3][3];
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
        T sx = T(0), sy = T(0), sz = T(0);
#pragma unroll
        for (int e1 = 0; e1 < 2; ++e1)
#pragma unroll
            for (int e2 = 0; e2 < 2; ++e2) {
                sx += C[comp][1][e1][e2] - C[comp][0][e1][e2];
                sy += C[comp][e1][1][e2] - C[comp][e1][0][e2];
                sz += C[comp][e1][e2][1] - C[comp][e1][e2][0];
            }
        d[0][comp] = sx * rdx4;
        d[1][comp] = sy * rdy4;
        d[2][comp] = sz * rdz4;
    }
    out[0] = d[1][2] - d[2][1];
    out[1] = d[2][0] - d[0][2];
    out[2] = d[0][1] - d[1][0];
}

// (M v) at node (i, j, k): its own 14 stored blocks times v at g + d(h), and
// the 13 neighbours' blocks M[g - d(h)][h] times v at g - d(h); with TR each
// block applied transposed
template <typename T, bool TR, typename F>
__device__ __forceinline__ void mv3(const T* __restrict__ M, int i, int j, int k, const GridP& g, F f, T (&out)[3])
{
    T r[3] = {T(0), T(0), T(0)};
    const T* Mg = M + node3(i, j, k, g) * kMBlock3;
#pragma unroll
    for (int h = 0; h < kHalf3; ++h) {
        int di, dj, dk;
        half_offset3(h, di, dj, dk);
        const T* Mo = Mg + h * 9;
        T vv[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) vv[s] = f(s, 1 + di, 1 + dj, 1 + dk);
#pragma unroll
        for (int rr = 0; rr < 3; ++rr)
#pragma unroll
            for (int s = 0; s < 3; ++s) r[rr] += ld(Mo + (TR ? s * 3 + rr : rr * 3 + s)) * vv[s];
        if (h == 0) continue;
        const T* Mn = M + node3(wrap1(i - di, g.nx), wrap1(j - dj, g.ny), wrap1(k - dk, g.nz), g) * kMBlock3 + h * 9;
#pragma unroll
        for (int s = 0; s < 3; ++s) vv[s] = f(s, 1 - di, 1 - dj, 1 - dk);
#pragma unroll
        for (int rr = 0; rr < 3; ++rr)
#pragma unroll
            for (int s = 0; s < 3; ++s) r[rr] += ld(Mn + (TR ? s * 3 + rr : rr * 3 + s)) * vv[s];
    }
    out[0] = r[0];
    out[1] = r[1];
    out[2] = r[2];
}

// The operator on tiles of 32 x 4 x 2 nodes, the input staged in T on the
// tile's 1-node halo (one FP64 load and conversion per staged value); the
// modes and the per-block partial sums are those of the 2D operator:
//   A:        out = in + B in
//   Residual: out = b - (in + B in), partial |out|^2
//   Arnoldi:  v = s in (to vj when vj is not null), out = B v, partials
//             <out, V_q> (q < nv), <out, v>, <out, out>
template <typename T, int MODE, bool TR>
__global__ void __launch_bounds__(kOpT3)
k_op3(const T* __restrict__ M, const double* __restrict__ in, double s, const double* __restrict__ b,
      double* __restrict__ out, double* __restrict__ vj, const double* __restrict__ V, int64_t ldv, int nv, GridP g,
      double* __restrict__ partial, const GmDyn* __restrict__ dyn)
{
    if (MODE == k3Arnoldi && dyn) {
        if (!dyn->live) return;
        in = dyn->in;
        s = dyn->s;
        vj = dyn->vj;
        out = dyn->out;
        nv = dyn->nv;
    }
    constexpr int HX = kOpX3 + 2, HY = kOpY3 + 2, HZ = kOpZ3 + 2;
    __shared__ T sv[3][HZ][HY][HX];
    __shared__ double buf[kOpChunk3][kOpT3];
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const int64_t nc = g.ncell;
    const int tx_n = (nx + kOpX3 - 1) / kOpX3, ty_n = (ny + kOpY3 - 1) / kOpY3;
    const int bx = blockIdx.x % tx_n, by = (blockIdx.x / tx_n) % ty_n, bz = blockIdx.x / (tx_n * ty_n);
    const int i0 = bx * kOpX3, j0 = by * kOpY3, k0 = bz * kOpZ3;
    const int tid = threadIdx.x, tx = tid % kOpX3, ty = (tid / kOpX3) % kOpY3, tz = tid / (kOpX3 * kOpY3);
    const int i = i0 + tx, j = j0 + ty, k = k0 + tz;
    const bool active = i < nx && j < ny && k < nz;
    const int64_t gidx = active ? node3(i, j, k, g) : 0;
    const T sT = (T)s;
    for (int q = tid; q < 3 * HZ * HY * HX; q += kOpT3) {
        const int comp = q / (HZ * HY * HX), rem = q % (HZ * HY * HX);
        const int zz = rem / (HY * HX), yy = (rem / HX) % HY, xx = rem % HX;
        const int gi = wrap1(min(i0 - 1 + xx, 2 * nx - 1), nx), gj = wrap1(min(j0 - 1 + yy, 2 * ny - 1), ny);
        const int gk = wrap1(min(k0 - 1 + zz, 2 * nz - 1), nz);
        T val = (T)__ldg(in + comp * nc + node3(gi, gj, gk, g));
        if (MODE == k3Arnoldi) val *= sT;
        sv[comp][zz][yy][xx] = val;
    }
    __syncthreads();
    double own[3] = {0.0, 0.0, 0.0}, wv[3] = {0.0, 0.0, 0.0};
    if (active) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            own[c] = __ldg(in + c * nc + gidx);
            if (MODE == k3Arnoldi && !is_one(s)) own[c] *= s;
        }
        auto f = [&](int comp, int a, int bb, int cc) -> T { return sv[comp][tz + cc][ty + bb][tx + a]; };
        T cc3[3], mv[3];
        curlcurl3<T>(f, gc<T>(g).qdx, gc<T>(g).qdy, gc<T>(g).qdz, cc3);
        mv3<T, TR>(M, i, j, k, g, f, mv);
        const T td = gc<T>(g).td;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double bv = (double)(td * td * cc3[c] + td * mv[c]);
            if (MODE == k3A) wv[c] = own[c] + bv;
            else if (MODE == k3Residual) wv[c] = b[c * nc + gidx] - (own[c] + bv);
            else wv[c] = bv;
            out[c * nc + gidx] = wv[c];
            if (MODE == k3Arnoldi && vj) vj[c * nc + gidx] = own[c];
        }
    }
    if (MODE == k3A) return;
    const int nq = MODE == k3Residual ? 1 : nv + 2;
    const int lane = tid & 31, wid = tid >> 5;
    for (int q0 = 0; q0 < nq; q0 += kOpChunk3) {
        const int kc = min(kOpChunk3, nq - q0);
        for (int c = 0; c < kc; ++c) {
            const int q = q0 + c;
            double d = 0.0;
            if (active) {
                if (MODE == k3Residual || q == nv + 1) d = wv[0] * wv[0] + wv[1] * wv[1] + wv[2] * wv[2];
                else if (q == nv) d = wv[0] * own[0] + wv[1] * own[1] + wv[2] * own[2];
                else {
                    const double* Vq = V + (int64_t)q * ldv + gidx;
                    d = wv[0] * __ldg(Vq) + wv[1] * __ldg(Vq + nc) + wv[2] * __ldg(Vq + 2 * nc);
                }
            }
            buf[c][tid] = d;
        }
        __syncthreads();
        for (int c = wid; c < kc; c += kOpT3 / 32) {
            double t = 0.0;
#pragma unroll
            for (int m = 0; m < kOpT3 / 32; ++m) t += buf[c][m * 32 + lane];
            t = warp_sum(t);
            if (lane == 0) partial[(int64_t)blockIdx.x * nq + q0 + c] = t;
        }
        __syncthreads();
    }
}

// b = E^n + theta dt curl_n B^n - theta dt Jhat
template <typename T>
__global__ void k_rhs3(const T* __restrict__ E, const T* __restrict__ B, const T* __restrict__ J,
                       double* __restrict__ b, GridP g)
{
    const int64_t nc = g.ncell;
    for (int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gi < nc; gi += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(gi % g.nx), j = (int)((gi / g.nx) % g.ny), k = (int)(gi / ((int64_t)g.nx * g.ny));
        const int ii[2] = {wrap1(i - 1, g.nx), i}, jj[2] = {wrap1(j - 1, g.ny), j}, kk[2] = {wrap1(k - 1, g.nz), k};
        T d[3][3];
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            const T* f = B + comp * nc;
            T sx = T(0), sy = T(0), sz = T(0);
#pragma unroll
            for (int e1 = 0; e1 < 2; ++e1)
#pragma unroll
                for (int e2 = 0; e2 < 2; ++e2) {
                    sx += f[node3(ii[1], jj[e1], kk[e2], g)] - f[node3(ii[0], jj[e1], kk[e2], g)];
                    sy += f[node3(ii[e1], jj[1], kk[e2], g)] - f[node3(ii[e1], jj[0], kk[e2], g)];
                    sz += f[node3(ii[e1], jj[e2], kk[1], g)] - f[node3(ii[e1], jj[e2], kk[0], g)];
                }
            d[0][comp] = sx * gc<T>(g).qdx;
            d[1][comp] = sy * gc<T>(g).qdy;
            d[2][comp] = sz * gc<T>(g).qdz;
        }
        const T cn[3] = {d[1][2] - d[2][1], d[2][0] - d[0][2], d[0][1] - d[1][0]};
        const T td = gc<T>(g).td;
#pragma unroll
        for (int comp = 0; comp < 3; ++comp)
            b[comp * nc + gi] = (double)(E[comp * nc + gi] + td * cn[comp] - td * J[comp * nc + gi]);
    }
}

constexpr int kFieldLedger3 = 6;

// E^{n+theta} (FP64 solution) -> Eth, E^{n+1}, B^{n+1} of cell (i,j,k) and the
// field ledger terms 0..4 (as the 2D field update); term 5 (the work) by
// k_work3 from Eth in T
template <typename T>
__global__ void __launch_bounds__(256)
k_field_update3(const double* __restrict__ x, T* __restrict__ Eth, T* __restrict__ E, const T* __restrict__ B0,
                T* __restrict__ B1, GridP g, double* __restrict__ partial)
{
    __shared__ double red[32 * 5];
    const int64_t nc = g.ncell;
    const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    T acc[5] = {T(0), T(0), T(0), T(0), T(0)};
    if (gidx < nc) {
        const int i = (int)(gidx % g.nx), j = (int)((gidx / g.nx) % g.ny), k = (int)(gidx / ((int64_t)g.nx * g.ny));
        const T th = gc<T>(g).theta, hdV = gc<T>(g).hdV;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T et = (T)x[c * nc + gidx];
            const T e0 = E[c * nc + gidx];
            const T e1 = (et - (T(1) - th) * e0) / th;
            Eth[c * nc + gidx] = et;
            E[c * nc + gidx] = e1;
            acc[0] += hdV * (e1 - e0) * (e1 + e0);
            acc[2] += (e1 - e0) * (e1 - e0);
            acc[3] += hdV * e1 * e1;
        }
        const int ii[2] = {i, wrap1(i + 1, g.nx)}, jj[2] = {j, wrap1(j + 1, g.ny)}, kk[2] = {k, wrap1(k + 1, g.nz)};
        T d[3][3];
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            T sx = T(0), sy = T(0), sz = T(0);
#pragma unroll
            for (int e1 = 0; e1 < 2; ++e1)
#pragma unroll
                for (int e2 = 0; e2 < 2; ++e2) {
                    sx += (T)x[comp * nc + node3(ii[1], jj[e1], kk[e2], g)] - (T)x[comp * nc + node3(ii[0], jj[e1], kk[e2], g)];
                    sy += (T)x[comp * nc + node3(ii[e1], jj[1], kk[e2], g)] - (T)x[comp * nc + node3(ii[e1], jj[0], kk[e2], g)];
                    sz += (T)x[comp * nc + node3(ii[e1], jj[e2], kk[1], g)] - (T)x[comp * nc + node3(ii[e1], jj[e2], kk[0], g)];
                }
            d[0][comp] = sx * gc<T>(g).qdx;
            d[1][comp] = sy * gc<T>(g).qdy;
            d[2][comp] = sz * gc<T>(g).qdz;
        }
        const T curl[3] = {d[1][2] - d[2][1], d[2][0] - d[0][2], d[0][1] - d[1][0]};
        const T dt = gc<T>(g).dt;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T b0 = B0[c * nc + gidx];
            const T b1 = b0 - dt * curl[c];
            B1[c * nc + gidx] = b1;
            acc[1] += hdV * (b1 - b0) * (b1 + b0);
            acc[2] += (b1 - b0) * (b1 - b0);
            acc[4] += hdV * b1 * b1;
        }
        acc[2] *= gc<T>(g).thdV;
    }
    double v[5], o[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) v[q] = (double)acc[q];
    block_sum<5>(v, red, o);
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < 5; ++q) partial[(int64_t)blockIdx.x * kFieldLedger3 + q] = o[q];
}

// ledger term 5: dt dV (Jhat + M E^{n+theta}) . E^{n+theta}, with the same
// blocks as k_field_update3
template <typename T>
__global__ void __launch_bounds__(256)
k_work3(const T* __restrict__ M, const T* __restrict__ J, const T* __restrict__ Eth, GridP g,
        double* __restrict__ partial)
{
    __shared__ double red[32];
    const int64_t nc = g.ncell;
    const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    T wk = T(0);
    if (gidx < nc) {
        const int i = (int)(gidx % g.nx), j = (int)((gidx / g.nx) % g.ny), k = (int)(gidx / ((int64_t)g.nx * g.ny));
        auto f = [&](int comp, int a, int b, int c) -> T {
            return ld(Eth + comp * nc + node3(wrap1(i - 1 + a, g.nx), wrap1(j - 1 + b, g.ny), wrap1(k - 1 + c, g.nz), g));
        };
        T mv[3];
        mv3<T, false>(M, i, j, k, g, f, mv);
#pragma unroll
        for (int c = 0; c < 3; ++c) wk += (J[c * nc + gidx] + mv[c]) * Eth[c * nc + gidx];
        wk *= gc<T>(g).dtdV;
    }
    double v[1] = {(double)wk}, o[1];
    block_sum<1>(v, red, o);
    if (threadIdx.x == 0) partial[(int64_t)blockIdx.x * kFieldLedger3 + 5] = o[0];
}

// ---------------------------------------------------------------------------
// push

// warps of a block: static shared memory below 48 KB
template <typename T>
struct PushCfg3 {
    static constexpr int warps = sizeof(T) == 4 ? 4 : 2;
};

// The explicit push with E^{n+theta} and B^n at x^{n+1/2}: ubar = alpha (u +
// beta E), u^{n+1} = 2 ubar - u^n, x^{n+3/2} = x^{n+1/2} + dt u^{n+1}/gamma^{n+1}
// as a cell shift plus offsets; the pushed particle goes to the same index
// of dst with its new cell in key. Ledger sums per block: dK, work,
// mismatch, K1 (as the 2D push). Warp per row segment of up to 32 cells, the
// lanes over the segment's particles. With rank non-null each particle also
// takes a slot among its new cell's particles, rank[p] = count[key]++ (one
// atomic per new cell and warp: the lanes with equal keys found by
// match-any), for the unstable counting sort that follows.
template <typename T>
__global__ void __launch_bounds__(32 * PushCfg3<T>::warps)
k_push3(PArrays<T> src, const T* __restrict__ sfz, PArrays<T> dst, T* __restrict__ dfz,
        const int32_t* __restrict__ start, int32_t* __restrict__ key, int32_t* __restrict__ rank,
        int32_t* __restrict__ count, const T* __restrict__ Eth, const T* __restrict__ B, GridP g, T beta, T qdt,
        T m, double* __restrict__ lsum, int uw)
{
    __shared__ int sst[PushCfg3<T>::warps][33];
    __shared__ PairTile3<T> stl[PushCfg3<T>::warps];
    __shared__ double red[32 * 4];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int nseg = (g.nx + uw - 1) / uw;
    const int64_t nunits = (int64_t)nseg * g.ny * g.nz;
    int* ss = sst[wib];
    const PairTile3<T>& tl = stl[wib];
    const T dtx = gc<T>(g).dt * gc<T>(g).rdx, dty = gc<T>(g).dt * gc<T>(g).rdy, dtz = gc<T>(g).dt * gc<T>(g).rdz;
    T acc[4] = {T(0), T(0), T(0), T(0)};
    // a batch whose slots are still on their way: its particle, the lanes that
    // share its new cell, and (the first of them) what the count was
    int wait_p = -1, wait_base = 0;
    unsigned wait_peers = 0u;
    auto settle = [&]() {
        const int b = __shfl_sync(0xffffffffu, wait_base, wait_peers ? __ffs(wait_peers) - 1 : lane);
        if (wait_p >= 0) rank[wait_p] = b + __popc(wait_peers & ((1u << lane) - 1u));
        wait_p = -1;
    };
    for (int64_t u = warp; u < nunits; u += nwarps) {
        const int i0 = (int)(u % nseg) * uw;
        const int jk = (int)(u / nseg);
        const int j = jk % g.ny, k = jk / g.ny;
        const int cn = min(uw, g.nx - i0);
        const int64_t c0 = node3(i0, j, k, g);
        __syncwarp();
        if (lane <= cn) ss[lane] = start[c0 + lane];
        if (lane == 0 && cn == 32) ss[32] = start[c0 + 32];
        load_pairs3<T>(stl[wib], Eth, B, i0, cn, j, k, g, lane);
        const int P0 = ss[0], P1 = ss[cn];
        int cl = 0;
        // the next batch is loaded while this one is pushed
        T nfx = T(0), nfy = T(0), nfz = T(0), nux = T(0), nuy = T(0), nuz = T(0), nw = T(0);
        auto fetch = [&](int q) {
            if (q < P1) {
                nfx = ld(src.fx + q);
                nfy = ld(src.fy + q);
                nfz = ld(sfz + q);
                nux = ld(src.ux + q);
                nuy = ld(src.uy + q);
                nuz = ld(src.uz + q);
                nw = ld(src.w + q);
            }
        };
        fetch(P0 + lane);
        for (int p0 = P0; p0 < P1; p0 += 32) {
            const int p = p0 + lane;
            const bool act = p < P1;
            const T fx = nfx, fy = nfy, fz = nfz, ux = nux, uy = nuy, uz = nuz, w = nw;
            fetch(p + 32);
            int newkey = -1 - lane;   // distinct for idle lanes
            if (act) {
                while (ss[cl + 1] <= p) ++cl;
                T E[3], Bp[3];
                tl.gather_E(cl, fx, fy, fz, E);
                tl.gather_B(cl, fx, fy, fz, Bp);
                const T u02 = ux * ux + uy * uy + uz * uz;
                const T g0 = sqrt(T(1) + u02), ig0 = T(1) / g0;
                const T bg = beta * ig0, ax = bg * Bp[0], ay = bg * Bp[1], az = bg * Bp[2];
                const T sa = T(1) / (T(1) + ax * ax + ay * ay + az * az);
                const T wx = ux + beta * E[0], wy = uy + beta * E[1], wz = uz + beta * E[2];
                const T wa = wx * ax + wy * ay + wz * az;
                const T ubx = sa * (wx + (wy * az - wz * ay) + wa * ax);
                const T uby = sa * (wy + (wz * ax - wx * az) + wa * ay);
                const T ubz = sa * (wz + (wx * ay - wy * ax) + wa * az);
                const T u1x = T(2) * ubx - ux, u1y = T(2) * uby - uy, u1z = T(2) * ubz - uz;
                const T u12 = u1x * u1x + u1y * u1y + u1z * u1z;
                const T g1 = sqrt(T(1) + u12), ig1 = T(1) / g1;
                const T t[3] = {fx + dtx * (u1x * ig1), fy + dty * (u1y * ig1), fz + dtz * (u1z * ig1)};
                const int nn[3] = {g.nx, g.ny, g.nz}, cc[3] = {i0 + cl, j, k};
                T fn[3];
                int cnew[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const T fl = floor(t[a]);
                    int sh = (int)fl;
                    T f = t[a] - fl;
                    if (f >= T(1)) { f -= T(1); sh += 1; }
                    fn[a] = f;
                    int q = cc[a] + sh;
                    if ((unsigned)q >= (unsigned)nn[a]) {   // across the box: any distance
                        q %= nn[a];
                        if (q < 0) q += nn[a];
                    }
                    cnew[a] = q;
                }
                dst.fx[p] = fn[0];
                dst.fy[p] = fn[1];
                dfz[p] = fn[2];
                dst.ux[p] = u1x;
                dst.uy[p] = u1y;
                dst.uz[p] = u1z;
                dst.w[p] = w;
                if (dst.id) dst.id[p] = src.id[p];
                newkey = (int32_t)node3(cnew[0], cnew[1], cnew[2], g);
                key[p] = newkey;
                // ledger: g0 - g1 = (u0 - u1).(u0 + u1)/(g0 + g1)
                const T ue = ubx * E[0] + uby * E[1] + ubz * E[2];
                const T du = (ux - u1x) * (ux + u1x) + (uy - u1y) * (uy + u1y) + (uz - u1z) * (uz + u1z);
                const T igs = T(1) / (g0 + g1), wk = qdt * w * ue * ig0;
                acc[0] -= w * m * du * igs;
                acc[1] += wk;
                acc[2] += wk * du * igs * igs;
                acc[3] += w * m * u12 / (g1 + T(1));
            }
            if (rank) {
                settle();   // the last batch's slots have had this one's time to arrive
                const unsigned peers = __match_any_sync(0xffffffffu, newkey);
                wait_peers = peers;
                if (act) {
                    wait_p = p;
                    if ((peers & ((1u << lane) - 1u)) == 0u) wait_base = atomicAdd(count + newkey, __popc(peers));
                }
            }
        }
        __syncwarp();
    }
    if (rank) settle();
    double v[4], o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = (double)acc[q];
    block_sum<4>(v, red, o);
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) lsum[(int64_t)blockIdx.x * 4 + q] = o[q];
}

// the counting sort's placement: particle p to start[key[p]] + rank[p]. Four
// particles a thread: each waits on a chain of loads (key, start, then the
// stores), and one at a time left the kernel bound by that wait
template <typename T>
__global__ void __launch_bounds__(256)
k_place3(PArrays<T> src, const T* __restrict__ sfz, PArrays<T> dst, T* __restrict__ dfz,
         const int32_t* __restrict__ key, const int32_t* __restrict__ rank, const int32_t* __restrict__ start,
         int64_t n)
{
    constexpr int U = 4;
    for (int64_t b = (int64_t)blockIdx.x * (256 * U) + threadIdx.x; b < n; b += (int64_t)gridDim.x * (256 * U)) {
        int64_t q[U], p[U];
        int kk[U], rr[U];
#pragma unroll
        for (int v = 0; v < U; ++v) {
            p[v] = b + 256 * v;
            const bool in = p[v] < n;
            kk[v] = in ? ld(key + p[v]) : 0;
            rr[v] = in ? ld(rank + p[v]) : 0;
            if (!in) p[v] = -1;
        }
#pragma unroll
        for (int v = 0; v < U; ++v) q[v] = (int64_t)ld(start + kk[v]) + rr[v];
        // one array at a time: its U loads in flight, then its stores
        auto move = [&](const T* a, T* o) {
            T x[U];
#pragma unroll
            for (int v = 0; v < U; ++v) x[v] = p[v] >= 0 ? ld(a + p[v]) : T(0);
#pragma unroll
            for (int v = 0; v < U; ++v)
                if (p[v] >= 0) o[q[v]] = x[v];
        };
        move(src.fx, dst.fx);
        move(src.fy, dst.fy);
        if (dfz) move(sfz, dfz);   // null for 2D particles
        move(src.ux, dst.ux);
        move(src.uy, dst.uy);
        move(src.uz, dst.uz);
        move(src.w, dst.w);
        if (dst.id)
#pragma unroll
            for (int v = 0; v < U; ++v)
                if (p[v] >= 0) dst.id[q[v]] = src.id[p[v]];
    }
}

}  // namespace

template <typename T>
cudaError_t load_convert3(const double* x, const double* u, const double* w, int64_t n, GridP g, PArrays<T> out,
                          T* ofz, int32_t* key, int32_t* val, int* bad, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    count_launches(1);
    k_load3<T><<<grid3(n, 256, 152 * 32), 256, 0, st>>>(x, u, w, n, g, out, ofz, key, val, bad);
    return cudaGetLastError();
}

template <typename T>
cudaError_t gather_particles3(const int32_t* perm, PArrays<T> src, const T* sfz, PArrays<T> dst, T* dfz, int64_t n,
                              bool ids_from_perm, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    count_launches(1);
    k_gather3<T><<<grid3(n, 256, 152 * 32), 256, 0, st>>>(perm, src, sfz, dst, dfz, n, ids_from_perm);
    return cudaGetLastError();
}

template <typename T>
cudaError_t export_particles3(PArrays<T> p, const T* fz, const int32_t* start, GridP g, double* x, double* u,
                              double* w, int32_t* id, cudaStream_t st)
{
    count_launches(1);
    k_export3<T><<<grid3((int64_t)g.ncell * 32, 256, 152 * 16), 256, 0, st>>>(p, fz, start, g, x, u, w, id);
    return cudaGetLastError();
}

// the width of the row segments a warp takes: 32 cells, halved while that
// leaves fewer than eight warps per SM
static int unit_width3(GridP g)
{
    int uw = 32;
    while (uw > 4 && (int64_t)((g.nx + uw - 1) / uw) * g.ny * g.nz < 152 * 8) uw /= 2;
    return uw;
}

template <typename T>
cudaError_t deposit3(const DepositSpecies<T>& ds, const FzArrays<T>& fz, const T* B, T* M, T* J, GridP g,
                     cudaStream_t st, int blocks)
{
    const int uw = unit_width3(g);
    const int64_t units = (int64_t)((g.nx + uw - 1) / uw) * g.ny * g.nz;
    count_launches(1);
    k_deposit3<T><<<grid3(units, DepCfg3<T>::warps, blocks > 0 ? blocks : 152 * 8), 32 * DepCfg3<T>::warps, 0, st>>>(
        ds, fz, B, M, J, g, uw);
    return cudaGetLastError();
}

int op_blocks3(GridP g)
{
    return ((g.nx + kOpX3 - 1) / kOpX3) * ((g.ny + kOpY3 - 1) / kOpY3) * ((g.nz + kOpZ3 - 1) / kOpZ3);
}

template <typename T, int MODE, bool TR>
cudaError_t launch_op3(const T* M, const double* in, double sc, const double* b, double* out, double* vj,
                       const double* V, int64_t ldv, int nv, GridP g, double* partial, cudaStream_t st,
                       const GmDyn* dyn)
{
    count_launches(1);
    k_op3<T, MODE, TR><<<op_blocks3(g), kOpT3, 0, st>>>(M, in, sc, b, out, vj, V, ldv, nv, g, partial, dyn);
    return cudaGetLastError();
}

template <typename T>
cudaError_t rhs3(const T* E, const T* B, const T* J, double* b, GridP g, cudaStream_t st)
{
    count_launches(1);
    k_rhs3<T><<<grid3(g.ncell, 256, 152 * 32), 256, 0, st>>>(E, B, J, b, g);
    return cudaGetLastError();
}

template <typename T>
cudaError_t field_update3(const double* x, const T* M, const T* J, T* Eth, T* E, const T* B0, T* B1, GridP g,
                          double* partial, int nblocks, cudaStream_t st)
{
    count_launches(2);
    k_field_update3<T><<<nblocks, 256, 0, st>>>(x, Eth, E, B0, B1, g, partial);
    k_work3<T><<<nblocks, 256, 0, st>>>(M, J, Eth, g, partial);
    return cudaGetLastError();
}

int push_blocks3(GridP g, int cap)
{
    const int uw = unit_width3(g);
    const int64_t units = (int64_t)((g.nx + uw - 1) / uw) * g.ny * g.nz;
    return (int)grid3(units, PushCfg3<float>::warps, cap > 0 ? cap : 152 * 16);
}

template <typename T>
cudaError_t push3(PArrays<T> src, const T* sfz, PArrays<T> dst, T* dfz, const int32_t* start, int32_t* key,
                  int32_t* rank, int32_t* count, const T* Eth, const T* B, GridP g, SpeciesConst sc, double* lsum,
                  int nblocks, cudaStream_t st)
{
    count_launches(1);
    k_push3<T><<<nblocks, 32 * PushCfg3<T>::warps, 0, st>>>(src, sfz, dst, dfz, start, key, rank, count, Eth, B, g,
                                                       (T)(sc.q * g.dt / (2.0 * sc.m)), (T)(sc.q * g.dt), (T)sc.m,
                                                       lsum, unit_width3(g));
    return cudaGetLastError();
}

template <typename T>
cudaError_t place3(PArrays<T> src, const T* sfz, PArrays<T> dst, T* dfz, const int32_t* key, const int32_t* rank,
                   const int32_t* start, int64_t n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    count_launches(1);
    k_place3<T><<<grid3(n, 256 * 4, 152 * 32), 256, 0, st>>>(src, sfz, dst, dfz, key, rank, start, n);
    return cudaGetLastError();
}

#define RELSIM_D3_INSTANTIATE(T)                                                                                   \
    template cudaError_t load_convert3<T>(const double*, const double*, const double*, int64_t, GridP, PArrays<T>, \
                                          T*, int32_t*, int32_t*, int*, cudaStream_t);                             \
    template cudaError_t gather_particles3<T>(const int32_t*, PArrays<T>, const T*, PArrays<T>, T*, int64_t, bool, \
                                              cudaStream_t);                                                       \
    template cudaError_t export_particles3<T>(PArrays<T>, const T*, const int32_t*, GridP, double*, double*,       \
                                              double*, int32_t*, cudaStream_t);                                    \
    template cudaError_t deposit3<T>(const DepositSpecies<T>&, const FzArrays<T>&, const T*, T*, T*, GridP,        \
                                     cudaStream_t, int);                                                                \
    template cudaError_t rhs3<T>(const T*, const T*, const T*, double*, GridP, cudaStream_t);                      \
    template cudaError_t field_update3<T>(const double*, const T*, const T*, T*, T*, const T*, T*, GridP, double*, \
                                          int, cudaStream_t);                                                      \
    template cudaError_t push3<T>(PArrays<T>, const T*, PArrays<T>, T*, const int32_t*, int32_t*, int32_t*,        \
                                  int32_t*, const T*, const T*, GridP, SpeciesConst, double*, int, cudaStream_t);  \
    template cudaError_t place3<T>(PArrays<T>, const T*, PArrays<T>, T*, const int32_t*, const int32_t*,           \
                                   const int32_t*, int64_t, cudaStream_t);                                         \
    template cudaError_t launch_op3<T, 0, false>(const T*, const double*, double, const double*, double*, double*, \
                                                 const double*, int64_t, int, GridP, double*, cudaStream_t,        \
                                                 const GmDyn*);                                                    \
    template cudaError_t launch_op3<T, 1, false>(const T*, const double*, double, const double*, double*, double*, \
                                                 const double*, int64_t, int, GridP, double*, cudaStream_t,        \
                                                 const GmDyn*);                                                    \
    template cudaError_t launch_op3<T, 2, false>(const T*, const double*, double, const double*, double*, double*, \
                                                 const double*, int64_t, int, GridP, double*, cudaStream_t,        \
                                                 const GmDyn*);                                                    \
    template cudaError_t launch_op3<T, 0, true>(const T*, const double*, double, const double*, double*, double*,  \
                                                const double*, int64_t, int, GridP, double*, cudaStream_t,         \
                                                const GmDyn*);                                                     \
    template cudaError_t launch_op3<T, 1, true>(const T*, const double*, double, const double*, double*, double*,  \
                                                const double*, int64_t, int, GridP, double*, cudaStream_t,         \
                                                const GmDyn*);                                                     \
    template cudaError_t launch_op3<T, 2, true>(const T*, const double*, double, const double*, double*, double*,  \
                                                const double*, int64_t, int, GridP, double*, cudaStream_t,         \
                                                const GmDyn*);

RELSIM_D3_INSTANTIATE(float)
RELSIM_D3_INSTANTIATE(double)

}  // namespace relsim
