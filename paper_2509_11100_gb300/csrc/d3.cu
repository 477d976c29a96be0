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
//   k_deposit3   warp per row segment of cells: its particles staged in shared
//                memory 32 at a time, the lanes sum the 27 distinct weight
//                products of a cell's node pairs
//   k_op3        the operator A = I + (theta dt)^2 curl_n curl_c + theta dt M on
//                32 x 2 x 2-node tiles, in the three modes of the 2D operator
//   k_rhs3, k_field_update3   the right-hand side, the field update with the
//                field ledger terms (on the operator's tiles)
//   k_push3      warp per row segment, the push with each particle's new cell
//                and its slot there (any move length), written as records;
//                k_places and k_place3 sort them
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
    const bool unit = is_one(g.dx) && is_one(g.dy) && is_one(g.dz);
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        double s[3] = {x[3 * p], x[3 * p + 1], x[3 * p + 2]};
        if (!unit) {
            s[0] /= g.dx;
            s[1] /= g.dy;
            s[2] /= g.dz;
        }
        const double ux = u[3 * p], uy = u[3 * p + 1], uz = u[3 * p + 2], ww = w[p];
        if (!finite_bits(s[0]) || !finite_bits(s[1]) || !finite_bits(s[2]) || !finite_bits(ux) || !finite_bits(uy) ||
            !finite_bits(uz) || !finite_bits(ww)) {
            atomicOr(bad, 1);
            s[0] = s[1] = s[2] = 0.0;
        }
        const int nn[3] = {g.nx, g.ny, g.nz};
        int c[3];
        T f[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) split_cell<T>(s[a], nn[a], c[a], f[a]);
        out.fx[p] = f[0];
        out.fy[p] = f[1];
        ofz[p] = f[2];
        out.ux[p] = narrow<T>(ux);
        out.uy[p] = narrow<T>(uy);
        out.uz[p] = narrow<T>(uz);
        out.w[p] = narrow<T>(ww);
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
    const bool unit = is_one(g.dx) && is_one(g.dy) && is_one(g.dz);
    for (int c = warp; c < g.ncell; c += nwarps) {
        const int i = c % g.nx, j = (c / g.nx) % g.ny, k = c / (g.nx * g.ny);
        const double id0 = (double)i, jd0 = (double)j, kd0 = (double)k;
        const int p1 = start[c + 1];
        for (int p = start[c] + lane; p < p1; p += 32) {
            if (x) {
                double xs = id0 + widen(pa.fx[p]), ys = jd0 + widen(pa.fy[p]), zs = kd0 + widen(fz[p]);
                if (!unit) {
                    xs *= g.dx;
                    ys *= g.dy;
                    zs *= g.dz;
                }
                x[3 * (int64_t)p] = xs;
                x[3 * (int64_t)p + 1] = ys;
                x[3 * (int64_t)p + 2] = zs;
            }
            if (u) {
                u[3 * (int64_t)p] = widen(pa.ux[p]);
                u[3 * (int64_t)p + 1] = widen(pa.uy[p]);
                u[3 * (int64_t)p + 2] = widen(pa.uz[p]);
            }
            if (w) w[p] = widen(pa.w[p]);
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
// (the 36 corner pairs take 27 distinct weight products), two moments per
// paired FP32 FMA. When a cell is done, its 36 blocks go to M from shared
// memory in address order, so that a warp's additions fall in few sectors, and
// the moments of the cell's upper x face start the next cell's lower face
// instead of being added to memory twice.
//
// Bound by shared memory (FP32: three quarters of its cycles) and issue. A
// particle is staged in 24 words, written and read 16 bytes at a time, and the
// current comes from the moments of a fourth column, c' alpha u beside alpha's
// three (a corner weight is the sum of eight products: X0 = XX0 + XX1, ..),
// with a batch's particles loaded while the batch before is added up: 7.4 ms
// on 256x128x128 with 32 particles a cell (four blocks of 128 registers an SM;
// five with spills 10.8, three 9.3). With 36 words in 4-byte stores of two
// particles side by side 9.1, 13.6 shared wavefronts a particle; with each
// lane owning one or two of the 36 pairs and batches per cell 11.5.
template <typename T>
struct DepCfg3 {
    static constexpr int warps = sizeof(T) == 4 ? 4 : 2;   // static shared memory < 48 KB
    static constexpr int blocks = 4;                       // an SM
};
constexpr int kItems3 = 36 * 9;        // a cell's additions to M
constexpr int kFace3 = 26 * 9;         // those not on the upper x face
constexpr int kMomZ3 = 86, kMomG3 = 255;   // words from ZZ to ZZ and from group to group (no bank conflicts)
// staged values of a particle, FP64: c alpha (rows of four), XX YY, corner
// weights (lower, upper z face), ZZ, current
enum { kS3E = 0, kS3XY = 12, kS3W = 22, kS3Z = 30, kS3V = 33, kS3N = 36 };

// the staged particles of a warp
template <typename T>
struct Stage3 {
    T v[32][kS3N + 1];
    __device__ __forceinline__ void put(int t, const T (&W)[8], const T (&XY)[9], const T (&Z)[3], const T (&ca)[9],
                                        const T (&cu)[3])
    {
        T* r = v[t];
#pragma unroll
        for (int e = 0; e < 9; ++e) r[kS3E + 4 * (e / 3) + e % 3] = ca[e];
#pragma unroll
        for (int e = 0; e < 9; ++e) r[kS3XY + e] = XY[e];
#pragma unroll
        for (int a = 0; a < 8; ++a) r[kS3W + a] = W[a];
#pragma unroll
        for (int e = 0; e < 3; ++e) r[kS3Z + e] = Z[e];
#pragma unroll
        for (int e = 0; e < 3; ++e) r[kS3V + e] = cu[e];
    }
};
// FP32: six pieces of 16 bytes (c alpha's rows with the current's component,
// XX YY, the ninth of them with ZZ) in a row of seven
template <>
struct Stage3<float> {
    float4 v[32][7];
    __device__ __forceinline__ void put(int t, const float (&)[8], const float (&XY)[9], const float (&Z)[3],
                                        const float (&ca)[9], const float (&cu)[3])
    {
        float4* r = v[t];
#pragma unroll
        for (int e = 0; e < 3; ++e) r[e] = make_float4(ca[3 * e], ca[3 * e + 1], ca[3 * e + 2], cu[e]);
        r[3] = make_float4(XY[0], XY[1], XY[2], XY[3]);
        r[4] = make_float4(XY[4], XY[5], XY[6], XY[7]);
        r[5] = make_float4(XY[8], Z[0], Z[1], Z[2]);
    }
};

// A lane's sums over a cell: lanes 0..26 are three groups of nine that take
// the staged particles in turn; a group's lane (zz, er) sums the nine moments
// (XX, YY) of its ZZ for row er of alpha and, FP64 at zz = 0 and 2, component
// er of the current at the four corners of the lower and upper z face, FP32
// the moments of that component. (What a staged particle costs is the bytes a
// lane loads, also where all lanes load the same ones: a tile of 9 products x
// 3 or 4 entries takes a third of the shared-memory traffic of one product x 9
// entries in each lane.)
template <typename T>
struct Acc3 {
    T m[9][3], j[4];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int k = 0; k < 9; ++k)
#pragma unroll
            for (int e = 0; e < 3; ++e) m[k][e] = T(0);
#pragma unroll
        for (int c = 0; c < 4; ++c) j[c] = T(0);
    }
    // staged particles t0 .. t1-1, every third from the grp-th of the batch
    __device__ __forceinline__ void add(const Stage3<T>& st, int t0, int t1, int grp, int zz, int er)
    {
        for (int t = t0 + (grp + 3 - t0 % 3) % 3; t < t1; t += 3) {
            const T* r = st.v[t];
            const T z = r[kS3Z + zz];
            T e[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) e[q] = z * r[kS3E + 4 * er + q];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const T w = r[kS3XY + k];
#pragma unroll
                for (int q = 0; q < 3; ++q) m[k][q] += w * e[q];
            }
            const T v = r[kS3V + er];
#pragma unroll
            for (int c = 0; c < 4; ++c) j[c] += r[kS3W + 2 * zz + c] * v;
        }
    }
    __device__ __forceinline__ T moment(int k, int e) const { return m[k][e]; }
    // corner c of the ZZ's z face (zz = 1 has none)
    __device__ __forceinline__ void currents(T (&o)[4]) const
    {
#pragma unroll
        for (int c = 0; c < 4; ++c) o[c] = j[c];
    }
    // a corner's current from what the lanes of a group left: value [zz][c]
    static __device__ __forceinline__ T corner(const T* o, int z, int at) { return o[24 * z + at]; }
    // the upper x face's sums become the next cell's lower face's
    __device__ __forceinline__ void carry()
    {
#pragma unroll
        for (int k = 0; k < 9; ++k)
#pragma unroll
            for (int e = 0; e < 3; ++e) m[k][e] = k < 3 ? m[k + 6][e] : T(0);
#pragma unroll
        for (int c = 0; c < 4; ++c) j[c] = (c & 1) == 0 ? j[c + 1] : T(0);
    }
};
template <>
struct Acc3<float> {
    float2 m[4][4];   // moments 2 k and 2 k + 1 of alpha's three entries and the current
    float m8[4];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int k = 0; k < 4; ++k) m[k][e] = make_float2(0.f, 0.f);
            m8[e] = 0.f;
        }
    }
    __device__ __forceinline__ void add(const Stage3<float>& st, int t0, int t1, int grp, int zz, int er)
    {
#pragma unroll 2
        for (int t = t0 + (grp + 3 - t0 % 3) % 3; t < t1; t += 3) {
            const float4* r = st.v[t];
            const float4 a = r[er], w0 = r[3], w1 = r[4];
            const float* s = reinterpret_cast<const float*>(r + 5);
            const float w8 = s[0], z = s[1 + zz];
            const float2 w[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                                 make_float2(w1.z, w1.w)};
            const float e[4] = {z * a.x, z * a.y, z * a.z, z * a.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 ee = make_float2(e[q], e[q]);
#pragma unroll
                for (int k = 0; k < 4; ++k) m[k][q] = __ffma2_rn(w[k], ee, m[k][q]);
                m8[q] += w8 * e[q];
            }
        }
    }
    __device__ __forceinline__ float moment(int k, int e) const
    {
        return k == 8 ? m8[e] : ((k & 1) ? m[(k >> 1) & 3][e].y : m[(k >> 1) & 3][e].x);
    }
    __device__ __forceinline__ void currents(float (&o)[4]) const
    {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int k = (c & 1) * 3 + (c >> 1);
            o[c] = (moment(k, 3) + moment(k + 1, 3)) + (moment(k + 3, 3) + moment(k + 4, 3));
        }
    }
    static __device__ __forceinline__ float corner(const float* o, int z, int at)
    {
        return o[12 * z + at] + o[12 * z + 12 + at];
    }
    __device__ __forceinline__ void carry()
    {
        // (the current's: the upper face's corner takes XX1 + XX2)
        float n[3][4];
#pragma unroll
        for (int y = 0; y < 3; ++y)
#pragma unroll
            for (int e = 0; e < 4; ++e) n[y][e] = e < 3 ? moment(6 + y, e) : moment(3 + y, e) + moment(6 + y, e);
        clear();
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            m[0][e] = make_float2(n[0][e], n[1][e]);
            m[1][e] = make_float2(n[2][e], 0.f);
        }
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
__global__ void __launch_bounds__(32 * DepCfg3<T>::warps, DepCfg3<T>::blocks)
k_deposit3(const __grid_constant__ DepositSpecies<T> ds, const __grid_constant__ FzArrays<T> fz,
           const T* __restrict__ B, T* __restrict__ M, T* __restrict__ J,
           GridP g, int uw)
{
    constexpr int kW = DepCfg3<T>::warps;
    __shared__ __align__(16) Stage3<T> sst[kW];
    __shared__ Tile3B<T> stl[kW];
    __shared__ T smom[kW][3 * kMomG3];   // a cell's moments (the three groups'), for the additions
    __shared__ T scur[kW][3][36];        // and its currents: ZZ, corner of the z face, component
    __shared__ int snode[kW][8];         // its corners' nodes
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
            item[rank * 9 + e] = (unsigned)at << 16 | (unsigned)(hs * 9 + e) << 8 | (unsigned)(mom / 9 * kMomZ3 + mom % 9 * 9 + e);
    }
    __syncthreads();
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int nseg = (g.nx + uw - 1) / uw;
    const int64_t nunits = (int64_t)nseg * g.ny * g.nz;
    const int nsp = ds.nsp, gcells = 32 / nsp;   // cells whose (cell, species) ranges fit the lanes
    Stage3<T>& st = sst[wib];
    const bool own = lane < 27;
    const int grp = own ? lane / 9 : 0, zz = own ? lane / 3 % 3 : 0, er = own ? lane % 3 : 0;
    for (int64_t u = warp; u < nunits; u += nwarps) {
        const int i0 = (int)(u % nseg) * uw;
        const int jk = (int)(u / nseg);
        const int j = jk % g.ny, k = jk / g.ny;
        const int cn = min(uw, g.nx - i0);
        __syncwarp();
        load_tile3B<T>(stl[wib], B, i0, cn, j, k, g, lane);
        Acc3<T> acc;
        acc.clear();
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
            // a batch's particles are loaded while the batch before is added up
            int nsg = 0;
            T nfx = T(0), nfy = T(0), nfz = T(0), nux = T(0), nuy = T(0), nuz = T(0), nwt = T(0);
            auto fetch = [&](int t) {
                // the range the lane's particle lies in (all lanes search)
                int seg = 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    if (__shfl_sync(0xffffffffu, incl, seg + o - 1) <= t) seg += o;
                const int p = __shfl_sync(0xffffffffu, base, seg) + t;
                nsg = seg;
                if (t < total) {
                    const int s = seg % nsp;
                    nfx = ld(ds.fx[s] + p);
                    nfy = ld(ds.fy[s] + p);
                    nfz = ld(fz.fz[s] + p);
                    nux = ld(ds.ux[s] + p);
                    nuy = ld(ds.uy[s] + p);
                    nuz = ld(ds.uz[s] + p);
                    nwt = ld(ds.w[s] + p);
                }
            };
            fetch(lane);
            for (int w0 = 0; cl < gc0; w0 += 32) {   // (every pass ends cells or takes 32 particles)
                const int t = w0 + lane;
                const int seg = nsg;
                const T fx = nfx, fy = nfy, fzz = nfz, ux = nux, uy = nuy, uz = nuz, wt = nwt;
                if (w0 + 32 < total) fetch(t + 32);
                if (t < total) {
                    const int s = seg % nsp, pc = cg + seg / nsp;
                    T W[8] = {}, Bp[3], al[9];
                    if (sizeof(T) == 8) corner_weights(fx, fy, fzz, W);
                    tile_B3(stl[wib].B, pc, fx, fy, fzz, Bp);
                    const T ig = T(1) / sqrt(T(1) + ux * ux + uy * uy + uz * uz);
                    alpha3(Bp, ds.beta[s] * ig, al);
                    const T cM = wt * ds.cM[s] * ig, cJ = wt * ds.cJ[s] * ig;
                    const T X[3] = {(T(1) - fx) * (T(1) - fx), (T(1) - fx) * fx, fx * fx};
                    const T Y[3] = {(T(1) - fy) * (T(1) - fy), (T(1) - fy) * fy, fy * fy};
                    const T Z[3] = {(T(1) - fzz) * (T(1) - fzz), (T(1) - fzz) * fzz, fzz * fzz};
                    T XY[9], ca[9], cu[3];
#pragma unroll
                    for (int e = 0; e < 9; ++e) {
                        ca[e] = cM * al[e];
                        XY[e] = X[e / 3] * Y[e % 3];
                    }
#pragma unroll
                    for (int r = 0; r < 3; ++r) cu[r] = cJ * (al[3 * r] * ux + al[3 * r + 1] * uy + al[3 * r + 2] * uz);
                    st.put(lane, W, XY, Z, ca, cu);
                }
                __syncwarp();
                const int wend = min(w0 + 32, total);
                int pos = w0;
                while (cl < gc0) {
                    const int upto = min(cend, wend);
                    if (upto > pos && own) acc.add(st, pos - w0, upto - w0, grp, zz, er);
                    pos = max(pos, upto);
                    if (cend > wend) break;   // the cell goes on in the next batch
                    // the cell is done
                    const int before = cl == 0 ? 0 : __shfl_sync(0xffffffffu, incl, cl * nsp - 1);
                    const bool last = cg + cl == cn - 1;
                    if (carry || cend > before) {
                        if (own) {
                            T* const o = smom[wib] + grp * kMomG3 + zz * kMomZ3 + er * 3;
#pragma unroll
                            for (int k = 0; k < 9; ++k)
                                if (k < 6 || last)
#pragma unroll
                                    for (int e = 0; e < 3; ++e) o[k * 9 + e] = acc.moment(k, e);
                            T cur[4];
                            acc.currents(cur);
#pragma unroll
                            for (int c = 0; c < 4; ++c) scur[wib][grp][(zz * 4 + c) * 3 + er] = cur[c];
                        }
                        const int i = i0 + cg + cl;
                        const int64_t nd = node3(wrap1(i + (lane & 1), g.nx), wrap1(j + ((lane >> 1) & 1), g.ny),
                                                 wrap1(k + ((lane >> 2) & 1), g.nz), g);
                        if (lane < 8) snode[wib][lane] = (int)nd;
                        __syncwarp();
                        const T* sm = &smom[wib][0];
                        auto give = [&](unsigned q) {
                            const unsigned v = q & 255u;
                            atomicAdd(M + (int64_t)snode[wib][q >> 16] * kMBlock3 + ((q >> 8) & 255u),
                                      sm[v] + sm[kMomG3 + v] + sm[2 * kMomG3 + v]);
                        };
#pragma unroll
                        for (int v = 0; v < (kFace3 + 31) / 32; ++v)
                            if (lane + 32 * v < kFace3) give(item[lane + 32 * v]);
                        if (last)
                            for (int it = kFace3 + lane; it < kItems3; it += 32) give(item[it]);
                        const int ja = lane / 3, jc = lane % 3;
                        if (lane < 24 && (last || (ja & 1) == 0)) {
                            const int at = (ja & 3) * 3 + jc, z = ja >> 2;
                            atomicAdd(J + (int64_t)jc * g.ncell + snode[wib][ja],
                                      Acc3<T>::corner(scur[wib][0], z, at) + Acc3<T>::corner(scur[wib][1], z, at) +
                                          Acc3<T>::corner(scur[wib][2], z, at));
                        }
                        __syncwarp();
                        carry = !last;
                    }
                    // the upper x face's sums start the next cell's lower face
                    if (last) acc.clear();
                    else acc.carry();
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
constexpr int kOpChunk3 = 8;

// the differences along each axis of three components at the 8 corners
// f(comp, a, b, c) of a cube, averaged over its 4 edges, as a curl: a cell
// from its nodes, or a node from the cells around it
template <typename T, typename F>
__device__ __forceinline__ void curl_cell3(F f, T rx, T ry, T rz, T (&C)[3])
{
    T d[3][3];   // d[axis][comp]
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
        T sx = T(0), sy = T(0), sz = T(0);
#pragma unroll
        for (int e1 = 0; e1 < 2; ++e1)
#pragma unroll
            for (int e2 = 0; e2 < 2; ++e2) {
                sx += f(comp, 1, e1, e2) - f(comp, 0, e1, e2);
                sy += f(comp, e1, 1, e2) - f(comp, e1, 0, e2);
                sz += f(comp, e1, e2, 1) - f(comp, e1, e2, 0);
            }
        d[0][comp] = sx * rx;
        d[1][comp] = sy * ry;
        d[2][comp] = sz * rz;
    }
    C[0] = d[1][2] - d[2][1];
    C[1] = d[2][0] - d[0][2];
    C[2] = d[0][1] - d[1][0];
}

// The operator's tiles: 32 x 2 x 2 nodes (FP64: 32 x 2 x 1). The tile's own mass-matrix rows (16 KB a row of 32 nodes in FP32) come
// into shared memory by asynchronous copies, all in flight together, while
// the input is staged; read straight from global memory (504 bytes from lane
// to lane) every load of a block touched 32 lines, and the operator was bound
// by their latency: 1.28 ms an application on 256x128x128 (FP32 form).
// Three tiles fit an SM's shared memory, and with a thread a node their twelve
// warps left it waiting (a third of the issue slots used, no unit above 45%):
// two threads share a node, one for its own blocks, one for its neighbours',
// and take the products with the basis in turn. 6.99 -> 6.5 ms for a step's
// seven applications, FP64 at 64x32x32 1.28 -> 1.05 ms a step. The field
// update keeps one thread a node: its neighbours' blocks need the registers
// (1.15 ms, with two 1.42). The neighbours' blocks from outside the tile,
// copied to shared memory like its own, leave two tiles an SM: slower, 8.1 ms.
template <typename T>
struct Op3 {
    static constexpr int X = 32, Y = 2, Z = sizeof(T) == 4 ? 2 : 1, nodes = X * Y * Z;
    static constexpr int share = 2;   // threads of a node in the operator (one in the field update)
    struct Shared {
        T Mm[Z * Y][X * kMBlock3];              // own blocks, row z Y + y
        T v[3][Z + 2][Y + 2][X + 2];            // the input on the 1-node halo
        T C[3][Z + 1][Y + 1][X + 1];            // its curl on the cells around the tile's nodes
        T part[3][nodes];                       // the neighbours' share of M v
    };
    static_assert(sizeof(Shared) >= sizeof(double) * (kOpChunk3 + 3) * nodes, "the dot products reuse it");
};
// a block's tile and this thread's node
template <typename T>
struct At3 {
    int i0, j0, k0, tw, th, td, tx, ty, tz, i, j, k, node;
    bool second;   // the node's second thread
    bool active;
    int64_t gidx;
    __device__ __forceinline__ explicit At3(const GridP& g)
    {
        using O = Op3<T>;
        const int nx = (g.nx + O::X - 1) / O::X, ny = (g.ny + O::Y - 1) / O::Y;
        const int bx = blockIdx.x % nx, by = (blockIdx.x / nx) % ny, bz = blockIdx.x / (nx * ny);
        i0 = bx * O::X;
        j0 = by * O::Y;
        k0 = bz * O::Z;
        tw = min(O::X, g.nx - i0);
        th = min(O::Y, g.ny - j0);
        td = min(O::Z, g.nz - k0);
        tx = threadIdx.x % O::X;
        ty = (threadIdx.x / O::X) % O::Y;
        node = threadIdx.x % O::nodes;
        second = threadIdx.x >= O::nodes;
        tz = node / (O::X * O::Y);
        i = i0 + tx;
        j = j0 + ty;
        k = k0 + tz;
        active = tx < tw && ty < th && tz < td;
        gidx = active ? node3(i, j, k, g) : 0;
    }
};

// start the copies of the tile's mass-matrix rows (16 bytes each where the
// rows are aligned to that, else 8)
template <typename T>
__device__ __forceinline__ void fetch_rows3(typename Op3<T>::Shared& S, const T* __restrict__ M, const At3<T>& t,
                                            const GridP& g)
{
    using O = Op3<T>;
    const bool wide = ((int64_t)g.nx * kMBlock3 * sizeof(T)) % 16 == 0;
    const int n = t.tw * kMBlock3 * (int)sizeof(T) / (wide ? 16 : 8);
#pragma unroll
    for (int r = 0; r < O::Y * O::Z; ++r) {
        const int y = r % O::Y, z = r / O::Y;
        if (y >= t.th || z >= t.td) continue;
        const char* src = reinterpret_cast<const char*>(M + node3(t.i0, t.j0 + y, t.k0 + z, g) * kMBlock3);
        char* dst = reinterpret_cast<char*>(&S.Mm[r][0]);
        if (wide)
            for (int q = threadIdx.x; q < n; q += blockDim.x) cp_async16(dst + 16 * q, src + 16 * q);
        else
            for (int q = threadIdx.x; q < n; q += blockDim.x) cp_async8(dst + 8 * q, src + 8 * q);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// the input (FP64) on the tile's halo in T, times s, and its curl on the
// cells around the tile's nodes (each formed once); the rows' copies land
template <typename T, bool SCALED>
__device__ __forceinline__ void stage_input3(typename Op3<T>::Shared& S, const double* __restrict__ in, T s,
                                             const At3<T>& t, const GridP& g)
{
    using O = Op3<T>;
    constexpr int HX = O::X + 2, HY = O::Y + 2, HZ = O::Z + 2;
    const int64_t nc = g.ncell;
    const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
    const int ga = wrap1(min(t.i0 - 1 + lane, 2 * g.nx - 1), g.nx), gb = wrap1(min(t.i0 + 31 + lane, 2 * g.nx - 1), g.nx);
    // a warp a row of 34 (a lane a column, the last two by two lanes), four
    // rows of loads in flight
    constexpr int rows = 3 * HZ * HY;
    const int W = blockDim.x / 32;
    for (int r0 = wid; r0 < rows; r0 += 4 * W) {
        double a[4], b[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = min(r0 + v * W, rows - 1), comp = r / (HZ * HY), zz = (r / HY) % HZ, yy = r % HY;
            const int gj = wrap1(min(t.j0 - 1 + yy, 2 * g.ny - 1), g.ny), gk = wrap1(min(t.k0 - 1 + zz, 2 * g.nz - 1), g.nz);
            const double* row = in + comp * nc + node3(0, gj, gk, g);
            a[v] = __ldg(row + ga);
            b[v] = lane < 2 ? __ldg(row + gb) : 0.0;
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = r0 + v * W;
            if (r >= rows) break;
            T* o = &S.v[0][0][0][0] + r * HX;
            T x = narrow<T>(a[v]);
            if (SCALED) x *= s;
            o[lane] = x;
            if (lane < 2) {
                T y = narrow<T>(b[v]);
                if (SCALED) y *= s;
                o[32 + lane] = y;
            }
        }
    }
    __syncthreads();
    const T rx = gc<T>(g).qdx, ry = gc<T>(g).qdy, rz = gc<T>(g).qdz;
    for (int q = threadIdx.x; q < (O::Z + 1) * (O::Y + 1) * (O::X + 1); q += blockDim.x) {
        const int c = q % (O::X + 1), y = (q / (O::X + 1)) % (O::Y + 1), z = q / ((O::X + 1) * (O::Y + 1));
        T C[3];
        curl_cell3<T>([&](int comp, int p, int o, int w) { return S.v[comp][z + w][y + o][c + p]; }, rx, ry, rz, C);
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) S.C[comp][z][y][c] = C[comp];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// the offset of stored block h (0..13)
__device__ __forceinline__ void half_offset3(int h, int& di, int& dj, int& dk)
{
    if (h < 2) { di = h; dj = 0; dk = 0; }
    else if (h < 5) { di = h - 3; dj = 1; dk = 0; }
    else { di = (h - 5) % 3 - 1; dj = (h - 5) / 3 - 1; dk = 1; }
}

// a stored block (9 values; even: the row starts on a pair of T) in registers
__device__ __forceinline__ void block3(const float* p, int h, float (&m)[9])
{
    if (h & 1) {
        m[0] = p[0];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 q = *reinterpret_cast<const float2*>(p + 1 + 2 * e);
            m[1 + 2 * e] = q.x;
            m[2 + 2 * e] = q.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 q = *reinterpret_cast<const float2*>(p + 2 * e);
            m[2 * e] = q.x;
            m[2 * e + 1] = q.y;
        }
        m[8] = p[8];
    }
}
__device__ __forceinline__ void block3(const double* p, int, double (&m)[9])
{
#pragma unroll
    for (int e = 0; e < 9; ++e) m[e] = p[e];
}

// (M v) at the thread's node: its own 14 stored blocks times v at g + d(h),
// and the 13 neighbours' blocks M[g - d(h)][h] times v at g - d(h) (from the
// tile where they lie in it, else from global memory); with TR each block
// applied transposed. With SHARE 2 a node's two threads take one sum each and the first
// gets both (every thread of the block calls)
template <typename T, bool TR, int SHARE>
__device__ __forceinline__ void mv3(typename Op3<T>::Shared& S, const T* __restrict__ M, const At3<T>& t,
                                    const GridP& g, T (&out)[3])
{
    using O = Op3<T>;
    T r[3] = {T(0), T(0), T(0)};
    const T* Mg = &S.Mm[t.tz * O::Y + t.ty][t.tx * kMBlock3];
    auto add = [&](const T (&m)[9], int di, int dj, int dk) {
        T vv[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) vv[s] = S.v[s][t.tz + 1 + dk][t.ty + 1 + dj][t.tx + 1 + di];
#pragma unroll
        for (int rr = 0; rr < 3; ++rr)
#pragma unroll
            for (int s = 0; s < 3; ++s) r[rr] += m[TR ? s * 3 + rr : rr * 3 + s] * vv[s];
    };
    auto neighbour = [&](int h, T (&m)[9]) {
        int di, dj, dk;
        half_offset3(h, di, dj, dk);
        const int x = t.tx - di, y = t.ty - dj, z = t.tz - dk;
        const T* Mn = x >= 0 && x < t.tw && y >= 0 && y < t.th && z >= 0
                          ? &S.Mm[z * O::Y + y][x * kMBlock3]
                          : M + node3(wrap1(t.i - di, g.nx), wrap1(t.j - dj, g.ny), wrap1(t.k - dk, g.nz), g) * kMBlock3;
        block3(Mn + h * 9, h, m);
    };
    // the neighbours' blocks three at a time (h = 2..4, 5..7, 8..10, 11..13),
    // each three on their way while the blocks before them are added
    T nb[2][3][9];
    auto begin = [&]() {
#pragma unroll
        for (int q = 0; q < 3; ++q) neighbour(2 + q, nb[0][q]);
    };
    auto others = [&]() {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (n < 3) neighbour(2 + 3 * (n + 1) + q, nb[(n + 1) & 1][q]);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                int di, dj, dk;
                half_offset3(2 + 3 * n + q, di, dj, dk);
                add(nb[n & 1][q], -di, -dj, -dk);
            }
        }
        T m[9];
        neighbour(1, m);
        add(m, -1, 0, 0);
    };
    auto mine = [&]() {
#pragma unroll
        for (int h = 0; h < kHalf3; ++h) {
            int di, dj, dk;
            half_offset3(h, di, dj, dk);
            T m[9];
            block3(Mg + h * 9, h, m);
            add(m, di, dj, dk);
        }
    };
    if (SHARE == 1) {
        if (t.active) {
            begin();
            mine();
            others();
        }
    } else {
        if (t.second && t.active) {
            begin();
            others();
#pragma unroll
            for (int c = 0; c < 3; ++c) S.part[c][t.node] = r[c];
        } else if (t.active) {
            mine();
        }
        __syncthreads();
        if (t.active && !t.second)
#pragma unroll
            for (int c = 0; c < 3; ++c) r[c] += S.part[c][t.node];
    }
    out[0] = r[0];
    out[1] = r[1];
    out[2] = r[2];
}

// The operator; the modes and the per-block partial sums are those of the 2D
// operator:
//   A:        out = in + B in
//   Residual: out = b - (in + B in), partial |out|^2
//   Arnoldi:  v = s in (to vj when vj is not null), out = B v, partials
//             <out, V_q> (q < nv), <out, v>, <out, out>
template <typename T, int MODE, bool TR>
__global__ void __launch_bounds__(Op3<T>::share * Op3<T>::nodes, 3)
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
    using O = Op3<T>;
    extern __shared__ __align__(128) unsigned char op3_smem[];
    typename O::Shared& S = *reinterpret_cast<typename O::Shared*>(op3_smem);
    const At3<T> t(g);
    const int64_t nc = g.ncell;
    const int tid = threadIdx.x;
    fetch_rows3<T>(S, M, t, g);
    double own[3] = {0.0, 0.0, 0.0}, wv[3] = {0.0, 0.0, 0.0};
    const bool owner = t.active && !t.second;
    if (owner) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            own[c] = __ldg(in + c * nc + t.gidx);
            if (MODE == k3Arnoldi && !is_one(s)) own[c] *= s;
        }
    }
    if (MODE == k3Arnoldi) stage_input3<T, true>(S, in, (T)s, t, g);
    else stage_input3<T, false>(S, in, T(1), t, g);
    T mv[3];
    mv3<T, TR, O::share>(S, M, t, g, mv);
    if (owner) {
        T cc3[3];
        curl_cell3<T>([&](int comp, int p, int o, int w) { return S.C[comp][t.tz + w][t.ty + o][t.tx + p]; },
                      gc<T>(g).qdx, gc<T>(g).qdy, gc<T>(g).qdz, cc3);
        const T td = gc<T>(g).td;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double bv = widen(td * td * cc3[c] + td * mv[c]);
            if (MODE == k3A) wv[c] = own[c] + bv;
            else if (MODE == k3Residual) wv[c] = b[c * nc + t.gidx] - (own[c] + bv);
            else wv[c] = bv;
            out[c * nc + t.gidx] = wv[c];
            if (MODE == k3Arnoldi && vj) vj[c * nc + t.gidx] = own[c];
        }
    }
    if (MODE == k3A) return;
    const int nq = MODE == k3Residual ? 1 : nv + 2;
    const int lane = tid & 31, wid = tid >> 5;
    double* buf = reinterpret_cast<double*>(op3_smem);   // [kOpChunk3][nodes]
    __syncthreads();   // the tile is no longer read
    if (MODE == k3Arnoldi && O::share == 2) {   // a node's threads take the products with the basis in turn
        double* const sw = buf + kOpChunk3 * O::nodes;
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (!t.second) sw[c * O::nodes + t.node] = wv[c];
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 3; ++c) wv[c] = sw[c * O::nodes + t.node];
    }
    for (int q0 = 0; q0 < nq; q0 += kOpChunk3) {
        const int kc = min(kOpChunk3, nq - q0);
        for (int c = 0; c < kc; ++c) {
            const int q = q0 + c;
            if (O::share == 2 && t.second != (MODE == k3Arnoldi && q < nv && (q & 1))) continue;
            double d = 0.0;
            if (t.active) {
                if (MODE == k3Residual || q == nv + 1) d = wv[0] * wv[0] + wv[1] * wv[1] + wv[2] * wv[2];
                else if (q == nv) d = wv[0] * own[0] + wv[1] * own[1] + wv[2] * own[2];
                else {
                    const double* Vq = V + (int64_t)q * ldv + t.gidx;
                    d = wv[0] * __ldg(Vq) + wv[1] * __ldg(Vq + nc) + wv[2] * __ldg(Vq + 2 * nc);
                }
            }
            buf[c * O::nodes + t.node] = d;
        }
        __syncthreads();
        for (int c = wid; c < kc; c += O::share * O::nodes / 32) {
            double sum = 0.0;
#pragma unroll
            for (int m = 0; m < O::nodes / 32; ++m) sum += buf[c * O::nodes + m * 32 + lane];
            sum = warp_sum(sum);
            if (lane == 0) partial[(int64_t)blockIdx.x * nq + q0 + c] = sum;
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
// field ledger terms, on the operator's tiles: the solution is staged in T
// once for the curl, the work and the update (as two kernels it was converted
// at every one of a node's 24 uses, on the FP64 pipe, and M was read from
// global memory: 1.7 ms on 256x128x128, FP32 form). Term 5 is the work
// dt dV (Jhat + M E^{n+theta}) . E^{n+theta}.
template <typename T>
__global__ void __launch_bounds__(Op3<T>::nodes, 3)
k_field_update3(const double* __restrict__ x, const T* __restrict__ M, const T* __restrict__ J, T* __restrict__ Eth,
                T* __restrict__ E, const T* __restrict__ B0, T* __restrict__ B1, GridP g, double* __restrict__ partial)
{
    using O = Op3<T>;
    extern __shared__ __align__(128) unsigned char op3_smem[];
    typename O::Shared& S = *reinterpret_cast<typename O::Shared*>(op3_smem);
    const At3<T> t(g);
    const int64_t nc = g.ncell;
    fetch_rows3<T>(S, M, t, g);
    stage_input3<T, false>(S, x, T(1), t, g);
    T acc[kFieldLedger3] = {T(0), T(0), T(0), T(0), T(0), T(0)};
    if (t.active) {
        const T th = gc<T>(g).theta, hdV = gc<T>(g).hdV, dt = gc<T>(g).dt;
        T mv[3], wk = T(0);
        mv3<T, false, 1>(S, M, t, g, mv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T et = S.v[c][t.tz + 1][t.ty + 1][t.tx + 1];
            const T e0 = E[c * nc + t.gidx];
            const T e1 = (et - (T(1) - th) * e0) / th;
            Eth[c * nc + t.gidx] = et;
            E[c * nc + t.gidx] = e1;
            acc[0] += hdV * (e1 - e0) * (e1 + e0);
            acc[2] += (e1 - e0) * (e1 - e0);
            acc[3] += hdV * e1 * e1;
            wk += (J[c * nc + t.gidx] + mv[c]) * et;
            // the cell's upper nodes: its curl is the one after the node's in x, y and z
            const T b0 = B0[c * nc + t.gidx];
            const T b1 = b0 - dt * S.C[c][t.tz + 1][t.ty + 1][t.tx + 1];
            B1[c * nc + t.gidx] = b1;
            acc[1] += hdV * (b1 - b0) * (b1 + b0);
            acc[2] += (b1 - b0) * (b1 - b0);
            acc[4] += hdV * b1 * b1;
        }
        acc[2] *= gc<T>(g).thdV;
        acc[5] = gc<T>(g).dtdV * wk;
    }
    double* red = reinterpret_cast<double*>(op3_smem);
    __syncthreads();   // the tile is no longer read
    double v[kFieldLedger3], o[kFieldLedger3];
#pragma unroll
    for (int q = 0; q < kFieldLedger3; ++q) v[q] = (double)acc[q];
    block_sum<kFieldLedger3>(v, red, o);
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < kFieldLedger3; ++q) partial[(int64_t)blockIdx.x * kFieldLedger3 + q] = o[q];
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
// lanes over the segment's particles. Each particle also takes a slot among
// its new cell's particles, rank[p] = count[key]++ (one atomic per new cell
// and warp: the lanes with equal keys found by match-any), for the unstable
// counting sort that follows.
template <typename T>
__global__ void __launch_bounds__(32 * PushCfg3<T>::warps)
k_push3(PArrays<T> src, const T* __restrict__ sfz, PRecords<T> dst,
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
        int nid = 0;
        auto fetch = [&](int q) {
            if (q < P1) {
                nfx = ld(src.fx + q);
                nfy = ld(src.fy + q);
                nfz = ld(sfz + q);
                nux = ld(src.ux + q);
                nuy = ld(src.uy + q);
                nuz = ld(src.uz + q);
                nw = ld(src.w + q);
                if (src.id) nid = ld(src.id + q);
            }
        };
        fetch(P0 + lane);
        for (int p0 = P0; p0 < P1; p0 += 32) {
            const int p = p0 + lane;
            const bool act = p < P1;
            const T fx = nfx, fy = nfy, fz = nfz, ux = nux, uy = nuy, uz = nuz, w = nw;
            const int pid = nid;
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
                dst.a[p] = PRecA<T>{fn[0], fn[1], u1x, u1y};
                dst.b[p] = PRecB<T>{u1z, w};
                dst.fz[p] = fn[2];
                if (dst.id) dst.id[p] = pid;
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
            settle();   // the last batch's slots have had this one's time to arrive
            const unsigned peers = __match_any_sync(0xffffffffu, newkey);
            wait_peers = peers;
            if (act) {
                wait_p = p;
                if ((peers & ((1u << lane) - 1u)) == 0u) wait_base = atomicAdd(count + newkey, __popc(peers));
            }
        }
        __syncwarp();
    }
    settle();
    double v[4], o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = (double)acc[q];
    block_sum<4>(v, red, o);
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) lsum[(int64_t)blockIdx.x * 4 + q] = o[q];
}

// The counting sort's placement in two passes: where each particle goes
// (perm[start[key[p]] + rank[p]] = p), then the particles in their new order,
// each record's pieces read where they lie and the arrays written in order.
// About half of the particles change cell, so one side of the sort goes to
// sectors of its own: written from arrays to arrays that was seven or eight
// scattered 4-byte stores a particle, 3.15 ms a species on 256x128x128 with
// 16 particles a cell (FP32 form, 67 million with ids). Now one scattered store and four
// loads of whole pieces, 0.31 + 1.22 ms (3.7 TB/s of algorithmic bytes, bound
// by sectors used in part). Both run several particles a thread: each waits on a
// chain of loads.
__global__ void __launch_bounds__(256)
k_places(const int32_t* __restrict__ key, const int32_t* __restrict__ rank, const int32_t* __restrict__ start,
         int32_t* __restrict__ perm, int64_t n)
{
    constexpr int U = 4;
    for (int64_t b = (int64_t)blockIdx.x * (256 * U) + threadIdx.x; b < n; b += (int64_t)gridDim.x * (256 * U)) {
        int kk[U], rr[U];
#pragma unroll
        for (int v = 0; v < U; ++v) {
            const int64_t p = b + 256 * v;
            kk[v] = p < n ? ld(key + p) : 0;
            rr[v] = p < n ? ld(rank + p) : 0;
        }
#pragma unroll
        for (int v = 0; v < U; ++v) kk[v] = ld(start + kk[v]);
#pragma unroll
        for (int v = 0; v < U; ++v) {
            const int64_t p = b + 256 * v;
            if (p < n) perm[(int64_t)kk[v] + rr[v]] = (int32_t)p;
        }
    }
}

constexpr int kPlace3 = 4;   // particles a thread
template <typename T>
__global__ void __launch_bounds__(256)
k_place3(PRecords<T> src, PArrays<T> dst, T* __restrict__ dfz, const int32_t* __restrict__ perm, int64_t n)
{
    constexpr int U = kPlace3;
    for (int64_t b = (int64_t)blockIdx.x * (256 * U) + threadIdx.x; b < n; b += (int64_t)gridDim.x * (256 * U)) {
        int p[U];
#pragma unroll
        for (int v = 0; v < U; ++v) p[v] = b + 256 * v < n ? ld(perm + b + 256 * v) : 0;
        PRecA<T> ra[U];
        PRecB<T> rb[U];
        T rz[U];
        int ri[U];
#pragma unroll
        for (int v = 0; v < U; ++v) {
            ra[v] = src.a[p[v]];
            rb[v] = src.b[p[v]];
            rz[v] = dfz ? src.fz[p[v]] : T(0);   // (no third offset for 2D particles)
            ri[v] = src.id ? src.id[p[v]] : 0;
        }
#pragma unroll
        for (int v = 0; v < U; ++v) {
            const int64_t q = b + 256 * v;
            if (q >= n) continue;
            dst.fx[q] = ra[v].fx;
            dst.fy[q] = ra[v].fy;
            dst.ux[q] = ra[v].ux;
            dst.uy[q] = ra[v].uy;
            dst.uz[q] = rb[v].uz;
            dst.w[q] = rb[v].w;
            if (dfz) dfz[q] = rz[v];
            if (dst.id) dst.id[q] = ri[v];
        }
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

template <typename T>
static int tiles3(const GridP& g)
{
    using O = Op3<T>;
    return ((g.nx + O::X - 1) / O::X) * ((g.ny + O::Y - 1) / O::Y) * ((g.nz + O::Z - 1) / O::Z);
}
int op_blocks3(GridP g, int precision) { return precision == 32 ? tiles3<float>(g) : tiles3<double>(g); }

template <typename T, int MODE, bool TR>
cudaError_t launch_op3(const T* M, const double* in, double sc, const double* b, double* out, double* vj,
                       const double* V, int64_t ldv, int nv, GridP g, double* partial, cudaStream_t st,
                       const GmDyn* dyn)
{
    const int smem = (int)sizeof(typename Op3<T>::Shared);
    const cudaError_t e = cudaFuncSetAttribute(k_op3<T, MODE, TR>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    count_launches(1);
    k_op3<T, MODE, TR><<<tiles3<T>(g), Op3<T>::share * Op3<T>::nodes, smem, st>>>(M, in, sc, b, out, vj, V, ldv, nv, g, partial, dyn);
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
    const int smem = (int)sizeof(typename Op3<T>::Shared);
    const cudaError_t e = cudaFuncSetAttribute(k_field_update3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    count_launches(1);
    k_field_update3<T><<<nblocks, Op3<T>::nodes, smem, st>>>(x, M, J, Eth, E, B0, B1, g, partial);
    return cudaGetLastError();
}

int push_blocks3(GridP g, int cap)
{
    const int uw = unit_width3(g);
    const int64_t units = (int64_t)((g.nx + uw - 1) / uw) * g.ny * g.nz;
    return (int)grid3(units, PushCfg3<float>::warps, cap > 0 ? cap : 152 * 16);
}

template <typename T>
cudaError_t push3(PArrays<T> src, const T* sfz, PRecords<T> dst, const int32_t* start, int32_t* key, int32_t* rank,
                  int32_t* count, const T* Eth, const T* B, GridP g, SpeciesConst sc, double* lsum, int nblocks,
                  cudaStream_t st)
{
    count_launches(1);
    k_push3<T><<<nblocks, 32 * PushCfg3<T>::warps, 0, st>>>(src, sfz, dst, start, key, rank, count, Eth, B, g,
                                                       (T)(sc.q * g.dt / (2.0 * sc.m)), (T)(sc.q * g.dt), (T)sc.m,
                                                       lsum, unit_width3(g));
    return cudaGetLastError();
}

template <typename T>
cudaError_t place3(PRecords<T> src, PArrays<T> dst, T* dfz, const int32_t* key, const int32_t* rank,
                   const int32_t* start, int32_t* perm, int64_t n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    count_launches(2);
    k_places<<<grid3(n, 256 * 4, 152 * 32), 256, 0, st>>>(key, rank, start, perm, n);
    k_place3<T><<<grid3(n, 256 * kPlace3, 152 * 32), 256, 0, st>>>(src, dst, dfz, perm, n);
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
    template cudaError_t push3<T>(PArrays<T>, const T*, PRecords<T>, const int32_t*, int32_t*, int32_t*, int32_t*, \
                                  const T*, const T*, GridP, SpeciesConst, double*, int, cudaStream_t);            \
    template cudaError_t place3<T>(PRecords<T>, PArrays<T>, T*, const int32_t*, const int32_t*, const int32_t*,    \
                                   int32_t*, int64_t, cudaStream_t);                                               \
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
