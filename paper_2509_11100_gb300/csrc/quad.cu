// quad.cu -- the 2D step with quadratic (triangular-shaped-cloud) shape
// functions, the higher-order variant of the linear shape of the other 2D
// kernels (same scheme, Sec. 2). Along each axis a particle at lattice
// coordinate s touches the nearest node n = floor(s + 1/2) and its two
// neighbours with weights 1/2 (1/2 - d)^2, 3/4 - d^2, 1/2 (1/2 + d)^2,
// d = s - n. In cell i with offset f that is nodes i-1 .. i+1 (f < 1/2, d =
// f) or i .. i+2 (f >= 1/2, d = f - 1); B on the centre lattice is gathered
// from centres i-1 .. i+1 with d = f - 1/2, whatever f. Node pairs of a
// particle lie up to two cells apart: 25 offsets, 13 stored per node in the
// order (0,0), (1,0), (2,0), (di,1) for di = -2..2, (di,2) for di = -2..2
// (a stored block serves both orders of its pair).
//
// Kernels:
//   k_deposit_q   warp per row segment of cells, the segment's B staged in
//                 shared memory; per cell the particles of all species staged
//                 in four groups by the half of the cell they sit in (each
//                 group touches a fixed 3 x 3 of the cell's 4 x 4 nodes), the
//                 lanes sum the groups' 36 weight products; a ring of four
//                 node columns in shared memory collects the cells' sums
//   k_op_q        the operator on 32 x 4-node tiles, the tile's mass-matrix
//                 rows and the input on a 2-node halo in shared memory, the
//                 modes and partial dot products of the other operators
//   k_field_update_q   the field update and the ledger terms on the same tiles
//   k_push_q      warp per row segment with E and B tiles, the push, the new
//                 cell and its slot for the counting sort (k_places, k_place3)
#include "launch.cuh"
#include "opcore.cuh"

namespace relsim {
namespace {

constexpr int kQX = 32;   // cells per row segment

unsigned gridq(int64_t n, int threads, int64_t cap)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > cap) b = cap;
    return (unsigned)(b > 0 ? b : 1);
}

// the stored index of offset (di, dj), or -1 when (-di, -dj) is stored
__host__ __device__ __forceinline__ int halfq(int di, int dj)
{
    if (dj == 2) return 8 + di + 2;
    if (dj == 1) return 3 + di + 2;
    if (dj == 0 && di >= 0) return di;
    return -1;
}

__device__ __forceinline__ void halfq_offset(int h, int& di, int& dj)
{
    if (h < 3) { di = h; dj = 0; }
    else if (h < 8) { di = h - 5; dj = 1; }
    else { di = h - 10; dj = 2; }
}

// the three weights of a particle along one axis (d in [-1/2, 1/2))
template <typename T>
__device__ __forceinline__ void quad3(T d, T (&w)[3])
{
    const T a = T(0.5) - d, b = T(0.5) + d;
    w[0] = T(0.5) * a * a;
    w[1] = T(0.75) - d * d;
    w[2] = T(0.5) * b * b;
}

// field tiles of a row segment (cells i0 .. i0+cn-1 of row j)
template <typename T>
struct TileBq {
    T B[3][3][kQX + 2];   // centre (i0 - 1 + c, j - 1 + r)
};
template <typename T>
struct TileQ : TileBq<T> {
    T E[3][4][kQX + 3];   // node (i0 - 1 + c, j - 1 + r)
};

template <typename T>
__device__ __forceinline__ void load_tileBq(TileBq<T>& tl, const T* __restrict__ B, int i0, int cn, int j,
                                            const GridP& g, int lane)
{
    const int nc = g.ncell;
    for (int q = lane; q < 3 * 3 * (kQX + 2); q += 32) {
        const int c = q % (kQX + 2), r = (q / (kQX + 2)) % 3, comp = q / (3 * (kQX + 2));
        if (c <= cn + 1)
            tl.B[comp][r][c] = ld(B + comp * nc + wrap1(j - 1 + r, g.ny) * g.nx + wrap1(i0 - 1 + c, g.nx));
    }
    __syncwarp();
}

template <typename T>
__device__ __forceinline__ void load_tileq(TileQ<T>& tl, const T* __restrict__ E, const T* __restrict__ B, int i0,
                                           int cn, int j, const GridP& g, int lane)
{
    const int nc = g.ncell;
    for (int q = lane; q < 3 * 4 * (kQX + 3); q += 32) {
            const int c = q % (kQX + 3), r = (q / (kQX + 3)) % 4, comp = q / (4 * (kQX + 3));
            if (c <= cn + 2)
                tl.E[comp][r][c] = ld(E + comp * nc + wrap1(j - 1 + r, g.ny) * g.nx + wrap1(i0 - 1 + c, g.nx));
        }
    load_tileBq<T>(tl, B, i0, cn, j, g, lane);
}

// B^n at a particle of local cell cl: centres cl-1 .. cl+1 (tile columns
// cl .. cl+2), rows j-1 .. j+1
template <typename T>
__device__ __forceinline__ void tile_Bq(const T (&B)[3][3][kQX + 2], int cl, T fx, T fy, T (&Bp)[3])
{
    T wx[3], wy[3];
    quad3(fx - T(0.5), wx);
    quad3(fy - T(0.5), wy);
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
        T b = T(0);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            T br = T(0);
#pragma unroll
            for (int c = 0; c < 3; ++c) br += wx[c] * B[comp][r][cl + c];
            b += wy[r] * br;
        }
        Bp[comp] = b;
    }
}

template <typename T>
__device__ __forceinline__ void alphaq(const T (&Bp)[3], T bg, T (&al)[9])   // bg = beta/gbar
{
    const T ax = bg * Bp[0], ay = bg * Bp[1], az = bg * Bp[2];
    const T ia = T(1) / (T(1) + ax * ax + ay * ay + az * az);
    al[0] = (T(1) + ax * ax) * ia; al[1] = (ax * ay + az) * ia; al[2] = (ax * az - ay) * ia;
    al[3] = (ax * ay - az) * ia; al[4] = (T(1) + ay * ay) * ia; al[5] = (ay * az + ax) * ia;
    al[6] = (ax * az + ay) * ia; al[7] = (ay * az - ax) * ia; al[8] = (T(1) + az * az) * ia;
}

// ---------------------------------------------------------------------------
// deposit

// A warp takes a row segment of cells; a cell's particles are staged 32 at a
// time, grouped by the half of the cell they sit in along x and y (hx, hy):
// a group touches the same 3 x 3 frame of the cell's 4 x 4 nodes. Along an
// axis the frame's node pairs have six weight products, so a particle adds
// c alpha_e to 36 products; 27 lanes each sum 2 x 2 of them for one row of
// alpha (4 products x 3 entries, two products per paired FP32 FMA), per
// group in registers over the cell. A cell's sums then go to the union's
// products in shared memory, held by the column of their left node in a ring
// of four columns: the next cell's union is this one's moved by a column, so
// only the column that falls out is added to M, its 37 blocks in address
// order (the sums of the others grow on).
//
// Bound by shared memory (FP32: 81% of its cycles when a particle's 36 values
// were stored 4 bytes at a time, two particles side by side: 1.25 ms on
// 512x256 with 128 particles a cell). A particle is staged in nine 16-byte
// pieces and a batch's particles are loaded while the batch before is added
// up: 1.02 ms (1.12 without the early loads; at five blocks an SM the spills
// make it 1.6). With each lane owning node pairs (45 a group, 106 a cell) and
// all 106 blocks of every cell added to M it took 1.85.
template <typename T>
struct DepCfgQ {
    static constexpr int warps = sizeof(T) == 4 ? 4 : 2;   // static shared memory below 48 KB
    static constexpr int blocks = 4;                       // an SM
};

// staged values of a particle: the six x and six y products, c alpha (rows of
// four, FP32 with the current's component as the fourth), the frame's nine
// weights, FP64 the current
enum { kQXX = 0, kQYY = 6, kQE = 12, kQW = 24, kQV = 33, kQRow = 38 };
template <typename T>
struct StageQ {
    T v[32][kQRow];
    __device__ __forceinline__ void put(int row, const T (&xx)[6], const T (&yy)[6], const T (&ca)[9], const T (&W)[9],
                                        const T (&cu)[3])
    {
        T* r = v[row];
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            r[kQXX + e] = xx[e];
            r[kQYY + e] = yy[e];
        }
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            r[kQE + 4 * (e / 3) + e % 3] = ca[e];
            r[kQW + e] = W[e];
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) r[kQV + e] = cu[e];
    }
};
template <>
struct StageQ<float> {
    float4 v[32][9];   // (an odd number of 16-byte pieces: rows start on different banks)
    __device__ __forceinline__ void put(int row, const float (&xx)[6], const float (&yy)[6], const float (&ca)[9],
                                        const float (&W)[9], const float (&cu)[3])
    {
        float4* r = v[row];
        r[0] = make_float4(xx[0], xx[1], xx[2], xx[3]);
        r[1] = make_float4(xx[4], xx[5], yy[0], yy[1]);
        r[2] = make_float4(yy[2], yy[3], yy[4], yy[5]);
#pragma unroll
        for (int e = 0; e < 3; ++e) r[3 + e] = make_float4(ca[3 * e], ca[3 * e + 1], ca[3 * e + 2], cu[e]);
        r[6] = make_float4(W[0], W[1], W[2], W[3]);
        r[7] = make_float4(W[4], W[5], W[6], W[7]);
        reinterpret_cast<float*>(r + 8)[0] = W[8];
    }
};

// a lane's sums over staged particles: product (x type 2 xg + (q & 1), y type
// 2 yg + (q >> 1)), entry e of its row of alpha, and its current
template <typename T>
struct SumQ {
    T a[12], j;
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int e = 0; e < 12; ++e) a[e] = T(0);
        j = T(0);
    }
    __device__ __forceinline__ void add(const StageQ<T>& st, int row, int xg, int yg, int er, int jf)
    {
        const T* r = st.v[row];
        const T x0 = r[kQXX + 2 * xg], x1 = r[kQXX + 2 * xg + 1], y0 = r[kQYY + 2 * yg], y1 = r[kQYY + 2 * yg + 1];
        const T w[4] = {x0 * y0, x1 * y0, x0 * y1, x1 * y1};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int e = 0; e < 3; ++e) a[3 * q + e] += w[q] * r[kQE + 4 * er + e];
        j += r[kQW + jf] * r[kQV + er];
    }
    __device__ __forceinline__ T value(int q, int e) const { return a[3 * q + e]; }
};
template <>
struct SumQ<float> {
    float2 a[2][3];   // [y type][entry], both x types
    float j;
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int y = 0; y < 2; ++y)
#pragma unroll
            for (int e = 0; e < 3; ++e) a[y][e] = make_float2(0.f, 0.f);
        j = 0.f;
    }
    __device__ __forceinline__ void add(const StageQ<float>& st, int row, int xg, int yg, int er, int jf)
    {
        const float* r = reinterpret_cast<const float*>(st.v[row]);
        const float2 x = *reinterpret_cast<const float2*>(r + kQXX + 2 * xg);
        const float2 y = *reinterpret_cast<const float2*>(r + kQYY + 2 * yg);
        const float4 e = *reinterpret_cast<const float4*>(r + kQE + 4 * er);
        const float2 w0 = make_float2(x.x * y.x, x.y * y.x), w1 = make_float2(x.x * y.y, x.y * y.y);
        const float2 e0 = make_float2(e.x, e.x), e1 = make_float2(e.y, e.y), e2 = make_float2(e.z, e.z);
        a[0][0] = __ffma2_rn(w0, e0, a[0][0]);
        a[0][1] = __ffma2_rn(w0, e1, a[0][1]);
        a[0][2] = __ffma2_rn(w0, e2, a[0][2]);
        a[1][0] = __ffma2_rn(w1, e0, a[1][0]);
        a[1][1] = __ffma2_rn(w1, e1, a[1][1]);
        a[1][2] = __ffma2_rn(w1, e2, a[1][2]);
        j += r[kQW + jf] * e.w;
    }
    __device__ __forceinline__ float value(int q, int e) const { return (q & 1) ? a[q >> 1][e].y : a[q >> 1][e].x; }
};

// the union's products: [column of the left node, a ring of four][dx][row c,
// dy: 3 c + dy][entry]
constexpr int kUY = 90;                 // values of one (column, dx)
constexpr int kUCol = 3 * kUY;          // and of a column
constexpr int kItemsQ = 37 * 9;         // additions to M of a column

// block q (0 .. 36) that holds a column's products: the node it is stored at
// (col columns right of the left node, union row), its offset index and the
// product's place (dx, 3 c + dy)
__device__ __forceinline__ void column_block(int q, int& col, int& row, int& hs, int& dx, int& yt)
{
    int n = 0;
    col = row = hs = dx = yt = 0;
    for (int x = 0; x < 3; ++x)
        for (int c = 0; c < 4; ++c)
            for (int dy = 0; dy < 3 && c + dy < 4; ++dy)
                for (int way = 0; way < (x > 0 && dy > 0 ? 2 : 1); ++way) {
                    // way 0: nodes (0, c) and (x, c + dy); 1: (x, c) and (0, c + dy)
                    if (n++ != q) continue;
                    col = way ? x : 0;
                    row = c;
                    hs = halfq(way ? -x : x, dy);
                    dx = x;
                    yt = 3 * c + dy;
                }
}

template <typename T>
__global__ void __launch_bounds__(32 * DepCfgQ<T>::warps, DepCfgQ<T>::blocks)
k_deposit_q(const __grid_constant__ DepositSpecies<T> ds, const T* __restrict__ B, T* __restrict__ M,
            T* __restrict__ J, GridP g, int uw)
{
    constexpr int kW = DepCfgQ<T>::warps;
    __shared__ __align__(16) StageQ<T> sst[kW];
    __shared__ T sum_[kW][4 * kUCol];
    __shared__ T sumj[kW][4][12];       // currents: [column][3 row + component]
    __shared__ TileBq<T> stl[kW];
    __shared__ int snode[kW][12];       // nodes (col, row) of a column's additions
    __shared__ unsigned item[kItemsQ];  // node << 20 | place in its blocks << 10 | value in the column
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < 37; q += blockDim.x) {
        int col, row, hs, dx, yt, rank = 0;
        column_block(q, col, row, hs, dx, yt);
        for (int o = 0; o < 37; ++o) {
            int c2, r2, h2, d2, y2;
            column_block(o, c2, r2, h2, d2, y2);
            rank += (c2 * 4 + r2) * kHalfQ + h2 < (col * 4 + row) * kHalfQ + hs ? 1 : 0;
        }
        for (int e = 0; e < 9; ++e)
            item[rank * 9 + e] = (unsigned)(col * 4 + row) << 20 | (unsigned)(hs * 9 + e) << 10 |
                                 (unsigned)(dx * kUY + yt * 9 + e);
    }
    for (int q = lane; q < 4 * kUCol; q += 32) sum_[wib][q] = T(0);
    for (int q = lane; q < 48; q += 32) (&sumj[wib][0][0])[q] = T(0);
    __syncthreads();
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int nseg = (g.nx + uw - 1) / uw;
    const int nunits = nseg * g.ny;
    StageQ<T>& st = sst[wib];
    T* const U = sum_[wib];
    // this lane's products (x types 2 xg, 2 xg + 1, y types 2 yg, 2 yg + 1),
    // row of alpha, and current (frame node, component)
    const bool own = lane < 27;
    const int er = own ? lane % 3 : 0, yg = own ? lane / 3 % 3 : 0, xg = own ? lane / 9 : 0;
    const int jf = own ? lane / 3 : 0, jc = own ? lane % 3 : 0;
    // pair type t of the frame's axis: its lower node and the distance
    auto low_of = [](int t) { return t < 3 ? 0 : (t < 5 ? 1 : 2); };
    auto dist_of = [](int t) { return t < 3 ? t : (t < 5 ? t - 3 : 0); };
    const int xl[2] = {low_of(2 * xg), low_of(2 * xg + 1)}, xd[2] = {dist_of(2 * xg), dist_of(2 * xg + 1)};
    const int yo[2] = {(3 * low_of(2 * yg) + dist_of(2 * yg)) * 9 + 3 * er,
                       (3 * low_of(2 * yg + 1) + dist_of(2 * yg + 1)) * 9 + 3 * er};
    for (int u = warp; u < nunits; u += nwarps) {
        const int i0 = (u % nseg) * uw, j = u / nseg;
        const int cn = min(uw, g.nx - i0);
        __syncwarp();
        load_tileBq<T>(stl[wib], B, i0, cn, j, g, lane);
        int live = 0;   // columns of the ring that hold sums
        for (int cl = 0; cl < cn + 3; ++cl) {   // the last three: only the columns left over
            const int i = i0 + cl;
            int cum[kMaxSpecies + 1], pst[kMaxSpecies];
            cum[0] = 0;
#pragma unroll
            for (int s = 0; s < kMaxSpecies; ++s) {
                pst[s] = 0;
                cum[s + 1] = cum[s];
                if (cl < cn && s < ds.nsp) {
                    pst[s] = ds.start[s][j * g.nx + i];
                    cum[s + 1] += ds.start[s][j * g.nx + i + 1] - pst[s];
                }
            }
            const int total = cum[kMaxSpecies];
            if (total > 0) {
                T acc[4][12], accj[4];   // per group
#pragma unroll
                for (int gq = 0; gq < 4; ++gq) {
                    accj[gq] = T(0);
#pragma unroll
                    for (int e = 0; e < 12; ++e) acc[gq][e] = T(0);
                }
                // a batch's particles are loaded while the batch before is added up
                int ns = 0;
                T nfx = T(0), nfy = T(0), nux = T(0), nuy = T(0), nuz = T(0), nwt = T(0);
                auto fetch = [&](int t) {
                    if (t >= total) return;
                    int s = 0, p = pst[0] + t;
#pragma unroll
                    for (int q = 1; q < kMaxSpecies; ++q)
                        if (t >= cum[q] && cum[q + 1] > cum[q]) {
                            s = q;
                            p = pst[q] + (t - cum[q]);
                        }
                    ns = s;
                    nfx = ld(ds.fx[s] + p);
                    nfy = ld(ds.fy[s] + p);
                    nux = ld(ds.ux[s] + p);
                    nuy = ld(ds.uy[s] + p);
                    nuz = ld(ds.uz[s] + p);
                    nwt = ld(ds.w[s] + p);
                };
                fetch(lane);
                for (int q0 = 0; q0 < total; q0 += 32) {
                    const int t = q0 + lane, s = ns;
                    const bool act = t < total;
                    const T fx = nfx, fy = nfy, ux = nux, uy = nuy, uz = nuz, wt = nwt;
                    fetch(t + 32);
                    const int hx = fx >= T(0.5), hy = fy >= T(0.5);
                    const int grp = act ? 2 * hy + hx : -1;
                    // rows of the groups, and this particle's place
                    int gr[5], row = 0;
                    gr[0] = 0;
#pragma unroll
                    for (int gq = 0; gq < 4; ++gq) {
                        const unsigned bal = __ballot_sync(0xffffffffu, grp == gq);
                        gr[gq + 1] = gr[gq] + __popc(bal);
                        if (grp == gq) row = gr[gq] + __popc(bal & ((1u << lane) - 1u));
                    }
                    if (act) {
                        T wx[3], wy[3], Bp[3], al[9];
                        quad3(hx ? fx - T(1) : fx, wx);
                        quad3(hy ? fy - T(1) : fy, wy);
                        tile_Bq(stl[wib].B, cl, fx, fy, Bp);
                        const T ig = T(1) / sqrt(T(1) + ux * ux + uy * uy + uz * uz);
                        alphaq(Bp, ds.beta[s] * ig, al);
                        const T cM = wt * ds.cM[s] * ig, cJ = wt * ds.cJ[s] * ig;
                        T xx[6], yy[6], W[9], cu[3];
                        int n = 0;
#pragma unroll
                        for (int a = 0; a < 3; ++a)
#pragma unroll
                            for (int b2 = a; b2 < 3; ++b2) {
                                xx[n] = wx[a] * wx[b2];
                                yy[n] = wy[a] * wy[b2];
                                ++n;
                            }
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
#pragma unroll
                            for (int c2 = 0; c2 < 3; ++c2) W[3 * r + c2] = wy[r] * wx[c2];
                            cu[r] = cJ * (al[3 * r] * ux + al[3 * r + 1] * uy + al[3 * r + 2] * uz);
                        }
#pragma unroll
                        for (int e = 0; e < 9; ++e) al[e] *= cM;
                        st.put(row, xx, yy, al, W, cu);
                    }
                    __syncwarp();
#pragma unroll
                    for (int gq = 0; gq < 4; ++gq) {
                        if (gr[gq + 1] == gr[gq]) continue;   // warp-uniform
                        SumQ<T> a;
                        a.clear();
                        #pragma unroll 2
                        for (int r = gr[gq]; r < gr[gq + 1]; ++r) a.add(st, r, xg, yg, er, jf);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
#pragma unroll
                            for (int e = 0; e < 3; ++e) acc[gq][3 * q + e] += a.value(q, e);
                        accj[gq] += a.j;
                    }
                    __syncwarp();
                }
                // the cell's sums into the union's products (distinct entries
                // per lane within a group)
#pragma unroll
                for (int gq = 0; gq < 4; ++gq) {
                    const int hx = gq & 1, hy = gq >> 1;
                    if (own) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            T* const o = U + ((cl + xl[q & 1] + hx) & 3) * kUCol + xd[q & 1] * kUY + yo[q >> 1] + 27 * hy;
#pragma unroll
                            for (int e = 0; e < 3; ++e) o[e] += acc[gq][3 * q + e];
                        }
                        sumj[wib][(cl + jf % 3 + hx) & 3][3 * (jf / 3 + hy) + jc] += accj[gq];
                    }
                    __syncwarp();   // another lane may own these entries in the next group
                }
                live = 4;
            }
            // the column of nodes i - 1 is complete
            if (live > 0) {
                if (lane < 12) snode[wib][lane] = column_node_q(i, j, lane, g.nx, g.ny);
                __syncwarp();
                T* const C = U + (cl & 3) * kUCol;
                for (int it = lane; it < kItemsQ; it += 32) {
                    const unsigned q = item[it];
                    atomicAdd(M + (int64_t)snode[wib][q >> 20] * kMBlockQ + ((q >> 10) & 1023u), C[q & 1023u]);
                }
                if (lane < 12) {
                    T& vj = sumj[wib][cl & 3][lane];
                    atomicAdd(J + (int64_t)(lane % 3) * g.ncell + snode[wib][lane / 3], vj);
                    vj = T(0);
                }
                __syncwarp();
                for (int q = lane; q < kUCol; q += 32) C[q] = T(0);
                __syncwarp();
                --live;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// the operator and the field update

enum { kqA = 0, kqResidual = 1, kqArnoldi = 2 };
constexpr int kOpChunkq = 8;

// The operator's tiles: 32 x 4 nodes (FP64: 32 x 2), one thread a node. The
// tile's own mass-matrix rows (15 KB a row in FP32) come into shared memory
// by asynchronous copies while the input is staged; read straight from global
// memory (468 bytes from lane to lane) every load of a block touched 32
// lines: 48 us an application on 512x256 (FP32 form).
template <typename T>
struct OpQ {
    static constexpr int X = 32, Y = sizeof(T) == 4 ? 4 : 2, threads = X * Y;
    struct Shared {
        T Mm[Y][X * kMBlockQ];          // own blocks
        T v[3][Y + 4][X + 4];           // the input on the 2-node halo
        T C[3][Y + 1][X + 1];           // its curl on the centres around the tile's nodes
    };
    static_assert(sizeof(Shared) >= sizeof(double) * kOpChunkq * threads, "the dot products reuse it");
};
// a block's tile and this thread's node
template <typename T>
struct AtQ {
    int i0, j0, tw, th, tx, ty, i, j;
    bool active;
    int64_t gidx;
    __device__ __forceinline__ explicit AtQ(const GridP& g)
    {
        using O = OpQ<T>;
        const int nx = (g.nx + O::X - 1) / O::X;
        i0 = (blockIdx.x % nx) * O::X;
        j0 = (blockIdx.x / nx) * O::Y;
        tw = min(O::X, g.nx - i0);
        th = min(O::Y, g.ny - j0);
        tx = threadIdx.x % O::X;
        ty = threadIdx.x / O::X;
        i = i0 + tx;
        j = j0 + ty;
        active = tx < tw && ty < th;
        gidx = active ? (int64_t)j * g.nx + i : 0;
    }
};

// start the copies of the tile's mass-matrix rows (16 bytes each where the
// rows are aligned to that, else 4)
template <typename T>
__device__ __forceinline__ void fetch_rowsq(typename OpQ<T>::Shared& S, const T* __restrict__ M, const AtQ<T>& t,
                                            const GridP& g)
{
    using O = OpQ<T>;
    const bool wide = ((int64_t)g.nx * kMBlockQ * sizeof(T)) % 16 == 0;
    const int n = t.tw * kMBlockQ * (int)sizeof(T) / (wide ? 16 : 4);
#pragma unroll
    for (int y = 0; y < O::Y; ++y) {
        if (y >= t.th) continue;
        const char* src = reinterpret_cast<const char*>(M + ((int64_t)(t.j0 + y) * g.nx + t.i0) * kMBlockQ);
        char* dst = reinterpret_cast<char*>(&S.Mm[y][0]);
        if (wide)
            for (int q = threadIdx.x; q < n; q += O::threads) cp_async16(dst + 16 * q, src + 16 * q);
        else
            for (int q = threadIdx.x; q < n; q += O::threads) cp_async4(dst + 4 * q, src + 4 * q);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// the input (FP64) on the tile's halo in T, times s, and its curl on the
// centres around the tile's nodes (each formed once); the rows' copies land
template <typename T, bool SCALED>
__device__ __forceinline__ void stage_inputq(typename OpQ<T>::Shared& S, const double* __restrict__ in, T s,
                                             const AtQ<T>& t, const GridP& g)
{
    using O = OpQ<T>;
    constexpr int HX = O::X + 4, HY = O::Y + 4;
    const int64_t nc = g.ncell;
    const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
    // a lane a column, the last four by four lanes; positions past the tile's
    // last used column or row are clamped (unused); four rows in flight
    const int ga = wrap1(min(t.i0 - 2 + lane, 2 * g.nx - 1), g.nx), gb = wrap1(min(t.i0 + 30 + lane, 2 * g.nx - 1), g.nx);
    constexpr int rows = 3 * HY, W = O::threads / 32;
    for (int r0 = wid; r0 < rows; r0 += 4 * W) {
        double a[4], b[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = min(r0 + v * W, rows - 1), comp = r / HY, yy = r % HY;
            const int gj = wrap1(min(t.j0 - 2 + yy, 2 * g.ny - 1), g.ny);
            const double* row = in + comp * nc + (int64_t)gj * g.nx;
            a[v] = __ldg(row + ga);
            b[v] = lane < 4 ? __ldg(row + gb) : 0.0;
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = r0 + v * W;
            if (r >= rows) break;
            T* o = &S.v[0][0][0] + r * HX;
            T x = narrow<T>(a[v]);
            if (SCALED) x *= s;
            o[lane] = x;
            if (lane < 4) {
                T y = narrow<T>(b[v]);
                if (SCALED) y *= s;
                o[32 + lane] = y;
            }
        }
    }
    __syncthreads();
    const T rx = gc<T>(g).hdx, ry = gc<T>(g).hdy;
    for (int q = threadIdx.x; q < (O::Y + 1) * (O::X + 1); q += O::threads) {
        const int c = q % (O::X + 1), y = q / (O::X + 1);
        T C[3];
        op_curl_c<T>([&](int comp, int p, int o) { return S.v[comp][y + 1 + o][c + 1 + p]; }, rx, ry, C);
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) S.C[comp][y][c] = C[comp];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// (M v) at the thread's node: its own 13 stored blocks times v at g + d(h),
// the 12 neighbours' blocks M[g - d(h)][h] times v at g - d(h) (from the tile
// where they lie in it, else from global memory); with TR each block
// transposed
template <typename T, bool TR>
__device__ __forceinline__ void mv_q(const typename OpQ<T>::Shared& S, const T* __restrict__ M, const AtQ<T>& t,
                                     const GridP& g, T (&out)[3])
{
    T r[3] = {T(0), T(0), T(0)};
    const T* Mg = &S.Mm[t.ty][t.tx * kMBlockQ];
    auto add = [&](const T* m, int di, int dj) {
        T vv[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) vv[s] = S.v[s][t.ty + 2 + dj][t.tx + 2 + di];
#pragma unroll
        for (int rr = 0; rr < 3; ++rr)
#pragma unroll
            for (int s = 0; s < 3; ++s) r[rr] += m[TR ? s * 3 + rr : rr * 3 + s] * vv[s];
    };
    auto neighbour = [&](int h, T (&m)[9]) {
        int di, dj;
        halfq_offset(h, di, dj);
        const int x = t.tx - di, y = t.ty - dj;
        const T* Mn = x >= 0 && x < t.tw && y >= 0
                          ? &S.Mm[y][x * kMBlockQ]
                          : M + ((int64_t)wrap1(t.j - dj, g.ny) * g.nx + wrap1(t.i - di, g.nx)) * kMBlockQ;
#pragma unroll
        for (int e = 0; e < 9; ++e) m[e] = Mn[h * 9 + e];
    };
    // the neighbours' blocks five at a time (h = 3..7, 8..12), each five on
    // their way while the blocks before them are added
    T nb[2][5][9];
#pragma unroll
    for (int q = 0; q < 5; ++q) neighbour(3 + q, nb[0][q]);
#pragma unroll
    for (int h = 0; h < kHalfQ; ++h) {
        int di, dj;
        halfq_offset(h, di, dj);
        add(Mg + h * 9, di, dj);
    }
#pragma unroll
    for (int n = 0; n < 2; ++n) {
#pragma unroll
        for (int q = 0; q < 5; ++q)
            if (n == 0) neighbour(8 + q, nb[1][q]);
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            int di, dj;
            halfq_offset(3 + 5 * n + q, di, dj);
            add(nb[n][q], -di, -dj);
        }
    }
#pragma unroll
    for (int h = 1; h < 3; ++h) {
        T m[9];
        neighbour(h, m);
        add(m, -h, 0);
    }
    out[0] = r[0];
    out[1] = r[1];
    out[2] = r[2];
}

template <typename T, int MODE, bool TR>
__global__ void __launch_bounds__(OpQ<T>::threads, 3)
k_op_q(const T* __restrict__ M, const double* __restrict__ in, double s, const double* __restrict__ b,
       double* __restrict__ out, double* __restrict__ vj, const double* __restrict__ V, int64_t ldv, int nv, GridP g,
       double* __restrict__ partial, const GmDyn* __restrict__ dyn)
{
    if (MODE == kqArnoldi && dyn) {
        if (!dyn->live) return;
        in = dyn->in;
        s = dyn->s;
        vj = dyn->vj;
        out = dyn->out;
        nv = dyn->nv;
    }
    using O = OpQ<T>;
    extern __shared__ __align__(128) unsigned char opq_smem[];
    typename O::Shared& S = *reinterpret_cast<typename O::Shared*>(opq_smem);
    const AtQ<T> t(g);
    const int64_t nc = g.ncell;
    const int tid = threadIdx.x;
    fetch_rowsq<T>(S, M, t, g);
    double own[3] = {0.0, 0.0, 0.0}, wv[3] = {0.0, 0.0, 0.0};
    if (t.active) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            own[c] = __ldg(in + c * nc + t.gidx);
            if (MODE == kqArnoldi && !is_one(s)) own[c] *= s;
        }
    }
    if (MODE == kqArnoldi) stage_inputq<T, true>(S, in, (T)s, t, g);
    else stage_inputq<T, false>(S, in, T(1), t, g);
    if (t.active) {
        T cc[3], mv[3];
        op_curl_n<T>([&](int comp, int p, int o) { return S.C[comp][t.ty + o][t.tx + p]; }, gc<T>(g).hdx, gc<T>(g).hdy,
                     cc);
        mv_q<T, TR>(S, M, t, g, mv);
        const T td = gc<T>(g).td;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double bv = widen(td * td * cc[c] + td * mv[c]);
            if (MODE == kqA) wv[c] = own[c] + bv;
            else if (MODE == kqResidual) wv[c] = b[c * nc + t.gidx] - (own[c] + bv);
            else wv[c] = bv;
            out[c * nc + t.gidx] = wv[c];
            if (MODE == kqArnoldi && vj) vj[c * nc + t.gidx] = own[c];
        }
    }
    if (MODE == kqA) return;
    const int nq = MODE == kqResidual ? 1 : nv + 2;
    const int lane = tid & 31, wid = tid >> 5;
    double* buf = reinterpret_cast<double*>(opq_smem);   // [kOpChunkq][threads]
    __syncthreads();   // the tile is no longer read
    for (int q0 = 0; q0 < nq; q0 += kOpChunkq) {
        const int kc = min(kOpChunkq, nq - q0);
        for (int c = 0; c < kc; ++c) {
            const int q = q0 + c;
            double d = 0.0;
            if (t.active) {
                if (MODE == kqResidual || q == nv + 1) d = wv[0] * wv[0] + wv[1] * wv[1] + wv[2] * wv[2];
                else if (q == nv) d = wv[0] * own[0] + wv[1] * own[1] + wv[2] * own[2];
                else {
                    const double* Vq = V + (int64_t)q * ldv + t.gidx;
                    d = wv[0] * __ldg(Vq) + wv[1] * __ldg(Vq + nc) + wv[2] * __ldg(Vq + 2 * nc);
                }
            }
            buf[c * O::threads + tid] = d;
        }
        __syncthreads();
        for (int c = wid; c < kc; c += O::threads / 32) {
            double sum = 0.0;
#pragma unroll
            for (int mm = 0; mm < O::threads / 32; ++mm) sum += buf[c * O::threads + mm * 32 + lane];
            sum = warp_sum(sum);
            if (lane == 0) partial[(int64_t)blockIdx.x * nq + q0 + c] = sum;
        }
        __syncthreads();
    }
}

constexpr int kFieldLedgerQ = 6;

// E^{n+theta} -> Eth, E^{n+1}, B^{n+1} of cell (i, j) and the ledger terms of
// the 2D field update, on the operator's tiles (term 5: the work dt dV
// (Jhat + M E^{n+theta}) . E^{n+theta})
template <typename T>
__global__ void __launch_bounds__(OpQ<T>::threads, 3)
k_field_update_q(const double* __restrict__ x, const T* __restrict__ M, const T* __restrict__ J, T* __restrict__ Eth,
                 T* __restrict__ E, const T* __restrict__ B0, T* __restrict__ B1, GridP g, double* __restrict__ partial)
{
    using O = OpQ<T>;
    extern __shared__ __align__(128) unsigned char opq_smem[];
    typename O::Shared& S = *reinterpret_cast<typename O::Shared*>(opq_smem);
    const AtQ<T> t(g);
    const int64_t nc = g.ncell;
    fetch_rowsq<T>(S, M, t, g);
    stage_inputq<T, false>(S, x, T(1), t, g);
    T acc[kFieldLedgerQ] = {T(0), T(0), T(0), T(0), T(0), T(0)};
    if (t.active) {
        const T th = gc<T>(g).theta, hdV = gc<T>(g).hdV, dt = gc<T>(g).dt;
        T mv[3], wk = T(0);
        mv_q<T, false>(S, M, t, g, mv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T et = S.v[c][t.ty + 2][t.tx + 2];
            const T e0 = E[c * nc + t.gidx];
            const T e1 = (et - (T(1) - th) * e0) / th;
            Eth[c * nc + t.gidx] = et;
            E[c * nc + t.gidx] = e1;
            acc[0] += hdV * (e1 - e0) * (e1 + e0);
            acc[2] += (e1 - e0) * (e1 - e0);
            acc[3] += hdV * e1 * e1;
            wk += (J[c * nc + t.gidx] + mv[c]) * et;
            // the cell's curl is that of the centre after the node's in x and y
            const T b0 = B0[c * nc + t.gidx];
            const T b1 = b0 - dt * S.C[c][t.ty + 1][t.tx + 1];
            B1[c * nc + t.gidx] = b1;
            acc[1] += hdV * (b1 - b0) * (b1 + b0);
            acc[2] += (b1 - b0) * (b1 - b0);
            acc[4] += hdV * b1 * b1;
        }
        acc[2] *= gc<T>(g).thdV;
        acc[5] = gc<T>(g).dtdV * wk;
    }
    double* red = reinterpret_cast<double*>(opq_smem);
    __syncthreads();   // the tile is no longer read
    double v[kFieldLedgerQ], o[kFieldLedgerQ];
#pragma unroll
    for (int q = 0; q < kFieldLedgerQ; ++q) v[q] = (double)acc[q];
    block_sum<kFieldLedgerQ>(v, red, o);
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < kFieldLedgerQ; ++q) partial[(int64_t)blockIdx.x * kFieldLedgerQ + q] = o[q];
}

// ---------------------------------------------------------------------------
// push

constexpr int kPushWarpsQ = 4;

template <typename T>
__global__ void __launch_bounds__(32 * kPushWarpsQ)
k_push_q(PArrays<T> src, PRecords<T> dst, const int32_t* __restrict__ start, int32_t* __restrict__ key,
         int32_t* __restrict__ rank, int32_t* __restrict__ count, const T* __restrict__ Eth, const T* __restrict__ B,
         GridP g, T beta, T qdt, T m, double* __restrict__ lsum, int uw)
{
    __shared__ int sst[kPushWarpsQ][kQX + 1];
    __shared__ TileQ<T> stl[kPushWarpsQ];
    __shared__ double red[32 * 4];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int nseg = (g.nx + uw - 1) / uw;
    const int nunits = nseg * g.ny;
    int* ss = sst[wib];
    const T dtx = gc<T>(g).dt * gc<T>(g).rdx, dty = gc<T>(g).dt * gc<T>(g).rdy;
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
    for (int u = warp; u < nunits; u += nwarps) {
        const int i0 = (u % nseg) * uw, j = u / nseg;
        const int cn = min(uw, g.nx - i0);
        const int c0 = j * g.nx + i0;
        __syncwarp();
        if (lane <= cn) ss[lane] = start[c0 + lane];
        if (lane == 0 && cn == kQX) ss[kQX] = start[c0 + kQX];
        load_tileq<T>(stl[wib], Eth, B, i0, cn, j, g, lane);
        const TileQ<T>& tl = stl[wib];
        const int P0 = ss[0], P1 = ss[cn];
        int cl = 0;
        // the next batch is loaded while this one is pushed
        T nfx = T(0), nfy = T(0), nux = T(0), nuy = T(0), nuz = T(0), nw = T(0);
        int nid = 0;
        auto fetch = [&](int q) {
            if (q < P1) {
                nfx = ld(src.fx + q);
                nfy = ld(src.fy + q);
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
            const T fx = nfx, fy = nfy, ux = nux, uy = nuy, uz = nuz, w = nw;
            const int pid = nid;
            fetch(p + 32);
            int newkey = -1 - lane;
            if (act) {
                while (ss[cl + 1] <= p) ++cl;
                // E from the particle's own 3 x 3 nodes of the cell's 4 x 4
                const int hx = fx >= T(0.5), hy = fy >= T(0.5);
                T wx[3], wy[3];
                quad3(hx ? fx - T(1) : fx, wx);
                quad3(hy ? fy - T(1) : fy, wy);
                T E[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    T e = T(0);
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        T er = T(0);
#pragma unroll
                        for (int cc = 0; cc < 3; ++cc) er += wx[cc] * tl.E[c][r + hy][cl + cc + hx];
                        e += wy[r] * er;
                    }
                    E[c] = e;
                }
                T Bp[3];
                tile_Bq(tl.B, cl, fx, fy, Bp);
                const T u02 = ux * ux + uy * uy + uz * uz;
                const T g0 = sqrt(T(1) + u02), ig0 = T(1) / g0;
                const T bg = beta * ig0, ax = bg * Bp[0], ay = bg * Bp[1], az = bg * Bp[2];
                const T sa = T(1) / (T(1) + ax * ax + ay * ay + az * az);
                const T wxv = ux + beta * E[0], wyv = uy + beta * E[1], wzv = uz + beta * E[2];
                const T wa = wxv * ax + wyv * ay + wzv * az;
                const T ubx = sa * (wxv + (wyv * az - wzv * ay) + wa * ax);
                const T uby = sa * (wyv + (wzv * ax - wxv * az) + wa * ay);
                const T ubz = sa * (wzv + (wxv * ay - wyv * ax) + wa * az);
                const T u1x = T(2) * ubx - ux, u1y = T(2) * uby - uy, u1z = T(2) * ubz - uz;
                const T u12 = u1x * u1x + u1y * u1y + u1z * u1z;
                const T g1 = sqrt(T(1) + u12), ig1 = T(1) / g1;
                const T t[2] = {fx + dtx * (u1x * ig1), fy + dty * (u1y * ig1)};
                const int nn[2] = {g.nx, g.ny}, cc0[2] = {i0 + cl, j};
                T fn[2];
                int cnew[2];
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const T fl = floor(t[a]);
                    int sh = (int)fl;
                    T f = t[a] - fl;
                    if (f >= T(1)) { f -= T(1); sh += 1; }
                    fn[a] = f;
                    int q = cc0[a] + sh;
                    if ((unsigned)q >= (unsigned)nn[a]) {   // across the box: any distance
                        q %= nn[a];
                        if (q < 0) q += nn[a];
                    }
                    cnew[a] = q;
                }
                dst.a[p] = PRecA<T>{fn[0], fn[1], u1x, u1y};
                dst.b[p] = PRecB<T>{u1z, w};
                if (dst.id) dst.id[p] = pid;
                newkey = cnew[1] * g.nx + cnew[0];
                key[p] = newkey;
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

}  // namespace

// the width of the row segments a warp takes: 32 cells, halved (to 8 at
// least: a segment adds three columns at its end) while that leaves fewer
// than eight warps per SM
static int unit_width_q(GridP g)
{
    int uw = kQX;
    while (uw > 8 && ((g.nx + uw - 1) / uw) * g.ny < 152 * 8) uw /= 2;
    return uw;
}

template <typename T>
cudaError_t deposit_q(const DepositSpecies<T>& ds, const T* B, T* M, T* J, GridP g, cudaStream_t st, int blocks)
{
    const int uw = unit_width_q(g);
    const int units = ((g.nx + uw - 1) / uw) * g.ny;
    count_launches(1);
    k_deposit_q<T><<<gridq(units, DepCfgQ<T>::warps, blocks > 0 ? blocks : 152 * 8), 32 * DepCfgQ<T>::warps, 0, st>>>(
        ds, B, M, J, g, uw);
    return cudaGetLastError();
}

template <typename T>
static int tiles_q(const GridP& g)
{
    using O = OpQ<T>;
    return ((g.nx + O::X - 1) / O::X) * ((g.ny + O::Y - 1) / O::Y);
}
int op_blocks_q(GridP g, int precision) { return precision == 32 ? tiles_q<float>(g) : tiles_q<double>(g); }

template <typename T, int MODE, bool TR>
cudaError_t launch_op_q(const T* M, const double* in, double sc, const double* b, double* out, double* vj,
                        const double* V, int64_t ldv, int nv, GridP g, double* partial, cudaStream_t st,
                        const GmDyn* dyn)
{
    const int smem = (int)sizeof(typename OpQ<T>::Shared);
    const cudaError_t e = cudaFuncSetAttribute(k_op_q<T, MODE, TR>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    count_launches(1);
    k_op_q<T, MODE, TR><<<tiles_q<T>(g), OpQ<T>::threads, smem, st>>>(M, in, sc, b, out, vj, V, ldv, nv, g, partial,
                                                                      dyn);
    return cudaGetLastError();
}

template <typename T>
cudaError_t field_update_q(const double* x, const T* M, const T* J, T* Eth, T* E, const T* B0, T* B1, GridP g,
                           double* partial, int nblocks, cudaStream_t st)
{
    const int smem = (int)sizeof(typename OpQ<T>::Shared);
    const cudaError_t e = cudaFuncSetAttribute(k_field_update_q<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    count_launches(1);
    k_field_update_q<T><<<nblocks, OpQ<T>::threads, smem, st>>>(x, M, J, Eth, E, B0, B1, g, partial);
    return cudaGetLastError();
}

int push_blocks_q(GridP g, int cap)
{
    const int uw = unit_width_q(g);
    const int64_t units = (int64_t)((g.nx + uw - 1) / uw) * g.ny;
    return (int)gridq(units, kPushWarpsQ, cap > 0 ? cap : 152 * 16);
}

template <typename T>
cudaError_t push_q(PArrays<T> src, PRecords<T> dst, const int32_t* start, int32_t* key, int32_t* rank,
                   int32_t* count, const T* Eth, const T* B, GridP g, SpeciesConst sc, double* lsum, int nblocks,
                   cudaStream_t st)
{
    count_launches(1);
    k_push_q<T><<<nblocks, 32 * kPushWarpsQ, 0, st>>>(src, dst, start, key, rank, count, Eth, B, g,
                                                        (T)(sc.q * g.dt / (2.0 * sc.m)), (T)(sc.q * g.dt), (T)sc.m,
                                                        lsum, unit_width_q(g));
    return cudaGetLastError();
}

#define RELSIM_Q_OP(T, MODE, TR)                                                                                  \
    template cudaError_t launch_op_q<T, MODE, TR>(const T*, const double*, double, const double*, double*,        \
                                                  double*, const double*, int64_t, int, GridP, double*,           \
                                                  cudaStream_t, const GmDyn*);
#define RELSIM_Q_INSTANTIATE(T)                                                                                   \
    template cudaError_t deposit_q<T>(const DepositSpecies<T>&, const T*, T*, T*, GridP, cudaStream_t, int);           \
    template cudaError_t field_update_q<T>(const double*, const T*, const T*, T*, T*, const T*, T*, GridP,        \
                                           double*, int, cudaStream_t);                                           \
    template cudaError_t push_q<T>(PArrays<T>, PRecords<T>, const int32_t*, int32_t*, int32_t*, int32_t*,        \
                                   const T*, const T*, GridP, SpeciesConst, double*, int, cudaStream_t);          \
    RELSIM_Q_OP(T, 0, false) RELSIM_Q_OP(T, 1, false) RELSIM_Q_OP(T, 2, false)                                   \
    RELSIM_Q_OP(T, 0, true) RELSIM_Q_OP(T, 1, true) RELSIM_Q_OP(T, 2, true)

RELSIM_Q_INSTANTIATE(float)
RELSIM_Q_INSTANTIATE(double)

}  // namespace relsim
