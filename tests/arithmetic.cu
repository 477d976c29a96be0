// The library's own FP32 <-> FP64 conversions and FP64 reciprocals against the
// operations they replace: counts of mismatches on standard output.
#include "common.cuh"

#include <cstdio>

using namespace relsim;

struct Counts {
    unsigned long long widen, narrow, rcp, rsqrt, special;
};

__device__ __forceinline__ bool nan_bits(double v) { return (__double_as_longlong(v) & 0x7fffffffffffffffll) > 0x7ff0000000000000ll; }
__device__ __forceinline__ bool nan_bits(float v) { return (__float_as_uint(v) & 0x7fffffffu) > 0x7f800000u; }

__device__ bool narrow_differs(double d)
{
    const float want = __double2float_rn(d), got = narrow<float>(d);
    return nan_bits(d) ? !nan_bits(got) : __float_as_uint(want) != __float_as_uint(got);
}

// a pseudorandom 64-bit word (the splitmix64 generator)
__device__ unsigned long long word(unsigned long long k)
{
    k += 0x9e3779b97f4a7c15ull;
    k = (k ^ (k >> 30)) * 0xbf58476d1ce4e5b9ull;
    k = (k ^ (k >> 27)) * 0x94d049bb133111ebull;
    return k ^ (k >> 31);
}

// every FP32 pattern: widened, and the FP64 values on, beside and halfway
// between FP32 neighbours narrowed
__global__ void k_all_floats(Counts* c)
{
    unsigned long long w = 0, m = 0;
    for (unsigned long long b = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; b < 1ull << 32;
         b += (unsigned long long)gridDim.x * blockDim.x) {
        const float f = __uint_as_float((unsigned)b);
        const double want = (double)f, got = widen(f);
        w += nan_bits(f) ? !nan_bits(got) : __double_as_longlong(want) != __double_as_longlong(got);
        const long long at = __double_as_longlong(got);
        const long long step[6] = {0, 1, (1ll << 28) - 1, 1ll << 28, (1ll << 28) + 1, (1ll << 29) - 1};
        for (int k = 0; k < 6; ++k) m += narrow_differs(__longlong_as_double(at + step[k]));
    }
    if (w) atomicAdd(&c->widen, w);
    if (m) atomicAdd(&c->narrow, m);
}

__device__ long long apart(double a, double b)   // representable values between two of one sign
{
    const long long d = __double_as_longlong(a) - __double_as_longlong(b);
    return d < 0 ? -d : d;
}

// random FP64 values of every exponent (subnormal to largest) and both signs
__global__ void k_random(Counts* c, int per)
{
    const int e = blockIdx.x;   // 0 .. 2046: the exponent field
    unsigned long long m = 0, r = 0, q = 0;
    for (int k = threadIdx.x; k < per; k += blockDim.x) {
        const unsigned long long h = word((unsigned long long)e * per + k);
        unsigned long long frac = h & 0xfffffffffffffull;
        if (k < 64) frac = k < 32 ? (unsigned long long)k : 0xfffffffffffffull - (k - 32);   // beside powers of two
        const double x = __longlong_as_double((long long)((unsigned long long)e << 52 | frac));
        m += narrow_differs(x) + narrow_differs(-x);
        if (x > 0.0) {
            r += apart(rcp_t(x), 1.0 / x) > 1;
            q += apart(rsqrt_t(x), 1.0 / sqrt(x)) > 2;
        }
    }
    if (m) atomicAdd(&c->narrow, m);
    if (r) atomicAdd(&c->rcp, r);
    if (q) atomicAdd(&c->rsqrt, q);
}

__global__ void k_special(Counts* c)
{
    const double inf = __longlong_as_double(0x7ff0000000000000ll), nan = __longlong_as_double(0x7ff8000000000000ll);
    const double x[8] = {0.0, -0.0, inf, -inf, nan, -1.5, -0x1p-1060, -0x1p901};
    for (int k = 0; k < 8; ++k) {
        const double a = rcp_t(x[k]), b = 1.0 / x[k], s = rsqrt_t(x[k]), t = 1.0 / sqrt(x[k]);
        c->special += nan_bits(b) ? !nan_bits(a) : __double_as_longlong(a) != __double_as_longlong(b);
        c->special += nan_bits(t) ? !nan_bits(s) : __double_as_longlong(s) != __double_as_longlong(t);
    }
}

int main()
{
    Counts* d = nullptr;
    Counts h;
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 1;
    k_all_floats<<<152 * 8, 256>>>(d);
    k_random<<<2047, 256>>>(d, 1 << 16);
    k_special<<<1, 1>>>(d);
    if (cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    std::printf("%llu %llu %llu %llu %llu\n", h.widen, h.narrow, h.rcp, h.rsqrt, h.special);
    return 0;
}
