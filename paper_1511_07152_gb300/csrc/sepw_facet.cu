// Image-plane faceting (Sec. 4.1): the visibilities of a facet centred at
// (l0, m0).  The linear term of the Taylor expansion of h about the facet
// centre is absorbed by u' = u - w l0 / n0, v' = v - w m0 / n0 (IEEE double,
// each operation rounded, in this order, so that locating u' agrees with the
// FP64 oracle bit for bit), and the phase centre moves to the facet centre:
// V' = V exp(2 pi i (u l0 + v m0 + w (n0 - 1))) (out of the facet: the
// conjugate phase).
//
// The kernel was bound by the FP64 pipe (about 1.3 operations per clock and
// SM; two divisions and the phase are some 30 of them: 60 us in and 18 us out
// for 1M visibilities, where memory alone takes 9 and 6; 26 us together now).  The phase is
// therefore summed exactly in 64-bit fixed point, in units of 2^-64 turns
// (whole turns drop out as the sum wraps), and the divisions by n0 are done on
// the integer significands with a reciprocal computed once on the host; only
// w l0, w m0 and the final subtractions use FP64.
#include <string.h>

#include "sepw_internal.cuh"

namespace sepw {

// x = (-1)^neg m 2^e, an integer significand below 2^53
struct Split {
    unsigned long long m;
    int32_t e;
    int32_t neg;
};

__host__ __device__ __forceinline__ Split split(double x)
{
    long long b;
#ifdef __CUDA_ARCH__
    b = __double_as_longlong(x);
#else
    memcpy(&b, &x, sizeof(b));
#endif
    const int eb = (int)((b >> 52) & 0x7FF);
    const unsigned long long f = (unsigned long long)b & 0x000FFFFFFFFFFFFFull;
    return {eb ? f | 0x0010000000000000ull : f, (eb ? eb : 1) - 1075, b < 0 ? 1 : 0};
}

// x c in units of 2^-64, modulo 2^64 (the fraction below a unit is cut off)
__device__ __forceinline__ unsigned long long turns(const Split &x, const Split &c)
{
    const unsigned long long lo = x.m * c.m, hi = __umul64hi(x.m, c.m);
    const int s = x.e + c.e + 64;  // left shift
    unsigned long long t;
    if (s >= 0)
        t = s < 64 ? lo << s : 0ull;
    else if (s > -64)
        t = lo >> -s | hi << (64 + s);
    else
        t = s > -128 ? hi >> (-s - 64) : 0ull;
    return x.neg != c.neg ? 0ull - t : t;
}

// Division by n0 (0 < n0 < 1 or = 1): with n0 = mb 2^eb, mb in [2^52, 2^53),
// recip = floor((2^116 - 1) / mb), at most 2^64 - 1
struct Divisor {
    double n0;
    unsigned long long recip;
    int32_t e;
};

// RN(a / n0).  q = floor(2^11 ma recip / 2^64) lies within 2 below 2^63 ma / mb,
// within 4 after normalising to 64 bits, so its upper 53 bits and the next
// give the rounding unless the 11 bits below are within 4 under the half way
// (the exact quotient of two 53-bit significands is never half way between
// two others); those, and operands or results that are not normal, take the
// FP64 division.  (A published method: division by an invariant through a
// precomputed reciprocal, T. Granlund and P. Montgomery, PLDI 1994.)
__device__ __forceinline__ double div_n0(double a, const Divisor &d)
{
    const long long b = __double_as_longlong(a);
    const int eb = (int)((b >> 52) & 0x7FF);
    const unsigned long long m = ((unsigned long long)b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    unsigned long long q = __umul64hi(m << 11, d.recip);
    int e = eb - d.e - 52;  // biased exponent of q's top bit, for q >= 2^63
    if (!(q >> 63)) {
        q <<= 1;
        --e;
    }
    const unsigned low = (unsigned)q & 0x7FFu;
    // (recip = 0: n0 is zero or not a number)
    if (!(q >> 63) || eb == 0 || eb == 0x7FF || e < 1 || e > 2045 ||
        (low >= 0x3FCu && low < 0x400u))
        return __ddiv_rn(a, d.n0);
    // the significand without its top bit, rounded; a carry moves into the exponent
    const unsigned long long r = ((q >> 11) & 0x000FFFFFFFFFFFFFull) + (low >> 10);
    return __longlong_as_double((long long)(((unsigned long long)b & 0x8000000000000000ull) |
                                            (((unsigned long long)e << 52) + r)));
}

struct FacetConst {
    double l0, m0;
    Split l, m, n;  // l0, m0, n0 - 1
    Divisor d;
    float sgn;
};

__global__ void __launch_bounds__(256) facet_shift_kernel(
    int64_t nvis, FacetConst f, const double *__restrict__ u, const double *__restrict__ v,
    const double *__restrict__ w, const float2 *vin, double *__restrict__ uo,
    double *__restrict__ vo, float2 *vout)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nvis)
        return;
    const double ui = u[i], vi = v[i], wi = w[i];
    if (uo) {
        uo[i] = __dadd_rn(ui, -div_n0(__dmul_rn(wi, f.l0), f.d));
        vo[i] = __dadd_rn(vi, -div_n0(__dmul_rn(wi, f.m0), f.d));
    }
    if (vout) {
        const Split su = split(ui), sv = split(vi), sw = split(wi);
        const unsigned long long ph = turns(su, f.l) + turns(sv, f.m) + turns(sw, f.n);
        float t = (float)(long long)ph * 5.4210108624275222e-20f;  // 2^-64: [-1/2, 1/2] turns
        if (max(max(su.e, sv.e), max(sw.e, f.n.e)) > 2046 - 1075)
            t = __int_as_float(0x7FC00000);  // a coordinate (or n0) is not finite
        float s, c;
        sincospif(2.f * t, &s, &c);
        s *= f.sgn;
        const float2 x = vin[i];
        vout[i] = make_float2(x.x * c - x.y * s, x.x * s + x.y * c);
    }
}

cudaError_t launch_facet_shift(int64_t nvis, double l0, double m0, int direction,
                               const double *u, const double *v, const double *w,
                               const float2 *vin, double *uo, double *vo, float2 *vout,
                               cudaStream_t s)
{
    if (nvis == 0)
        return cudaSuccess;
    const double n0 = sqrt(1.0 - l0 * l0 - m0 * m0);
    FacetConst f;
    f.l0 = l0;
    f.m0 = m0;
    f.l = split(l0);
    f.m = split(m0);
    f.n = split(n0 - 1.0);
    const Split b = split(n0);  // normal if positive: its square is at least 2^-53
    f.d.n0 = n0;
    f.d.e = b.e;
    f.d.recip = n0 > 0.0 ? (unsigned long long)((((unsigned __int128)1 << 116) - 1) / b.m) : 0ull;
    f.sgn = direction == 0 ? 1.f : -1.f;
    facet_shift_kernel<<<(unsigned)((nvis + 255) / 256), 256, 0, s>>>(nvis, f, u, v, w, vin, uo,
                                                                      vo, vout);
    return cudaGetLastError();
}

}  // namespace sepw
