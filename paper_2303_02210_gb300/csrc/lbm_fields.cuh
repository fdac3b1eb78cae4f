// Density and velocity fields (Eq. 1: rho = sum_i f_i, u = sum_i f_i e_i /
// rho, u = 0 where rho = 0) of one population copy into arrays of doubles,
// for D2Q9 (Lat9) and D2Q7 (Lat7).
//
// What bounds it: the GB300's FP64 pipe issues about two operations per clock
// and SM, so the plain form (nine conversions, 18 additions and two divisions
// in FP64 per node, about 120 clocks per SM and node) took 878 us at 4096 x
// 2048 FP32 with 4.1M tissue nodes, where the memory traffic (7 or 9
// populations read, 24 bytes written) takes about 55 us at the copy rate.
// Populations stored in 32 or 16 bits are 24-bit integers times a power of
// two, so the sums are formed exactly in 64-bit integers, the conversions are
// bit operations, and nine FP64 operations are left per node: a reciprocal
// shared by both quotients and three per quotient (fields_quotient): 85 us there,
// 163 us instead of 1743 at 8192 x 2048.
//
// Every value is the one the plain form gives, bit for bit:
//  * with all populations non-negative and the largest less than 2^22 times
//    the smallest non-zero one, they are integers m_i 2^s_i (0 <= s_i <= 21)
//    of one unit; their sum is below 9 2^45 < 2^49 units, so FP64 additions of
//    them in any order are exact, as the integer ones are;
//  * a correctly rounded quotient, by the argument at fields_quotient.
// Nodes that are not so (a range of 2^22 or more, a negative zero, an infinity
// or a NaN) take the plain form.
// Rows from y_hi on hold no mass (the active window's top): written as zeros
// without being read.
#pragma once

#include "lbm_d2q7.cuh"
#include "lbm_kernels.cuh"

namespace lbm {

// The momentum in FP64, in the oracle's order of operations.
__device__ __forceinline__ void fields_momentum(const double (&g)[NQ], double &jx, double &jy)
{
    jx = ((((g[1] - g[3]) + g[5]) - g[6]) - g[7]) + g[8];
    jy = ((((g[2] - g[4]) + g[5]) + g[6]) - g[7]) - g[8];
}
__device__ __forceinline__ void fields_momentum(const double (&g)[NQ7], double &jx, double &jy)
{
    momentum7<double>(g, jx, jy);
}

// |v| 2^k with v's sign as a double, for |v| < 2^53 (exact; v = 0 gives +0).
__device__ __forceinline__ double fields_i2d(long long v, int k)
{
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int lz = __clzll((long long)a);
    const unsigned long long m = (a << lz) << 1; // the bits below the leading one, at the top
    const unsigned long long e = (unsigned long long)(1023 + 63 - lz + k) << 52;
    const unsigned long long s = v < 0 ? 0x8000000000000000ull : 0ull;
    return a == 0ull ? 0.0 : __longlong_as_double((long long)(s | e | (m >> 12)));
}

// a / b correctly rounded, b in [1, 2) with at most 49 significant bits, y an
// approximation of 1 / b within 2^-52 (relative), a of any magnitude away from
// the underflow threshold. One corrected quotient (Markstein, IBM J. Res.
// Dev. 34, 1990): q0 = a y is within two ulps of a / b, the remainder a - q0 b
// is exact in one fused multiply-add, and q0 + remainder y differs from a / b
// by at most 2 ulp 2^-52 before its one rounding. a / b is no midpoint m of
// two neighbouring doubles, and |a / b - m| = |a - m b| / b is at least
// (ulp / 2) 2^-48 / b > ulp 2^-50, since m is a multiple of ulp / 2 and b one
// of 2^-48 (a is a multiple of their product): so it rounds as a / b does.
__device__ __forceinline__ double fields_quotient(double a, double b, double y)
{
    const double q0 = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-b, q0, a), y, q0);
}

// rho and u of a node from its populations as floats; false if they do not
// fit the integer form.
template <typename LT>
__device__ __forceinline__ bool fields_int(const float (&g)[LT::Q], double &rho, double &ux, double &uy)
{
    constexpr int Q = LT::Q, S = 21;
    uint32_t any = 0u, top = 0u;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const uint32_t b = __float_as_uint(g[i]);
        any |= b;
        top = max(top, b & 0x7FFFFFFFu);
    }
    if (top == 0u && any == 0u) {
        rho = ux = uy = 0.0;
        return true;
    }
    const int emax = (int)(top >> 23);
    bool ok = (int)any >= 0 && emax < 255;
    int m[Q], p[Q]; // population i is m p units of 2^(emax - S - 150)
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const uint32_t b = __float_as_uint(g[i]);
        const int s = (int)(b >> 23) - emax + S;
        ok = ok && (b == 0u || (s >= 0 && b >= 0x00800000u));
        m[i] = b == 0u ? 0 : (int)((b & 0x7FFFFFu) | 0x800000u);
        p[i] = 1 << (s & 31);
    }
    if (!ok) return false;
    long long r = 0, jx = 0, jy = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) r += (long long)m[i] * p[i];
    if constexpr (Q == 9) {
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if (ex(i) != 0) jx += (long long)m[i] * (ex(i) * p[i]);
            if (ey(i) != 0) jy += (long long)m[i] * (ey(i) * p[i]);
        }
    } else { // twice jx, and jy before its factor sqrt(3)/2
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            jx += (long long)m[i] * ((i == 1 ? 2 : (i == 4 ? -2 : (i == 2 || i == 6 ? 1 : -1))) * p[i]);
            if (i != 1 && i != 4) jy += (long long)m[i] * ((i == 2 || i == 3 ? 1 : -1) * p[i]);
        }
    }
    // rho = b 2^k units with b in [1, 2)
    const int k = 63 - __clzll(r);
    const double b = fields_i2d(r, -k);
    rho = __longlong_as_double(__double_as_longlong(b) + ((long long)(k + emax - S - 150) << 52));
    // 1 / b: the float reciprocal of b's upper bits (within 2^-21), then one
    // third-order step
    const uint32_t hi = (uint32_t)__double2hiint(b), lo = (uint32_t)__double2loint(b);
    const float bf = __uint_as_float(0x3F800000u | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(bf));
    const uint32_t yb = __float_as_uint(yf);
    const double y0 = __hiloint2double((int)((yb >> 3) + (896u << 20)), (int)(yb << 29));
    const double e = __fma_rn(-b, y0, 1.0);
    const double y = __fma_rn(y0, __fma_rn(e, e, e), y0);
    if constexpr (Q == 9) {
        ux = fields_quotient(fields_i2d(jx, -k), b, y);
        uy = fields_quotient(fields_i2d(jy, -k), b, y);
    } else {
        ux = fields_quotient(fields_i2d(jx, -k - 1), b, y);
        uy = fields_quotient(__dmul_rn(fields_i2d(jy, -k), HALF_SQRT3), b, y);
    }
    return true;
}

// One node per thread: nine loads in flight per thread, coalesced stores
// whatever the width.
template <typename S, typename LT>
__global__ void __launch_bounds__(256) k_fields(SimDev d, int cur, double *__restrict__ rho, double *__restrict__ ux,
                                                double *__restrict__ uy)
{
    const uint32_t total = (uint32_t)d.W * (uint32_t)d.H;
    const uint32_t k = blockIdx.x * 256u + threadIdx.x;
    if (k >= total) return;
    const int y = (int)(k / (uint32_t)d.W), x = (int)(k % (uint32_t)d.W);
    double r = 0.0, vx = 0.0, vy = 0.0;
    if (y < d.sc->y_hi) {
        const Pop<S> pc(d);
        const S *f = (const S *)d.f[cur] + (long long)y * d.Wp + x;
        bool done = false;
        arith_t<S> g[LT::Q];
#pragma unroll
        for (int i = 0; i < LT::Q; ++i) g[i] = pc.ld(f[i * d.P], i);
        if constexpr (sizeof(S) < 8) done = fields_int<LT>(g, r, vx, vy);
        if (!done) {
            double h[LT::Q];
#pragma unroll
            for (int i = 0; i < LT::Q; ++i) h[i] = (double)g[i];
            r = h[0];
#pragma unroll
            for (int i = 1; i < LT::Q; ++i) r = r + h[i];
            double jx, jy;
            fields_momentum(h, jx, jy);
            vx = r != 0.0 ? jx / r : 0.0;
            vy = r != 0.0 ? jy / r : 0.0;
        }
    }
    rho[k] = r;
    ux[k] = vx;
    uy[k] = vy;
}

template <typename S, typename LT>
cudaError_t launch_fields(const SimDev &d, int cur, double *rho, double *ux, double *uy, cudaStream_t s)
{
    const unsigned blocks = ((unsigned)d.W * (unsigned)d.H + 255u) / 256u;
    k_fields<S, LT><<<blocks, 256, 0, s>>>(d, cur, rho, ux, uy);
    return cudaGetLastError();
}

} // namespace lbm
