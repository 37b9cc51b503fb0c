// rotation.cuh -- the Jacobi rotation of a symmetric 2 x 2 block and a reciprocal, without the
// FP64 divisions and square roots whose dependent chains (about 2 us a rotation on GB300's
// FP64 pipe) would dominate a round.
#pragma once
#include <cuda_runtime.h>

namespace sparc {

// c, s with c^2 + s^2 = 1 to FP64 accuracy and J^T [app apq; apq aqq] J diagonal up to a relative
// 2^-22 of apq (apq != 0, finite): the tangent of Golub & Van Loan's sym.schur2, t = sgn / (|tau| +
// sqrt(1 + tau^2)) with tau = (aqq - app) / (2 apq), is formed in FP32 from operands scaled by
// a power of two. A rotation need not annihilate its entry exactly (the entry is recomputed by
// the update, and sweeps repeat until all entries are below the threshold), but it must be
// orthogonal: 1 / sqrt(1 + t^2) starts from FP32 and takes two Newton steps in FP64.
__device__ __forceinline__ void jacobi_angle(double app, double aqq, double apq, double &c, double &s)
{
    const double num = aqq - app, den = 2.0 * apq;
    const int en = (__double2hiint(num) >> 20) & 0x7ff, ed = (__double2hiint(den) >> 20) & 0x7ff;
    const int e = min(max(max(en, ed), 1), 2045);
    const double sc = __hiloint2double((2046 - e) << 20, 0);
    const float fn = (float)(num * sc), fd = (float)(den * sc);
    const float h = sqrtf(fmaf(fn, fn, fd * fd));
    // tau >= 0 (num and den of one sign, or num = 0): t > 0
    float t = fabsf(fd) / (fabsf(fn) + h);
    if ((fn < 0.0f) != (fd < 0.0f) && fn != 0.0f) t = -t;
    const double td = (double)t, x = fma(td, td, 1.0);
    double y = (double)rsqrtf((float)x);
    y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    c = y;
    s = td * y;
}

// 1 / d for a normal positive d: FP32 reciprocal of the significand, two Newton steps.
__device__ __forceinline__ double fast_reciprocal(double d)
{
    const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
    if (hi < 0 || e < 2 || e > 2044) return 1.0 / d;
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(d));
    double y = (double)(1.0f / (float)m);
    y = fma(y, fma(-m, y, 1.0), y);
    y = fma(y, fma(-m, y, 1.0), y);
    return y * __hiloint2double((2046 - e) << 20, 0);
}

// a / b to about an ulp (a short chain; b as for fast_reciprocal, else a plain division: the
// reciprocal of a subnormal b may overflow where the quotient does not)
__device__ __forceinline__ double fast_quotient(double a, double b)
{
    const int e = (__double2hiint(b) >> 20) & 0x7ff;
    if (e < 2 || e > 2044) return a / b;
    const double y = fast_reciprocal(fabs(b));
    const double q = a * y, d = fabs(b);
    const double z = isfinite(q) ? fma(y, fma(-q, d, a), q) : q;
    return b < 0.0 ? -z : z;
}

}  // namespace sparc
