// poisson.cu -- the electrostatic potential (Sec. 3.3): pseudocharges (Eq.
// PseudochargeDiscrete, Algorithm PseudochargeCalculation), multipole boundary values (Eq.
// phi:BC:discrete, l_max = 6 as in Sec. 4), the charge correction (Eq. Phi:correction)
// and the linear system -(1/4 pi) L_h phi = rho + b - d (Eq. FD:PoissonDiscrete) solved by
// conjugate gradients with a Jacobi preconditioner, all on the device in FP64 (the operator
// as exact integer sums, below).
//
// The multipole terms use real solid harmonics R_lm(x) = |x|^l Y_lm(x/|x|), evaluated as
// polynomials: with Pi_l^m(z, r^2) the associated-Legendre recurrence in solid form
// (Pi_m^m = (2m-1)!!, Pi_{m+1}^m = (2m+1) z Pi_m^m, (l-m) Pi_l^m = (2l-1) z Pi_{l-1}^m -
// (l+m-1) r^2 Pi_{l-2}^m) and (x + iy)^m = A_m + i B_m, R_l0 = N_l0 Pi_l^0, R_lm = N_lm
// Pi_l^m A_m and R_l,-m = N_lm Pi_l^m B_m (m > 0), N the orthonormalisation constants.
// The boundary potential sum_m Y_lm(x) Q_lm depends only on the span of the degree-l
// harmonics, so any orthonormal real basis gives the same values.
//
// Every reduction (moments, CG dot products) runs in a fixed order: a block-level tree,
// then one CTA over the block partials, so results repeat bit for bit.
#include "device_once.cuh"
#include "fx.cuh"
#include "grid.cuh"
#include "internal.cuh"
#include "rotation.cuh"

#include <algorithm>
#include <cmath>

namespace sparc {

namespace {
constexpr int kLmax = 6;
constexpr int kNQ = (kLmax + 1) * (kLmax + 1);  // 49 moments
constexpr int kPT = 256;                         // threads of the grid-wide kernels
constexpr double kInv4Pi = 0.07957747154594767;  // 1 / (4 pi)
constexpr double kSqrtPi = 1.7724538509055159;
constexpr int kMomPer = 8;                       // nodes per thread of the moments
}  // namespace

// R_lm(x, y, z) for l <= 6 into S[l*l + l + m] (N: the 49 normalisation constants, same
// index).
__device__ __forceinline__ void solid_harmonics(double x, double y, double z, const double *N,
                                                double *S)
{
    const double r2 = x * x + y * y + z * z;
    double A = 1.0, B = 0.0;  // Re and Im of (x + iy)^m
    double pmm = 1.0;         // Pi_m^m = (2m-1)!!
#pragma unroll
    for (int m = 0; m <= kLmax; ++m) {
        if (m > 0) {
            const double a = A * x - B * y, b = A * y + B * x;
            A = a;
            B = b;
            pmm *= (double)(2 * m - 1);
        }
        double p2 = 0.0, p1 = pmm;  // Pi_{l-2}^m, Pi_{l-1}^m
#pragma unroll
        for (int l = m; l <= kLmax; ++l) {
            double pl;
            if (l == m)
                pl = pmm;
            else if (l == m + 1)
                pl = (double)(2 * m + 1) * z * pmm;
            else
                pl = ((double)(2 * l - 1) * z * p1 - (double)(l + m - 1) * r2 * p2) /
                     (double)(l - m);
            if (l > m) {
                p2 = p1;
                p1 = pl;
            }
            const int c = l * l + l;
            if (m == 0) {
                S[c] = N[c] * pl;
            } else {
                S[c + m] = N[c + m] * pl * A;
                S[c - m] = N[c + m] * pl * B;
            }
        }
    }
}

struct PoisCoef {
    double w[kRadius + 1];  // Laplacian weights (1/h^2 included); 6 w[0] is the centre's
    double N[kNQ];          // solid-harmonic normalisation
    double cx, cy, cz;      // expansion centre
    double h;
    int radius;
};

// V_ext on the grid extended by `radius` nodes beyond each face: sum_J -Z_J erf(r/rc)/r
// (r -> 0: -2 Z_J / (sqrt(pi) rc); r >= 6 rc: -Z_J / r, where erf rounds to 1).
__global__ void __launch_bounds__(kPT)
k_vext(double *__restrict__ Ve, int e0, int e1, int e2, int radius, double h,
       const double *__restrict__ R, const double *__restrict__ Z, int natoms, double rc)
{
    const long t = (long)blockIdx.x * kPT + threadIdx.x;
    const long ne = (long)e0 * e1 * e2;
    if (t >= ne) return;
    const int i = (int)(t % e0) - radius, j = (int)((t / e0) % e1) - radius,
              k = (int)(t / ((long)e0 * e1)) - radius;
    const double x = i * h, y = j * h, z = k * h;
    double v = 0.0;
    for (int J = 0; J < natoms; ++J) {
        const double dx = x - R[3 * J], dy = y - R[3 * J + 1], dz = z - R[3 * J + 2];
        const double r = sqrt(dx * dx + dy * dy + dz * dz);
        if (r < 1e-12)
            v -= 2.0 * Z[J] / (kSqrtPi * rc);
        else if (r >= 6.0 * rc)
            v -= Z[J] / r;
        else
            v -= Z[J] * erf(r / rc) / r;
    }
    Ve[t] = v;
}

// b = -(1/4 pi) L_h V_ext at the grid nodes (Eq. PseudochargeDiscrete).
__global__ void __launch_bounds__(kPT)
k_pseudocharge(const double *__restrict__ Ve, double *__restrict__ b, int n0, int n1, int n2,
               PoisCoef pc)
{
    const long t = (long)blockIdx.x * kPT + threadIdx.x;
    const long nd = (long)n0 * n1 * n2;
    if (t >= nd) return;
    const int R = pc.radius;
    const int i = (int)(t % n0), j = (int)((t / n0) % n1), k = (int)(t / ((long)n0 * n1));
    const long e0 = n0 + 2 * R, e01 = e0 * (n1 + 2 * R);
    const long c = (i + R) + (j + R) * e0 + (k + R) * e01;
    double L = 6.0 * pc.w[0] * Ve[c];
    for (int p = 1; p <= R; ++p)
        L += pc.w[p] * (Ve[c + p] + Ve[c - p] + Ve[c + p * e0] + Ve[c - p * e0] +
                        Ve[c + p * e01] + Ve[c - p * e01]);
    b[t] = -kInv4Pi * L;
}

// Block partials of sum (rho + b) R_lm(x - centre) over the grid: part[block * 49 + q]. A
// thread sums kMomPer nodes before the 49 block reductions.
__global__ void __launch_bounds__(kPT)
k_moments(const double *__restrict__ rho, const double *__restrict__ b, int n0, int n1, int n2,
          PoisCoef pc, double *__restrict__ part)
{
    __shared__ double sh[kPT / 32][kNQ];
    const long nd = (long)n0 * n1 * n2;
    double A[kNQ];
#pragma unroll
    for (int q = 0; q < kNQ; ++q) A[q] = 0.0;
    for (int u = 0; u < kMomPer; ++u) {
        const long t = ((long)blockIdx.x * kMomPer + u) * kPT + threadIdx.x;
        if (t >= nd) break;
        double S[kNQ];
        const double f = (rho ? rho[t] : 0.0) + b[t];
        const int i = (int)(t % n0), j = (int)((t / n0) % n1), k = (int)(t / ((long)n0 * n1));
        solid_harmonics(i * pc.h - pc.cx, j * pc.h - pc.cy, k * pc.h - pc.cz, pc.N, S);
#pragma unroll
        for (int q = 0; q < kNQ; ++q) A[q] = fma(f, S[q], A[q]);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < kNQ; ++q) {
        double v = A[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) sh[warp][q] = v;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < kNQ; q += kPT) {
        double v = 0.0;
        for (int w = 0; w < kPT / 32; ++w) v += sh[w][q];
        part[(long)blockIdx.x * kNQ + q] = v;
    }
}

// out[q] = scale * sum_b part[b * nq + q] over nblk blocks (CTA q, fixed order).
__global__ void __launch_bounds__(kPT)
k_sum_partials(const double *__restrict__ part, int nblk, int nq, double scale, double *out)
{
    __shared__ double sh[kPT];
    const int q = blockIdx.x;
    double v = 0.0;
    for (int b = threadIdx.x; b < nblk; b += kPT) v += part[(long)b * nq + q];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = kPT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[q] = scale * sh[0];
}

// phi at the nodes outside the grid that a grid node's stencil reaches: face f (0: i < 0,
// 1: i >= n0, 2: j < 0, 3: j >= n1, 4: k < 0, 5: k >= n2), layer p = 1..radius, and the
// face's two in-grid coordinates (a fastest). Eq. (phi:BC:discrete):
// phi = sum_l 4 pi / (2l + 1) r^-(2l+1) sum_m R_lm(x) Q_lm.
__global__ void __launch_bounds__(kPT)
k_phi_ext(double *__restrict__ pe, int n0, int n1, int n2, PoisCoef pc,
          const double *__restrict__ Q, long total)
{
    const long t = (long)blockIdx.x * kPT + threadIdx.x;
    if (t >= total) return;
    const int R = pc.radius;
    const long s01 = (long)n1 * n2 * R, s23 = (long)n0 * n2 * R;
    int f;
    long u;
    if (t < 2 * s01) {
        f = (int)(t / s01);
        u = t % s01;
    } else if (t < 2 * s01 + 2 * s23) {
        f = 2 + (int)((t - 2 * s01) / s23);
        u = (t - 2 * s01) % s23;
    } else {
        const long s45 = (long)n0 * n1 * R;
        f = 4 + (int)((t - 2 * s01 - 2 * s23) / s45);
        u = (t - 2 * s01 - 2 * s23) % s45;
    }
    const int na = f < 2 ? n1 : n0, nb = f < 4 ? n2 : n1;
    const int a = (int)(u % na), bb = (int)((u / na) % nb), p = (int)(u / ((long)na * nb)) + 1;
    int i, j, k;
    switch (f) {
    case 0: i = -p; j = a; k = bb; break;
    case 1: i = n0 - 1 + p; j = a; k = bb; break;
    case 2: i = a; j = -p; k = bb; break;
    case 3: i = a; j = n1 - 1 + p; k = bb; break;
    case 4: i = a; j = bb; k = -p; break;
    default: i = a; j = bb; k = n2 - 1 + p; break;
    }
    const double x = i * pc.h - pc.cx, y = j * pc.h - pc.cy, z = k * pc.h - pc.cz;
    double S[kNQ];
    solid_harmonics(x, y, z, pc.N, S);
    const double r2 = x * x + y * y + z * z, r = sqrt(r2);
    double phi = 0.0, rp = r;  // rp = r^(2l+1)
#pragma unroll
    for (int l = 0; l <= kLmax; ++l) {
        double s = 0.0;
#pragma unroll
        for (int m = -l; m <= l; ++m) s += S[l * l + l + m] * Q[l * l + l + m];
        phi += 4.0 * M_PI / (double)(2 * l + 1) * s / rp;
        rp *= r2;
    }
    pe[t] = phi;
}

// rhs = rho + b - d, d = -(1/4 pi) sum_p w_p (phi at the outside neighbours at distance p)
// (Eq. Phi:correction).
__global__ void __launch_bounds__(kPT)
k_poisson_rhs(const double *__restrict__ rho, const double *__restrict__ b,
              const double *__restrict__ pe, int n0, int n1, int n2, PoisCoef pc,
              double *__restrict__ rhs)
{
    const long t = (long)blockIdx.x * kPT + threadIdx.x;
    const long nd = (long)n0 * n1 * n2;
    if (t >= nd) return;
    const int R = pc.radius;
    const int i = (int)(t % n0), j = (int)((t / n0) % n1), k = (int)(t / ((long)n0 * n1));
    const long s01 = (long)n1 * n2 * R, s23 = (long)n0 * n2 * R, s45 = (long)n0 * n1 * R;
    const long o[6] = {0, s01, 2 * s01, 2 * s01 + s23, 2 * s01 + 2 * s23,
                       2 * s01 + 2 * s23 + s45};
    // the neighbour at distance p beyond a face lies in that face's layer q (1..R): q = p - i
    // below the grid, q = i + p - (n0 - 1) above it (likewise for j, k)
    double d = 0.0;
    for (int p = 1; p <= R; ++p) {
        double s = 0.0;
        if (i - p < 0) s += pe[o[0] + (long)(p - i - 1) * n1 * n2 + j + (long)k * n1];
        if (i + p >= n0) s += pe[o[1] + (long)(i + p - n0) * n1 * n2 + j + (long)k * n1];
        if (j - p < 0) s += pe[o[2] + (long)(p - j - 1) * n0 * n2 + i + (long)k * n0];
        if (j + p >= n1) s += pe[o[3] + (long)(j + p - n1) * n0 * n2 + i + (long)k * n0];
        if (k - p < 0) s += pe[o[4] + (long)(p - k - 1) * n0 * n1 + i + (long)j * n0];
        if (k + p >= n2) s += pe[o[5] + (long)(k + p - n2) * n0 * n1 + i + (long)j * n0];
        d += pc.w[p] * s;
    }
    d *= -kInv4Pi;
    rhs[t] = (rho ? rho[t] : 0.0) + b[t] - d;
}

// ---- conjugate gradients in one cooperative kernel ---------------------------------------
// The Jacobi preconditioner of this operator is one number (its diagonal is constant), which
// cancels from the iteration: x, r, alpha p and the iteration count are those of
//   alpha = r.r / p.Ap;  x += alpha p;  r -= alpha A p;  beta = r'.r' / r.r;  p = r' + beta p.
// Three phases per iteration, a grid barrier after each:
//   A  A p on bricks of 16 x 16 x bz nodes, one or more per CTA, and partial sums of p.Ap;
//   B  r -= alpha A p, partial sums of r.r and the largest |r|;
//   C  x += alpha p, p = r + beta p, p's grid form and its largest magnitude.
// The operator works on a fixed-point grid, as the FP64 stencil does (stencil_df.cu), but p is
// kept to 2^-57 of its largest value, as two whole numbers d and r of 28 bits, both summed over
// the neighbours and weighted in integers without rounding; the result is rounded to 2^-61 of
// the largest term and then to FP64. That is two FP64 operations a node instead of 37, and closer
// to the exact operator than those (40^3, radius 6, relative error in the 2-norm: over CG's
// own p 6e-17 in the median and 2e-15 at most, FP64 5e-16 and 2.7e-15), which CG needs: the
// recursion follows the operator it is given, so a coarser one (26 bits and an FP32
// remainder: 7e-15 and 1.9e-13) leaves f - A x at 2.2e-13 of f whatever tol, and this one,
// like FP64, at 3e-14. Phase C writes that form, with the exponent from |p_new| <= max |r| +
// beta max |p|, so phase A converts nothing. Every CTA adds the CTAs' partial sums itself, in
// the same order.
//
// Bound by latency: three barriers, the brick's loads from L2 and short FP64 chains (an FP64
// warp instruction holds its quarter of the SM for 64 cycles). 64^3: 85 us an iteration with
// seven launches (the FP64 operator 27 us, two dot products and their one-CTA sums 37 us), 19
// us so.
namespace {
constexpr int kCgThreads = 512;
constexpr int kBr = 16;                        // brick edge along x and y
constexpr int kBrH = kBr + 2 * kRadius;        // with the halo
constexpr int kCgSmemMax = 200 * 1024;
constexpr int kCgMaxGrid = 152;                // one CTA per SM (all resident: grid barriers)
constexpr int kCgPerLaunch = 512;              // iterations of one launch

// shared memory of a brick bz planes high: the planes with their x and y halos, then the
// columns without them, z halo included (so that every neighbour is at a constant offset)
constexpr long cg_smem(int bz) { return 8L * (kBrH * kBrH * bz + kBr * kBr * (bz + 2 * kRadius)); }

struct CgState {
    double ff, rr;      // |f|^2, r.r
    int E;              // p's grid exponent: |p| < 2^E
    int done, iters;
    GridBarrier bar;
};

struct CgArgs {
    double *x, *r, *p, *Ap;
    int2 *q;            // p on its grid
    const double *f;
    double *part;       // kCgMaxGrid sums
    unsigned *pmax;     // kCgMaxGrid maxima
    CgState *s;
    int n0, n1, n2, bz;
    int W[kRadius + 1];
    double scale;       // -(1/4 pi) / (D h^2)
    double tol2;
    int first, last;    // iterations of this launch
};

// The CTA's sum of v and maximum of m into *part and *pmax, in a fixed order. An FP64 add
// holds its quarter of the SM for 64 cycles whatever its active lanes, so the sum halves
// through shared memory (20 warp-wide adds) rather than by shuffles in all 16 warps (84).
__device__ __forceinline__ void cg_put(double v, unsigned m, double *part, unsigned *pmax)
{
    __shared__ double sv[kCgThreads];
    __shared__ unsigned sm[kCgThreads / 32];
    const int tid = threadIdx.x;
    sv[tid] = v;
    m = __reduce_max_sync(0xffffffffu, m);
    if ((tid & 31) == 0) sm[tid >> 5] = m;
    __syncthreads();
    for (int h = kCgThreads / 2; h >= 32; h >>= 1) {
        if (tid < h) sv[tid] = v = v + sv[tid + h];
        if (h > 32) __syncthreads();
    }
    if (tid < 32) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        m = __reduce_max_sync(0xffffffffu, tid < kCgThreads / 32 ? sm[tid] : 0u);
        if (tid == 0) *part = v, *pmax = m;
    }
}

// The CTA's maximum alone
__device__ __forceinline__ void cg_put_max(unsigned m, unsigned *pmax)
{
    __shared__ unsigned sm[kCgThreads / 32];
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = __reduce_max_sync(0xffffffffu, threadIdx.x < kCgThreads / 32 ? sm[threadIdx.x] : 0u);
        if (threadIdx.x == 0) *pmax = m;
    }
}

// The sum of part and the maxima of pa and pb over all CTAs (after a grid barrier), handed to
// `fin` in thread 0, which leaves the iteration's scalars in shared memory: one thread does the
// FP64 divisions. Ends with a CTA barrier.
template <typename F>
__device__ __forceinline__ void cg_get(const double *part, const unsigned *pa, const unsigned *pb,
                                       F fin)
{
    if (threadIdx.x < 32) {
        double t[kCgMaxGrid / 32 + 1];
        unsigned x = 0u, y = 0u;
#pragma unroll
        for (int k = 0; k <= kCgMaxGrid / 32; ++k) {
            const int b = threadIdx.x + 32 * k;
            const bool in = b < (int)gridDim.x;
            t[k] = in ? __ldcg(part + b) : 0.0;
            x = max(x, in ? __ldcg(pa + b) : 0u);
            y = max(y, in ? __ldcg(pb + b) : 0u);
        }
        double u = t[0];
#pragma unroll
        for (int k = 1; k <= kCgMaxGrid / 32; ++k)
            if (32 * k < (int)gridDim.x) u += t[k];
        for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
        x = __reduce_max_sync(0xffffffffu, x);
        y = __reduce_max_sync(0xffffffffu, y);
        if (threadIdx.x == 0) fin(u, x, y);
    }
    __syncthreads();
}

// y on the grid of exponent E, |y| < 2^E: y 2^(28-E) = d + 2^-28 r, both of y's sign, |d| < 2^28,
// |r| <= 2^28 (rounded to nearest). With the significand at the top of 64 bits, y = (h:l)
// 2^(e-1086), and (h:l) >> (1026 + E - e) (4 or more) is |y| 2^(60-E). Zero and subnormal y give 0.
__device__ __forceinline__ int2 cg_grid(double y, int E)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(y);
    const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
    const int e = (int)((hw >> 20) & 0x7ffu);
    const unsigned h = e ? __funnelshift_l(lw, hw, 11) | 0x80000000u : 0u;
    const unsigned l = e ? lw << 11 : 0u;
    const unsigned long long N = (((unsigned long long)h << 32) | l) >> min(1026 + E - e, 63);
    const unsigned f = (unsigned)N;
    const int sm = (int)hw >> 31;  // 0 or -1
    return make_int2(((int)(N >> 32) ^ sm) - sm, ((int)((f >> 4) + ((f >> 3) & 1u)) ^ sm) - sm);
}

// scale 2^(E - 38): the operator's factor for T in 2^-10 of a grid unit 2^(E-28)
__device__ __forceinline__ double cg_scale(double scale, int E)
{
    const int e = E - 38 + 1023;
    return e > 0 && e < 2047 ? scale * __hiloint2double(e << 20, 0) : ldexp(scale, E - 38);
}

// tol^2 |f|^2, or -1 (never reached) where f is so small (its norm below 1e-144) that this
// vanishes: the last values of r.r would be a few units of the smallest number and then 0, which
// is no residual below the tolerance
__device__ __forceinline__ double cg_stop(double tol2, double ff)
{
    const double s = tol2 * ff;
    return s < 0x1p-1060 && ff < 0x1p-960 ? -1.0 : s;
}

// E with |y| < 2^E for |y| <= a + b c, from the high words of a and c (each at most 2^-20
// above its value's truncation) and b >= 0
__device__ __forceinline__ int cg_exponent(unsigned a, double b, unsigned c)
{
    const double x = __hiloint2double((int)a + 1, 0), y = __hiloint2double((int)c + 1, 0);
    return bound_exponent(abs_hi_word(fma(b, y, x) * (1.0 + 0x1p-40)));
}
}  // namespace

__global__ void __launch_bounds__(kCgThreads, 1) k_cg(const CgArgs g)
{
    extern __shared__ int2 sm[];
    constexpr int R = kRadius, kU = 4, kL = 8, kWarps = kCgThreads / 32;
    const unsigned nb = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long nd = (long)g.n0 * g.n1 * g.n2, plane = (long)g.n0 * g.n1;
    const long gt = (long)blockIdx.x * kCgThreads + tid, gs = (long)nb * kCgThreads;
    CgState *s = g.s;
    // sums and maxima of the phases: 0 p.Ap, 1 r.r and |r|, 2 |p|; each is written by its CTA
    // and read by all after a barrier, and written again only two barriers later
    double *part1 = g.part + kCgMaxGrid;
    unsigned *pmax0 = g.pmax, *pmax1 = g.pmax + kCgMaxGrid, *pmax2 = g.pmax + 2 * kCgMaxGrid;
    // the iteration's scalars; thread 0 writes them between barriers that all threads pass
    // before they read or after they have read them
    __shared__ struct {
        double rr, ff, alpha, as, beta, sc, stop;  // sc: Ap = sc T; stop: of r.r
        int E, done;
    } S;
    unsigned m, epoch = 0;
    if (g.first == 0) {
        // r = p = f, x = 0
        double v = 0.0;
        m = 0u;
        for (long t = gt; t < nd; t += gs) {
            const double f = g.f[t];
            g.x[t] = 0.0;
            g.r[t] = f;
            g.p[t] = f;
            v = fma(f, f, v);
            m = max(m, abs_hi_word(f));
        }
        cg_put(v, m, part1 + blockIdx.x, pmax2 + blockIdx.x);
        if (!grid_barrier(&s->bar, nb, epoch)) return;
        cg_get(part1, pmax2, pmax2, [&](double u, unsigned x, unsigned) {
            S.rr = S.ff = u;
            S.stop = cg_stop(g.tol2, u);
            S.E = bound_exponent(x);
            S.sc = cg_scale(g.scale, S.E);
        });
        if (S.rr == 0.0) {
            if (gt == 0) s->ff = s->rr = 0.0, s->done = 1, s->iters = 0;
            return;
        }
        for (long t = gt; t < nd; t += gs) g.q[t] = cg_grid(g.p[t], S.E);
        if (!grid_barrier(&s->bar, nb, epoch)) return;
    } else {
        if (tid == 0) {
            S.rr = s->rr;
            S.ff = s->ff;
            S.stop = cg_stop(g.tol2, S.ff);
            S.E = s->E;
            S.sc = cg_scale(g.scale, S.E);
        }
        __syncthreads();
    }
    const int gx = (g.n0 + kBr - 1) / kBr, gy = (g.n1 + kBr - 1) / kBr;
    const int gz = (g.n2 + g.bz - 1) / g.bz;
    const int nbrick = gx * gy * gz;
    const int slab = kBrH * kBrH;                      // a plane with its halo
    int2 *zc = sm + (long)slab * g.bz + R * kBr * kBr;  // columns; plane 0 (halo from -6 on)
    int it = g.first, done = 0;
    for (; it < g.last && !done; ++it) {
        // ---- A: T = Ap / sc, Ap = -(1/4 pi) L_h p, and p.T
        double v = 0.0;
        for (int br = blockIdx.x; br < nbrick; br += nb) {
            const int i0 = (br % gx) * kBr, j0 = (br / gx % gy) * kBr, k0 = br / (gx * gy) * g.bz;
            const int bz = min(g.bz, g.n2 - k0);
            __syncthreads();  // the previous brick's reads are done
            auto at = [&](int i, int j, int k) -> int2 {
                const bool in = i >= 0 && i < g.n0 && j >= 0 && j < g.n1 && k >= 0 && k < g.n2;
                return in ? __ldcg(g.q + (i + (long)g.n0 * j + plane * k)) : make_int2(0, 0);
            };
            // rows of the brick with their x halo: a warp per row, 28 lanes (kL rows a trip, all
            // their loads in flight); then, 16 lanes a row, the y halo and the z halo
            for (int row0 = warp; row0 < bz * kBr; row0 += kL * kWarps) {
                int2 w[kL];
#pragma unroll
                for (int u = 0; u < kL; ++u) {
                    const int row = row0 + u * kWarps;
                    w[u] = lane < kBrH && row < bz * kBr
                               ? at(i0 - R + lane, j0 + row % kBr, k0 + row / kBr)
                               : make_int2(0, 0);
                }
#pragma unroll
                for (int u = 0; u < kL; ++u) {
                    const int row = row0 + u * kWarps, y = row % kBr, z = row / kBr;
                    if (lane < kBrH && row < bz * kBr) {
                        sm[z * slab + (y + R) * kBrH + lane] = w[u];
                        if (lane >= R && lane < R + kBr) zc[(z * kBr + y) * kBr + lane - R] = w[u];
                    }
                }
            }
            const int hx = tid % kBr, nyh = bz * 2 * R, nh = nyh + 2 * R * kBr;
            for (int row0 = tid / kBr; row0 < nh; row0 += kL * (kCgThreads / kBr)) {
                int2 w[kL];
#pragma unroll
                for (int u = 0; u < kL; ++u) {
                    const int row = row0 + u * (kCgThreads / kBr);
                    int y, z;  // the halo row in the brick's coordinates
                    if (row < nyh) {
                        z = row / (2 * R);
                        y = row - z * (2 * R);
                        y = y < R ? y - R : y - R + kBr;
                    } else {
                        z = (row - nyh) / kBr;
                        y = (row - nyh) % kBr;
                        z = z < R ? z - R : z - R + bz;
                    }
                    w[u] = row < nh ? at(i0 + hx, j0 + y, k0 + z) : make_int2(0, 0);
                }
#pragma unroll
                for (int u = 0; u < kL; ++u) {
                    const int row = row0 + u * (kCgThreads / kBr);
                    if (row < nyh) {
                        const int z = row / (2 * R), h = row - z * (2 * R);
                        sm[z * slab + (h < R ? h : h + kBr) * kBrH + hx + R] = w[u];
                    } else if (row < nh) {
                        const int z = (row - nyh) / kBr, y = (row - nyh) % kBr;
                        zc[((z < R ? z - R : z - R + bz) * kBr + y) * kBr + hx] = w[u];
                    }
                }
            }
            __syncthreads();
            const int y = tid / kBr % kBr, zl = tid / (kBr * kBr);
            if (i0 + hx < g.n0 && j0 + y < g.n1) {
                constexpr int kZ = kCgThreads / (kBr * kBr);
                const long o0 = (i0 + hx) + (long)g.n0 * (j0 + y) + plane * k0;
                for (int z0 = zl; z0 < bz; z0 += kU * kZ) {
                    double pv[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int z = z0 + u * kZ;
                        pv[u] = z < bz ? __ldcg(g.p + (o0 + plane * z)) : 0.0;
                    }
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int z = z0 + u * kZ;
                        if (z >= bz) break;
                        const int2 *c = sm + z * slab + (y + R) * kBrH + hx + R;
                        const int2 *cz = zc + (z * kBr + y) * kBr + hx;
                        // (six terms of 28 bits fit 32; the weights' sum is below 2^24.1)
                        long long A = (long long)g.W[0] * c->x, B = (long long)g.W[0] * c->y;
#pragma unroll
                        for (int r = R; r >= 1; --r) {
                            const int2 xa = c[r], xb = c[-r], ya = c[r * kBrH], yb = c[-r * kBrH];
                            const int2 za = cz[r * kBr * kBr], zb = cz[-r * kBr * kBr];
                            A += (long long)g.W[r] * ((xa.x + xb.x + ya.x) + (yb.x + za.x + zb.x));
                            B += (long long)g.W[r] * ((xa.y + xb.y + ya.y) + (yb.y + za.y + zb.y));
                        }
                        // T = (A + 2^-28 B) 2^10, below 2^62.2
                        const double T = (double)(A * 1024 + ((B + (1 << 17)) >> 18));
                        g.Ap[o0 + plane * z] = T;
                        v = fma(pv[u], T, v);
                    }
                }
            }
        }
        cg_put(v, 0u, g.part + blockIdx.x, pmax0 + blockIdx.x);
        if (!grid_barrier(&s->bar, nb, epoch)) return;
        // ---- B: r -= alpha Ap, r.r, max |r|
        cg_get(g.part, pmax0, pmax0, [&](double u, unsigned, unsigned) {
            S.alpha = fast_quotient(S.rr, S.sc * u);
            S.as = S.alpha * S.sc;
        });
        const double mas = -S.as;
        v = 0.0;
        m = 0u;
        // (kU nodes a trip: their loads are in flight together)
        for (long t0 = gt; t0 < nd; t0 += kU * gs) {
            double a[kU], r[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const long t = t0 + u * gs;
                a[u] = t < nd ? __ldcg(g.Ap + t) : 0.0;
                r[u] = t < nd ? g.r[t] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const long t = t0 + u * gs;
                if (t >= nd) break;
                const double x = fma(mas, a[u], r[u]);
                g.r[t] = x;
                v = fma(x, x, v);
                m = max(m, abs_hi_word(x));
            }
        }
        cg_put(v, m, part1 + blockIdx.x, pmax1 + blockIdx.x);
        if (!grid_barrier(&s->bar, nb, epoch)) return;
        // ---- C: x += alpha p, p = r + beta p
        cg_get(part1, pmax1, pmax2, [&](double u, unsigned maxr, unsigned maxp) {
            S.beta = fast_quotient(u, S.rr);
            S.rr = u;
            S.done = !(u > S.stop);  // converged, or not a number
            S.E = cg_exponent(maxr, S.beta, maxp);
            S.sc = cg_scale(g.scale, S.E);
        });
        const double alpha = S.alpha, beta = S.beta;
        const int E = S.E;
        done = S.done;
        m = 0u;
        for (long t0 = gt; t0 < nd; t0 += kU * gs) {
            double po[kU], x[kU], r[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const long t = t0 + u * gs;
                po[u] = t < nd ? g.p[t] : 0.0;
                x[u] = t < nd ? g.x[t] : 0.0;
                r[u] = t < nd ? g.r[t] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const long t = t0 + u * gs;
                if (t >= nd) break;
                g.x[t] = fma(alpha, po[u], x[u]);
                const double pn = fma(beta, po[u], r[u]);
                g.p[t] = pn;
                g.q[t] = cg_grid(pn, E);
                m = max(m, abs_hi_word(pn));
            }
        }
        if (done) continue;
        if (!grid_barrier(&s->bar, nb, epoch)) return;
        // (after the barrier: other CTAs were reading the last maxima before it)
        cg_put_max(m, pmax2 + blockIdx.x);
    }
    if (gt == 0) {
        s->ff = S.ff;
        s->rr = S.rr;
        s->E = S.E;
        s->done = done;
        s->iters = it;
    }
}

namespace {
long pois_partials(long nd)
{
    const long nblk = (nd + (long)kPT * kMomPer - 1) / ((long)kPT * kMomPer);
    const long cg = 3 * kCgMaxGrid + (3 * kCgMaxGrid + 1) / 2;
    return nblk * kNQ > cg ? nblk * kNQ : cg;
}
}  // namespace

size_t poisson_workspace(int n0, int n1, int n2, int radius)
{
    const long nd = (long)n0 * n1 * n2;
    const long ne = (long)(n0 + 2 * radius) * (n1 + 2 * radius) * (n2 + 2 * radius);
    const long nshell = 2L * radius * ((long)n1 * n2 + (long)n0 * n2 + (long)n0 * n1);
    // b, rhs, r, q, p, Ap; V_ext; shell; partials; Q (49); the CG state
    return sizeof(double) * (size_t)(6 * nd + ne + nshell + pois_partials(nd) + kNQ) +
           sizeof(CgState) + 64;
}

// Brick height: bricks one CTA takes per iteration x (its nodes + the halo's loads), fewest
// node-times, within the shared memory.
static int cg_brick_height(int n0, int n1, int n2)
{
    const long t = (long)((n0 + kBr - 1) / kBr) * ((n1 + kBr - 1) / kBr);
    long best = -1;
    int bz = 1;
    for (int z = 1; z <= n2 && cg_smem(z) <= kCgSmemMax; ++z) {
        const long per = (t * ((n2 + z - 1) / z) + kCgMaxGrid - 1) / kCgMaxGrid;
        const long cost = per * (kBrH * kBrH * (long)z + 2 * kRadius * kBr * kBr + 1024);
        if (best < 0 || cost < best) best = cost, bz = z;
    }
    return bz;
}

cudaError_t poisson_solve(const DevHam &H, const double *R, const double *Z, int natoms,
                          double rc, const double *rho, double *phi, double *b_out, double tol,
                          int maxit, void *ws, int *iters_host, double *relres_host,
                          cudaStream_t st)
{
    const int n0 = H.n0, n1 = H.n1, n2 = H.n2, Rr = H.radius;
    const long nd = (long)n0 * n1 * n2;
    const long ne = (long)(n0 + 2 * Rr) * (n1 + 2 * Rr) * (n2 + 2 * Rr);
    const long nshell = 2L * Rr * ((long)n1 * n2 + (long)n0 * n2 + (long)n0 * n1);
    const long nblk = (nd + kPT - 1) / kPT;
    const long nmom = (nd + (long)kPT * kMomPer - 1) / ((long)kPT * kMomPer);
    double *w = (double *)ws;
    double *b = w, *rhs = b + nd, *r = rhs + nd, *q = r + nd, *p = q + nd, *Ap = p + nd;
    double *Ve = Ap + nd, *pe = Ve + ne, *part = pe + nshell, *Q = part + pois_partials(nd);
    CgState *cs = (CgState *)(((uintptr_t)(Q + kNQ) + 15) & ~(uintptr_t)15);

    PoisCoef pc;
    for (int q = 0; q <= kRadius; ++q) pc.w[q] = H.w[q];
    pc.h = H.h;
    pc.radius = Rr;
    pc.cx = 0.5 * (n0 - 1) * H.h;
    pc.cy = 0.5 * (n1 - 1) * H.h;
    pc.cz = 0.5 * (n2 - 1) * H.h;
    for (int l = 0; l <= kLmax; ++l) {
        for (int m = 0; m <= l; ++m) {
            double ratio = 1.0;  // (l - m)! / (l + m)!
            for (int q = l - m + 1; q <= l + m; ++q) ratio /= (double)q;
            const double nlm = sqrt((2.0 * l + 1.0) / (4.0 * M_PI) * ratio * (m ? 2.0 : 1.0));
            pc.N[l * l + l + m] = nlm;
            pc.N[l * l + l - m] = nlm;
        }
    }
    cudaError_t e;
    // pseudocharge, moments, boundary values, right-hand side
    k_vext<<<(unsigned)((ne + kPT - 1) / kPT), kPT, 0, st>>>(Ve, n0 + 2 * Rr, n1 + 2 * Rr,
                                                             n2 + 2 * Rr, Rr, H.h, R, Z, natoms,
                                                             rc);
    note_launch();
    k_pseudocharge<<<(unsigned)nblk, kPT, 0, st>>>(Ve, b, n0, n1, n2, pc);
    note_launch();
    k_moments<<<(unsigned)nmom, kPT, 0, st>>>(rho, b, n0, n1, n2, pc, part);
    note_launch();
    k_sum_partials<<<kNQ, kPT, 0, st>>>(part, (int)nmom, kNQ, H.h * H.h * H.h, Q);
    note_launch();
    k_phi_ext<<<(unsigned)((nshell + kPT - 1) / kPT), kPT, 0, st>>>(pe, n0, n1, n2, pc, Q,
                                                                    nshell);
    note_launch();
    k_poisson_rhs<<<(unsigned)nblk, kPT, 0, st>>>(rho, b, pe, n0, n1, n2, pc, rhs);
    note_launch();
    if (b_out) {
        if ((e = cudaMemcpyAsync(b_out, b, sizeof(double) * nd, cudaMemcpyDeviceToDevice, st)) !=
            cudaSuccess)
            return e;
    }
    // CG from phi = 0
    CgArgs g;
    g.x = phi;
    g.r = r;
    g.p = p;
    g.Ap = Ap;
    g.q = (int2 *)q;
    g.f = rhs;
    g.part = part;
    g.pmax = (unsigned *)(part + 3 * kCgMaxGrid);
    g.s = cs;
    g.n0 = n0;
    g.n1 = n1;
    g.n2 = n2;
    g.bz = cg_brick_height(n0, n1, n2);
    for (int t = 0; t <= kRadius; ++t) {
        g.W[t] = H.wint[t];
    }
    g.scale = -kInv4Pi * H.wunit;
    g.tol2 = tol * tol;
    static DeviceOnce smem, count;
    int sms;
    if ((e = smem.allow_smem(kCgSmemMax, k_cg)) != cudaSuccess) return e;
    if ((e = count.get(sms, [](int dev, int &n) {
             return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
         })) != cudaSuccess)
        return e;
    // enough CTAs for the bricks, and for the vector phases (four nodes per thread)
    const long bricks = (long)((n0 + kBr - 1) / kBr) * ((n1 + kBr - 1) / kBr) * ((n2 + g.bz - 1) / g.bz);
    const long vec = (nd + 4 * kCgThreads - 1) / (4 * kCgThreads);
    const int grid = (int)std::min<long>(std::min(kCgMaxGrid, sms), std::max(bricks, vec));
    if ((e = cudaMemsetAsync(cs, 0, sizeof(CgState), st)) != cudaSuccess) return e;
    CgState h;
    for (int it = 0; it < maxit; it += kCgPerLaunch) {
        g.first = it;
        g.last = maxit - it < kCgPerLaunch ? maxit : it + kCgPerLaunch;
        if ((e = cudaMemsetAsync(&cs->bar, 0, sizeof(GridBarrier), st)) != cudaSuccess) return e;
        void *args[] = {&g};
        e = cudaLaunchCooperativeKernel((const void *)k_cg, dim3(grid), dim3(kCgThreads), args,
                                        (size_t)cg_smem(g.bz), st);
        note_launch();
        if (e != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(&h, cs, sizeof h, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
            return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
        if (h.done || h.bar.err) break;
    }
    // a NaN never meets the tolerance: the iterations left after it would change nothing
    *iters_host = std::isnan(h.rr) ? maxit : h.iters;
    // a barrier that gave up counts as no convergence; with a right-hand side of zeros, or with NaN
    // in it, there is nothing to compare with
    *relres_host = h.bar.err ? INFINITY : h.ff > 0.0 ? std::sqrt(h.rr / h.ff) : 0.0;
    // and below cg_stop's range r.r says nothing any more
    if (!h.done && *relres_host <= tol) *relres_host = NAN;
    return cudaGetLastError();
}

}  // namespace sparc
