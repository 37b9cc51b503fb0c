// observables.cu -- the steps after the subspace rotation: occupations and the Fermi level
// (Eq. FermiEnergyConstraintFormulation), the electron density (Sec. 3.4, the equation
// after Eq. OrbitalTransformation) and the non-local atomic force (Eq. NonlocForce:Discrete
// with Y and W of Eq. NonLocForce:U:W, Algorithm non-localForceCalculation), all in FP64.
#include "internal.cuh"

#include <cmath>

namespace sparc {

namespace {
constexpr int kFermiThreads = 256;
constexpr int kFermiMaxIter = 200;
constexpr int kDensityThreads = 256;
constexpr int kForceThreads = 256;

// Sums of a and b over the block in a fixed order (same result on every launch).
template <int NT>
__device__ __forceinline__ void block_sum2(double &a, double &b, double (*sh)[NT])
{
    sh[0][threadIdx.x] = a;
    sh[1][threadIdx.x] = b;
    __syncthreads();
#pragma unroll
    for (int s = NT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + s];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    a = sh[0][0];
    b = sh[1][0];
    __syncthreads();
}
}  // namespace

// One CTA. F(mu) = 2 sum_n g_n(mu) - N_e increases with mu; F' = (2 / kT) sum g (1 - g).
// A bracket [lo, hi] with F(lo) <= 0 <= F(hi) is grown from [min lambda - 1, max lambda + 1];
// from its midpoint, Newton steps are taken while they land inside the bracket and the
// bracket at least halves every two steps, bisection otherwise (the paper finds the same
// root with Brent's method, Sec. 4). Stops when the Newton step is below 2 ulp of mu,
// F(mu) = 0, or the bracket is 4 ulp wide. status: 0 converged, 1 no convergence, 2 a
// non-finite eigenvalue.
__global__ void __launch_bounds__(kFermiThreads)
k_fermi(const double *__restrict__ lam, int ns, double nelec, double kT, double *mu_out,
        double *g, int *status)
{
    __shared__ double red[2][kFermiThreads];
    const double eps = 2.220446049250313e-16;
    auto eval = [&](double mu, double &F, double &dF) {
        double a = 0.0, b = 0.0;
        for (int i = threadIdx.x; i < ns; i += kFermiThreads) {
            const double gi = 1.0 / (1.0 + exp((lam[i] - mu) / kT));
            a += gi;
            b += gi * (1.0 - gi);
        }
        block_sum2<kFermiThreads>(a, b, red);
        F = 2.0 * a - nelec;
        dF = 2.0 * b / kT;
    };
    // extremes of the spectrum
    double lmin = INFINITY, lmax = -INFINITY;
    bool finite = true;
    for (int i = threadIdx.x; i < ns; i += kFermiThreads) {
        const double v = lam[i];
        finite = finite && isfinite(v);
        lmin = fmin(lmin, v);
        lmax = fmax(lmax, v);
    }
    finite = __syncthreads_and(finite);
    red[0][threadIdx.x] = lmin;
    red[1][threadIdx.x] = lmax;
    __syncthreads();
    for (int s = kFermiThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] = fmin(red[0][threadIdx.x], red[0][threadIdx.x + s]);
            red[1][threadIdx.x] = fmax(red[1][threadIdx.x], red[1][threadIdx.x + s]);
        }
        __syncthreads();
    }
    lmin = red[0][0];
    lmax = red[1][0];
    __syncthreads();
    if (!finite) {
        if (threadIdx.x == 0) *status = 2;
        return;
    }
    double lo = lmin - 1.0, hi = lmax + 1.0, F, dF;
    double width = hi - lo;
    for (int t = 0; t < 64; ++t) {  // F(lo) <= 0 (N_e > 0)
        eval(lo, F, dF);
        if (F <= 0.0) break;
        lo -= width;
        width *= 2.0;
    }
    width = hi - lo;
    for (int t = 0; t < 64; ++t) {  // F(hi) >= 0 (N_e < 2 Ns)
        eval(hi, F, dF);
        if (F >= 0.0) break;
        hi += width;
        width *= 2.0;
    }
    double mu = 0.5 * (lo + hi);
    eval(mu, F, dF);
    double w_prev2 = INFINITY, w_prev = INFINITY;
    int st = 1;
    for (int it = 0; it < kFermiMaxIter; ++it) {
        if (F == 0.0) {
            st = 0;
            break;
        }
        if (F < 0.0)
            lo = mu;
        else
            hi = mu;
        const double w = hi - lo;
        if (w <= 4.0 * eps * fmax(fabs(lo), fabs(hi))) {
            st = 0;
            break;
        }
        const double nx = dF > 0.0 ? mu - F / dF : NAN;  // NaN fails the range test
        const bool newton = nx > lo && nx < hi && (it < 2 || w <= 0.5 * w_prev2);
        if (newton && fabs(nx - mu) <= 2.0 * eps * fabs(mu)) {
            mu = nx;
            st = 0;
            break;
        }
        w_prev2 = w_prev;
        w_prev = w;
        mu = newton ? nx : 0.5 * (lo + hi);
        eval(mu, F, dF);
    }
    for (int i = threadIdx.x; i < ns; i += kFermiThreads)
        g[i] = 1.0 / (1.0 + exp((lam[i] - mu) / kT));
    if (threadIdx.x == 0) {
        *mu_out = mu;
        *status = st;
    }
}

cudaError_t fermi_level(const double *lam, int ns, double nelec, double kT, double *mu,
                        double *g, int *status, cudaStream_t st)
{
    k_fermi<<<1, kFermiThreads, 0, st>>>(lam, ns, nelec, kT, mu, g, status);
    note_launch();
    return cudaGetLastError();
}

// rho[p] = scale * sum_n g_n x_n[p]^2, columns in ascending order; one node per thread, eight
// column loads in flight. Bounded by the FP64 pipe (two operations per value, 0.41 ms for
// 96^3 x 128 FP64, whose read alone takes 0.13 ms): where eight g_n in a row are exactly 1,
// as they are for all levels more than 37 kT below the Fermi level, the products by them are left
// out (same bits; 0.32 ms with 55% such levels).
template <typename T>
__global__ void __launch_bounds__(kDensityThreads)
k_density(const T *__restrict__ X, long ld, int ncols, long nd, const double *__restrict__ g,
          double scale, double *__restrict__ rho)
{
    const long p = (long)blockIdx.x * kDensityThreads + threadIdx.x;
    if (p >= nd) return;
    const T *x = X + p;
    double acc = 0.0;
    int n = 0;
    for (; n + 8 <= ncols; n += 8) {
        T v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = x[(long)(n + u) * ld];
        bool ones = true;  // (the same for all threads)
#pragma unroll
        for (int u = 0; u < 8; ++u)
            ones = ones && __double_as_longlong(g[n + u]) == 0x3ff0000000000000ll;
        if (ones) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const double d = (double)v[u];
                acc = fma(d, d, acc);
            }
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const double d = (double)v[u];
                acc = fma(g[n + u] * d, d, acc);
            }
        }
    }
    for (; n < ncols; ++n) {
        const double d = (double)x[(long)n * ld];
        acc = fma(g[n] * d, d, acc);
    }
    rho[p] = scale * acc;
}

template <typename T>
cudaError_t density(const T *X, long ld, int ncols, long nd, const double *g, double h,
                    double *rho, cudaStream_t st)
{
    const long blocks = (nd + kDensityThreads - 1) / kDensityThreads;
    k_density<T><<<(unsigned)blocks, kDensityThreads, 0, st>>>(X, ld, ncols, nd, g,
                                                               2.0 / (h * h * h), rho);
    note_launch();
    return cudaGetLastError();
}
template cudaError_t density<double>(const double *, long, int, long, const double *, double,
                                     double *, cudaStream_t);
template cudaError_t density<float>(const float *, long, int, long, const double *, double,
                                    double *, cudaStream_t);

// ---- non-local force --------------------------------------------------------------------
// A component of the discrete gradient of a column at a node, sum_r w_r (x(p + r) - x(p - r)),
// is formed in integers. With E the largest exponent of the 12 values, each is a whole number
// N = x 2^(60 - E) below 2^60 (bits under 2^-60 of the largest value fall away; FP64 sums of
// the same terms round at 2^-53), the weights are whole numbers over a common denominator, and
// the differences N(p + r) - N(p - r) = a 2^30 + b enter two 64-bit sums by one multiply-add
// each, exactly. The result is rounded once to FP64, packed by integer operations.
// 64 <= E <= kGradMaxExp keeps every intermediate normal; other components (all values tiny or
// zero, huge, Inf, NaN) take the plain FP64 sums.
constexpr int kGradMaxExp = 1982;

// v >> s for any s (0 from 64 on)
__device__ __forceinline__ unsigned long long shift_right(unsigned long long v, unsigned s)
{
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}

template <typename T> struct GradBits;
template <> struct GradBits<double> {
    static constexpr int kOff = 1082;  // x = N 2^(E - kOff)
    static constexpr int kShift = 20;  // exponent's place in the word whose maximum gives E
    unsigned hw, lw;
    __device__ __forceinline__ void set(double x)
    {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x);
        hw = (unsigned)(b >> 32), lw = (unsigned)b;
    }
    __device__ __forceinline__ unsigned magnitude() const { return hw & 0x7fffffffu; }
    // (zero and subnormal values are shifted out, E >= 64)
    __device__ __forceinline__ long long grid(int E) const
    {
        const unsigned e = magnitude() >> kShift;
        const unsigned h = __funnelshift_l(lw, hw, 11) | 0x80000000u;
        const long long N = (long long)shift_right(((unsigned long long)h << 32) | (lw << 11),
                                                   (unsigned)(E + 4) - e);
        return (int)hw < 0 ? -N : N;
    }
};
template <> struct GradBits<float> {
    static constexpr int kOff = 186;
    static constexpr int kShift = 23;
    unsigned u;
    __device__ __forceinline__ void set(float x) { u = __float_as_uint(x); }
    __device__ __forceinline__ unsigned magnitude() const { return u & 0x7fffffffu; }
    __device__ __forceinline__ long long grid(int E) const
    {
        const unsigned e = magnitude() >> kShift;
        const long long N = (long long)shift_right(
            (unsigned long long)((u << 8) | 0x80000000u) << 32, (unsigned)(E + 4) - e);
        return (int)u < 0 ? -N : N;
    }
};

// (ga 2^30 + gb) 2^k rounded to nearest; |ga| < 2^48, |gb| < 2^47, the result in FP64's range
__device__ __forceinline__ double grad_to_double(long long ga, long long gb, int k)
{
    long long t = ga + (gb >> 30);
    unsigned f = (unsigned)gb & 0x3fffffffu;
    const unsigned neg = (unsigned)(t >> 63) & 0x80000000u;
    if (neg) {
        t = -t - (f ? 1 : 0);
        f = (0x40000000u - f) & 0x3fffffffu;
    }
    // t 2^30 + f with its leading one moved to bit 63 (t < 2^49; t = 0: f alone)
    const bool small = t == 0;
    const unsigned long long hi = small ? (unsigned long long)f : (unsigned long long)t;
    if (hi == 0) return 0.0;
    const int lz = __clzll((long long)hi);
    unsigned long long u = hi << lz;
    if (!small) u |= ((unsigned long long)f << 34) >> (64 - lz);
    const int e = (small ? 0 : 30) + 63 - lz + k + 1023;  // biased exponent
    const unsigned long long m = (u >> 11) + ((u >> 10) & 1ull);
    const unsigned long long bits = ((unsigned long long)(e - 1) << 52) + m;  // a carry raises e
    return __longlong_as_double((long long)(bits | ((unsigned long long)neg << 32)));
}

// One CTA per (atom J, column n). Over the atom's support entries: y_l = sum x chi_l and
// w_dl = sum (grad_h x)_d chi_l, with grad_h of Eq. (gradient:approximate) evaluated at the
// entry's node from the column (zero outside the grid); out[(J ncols + n) 16 + k]:
// k = l (y), 4 + 4 d + l (w). Bounded by the FP64 pipe (a warp instruction holds its quarter
// 64 cycles): the 16 multiply-adds per entry are left on it, the 36 operations of the gradient
// are not, and the sums over the threads are formed by 16 threads a value, not one by one.
// 40 atoms, 96^3 x 128 FP64: 2.37 ms with all of it in FP64, 1.05 ms so (0.6 ms of it the 16;
// about 1200 instructions an entry, 900 of them on the 36 values).
template <typename T>
__global__ void __launch_bounds__(kForceThreads, 3)
k_force_yw(const T *__restrict__ X, long ld, const int *__restrict__ atom_ptr,
           const int *__restrict__ idx, const double *__restrict__ chi, int n0, int n1, int n2,
           int radius, GradCoef wg, double *__restrict__ out)
{
    __shared__ double red[16][kForceThreads + 1];
    const int J = blockIdx.x, n = blockIdx.y, ncols = gridDim.y;
    const T *x = X + (long)n * ld;
    const int e0 = atom_ptr[J], e1 = atom_ptr[J + 1];
    const long plane = (long)n0 * n1;
    double acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.0;
    for (int e = e0 + threadIdx.x; e < e1; e += kForceThreads) {
        const unsigned p = (unsigned)idx[e];
        const unsigned row = p / (unsigned)n0;
        const int i = (int)(p - row * (unsigned)n0);
        const int k = (int)(row / (unsigned)n1);
        const int j = (int)(row - (unsigned)k * (unsigned)n1);
        const T *xp = x + p;
        const double xc = (double)xp[0];
        double gd[3];
        const bool inner = radius == kRadius && i >= kRadius && i + kRadius < n0 && j >= kRadius &&
                           j + kRadius < n1 && k >= kRadius && k + kRadius < n2;
        const bool whole = __all_sync(__activemask(), inner);  // no bounds to look at
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const long st = d == 0 ? 1 : d == 1 ? n0 : plane;
            const int at = d == 0 ? i : d == 1 ? j : k, m = d == 0 ? n0 : d == 1 ? n1 : n2;
            GradBits<T> v[2 * kRadius];
            if (whole) {
#pragma unroll
                for (int r = 1; r <= kRadius; ++r) {
                    v[2 * r - 2].set(xp[r * st]);
                    v[2 * r - 1].set(xp[-r * st]);
                }
            } else {
#pragma unroll
                for (int r = 1; r <= kRadius; ++r) {
                    v[2 * r - 2].set(r <= radius && at + r < m ? xp[r * st] : (T)0);
                    v[2 * r - 1].set(r <= radius && at - r >= 0 ? xp[-r * st] : (T)0);
                }
            }
            unsigned mx = 0;
#pragma unroll
            for (int r = 0; r < 2 * kRadius; ++r) mx = max(mx, v[r].magnitude());
            const int E = (int)(mx >> GradBits<T>::kShift);
            if (E >= 64 && E <= kGradMaxExp && !(sizeof(T) == 4 && E == 0xff)) {
                long long ga = 0, gb = 0;
#pragma unroll
                for (int r = 1; r <= kRadius; ++r) {
                    const long long D = v[2 * r - 2].grid(E) - v[2 * r - 1].grid(E);
                    ga += (long long)wg.iw[r] * (int)(D >> 30);
                    gb += (long long)wg.iw[r] * (int)((unsigned)D & 0x3fffffffu);
                }
                gd[d] = grad_to_double(ga, gb, E - GradBits<T>::kOff);
            } else {
                gd[d] = 0.0;
#pragma unroll 1
                for (int r = 1; r <= radius; ++r)
                    gd[d] = fma((double)wg.iw[r], (at + r < m ? (double)xp[r * st] : 0.0) -
                                                      (at - r >= 0 ? (double)xp[-r * st] : 0.0),
                                gd[d]);
            }
        }
        const double2 c01 = reinterpret_cast<const double2 *>(chi)[2L * e];
        const double2 c23 = reinterpret_cast<const double2 *>(chi)[2L * e + 1];
        const double cl[4] = {c01.x, c01.y, c23.x, c23.y};
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            acc[l] = fma(xc, cl[l], acc[l]);
#pragma unroll
            for (int d = 0; d < 3; ++d) acc[4 + 4 * d + l] = fma(gd[d], cl[l], acc[4 + 4 * d + l]);
        }
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) red[k][threadIdx.x] = acc[k];
    __syncthreads();
    static_assert(kForceThreads == 256, "16 threads per value");
    const int k = threadIdx.x >> 4, q = threadIdx.x & 15;
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < kForceThreads / 16; ++m) s += red[k][q + 16 * m];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (q == 0) out[((long)J * ncols + n) * 16 + k] = k < 4 ? s : s * wg.scale;
}

// f_Jd = -4 h^3 sum_n g_n sum_lm gamma_Jl y_nl w_ndl. One CTA per atom, a thread per column
// (strided), the threads' sums combined in a fixed order (one thread per atom and direction
// walking all columns: 103 us for 40 atoms x 128 columns, a chain of loads; 6 us so).
constexpr int kForceSumThreads = 128;
__global__ void __launch_bounds__(kForceSumThreads)
k_force_sum(const double *__restrict__ yw, const double *__restrict__ g,
            const double *__restrict__ gamma, int ncols, double h3, double *__restrict__ f)
{
    __shared__ double red[kForceSumThreads / 32][3];
    const int J = blockIdx.x;
    const double *gm = gamma + 4L * J;
    double s[3] = {0.0, 0.0, 0.0};
    for (int n = threadIdx.x; n < ncols; n += kForceSumThreads) {
        const double *v = yw + ((long)J * ncols + n) * 16;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double a = 0.0;
#pragma unroll
            for (int l = 0; l < 4; ++l) a = fma(gm[l] * v[l], v[4 + 4 * d + l], a);
            s[d] = fma(g[n], a, s[d]);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[d] += __shfl_xor_sync(0xffffffffu, s[d], o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][d] = s[d];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < kForceSumThreads / 32; ++w) t += red[w][threadIdx.x];
        f[3L * J + threadIdx.x] = -4.0 * h3 * t;
    }
}

template <typename T>
cudaError_t nonlocal_force(const DevHam &H, const T *X, long ld, int ncols, const double *g,
                           const double *gamma, const GradCoef &wg, double *yw, double *f,
                           cudaStream_t st)
{
    if (H.natoms <= 0) return cudaSuccess;
    dim3 grid(H.natoms, ncols);
    k_force_yw<T><<<grid, kForceThreads, 0, st>>>(X, ld, H.atom_ptr, H.idx, H.chi, H.n0, H.n1,
                                                  H.n2, H.radius, wg, yw);
    note_launch();
    k_force_sum<<<H.natoms, kForceSumThreads, 0, st>>>(yw, g, gamma, ncols, H.h * H.h * H.h, f);
    note_launch();
    return cudaGetLastError();
}
template cudaError_t nonlocal_force<double>(const DevHam &, const double *, long, int,
                                            const double *, const double *, const GradCoef &,
                                            double *, double *, cudaStream_t);
template cudaError_t nonlocal_force<float>(const DevHam &, const float *, long, int,
                                           const double *, const double *, const GradCoef &,
                                           double *, double *, cudaStream_t);

GradCoef grad_coef(int radius, double h)
{
    // w~_p = (-1)^(p+1) / (h p) (n_o!)^2 / ((n_o - p)! (n_o + p)!), the ratio formed as the
    // product over q = 1..p of (n_o - q + 1) / (n_o + q)
    // The weights over 27720 / h are whole numbers for every radius up to 6 (1 / (p ratio) at
    // p = n_o is n_o (2 n_o)! / (n_o!)^2: 2, 12, 60, 280, 1260, 5544).
    constexpr double kGradDenom = 27720.0;
    static_assert(kRadius == 6, "the common denominator covers radii up to 6");
    GradCoef c;
    for (int p = 0; p <= kRadius; ++p) c.iw[p] = 0;
    c.scale = 1.0 / (kGradDenom * h);
    for (int p = 1; p <= radius; ++p) {
        double ratio = 1.0;
        for (int q = 1; q <= p; ++q) ratio *= (double)(radius - q + 1) / (double)(radius + q);
        c.iw[p] = (int)std::lround(((p % 2) ? kGradDenom : -kGradDenom) * ratio / p);
    }
    return c;
}

}  // namespace sparc
