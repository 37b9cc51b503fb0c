// lanczos.cu -- spectral bounds for the Chebyshev filter (Sec. 4: the extremal
// eigenvalues of H come from a few iterations of the Lanczos method).
//
// Plain Lanczos on one vector, all scalars kept on the device (no host round trip per
// step):  w = H v_j;  alpha_j = <w, v_j>;  w -= alpha_j v_j + beta_{j-1} v_{j-1};
//         beta_j = ||w||;  v_{j+1} = w / beta_j.
// If beta_j is zero or not finite the iteration stops there (an invariant subspace was
// found); the remaining kernels see the stop flag and do nothing.
// Start vector: v0[p] = u(splitmix64(seed ^ p)) - 0.5 with u(z) = (z >> 11) 2^-53, the
// SplitMix64 generator as published by Vigna (mixing constants of Stafford's Mix13).
// Dot products are two-level fixed-order reductions, so results are reproducible.
//
// On one vector every kernel is short (a 64^3 step's six take 5 to 20 us each), so a step is as
// few launches as its global sums allow: apply, <w, v>, the subtraction with ||w||^2, the scaling.
// The CTA that finishes last adds the partial sums and forms the scalars that follow from them
// (a reciprocal or square root in every thread holds the FP64 pipe longer than the vector
// update itself), and the scaling takes the new vector's magnitude bound for the next apply. Ten
// steps on 64^3, 20 atoms: 0.95 ms as eleven launches a step with a separate bound pass (20 us)
// and reduction launches, 0.62 ms so.
#include "fx.cuh"
#include "internal.cuh"

namespace sparc {

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z)
{
    z += 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

__global__ void k_lanczos_start(double *v, long n, unsigned long long seed)
{
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long)gridDim.x * blockDim.x)
        v[p] = (double)(splitmix64(seed ^ (unsigned long long)p) >> 11) *
                   (1.0 / 9007199254740992.0) - 0.5;
}

cudaError_t lanczos_start(double *v, long n, unsigned long long seed, cudaStream_t st)
{
    k_lanczos_start<<<152 * 8, 256, 0, st>>>(v, n, seed);
    note_launch();
    return cudaGetLastError();
}

namespace {
// This CTA's partial sum into part; true in the CTA that stored last, with the sum of all the
// partials (in a fixed order) in `total` of thread 0. ticket returns to zero.
__device__ __forceinline__ bool sum_by_last(double s, double *part, unsigned *ticket, double &total)
{
    __shared__ double red[8];
    __shared__ bool last;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    s = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 256) s += __ldcg(part + b);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        total = 0.0;
        for (int w = 0; w < 8; ++w) total += red[w];
        *ticket = 0u;
    }
    return true;
}

// Raises *b by the largest high word m of the CTA's threads (all CTAs raise one word: by warps,
// the reads of it took longer than the vector update).
__device__ __forceinline__ void raise_by_cta(unsigned *b, unsigned m)
{
    __shared__ unsigned red[8];
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = max(m, red[w]);
        if (m) raise_bound(b, m);
    }
}
}  // namespace

// *r = <x, y>, or 1 / sqrt(<x, y>) (RSQRT).
template <bool RSQRT>
__global__ void __launch_bounds__(256)
k_dot(const double *__restrict__ x, const double *__restrict__ y, long n, double *part,
      unsigned *ticket, double *r)
{
    double s = 0.0, t;
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long)gridDim.x * blockDim.x)
        s += x[p] * y[p];
    if (sum_by_last(s, part, ticket, t) && threadIdx.x == 0) *r = RSQRT ? 1.0 / sqrt(t) : t;
}

cudaError_t dot_f64(const double *x, const double *y, long n, double *part, unsigned *ticket,
                    bool rsqrt, double *r, cudaStream_t st)
{
    if (rsqrt)
        k_dot<true><<<kDotBlocks, 256, 0, st>>>(x, y, n, part, ticket, r);
    else
        k_dot<false><<<kDotBlocks, 256, 0, st>>>(x, y, n, part, ticket, r);
    note_launch();
    return cudaGetLastError();
}

// v *= *f, *b raised to the new values' bound
__global__ void __launch_bounds__(256)
k_lanczos_scale(double *__restrict__ v, long n, const double *f, unsigned *b)
{
    const double s = *f;
    unsigned m = 0u;
#pragma unroll 4
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long)gridDim.x * blockDim.x) {
        const double x = v[p] * s;
        v[p] = x;
        m = max(m, abs_hi_word(x));
    }
    raise_by_cta(b, m);
}

cudaError_t lanczos_scale(double *v, long n, const double *f, unsigned *b, cudaStream_t st)
{
    k_lanczos_scale<<<152 * 2, 256, 0, st>>>(v, n, f, b);
    note_launch();
    return cudaGetLastError();
}

// w -= alpha_j v + beta_{j-1} vp; beta_j = ||w||, inv = 1 / beta_j; stop = j + 1 where beta_j is
// zero or not finite.
__global__ void __launch_bounds__(256)
k_lanczos_orth(double *__restrict__ w, const double *__restrict__ v,
               const double *__restrict__ vp, long n, const double *alpha,
               double *beta, int j, double *part, unsigned *ticket, double *inv, int *stop)
{
    if (*stop) return;
    const double a = alpha[j];
    const double b = j > 0 ? beta[j - 1] : 0.0;
    double s = 0.0, t;
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long)gridDim.x * blockDim.x) {
        double x = w[p] - a * v[p];
        if (j > 0) x -= b * vp[p];  // (vp is not set before the first step)
        w[p] = x;
        s += x * x;
    }
    if (sum_by_last(s, part, ticket, t) && threadIdx.x == 0) {
        const double bj = sqrt(t);
        beta[j] = bj;
        *inv = 1.0 / bj;
        if (!(bj > 0.0) || !isfinite(bj)) *stop = j + 1;
    }
}

cudaError_t lanczos_orth(double *w, const double *v, const double *vp, long n,
                         const double *alpha, double *beta, int j, double *part, unsigned *ticket,
                         double *inv, int *stop, cudaStream_t st)
{
    k_lanczos_orth<<<kDotBlocks, 256, 0, st>>>(w, v, vp, n, alpha, beta, j, part, ticket, inv, stop);
    note_launch();
    return cudaGetLastError();
}

// vp = v, v = w inv; b[1] raised to the new v's bound (after a stop v and its bound b[0] stay)
__global__ void __launch_bounds__(256)
k_lanczos_next(double *__restrict__ v, double *__restrict__ vp, const double *__restrict__ w, long n, const double *inv, unsigned *b,
               const int *stop)
{
    if (*stop) {
        if (blockIdx.x == 0 && threadIdx.x == 0) b[1] = b[0];
        return;
    }
    const double f = *inv;
    unsigned m = 0u;
#pragma unroll 4
    for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long)gridDim.x * blockDim.x) {
        vp[p] = v[p];
        const double x = w[p] * f;
        v[p] = x;
        m = max(m, abs_hi_word(x));
    }
    raise_by_cta(b + 1, m);
}

cudaError_t lanczos_next(double *v, double *vp, const double *w, long n, const double *inv,
                         unsigned *b, const int *stop, cudaStream_t st)
{
    k_lanczos_next<<<152 * 2, 256, 0, st>>>(v, vp, w, n, inv, b, stop);
    note_launch();
    return cudaGetLastError();
}

// T (keff x keff, column-major) from alpha/beta; keff = steps completed.
__global__ void k_lanczos_tridiag(const double *alpha, const double *beta, int k, const int *stop,
                                  double *T, int *keff)
{
    const int m = *stop ? *stop : k;
    if (threadIdx.x == 0) *keff = m;
    for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
        const int i = t % m, j = t / m;
        double v = 0.0;
        if (i == j) v = alpha[i];
        else if (i == j + 1) v = beta[j];
        else if (j == i + 1) v = beta[i];
        T[t] = v;
    }
}

cudaError_t lanczos_tridiag(const double *alpha, const double *beta, int k, const int *stop,
                            double *T, int *keff, cudaStream_t st)
{
    k_lanczos_tridiag<<<1, 256, 0, st>>>(alpha, beta, k, stop, T, keff);
    note_launch();
    return cudaGetLastError();
}

// out[0] = theta_min; out[1] = max(1.01 theta_max, theta_max + |beta_last s_last|).
__global__ void k_lanczos_final(const double *ev, const double *Q, const double *beta, int k,
                                const int *keff, double *out)
{
    const int m = *keff;
    const double tmax = ev[m - 1];
    const double s = Q[(m - 1) + (long)(m - 1) * m];
    const double g = tmax + fabs(beta[m - 1] * s);
    const double b = 1.01 * tmax;
    out[0] = ev[0];
    out[1] = b > g ? b : g;
}

cudaError_t lanczos_bounds_final(const double *ev, const double *Q, const double *beta, int k,
                                 const int *keff, double *out, cudaStream_t st)
{
    k_lanczos_final<<<1, 1, 0, st>>>(ev, Q, beta, k, keff, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace sparc
