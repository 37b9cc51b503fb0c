// dense.cu -- the Ns x Ns steps of CheFSI on the device (Sec. 3.4; the paper solves
// the generalized eigenproblem H_s y = lambda M_s y with LAPACK, Sec. 4, serially on
// the host, and names it the next bottleneck in Sec. 5).
//
// Reduction (the one LAPACK's dsygv performs): M_s = L L^T (Cholesky), A = L^-1 H_s L^-T,
// A = Q diag(lambda) Q^T, and the coefficient matrix of the rotation Y = L^-T Q.
// The symmetric eigensolve ends in the cyclic Jacobi method with the round-robin (chess
// tournament) parallel ordering of Brent & Luk (1985): in each round the Ns/2 disjoint
// (p, q) pairs are rotated at once; rotation angles follow Golub & Van Loan's symmetric
// Schur decomposition (Algorithm 8.4.1, "sym.schur2"); a rotation is skipped when
// |a_pq| <= 4 eps ||A||_F (an absolute threshold, so rounding noise near zero diagonal
// entries cannot keep the sweeps going) and the sweeps stop when a sweep skips all of
// them. Off-diagonal entries left below that threshold move the eigenvalues only at
// second order (|a_pq|^2 / gap).
// Eigenvalues are sorted ascending and each eigenvector column is signed so that its
// largest-magnitude entry is positive (lowest index on ties).
//
// At every size the problem is solved approximately in FP32 (64 times the FP64 rate), refined
// to FP64 by products, and checked by the FP64 Jacobi, which does what is left: up to kSmallEig
// states (and the k x k Lanczos problem) in one CTA's shared memory, above on many SMs
// (jacobi.cu). Matrices are column-major in global memory (L2-resident for the sizes used). All
// loops and waits are bounded.
#include "device_once.cuh"
#include "df.cuh"
#include "fx.cuh"
#include "grid.cuh"
#include "internal.cuh"
#include "rotation.cuh"

#include <type_traits>

namespace sparc {

namespace {
constexpr int kMaxSweeps = 60;
constexpr double kEps = 2.220446049250313e-16;
constexpr int kSmallEig = 32;   // largest Ns solved in one CTA in FP64
constexpr int kMaxSmall = 64;   // largest size of the one-CTA kernel (Lanczos steps)
constexpr int kEigArrays = 6;   // shared-memory matrices of the one-CTA eigensolve
constexpr int kMaxSweeps32 = 20;
constexpr int kRefine = 2;

// M_s and H_s are taken between 2^-136 (M_s's diagonal; below: status 1, no basis) and 2^136 (any
// entry; beyond, and NaN: status 2), which is the range of FP32 products. Blocks beyond it are
// not orbitals, and the squares of their overlaps in the Cholesky step would leave FP64's range
// (columns of 1e-140 came out 1e-2 from orthonormal), as their FP32 values do H's.
__device__ __forceinline__ bool in_range(double x) { return fabs(x) <= 0x1p136; }
__device__ __forceinline__ bool pivot_ok(double pivot, double diag, int n)
{
    return pivot > 4.0 * n * kEps * diag && diag >= 0x1p-136 && isfinite(pivot);
}

// Entry (i, j) of the refinement rotation: a / (a_jj - a_ii), or 0 where the two are too close
// for two Newton-Schulz steps to make I + E orthogonal again: |E_ij| > 1/64, or a gap below
// 2^-16 of the matrix (mx: high word of its largest entry), where whole multiplets of
// rounding-sized entries could pass the first test and add up.
__device__ __forceinline__ double refine_entry(double a, double aii, double ajj, bool diag,
                                               unsigned mx)
{
    const double gap = ajj - aii;
    const bool wide = (int)(abs_hi_word(gap) >> 20) >= (int)(mx >> 20) - 16;
    return (!diag && wide && fabs(a) <= 0.015625 * fabs(gap)) ? a / gap : 0.0;
}

__device__ __forceinline__ void pair_of(int r, int k, int m, int &p, int &q)
{
    // circle method: player m-1 is fixed; round r pairs (r, m-1) and
    // ((r + k) mod (m-1), (r - k) mod (m-1)) for k = 1..m/2-1.
    if (k == 0) {
        p = r;
        q = m - 1;
    } else {
        p = (r + k) % (m - 1);
        q = (r - k + (m - 1)) % (m - 1);
    }
    if (p > q) {
        const int t = p;
        p = q;
        q = t;
    }
}

// One warp: where eigenpair i goes and how it is signed. d: the n eigenvalues; v: its
// eigenvector. rank = the number of smaller eigenvalues (ties by index); neg = the entry of
// largest magnitude (lowest index on ties) is negative.
__device__ __forceinline__ void rank_and_sign(const double *d, const double *v, int n, int i,
                                              int &rank, bool &neg)
{
    const int lane = threadIdx.x & 31;
    const double di = d[i];
    int r = 0, arg = -1;
    double best = -1.0;
    for (int j = lane; j < n; j += 32) {
        const double dj = d[j], a = fabs(v[j]);
        r += dj < di || (dj == di && j < i);
        if (a > best) best = a, arg = j;
    }
    for (int o = 16; o > 0; o >>= 1) {
        r += __shfl_xor_sync(0xffffffffu, r, o);
        const double b2 = __shfl_xor_sync(0xffffffffu, best, o);
        const int a2 = __shfl_xor_sync(0xffffffffu, arg, o);
        if (b2 > best || (b2 == best && (unsigned)a2 < (unsigned)arg)) best = b2, arg = a2;
    }
    rank = r;
    neg = arg >= 0 && v[arg] < 0.0;
}
}  // namespace

// Cyclic Jacobi of an n x n matrix, n <= NMAX, by one CTA of NT threads: S and V in shared
// memory (column-major, leading dimension NMAX + 1; rows and columns n .. NMAX - 1 of S are
// not touched); on return S is diagonal and V holds the eigenvectors. Thread (pair k1, pair k2)
// updates the 2 x 2 block of S in place on both sides, then V's columns. Bound by the chain
// angles - barrier - update - barrier of a round. Returns false after kMaxSweeps.
template <int NMAX, int NT>
struct JacobiShared {
    int sp[NMAX / 2], sq[NMAX / 2];
    double sc[NMAX / 2], ss[NMAX / 2], red[NT / 32];
    float fc[NMAX / 2], fs[NMAX / 2];  // the FP32 phase's rotations
    int any, round_rot, rotated;
};

template <int NMAX, int NT>
__device__ __forceinline__ bool jacobi_cta(double *S, double *V, int n, JacobiShared<NMAX, NT> &J)
{
    constexpr int LD = NMAX + 1;
    const int tid = threadIdx.x, lane = tid & 31;
    double f = 0.0;
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        const double a = S[i + j * LD];
        V[i + j * LD] = i == j ? 1.0 : 0.0;
        f += a * a;
    }
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0) J.red[tid >> 5] = f;
    __syncthreads();
    f = 0.0;
    for (int w = 0; w < NT / 32; ++w) f += J.red[w];
    const double thr = 4.0 * kEps * sqrt(f);
    const int m = n + (n & 1), half = m / 2;
    bool ok = false;
    if (tid == 0) J.rotated = 0;
    for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        // a sweep starts with a look for entries above the threshold
        int found = 0;
        for (int t = tid; t < n * n; t += NT) {
            const int i = t % n, j = t / n;
            if (i != j && !(fabs(S[i + j * LD]) <= thr)) found = 1;
        }
        ok = !__syncthreads_or(found);
        if (ok) break;
        if (tid == 0) J.rotated = 1;
        for (int r = 0; r < m - 1; ++r) {
            if (tid < 32) {
                bool rot = false;
                if (lane < half) {
                    int p, q;
                    pair_of(r, lane, m, p, q);
                    double c = 1.0, s = 0.0;
                    const double apq = q < n ? S[p + q * LD] : 0.0;
                    if (fabs(apq) > thr) {
                        jacobi_angle(S[p + p * LD], S[q + q * LD], apq, c, s);
                        rot = true;
                    }
                    J.sp[lane] = p;
                    J.sq[lane] = q < n ? q : p;
                    J.sc[lane] = c;
                    J.ss[lane] = s;
                }
                rot = __any_sync(0xffffffffu, rot);
                if (lane == 0) J.round_rot = rot;
            }
            __syncthreads();
            if (J.round_rot) {
                // block (k1, k2): the pair of an odd size's missing index has q = p and s = 0,
                // and its second row and column are left out
                for (int t = tid; t < half * half; t += NT) {
                    const int k1 = t % half, k2 = t / half;
                    const int p1 = J.sp[k1], q1 = J.sq[k1], p2 = J.sp[k2], q2 = J.sq[k2];
                    const double c1 = J.sc[k1], s1 = J.ss[k1], c2 = J.sc[k2], s2 = J.ss[k2];
                    const double app = S[p1 + p2 * LD], apq = S[p1 + q2 * LD];
                    const double aqp = S[q1 + p2 * LD], aqq = S[q1 + q2 * LD];
                    const double bpp = c1 * app - s1 * aqp, bpq = c1 * apq - s1 * aqq;
                    const double bqp = s1 * app + c1 * aqp, bqq = s1 * apq + c1 * aqq;
                    S[p1 + p2 * LD] = c2 * bpp - s2 * bpq;
                    if (q2 != p2) S[p1 + q2 * LD] = s2 * bpp + c2 * bpq;
                    if (q1 != p1) S[q1 + p2 * LD] = c2 * bqp - s2 * bqq;
                    if (q1 != p1 && q2 != p2) S[q1 + q2 * LD] = s2 * bqp + c2 * bqq;
                }
                for (int t = tid; t < half * n; t += NT) {
                    const int row = t % n, k = t / n;
                    const double s = J.ss[k], c = J.sc[k];
                    if (s == 0.0) continue;
                    const double x = V[row + J.sp[k] * LD], y = V[row + J.sq[k] * LD];
                    V[row + J.sp[k] * LD] = c * x - s * y;
                    V[row + J.sq[k] * LD] = s * x + c * y;
                }
            }
            __syncthreads();
        }
    }
    __syncthreads();
    return ok;
}

// C = op(A) B in one CTA (n x n, leading dimension NMAX + 1, shared memory): TA transposes A;
// MODE 0: the product, 1: A + the product, 2: 1.5 I - 0.5 times it. Ends with a barrier.
template <int NMAX, int NT, bool TA, int MODE>
__device__ __forceinline__ void mm_cta(const double *A, const double *B, double *C, int n)
{
    constexpr int LD = NMAX + 1;
    for (int t = threadIdx.x; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        double v0 = 0.0, v1 = 0.0;
        int k = 0;
        for (; k + 1 < n; k += 2) {
            v0 = fma(TA ? A[k + i * LD] : A[i + k * LD], B[k + j * LD], v0);
            v1 = fma(TA ? A[k + 1 + i * LD] : A[i + (k + 1) * LD], B[k + 1 + j * LD], v1);
        }
        if (k < n) v0 = fma(TA ? A[k + i * LD] : A[i + k * LD], B[k + j * LD], v0);
        double v = v0 + v1;
        if (MODE == 1) v += A[i + j * LD];
        if (MODE == 2) v = (i == j ? 1.5 : 0.0) - 0.5 * v;
        C[i + j * LD] = v;
    }
    __syncthreads();
}

// Eigenvalues (the diagonal of D on return) and eigenvectors (P) of the symmetric A (n x n,
// n <= NMAX, kept) by one CTA: the steps of the large solve below (FP32 Jacobi, Newton-Schulz,
// one or two refinements, FP64 Jacobi for what is left) in shared memory. An FP64 instruction
// occupies its quarter of the SM for 64 cycles whether one lane or 32 are active, so an FP64 Jacobi
// round takes more than 2 us however small the matrix; an FP32 round takes a tenth of it. W: three more
// n x n arrays (W[0] holds the two FP32 matrices). Returns false if the last step did not
// converge.
template <int NMAX, int NT>
__device__ __forceinline__ bool eig_cta(const double *A, double *P, double *D, double *const *W,
                                        int n, JacobiShared<NMAX, NT> &J)
{
    constexpr int LD = NMAX + 1;
    const int tid = threadIdx.x, lane = tid & 31;
    float *S = reinterpret_cast<float *>(W[0]), *Q = S + NMAX * LD;
    // scaled by a power of two to a largest entry in [1/2, 1)
    unsigned mx = 0u;
    for (int t = tid; t < n * n; t += NT) mx = max(mx, abs_hi_word(A[t % n + (t / n) * LD]));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (tid == 0) J.any = 0;
    __syncthreads();
    if (lane == 0) atomicMax(&J.any, (int)mx);
    __syncthreads();
    const unsigned amax = (unsigned)J.any;
    const int ex = (int)(amax >> 20);
    const double scale = (ex == 0 || ex >= 0x7ff) ? 1.0 : ldexp(1.0, 1022 - ex);
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        S[i + j * LD] = (float)(A[i + j * LD] * scale);
        Q[i + j * LD] = i == j ? 1.0f : 0.0f;
    }
    const float thr = 8.0f * 1.1920928955078125e-07f;
    const int m = n + (n & 1), half = m / 2;
    // this thread's 2 x 2 blocks and rows never change; pairs advance by one per round
    for (int sweep = 0; sweep < kMaxSweeps32; ++sweep) {
        __syncthreads();
        if (tid == 0) J.any = 0;
        int a = lane, b = (lane == 0 ? m - 1 : m - 1 - lane);
        for (int r = 0; r < m - 1; ++r) {
            if (tid < 32) {
                bool rot = false, big = false;
                if (lane < half) {
                    const int p = min(a, b), q = max(a, b);
                    float c = 1.0f, s = 0.0f;
                    const float apq = q < n ? S[p + q * LD] : 0.0f;
                    if (fabsf(apq) > thr) {
                        const float num = S[q + q * LD] - S[p + p * LD], den = 2.0f * apq;
                        const float h2 = fmaf(num, num, den * den);
                        float t = __fdividef(fabsf(den), fabsf(num) + h2 * rsqrtf(h2));
                        if ((num < 0.0f) != (den < 0.0f) && num != 0.0f) t = -t;
                        c = rsqrtf(fmaf(t, t, 1.0f));
                        s = t * c;
                        rot = true;
                        big = fabsf(apq) > 8.0f * thr;
                    }
                    J.sp[lane] = p;
                    J.sq[lane] = q < n ? q : p;
                    J.fc[lane] = c;
                    J.fs[lane] = s;
                }
                if (++a == m - 1) a = 0;
                if (lane != 0 && ++b == m - 1) b = 0;
                rot = __any_sync(0xffffffffu, rot);
                big = __any_sync(0xffffffffu, big);
                if (lane == 0) {
                    J.round_rot = rot;
                    if (big) J.any = 1;
                }
            }
            __syncthreads();
            if (J.round_rot) {
                for (int t = tid; t < half * half; t += NT) {
                    const int k1 = t % half, k2 = t / half;
                    const int p1 = J.sp[k1], q1 = J.sq[k1], p2 = J.sp[k2], q2 = J.sq[k2];
                    const float c1 = J.fc[k1], s1 = J.fs[k1], c2 = J.fc[k2], s2 = J.fs[k2];
                    const float app = S[p1 + p2 * LD], apq = S[p1 + q2 * LD];
                    const float aqp = S[q1 + p2 * LD], aqq = S[q1 + q2 * LD];
                    const float bpp = c1 * app - s1 * aqp, bpq = c1 * apq - s1 * aqq;
                    const float bqp = s1 * app + c1 * aqp, bqq = s1 * apq + c1 * aqq;
                    S[p1 + p2 * LD] = c2 * bpp - s2 * bpq;
                    if (q2 != p2) S[p1 + q2 * LD] = s2 * bpp + c2 * bpq;
                    if (q1 != p1) S[q1 + p2 * LD] = c2 * bqp - s2 * bqq;
                    if (q1 != p1 && q2 != p2) S[q1 + q2 * LD] = s2 * bqp + c2 * bqq;
                }
                for (int t = tid; t < half * n; t += NT) {
                    const int row = t % n, k = t / n;
                    const float c = J.fc[k], s = J.fs[k];
                    if (s == 0.0f) continue;
                    const float x = Q[row + J.sp[k] * LD], y = Q[row + J.sq[k] * LD];
                    Q[row + J.sp[k] * LD] = c * x - s * y;
                    Q[row + J.sq[k] * LD] = s * x + c * y;
                }
            }
            __syncthreads();
        }
        if (!J.any) break;
    }
    __syncthreads();
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        P[i + j * LD] = (double)Q[i + j * LD];
    }
    __syncthreads();
    for (int it = 0; it <= kRefine; ++it) {
        if (it > 0) {
            for (int t = tid; t < n * n; t += NT) {
                const int i = t % n, j = t / n;
                W[1][i + j * LD] = refine_entry(D[i + j * LD], D[i + i * LD], D[j + j * LD], i == j, amax);
            }
            __syncthreads();
            mm_cta<NMAX, NT, false, 1>(P, W[1], W[2], n);  // P (I + E)
            for (int t = tid; t < n * n; t += NT) P[t % n + (t / n) * LD] = W[2][t % n + (t / n) * LD];
            __syncthreads();
        }
        mm_cta<NMAX, NT, true, 2>(P, P, W[1], n);
        mm_cta<NMAX, NT, false, 0>(P, W[1], W[2], n);
        mm_cta<NMAX, NT, true, 2>(W[2], W[2], W[1], n);
        mm_cta<NMAX, NT, false, 0>(W[2], W[1], P, n);
        mm_cta<NMAX, NT, false, 0>(A, P, W[1], n);
        mm_cta<NMAX, NT, true, 0>(P, W[1], D, n);
    }
    // exactly symmetric, then the FP64 Jacobi (usually one sweep without a rotation)
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        if (i < j) D[j + i * LD] = D[i + j * LD];
    }
    __syncthreads();
    if (!jacobi_cta<NMAX, NT>(D, W[1], n, J)) return false;
    if (J.rotated) {
        mm_cta<NMAX, NT, false, 0>(P, W[1], W[2], n);
        for (int t = tid; t < n * n; t += NT) P[t % n + (t / n) * LD] = W[2][t % n + (t / n) * LD];
        __syncthreads();
    }
    return true;
}

// The eigensolve of an n x n matrix, n <= NMAX, in one CTA (*n_dev if not null, else nmax).
// Sets *status to 0, 2 (size) or 3 (no convergence). The 10 x 10 Lanczos problem: 185 us with
// FP64 divisions and square roots per angle and A, V in global memory, 70 us so.
template <int NMAX, int NT>
__global__ void __launch_bounds__(NT)
k_eig_small(const double *__restrict__ A, int nmax, const int *n_dev, double *ev, double *Q,
            int *status)
{
    constexpr int LD = NMAX + 1;
    extern __shared__ double sh[];  // kEigArrays arrays
    double *S = sh, *V = sh + NMAX * LD, *D = sh + 2 * NMAX * LD;
    double *const W[3] = {sh + 3 * NMAX * LD, sh + 4 * NMAX * LD, sh + 5 * NMAX * LD};
    __shared__ JacobiShared<NMAX, NT> J;
    __shared__ double dg[NMAX];
    const int n = n_dev ? *n_dev : nmax;
    const int tid = threadIdx.x, lane = tid & 31;
    if (n < 1 || n > nmax || n > NMAX) {
        if (tid == 0) *status = 2;
        return;
    }
    for (int t = tid; t < n * n; t += NT) S[t % n + (t / n) * LD] = A[t];
    __syncthreads();
    if (!eig_cta<NMAX, NT>(S, V, D, W, n, J)) {
        if (tid == 0) *status = 3;
        return;
    }
    for (int i = tid; i < n; i += NT) dg[i] = D[i + i * LD];
    __syncthreads();
    for (int i = tid >> 5; i < n; i += NT / 32) {
        int r;
        bool neg;
        rank_and_sign(dg, V + i * LD, n, i, r, neg);
        if (lane == 0) ev[r] = dg[i];
        for (int row = lane; row < n; row += 32) {
            const double v = V[row + i * LD];
            Q[row + (long)r * n] = neg ? -v : v;
        }
    }
    if (tid == 0) *status = 0;
}

template <int NMAX, int NT>
static cudaError_t eig_small(const double *A, int n, const int *n_dev, double *ev, double *Q,
                             int *status, cudaStream_t st)
{
    const int smem = kEigArrays * NMAX * (NMAX + 1) * (int)sizeof(double);
    static DeviceOnce once;
    const cudaError_t e = once.allow_smem(smem, k_eig_small<NMAX, NT>);
    if (e != cudaSuccess) return e;
    k_eig_small<NMAX, NT><<<1, NT, smem, st>>>(A, n, n_dev, ev, Q, status);
    note_launch();
    return cudaGetLastError();
}

// The whole reduction and eigensolve for n <= kSmallEig states in one CTA and its shared memory,
// in FP64 but for the eigensolve's FP32 start (eig_cta): M_s and H_s symmetrised and checked
// (status 2), Cholesky with the pivot rule of k_chol_grid (status 1), U = L^-T, A = U^T H_s U, the
// eigensolve (status 3), sort and sign, and Cf = U Q. Six launches and a grid barrier per column and per rotation round otherwise: 12
// states, 380 us -> 100 us.
namespace {
constexpr int kRrThreads = 256;
constexpr int kRrArrays = 8;
constexpr int kRrSmem = kRrArrays * kSmallEig * (kSmallEig + 1) * (int)sizeof(double);
}
__global__ void __launch_bounds__(kRrThreads)
k_rr_small(const double *__restrict__ M, const double *__restrict__ Hs, int n,
           double *__restrict__ ritz, double *__restrict__ Cf, int *status)
{
    constexpr int NM = kSmallEig, LD = NM + 1, NT = kRrThreads;
    extern __shared__ double sh[];  // kRrArrays arrays
    constexpr int SZ = NM * LD;
    double *A = sh, *B = sh + SZ, *W = sh + 2 * SZ, *U = sh + 3 * SZ, *D = sh + 4 * SZ;
    double *const X[3] = {sh + 5 * SZ, sh + 6 * SZ, sh + 7 * SZ};
    __shared__ double piv[NM], od[NM];
    __shared__ JacobiShared<NM, NT> J;
    __shared__ int bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) bad = 0;
    __syncthreads();
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        const double m = 0.5 * (M[t] + M[j + (long)i * n]);
        const double h = 0.5 * (Hs[t] + Hs[j + (long)i * n]);
        A[i + j * LD] = m;
        B[i + j * LD] = h;
        if (i == j) od[i] = m;
        if (!in_range(m) || !in_range(h)) bad = 1;
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) *status = 2;
        return;
    }
    // M = L L^T: column j of A below the diagonal keeps M_rj of the Schur complement, piv its
    // pivot; L_rj = A_rj / sqrt(piv_j)
    for (int j = 0; j < n; ++j) {
        const double d = A[j + j * LD];
        if (!pivot_ok(d, od[j], n)) {
            if (tid == 0) *status = 1;
            return;
        }
        if (tid == 0) piv[j] = d;
        const double inv = fast_reciprocal(d);
        const int m = n - 1 - j;
        for (int t = tid; t < m * m; t += NT) {
            const int r = j + 1 + t % m, c = j + 1 + t / m;
            if (r >= c) A[r + c * LD] -= A[r + j * LD] * A[c + j * LD] * inv;
        }
        __syncthreads();
    }
    if (tid < n) {
        const double l = sqrt(piv[tid]);
        piv[tid] = 1.0 / l;  // 1 / L_jj
    }
    __syncthreads();
    for (int t = tid; t < n * n; t += NT) {
        const int r = t % n, c = t / n;
        if (r > c) A[r + c * LD] *= piv[c];  // L
    }
    __syncthreads();
    // U = L^-T: warp c solves L x = e_c (lanes share each row's dot product), U_cr = x_r
    for (int c = warp; c < n; c += NT / 32) {
        for (int r = lane; r < c; r += 32) U[c + r * LD] = 0.0;
        for (int r = c; r < n; ++r) {
            double sum = (lane >= c && lane < r) ? A[r + lane * LD] * U[c + lane * LD] : 0.0;
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0) U[c + r * LD] = ((r == c ? 1.0 : 0.0) - sum) * piv[r];
            __syncwarp();
        }
    }
    __syncthreads();
    // W = H U, A = U^T W (U upper triangular)
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        double v = 0.0;
        for (int k = 0; k <= j; ++k) v = fma(B[i + k * LD], U[k + j * LD], v);
        W[i + j * LD] = v;
    }
    __syncthreads();
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        if (i > j) continue;
        double v = 0.0;
        for (int k = 0; k <= i; ++k) v = fma(U[k + i * LD], W[k + j * LD], v);
        A[i + j * LD] = v;
        A[j + i * LD] = v;
    }
    __syncthreads();
    if (!eig_cta<NM, NT>(A, W, D, X, n, J)) {
        if (tid == 0) *status = 3;
        return;
    }
    for (int i = tid; i < n; i += NT) od[i] = D[i + i * LD];
    __syncthreads();
    for (int i = warp; i < n; i += NT / 32) {
        int r;
        bool neg;
        rank_and_sign(od, W + i * LD, n, i, r, neg);
        if (lane == 0) ritz[r] = od[i];
        for (int row = lane; row < n; row += 32) {
            const double v = W[row + i * LD];
            B[row + r * LD] = neg ? -v : v;
        }
    }
    __syncthreads();
    for (int t = tid; t < n * n; t += NT) {
        const int i = t % n, j = t / n;
        double v = 0.0;
        for (int k = i; k < n; ++k) v = fma(U[i + k * LD], B[k + j * LD], v);
        Cf[t] = v;
    }
}

// nine n x n matrices and the FP32 pair, vectors, the block Jacobi's scratch
long dense_work_elems(int ns)
{
    return 9L * ns * ns + 8L * ns + 64 + (long)(block_jacobi_f32_scratch(ns) / sizeof(double)) + 1;
}

// ---- multi-SM reduction of the generalized problem ----------------------------------
// Cholesky M_s = L L^T on a cooperative grid (right-looking, one bounded grid barrier per
// column), the triangular inverse U = L^-T (one warp per column, no barrier), and the
// products A = U^T (H_s U) and Cf = U Q as small products (k_gemm_small).
namespace {
constexpr int CT = 256;       // threads per CTA of the cooperative Cholesky
constexpr int kInvWarps = 4;  // columns per CTA of the triangular inverse
}  // namespace

// Symmetrise M_s and H_s and check them for entries out of range (status 2); Cholesky with
// the pivot rule pivot_j > 4 n eps M_jj (pivot_ok; status 1 otherwise); writes L row-major into Lr
// (Lr[k + r n] = L_rk, zero above the diagonal) and 1 / L_jj into dinv. Every CTA reads
// the same pivot after the barrier, so all take the same decision. M is overwritten by the
// Schur complements; odiag holds the original diagonal. A barrier that times out sets
// status 4.
__global__ void __launch_bounds__(CT)
k_chol_grid(double *M, double *Hs, int n, double *Lr, double *dinv, double *odiag,
            GridBarrier *bar, int *status)
{
    const unsigned nb = gridDim.x;
    const long gtid = (long)blockIdx.x * CT + threadIdx.x, gs = (long)nb * CT;
    const long nn = (long)n * n;
    unsigned epoch = 0;
    auto sync = [&]() -> bool {
        if (grid_barrier(bar, nb, epoch)) return true;
        if (threadIdx.x == 0) atomicExch(status, 4);
        return false;
    };
    for (long t = gtid; t < nn; t += gs) {
        const int i = (int)(t % n), j = (int)(t / n);
        if (i < j) {
            const long tt = j + (long)i * n;
            const double m = 0.5 * (M[t] + M[tt]), h = 0.5 * (Hs[t] + Hs[tt]);
            M[t] = m;
            M[tt] = m;
            Hs[t] = h;
            Hs[tt] = h;
            if (!in_range(m) || !in_range(h)) atomicExch(status, 2);
        } else if (i == j) {
            if (!in_range(M[t]) || !in_range(Hs[t])) atomicExch(status, 2);
            odiag[i] = M[t];
        }
    }
    if (!sync()) return;
    if (*((volatile int *)status) != 0) return;
    for (int j = 0; j < n; ++j) {
        const double d = __ldcg(M + j + (long)j * n);
        if (!pivot_ok(d, __ldcg(odiag + j), n)) {
            if (gtid == 0) atomicExch(status, 1);
            return;
        }
        const double inv = fast_reciprocal(d);
        const int m = n - 1 - j;
        for (long t = gtid; t < (long)m * m; t += gs) {
            const int rr = j + 1 + (int)(t % m), cc = j + 1 + (int)(t / m);
            if (rr >= cc) {
                const double a = __ldcg(M + rr + (long)j * n), b = __ldcg(M + cc + (long)j * n);
                M[rr + (long)cc * n] = __ldcg(M + rr + (long)cc * n) - a * b * inv;
            }
        }
        if (!sync()) return;
    }
    // L_jj = sqrt(pivot_j), L_rj = M_rj / L_jj
    for (long t = gtid; t < n; t += gs) {
        const double l = sqrt(__ldcg(M + t + t * n));
        odiag[t] = l;
        dinv[t] = 1.0 / l;
    }
    if (!sync()) return;
    for (long t = gtid; t < nn; t += gs) {
        const int r = (int)(t % n), k = (int)(t / n);  // column-major walk of M
        double v = 0.0;
        if (k < r)
            v = __ldcg(M + t) * __ldcg(dinv + k);
        else if (k == r)
            v = __ldcg(odiag + r);
        Lr[k + (long)r * n] = v;
    }
}

// U = L^-T: warp c solves L x = e_c by forward substitution (rows c .. n-1; each row's dot
// product is split over the lanes in a fixed order and lane 0's sum is used), then writes
// row c of U (U_cr = x_r, zero for r < c).
__global__ void __launch_bounds__(32 * kInvWarps)
k_tri_inv(const double *__restrict__ Lr, const double *__restrict__ dinv, int n, double *U,
          const int *status)
{
    __shared__ double xs[kInvWarps][kMaxDense];
    if (*((volatile const int *)status) != 0) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x * kInvWarps + warp;
    if (c >= n) return;
    double *x = xs[warp];
    for (int r = c; r < n; ++r) {
        const double *row = Lr + (long)r * n;
        double sum = 0.0;
        for (int k = c + lane; k < r; k += 32) sum += row[k] * x[k];
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        sum = __shfl_sync(0xffffffffu, sum, 0);
        if (lane == 0) x[r] = ((r == c ? 1.0 : 0.0) - sum) * dinv[r];
        __syncwarp();
    }
    for (int r = lane; r < n; r += 32) U[c + (long)r * n] = r >= c ? x[r] : 0.0;
}

// After the multi-SM Jacobi: sort the eigenvalues ascending and sign the eigenvectors
// (largest |entry| positive, lowest index on ties) into Q; a warp per eigenpair.
__global__ void __launch_bounds__(256)
k_dense_sort(int n, const double *__restrict__ diag, const double *__restrict__ V, double *ritz,
             double *Q, int *status, const GridBarrier *bar)
{
    if (*((volatile int *)status) != 0) return;
    if (bar->err) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *status = 4;
        return;
    }
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    const double *v = V + (long)i * n;
    int r;
    bool neg;
    rank_and_sign(diag, v, n, i, r, neg);
    if (lane == 0) ritz[r] = diag[i];
    for (int row = lane; row < n; row += 32) Q[row + (long)r * n] = neg ? -v[row] : v[row];
}

// ---- small products --------------------------------------------------------------------
// C = op(A) B, all n x n, column-major; op(A) = A or A^T (TA). MODE 0: the product; 1: D + the
// product; 2: 1.5 I - 0.5 times it (the Newton-Schulz coefficients of A^T A). SYM: the product
// is symmetric, only tiles on and above the diagonal are computed and mirrored. A CTA of 16 x
// 16 threads owns a TS x TS tile. Up to 256 states FP64 multiply-adds in tiles of 16 (a 128 x
// 128 product spreads over 64 SMs: 8 us, as in pair arithmetic, and 46 to 72 us on four CTAs
// of 64 x 64); above, tiles of 32 in FP32-pair arithmetic, whose sums go to FP64 every 64
// products as in gram_df.cu (512 states: 0.09 ms against 0.22), except where the result's
// last bits decide how much the FP64 Jacobi finds to rotate (`exact`).
template <int TS, bool NATIVE, bool TA, int MODE, bool SYM>
__global__ void __launch_bounds__(256)
k_gemm_small(const double *__restrict__ A, const double *__restrict__ B,
             const double *__restrict__ D, double *__restrict__ C, int n)
{
    constexpr int KT = 32, U = TS / 16, L = TS * KT / 256;
    static_assert(64 % KT == 0, "flush period");
    if (SYM && blockIdx.x > blockIdx.y) return;
    using Elem = std::conditional_t<NATIVE, double, float2>;
    __shared__ Elem As[KT][TS + 1], Bs[KT][TS + 1];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int i0 = blockIdx.x * TS, j0 = blockIdx.y * TS;
    float sh[U][U], sl[U][U];
    double acc[U][U];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) sh[u][v] = sl[u][v] = 0.0f, acc[u][v] = 0.0;
    double ra[L], rb[L];
    // a tile's elements, the contiguous index fastest over the threads
    auto load = [&](int k0) {
#pragma unroll
        for (int x = 0; x < L; ++x) {
            const int t = tid + 256 * x;
            const int k = TA ? t % KT : t / TS, i = TA ? t / KT : t % TS;
            ra[x] = (k0 + k < n && i0 + i < n)
                        ? (TA ? A[(k0 + k) + (long)(i0 + i) * n] : A[(i0 + i) + (long)(k0 + k) * n])
                        : 0.0;
            const int kb = t % KT, j = t / KT;
            rb[x] = (k0 + kb < n && j0 + j < n) ? B[(k0 + kb) + (long)(j0 + j) * n] : 0.0;
        }
    };
    load(0);
    for (int k0 = 0; k0 < n; k0 += KT) {
#pragma unroll
        for (int x = 0; x < L; ++x) {
            const int t = tid + 256 * x;
            const int k = TA ? t % KT : t / TS, i = TA ? t / KT : t % TS;
            if constexpr (NATIVE) {
                As[k][i] = ra[x];
                Bs[t % KT][t / KT] = rb[x];
            } else {
                As[k][i] = split_double(ra[x]);
                Bs[t % KT][t / KT] = split_double(rb[x]);
            }
        }
        __syncthreads();
        if (k0 + KT < n) load(k0 + KT);
#pragma unroll 8
        for (int k = 0; k < KT; ++k) {
            Elem a[U], b[U];
#pragma unroll
            for (int u = 0; u < U; ++u) a[u] = As[k][tx + 16 * u], b[u] = Bs[k][ty + 16 * u];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int v = 0; v < U; ++v) {
                    if constexpr (NATIVE)
                        acc[u][v] = fma(a[u], b[v], acc[u][v]);
                    else
                        mac(a[u], b[v], sh[u][v], sl[u][v]);
                }
        }
        if (!NATIVE && (k0 / KT) % (64 / KT) == 64 / KT - 1) {
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int v = 0; v < U; ++v) {
                    acc[u][v] += pair_to_double(sh[u][v], sl[u][v]);
                    sh[u][v] = sl[u][v] = 0.0f;
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) {
            const int i = i0 + tx + 16 * u, j = j0 + ty + 16 * v;
            if (i >= n || j >= n) continue;
            const long o = i + (long)j * n;
            double c = NATIVE ? acc[u][v] : acc[u][v] + pair_to_double(sh[u][v], sl[u][v]);
            if (MODE == 1) c += D[o];
            if (MODE == 2) c = (i == j ? 1.5 : 0.0) - 0.5 * c;
            if (SYM) {
                // a diagonal tile's lower half takes the upper half's values
                if (i <= j || i0 != j0) {
                    C[o] = c;
                    if (i != j) C[j + (long)i * n] = c;
                }
            } else {
                C[o] = c;
            }
        }
}

template <bool TA, int MODE, bool SYM>
static cudaError_t gemm_small(const double *A, const double *B, const double *D, double *C, int n,
                              cudaStream_t st, bool exact = false)
{
    const unsigned g16 = (n + 15) / 16, g32 = (n + 31) / 32;
    if (n <= 256)
        k_gemm_small<16, true, TA, MODE, SYM><<<dim3(g16, g16), 256, 0, st>>>(A, B, D, C, n);
    else if (exact)
        k_gemm_small<32, true, TA, MODE, SYM><<<dim3(g32, g32), 256, 0, st>>>(A, B, D, C, n);
    else
        k_gemm_small<32, false, TA, MODE, SYM><<<dim3(g32, g32), 256, 0, st>>>(A, B, D, C, n);
    note_launch();
    return cudaGetLastError();
}

// ---- eigensolve of A = U^T H_s U for Ns > kSmallEig ---------------------------------------
// FP32 block Jacobi (jacobi.cu) -> P, made orthogonal to FP64 accuracy by two Newton-Schulz steps P
// <- P (3 I - P^T P) / 2; A' = P^T A P is then diagonal to about the FP32 level. kRefine times: the
// first-order rotation that removes A's off-diagonal part, P <- P (I + E) with E_ij = a'_ij /
// (a'_jj - a'_ii), re-orthogonalised, and A' again (each step squares the relative off-diagonal
// size, as in the refinement of T. Ogita and K. Aishima, "Iterative refinement for symmetric
// eigenvalue decomposition", Japan J. Indust. Appl. Math. 35, 2018). Pairs too close for it
// keep E_ij = 0 (refine_entry). The FP64 Jacobi on A' removes whatever is above its threshold,
// usually nothing; the eigenvectors of A are P V'. The products cost a few launches where the
// FP64 Jacobi alone needs a grid barrier per round of each of its sweeps: 128 states from 6.6 to
// 2.0 ms; 512 states, where the FP32 phase was there before, from 40 to 15 ms.
__global__ void k_f32_to_f64(const float *a, double *b, long n)
{
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x)
        b[t] = (double)a[t];
}

__global__ void k_refine_rotation(const double *__restrict__ A, double *__restrict__ E, int n, const unsigned *mx)
{
    const long nn = (long)n * n;
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < nn; t += (long)gridDim.x * blockDim.x) {
        const long i = t % n, j = t / n;
        E[t] = refine_entry(A[t], A[i + i * n], A[j + j * n], i == j, *mx);
    }
}

cudaError_t dense_rr(double *M, double *Hs, int ns, double *ritz, double *Cf, double *work,
                     int *status, cudaStream_t st)
{
    if (ns <= 0 || ns > kMaxDense) return cudaErrorInvalidValue;
    cudaError_t e;
    if ((e = cudaMemsetAsync(status, 0, sizeof(int), st)) != cudaSuccess) return e;
    if (ns <= kSmallEig) {
        static DeviceOnce once;
        if ((e = once.allow_smem(kRrSmem, k_rr_small)) != cudaSuccess) return e;
        k_rr_small<<<1, kRrThreads, kRrSmem, st>>>(M, Hs, ns, ritz, Cf, status);
        note_launch();
        return cudaGetLastError();
    }
    const long nn = (long)ns * ns;
    double *R0 = work;            // L row-major, H_s U, a Newton-Schulz step, Jacobi's copy, Q
    double *A = work + nn;        // U^T H_s U
    double *V = work + 2 * nn;    // refinement rotation, then FP64 Jacobi eigenvectors of A'
    double *U = work + 3 * nn;    // L^-T
    double *Ap = work + 4 * nn;   // A' = P^T A P (Jacobi's working copy)
    double *P = work + 5 * nn;    // eigenvectors, ping-pong with P2
    double *G = work + 6 * nn;    // Newton-Schulz coefficients / A P / P V'
    double *P2 = work + 7 * nn;
    float *A32 = (float *)(work + 8 * nn), *V32 = A32 + nn;
    double *diag = work + 9 * nn, *dinv = diag + ns, *odiag = dinv + ns;
    void *scratch = diag + 8L * ns + 64;
    GridBarrier *bar = (GridBarrier *)(status + 8);
    unsigned *mx = (unsigned *)(status + 13);
    static DeviceOnce coop;
    int cb;  // co-resident CTAs of k_chol_grid
    if ((e = coop.get(cb, [](int dev, int &n) {
             return coop_blocks((const void *)k_chol_grid, CT, dev, n);
         })) != cudaSuccess)
        return e;
    long want = (nn / 2 + CT - 1) / CT;
    if (want < 1) want = 1;
    int G0 = (int)(want < cb ? want : cb);
    if (G0 > 152) G0 = 152;
    if ((e = cudaMemsetAsync(bar, 0, sizeof(GridBarrier), st)) != cudaSuccess) return e;
    {
        void *args[] = {&M, &Hs, &ns, &R0, &dinv, &odiag, &bar, &status};
        e = cudaLaunchCooperativeKernel((const void *)k_chol_grid, dim3(G0), dim3(CT), args, 0, st);
        note_launch();
        if (e != cudaSuccess) return e;
    }
    k_tri_inv<<<(ns + kInvWarps - 1) / kInvWarps, 32 * kInvWarps, 0, st>>>(R0, dinv, ns, U,
                                                                            status);
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = gemm_small<false, 0, false>(Hs, U, nullptr, R0, ns, st)) != cudaSuccess) return e;
    if ((e = gemm_small<true, 0, true>(U, R0, nullptr, A, ns, st)) != cudaSuccess) return e;
    // FP32 phase -> P
    const int cg = (int)((nn + 255) / 256 < 152 * 4 ? (nn + 255) / 256 : 152 * 4);
    if ((e = block_jacobi_f32(A, A32, V32, ns, mx, scratch, status + 14 + 1, kMaxSweeps32, st)) !=
        cudaSuccess)
        return e;
    k_f32_to_f64<<<cg, 256, 0, st>>>(V32, P, nn);
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // closer eigenvalues need one step more
    const int refine = ns <= 128 ? kRefine : kRefine + 1;
    for (int it = 0; it <= refine; ++it) {
        if (it > 0) {
            k_refine_rotation<<<cg, 256, 0, st>>>(Ap, V, ns, mx);
            note_launch();
            if ((e = gemm_small<false, 1, false>(P2, V, P2, P, ns, st)) != cudaSuccess) return e;
        }
        // P <- P (1.5 I - 0.5 P^T P) twice (into R0, then P2), A' = P2^T (A P2)
        if ((e = gemm_small<true, 2, true>(P, P, nullptr, G, ns, st)) != cudaSuccess) return e;
        if ((e = gemm_small<false, 0, false>(P, G, nullptr, R0, ns, st)) != cudaSuccess) return e;
        // (the last orthogonalisation and A' decide what is left above the Jacobi's threshold
        // of 4 eps; pair arithmetic leaves 2^-45)
        const bool last = it == refine;
        if ((e = gemm_small<true, 2, true>(R0, R0, nullptr, G, ns, st, last)) != cudaSuccess) return e;
        if ((e = gemm_small<false, 0, false>(R0, G, nullptr, P2, ns, st, last)) != cudaSuccess) return e;
        if ((e = gemm_small<false, 0, false>(A, P2, nullptr, G, ns, st, last)) != cudaSuccess) return e;
        if ((e = gemm_small<true, 0, true>(P2, G, nullptr, Ap, ns, st, last)) != cudaSuccess) return e;
    }
    if ((e = jacobi_grid(Ap, R0, V, diag, ns, bar, status, status + 12, st)) != cudaSuccess)
        return e;
    if ((e = gemm_small<false, 0, false>(P2, V, nullptr, G, ns, st)) != cudaSuccess) return e;  // P V'
    k_dense_sort<<<(ns + 7) / 8, 256, 0, st>>>(ns, diag, G, ritz, R0, status, bar);
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return gemm_small<false, 0, false>(U, R0, nullptr, Cf, ns, st);  // Cf = U Q
}

cudaError_t dense_syev(const double *A, int ns, const int *ns_dev, double *ev, double *Q,
                       int *status, cudaStream_t st)
{
    if (ns <= 0 || ns > kMaxSmall) return cudaErrorInvalidValue;
    if (ns <= kSmallEig) return eig_small<kSmallEig, 256>(A, ns, ns_dev, ev, Q, status, st);
    return eig_small<kMaxSmall, 1024>(A, ns, ns_dev, ev, Q, status, st);
}

}  // namespace sparc
