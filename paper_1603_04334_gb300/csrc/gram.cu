// gram.cu -- subspace contractions of CheFSI (Sec. 3.4):
//   projection  M_s = Psi_f^T Psi_f,  H_s = Psi_f^T (H Psi_f)   (Eq. after
//               SubspaceGeneralizedEigenproblem), G = A^T B over Nd rows;
//   residuals   r_n = || H x_n - lambda_n x_n ||_2.
// All accumulate in FP64. A product of two FP32 values is exact in FP64, so the FP32
// blocks of the mixed-precision form lose nothing at the product step.
//
// Gram: a CTA computes a 64 x 64 tile of G over one slice of the Nd rows (split-K);
// the slices are summed by a second kernel in a fixed order (deterministic).
#include "df.cuh"
#include "internal.cuh"

namespace sparc {

namespace {
constexpr int GT = 64;     // Gram tile (rows and columns of G)
constexpr int kSplitTarget = 152 * 4;  // CTAs wanted per launch
constexpr long kMinRowsPerSplit = 2048;

int gram_splits(int ns, long nd)
{
    const long tiles = (long)((ns + GT - 1) / GT) * ((ns + GT - 1) / GT);
    long s = (kSplitTarget + tiles - 1) / tiles;
    const long smax = (nd + kMinRowsPerSplit - 1) / kMinRowsPerSplit;
    if (s > smax) s = smax;
    if (s < 1) s = 1;
    if (s > 4096) s = 4096;
    return (int)s;
}
}  // namespace

long gram_part_elems(int ns, long nd) { return (long)gram_splits(ns, nd) * ns * ns; }

// All Gram contractions run in FP32-pair arithmetic (gram_df.cu); for FP32 inputs the
// products are exact there.
template <typename TA, typename TB>
static cudaError_t gram(const TA *A, long lda, const TB *B, long ldb, long nd, int ns, double *G,
                        double *part, cudaStream_t st, bool sym)
{
    return gram_df_launch<TA, TB>(A, lda, B, ldb, nd, ns, G, part, gram_splits(ns, nd), sym, st);
}

cudaError_t gram_f64(const double *A, long lda, const double *B, long ldb, long nd, int ns,
                     double *G, double *part, cudaStream_t st, bool sym)
{
    return gram<double, double>(A, lda, B, ldb, nd, ns, G, part, st, sym);
}
int gram_default_splits(int ns, long nd) { return gram_splits(ns, nd); }

cudaError_t gram_f64_nsplit(const double *A, long lda, const double *B, long ldb, long nd, int ns,
                            double *G, double *part, int nsplit, cudaStream_t st)
{
    return gram_df_launch<double, double>(A, lda, B, ldb, nd, ns, G, part, nsplit, false, st);
}

cudaError_t gram_f32_f32(const float *A, long lda, const float *B, long ldb, long nd, int ns,
                         double *G, double *part, cudaStream_t st, bool sym)
{
    return gram<float, float>(A, lda, B, ldb, nd, ns, G, part, st, sym);
}
cudaError_t gram_f32_f64(const float *A, long lda, const double *B, long ldb, long nd, int ns,
                         double *G, double *part, cudaStream_t st, bool sym)
{
    return gram<float, double>(A, lda, B, ldb, nd, ns, G, part, st, sym);
}

// ---- residual norms ------------------------------------------------------------------
// A column's rows are cut into kResidParts ranges, one CTA each; the partial sums of squares
// are added in range order (deterministic). One pass over both blocks; with one CTA per column
// it read them at 1.8 TB/s (96^3 x 128 FP64: 0.99 ms), with ranges at the memory's rate
// (0.31 ms).
// FP64 blocks take two FP64 operations a value. FP32 blocks would take four (two of them
// conversions), which the FP64 pipe makes seven times the memory time (128^3 x 512: 9.2 ms), so
// r = h - lambda x and its square are formed as exact FP32 pairs (products by FMA, sums by
// two_sum; about 2^-46 relative) and added to FP64 every kResidFlush values (1.5 ms). A range
// whose sum leaves the range where pairs of FP32 hold is done again in FP64.
namespace {
constexpr int kResidParts = 16;
constexpr int kResidFlush = 16;  // values of a thread per FP32-pair partial sum
}  // namespace

long resid_part_elems(int ncols) { return (long)kResidParts * ncols; }

template <typename T>
__device__ __forceinline__ double resid_range(const T *x, const T *hx, double lam, long b, long e)
{
    double s0 = 0.0, s1 = 0.0;
    long p = b + threadIdx.x;
    for (; p + 256 < e; p += 512) {
        const double r0 = (double)hx[p] - lam * (double)x[p];
        const double r1 = (double)hx[p + 256] - lam * (double)x[p + 256];
        s0 += r0 * r0;
        s1 += r1 * r1;
    }
    if (p < e) {
        const double r = (double)hx[p] - lam * (double)x[p];
        s0 += r * r;
    }
    return s0 + s1;
}

__device__ __forceinline__ double resid_range_pair(const float *x, const float *hx, double lam,
                                                   long b, long e)
{
    const float lh = (float)lam, ll = (float)(lam - (double)lh);
    double acc = 0.0;
    for (long p = b + threadIdx.x; p < e; p += 256 * kResidFlush) {
        float sh = 0.0f, sl = 0.0f;
#pragma unroll
        for (int u = 0; u < kResidFlush; ++u) {
            const long q = p + 256 * u;
            const float xv = q < e ? x[q] : 0.0f, hv = q < e ? hx[q] : 0.0f;
            const float m = lh * xv;
            float r, re, t, te;
            two_sum(hv, -m, r, re);                          // h - fl(lambda x), exactly
            re -= fmaf(lh, xv, -m) + ll * xv;                // and the product's low part
            const float w = r * r;
            two_sum(sh, w, t, te);
            sh = t;
            sl += te + fmaf(2.0f * r, re, fmaf(r, r, -w));
        }
        acc += pair_to_double(sh, sl);
    }
    return acc;
}

template <typename T>
__global__ void __launch_bounds__(256)
k_resid(const T *__restrict__ X, const T *__restrict__ HX, long ld, long nd,
        const double *__restrict__ ritz, double *__restrict__ part)
{
    __shared__ double red[8];
    const int c = blockIdx.y;
    const double lam = ritz[c];
    const T *x = X + (long)c * ld;
    const T *hx = HX + (long)c * ld;
    const long per = (nd + kResidParts - 1) / kResidParts;
    const long b = (long)blockIdx.x * per, e = min(nd, b + per);
    double s = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        if constexpr (sizeof(T) == 4)
            s = pass == 0 ? resid_range_pair(x, hx, lam, b, e) : resid_range(x, hx, lam, b, e);
        else
            s = resid_range(x, hx, lam, b, e);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        s = 0.0;
        for (int w = 0; w < 8; ++w) s += red[w];
        __syncthreads();
        // FP32 squares neither overflow nor lose their low parts in between
        if (sizeof(T) == 8 || (s > 1e-24 && s < 1e30)) break;
    }
    if (threadIdx.x == 0) part[(long)c * kResidParts + blockIdx.x] = s;
}

__global__ void k_resid_sum(const double *__restrict__ part, int ncols, double *__restrict__ resid)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncols) return;
    double s = 0.0;
    for (int t = 0; t < kResidParts; ++t) s += part[(long)c * kResidParts + t];
    resid[c] = sqrt(s);
}

template <typename T>
static cudaError_t resid(const T *X, const T *HX, long ld, long nd, int ncols, const double *ritz,
                         double *part, double *out, cudaStream_t st)
{
    if (ncols <= 0) return cudaSuccess;
    k_resid<T><<<dim3(kResidParts, ncols), 256, 0, st>>>(X, HX, ld, nd, ritz, part);
    note_launch();
    k_resid_sum<<<(ncols + 127) / 128, 128, 0, st>>>(part, ncols, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t resid_f64(const double *X, const double *HX, long ld, long nd, int ncols,
                      const double *ritz, double *part, double *out, cudaStream_t st)
{
    return resid<double>(X, HX, ld, nd, ncols, ritz, part, out, st);
}
cudaError_t resid_f32(const float *X, const float *HX, long ld, long nd, int ncols,
                      const double *ritz, double *part, double *out, cudaStream_t st)
{
    return resid<float>(X, HX, ld, nd, ncols, ritz, part, out, st);
}

}  // namespace sparc
