// bounds.cu -- per-column magnitude bounds of a block (the FP64 stencil's and projection's
// fixed-point grid).
#include "fx.cuh"
#include "internal.cuh"

#include <cstdint>

namespace sparc {

// Column bounds: b[c] = max(b[c], largest high word of |y| over column c). Bounded by the read.
// Several CTAs per column stride over it, 16 bytes a load where the columns allow it (VEC),
// eight loads in flight per thread, and raise the bound once each: a few atomics per column, not
// one per warp. FP32 values are compared as their magnitude bits, which the high word follows
// monotonically, and converted once at the end (converted one by one and loaded four bytes at a
// time, 128^3 x 512 took 2.0 ms, three times its read).
namespace {
constexpr int kColmaxThreads = 256, kColmaxPer = 8;
constexpr long kColmaxCtas = 152 * 8;  // CTAs that fill the chip, shared out over the columns

__device__ __forceinline__ unsigned magnitude(double x) { return abs_hi_word(x); }
__device__ __forceinline__ unsigned magnitude(float x) { return __float_as_uint(x) & 0x7fffffffu; }
template <typename T> __device__ __forceinline__ unsigned to_high_word(unsigned m)
{
    return sizeof(T) == 8 ? m : abs_hi_word(__uint_as_float(m));
}
}  // namespace

template <typename T, bool VEC>
__global__ void __launch_bounds__(kColmaxThreads)
k_colmax(const T *__restrict__ Y, long ld, long nd, unsigned *b)
{
    __shared__ unsigned red[kColmaxThreads / 32];
    constexpr int W = VEC ? 16 / (int)sizeof(T) : 1;  // values per load
    const T *Yc = Y + (long)blockIdx.y * ld;
    constexpr long span = (long)kColmaxThreads * kColmaxPer;
    const long nv = nd / W;  // whole loads
    unsigned m = 0u;
    for (long base = (long)blockIdx.x * span + threadIdx.x; base < nv;
         base += (long)gridDim.x * span) {
        if constexpr (VEC) {
            uint4 v[kColmaxPer];
#pragma unroll
            for (int t = 0; t < kColmaxPer; ++t) {
                const long p = base + (long)t * kColmaxThreads;
                v[t] = p < nv ? reinterpret_cast<const uint4 *>(Yc)[p] : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int t = 0; t < kColmaxPer; ++t) {
                m = max(m, max(v[t].y & 0x7fffffffu, v[t].w & 0x7fffffffu));
                if (sizeof(T) == 4) m = max(m, max(v[t].x & 0x7fffffffu, v[t].z & 0x7fffffffu));
            }
        } else {
#pragma unroll
            for (int t = 0; t < kColmaxPer; ++t) {
                const long p = base + (long)t * kColmaxThreads;
                if (p < nv) m = max(m, magnitude(Yc[p]));
            }
        }
    }
    if (VEC && blockIdx.x == 0)
        for (long p = nv * W + threadIdx.x; p < nd; p += kColmaxThreads) m = max(m, magnitude(Yc[p]));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kColmaxThreads / 32; ++w) m = max(m, red[w]);
        m = to_high_word<T>(m);
        if (m) raise_bound(b + blockIdx.y, m);
    }
}

template <typename T>
static cudaError_t colmax_launch(const T *Y, int ncols, long ld, long nd, unsigned *b,
                                 cudaStream_t st)
{
    if (ncols <= 0 || nd <= 0) return cudaSuccess;
    if (ncols > 65535) return cudaErrorInvalidValue;
    const int W = 16 / (int)sizeof(T);
    const bool vec = ((uintptr_t)Y & 15u) == 0 && ld % W == 0;
    const long per = (long)kColmaxThreads * kColmaxPer * (vec ? W : 1);
    const long chunks = (nd + per - 1) / per;
    const long share = (kColmaxCtas + ncols - 1) / ncols;
    dim3 grid((unsigned)(chunks < share ? chunks : share), (unsigned)ncols);
    if (vec)
        k_colmax<T, true><<<grid, kColmaxThreads, 0, st>>>(Y, ld, nd, b);
    else
        k_colmax<T, false><<<grid, kColmaxThreads, 0, st>>>(Y, ld, nd, b);
    note_launch();
    return cudaGetLastError();
}

cudaError_t colmax_f64(const double *Y, int ncols, long ld, long nd, unsigned *b,
                       cudaStream_t st)
{
    return colmax_launch<double>(Y, ncols, ld, nd, b, st);
}

cudaError_t colmax_f32(const float *Y, int ncols, long ld, long nd, unsigned *b,
                       cudaStream_t st)
{
    return colmax_launch<float>(Y, ncols, ld, nd, b, st);
}

}  // namespace sparc
