// gram_tc.cu -- the subspace contractions on the tensor cores (tcgen05):
//   M_s = Y^T Y  and  H_s = Y^T (H Y)   (projection onto the filtered block, Sec. 3.4),
// G = A^T B over the Nd grid rows, and the rotation X = Y (L^-T Q) (Eq.
// OrbitalTransformation). Two digit representations share one kernel: 47 bits (six digits;
// the Gram pair of both forms, FP64 or FP32 Y, and the FP64 form's rotation) and 23 bits
// (three digits; sparc_gram_tc and the mixed form's FP32 rotation). The description below
// is of the 23-bit form; the 47-bit form differs as stated at struct Tc47.
//
// The scheme is a fixed-point form of the error-free splitting of a matrix product into
// slices whose products the hardware forms exactly (the Ozaki scheme: K. Ozaki, T. Ogita,
// S. Oishi and S. M. Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication and its applicability", Numer. Algorithms 59,
// 2012), with per-chunk scaling so that the slices are small integers and the tensor
// core's FP32 accumulator sums them exactly, in the manner of the integer-unit emulations of
// FP64 products (H. Ootomo, K. Ozaki and R. Yokota, "DGEMM on integer matrix
// multiplication unit", IJHPCA 2024).
//
// Representation. The rows are cut into chunks of kChunk = 256. For chunk c and column j
// of an operand, e = e(c, j) is the smallest integer with max_{k in c} |x_kj| < 2^e, and
// each entry is rounded to N = round(|x| 2^(23 - e)), an integer in [0, 2^23], written in
// three balanced base-256 digits N = d1 2^16 + d2 2^8 + d3 with 0 <= d1 <= 128 and
// -128 <= d2, d3 <= 127 (signs carried by the digits). Every digit is an integer of at most
// 8 bits, held exactly by BF16. So x = 2^(e - 23) (d1 2^16 + d2 2^8 + d3) up to 2^-24 of
// the chunk's largest entry (about the rounding the FP32 block already carries).
//
// Exact accumulation. A product of two digits is an integer below 2^14 in magnitude,
// exact in the tensor core's FP32 accumulator. The digit pairs (s, t) are grouped by
// class w = s + t (0-based digits), whose weight is 2^(-8 w) relative to class 0; classes
// 0, 1, 2 are kept (6 digit products per 16 rows, one tensor-memory accumulator per class)
// and classes 3, 4 (products below 2^-22 of the leading term) are dropped. Per chunk a class
// accumulator holds at most 3 x 2^14 x 256 < 2^24 in magnitude, so its FP32 sums are
// exact integers. After each chunk the epilogue warps read the three accumulators from
// tensor memory, combine them into an FP32 pair, apply 2^(e_i + e_j) exactly and add them
// into a running FP32-pair sum (errors of a few 2^-39 of the chunk's largest product, no
// FP64 pipe). The result is the Gram matrix of the 23-bit rounded block with no error growth
// along Nd; the FP32-pair Gram of gram_df.cu remains the exact one. The 47-bit form combines a
// chunk's accumulators into one 64-bit integer, shifts it right by the chunk's exponents'
// distance from the columns' largest (E_i - e_i + E_j - e_j, rounded) and adds it to a 64-bit
// integer sum. A chunk is rounded to one unit of that sum, 2^(E_i + E_j - 54 + drop) (drop:
// log2 of a split's chunks, 8 at 96^3 x 128), also where the large values of the two columns
// lie in different chunks: the entry's error is absolute, over 6912 chunks about 2^-41 max|x_i|
// max|x_j|, which against the columns' norms is below FP64's rounding once they spread over some
// thousands of nodes.
//
// Layout and pipeline. A pre-pass (k_tc_digits) writes the digits of an operand in the
// shared-memory order the MMA reads (no swizzle, K-major, 8-row x 16-byte core matrices)
// as 8 KB blobs, one per (128-column block, 32-row step, digit), plus the exponents
// e(c, j). A CTA owns one 128 x 128 tile of G (Tc47: 128 x 64) over a range of chunks
// (split-K): warp 0 streams a step's blobs into a three-stage ring, A by one untiled bulk
// copy, B by one tiled copy that lays its digits side by side along N. One thread of warp 1
// issues the tcgen05.mma (M = 128, K = 16): per A digit s one MMA over the kept B digits
// 0 .. at once (Tc23: N = 384 as 256 + 128, then 256, then 128), which writes the class
// accumulators s .. side by side (384 tensor-memory columns) and reads the A digit once
// instead of once per product; it commits stage releases and chunk completions to mbarriers,
// and sixteen epilogue warps (four per tensor-memory lane quarter, the running sums in
// registers) flush every chunk. Partial tiles of the K splits are summed by a second kernel
// in a fixed order (deterministic). Every wait is bounded; on a timeout the kernel raises
// *err, drains its copies and MMAs (bounded), frees its tensor memory and returns.
//
// What bounds it. The MMAs of a 96^3 x 128 Tc47 launch need 0.26 ms at the tensor pipe's
// rate (21 products, N = 64 .. 256). Of its 0.73 ms the pipe was busy 44%: the issuing thread
// formed descriptors and tested barriers for longer than a step's MMAs took, B's 1 KB pieces
// came in twelve requests a step, and every chunk waited for the epilogue's sums of pairs.
// Uniform issue, one copy for B, 32-row steps and 64-bit integer sums of which only the
// combination is waited for: 0.47 ms (128^3 x 512, two slabs, M and H: 33.8 -> 21 ms). What
// is left is that wait, about 2000 cycles a chunk beside 5400 of MMAs (the class accumulators
// fill 384 of the 512 columns, so no second set fits).
#include "device_once.cuh"
#include "internal.cuh"

#include <algorithm>
#include <cstring>
#include "tma.cuh"

#include <cstdint>
#include <cuda_bf16.h>

namespace sparc {

namespace {
constexpr int kTile = 128;                     // MMA M (A columns per tile)
constexpr int kEpiWarps = 16;                  // four per tensor-memory lane quarter
constexpr int kThreads = 32 * (2 + kEpiWarps);
constexpr unsigned kWaitLimit = 1u << 22;
constexpr int kTmemCols = 512;
constexpr int kNonFinite = INT32_MAX;          // exponent sentinel of a chunk with Inf/NaN
constexpr int kZeroExp = -4096;                // exponent of an all-zero chunk column
// core-matrix offsets inside a blob (elements): K-adjacent cores 2048 B apart, M/N-adjacent
// cores 128 B apart
constexpr unsigned kLbo = 2048, kSbo = 128;
}  // namespace

// The representations. Tc23: entries rounded to 23 bits of the chunk's largest, three
// base-256 digits, classes 0..2, 256-row chunks, 128 x 128 tiles (sparc_gram_tc, the mixed
// form's rotation). Tc47: 47 bits, six base-256 digits, classes 0..5 (21 digit products per
// 16 rows, issued as 8 MMAs of N = 64 .. 256 over the digit-concatenated B; a class sums at
// most six digit products, so 128-row chunks keep it below 2^24), 128 x 64 half tiles (six
// class accumulators of 64 columns fit the 512 tensor-memory columns): the Gram pairs of
// both forms and the FP64 form's rotation. The digit base is a
// parameter (kBase bits); kScale = kBits - kBase (kDigits - 1), so that
// x = 2^(e - kScale) sum_s d_s 2^(-kBase s).
struct Tc23 {
    static constexpr int kDigits = 3, kClasses = 3, kBits = 23, kChunk = 256, kStep = 32,
                         kN = 128, kStages = 3, kBase = 8;
    static constexpr bool kPair = true;   // epilogue sums as FP32 pairs
};
struct Tc47 {
    static constexpr int kDigits = 6, kClasses = 6, kBits = 47, kChunk = 128, kStep = 32,
                         kN = 64, kStages = 3, kBase = 8;
    static constexpr bool kPair = false;  // as 64-bit integers
};
// A stage holds A's blobs (all 128 columns of each digit) and the kN columns of B's blobs
// this CTA multiplies. B is stored digit-concatenated: per 8-row K group, the kN / 8 core
// matrices of digit 0, then those of digit 1, ... (kDigits kN columns, each piece copied
// from one contiguous run of a blob's K group), so that one MMA with N = nb kN multiplies
// an A digit by nb consecutive B digits at once and writes the nb class accumulators that
// sit side by side in tensor memory. B's K-adjacent cores are kDigits kN 16 B apart.
template <class C> struct TcDims {
    static constexpr int kStepsPerChunk = C::kChunk / C::kStep;
    static constexpr int kBlobElems = kTile * C::kStep;                    // BF16 per blob
    static constexpr unsigned kOperandBytes = C::kDigits * kBlobElems * 2;
    static constexpr unsigned kBPiece = C::kN * 16;            // one digit's cores of a K group
    static constexpr unsigned kBLbo = C::kDigits * kBPiece;     // B K-group stride
    static constexpr unsigned kBOperandBytes = C::kDigits * C::kN * C::kStep * 2;
    static constexpr unsigned kStageBytes = kOperandBytes + kBOperandBytes;
    static constexpr int kHalves = kTile / C::kN;                          // CTAs per tile
    static constexpr int kEpiCols = C::kN / (kEpiWarps / 4);              // per epilogue warp
    // ring, then (Tc23) the low parts of the epilogue's running pair sums ([warp][column][lane])
    static constexpr unsigned kLowBytes = C::kPair ? kEpiWarps * kEpiCols * 32 * 4 : 0;
    static constexpr unsigned kSmemBytes = C::kStages * kStageBytes + kLowBytes + 1024;
    static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
    static_assert(C::kClasses * C::kN <= kTmemCols, "class accumulators exceed tensor memory");
    static_assert(C::kBits <= C::kBase * C::kDigits - 1,
                  "top digit must stay within [0, 2^(kBase - 1)]");
    // a class sums at most kClasses digit products of magnitude <= 2^(2 kBase - 2) per row:
    // exact in the FP32 accumulator over a chunk
    static_assert(((long)C::kClasses << (2 * C::kBase - 2)) * C::kChunk < (1L << 24),
                  "class sums of a chunk must stay exact in FP32");
    static constexpr int kScale = C::kBits - C::kBase * (C::kDigits - 1);
    // Tc47: the epilogue's integer T = sum_w class_w 2^(8 (5 - w)), below 2^61.1, counts
    // 2^(e_i + e_j - kUnit)
    static constexpr int kUnit = 2 * kScale + C::kBase * (C::kClasses - 1);
};

namespace {
template <class C>
__device__ __forceinline__ long blob_offset(int cb, long step, int s, long nstep)
{
    return (((long)cb * nstep + step) * C::kDigits + s) * TcDims<C>::kBlobElems;
}

__device__ __forceinline__ int in_blob(int k, int c)  // k: row in step, c: column (0..127)
{
    return ((((k >> 3) * 16 + (c >> 3)) * 8 + (c & 7)) * 8) + (k & 7);
}

// |x| as an unsigned integer (monotonic in |x| for finite x), exponent bits and significand
template <typename T> struct FBits;
template <> struct FBits<float> {
    using U = uint32_t;
    static constexpr int kMant = 23, kBias = 127, kExpMask = 0xFF;
    __device__ static U mag(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
    __device__ static bool neg(float x) { return (__float_as_uint(x) >> 31) != 0; }
};
template <> struct FBits<double> {
    using U = unsigned long long;
    static constexpr int kMant = 52, kBias = 1023, kExpMask = 0x7FF;
    __device__ static U mag(double x) { return (U)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull; }
    __device__ static bool neg(double x) { return __double_as_longlong(x) < 0; }
};
}  // namespace

// |x| (bit pattern mag) on the grid of exponent e: round(|x| 2^(kBits - e)), in [0, 2^kBits].
template <class C, typename T>
__device__ __forceinline__ unsigned long long grid_value(typename FBits<T>::U mag, int e)
{
    using B = FBits<T>;
    using U = typename B::U;
    if (mag == 0) return 0ull;
    const int bx = (int)(mag >> B::kMant);
    const U m = (mag & (((U)1 << B::kMant) - 1)) | (bx ? ((U)1 << B::kMant) : 0);
    const int sh = e + B::kBias + B::kMant - C::kBits - (bx ? bx : 1);
    if (sh <= 0) return (unsigned long long)m << (-sh);  // exact: FP32 inputs of the 47-bit form
    if (sh < 8 * (int)sizeof(U)) return (unsigned long long)((m + ((U)1 << (sh - 1))) >> sh);
    return 0ull;
}

// exponent of a chunk column from its largest magnitude: |x| < 2^e
template <typename T>
__device__ __forceinline__ int chunk_exponent(typename FBits<T>::U mx)
{
    using B = FBits<T>;
    const int bx = (int)(mx >> B::kMant);
    return mx == 0 ? kZeroExp : (bx == 0 ? 2 - B::kBias : bx - B::kBias + 1);
}

// The digits of eight grid values N (sign bit t of neg) as BF16, eight K-adjacent elements (16
// bytes) per digit, digit s to dst + s stride. Adding 128 at every lower digit's place makes the
// balanced digits the bytes of the sum minus 128 (the top digit, at most 128, is the byte as it
// is): a byte permutation puts each into the significand of 1.5 2^23, one multiply-add takes
// the offset off and applies the sign, and the upper half of the FP32 result is the BF16.
template <class C>
__device__ __forceinline__ void store_digits(const unsigned long long (&N)[8], unsigned neg,
                                             __nv_bfloat16 *dst, long stride)
{
    static_assert(C::kBase == 8 && C::kDigits <= 8, "byte digits");
    constexpr unsigned long long kBias = 0x8080808080808080ull >> (64 - 8 * (C::kDigits - 1));
    constexpr float kM = 12582912.0f;  // 1.5 * 2^23, bits 0x4B400000
    unsigned lo[8], hi[8];
    float sg[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const unsigned long long n = N[t] + kBias;
        lo[t] = (unsigned)n;
        hi[t] = (unsigned)(n >> 32);
        sg[t] = ((neg >> t) & 1u) ? -1.0f : 1.0f;
    }
#pragma unroll
    for (int s = 0; s < C::kDigits; ++s) {
        const int byte = C::kDigits - 1 - s;
        const float off = -(kM + (s ? 128.0f : 0.0f));
        unsigned f[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const unsigned x = __byte_perm(byte < 4 ? lo[t] : hi[t], 0x4B400000u, 0x7650u | (byte & 3));
            f[t] = __float_as_uint(fmaf(__uint_as_float(x), sg[t], off * sg[t]));
        }
        uint4 v;
        v.x = __byte_perm(f[0], f[1], 0x7632);
        v.y = __byte_perm(f[2], f[3], 0x7632);
        v.z = __byte_perm(f[4], f[5], 0x7632);
        v.w = __byte_perm(f[6], f[7], 0x7632);
        *reinterpret_cast<uint4 *>(dst + s * stride) = v;
    }
}

// Eight consecutive rows of a column from row k (zero past nd); vec: 16-byte loads allowed.
template <typename T>
__device__ __forceinline__ void load8(const T *X, long k, long nd, bool live, bool vec, T (&x)[8])
{
    if (live && vec && k + 8 <= nd) {
        constexpr int W = 16 / sizeof(T);
#pragma unroll
        for (int u = 0; u < 8 / W; ++u) {
            const uint4 v = *reinterpret_cast<const uint4 *>(X + k + W * u);
            memcpy(&x[W * u], &v, 16);
        }
    } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = live && k + t < nd ? X[k + t] : (T)0;
    }
}

// Digits and exponents of one operand. CTA: one chunk (blockIdx.y) x 8 or 16 columns
// (blockIdx.x); a thread takes eight consecutive rows of a column, so its loads are whole
// sectors and its stores 16 bytes per digit, 128 contiguous bytes per eight columns (a row
// per lane stored two bytes at a time: 0.50 ms for a 96^3 x 128 FP64 block, 0.38 ms so).
// Rows past nd and columns past ns are zero; a chunk column holding Inf or NaN gets the
// exponent kNonFinite. EX[col] is raised to the column's largest exponent.
template <class C, typename T>
__global__ void __launch_bounds__(256)
k_tc_digits(const T *__restrict__ X, long ld, long nd, int ns, long nstep, bool vec,
            __nv_bfloat16 *__restrict__ D, int *__restrict__ E, int *__restrict__ EX, int ns_pad)
{
    using B = FBits<T>;
    using U = typename B::U;
    constexpr int kKg = C::kChunk / 8, kCols = 256 / kKg, kWarpsPer = C::kChunk / 32;
    static_assert(kCols * kKg == 256 && kCols % 8 == 0, "threads of a chunk");
    __shared__ U red[8][8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c8 = tid & 7, kg = (tid >> 3) % kKg, grp = tid / (8 * kKg);
    const int col = blockIdx.x * kCols + grp * 8 + c8;
    const long chunk = blockIdx.y, k = chunk * C::kChunk + kg * 8;
    T x[8];
    load8(X + (long)(col < ns ? col : 0) * ld, k, nd, col < ns, vec, x);
    U mx = 0;
    unsigned neg = 0u;
    const U inf = (U)B::kExpMask << B::kMant;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const U m = B::mag(x[t]);
        mx = m > mx ? m : mx;
        neg |= (B::neg(x[t]) ? 1u : 0u) << t;
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
        const U t = (U)__shfl_xor_sync(0xffffffffu, (unsigned long long)mx, o);
        mx = t > mx ? t : mx;
    }
    if (lane < 8) red[warp][lane] = mx;
    __syncthreads();
    const int w0 = grp * kWarpsPer;
#pragma unroll
    for (int w = 0; w < kWarpsPer; ++w) mx = red[w0 + w][c8] > mx ? red[w0 + w][c8] : mx;
    const bool bad = mx >= inf;
    const int e = chunk_exponent<T>(mx);
    if (kg == 0 && col < ns_pad) {
        E[chunk * ns_pad + col] = bad ? kNonFinite : e;
        if (!bad && e > *(volatile int *)(EX + col)) atomicMax(EX + col, e);
    }
    if (col >= ns_pad) return;
    unsigned long long N[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) N[t] = bad ? 0ull : grid_value<C, T>(B::mag(x[t]), e);
    const int cb = col >> 7, c = col & 127;
    store_digits<C>(N, neg,
                    D + blob_offset<C>(cb, k / C::kStep, 0, nstep) + in_blob((int)(k % C::kStep), c),
                    TcDims<C>::kBlobElems);
}

// 2^(e - kScale) as an FP32 factor (the chunk scale 2^(e_i + e_j - 2 kScale) is applied as
// two such factors, each exact); 0 below the FP32 normal range, NaN for a non-finite chunk.
template <class C>
__device__ __forceinline__ float pow2_factor(int e)
{
    if (e == kNonFinite) return __int_as_float(0x7FC00000);
    const int b = e - TcDims<C>::kScale + 127;
    if (b <= 0) return 0.0f;
    if (b >= 255) return __int_as_float(0x7F800000);
    return __int_as_float(b << 23);
}

__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// a 2^sc as FP64, rounded to nearest, by integer operations (an FP64 instruction per output
// would load the FP64 pipe); below the normal range 0, above it Inf.
__device__ __forceinline__ double scaled_to_double(long long a, int sc)
{
    const unsigned long long sgn = (unsigned long long)a & 0x8000000000000000ull;
    const unsigned long long m = (unsigned long long)(a < 0 ? -a : a);
    if (m == 0) return 0.0;
    const int lz = __clzll((long long)m);
    const unsigned long long t = m << lz;
    const unsigned long long r = (t >> 11) + ((t >> 10) & 1ull);  // 53 bits, hidden bit included
    const int e = 1023 + 63 - lz + sc;
    if (e <= 0) return 0.0;
    if (e >= 2047) return __longlong_as_double((long long)(sgn | 0x7ff0000000000000ull));
    return __longlong_as_double((long long)(sgn | (((unsigned long long)(e - 1) << 52) + r)));
}

// The chunk's integer T from Tc47's class sums (exact integers in FP32, below 2^21, 2^22, 2^22.6,
// 2^23, 2^23.4, 2^23.6). Integers up to 2^22 come out of the significand of 1.5 2^23 + v, larger
// ones by conversion; the last two classes, as 2^8 f4 + f5 = 2^10 t + g with t = f4 / 4 rounded
// and the exact remainder g, are rounded to 4 units, 2^-50 of the largest product (rounded to
// 2^10 in one step they cost four operations less, and columns whose largest values stand out by
// 2^20 and more, where the sums are far below T's range, lost bits that the digits hold).
__device__ __forceinline__ long long class_sum47(const uint32_t (&v)[6])
{
    constexpr float kM = 12582912.0f;
    auto f = [&](int w) { return __uint_as_float(v[w]); };
    const int b0 = __float_as_int(f(0) + kM), b1 = __float_as_int(f(1) + kM);
    const int i1 = (int)(((unsigned)b0 << 8) + (unsigned)b1 - (0x40000000u + 0x4B400000u));
    const int i2 = (int)(((unsigned)__float2int_rn(f(2)) << 8) + (unsigned)__float2int_rn(f(3)));
    const float t = fmaf(f(4), 0.25f, kM);
    const float g = fmaf(fmaf(t - kM, -4.0f, f(4)), 256.0f, f(5));  // below 2^23.7: exact
    const float l = fmaf(g, 0.25f, kM);
    const int i3 = (int)(((unsigned)__float_as_int(t) << 8) + (unsigned)__float_as_int(l) -
                         (0x40000000u + 0x4B400000u));
    return ((long long)i1 << 32) + ((long long)i2 * 65536 + (long long)i3 * 4);
}

// Digits of the transposed operand: B = Y^T for the rotation, so the K dimension runs over
// Y's columns and each Y row gets its own exponent per chunk of kChunk columns. CTA: 32
// rows (lanes) x 16 warps, each with one or two groups of 8 columns: loads are coalesced
// across lanes, the row's largest entry (as the word that holds its exponent) is found by shared
// memory maxima, and each thread writes its 8 values of a digit as one 16-byte store (the 8
// K-adjacent elements of a core matrix row are contiguous, and the 32 rows of a warp fill 512
// contiguous bytes). Rows past nd and columns past ns are zero. Bounded by its reads and writes;
// with every thread reading all warps' 64-bit maxima, and the 256-column chunks in CTAs of 1024
// threads of which one fits an SM, 2.7 ms for half of 128^3 x 512 FP64 to 23 bits, 1.23 ms so.
constexpr int kDigitTWarps = 16;
template <class C, typename T>
__global__ void __launch_bounds__(32 * kDigitTWarps)
k_tc_digits_t(const T *__restrict__ Y, long ld, long nd, int ns, long nstep,
              __nv_bfloat16 *__restrict__ D, int *__restrict__ E, long nd_pad)
{
    using B = FBits<T>;
    using U = typename B::U;
    constexpr int P = C::kChunk / 8 / kDigitTWarps;  // column groups of a thread
    static_assert(P * 8 * kDigitTWarps == C::kChunk, "whole groups");
    constexpr int kWordShift = 8 * (int)sizeof(T) - 32;
    __shared__ unsigned red[32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    if (g == 0) red[lane] = 0u;
    const long row = (long)blockIdx.x * 32 + lane;
    const long chunk = blockIdx.y;
    const bool live = row < nd;
    T x[P][8];
    U mx = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int kb = (int)(chunk * C::kChunk) + (g + kDigitTWarps * q) * 8;
#pragma unroll
        for (int t = 0; t < 8; ++t)
            x[q][t] = (live && kb + t < ns) ? Y[row + (long)(kb + t) * ld] : (T)0;
    }
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const U m = B::mag(x[q][t]);
            mx = m > mx ? m : mx;
        }
    // the word with the exponent; a value below its last bit counts as that bit (not zero)
    const unsigned word = (unsigned)(mx >> kWordShift);
    __syncthreads();
    atomicMax(&red[lane], word ? word : mx != 0 ? 1u : 0u);
    __syncthreads();
    const unsigned top = red[lane];
    const bool bad = top >= (unsigned)(((U)B::kExpMask << B::kMant) >> kWordShift);
    const int e = top == 1u ? 2 - B::kBias : chunk_exponent<T>((U)top << kWordShift);
    if (g == 0 && row < nd_pad) E[chunk * nd_pad + row] = bad ? kNonFinite : e;
    if (row >= nd_pad) return;
    const int cb = (int)(row >> 7), c = (int)(row & 127);
#pragma unroll
    for (int q = 0; q < P; ++q) {
        unsigned long long N[8];
        unsigned neg = 0u;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            N[t] = bad ? 0ull : grid_value<C, T>(B::mag(x[q][t]), e);
            neg |= (B::neg(x[q][t]) ? 1u : 0u) << t;
        }
        // the 8 columns kb .. kb+7 lie in one K-step (kStep is a multiple of 8) and one core
        const int kb = (int)(chunk * C::kChunk) + (g + kDigitTWarps * q) * 8;
        store_digits<C>(N, neg,
                        D + blob_offset<C>(cb, kb / C::kStep, 0, nstep) + in_blob(kb % C::kStep, c),
                        TcDims<C>::kBlobElems);
    }
}

// tiles[t] = (A column block, B column block); a tile is computed by kHalves CTAs, each
// for kN of its 128 B columns. part: nsplit x ntiles x 128 x 128 doubles, element (r, c) of
// a tile at r * 128 + c (r: A column, c: B column).
// Work units: a unit is one tile half (kN of the tile's 128 B columns) over a range of
// chunks. Gram mode: CTA b owns unit b (units = halves x tiles x splits); the tiles from ntiles1
// on are those of a second Gram with the same A (M_s and H_s of a Rayleigh-Ritz step in one
// launch: half as many splits to add up, and one launch and reduction less, a tenth of the step
// at 24^3 x 12). ROT (the rotation,
// see rotate_tc below): tile t is (t / mblk, t % mblk) over all chunks (mblk = B blocks, so
// the units that share an A block run side by side and find it in L2), the CTAs are
// persistent and walk units b, b + gridDim.x, ... with the ring, the MMAs and the epilogue
// running on across units; A's and B's exponents have the row strides ea_ld and eb_ld, and
// the epilogue writes out[i + j ldo] (i: A column, j: B column) for i < nrow, j < ncol, a
// warp's lanes covering 32 consecutive i (coalesced).
template <class C, bool ROT, typename TO = double>
__global__ void __launch_bounds__(kThreads, 1)
k_gram_tc(const __nv_bfloat16 *__restrict__ DA, const int *__restrict__ EA,
          const __grid_constant__ CUtensorMap mapB, const int *__restrict__ EB, int ns_pad, long nstep,
          const int2 *__restrict__ tiles, int ntiles, int nsplit, double *__restrict__ part,
          int drop, int *err, const int *__restrict__ EXA, const int *__restrict__ EXB,
          const __grid_constant__ CUtensorMap mapB2, const int *__restrict__ EB2,
          const int *__restrict__ EXB2, int ntiles1, int eb_ld = 0, int mblk = 1, TO *__restrict__ out = nullptr, long ldo = 0,
          long nrow = 0, int ncol = 0, long ea_ld = 0)
{
    using Dm = TcDims<C>;
    constexpr int kStages = C::kStages, kStepsPerChunk = Dm::kStepsPerChunk;
    constexpr unsigned kStageBytes = Dm::kStageBytes, kOperandBytes = Dm::kOperandBytes;
    constexpr unsigned kBLbo = Dm::kBLbo;
    constexpr int kEpiCols = Dm::kEpiCols;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], acc_full, acc_empty, drain;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;

    unsigned char *smem =
        (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long nchunk = nstep / kStepsPerChunk;
    const long ea_stride = ROT ? ea_ld : ns_pad;
    const int nunits = ROT ? ntiles * Dm::kHalves : (int)gridDim.x;
    const int ustride = ROT ? (int)gridDim.x : nunits;
    struct Unit {
        int hf, tile, split;
        bool second;  // of the two Grams A^T B, A^T B2
        int2 tb;
        long c0, c1;
    };
    auto unit = [&](int u) {
        Unit w;
        w.hf = u % Dm::kHalves;
        w.tile = (u / Dm::kHalves) % ntiles;
        w.split = u / (Dm::kHalves * ntiles);
        w.second = !ROT && w.tile >= ntiles1;
        w.tb = ROT ? make_int2(w.tile / mblk, w.tile % mblk)
                   : tiles[w.second ? w.tile - ntiles1 : w.tile];
        w.c0 = ROT ? 0 : (long)w.split * nchunk / nsplit;
        w.c1 = ROT ? nchunk : (long)(w.split + 1) * nchunk / nsplit;
        return w;
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&acc_full, 1);
        mbar_init(&acc_empty, kEpiWarps);
        mbar_init(&drain, 1);
        mbar_fence_init();
        abort_flag = 0;
    }
    if (warp == 1) tmem_alloc(&tmem_base, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    auto fail = [&]() {
        abort_flag = 1;
        atomicExch(err, 1);
    };

    // Warps 0 and 1 run their loops whole, so that the counters and the operand descriptors are
    // uniform values; one lane issues. A step's MMAs take 672 (Tc47) or 768 cycles (Tc23), and a
    // single thread that formed 14 descriptors and tested two barriers between steps needed more
    // than that: the tensor pipe was idle 55% of the time.
    if (warp == 0) {
        // ---- producer: A and B blobs of each step into the ring, unit after unit ----
        // A's blobs are one run of memory; this unit's kN columns of B's digits come by one tiled
        // copy that puts them digit by digit within each K group (copied piece by piece they were
        // kDigits kGroups requests of 1 KB a step, which the copy unit does not serve in the time
        // of the MMAs: 605 us for the 96^3 x 128 block below, 524 us by one copy)
        unsigned j = 0;  // steps handed to the ring over all units
        int s = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < nunits && ok; u += ustride) {
            const Unit w = unit(u);
            const __nv_bfloat16 *src = DA + blob_offset<C>(w.tb.x, w.c0 * kStepsPerChunk, 0, nstep);
            int row = (int)((w.tb.y * nstep + w.c0 * kStepsPerChunk) * C::kDigits);
            const long n = (w.c1 - w.c0) * kStepsPerChunk;
            for (long st = 0; st < n; ++st) {
                ok = j < kStages || mbar_wait(&empty[s], (j / kStages & 1u) ^ 1u, kWaitLimit);
                ok = __all_sync(0xffffffffu, ok && !abort_flag);
                if (!ok) {
                    if (lane == 0) fail();
                    break;
                }
                if (lane == 0) {
                    unsigned char *dst = smem + (size_t)s * kStageBytes;
                    mbar_arrive_expect_tx(&full[s], kStageBytes);
                    bulk_load(dst, src, kOperandBytes, &full[s]);
                    tma_load_3d(dst + kOperandBytes, w.second ? &mapB2 : &mapB, &full[s], w.hf * (C::kN * 2), row, 0);
                }
                __syncwarp();
                src += C::kDigits * Dm::kBlobElems;
                row += C::kDigits;
                ++j;
                s = s + 1 == kStages ? 0 : s + 1;
            }
        }
        if (abort_flag) {
            // wait (bounded) for the last copy issued into each stage
            for (int q = 0; q < kStages; ++q) {
                if (j <= (unsigned)q) break;
                const unsigned last = j - 1 - (j - 1 - q) % kStages;  // j-1 or less, = q mod kStages
                mbar_wait(&full[q], last / kStages & 1u, kWaitLimit);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issuer ----
        const uint64_t ad0 = smem_desc(smem, kLbo, kSbo);
        const uint64_t bd0 = smem_desc(smem + kOperandBytes, kBLbo, kSbo);
        const bool leader = lane == 0;
        unsigned j = 0, cc = 0;  // steps and chunks over all units
        int s = 0;
        bool ok = true, ready = false;  // ready: stage s is known to be full
        for (int u = blockIdx.x; u < nunits && ok; u += ustride) {
            const Unit w = unit(u);
            for (long c = w.c0; c < w.c1; ++c, ++cc) {
                if (cc > 0) {
                    ok = mbar_wait(&acc_empty, (cc - 1) & 1u, kWaitLimit) && !abort_flag;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_fence_after();
                }
#pragma unroll 1
                for (int kin = 0; kin < kStepsPerChunk; ++kin) {
                    if (!ready) {
                        ok = __all_sync(0xffffffffu,
                                        mbar_wait(&full[s], j / kStages & 1u, kWaitLimit));
                        if (!ok) break;
                    }
                    const uint64_t ads = ad0 + (unsigned)s * (kStageBytes >> 4);
                    const uint64_t bds = bd0 + (unsigned)s * (kStageBytes >> 4);
                    if (leader) {
#pragma unroll
                        for (int ks = 0; ks < C::kStep / 16; ++ks) {
#pragma unroll
                            for (int sa = 0; sa < C::kDigits; ++sa) {
                                // A digit sa times B digits 0 .. nb-1 (classes sa .. sa+nb-1, the
                                // kept ones), as MMAs of N <= 256 over the digit-concatenated B
                                const int nb = C::kClasses - sa < C::kDigits ? C::kClasses - sa
                                                                             : C::kDigits;
#pragma unroll
                                for (int n0 = 0; n0 < nb * C::kN; n0 += 256) {
                                    const int nl = nb * C::kN - n0 < 256 ? nb * C::kN - n0 : 256;
                                    // the sa = 0 MMAs cover every class: at a chunk start they
                                    // overwrite the accumulators, all later ones accumulate
                                    tc_mma_bf16(
                                        tmem + (uint32_t)(sa * C::kN + n0),
                                        ads + ((sa * Dm::kBlobElems * 2 + ks * 2 * kLbo) >> 4),
                                        bds + ((ks * 2 * kBLbo + (n0 / 8) * kSbo) >> 4),
                                        idesc_bf16_f32(kTile, nl), kin > 0 || ks > 0 || sa > 0);
                                }
                            }
                        }
                        tc_commit(&empty[s]);  // stage free once these MMAs are done
                        if (kin == kStepsPerChunk - 1) tc_commit(&acc_full);  // chunk complete
                    }
                    __syncwarp();
                    ++j;
                    s = s + 1 == kStages ? 0 : s + 1;
                    // (a stage past the last one never fills)
                    ready = __all_sync(0xffffffffu, mbar_test(&full[s], j / kStages & 1u));
                }
                if (!ok) break;
            }
        }
        if (leader) {
            if (!ok) fail();
            // all MMAs issued by this thread are complete before tensor memory is freed
            tc_commit(&drain);
            if (!mbar_wait(&drain, 0u, kWaitLimit)) fail();
        }
        __syncwarp();
    } else {
        const int q = warp & 3;                 // tensor-memory lane quarter of this warp
        const int hw = (warp - 2) >> 2;         // columns kEpiCols hw .. of this CTA's kN
        const int r = q * 32 + lane;            // tile row = A column within the block
        if constexpr (C::kPair) {
        // ---- epilogue: flush each chunk's class accumulators into FP32-pair sums ----
        float H[kEpiCols];
        float *Lw = reinterpret_cast<float *>(smem + (size_t)kStages * kStageBytes) +
                    (size_t)(warp - 2) * kEpiCols * 32 + lane;  // Lw[u * 32]: column u
        long cc = 0;  // chunks over all units
        bool ok = true;
        // the chunk exponents are loaded one chunk ahead (they do not depend on the MMAs):
        // this thread's A column, and kEpiCols / 32 of the warp's B columns per lane, whose
        // factors reach the other lanes by shuffle
        constexpr int kEB = kEpiCols / 32;
        const long eb_stride = ROT ? eb_ld : ns_pad;
        for (int u = blockIdx.x; u < nunits && ok; u += ustride) {
            const Unit w = unit(u);
            const long colA = (long)w.tb.x * kTile + r;
            const int *ebw = (w.second ? EB2 : EB) + (long)w.tb.y * kTile + w.hf * C::kN +
                             hw * kEpiCols + lane;
            int ea_n = EA[w.c0 * ea_stride + colA], eb_n[kEB];
#pragma unroll
            for (int k = 0; k < kEB; ++k) eb_n[k] = ebw[w.c0 * eb_stride + 32 * k];
            for (long c = w.c0; c < w.c1; ++c, ++cc) {
                const float fA = pow2_factor<C>(ea_n);
                float fb[kEB];
#pragma unroll
                for (int k = 0; k < kEB; ++k) fb[k] = pow2_factor<C>(eb_n[k]);
                if (c + 1 < w.c1) {
                    ea_n = EA[(c + 1) * ea_stride + colA];
#pragma unroll
                    for (int k = 0; k < kEB; ++k) eb_n[k] = ebw[(c + 1) * eb_stride + 32 * k];
                }
                ok = mbar_wait(&acc_full, (unsigned)(cc & 1), kWaitLimit) && !abort_flag;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    if (lane == 0) fail();
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < kEpiCols / 4; ++g) {
                    const uint32_t ta =
                        tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hw * kEpiCols + g * 4);
                    uint32_t v[C::kClasses][4];
#pragma unroll
                    for (int cl = 0; cl < C::kClasses; ++cl)
                        tmem_ld4(ta + (uint32_t)(cl * C::kN), v[cl]);
                    tmem_wait_ld();
                    if (g == kEpiCols / 4 - 1) {
                        // all sums are in registers: the next chunk's MMAs may start
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&acc_empty);
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        // class_0 + class_1 2^-8 + class_2 2^-16 as a pair: h rounds the
                        // first two, and h - class_0 is exact (a multiple of 2^-8 below 2^16),
                        // so the rest of class_1 is too; l is rounded to 2^-17 or better,
                        // 2^-39 of the largest sum
                        const float c0 = __uint_as_float(v[0][x]), c1 = __uint_as_float(v[1][x]);
                        const float h = fmaf(c1, 0x1p-8f, c0);
                        const float l = fmaf(__uint_as_float(v[2][x]), 0x1p-16f,
                                             fmaf(c1, 0x1p-8f, c0 - h));
                        const float f =
                            fA * __shfl_sync(0xffffffffu, fb[(g * 4 + x) / 32], (g * 4 + x) % 32);
                        if (c == w.c0) {  // the unit's first chunk: the sums are its own
                            H[g * 4 + x] = h * f;
                            Lw[(g * 4 + x) * 32] = l * f;
                        } else {
                            float sh, se;
                            two_sum_f(H[g * 4 + x], h * f, sh, se);
                            H[g * 4 + x] = sh;
                            Lw[(g * 4 + x) * 32] += fmaf(l, f, se);
                        }
                    }
                }
            }
            if (!ok) break;
            if (ROT) {
                const long i = (long)w.tb.x * kTile + r;
                const long j0 = (long)w.tb.y * kTile + w.hf * C::kN + hw * kEpiCols;
                if (i < nrow) {
                    TO *o = out + i + j0 * ldo;
#pragma unroll
                    for (int x = 0; x < kEpiCols; ++x) {
                        if (j0 + x >= ncol) continue;
                        o[(long)x * ldo] = H[x] + Lw[x * 32];  // the pair rounded to FP32
                    }
                }
            } else {
                double *o = part + ((long)w.split * ntiles + w.tile) * kTile * kTile +
                            (long)r * kTile + w.hf * C::kN + hw * kEpiCols;
#pragma unroll
                for (int x = 0; x < kEpiCols; ++x) o[x] = (double)H[x] + (double)Lw[x * 32];
            }
        }
        } else {
        // ---- epilogue: each chunk's class accumulators into 64-bit integer sums ----
        long long S[kEpiCols];
        long cc = 0;  // chunks over all units
        bool ok = true;
        // the chunk exponents are loaded one chunk ahead (they do not depend on the MMAs):
        // this thread's A column, and one of the warp's B columns per lane (lane mod kEpiCols),
        // whose shifts reach the other lanes by shuffle
        const long eb_stride = ROT ? eb_ld : ns_pad;
        for (int u = blockIdx.x; u < nunits && ok; u += ustride) {
            const Unit w = unit(u);
            const long colA = (long)w.tb.x * kTile + r;
            const long colB = (long)w.tb.y * kTile + w.hf * C::kN + hw * kEpiCols + lane % kEpiCols;
            const int *ebw = (w.second ? EB2 : EB) + colB;
#pragma unroll
            for (int x = 0; x < kEpiCols; ++x) S[x] = 0;
            // largest exponents over the chunks (the rotation's few chunks are looked at here)
            int xa = kZeroExp, xb = kZeroExp, bad = 0;
            if (ROT) {
                for (long c = w.c0; c < w.c1; ++c) {
                    const int e = EA[c * ea_stride + colA];
                    xa = max(xa, e == kNonFinite ? kZeroExp : e);
                    const int f = ebw[c * eb_stride];
                    xb = max(xb, f == kNonFinite ? kZeroExp : f);
                }
            } else {
                xa = max(xa, EXA[colA]);
                xb = max(xb, (w.second ? EXB2 : EXB)[colB]);
            }
            int ea_n = EA[w.c0 * ea_stride + colA], eb_n = ebw[w.c0 * eb_stride];
            for (long c = w.c0; c < w.c1; ++c, ++cc) {
                // shifts less one, and flags of chunks holding Inf or NaN (bit 0 this row's, bit 1
                // the lane's column)
                if (ea_n == kNonFinite) bad |= 1, ea_n = xa;
                const int sa = xa - ea_n + drop - 1;
                if (eb_n == kNonFinite) bad |= 2, eb_n = xb;
                const int sb = xb - eb_n;
                if (c + 1 < w.c1) {
                    ea_n = EA[(c + 1) * ea_stride + colA];
                    eb_n = ebw[(c + 1) * eb_stride];
                }
                ok = mbar_wait(&acc_full, (unsigned)(cc & 1), kWaitLimit) && !abort_flag;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    if (lane == 0) fail();
                    break;
                }
                tc_fence_after();
                // all of the chunk's integers first, so that the next chunk's MMAs may start ...
                long long T[kEpiCols];
#pragma unroll
                for (int g = 0; g < kEpiCols / 4; ++g) {
                    const uint32_t ta =
                        tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hw * kEpiCols + g * 4);
                    uint32_t v[C::kClasses][4];
#pragma unroll
                    for (int cl = 0; cl < C::kClasses; ++cl)
                        tmem_ld4(ta + (uint32_t)(cl * C::kN), v[cl]);
                    tmem_wait_ld();
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        uint32_t vx[C::kClasses];
#pragma unroll
                        for (int cl = 0; cl < C::kClasses; ++cl) vx[cl] = v[cl][x];
                        T[g * 4 + x] = class_sum47(vx);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty);
                // ... then, beside them, T 2^-(sh + 1), rounded, into the sums
#pragma unroll
                for (int x = 0; x < kEpiCols; ++x) {
                    const int sh = sa + __shfl_sync(0xffffffffu, sb, x);
                    S[x] += ((T[x] >> min((unsigned)sh, 62u)) + 1) >> 1;
                }
            }
            if (!ok) break;
            const int unit_e = xa - Dm::kUnit + drop;  // 2^(unit_e + xb): the value of one
            const long i = (long)w.tb.x * kTile + r;
            const long j0 = (long)w.tb.y * kTile + w.hf * C::kN + hw * kEpiCols;
            TO *o = ROT ? out + i + j0 * ldo : nullptr;
            double *pt = ROT ? nullptr
                             : part + ((long)w.split * ntiles + w.tile) * kTile * kTile +
                                   (long)r * kTile + w.hf * C::kN + hw * kEpiCols;
#pragma unroll
            for (int x = 0; x < kEpiCols; ++x) {
                const int sc = unit_e + __shfl_sync(0xffffffffu, xb, x);
                const int fb = __shfl_sync(0xffffffffu, bad, x);
                const bool nan = (bad & 1) || (fb & 2);
                if (ROT) {
                    if (i >= nrow || j0 + x >= ncol) continue;
                    o[(long)x * ldo] = nan ? __longlong_as_double(0x7ff8000000000000ll)
                                           : scaled_to_double(S[x], sc);
                } else {
                    pt[x] = nan ? __longlong_as_double(0x7ff8000000000000ll)
                                : scaled_to_double(S[x], sc);
                }
            }
        }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// G (tiles below ntiles1) and G2 from the split partials, summed in split order, eight loads in
// flight; sym mirrors each off-diagonal tile.
__global__ void k_gram_tc_reduce(const double *__restrict__ part, const int2 *__restrict__ tiles,
                                 int ntiles, int ntiles1, int nsplit, int ns, bool sym, double *G,
                                 double *G2)
{
    constexpr int kU = 8;
    const long tot = (long)ntiles * kTile * kTile;
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < tot;
         t += (long)gridDim.x * blockDim.x) {
        const int tile = (int)(t / (kTile * kTile));
        const int e = (int)(t % (kTile * kTile));
        const int r = e / kTile, c = e % kTile;
        const int2 tb = tiles[tile < ntiles1 ? tile : tile - ntiles1];
        const int i = tb.x * kTile + r, j = tb.y * kTile + c;
        if (i >= ns || j >= ns) continue;
        const double *p = part + (long)tile * kTile * kTile + e;
        const long step = (long)ntiles * kTile * kTile;
        double v = 0.0;
        for (int s0 = 0; s0 < nsplit; s0 += kU) {
            double x[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) x[u] = s0 + u < nsplit ? p[(s0 + u) * step] : 0.0;
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (s0 + u < nsplit) v += x[u];
        }
        double *g = tile < ntiles1 ? G : G2;
        g[i + (long)j * ns] = v;
        if (sym && tb.x != tb.y) g[j + (long)i * ns] = v;
    }
}

// ---- host side -------------------------------------------------------------------------

namespace {
struct TcPlan {
    int ns_pad, nblk, ntiles1, ntiles, nsplit;  // tiles of one Gram, of all
    int drop;  // right shift of a chunk's integer: the chunks of a unit add up below 2^63
    long nstep, nchunk;
    size_t digits_bytes, exps_bytes, part_bytes, tiles_bytes;
};

int log2_ceil(long n)
{
    int b = 0;
    while ((1L << b) < n) ++b;
    return b;
}

template <class C>
TcPlan tc_plan(long nd, int ns, bool sym, int grams = 1)
{
    TcPlan p;
    p.nblk = (ns + kTile - 1) / kTile;
    p.ns_pad = p.nblk * kTile;
    p.nchunk = (nd + C::kChunk - 1) / C::kChunk;
    p.nstep = p.nchunk * TcDims<C>::kStepsPerChunk;
    p.ntiles1 = sym ? p.nblk * (p.nblk + 1) / 2 : p.nblk * p.nblk;
    p.ntiles = grams * p.ntiles1;
    // K splits: one CTA per SM (the ring and the class accumulators fill an SM), so the
    // kernel takes (waves of 152 CTAs) x (chunks per split). Pick the split count with the
    // fewest chunk-times, counting about two chunks of fixed cost per CTA (set-up and the
    // partial tile's store), and keep the partial tiles within 256 MB.
    const long ctas = (long)p.ntiles * TcDims<C>::kHalves;
    const long smax_mem = ((long)256 << 20) / ((long)p.ntiles * kTile * kTile * 8);
    long smax = p.nchunk < smax_mem ? p.nchunk : smax_mem;
    if (smax > 1024) smax = 1024;
    long best_s = 1, best = -1;
    for (long s = 1; s <= smax; ++s) {
        const long waves = (ctas * s + 151) / 152;
        const long cost = waves * ((p.nchunk + s - 1) / s + 2);
        if (best < 0 || cost < best) best = cost, best_s = s;
    }
    p.nsplit = (int)best_s;
    p.drop = std::max(1, log2_ceil((p.nchunk + best_s - 1) / best_s));
    p.digits_bytes = (size_t)C::kDigits * p.ns_pad * p.nstep * C::kStep * 2;
    p.exps_bytes = (size_t)(p.nchunk + 1) * p.ns_pad * sizeof(int);  // then the largest per column
    p.part_bytes = (size_t)p.nsplit * p.ntiles * kTile * kTile * sizeof(double);
    p.tiles_bytes = (size_t)p.ntiles1 * sizeof(int2);
    return p;
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

template <class C>
size_t tc_workspace(long nd, int ns, bool same_operand, bool sym, int grams = 1)
{
    const TcPlan p = tc_plan<C>(nd, ns, sym, grams);
    const int nops = same_operand ? 1 : 2;
    return nops * (align256(p.digits_bytes) + align256(p.exps_bytes)) + align256(p.part_bytes) +
           align256(p.tiles_bytes);
}
}  // namespace

size_t gram_tc_workspace(long nd, int ns, bool same_operand, bool sym)
{
    return tc_workspace<Tc23>(nd, ns, same_operand, sym);
}
size_t gram_tc47_workspace(long nd, int ns) { return tc_workspace<Tc47>(nd, ns, false, true, 2); }

// 16-byte loads along a column
template <typename T>
static bool tc_vec(const T *X, long ld)
{
    return ((uintptr_t)X & 15u) == 0 && ld % (long)(16 / sizeof(T)) == 0;
}

template <class C, typename T>
static cudaError_t tc_digits(const T *X, long ld, long nd, int ns, const TcPlan &p,
                             __nv_bfloat16 *D, int *E, cudaStream_t st)
{
    if (p.nchunk > 65535) return cudaErrorInvalidValue;
    int *EX = E + p.nchunk * p.ns_pad;
    const cudaError_t e = cudaMemsetAsync(EX, 0x80, sizeof(int) * (size_t)p.ns_pad, st);
    if (e != cudaSuccess) return e;
    dim3 grid(p.ns_pad / (2048 / C::kChunk), (unsigned)p.nchunk);
    k_tc_digits<C, T><<<grid, 256, 0, st>>>(X, ld, nd, ns, p.nstep, tc_vec(X, ld), D, E, EX,
                                            p.ns_pad);
    note_launch();
    return cudaGetLastError();
}

// A digit buffer of nblk column blocks as (16-byte units of a K group's 128 columns taken as
// 8-byte words, digit of a step, K group of a step), with the box of one CTA's B operand. The
// box starts at a multiple of its width, so the x coordinate is a multiple of 1 KB.
template <class C>
static cudaError_t tc_map(CUtensorMap &m, const __nv_bfloat16 *D, long nblk, long nstep)
{
    constexpr int kGroups = C::kStep / 8;
    PFN_cuTensorMapEncodeTiled_v12000 enc;
    const cudaError_t e = tensor_map_encoder(enc);
    if (e != cudaSuccess) return e;
    const long rows = nblk * nstep * C::kDigits;
    if (rows > 0x7fffffffL) return cudaErrorInvalidValue;
    cuuint64_t dims[3] = {kTile * 2, (cuuint64_t)rows, kGroups};
    cuuint64_t strides[2] = {(cuuint64_t)TcDims<C>::kBlobElems * 2, kTile * 16};
    cuuint32_t box[3] = {C::kN * 2, C::kDigits, kGroups}, estr[3] = {1, 1, 1};
    return enc(&m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, (void *)D, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess
               : cudaErrorInvalidValue;
}

// Tile list (host-built, uploaded) and the kernel's shared-memory attribute.
template <class C>
static cudaError_t tc_prepare(const TcPlan &p, bool sym, int2 *tiles, cudaStream_t st)
{
    static DeviceOnce once;
    const cudaError_t e = once.allow_smem((int)TcDims<C>::kSmemBytes, k_gram_tc<C, false>);
    if (e != cudaSuccess) return e;
    static thread_local int2 host_tiles[64 * 65 / 2 + 64 * 64];
    if (p.ntiles1 > (int)(sizeof(host_tiles) / sizeof(int2))) return cudaErrorInvalidValue;
    int n = 0;
    for (int a = 0; a < p.nblk; ++a)
        for (int b = (sym ? a : 0); b < p.nblk; ++b) host_tiles[n++] = make_int2(a, b);
    return cudaMemcpyAsync(tiles, host_tiles, p.tiles_bytes, cudaMemcpyHostToDevice, st);
}

// G = A^T B and, for a plan of two Grams, G2 = A^T B2
template <class C>
static cudaError_t tc_run(const TcPlan &p, const __nv_bfloat16 *DA, const int *EA,
                          const __nv_bfloat16 *DB, const int *EB, const __nv_bfloat16 *DB2,
                          const int *EB2, const int2 *tiles, double *part, int ns, bool sym,
                          double *G, double *G2, int *err, cudaStream_t st)
{
    const int ctas = p.ntiles * p.nsplit * TcDims<C>::kHalves;
    const long ex = p.nchunk * p.ns_pad;
    CUtensorMap mapB, mapB2;
    cudaError_t e = tc_map<C>(mapB, DB, p.nblk, p.nstep);
    if (e == cudaSuccess) e = tc_map<C>(mapB2, DB2, p.nblk, p.nstep);
    if (e != cudaSuccess) return e;
    k_gram_tc<C, false><<<ctas, kThreads, TcDims<C>::kSmemBytes, st>>>(
        DA, EA, mapB, EB, p.ns_pad, p.nstep, tiles, p.ntiles, p.nsplit, part, p.drop, err, EA + ex,
        EB + ex, mapB2, EB2, EB2 + ex, p.ntiles1);
    note_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_gram_tc_reduce<<<152 * 4, 256, 0, st>>>(part, tiles, p.ntiles, p.ntiles1, p.nsplit, ns, sym,
                                              G, G2);
    note_launch();
    return cudaGetLastError();
}

template <class C, typename TA, typename TB>
static cudaError_t gram_tc_impl(const TA *A, long lda, const TB *B, long ldb, long nd, int ns,
                                double *G, void *ws, size_t ws_bytes, bool sym, int *err,
                                cudaStream_t st)
{
    if (ns <= 0 || nd <= 0) return cudaErrorInvalidValue;
    const bool same = (const void *)A == (const void *)B && sizeof(TA) == sizeof(TB) && lda == ldb;
    const TcPlan p = tc_plan<C>(nd, ns, sym);
    if (ws_bytes < tc_workspace<C>(nd, ns, same, sym)) return cudaErrorInvalidValue;
    unsigned char *w = (unsigned char *)ws;
    auto take = [&](size_t b) {
        unsigned char *r = w;
        w += align256(b);
        return r;
    };
    __nv_bfloat16 *DA = (__nv_bfloat16 *)take(p.digits_bytes);
    int *EA = (int *)take(p.exps_bytes);
    __nv_bfloat16 *DB = DA;
    int *EB = EA;
    if (!same) {
        DB = (__nv_bfloat16 *)take(p.digits_bytes);
        EB = (int *)take(p.exps_bytes);
    }
    double *part = (double *)take(p.part_bytes);
    int2 *tiles = (int2 *)take(p.tiles_bytes);

    cudaError_t e;
    if ((e = tc_prepare<C>(p, sym, tiles, st)) != cudaSuccess) return e;
    if ((e = tc_digits<C, TA>(A, lda, nd, ns, p, DA, EA, st)) != cudaSuccess) return e;
    if (!same && (e = tc_digits<C, TB>(B, ldb, nd, ns, p, DB, EB, st)) != cudaSuccess) return e;
    return tc_run<C>(p, DA, EA, DB, EB, DB, EB, tiles, part, ns, sym, G, nullptr, err, st);
}

template <class C, typename TA, typename TB>
static cudaError_t gram_tc_pair_impl(const TA *A, long lda, const TB *B, long ldb, long nd,
                                     int ns, double *M, double *Hm, void *ws, size_t ws_bytes,
                                     int *err, cudaStream_t st)
{
    if (ns <= 0 || nd <= 0) return cudaErrorInvalidValue;
    const TcPlan p = tc_plan<C>(nd, ns, true, 2);
    if (ws_bytes < tc_workspace<C>(nd, ns, false, true, 2)) return cudaErrorInvalidValue;
    unsigned char *w = (unsigned char *)ws;
    auto take = [&](size_t b) {
        unsigned char *r = w;
        w += align256(b);
        return r;
    };
    __nv_bfloat16 *DA = (__nv_bfloat16 *)take(p.digits_bytes);
    int *EA = (int *)take(p.exps_bytes);
    __nv_bfloat16 *DB = (__nv_bfloat16 *)take(p.digits_bytes);
    int *EB = (int *)take(p.exps_bytes);
    double *part = (double *)take(p.part_bytes);
    int2 *tiles = (int2 *)take(p.tiles_bytes);
    cudaError_t e;
    if ((e = tc_prepare<C>(p, true, tiles, st)) != cudaSuccess) return e;
    if ((e = tc_digits<C, TA>(A, lda, nd, ns, p, DA, EA, st)) != cudaSuccess) return e;
    if ((e = tc_digits<C, TB>(B, ldb, nd, ns, p, DB, EB, st)) != cudaSuccess) return e;
    return tc_run<C>(p, DA, EA, DA, EA, DB, EB, tiles, part, ns, true, M, Hm, err, st);
}

template <typename TA, typename TB>
cudaError_t gram_tc(const TA *A, long lda, const TB *B, long ldb, long nd, int ns, double *G,
                    void *ws, size_t ws_bytes, bool sym, int *err, cudaStream_t st)
{
    return gram_tc_impl<Tc23, TA, TB>(A, lda, B, ldb, nd, ns, G, ws, ws_bytes, sym, err, st);
}


template <typename TA>
cudaError_t gram_tc47_pair(const TA *A, long lda, const double *B, long ldb, long nd, int ns,
                           double *M, double *Hm, void *ws, size_t ws_bytes, int *err,
                           cudaStream_t st)
{
    return gram_tc_pair_impl<Tc47, TA, double>(A, lda, B, ldb, nd, ns, M, Hm, ws, ws_bytes, err,
                                               st);
}
template cudaError_t gram_tc47_pair<double>(const double *, long, const double *, long, long, int,
                                            double *, double *, void *, size_t, int *,
                                            cudaStream_t);
template cudaError_t gram_tc47_pair<float>(const float *, long, const double *, long, long, int,
                                           double *, double *, void *, size_t, int *,
                                           cudaStream_t);

// ---- rotation out = Y C on the tensor cores -----------------------------------------------
// Written as the contraction G = A^T B with A = Y^T (K = Ns: Y's columns, M = Nd: Y's rows)
// and B = C (N = Ns): G(i, j) = sum_k Y_ik C_kj = out(i, j). Y gets exponents per (K chunk,
// row), C per (K chunk, column), so every product in a class accumulator shares one scale.
// K = Ns is short, so a unit is one tile (Tc47: a 128 x 64 half tile) over all of K; the
// tensor-memory lanes hold Y's rows, so each store of the epilogue covers 32 consecutive rows
// of a column. The FP64 form uses the 47-bit digits (FP64 blocks, FP64 output); the mixed
// form the 23-bit digits (FP32 block or the FP64 H Y of its residuals, FP32 output): each
// entry of Y and C is rounded to 2^-24 of its chunk's largest, the rounding an FP32 result
// carries anyway, for 6 digit products per 16 K instead of 21.
namespace {
struct RotPlan {
    int ns_pad, mblk;
    long nblk, nd_pad, nchunk, nstep;
    size_t da_bytes, ea_bytes, db_bytes, eb_bytes;
};
template <class C>
RotPlan rot_plan(long nd, int ns)
{
    RotPlan p;
    p.mblk = (ns + kTile - 1) / kTile;
    p.ns_pad = p.mblk * kTile;
    p.nblk = (nd + kTile - 1) / kTile;
    p.nd_pad = p.nblk * kTile;
    p.nchunk = (ns + C::kChunk - 1) / C::kChunk;
    p.nstep = p.nchunk * TcDims<C>::kStepsPerChunk;
    p.da_bytes = (size_t)C::kDigits * p.ns_pad * p.nstep * C::kStep * 2;
    p.ea_bytes = (size_t)(p.nchunk + 1) * p.ns_pad * sizeof(int);
    p.db_bytes = (size_t)C::kDigits * p.nd_pad * p.nstep * C::kStep * 2;
    p.eb_bytes = (size_t)p.nchunk * p.nd_pad * sizeof(int);
    return p;
}
template <class C>
size_t rot_workspace(long nd, int ns)
{
    const RotPlan p = rot_plan<C>(nd, ns);
    return align256(p.da_bytes) + align256(p.ea_bytes) + align256(p.db_bytes) +
           align256(p.eb_bytes);
}

template <class C, typename TY, typename TO>
cudaError_t rotate_tc_impl(const TY *Y, long ldy, long nd, int ns, const double *Cm, TO *out,
                           long ldo, void *ws, size_t ws_bytes, int *err, cudaStream_t st)
{
    if (ns <= 0 || nd <= 0) return cudaSuccess;
    const RotPlan p = rot_plan<C>(nd, ns);
    if (ws_bytes < rot_workspace<C>(nd, ns)) return cudaErrorInvalidValue;
    const long ctas = (long)p.mblk * p.nblk * TcDims<C>::kHalves;
    if (p.nchunk > 65535 || ctas > 0x7fffffffL || p.nd_pad / 32 > 0x7fffffffL)
        return cudaErrorInvalidValue;
    unsigned char *w = (unsigned char *)ws;
    auto take = [&](size_t b) {
        unsigned char *r = w;
        w += align256(b);
        return r;
    };
    __nv_bfloat16 *DA = (__nv_bfloat16 *)take(p.da_bytes);
    int *EA = (int *)take(p.ea_bytes);
    __nv_bfloat16 *DB = (__nv_bfloat16 *)take(p.db_bytes);
    int *EB = (int *)take(p.eb_bytes);
    static DeviceOnce once;
    cudaError_t e = once.allow_smem((int)TcDims<C>::kSmemBytes, k_gram_tc<C, true, TO>);
    if (e != cudaSuccess) return e;
    {   // A = C: K = Ns rows, M = Ns columns
        dim3 grid(p.ns_pad / (2048 / C::kChunk), (unsigned)p.nchunk);
        int *EX = EA + p.nchunk * p.ns_pad;  // (not used by the rotation)
        if ((e = cudaMemsetAsync(EX, 0x80, sizeof(int) * (size_t)p.ns_pad, st)) != cudaSuccess)
            return e;
        k_tc_digits<C, double><<<grid, 256, 0, st>>>(Cm, ns, ns, ns, p.nstep, tc_vec(Cm, ns), DA, EA,
                                                     EX, p.ns_pad);
        note_launch();
    }
    {   // B = Y^T: K = Ns (Y's columns), N = Nd (Y's rows)
        dim3 grid((unsigned)(p.nd_pad / 32), (unsigned)p.nchunk);
        k_tc_digits_t<C, TY><<<grid, 32 * kDigitTWarps, 0, st>>>(Y, ldy, nd, ns, p.nstep, DB,
                                                                    EB, p.nd_pad);
        note_launch();
    }
    const unsigned grid = (unsigned)(ctas < 152 ? ctas : 152);  // persistent, one per SM
    CUtensorMap mapB;
    if ((e = tc_map<C>(mapB, DA, p.mblk, p.nstep)) != cudaSuccess) return e;
    // A: Y's digits (nblk row blocks, exponent stride nd_pad); B: C's (mblk column blocks,
    // the fastest tile index)
    k_gram_tc<C, true, TO><<<grid, kThreads, TcDims<C>::kSmemBytes, st>>>(
        DB, EB, mapB, EA, p.ns_pad, p.nstep, nullptr, (int)(p.mblk * p.nblk), 1, nullptr,
        std::max(1, log2_ceil(p.nchunk)), err, nullptr, nullptr,
        mapB, EA, nullptr, 0, p.ns_pad, p.mblk, out, ldo, nd, ns, p.nd_pad);
    note_launch();
    return cudaGetLastError();
}
}  // namespace

size_t rotate_tc_workspace(long nd, int ns) { return rot_workspace<Tc47>(nd, ns); }
size_t rotate_tc23_workspace(long nd, int ns) { return rot_workspace<Tc23>(nd, ns); }

cudaError_t rotate_tc(const double *Y, long ldy, long nd, int ns, const double *Cm, double *out,
                      long ldo, void *ws, size_t ws_bytes, int *err, cudaStream_t st)
{
    return rotate_tc_impl<Tc47, double, double>(Y, ldy, nd, ns, Cm, out, ldo, ws, ws_bytes, err,
                                                st);
}

template <typename TY>
cudaError_t rotate_tc23(const TY *Y, long ldy, long nd, int ns, const double *Cm, float *out,
                        long ldo, void *ws, size_t ws_bytes, int *err, cudaStream_t st)
{
    return rotate_tc_impl<Tc23, TY, float>(Y, ldy, nd, ns, Cm, out, ldo, ws, ws_bytes, err, st);
}
template cudaError_t rotate_tc23<float>(const float *, long, long, int, const double *, float *,
                                        long, void *, size_t, int *, cudaStream_t);
template cudaError_t rotate_tc23<double>(const double *, long, long, int, const double *, float *,
                                         long, void *, size_t, int *, cudaStream_t);

__global__ void k_add_into(double *__restrict__ dst, const double *__restrict__ src, long n)
{
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long)gridDim.x * blockDim.x)
        dst[t] += src[t];
}

cudaError_t add_into(double *dst, const double *src, long n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const long b = (n + 255) / 256;
    k_add_into<<<(unsigned)(b < 1216 ? b : 1216), 256, 0, st>>>(dst, src, n);
    note_launch();
    return cudaGetLastError();
}

template cudaError_t gram_tc<float, float>(const float *, long, const float *, long, long, int,
                                           double *, void *, size_t, bool, int *, cudaStream_t);
template cudaError_t gram_tc<float, double>(const float *, long, const double *, long, long, int,
                                            double *, void *, size_t, bool, int *, cudaStream_t);
template cudaError_t gram_tc<double, double>(const double *, long, const double *, long, long,
                                             int, double *, void *, size_t, bool, int *,
                                             cudaStream_t);

}  // namespace sparc
