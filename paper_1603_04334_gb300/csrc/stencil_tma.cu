// stencil_tma.cu -- the FP32 fused stencil step (Eq. FD:Laplacian, weights Eq. weightsLap,
// zero-Dirichlet boundaries, V_eff, Chebyshev recurrence of Algorithm ChebychevFilter,
// Sec. 3.4) fed by the Tensor Memory Accelerator.
//
// The FP32 filter step moves 12 B per point-orbital and should run at HBM speed. A CTA owns
// a 32 x 16 tile of (x, y) for one column and streams along z. Thread 0 keeps a ring of
// kStages shared-memory planes filled with 4-D tiled TMA loads (cp.async.bulk.tensor) of
// the tile plus its radius-6 halo: the box starts 8 nodes left of the tile so that the x
// coordinate stays 16-byte aligned, and nodes outside the grid are zero-filled by the TMA
// unit, which is exactly the zero-Dirichlet boundary. Each plane's arrival is signalled
// through an mbarrier (expect-tx); after the CTA barrier that ends the compute of a plane,
// thread 0 refills that plane's stage. All waits are bounded and report a timeout through
// a device flag instead of hanging.
//
// Each thread takes 4 consecutive x nodes of one row with 128-bit shared loads (5 loads
// cover x-6 .. x+9 of the four nodes, 12 more the y neighbours) and keeps the z neighbours
// of its four nodes in a 13-deep register queue of float4, filled from each newly arrived
// plane. The arithmetic runs on packed FP32 pairs (two nodes per add or fused
// multiply-add), each operation rounded as the scalar form would round it, and the plane
// loop is unrolled 13 times, one copy per rotation of the queue, so the queue is never
// shifted. The queue needs planes t .. t+6 of the ring, so with kStages = 9 the loads run
// 2 planes ahead of the compute.
//
// Y_{j-1} (one third of the step's traffic) rides in the same ring: the TMA load that
// brings plane t of Y also brings the halo-free tile of Y_{j-1} at the plane whose compute
// first needs plane t (z - 6), completing on the same mbarrier, so every HBM stream of the
// step is an asynchronous bulk copy. V_eff (one plane shared by all columns, L2-resident)
// is prefetched into registers two planes ahead.
//
// Requirements (checked on the host, else k_stencil_f32_copy runs): n0 and ld
// multiples of 4 and 16-byte aligned block pointers (TMA strides and float4 accesses).
#include "device_once.cuh"
#include "internal.cuh"

#include <type_traits>
#include "tma.cuh"

#include <cudaTypedefs.h>

namespace sparc {

namespace {
constexpr int kTX = 8;       // threads along x, 4 nodes each
constexpr int kTY = 16;      // rows per tile
constexpr int kBX = 4 * kTX; // 32 nodes along x
constexpr int kR = kRadius;  // 6
constexpr int kW = kBX + 16; // box width: 8 left (aligned) + 32 + 8 right
constexpr int kH = kTY + 2 * kR;
constexpr int kStages = 9;
// Y_{j-1} tiles: one arrives with plane t and is used when that plane enters the z queue, kPrev
// steps after it was issued (a plane stays kR steps longer), so they need fewer slots
constexpr int kPrev = kStages - kR;
constexpr int kPlaneBytes = kW * kH * 4;   // Y plane with halo
constexpr int kTileBytes = kBX * kTY * 4;  // Y_{j-1} tile, no halo
constexpr int kStageFloats = kW * kH;
constexpr int kTileFloats = kBX * kTY;
// 54.5 KB: four CTAs (16 warps) per SM; with a tile slot in each of ten stages it was three
constexpr int kSmemBytes = kStages * kPlaneBytes + kPrev * kTileBytes;
constexpr unsigned kWaitLimit = 1u << 22;
}  // namespace

// Step coefficients as packed pairs for the FP32x2 instructions (both lanes equal).
struct StepCoef2 {
    float2 w[kR + 1];
    float2 c0, alpha, nbeta;
};

__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }

// One plane of the step for the thread's four nodes, as two packed pairs (nodes 0-1 and
// 2-3). row: the plane row at node i - 8 (20 values cover i - 8 .. i + 11); the z queue
// slot of logical entry k (plane tc - 6 + k) is (PH + k) % 13, a compile-time index. Per
// node: (c0 + alpha V) y + sum_r w_r ((x+r + x-r) + (y+r + y-r) + (z+r + z-r)), each
// operation rounded as in the scalar form (the x sums of odd radii, whose pairs straddle
// a register pair boundary, stay scalar).
template <int PH>
__device__ __forceinline__ void plane_math(const float *row, const float4 (&q)[2 * kR + 1],
                                           const float4 &vv, const StepCoef2 &cf, float2 &aA,
                                           float2 &aB)
{
    constexpr int Q = 2 * kR + 1;
    float f[20];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        const float4 v = *reinterpret_cast<const float4 *>(row + 4 * m);
        f[4 * m] = v.x;
        f[4 * m + 1] = v.y;
        f[4 * m + 2] = v.z;
        f[4 * m + 3] = v.w;
    }
    const float4 c = q[(PH + kR) % Q];
    aA = __fmul2_rn(__ffma2_rn(cf.alpha, lo2(vv), cf.c0), lo2(c));
    aB = __fmul2_rn(__ffma2_rn(cf.alpha, hi2(vv), cf.c0), hi2(c));
#pragma unroll
    for (int r = 1; r <= kR; ++r) {
        const float4 yp = *reinterpret_cast<const float4 *>(row + r * kW + 8);
        const float4 ym = *reinterpret_cast<const float4 *>(row - r * kW + 8);
        const float4 zp = q[(PH + kR + r) % Q], zm = q[(PH + kR - r) % Q];
        float2 xA, xB;
        if (r % 2 == 0) {
            xA = __fadd2_rn(make_float2(f[8 + r], f[9 + r]), make_float2(f[8 - r], f[9 - r]));
            xB = __fadd2_rn(make_float2(f[10 + r], f[11 + r]), make_float2(f[10 - r], f[11 - r]));
        } else {
            xA = make_float2(f[8 + r] + f[8 - r], f[9 + r] + f[9 - r]);
            xB = make_float2(f[10 + r] + f[10 - r], f[11 + r] + f[11 - r]);
        }
        const float2 tA = __fadd2_rn(__fadd2_rn(xA, __fadd2_rn(lo2(yp), lo2(ym))),
                                     __fadd2_rn(lo2(zp), lo2(zm)));
        const float2 tB = __fadd2_rn(__fadd2_rn(xB, __fadd2_rn(hi2(yp), hi2(ym))),
                                     __fadd2_rn(hi2(zp), hi2(zm)));
        aA = __ffma2_rn(cf.w[r], tA, aA);
        aB = __ffma2_rn(cf.w[r], tB, aB);
    }
}

// The x sums of radius r of a row's four nodes from the 20 values around them.
template <int r>
__device__ __forceinline__ void x_sums(const float (&f)[20], float2 &xA, float2 &xB)
{
    if constexpr (r % 2 == 0) {
        xA = __fadd2_rn(make_float2(f[8 + r], f[9 + r]), make_float2(f[8 - r], f[9 - r]));
        xB = __fadd2_rn(make_float2(f[10 + r], f[11 + r]), make_float2(f[10 - r], f[11 - r]));
    } else {
        xA = make_float2(f[8 + r] + f[8 - r], f[9 + r] + f[9 - r]);
        xB = make_float2(f[10 + r] + f[10 - r], f[11 + r] + f[11 - r]);
    }
}

// plane_math for two rows at once (row: the upper one's; q, vv and a: of the rows in turn): the
// y neighbours of the pair are 12 loads instead of 24, and each is used by both rows. The values
// are those of plane_math, operation by operation.
template <int PH>
__device__ __forceinline__ void plane_math2(const float *row, const float4 (&q)[2][2 * kR + 1],
                                            const float4 (&vv)[2], const StepCoef2 &cf,
                                            float2 (&a)[2][2])
{
    constexpr int Q = 2 * kR + 1;
    float f[2][20];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const float4 v = *reinterpret_cast<const float4 *>(row + h * kW + 4 * m);
            f[h][4 * m] = v.x;
            f[h][4 * m + 1] = v.y;
            f[h][4 * m + 2] = v.z;
            f[h][4 * m + 3] = v.w;
        }
    const float4 c0 = q[0][(PH + kR) % Q], c1 = q[1][(PH + kR) % Q];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float4 c = h ? c1 : c0;
        a[h][0] = __fmul2_rn(__ffma2_rn(cf.alpha, lo2(vv[h]), cf.c0), lo2(c));
        a[h][1] = __fmul2_rn(__ffma2_rn(cf.alpha, hi2(vv[h]), cf.c0), hi2(c));
    }
    float4 up = c0, dn = c1;  // the rows at distance r - 1 above row 0 and below row 1
    auto radius = [&](auto rr) {
        constexpr int r = decltype(rr)::value;
        const float4 un = *reinterpret_cast<const float4 *>(row - r * kW + 8);
        const float4 dm = *reinterpret_cast<const float4 *>(row + (1 + r) * kW + 8);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 yp = h ? dm : dn, ym = h ? up : un;
            const float4 zp = q[h][(PH + kR + r) % Q], zm = q[h][(PH + kR - r) % Q];
            float2 xA, xB;
            x_sums<r>(f[h], xA, xB);
            const float2 tA = __fadd2_rn(__fadd2_rn(xA, __fadd2_rn(lo2(yp), lo2(ym))),
                                         __fadd2_rn(lo2(zp), lo2(zm)));
            const float2 tB = __fadd2_rn(__fadd2_rn(xB, __fadd2_rn(hi2(yp), hi2(ym))),
                                         __fadd2_rn(hi2(zp), hi2(zm)));
            a[h][0] = __ffma2_rn(cf.w[r], tA, a[h][0]);
            a[h][1] = __ffma2_rn(cf.w[r], tB, a[h][1]);
        }
        up = un;
        dn = dm;
    };
    radius(std::integral_constant<int, 1>{});
    radius(std::integral_constant<int, 2>{});
    radius(std::integral_constant<int, 3>{});
    radius(std::integral_constant<int, 4>{});
    radius(std::integral_constant<int, 5>{});
    radius(std::integral_constant<int, 6>{});
    static_assert(kR == 6, "the radii above");
}

// State of one thread of k_stencil_f32_tma.
struct TmaThread {
    float *sm;
    uint64_t *full;
    float *Oc;
    const float *V;
    const CUtensorMap *tmY, *tmP;
    long p, plane;  // p: the thread's node offset at the current compute plane
    int k, k1, T;   // current compute z, end of the chunk, planes of the CTA
    int i0, j0, k0, col;
    int sc;         // stage of the compute plane tc
    int sn;         // stage of plane tc + 6 (its centre enters the queue)
    int sp;         // slot of its Y_{j-1} tile
    unsigned pn;    // parity of plane tc + 6's current use of its stage
    int tc;         // current compute plane
    int row;        // offset of the thread's upper row and first node in a plane's box, less 8
    int tile;       // the same in a Y_{j-1} tile
    int n0, tid;
    bool act[2], hasP;
};

// plane t of Y (z = k0 - 6 + t) into stage t % kStages, with the Y_{j-1} tile of the plane
// computed when plane t completes the z queue (z - 6); thread 0 only
__device__ __forceinline__ void tma_issue(TmaThread &s, int t)
{
    const int st = t % kStages;
    const bool p = s.hasP && t >= 2 * kR;
    float *dst = s.sm + (long)st * kStageFloats;
    mbar_arrive_expect_tx(&s.full[st], kPlaneBytes + (p ? kTileBytes : 0));
    tma_load_4d(dst, s.tmY, &s.full[st], s.i0 - 8, s.j0 - kR, s.k0 - kR + t, s.col);
    if (p)
        tma_load_4d(s.sm + kStages * kStageFloats + t % kPrev * kTileFloats, s.tmP, &s.full[st],
                    s.i0, s.j0, s.k0 - 2 * kR + t, s.col);
}

template <int PH, int NR>
__device__ __forceinline__ bool plane_step(TmaThread &s, float4 (&q)[NR][2 * kR + 1],
                                           float4 (&vv)[NR], float4 (&v1)[NR], const StepCoef2 &cf,
                                           int *timed_out)
{
    constexpr int Q = 2 * kR + 1;
    float4 v2[NR];
#pragma unroll
    for (int h = 0; h < NR; ++h) {
        v2[h] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s.act[h] && s.k + 2 < s.k1)
            v2[h] = *reinterpret_cast<const float4 *>(s.V + s.p + h * s.n0 + 2 * s.plane);
    }
    const bool got = mbar_wait(&s.full[s.sn], s.pn, kWaitLimit);
    const float *stn = s.sm + (long)s.sn * kStageFloats + s.row + 8;
#pragma unroll
    for (int h = 0; h < NR; ++h)
        q[h][(PH + 2 * kR) % Q] = *reinterpret_cast<const float4 *>(stn + h * kW);
    float2 a[NR][2];
    const float *row = s.sm + (long)s.sc * kStageFloats + s.row;
    if constexpr (NR == 2)
        plane_math2<PH>(row, q, vv, cf, a);
    else
        plane_math<PH>(row, q[0], vv[0], cf, a[0][0], a[0][1]);
#pragma unroll
    for (int h = 0; h < NR; ++h) {
        if (s.act[h] && got) {
            if (s.hasP) {
                const float4 pv = *reinterpret_cast<const float4 *>(
                    s.sm + kStages * kStageFloats + s.sp * kTileFloats + s.tile + h * kBX);
                a[h][0] = __ffma2_rn(cf.nbeta, lo2(pv), a[h][0]);
                a[h][1] = __ffma2_rn(cf.nbeta, hi2(pv), a[h][1]);
            }
            *reinterpret_cast<float4 *>(s.Oc + s.p + h * s.n0) =
                make_float4(a[h][0].x, a[h][0].y, a[h][1].x, a[h][1].y);
        }
        vv[h] = v1[h];
        v1[h] = v2[h];
    }
    if (!got) *timed_out = 1;
    __syncthreads();  // every thread is done with plane tc's stage
    if (*(volatile int *)timed_out) return false;
    if (s.tid == 0 && s.tc + kStages < s.T) tma_issue(s, s.tc + kStages);
    if (++s.sc == kStages) s.sc = 0;
    if (++s.sn == kStages) {
        s.sn = 0;
        s.pn ^= 1u;
    }
    if (++s.sp == kPrev) s.sp = 0;
    ++s.k;
    ++s.tc;
    s.p += s.plane;
    return true;
}

// Block: 8 x 16 / NR threads (4 x-nodes of NR neighbouring rows each). Thread 0 keeps the ring kStages planes ahead:
// after the barrier that ends the compute of plane tc, it refills that plane's stage with
// plane tc + kStages. The plane loop is unrolled 13 times, one copy per rotation of the z
// queue, so the queue is never shifted.
template <int NR>
__global__ void __launch_bounds__(kTX *kTY / NR, 4)
k_stencil_f32_tma(const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmP,
                  bool hasP, float *out, const float *__restrict__ V, int n0, int n1, int n2,
                  long ld, int nzc, int zchunk, StepCoef2 cf, int *err)
{
    // kStages Y planes [kH][kW], then kPrev Y_{j-1} tiles [kTY][kBX]
    extern __shared__ __align__(128) float sm[];
    __shared__ __align__(8) uint64_t full[kStages];
    __shared__ int timed_out;
    TmaThread s;
    s.tid = threadIdx.y * kTX + threadIdx.x;
    s.row = (kR + NR * threadIdx.y) * kW + 4 * threadIdx.x;
    s.tile = NR * threadIdx.y * kBX + 4 * threadIdx.x;
    s.n0 = n0;
    s.i0 = blockIdx.x * kBX;
    s.j0 = blockIdx.y * kTY;
    s.col = blockIdx.z / nzc;
    s.k0 = (blockIdx.z % nzc) * zchunk;
    s.k1 = min(n2, s.k0 + zchunk);
    s.T = (s.k1 - s.k0) + 2 * kR;  // planes k0-6 .. k1+5
    s.sm = sm;
    s.full = full;
    s.tmY = &tmY;
    s.tmP = &tmP;
    s.hasP = hasP;
    const int i = s.i0 + 4 * threadIdx.x, j = s.j0 + NR * threadIdx.y;
#pragma unroll
    for (int h = 0; h < NR; ++h) s.act[h] = (i < n0) && (j + h < n1);
    s.plane = (long)n0 * n1;
    s.k = s.k0;
    s.p = (long)i + (long)n0 * j + (long)s.k0 * s.plane;
    s.Oc = out + (long)s.col * ld;
    s.V = V;
    if (s.tid == 0) {
        tma_prefetch_desc(&tmY);
        if (hasP) tma_prefetch_desc(&tmP);
        for (int t = 0; t < kStages; ++t) mbar_init(&full[t], 1);
        mbar_fence_init();
        timed_out = 0;
    }
    __syncthreads();
    if (s.tid == 0)
        for (int t = 0; t < kStages && t < s.T; ++t) tma_issue(s, t);
    auto center = [&](int t, int h) -> float4 {
        return *reinterpret_cast<const float4 *>(sm + (long)(t % kStages) * kStageFloats + s.row +
                                                 h * kW + 8);
    };
    bool ok = true;
    float4 q[NR][2 * kR + 1];
    // planes 0..5 only feed the queue: read them, then hand their stages to planes
    // kStages .. kStages+5
    for (int t = 0; t < kR; ++t) {
        ok = ok && mbar_wait(&full[t % kStages], (unsigned)((t / kStages) & 1), kWaitLimit);
#pragma unroll
        for (int h = 0; h < NR; ++h) q[h][t] = center(t, h);
    }
    if (!ok) timed_out = 1;
    __syncthreads();
    if (s.tid == 0 && !timed_out)
        for (int t = kStages; t < kStages + kR && t < s.T; ++t) tma_issue(s, t);
    for (int t = kR; t < 2 * kR; ++t) {
        ok = ok && mbar_wait(&full[t % kStages], (unsigned)((t / kStages) & 1), kWaitLimit);
#pragma unroll
        for (int h = 0; h < NR; ++h) q[h][t] = center(t, h);
    }
    if (!ok) timed_out = 1;
    __syncthreads();
    s.sc = kR % kStages;
    s.sn = (2 * kR) % kStages;
    s.pn = (unsigned)(((2 * kR) / kStages) & 1);
    s.sp = (2 * kR) % kPrev;
    s.tc = kR;
    float4 vv[NR], v1[NR];
#pragma unroll
    for (int h = 0; h < NR; ++h) {
        vv[h] = v1[h] = make_float4(0.f, 0.f, 0.f, 0.f);
        const float *v = V + s.p + h * n0;
        if (s.act[h]) vv[h] = *reinterpret_cast<const float4 *>(v);
        if (s.act[h] && s.k0 + 1 < s.k1) v1[h] = *reinterpret_cast<const float4 *>(v + s.plane);
    }
    const int tend = s.T - kR;
    if (!timed_out) {
#define SPARC_PLANE(PH)                                                                  \
    if (s.tc >= tend) break;                                                             \
    if (!plane_step<PH, NR>(s, q, vv, v1, cf, &timed_out)) break;
        for (;;) {
            SPARC_PLANE(0) SPARC_PLANE(1) SPARC_PLANE(2) SPARC_PLANE(3) SPARC_PLANE(4)
            SPARC_PLANE(5) SPARC_PLANE(6) SPARC_PLANE(7) SPARC_PLANE(8) SPARC_PLANE(9)
            SPARC_PLANE(10) SPARC_PLANE(11) SPARC_PLANE(12)
        }
#undef SPARC_PLANE
    }
    if (timed_out) {
        // leave no TMA write in flight into this CTA's shared memory: wait (bounded) for
        // the latest issued plane of every stage, then report
        if (s.tid == 0) {
            atomicExch(err, 1);
            const int issued = min(s.T, s.tc + kStages);  // planes handed to the TMA unit
            for (int st = 0; st < kStages; ++st) {
                int last = -1;  // latest plane issued into stage st
                for (int t = st; t < issued; t += kStages) last = t;
                if (last >= 0) mbar_wait(&full[st], (unsigned)((last / kStages) & 1), kWaitLimit);
            }
        }
        __syncthreads();
    }
}

// The same step for rows that TMA cannot address (n0 or ld not a multiple of 4, a block off a
// 16-byte boundary): the ring is filled by 4-byte asynchronous copies (cp.async, zero-filled
// outside the grid) that consecutive lanes issue along rows, and the output row goes through
// shared memory so that its stores are consecutive too; the arithmetic and the queue are
// those of k_stencil_f32_tma, plane by plane. One barrier per plane: it follows the wait for
// this thread's copies of the step's planes and precedes the copies into the stage that the
// previous step released. Bound by latency (about 80 thread instructions a node slot, issue
// 46% busy at 12 warps per SM) where the row-per-thread
// kernel it replaces needed 207: 75 x 61 x 53 x 40, 92 us -> 84 us a step.
namespace {
constexpr int kWarpsC = kTX * kTY / 32;
}

__device__ __forceinline__ void copy4(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(in ? 4 : 0)
                 : "memory");
}

__global__ void __launch_bounds__(kTX *kTY, 4)
k_stencil_f32_copy(const float *Yb, const float *Pb, float *out, const float *__restrict__ V,
                   int n0, int n1, int n2, long ld, int nzc, int zchunk, StepCoef2 cf)
{
    extern __shared__ __align__(128) float sm[];
    float *const prev = sm + kStages * kStageFloats;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kTX + tx;
    const int lane = tid & 31, warp = tid >> 5;
    const int i0 = blockIdx.x * kBX, j0 = blockIdx.y * kTY;
    const int col = blockIdx.z / nzc;
    const int k0 = (blockIdx.z % nzc) * zchunk, k1 = min(n2, k0 + zchunk);
    const unsigned plane = (unsigned)n0 * (unsigned)n1;
    const float *Y = Yb + (long)col * ld;
    const float *P = Pb ? Pb + (long)col * ld : nullptr;
    float *O = out + (long)col * ld;
    // plane z of Y into stage st: the 32 columns of the tile for all 28 rows, a warp per row,
    // then the 6 columns left and right of its 16 rows
    const bool xin = i0 + lane < n0;
    auto copy_plane = [&](int z, int st) {
        const bool zin = z >= 0 && z < n2;
        const float *src = Y + (zin ? (unsigned)z * plane : 0u);
        float *dst = sm + st * kStageFloats;
#pragma unroll
        for (int u = 0; u < kH / kWarpsC; ++u) {
            const int r = warp + u * kWarpsC, j = j0 - kR + r;
            const bool in = zin && xin && j >= 0 && j < n1;
            copy4(dst + r * kW + 8 + lane, src + (in ? (unsigned)(i0 + lane) + (unsigned)n0 * (unsigned)j : 0u), in);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = tid + u * kTX * kTY;
            if (e < 2 * kR * kTY) {
                const int r = e / (2 * kR), h = e - r * (2 * kR);
                const int x = h < kR ? h - kR : h - kR + kBX, i = i0 + x, j = j0 + r;
                const bool in = zin && i >= 0 && i < n0 && j < n1;
                copy4(dst + (kR + r) * kW + 8 + x, src + (in ? (unsigned)i + (unsigned)n0 * (unsigned)j : 0u), in);
            }
        }
    };
    auto copy_prev = [&](int z, int slot) {
        float *dst = prev + slot * kTileFloats;
#pragma unroll
        for (int u = 0; u < kTY / kWarpsC; ++u) {
            const int r = warp + u * kWarpsC, j = j0 + r;
            const bool in = xin && j < n1;
            copy4(dst + r * kBX + lane,
                  P + (in ? (unsigned)(i0 + lane) + (unsigned)n0 * (unsigned)j + (unsigned)z * plane : 0u), in);
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    // planes are numbered from k0 - 6; plane t goes to stage t % kStages, the Y_{j-1} tile of
    // step t (compute plane t) to slot t % kPrev. Step t starts with planes t .. t + 6 and its
    // tile present and issues plane t - 1 + kStages and the tile of step t + kPrev - 1.
    const int T = (k1 - k0) + 2 * kR;
    for (int t = 0; t < kStages; ++t) copy_plane(k0 - kR + t, t);  // (T >= 13)
    commit();
    const float *vp = V + ((unsigned)min(i0 + 4 * tx, n0 - 1) + (unsigned)n0 * (unsigned)min(j0 + ty, n1 - 1));
    const int nv = min(n0 - 1 - min(i0 + 4 * tx, n0 - 1), 3);  // further nodes of the row
    auto load_v = [&](int z) {
        const float *q = vp + (unsigned)z * plane;
        float4 v;
        v.x = q[0];
        v.y = q[min(1, nv)];
        v.z = q[min(2, nv)];
        v.w = q[nv];
        return v;
    };
    float4 q[2 * kR + 1];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    auto center = [&](int st) {
        return *reinterpret_cast<const float4 *>(sm + st * kStageFloats + (kR + ty) * kW + 8 + 4 * tx);
    };
    // planes 0 .. 5 only feed the queue: their stages take the planes up to 12, which step 6
    // needs, and 13, with the first two tiles
#pragma unroll
    for (int t = 0; t < kStages; ++t) q[t] = center(t);
    __syncthreads();
    for (int t = kStages; t <= 2 * kR; ++t) copy_plane(k0 - kR + t, t % kStages);
    if (P) copy_prev(k0, kR % kPrev);
    commit();
    if (2 * kR + 1 < T) copy_plane(k0 + kR + 1, (2 * kR + 1) % kStages);
    if (P && k0 + 1 < k1) copy_prev(k0 + 1, (kR + 1) % kPrev);
    commit();
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int t = kStages; t < 2 * kR; ++t) q[t] = center(t % kStages);
    int sc = kR % kStages, sn = (2 * kR) % kStages, sp = kR % kPrev, k = k0;
    float4 vv = load_v(k0), v1 = load_v(min(k0 + 1, k1 - 1));
    auto step = [&](auto phase) {
        constexpr int PH = decltype(phase)::value;
        constexpr int Q = 2 * kR + 1;
        const int tc = k - k0 + kR;
        // all but the newest group are here; every thread is done with the previous step
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        {
            const int t = tc - 1 + kStages;  // into the stage of plane tc - 1
            if (t < T) copy_plane(k0 - kR + t, sc == 0 ? kStages - 1 : sc - 1);
            if (P && k + kPrev - 1 < k1) copy_prev(k + kPrev - 1, sp == 0 ? kPrev - 1 : sp - 1);
            commit();
        }
        const float4 v2 = load_v(min(k + 2, k1 - 1));
        q[(PH + 2 * kR) % Q] = center(sn);
        const float *row = sm + sc * kStageFloats + (kR + ty) * kW + 4 * tx;
        float2 aA, aB;
        plane_math<PH>(row, q, vv, cf, aA, aB);
        // the tile's slot takes the result in place of Y_{j-1}: a warp writes its four rows as
        // its threads own them and stores them row by row
        float *const ot = prev + sp * kTileFloats;
        float4 *const mine = reinterpret_cast<float4 *>(ot + ty * kBX + 4 * tx);
        if (P) {
            const float4 pv = *mine;
            aA = __ffma2_rn(cf.nbeta, lo2(pv), aA);
            aB = __ffma2_rn(cf.nbeta, hi2(pv), aB);
        }
        *mine = make_float4(aA.x, aA.y, aB.x, aB.y);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = 4 * warp + u;
            if (xin && j0 + r < n1)
                O[(unsigned)(i0 + lane) + (unsigned)n0 * (unsigned)(j0 + r) + (unsigned)k * plane] =
                    ot[r * kBX + lane];
        }
        vv = v1;
        v1 = v2;
        if (++sc == kStages) sc = 0;
        if (++sn == kStages) sn = 0;
        if (++sp == kPrev) sp = 0;
        ++k;
    };
#define SPARC_COPY_STEP(PH)                                                              \
    if (k >= k1) break;                                                                  \
    step(std::integral_constant<int, PH>{});
    for (;;) {
        SPARC_COPY_STEP(0) SPARC_COPY_STEP(1) SPARC_COPY_STEP(2) SPARC_COPY_STEP(3)
        SPARC_COPY_STEP(4) SPARC_COPY_STEP(5) SPARC_COPY_STEP(6) SPARC_COPY_STEP(7)
        SPARC_COPY_STEP(8) SPARC_COPY_STEP(9) SPARC_COPY_STEP(10) SPARC_COPY_STEP(11)
        SPARC_COPY_STEP(12)
    }
#undef SPARC_COPY_STEP
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

namespace {
// State of one thread of k_batch_stencil_tma within an item.
struct BatchThread {
    float *Oc;
    const float *V;
    long p, plane;  // p: the thread's node offset at the current plane
    int k, k1;      // current z, end of the range
    int sn;         // stage of the plane entering the queue (its Y_{j-1} slot is sn mod kPrev)
    unsigned pn;    // parity of its current use
    int row, tile;  // offsets of the thread's rows in a plane's box (less 8) and in a tile
    int n0;
    bool act[2], hasP;
};
static_assert(kStages % kPrev == 0, "a plane's Y_{j-1} slot follows from its stage");

template <int PH, int NR>
__device__ __forceinline__ bool batch_plane(BatchThread &s, float4 (&q)[NR][2 * kR + 1],
                                            float4 (&vv)[NR], float4 (&v1)[NR], const StepCoef2 &cf,
                                            float *sm, uint64_t *full, int *timed_out)
{
    constexpr int Q = 2 * kR + 1;
    float4 v2[NR];
#pragma unroll
    for (int h = 0; h < NR; ++h) {
        v2[h] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s.act[h] && s.k + 2 < s.k1)
            v2[h] = *reinterpret_cast<const float4 *>(s.V + s.p + h * s.n0 + 2 * s.plane);
    }
    const bool got = mbar_wait(&full[s.sn], s.pn, kWaitLimit);
#pragma unroll
    for (int h = 0; h < NR; ++h)
        q[h][(PH + 2 * kR) % Q] = *reinterpret_cast<const float4 *>(
            sm + s.sn * kStageFloats + s.row + h * kW + 8);
    const int sc = s.sn >= kR ? s.sn - kR : s.sn + kStages - kR;
    float2 a[NR][2];
    const float *row = sm + sc * kStageFloats + s.row;
    if constexpr (NR == 2)
        plane_math2<PH>(row, q, vv, cf, a);
    else
        plane_math<PH>(row, q[0], vv[0], cf, a[0][0], a[0][1]);
#pragma unroll
    for (int h = 0; h < NR; ++h) {
        if (s.act[h] && got) {
            if (s.hasP) {
                const float4 pv = *reinterpret_cast<const float4 *>(
                    sm + kStages * kStageFloats + s.sn % kPrev * kTileFloats + s.tile + h * kBX);
                a[h][0] = __ffma2_rn(cf.nbeta, lo2(pv), a[h][0]);
                a[h][1] = __ffma2_rn(cf.nbeta, hi2(pv), a[h][1]);
            }
            *reinterpret_cast<float4 *>(s.Oc + s.p + h * s.n0) =
                make_float4(a[h][0].x, a[h][0].y, a[h][1].x, a[h][1].y);
        }
        vv[h] = v1[h];
        v1[h] = v2[h];
    }
    if (!got) *timed_out = 1;
    if (++s.sn == kStages) {
        s.sn = 0;
        s.pn ^= 1u;
    }
    ++s.k;
    s.p += s.plane;
    __syncthreads();  // the plane's stage is free
    return !*(volatile int *)timed_out;
}
}  // namespace

// Work-list form for a batch of clusters: a persistent CTA walks its items (cluster,
// column, 32 x 16 tile, z range) in order, and its ring runs on across item boundaries: the
// planes of all its items form one sequence (item i contributes (k1 - k0) + 12 planes),
// thread 0 issues that sequence kStages planes ahead of the planes released, and the
// consumers take the planes in the same order. Each cluster's tensor maps (Y_j with halo,
// Y_{j-1} tile) live in device memory, its sizes, pointers and coefficients in its
// BatchTma entry (the current item's coefficients in shared memory). A plane is computed as in
// k_stencil_f32_tma, two rows per thread where the launch is more than a wave (the scalar form
// with a shifted queue it replaces: 445 us a step for 12 clusters of 32 to 48 nodes an edge, 400 us
// so; one cluster 31.7 -> 27.7 us, 40 clusters 1.28 -> 1.12 ms).
template <int NR>
__global__ void __launch_bounds__(kTX *kTY / NR, NR == 1 ? 2 : 4)
k_batch_stencil_tma(const BatchItem *__restrict__ items, int nitems, const BatchTma *cs, int *err)
{
    extern __shared__ __align__(128) float sm[];
    __shared__ __align__(8) uint64_t full[kStages];
    __shared__ int timed_out;
    __shared__ __align__(16) StepCoef2 cf;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int tid = ty * kTX + tx;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(&full[s], 1);
        mbar_fence_init();
        timed_out = 0;
    }
    __syncthreads();
    // producer state (thread 0): next plane to hand to the TMA unit; the item being issued
    // is held in registers (read from global memory once per item, not once per plane)
    int p_it = blockIdx.x, p_t = 0, p_T = 0, p_x = 0, p_y = 0, p_z = 0, p_col = 0;
    const CUtensorMap *p_mY = nullptr, *p_mP = nullptr;
    unsigned issued = 0;  // planes handed to the TMA unit (fewer than 2^31 per CTA: host check)
    auto issue_upto = [&](unsigned limit) {
        while (issued < limit && p_it < nitems) {
            if (p_t == 0) {  // a new item: read it and bring its descriptors close
                const BatchItem w = items[p_it];
                const BatchTma &C = cs[w.cluster];
                p_mY = (const CUtensorMap *)C.mY;
                p_mP = (const CUtensorMap *)C.mP;
                p_T = (w.k1 - w.k0) + 2 * kR;
                p_x = w.a * kBX;
                p_y = w.b * kTY;
                p_z = w.k0 - kR;
                p_col = w.col;
                tma_prefetch_desc(p_mY);
                if (p_mP) tma_prefetch_desc(p_mP);
            }
            const unsigned s = issued % kStages;
            const bool p = p_mP != nullptr && p_t >= 2 * kR;
            float *st = sm + (long)s * kStageFloats;
            mbar_arrive_expect_tx(&full[s], kPlaneBytes + (p ? kTileBytes : 0));
            tma_load_4d(st, p_mY, &full[s], p_x - 8, p_y - kR, p_z + p_t, p_col);
            if (p)
                tma_load_4d(sm + kStages * kStageFloats + issued % kPrev * kTileFloats, p_mP,
                            &full[s], p_x, p_y, p_z - kR + p_t, p_col);
            ++issued;
            if (++p_t == p_T) {
                p_t = 0;
                p_it += gridDim.x;
            }
        }
    };
    auto wait = [&](unsigned g) -> bool {
        return mbar_wait(&full[g % kStages], (g / kStages) & 1u, kWaitLimit);
    };
    if (tid == 0) issue_upto(kStages);
    unsigned g0 = 0;  // sequence index of the current item's first plane
    for (int it = blockIdx.x; it < nitems && !timed_out; it += gridDim.x) {
        const BatchItem w = items[it];
        const BatchTma &C = cs[w.cluster];
        const int n0 = C.n0, n1 = C.n1;
        const int T = (w.k1 - w.k0) + 2 * kR;
        const int i = w.a * kBX + 4 * tx, j = w.b * kTY + NR * ty;
        if (tid <= kR) cf.w[tid] = make_float2(C.cf.w[tid], C.cf.w[tid]);
        if (tid == 0) {
            cf.c0 = make_float2(C.cf.c0, C.cf.c0);
            cf.alpha = make_float2(C.cf.alpha, C.cf.alpha);
            cf.nbeta = make_float2(-C.cf.beta, -C.cf.beta);
        }
        BatchThread b;
        b.row = (kR + NR * ty) * kW + 4 * tx;
        b.tile = NR * ty * kBX + 4 * tx;
        auto center = [&](unsigned g, int h) -> float4 {
            return *reinterpret_cast<const float4 *>(sm + (g % kStages) * kStageFloats + b.row +
                                                     h * kW + 8);
        };
        bool ok = true;
        float4 q[NR][2 * kR + 1];
        for (int t = 0; t < kR; ++t) {
            ok = ok && wait(g0 + t);
#pragma unroll
            for (int h = 0; h < NR; ++h) q[h][t] = center(g0 + t, h);
        }
        if (!ok) timed_out = 1;
        __syncthreads();
        if (tid == 0 && !timed_out) issue_upto(g0 + kR + kStages);
        for (int t = kR; t < 2 * kR; ++t) {
            ok = ok && wait(g0 + t);
#pragma unroll
            for (int h = 0; h < NR; ++h) q[h][t] = center(g0 + t, h);
        }
        if (!ok) timed_out = 1;
        __syncthreads();
        b.n0 = n0;
        b.Oc = C.out + (long)w.col * C.ld;
        b.V = C.V;
        b.plane = (long)n0 * n1;
        b.p = (long)i + (long)n0 * j + (long)w.k0 * b.plane;
        b.k = w.k0;
        b.k1 = w.k1;
        b.sn = (int)((g0 + 2 * kR) % kStages);
        b.pn = (g0 + 2 * kR) / kStages & 1u;
        b.hasP = C.mP != nullptr;
        float4 vv[NR], v1[NR];
#pragma unroll
        for (int h = 0; h < NR; ++h) {
            b.act[h] = (i < n0) && (j + h < n1);
            vv[h] = v1[h] = make_float4(0.f, 0.f, 0.f, 0.f);
            const float *v = b.V + b.p + h * n0;
            if (b.act[h]) vv[h] = *reinterpret_cast<const float4 *>(v);
            if (b.act[h] && b.k + 1 < b.k1)
                v1[h] = *reinterpret_cast<const float4 *>(v + b.plane);
        }
        for (bool more = !timed_out && b.k < b.k1; more;) {
            // (each plane that is done makes room for one)
#define SPARC_BATCH_STEP(PH)                                                                   \
    more = batch_plane<PH, NR>(b, q, vv, v1, cf, sm, full, &timed_out);                             \
    if (tid == 0 && more) issue_upto(issued + 1);                                               \
    if (!(more = more && b.k < b.k1)) break
            SPARC_BATCH_STEP(0);
            SPARC_BATCH_STEP(1);
            SPARC_BATCH_STEP(2);
            SPARC_BATCH_STEP(3);
            SPARC_BATCH_STEP(4);
            SPARC_BATCH_STEP(5);
            SPARC_BATCH_STEP(6);
            SPARC_BATCH_STEP(7);
            SPARC_BATCH_STEP(8);
            SPARC_BATCH_STEP(9);
            SPARC_BATCH_STEP(10);
            SPARC_BATCH_STEP(11);
            SPARC_BATCH_STEP(12);
#undef SPARC_BATCH_STEP
        }
        g0 += T;
        __syncthreads();  // the item's last planes (z halo) are free
        if (tid == 0 && !timed_out) issue_upto(g0 + kStages);
    }
    if (timed_out) {
        if (tid == 0) {
            atomicExch(err, 1);
            for (unsigned s = 0; s < kStages; ++s) {
                if (s >= issued) continue;
                const unsigned last = s + (issued - 1 - s) / kStages * kStages;  // latest in s
                mbar_wait(&full[s], (last / kStages) & 1u, kWaitLimit);
            }
        }
        __syncthreads();
    }
}

// The two tensor maps of a block: with the halo box (the Y_j loads) and with the tile box
// (the Y_{j-1} loads); maps[0], maps[1].
cudaError_t encode_f32_maps(const DevHam &H, const float *base, int ncols, long ld, void *maps)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc;
    const cudaError_t e = tensor_map_encoder(enc);
    if (e != cudaSuccess) return e;
    CUtensorMap *m = reinterpret_cast<CUtensorMap *>(maps);
    cuuint64_t dims[4] = {(cuuint64_t)H.n0, (cuuint64_t)H.n1, (cuuint64_t)H.n2, (cuuint64_t)ncols};
    cuuint64_t strides[3] = {(cuuint64_t)H.n0 * 4, (cuuint64_t)H.n0 * H.n1 * 4,
                             (cuuint64_t)ld * 4};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    cuuint32_t boxY[4] = {(cuuint32_t)kW, (cuuint32_t)kH, 1, 1};
    cuuint32_t boxP[4] = {(cuuint32_t)kBX, (cuuint32_t)kTY, 1, 1};
    if (enc(&m[0], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void *)base, dims, strides, boxY,
                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
        enc(&m[1], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void *)base, dims, strides, boxP,
                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

size_t tensor_map_bytes() { return sizeof(CUtensorMap); }
void batch_tma_tile(int &bx, int &by)
{
    bx = kBX;
    by = kTY;
}

cudaError_t batch_stencil_tma(const BatchItem *items, int nitems, const BatchTma *cs, int grid,
                              int *err, cudaStream_t st)
{
    if (nitems <= 0) return cudaSuccess;
    static DeviceOnce once;
    const int smem = kSmemBytes;
    const cudaError_t e = once.allow_smem(smem, k_batch_stencil_tma<1>, k_batch_stencil_tma<2>);
    if (e != cudaSuccess) return e;
    // one row per thread while all items are resident at two CTAs per SM (as in stencil_f32_tma)
    if (nitems <= 2 * 152)
        k_batch_stencil_tma<1><<<grid, dim3(kTX, kTY), smem, st>>>(items, nitems, cs, err);
    else
        k_batch_stencil_tma<2><<<grid, dim3(kTX, kTY / 2), smem, st>>>(items, nitems, cs, err);
    note_launch();
    return cudaGetLastError();
}

bool stencil_tma_ok(const DevHam &H, const void *Y, const void *Yprev, const void *out, long ld)
{
    auto al = [](const void *p) { return ((uintptr_t)p & 15u) == 0; };
    return (H.n0 % 4 == 0) && (ld % 4 == 0) && al(Y) && al(out) && (!Yprev || al(Yprev)) &&
           al(H.Vf) && H.n0 <= (1 << 24) && H.n1 <= (1 << 24);
}

// z ranges per column of the two kernels above: 608 CTAs (four per SM) run at a time, each for
// its planes plus about eight plane-times for the twelve it reads ahead; the count with the
// fewest plane-times over all waves, of at least eight planes each.
static void f32_z_split(int n2, long tiles, int ncols, int &nzc, int &zchunk)
{
    constexpr int kFill = 8, kMinPlanes = 8;
    const long per = tiles * ncols;
    long best = -1;
    nzc = 1;
    zchunk = n2;
    for (int z = 1; z == 1 || (n2 / z >= kMinPlanes && (long)z * ncols <= 65535); ++z) {
        const int zc = (n2 + z - 1) / z, used = (n2 + zc - 1) / zc;
        const long cost = (per * used + 607) / 608 * (zc + kFill);
        if (best < 0 || cost < best) best = cost, nzc = used, zchunk = zc;
    }
}

static StepCoef2 pair_coef(const StepCoef<float> &cf)
{
    StepCoef2 c2;
    for (int r = 0; r <= kR; ++r) c2.w[r] = make_float2(cf.w[r], cf.w[r]);
    c2.c0 = make_float2(cf.c0, cf.c0);
    c2.alpha = make_float2(cf.alpha, cf.alpha);
    c2.nbeta = make_float2(-cf.beta, -cf.beta);
    return c2;
}

cudaError_t stencil_f32_copy(const DevHam &H, const float *Y, const float *Yprev, float *out,
                             int ncols, long ld, const StepCoef<float> &cf, cudaStream_t st)
{
    if (ncols <= 0) return cudaSuccess;
    if (ncols > 65535) return cudaErrorInvalidValue;
    static DeviceOnce once;
    const cudaError_t e = once.allow_smem(kSmemBytes, k_stencil_f32_copy);
    if (e != cudaSuccess) return e;
    const int gx = (H.n0 + kBX - 1) / kBX, gy = (H.n1 + kTY - 1) / kTY;
    int nzc, zchunk;
    f32_z_split(H.n2, (long)gx * gy, ncols, nzc, zchunk);
    k_stencil_f32_copy<<<dim3(gx, gy, ncols * nzc), dim3(kTX, kTY), kSmemBytes, st>>>(
        Y, Yprev, out, H.Vf, H.n0, H.n1, H.n2, ld, nzc, zchunk, pair_coef(cf));
    note_launch();
    return cudaGetLastError();
}

cudaError_t stencil_f32_tma(const DevHam &H, const float *Y, const float *Yprev, float *out,
                            int ncols, long ld, const StepCoef<float> &cf, int *err,
                            cudaStream_t st)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc;
    cudaError_t e = tensor_map_encoder(enc);
    if (e != cudaSuccess) return e;
    static DeviceOnce once;
    const int smem = kSmemBytes;
    e = once.allow_smem(smem, k_stencil_f32_tma<1>, k_stencil_f32_tma<2>);
    if (e != cudaSuccess) return e;
    // both maps view a block as (x, y, z, column); they differ in base and box
    auto encode = [&](CUtensorMap *m, const float *base, cuuint32_t bx, cuuint32_t by) {
        cuuint64_t dims[4] = {(cuuint64_t)H.n0, (cuuint64_t)H.n1, (cuuint64_t)H.n2,
                              (cuuint64_t)ncols};
        cuuint64_t strides[3] = {(cuuint64_t)H.n0 * 4, (cuuint64_t)H.n0 * H.n1 * 4,
                                 (cuuint64_t)ld * 4};
        cuuint32_t box[4] = {bx, by, 1, 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void *)base, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUtensorMap mapY, mapP;
    if (encode(&mapY, Y, kW, kH) != CUDA_SUCCESS) return cudaErrorInvalidValue;
    if (Yprev) {
        if (encode(&mapP, Yprev, kBX, kTY) != CUDA_SUCCESS) return cudaErrorInvalidValue;
    } else {
        mapP = mapY;  // never dereferenced: the kernel issues no Y_{j-1} load
    }
    const int gx = (H.n0 + kBX - 1) / kBX, gy = (H.n1 + kTY - 1) / kTY;
    int nzc, zchunk;
    f32_z_split(H.n2, (long)gx * gy, ncols, nzc, zchunk);
    dim3 grid(gx, gy, ncols * nzc);
    // Two rows per thread read 26 16-byte values from shared memory for eight nodes where one
    // row reads 19 for four, which is what bounds a full chip; a launch of one wave is
    // bound by its planes' latency, and the more threads are the faster: 96^3 x 128 380 -> 335 us,
    // 128^3 x 64 444 -> 403, 160^3 x 256 3.22 -> 3.07 ms; 32^3 x 16 (256 CTAs) 9.3 us with one
    // row, 9.8 with two, 48 x 40 x 36 x 60 (720 CTAs) 34 either way.
    auto launch = [&](auto nr) {
        constexpr int NR = decltype(nr)::value;
        k_stencil_f32_tma<NR><<<grid, dim3(kTX, kTY / NR), smem, st>>>(
            mapY, mapP, Yprev != nullptr, out, H.Vf, H.n0, H.n1, H.n2, ld, nzc, zchunk,
            pair_coef(cf), err);
    };
    if ((long)gx * gy * ncols * nzc > 4 * 152)
        launch(std::integral_constant<int, 2>{});
    else
        launch(std::integral_constant<int, 1>{});
    note_launch();
    return cudaGetLastError();
}

// Failure-detection self-test of the bounded mbarrier wait used above: the barrier expects
// two arrivals and gets one, so every thread's wait ends through its probe limit
// (~65 ms here); *err is set to 1 exactly as the stencil does on a lost TMA load.
__global__ void __launch_bounds__(32) k_mbar_selftest(int *err)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 2);
        mbar_fence_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_arrive(&bar);
    const bool ok = mbar_wait(&bar, 0u, 1u << 20);
    if (!ok && threadIdx.x == 0) atomicExch(err, 1);
}

cudaError_t mbar_selftest(int *err, cudaStream_t st)
{
    k_mbar_selftest<<<1, 32, 0, st>>>(err);
    note_launch();
    return cudaGetLastError();
}

}  // namespace sparc
