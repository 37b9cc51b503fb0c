// stencil_df.cu -- the FP64 fused stencil step on the integer, FP32 and FP64 pipes.
//
// The operation of stencil.cu (Eq. FD:Laplacian with the weights of Eq. weightsLap,
// zero-Dirichlet boundaries, V_eff and the Chebyshev three-term recurrence of Algorithm
// ChebychevFilter, Sec. 3.4), for FP64 blocks. GB300 issues FP64 at 1/64 of its FP32 rate, so a
// native FP64 stencil (37 FP64 multiply-adds per point) is bound by the FP64 pipe at a few per
// cent of HBM bandwidth. This kernel spends three FP64 operations per point:
//   * The Laplacian weights of radius n_o are rationals with one small common
//     denominator D (h^2 w_p = W_p / D, W_p integers, D = 831600 for every n_o), so
//     h^2 D L_h y = sum_p W_p S_p is an integer combination of the neighbour sums S_p.
//   * Every value of a column is put on a fixed-point grid: with |y| < 2^E over the
//     column (E from a per-column bound), y 2^(26-E) = d + 2^-32 r with d an integer truncated
//     toward zero (|d| < 2^26) and r the rest (|r| <= 2^32, same sign) rounded to FP32.
//   * Each radius sums its six neighbours' d in int32 (exact: |sum| < 6 * 2^26) and
//     applies W_p with one 32 x 32 -> 64-bit integer multiply-add (exact); the r parts are
//     summed and weighted in FP32 and the FP32 sum is rounded to an integer. The total
//     T ~ h^2 D L_h y 2^(26-E) is an int64 below 2^51 in magnitude (sum |W_p| < 2^24.1),
//     converted to FP64 exactly by one FP64 add (the 1.5 * 2^52 offset).
//   * The potential joins the integer sum: T += U y with U = (V_p - shift) / g, g =
//     (-1/2) / (D h^2), an integer plus a 30-bit fraction (V / g is tabulated once per context;
//     the shift is a launch constant), which leaves out = alpha g 2^(E-26) T - beta Y_{j-1}: two
//     more FP64 operations a point. Where that does not fit (a kinetic scale other than 1, a
//     potential beyond 2^25 units) the general form computes alpha (V_p - shift) y_p in FP64.
// Error: the rounding of r (2^-51 of the column's largest value per value) and the FP32
// rounding of the r sum and of the potential's product (about a unit of 2^(E-26), weighted by g ~
// 1e-5 at h = 0.3, at every radius): about 2^-42 of the column's largest value in the worst case,
// 1.3e-15 to 1.8e-15 of the largest |H X| measured at radii 1 to 6. The potential term, an FP64
// product of y itself in the general form, is thereby absolute in the column, as the
// Laplacian's part always is. A column
// whose bound is not finite (Inf or NaN anywhere in Y_j) gives NaN in every output value of
// the column. Each launch can raise the output's column bounds (atomicMax), which is how
// the filter hands the bound of Y_{j+1} to the next step without another pass over the
// block.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <type_traits>

#include "df.cuh"
#include "fx.cuh"
#include "internal.cuh"

namespace sparc {

// Coefficients of one launch. W, Wf: integer weights of h^2 D L_h (W[0]: the 3-D centre) and
// the same as FP32 (exact: |W| < 2^24).
struct FxCoef {
    int W[kRadius + 1];
    float Wf[kRadius + 1];
    int c0;        // integer-potential form: W[0] + floor(C), C the shift in units of 1 / vscale
    int c1;        // and the 30-bit fraction of C
    double ag;     // alpha (-1/2) ks / (D h^2)
    double mbeta;  // -beta
    double alpha, shift;  // the general form's potential factor
};

__device__ __forceinline__ double as_f64(double y) { return y; }
__device__ __forceinline__ double as_f64(float y) { return (double)y; }

constexpr double kMagic = 6755399441055744.0;  // 1.5 * 2^52 (the integer sums start at its bits)
constexpr long long kMagicBits = 0x4338000000000000ll;
constexpr int kDfPX = 16, kDfBY = 16;  // tile: 16 pairs (32 nodes) along x, 16 rows

// Two x-adjacent values; nv of them are inside the grid. VEC: rows are an even number of
// elements and the block is aligned to a pair, so nv is 0 or 2 and one load takes both.
template <typename TI>
struct Pair {
    TI a, b;
};
template <typename TI, bool VEC>
__device__ __forceinline__ Pair<TI> load_pair(const TI *p, int nv)
{
    Pair<TI> v = {(TI)0, (TI)0};
    if constexpr (VEC) {
        if (nv) {
            if constexpr (sizeof(TI) == 8) {
                const double2 d = *reinterpret_cast<const double2 *>(p);
                v.a = d.x, v.b = d.y;
            } else {
                const float2 d = *reinterpret_cast<const float2 *>(p);
                v.a = d.x, v.b = d.y;
            }
        }
    } else {
        if (nv > 0) v.a = p[0];
        if (nv > 1) v.b = p[1];
    }
    return v;
}

// A pair on the column's grid: (d_0, d_1, r_0, r_1).
template <typename TI>
__device__ __forceinline__ int4 to_grid_pair(Pair<TI> v, int E)
{
    const int2 x = to_grid(v.a, E), y = to_grid(v.b, E);
    return make_int4(x.x, y.x, x.y, y.y);
}

__device__ __forceinline__ float2 r_pair(const int4 &v)
{
    return make_float2(__int_as_float(v.z), __int_as_float(v.w));
}

// TI is the input block's type: FP64, or FP32 (the mixed-precision Rayleigh-Ritz step
// applies H in FP64 to the FP32 filtered block). A thread owns two x-adjacent nodes of a
// 32 x 16 tile and walks the tile's z range of one column; the 13 planes around it stay in
// registers on the column's grid, the current plane's tile with its x and y halos in shared
// memory as 16-byte pairs (d_0, d_1, r_0, r_1). The halo pairs (3 per row and side, 16 per
// row above and below: 288 for 256 threads) are loaded and converted by all threads, the
// last 32 by warp 0 alone. The next plane's halo pairs, queue entry, potential and Y_{j-1}
// are loaded during the current plane's compute (loading the potential and Y_{j-1} of the same
// plane at the start of its step instead took 1.6 ms against 1.13 for 96^3 x 128).
//
// What bounds it: latency (shared-memory reads and the FP64 pipe; issue slots 42% busy, the
// shared-memory pipe 58%, FP64 50%) at the 16 warps that 128 registers leave, which is also less
// than it wants: the usual form spills 128 bytes of stores and 312 of loads a thread over the 13
// unrolled planes (FP32 input 148 and 468, the general form 136 and 340). The pair
// form reads 18 16-byte values for the neighbours of two nodes (a thread per node: 48 of 8
// bytes), the r sums run on packed FP32 pairs, addresses, predicates and the barrier are shared
// by two nodes and the loads and stores are 16 bytes wide: about 162 thread instructions per
// node against 282. VINT (the integer potential, the usual form) takes alpha (V - shift) y out
// of the FP64 pipe: V / g on a 2^-30 grid of the weights' units (DevHam::uq) joins the centre
// weight, so a point costs three FP64 operations instead of four and no second read of y.
// A filter step of 96^3 x 128: 1.435 ms with one node per thread, 1.13 ms in this form; the
// degree-20 filter's error against 64-bit arithmetic went from 2.0e-14 to 1.4e-14 of its norm.
template <typename TI, bool VEC, bool VINT>
__global__ void __launch_bounds__(kDfPX *kDfBY, 2)
k_stencil_df(const TI *__restrict__ Yb, const double *Yprev, double *outb,
             const int2 *__restrict__ uq, const double *__restrict__ V, int n0, int n1, int n2,
             long ld, int nzc, int zchunk, FxCoef cf, const unsigned *__restrict__ bY,
             unsigned *bOut)
{
    constexpr int R = kRadius, PX = kDfPX, BY = kDfBY, NT = PX * BY, HP = R / 2;
    constexpr int SX = PX + 2 * HP, SY = BY + 2 * R;    // a plane's pairs and rows
    constexpr int NH = 2 * HP * BY + 2 * R * PX;        // halo pairs of a plane
    constexpr int NH2 = NH - NT;                        // second halo pairs: one warp's
    static_assert(R % 2 == 0 && NH2 > 0 && NH2 <= 32, "halo duties");
    // plane k is read from buffer b while plane k+1 is staged into buffer b ^ 1: one barrier
    // per plane
    __shared__ int4 s[2 * SY * SX];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * PX + tx;
    const int i0 = blockIdx.x * 2 * PX, j0 = blockIdx.y * BY;
    const int i = i0 + 2 * tx, j = j0 + ty;
    const int col = blockIdx.z / nzc;
    const int k0 = (blockIdx.z % nzc) * zchunk;
    const int k1 = min(n2, k0 + zchunk);
    const unsigned plane = (unsigned)n0 * (unsigned)n1;  // offsets in a column fit 32 bits
    const TI *Y = Yb + (long)col * ld;
    const double *P = Yprev ? Yprev + (long)col * ld : nullptr;
    double *out = outb + (long)col * ld;
    // nodes of this thread's pair inside the grid
    const int nv = (j < n1 && i < n0) ? min(n0 - i, 2) : 0;
    const unsigned pij = nv ? (unsigned)i + (unsigned)n0 * (unsigned)j : 0u;
    const int4 zero = make_int4(0, 0, 0, 0);
    // the column's scale: grid values in units of 2^(EY-26)
    const unsigned uy = bY[col];
    const bool nonfinite = ((uy >> 20) & 0x7ffu) == 0x7ffu;
    const int EY = bound_exponent(uy);
    // alpha g 2^(EY-26); NaN for a column whose bound is not finite, which makes every output
    // of the column NaN without a test per point
    const double gs = nonfinite ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(cf.ag, EY - 26);
    // halo duties: pair tid of the strips (left, right: HP x BY each; top, bottom: PX x R
    // each), and for warp 0 pair NT + tid; hs = shared-memory index, hn = nodes of the pair
    // inside the grid, hg = offset in the plane
    auto duty = [&](int h, int &hs, int &hn, unsigned &hg) {
        int sx, sy;
        if (h < 2 * HP * BY) {
            const int side = h / (HP * BY), rr = h % (HP * BY);
            sy = R + rr / HP;
            sx = side ? HP + PX + rr % HP : rr % HP;
        } else {
            const int w = h - 2 * HP * BY;
            const int side = w / (R * PX), rr = w % (R * PX);
            sx = HP + rr % PX;
            sy = side ? BY + R + rr / PX : rr / PX;
        }
        const int gx = i0 - R + 2 * sx, gy = j0 - R + sy;
        hs = sy * SX + sx;
        hn = (gx >= 0 && gx < n0 && gy >= 0 && gy < n1) ? min(n0 - gx, 2) : 0;
        hg = hn ? (unsigned)gx + (unsigned)n0 * (unsigned)gy : 0u;
    };
    int hs0, hn0, hs1 = 0, hn1 = 0;
    unsigned hg0, hg1 = 0u;
    duty(tid, hs0, hn0, hg0);
    const bool two = tid < NH2;
    if (two) duty(NT + tid, hs1, hn1, hg1);
    const int me = (ty + R) * SX + tx + HP;  // this thread's pair in a plane buffer

    int4 q[2 * R + 1];
#pragma unroll
    for (int t = 0; t < 2 * R + 1; ++t) {
        const int kk = k0 - R + t;
        const bool in = kk >= 0 && kk < n2;
        q[t] = to_grid_pair(load_pair<TI, VEC>(Y + (pij + (unsigned)(in ? kk : 0) * plane),
                                               in ? nv : 0), EY);
    }
    {
        const unsigned pk = (unsigned)k0 * plane;
        s[me] = q[R];
        s[hs0] = to_grid_pair(load_pair<TI, VEC>(Y + (hg0 + pk), hn0), EY);
        if (two) s[hs1] = to_grid_pair(load_pair<TI, VEC>(Y + (hg1 + pk), hn1), EY);
    }
    // the potential of the pair: (floor, fraction) of both nodes, or alpha (V - shift)
    auto load_u = [&](unsigned off, int4 &ui, double2 &uf) {
        if constexpr (VINT) {
            if constexpr (VEC) {
                if (nv) ui = *reinterpret_cast<const int4 *>(uq + off);
            } else {
                int2 a = make_int2(0, 0), b = a;
                if (nv > 0) a = uq[off];
                if (nv > 1) b = uq[off + 1];
                ui = make_int4(a.x, a.y, b.x, b.y);
            }
        } else {
            if (nv > 0) uf.x = cf.alpha * (V[off] - cf.shift);
            if (nv > 1) uf.y = cf.alpha * (V[off + 1] - cf.shift);
        }
    };
    int4 ui = zero;
    double2 uf = make_double2(0.0, 0.0);
    Pair<double> pc = {0.0, 0.0};
    load_u(pij + (unsigned)k0 * plane, ui, uf);
    if (P) pc = load_pair<double, VEC>(P + (pij + (unsigned)k0 * plane), nv);
    unsigned omax = 0u;
    __syncthreads();
    // The plane loop is unrolled 13 times, one copy per rotation of the z queue: in the
    // copy of phase PH, logical queue entry t (plane k - R + t) sits in q[(PH + t) % 13], so
    // the queue is never shifted.
    int k = k0;
    auto step = [&](auto phase) {
        constexpr int PH = decltype(phase)::value;
        constexpr int Q = 2 * R + 1;
        const int b = (k - k0) & 1;
        const unsigned pk = (unsigned)k * plane;
        // loads for plane k+1 (and the queue entry k+R+1), consumed after the compute
        const bool more = k + 1 < k1;
        const unsigned pk1 = pk + plane;
        Pair<TI> g0 = {(TI)0, (TI)0}, g1 = {(TI)0, (TI)0}, gq = {(TI)0, (TI)0};
        int4 un = zero;
        double2 ufn = make_double2(0.0, 0.0);
        Pair<double> pn = {0.0, 0.0};
        if (more) {
            load_u(pij + pk1, un, ufn);
            if (P) pn = load_pair<double, VEC>(P + (pij + pk1), nv);
            g0 = load_pair<TI, VEC>(Y + (hg0 + pk1), hn0);
            if (two) g1 = load_pair<TI, VEC>(Y + (hg1 + pk1), hn1);
        }
        const int kn = k + R + 1;
        if (kn < n2) gq = load_pair<TI, VEC>(Y + (pij + (unsigned)kn * plane), nv);
        if (nv) {
            // h^2 D L_h y in units of 2^(EY-26): exact integer sums of d, FP32 sums of r,
            // from the outermost radius (smallest weight) inwards, so that the FP32 sum is
            // rounded at its full magnitude only by its last terms. x values: index m is node
            // i - 6 + m, the pair itself m = 6, 7.
            const int4 *row = s + b * (SY * SX) + me;
            const int4 c = q[(PH + R) % Q];
            long long A0 = kMagicBits, A1 = kMagicBits;
            float2 rs = make_float2(0.0f, 0.0f);
            int xd[14];
            float xr[14];
            auto take = [&](int m, const int4 &v) {
                xd[m] = v.x, xd[m + 1] = v.y;
                xr[m] = __int_as_float(v.z), xr[m + 1] = __int_as_float(v.w);
            };
            take(6, c);
#pragma unroll
            for (int r = R; r >= 1; --r) {
                if (r % 2 == 0) {  // pairs -r/2 and r/2: nodes m = 6 - r, 7 - r and 6 + r, 7 + r
                    take(6 - r, row[-(r / 2)]);
                    take(6 + r, row[r / 2]);
                }
                // (an odd radius also needs the pairs one step further in)
                if (r % 2 == 1 && r > 1) {
                    take(6 - r + 1, row[-(r / 2)]);
                    take(6 + r - 1, row[r / 2]);
                }
                const int4 ya = row[r * SX], yb = row[-r * SX];
                const int4 za = q[(PH + R + r) % Q], zb = q[(PH + R - r) % Q];
                const int s0 = (xd[6 + r] + xd[6 - r] + ya.x) + (yb.x + za.x + zb.x);
                const int s1 = (xd[7 + r] + xd[7 - r] + ya.y) + (yb.y + za.y + zb.y);
                float2 xs;
                if (r % 2 == 0)
                    xs = __fadd2_rn(make_float2(xr[6 + r], xr[7 + r]),
                                    make_float2(xr[6 - r], xr[7 - r]));
                else
                    xs = make_float2(xr[6 + r] + xr[6 - r], xr[7 + r] + xr[7 - r]);
                const float2 sr = __fadd2_rn(__fadd2_rn(xs, __fadd2_rn(r_pair(ya), r_pair(yb))),
                                             __fadd2_rn(r_pair(za), r_pair(zb)));
                A0 += (long long)cf.W[r] * s0;
                A1 += (long long)cf.W[r] * s1;
                rs = __ffma2_rn(make_float2(cf.Wf[r], cf.Wf[r]), sr, rs);
            }
            double y0 = 0.0, y1 = 0.0;  // alpha (V - shift) y of the general form
            if constexpr (VINT) {
                // centre weight with the potential: integer part times d, the fraction times
                // d rounded to a unit, and both times r in FP32
                const int w0 = cf.c0 + ui.x, w1 = cf.c0 + ui.z;
                A0 += (long long)w0 * c.x;
                A1 += (long long)w1 * c.y;
                const int v0 = cf.c1 + ui.y, v1 = cf.c1 + ui.w;
                const long long f0 = (long long)v0 * c.x;
                const long long f1 = (long long)v1 * c.y;
                rs = __ffma2_rn(__fmul2_rn(make_float2((float)v0, (float)v1),
                                           make_float2(0x1p-30f, 0x1p-30f)), r_pair(c), rs);
                rs = __ffma2_rn(make_float2((float)w0, (float)w1), r_pair(c), rs);
                rs = __fmul2_rn(rs, make_float2(0x1p-29f, 0x1p-29f));
                // r sum and fraction in eighths of a unit, rounded to a unit together
                A0 += (long long)((__float2int_rn(rs.x) + (int)(f0 >> 27) + 4) >> 3);
                A1 += (long long)((__float2int_rn(rs.y) + (int)(f1 >> 27) + 4) >> 3);
            } else {
                A0 += (long long)cf.W[0] * c.x;
                A1 += (long long)cf.W[0] * c.y;
                rs = __ffma2_rn(make_float2(cf.Wf[0], cf.Wf[0]), r_pair(c), rs);
                rs = __fmul2_rn(rs, make_float2(0x1p-32f, 0x1p-32f));
                A0 += (long long)__float2int_rn(rs.x);
                A1 += (long long)__float2int_rn(rs.y);
                const Pair<TI> yc = load_pair<TI, VEC>(Y + (pij + pk), nv);  // (cached)
                y0 = uf.x * as_f64(yc.a);
                y1 = uf.y * as_f64(yc.b);
            }
            // T from the bits of T + 1.5 2^52, exactly
            const double T0 = __longlong_as_double(A0) - kMagic;
            const double T1 = __longlong_as_double(A1) - kMagic;
            const double o0 = fma(gs, T0, VINT ? cf.mbeta * pc.a : fma(cf.mbeta, pc.a, y0));
            const double o1 = fma(gs, T1, VINT ? cf.mbeta * pc.b : fma(cf.mbeta, pc.b, y1));
            double *o = out + (pij + pk);
            omax = max(omax, abs_hi_word(o0));
            if constexpr (VEC) {
                omax = max(omax, abs_hi_word(o1));
                *reinterpret_cast<double2 *>(o) = make_double2(o0, o1);
            } else {
                o[0] = o0;
                if (nv > 1) {
                    omax = max(omax, abs_hi_word(o1));
                    o[1] = o1;
                }
            }
        }
        // plane k - R leaves the queue; its slot takes plane k + R + 1 (logical entry 2R
        // of the next phase), and the next phase's centre is plane k + 1
        q[PH % Q] = to_grid_pair(gq, EY);
        ui = un;
        uf = ufn;
        pc = pn;
        if (more) {
            int4 *nb = s + (b ^ 1) * (SY * SX);
            nb[me] = q[(PH + 1 + R) % Q];
            nb[hs0] = to_grid_pair(g0, EY);
            if (two) nb[hs1] = to_grid_pair(g1, EY);
        }
        __syncthreads();
        ++k;
    };
#define SPARC_DF_STEP(P)                                                                 \
    if (k >= k1) break;                                                                  \
    step(std::integral_constant<int, P>{});
    for (;;) {
        SPARC_DF_STEP(0) SPARC_DF_STEP(1) SPARC_DF_STEP(2) SPARC_DF_STEP(3) SPARC_DF_STEP(4)
        SPARC_DF_STEP(5) SPARC_DF_STEP(6) SPARC_DF_STEP(7) SPARC_DF_STEP(8) SPARC_DF_STEP(9)
        SPARC_DF_STEP(10) SPARC_DF_STEP(11) SPARC_DF_STEP(12)
    }
#undef SPARC_DF_STEP
    if (bOut) {
        omax = __reduce_max_sync(0xffffffffu, omax);
        if ((tid & 31) == 0 && omax) raise_bound(bOut + col, omax);
    }
}

// uq = V vscale (vscale = -2 D h^2) as floor and 30-bit fraction; lim[0], lim[1]: smallest and
// largest floor, clamped to +-2^30 (what lies beyond, and NaN, counts as +-2^30: the host then
// takes the general form).
__global__ void __launch_bounds__(256)
k_potential_grid(const double *__restrict__ V, double vscale, int2 *__restrict__ uq, long n,
                 int *lim)
{
    constexpr int kBig = 1 << 30;
    int lo = kBig, hi = -kBig;
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long)gridDim.x * blockDim.x) {
        const double x = V[t] * vscale, f = floor(x);
        int a = kBig, b = 0;
        if (f > -(double)kBig && f < (double)kBig) {
            a = (int)f;
            b = (int)rint((x - f) * (double)kBig);
            if (b == kBig) ++a, b = 0;
        } else if (f <= -(double)kBig) {
            a = -kBig;
        }
        uq[t] = make_int2(a, b);
        lo = min(lo, a);
        hi = max(hi, a);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(lim, lo);
        atomicMax(lim + 1, hi);
    }
}

cudaError_t potential_grid(const double *V, double vscale, int2 *uq, long n, int *lim,
                           cudaStream_t st)
{
    const long b = (n + 255) / 256;
    k_potential_grid<<<(unsigned)(b < 152 * 8 ? b : 152 * 8), 256, 0, st>>>(V, vscale, uq, n, lim);
    note_launch();
    return cudaGetLastError();
}

// Whether the potential V - shift fits the integer centre weight (kinetic scale 1, and
// |W_0 + U| + 6 sum |W_p| within 2^25, so that |T| stays below 2^51), and the shift's parts.
static bool integer_potential(const DevHam &H, double shift, FxCoef &cf)
{
    if (H.kscale != 1.0 || !H.uq) return false;
    const double C = -shift * H.vscale, f = std::floor(C);
    if (!(std::fabs(C) < 1073741824.0)) return false;
    long long w = 0;
    for (int r = 1; r <= kRadius; ++r) w += 6ll * std::abs(H.wint[r]);
    const long long c = H.wint[0] + (long long)f;
    const long long lo = c + H.umin, hi = c + H.umax + 2;
    const long long m = std::max(lo < 0 ? -lo : lo, hi < 0 ? -hi : hi);
    if (m + w + 2 > (1ll << 25)) return false;
    cf.c0 = (int)c;
    cf.c1 = (int)std::min(1073741823.0, std::rint((C - f) * 1073741824.0));
    return true;
}

// z ranges per column: a CTA takes about (planes + kFill) plane-times (kFill: the 13 planes
// of its queue, read before the first one), and 304 CTAs (two per SM) run at a time. The count
// with the fewest plane-times over all waves is taken, with at least kMinPlanes planes each
// (H X of 24^3 x 12, whose 24 tiles leave most SMs idle as one range each: 66 us with ranges of
// at least 16 planes, 35 us so; a 70 x 61 x 53 x 33 filter of degree 10: 2.19 ms, 1.67 ms).
static void df_z_split(int n2, long tiles, int ncols, int &nzc, int &zchunk)
{
    constexpr int kFill = 5, kMinPlanes = 4;
    const long per = tiles * ncols;
    long best = -1;
    nzc = 1;
    zchunk = n2;
    for (int z = 1; z == 1 || (n2 / z >= kMinPlanes && (long)z * ncols <= 65535); ++z) {
        const int zc = (n2 + z - 1) / z;
        const int used = (n2 + zc - 1) / zc;
        const long cost = (per * used + 303) / 304 * (zc + kFill);
        if (best < 0 || cost < best) best = cost, nzc = used, zchunk = zc;
    }
}

template <typename TI>
static cudaError_t stencil_df_launch(const DevHam &H, const TI *Y, const double *Yprev,
                                     double *out, int ncols, long ld, double alpha,
                                     double shift, double beta, const unsigned *bY,
                                     unsigned *bOut, cudaStream_t st)
{
    if (ncols <= 0) return cudaSuccess;
    if (ncols > 65535 || !bY) return cudaErrorInvalidValue;
    FxCoef cf;
    for (int r = 0; r <= kRadius; ++r) {
        cf.W[r] = H.wint[r];
        cf.Wf[r] = (float)H.wint[r];
    }
    cf.ag = alpha * (-0.5 * H.kscale * H.wunit);
    cf.mbeta = -beta;
    cf.alpha = alpha;
    cf.shift = shift;
    cf.c0 = cf.c1 = 0;
    const bool vint = integer_potential(H, shift, cf);
    const int gx = (H.n0 + 2 * kDfPX - 1) / (2 * kDfPX), gy = (H.n1 + kDfBY - 1) / kDfBY;
    int nzc, zchunk;
    df_z_split(H.n2, (long)gx * gy, ncols, nzc, zchunk);
    dim3 grid(gx, gy, ncols * nzc), block(kDfPX, kDfBY);
    // pairs load as one when every row starts on a pair boundary
    auto al = [](const void *p, size_t b) { return ((uintptr_t)p & (b - 1)) == 0; };
    const bool vec = H.n0 % 2 == 0 && ld % 2 == 0 && al(Y, 2 * sizeof(TI)) && al(out, 16) &&
                     (!Yprev || al(Yprev, 16));
    auto go = [&](auto kernel) {
        kernel<<<grid, block, 0, st>>>(Y, Yprev, out, H.uq, H.V, H.n0, H.n1, H.n2, ld, nzc, zchunk,
                                       cf, bY, bOut);
    };
    if (vint && vec)
        go(k_stencil_df<TI, true, true>);
    else if (vint)
        go(k_stencil_df<TI, false, true>);
    else if (vec)
        go(k_stencil_df<TI, true, false>);
    else
        go(k_stencil_df<TI, false, false>);
    note_launch();
    return cudaGetLastError();
}

cudaError_t stencil_f64(const DevHam &H, const double *Y, const double *Yprev, double *out,
                        int ncols, long ld, double alpha, double shift, double beta,
                        const unsigned *bY, unsigned *bOut, cudaStream_t st)
{
    return stencil_df_launch<double>(H, Y, Yprev, out, ncols, ld, alpha, shift, beta, bY, bOut,
                                     st);
}

cudaError_t stencil_f32in_f64(const DevHam &H, const float *Y, double *out, int ncols, long ld,
                              const unsigned *bY, cudaStream_t st)
{
    return stencil_df_launch<float>(H, Y, nullptr, out, ncols, ld, 1.0, 0.0, 0.0, bY, nullptr,
                                    st);
}

}  // namespace sparc
