// evfdlb_2d.cu -- the two-dimensional tensor-product extension of the EV1
// time step (a plane periodic domain, homogeneous along z), FP32 with FP64
// conserved sums (and an FP64 build for parity checks).  The paper solves a
// 1D slab and names 2D as future work (Sec. IV); the 2D model extends its
// Sec. II-III statement:
//   * reduced distributions over p_z: F = int f dp_z, G = int f p_z^2/2 dp_z,
//     on the tensor product of the full-range Gauss-Hermite set of order Q
//     per axis, projected to order Q-1 per axis;
//   * reduced Shakhov equilibria and J1 (one transverse direction), written
//     as F_MB times a cubic polynomial in the peculiar velocity c, so that
//     their Hermite coefficients are sums of products of one-axis Gaussian
//     moments E[c^a psi_l(u + c)] (Stein's identity);
//   * the Eq. (force) integral over z as the in-plane kernel
//     g2(rho) = rho_vec gamma phi sigma^gamma int_{r > sigma} r^-(gamma+2) dz,
//     summed over the grid offsets inside the r_cut disc (rectangle rule);
//   * the Fischer-Methfessel average with chord weights 2 sqrt(sigma^2 - rho^2),
//     normalised; fourth-order gradients and WENO-5 along each axis.
// One RK stage is four launches:
//   k2_moments  raw moment sums of the stage input per node (the conserved
//               ones -- mass, momentum, energy -- to FP64 accuracy);
//   k2_fields   node fields per 16x16 node tile (force disc, FM average, chi,
//               gradients, transport) and the polynomial coefficients of the
//               equilibria;
//   k2_coll     per group of 16 nodes, all Q^2 velocities: force and collision
//               in velocity space, written with the Runge-Kutta base as the
//               stage's local increment V into the stage's output;
//   k2_adv      per 32x32 node tile and a run of velocities: WENO-5 faces along
//               x and y, added to V and the input in place.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "evfdlb_device.cuh"
#include "evfdlb_internal.h"

namespace evfdlb {

struct Slab2 {
    int nx, ny, Q, relax;
    long long N;          // nodes, nx * ny
    int nft, nfm;         // force and Fischer-Methfessel taps
    int fm_staged;        // whether k2_fields stages the latter in shared memory
    int Mf, mfm;          // their radii in nodes
    double dx;
};

// The model constants a kernel multiplies by, in its precision R, rounded on
// the host.  An FP32 kernel that takes them as doubles converts them on the
// FP64 pipe, and the compiler forms such conversions (and a compare of a
// double stage weight) again inside the plane loop instead of holding their
// results: they kept that pipe 65 % busy in the FP32 advection.
template <typename R>
struct Par2 {
    R k12, weno_eps, b, eta_coef, mu0_coef;               // k12 = 1 / (12 dx)
    // one Shu-Osher stage alpha base + beta (h + dt R) in increment form,
    //   h + (V + ca (xi_x df_x + xi_y df_y)),  V = alpha (base - h) + cb RL
    // (alpha + beta = 1): cb = beta dt, ca = -beta dt / dx.  The right-hand
    // side itself is cb = 1, ca = -1 / dx without h.
    R alpha, cb, ca, hs;                                   // hs: 1 for a stage, 0 for a right-hand side
    int with_base;                                         // alpha != 0
};

// The 2D state interleaves the distributions: pair (F, G) of velocity k at
// node i is element k N + i of an R2 array, so that every kernel moves both
// with one 8-byte (FP32) or 16-byte (FP64) access.
template <typename R>
using Pair = typename std::conditional<std::is_same<R, float>::value, float2, double2>::type;

// Arithmetic on pairs: FP32 in packed instructions (two lanes each; one may
// take a literal for both), FP64 componentwise.
__device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }
__device__ __forceinline__ double2 splat(double a) { return make_double2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, splat(-1.f), a); }
__device__ __forceinline__ double2 sub2(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double2 mul2(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}

// raw moment sums per node ([kNumMom2][N], FP64)
enum { M2_S0 = 0, M2_S1X, M2_S1Y, M2_S2XX, M2_S2YY, M2_G0, M2_S2XY, M2_S3X, M2_S3Y, M2_G1X, M2_G1Y, kNumMom2 };
// node outputs of k2_fields ([kNumFld2][N], precision R): n, ux, uy, T, nu,
// Fx, Fy, then the coefficients P_ab (times n) of the F and G polynomials in
// the order (a,b) = (0,0) (1,0) (0,1) (2,0) (1,1) (0,2) (3,0) (2,1) (1,2) (0,3)
enum { F2_N = 0, F2_UX, F2_UY, F2_T, F2_NU, F2_FX, F2_FY, F2_PF = 7, F2_PG = 17, kNumFld2 = 27 };

constexpr int kTile2 = 16;     // k2_fields tile edge
constexpr int kNB = 16;        // nodes per k2_coll CTA (half a warp: a lane per node and distribution)
static_assert(kNB == 16, "k2_coll maps the 32 lanes of a warp to 16 nodes x 2 distributions");

__device__ __forceinline__ int wrapi(int i, int n) {
    int r = i % n;
    return r < 0 ? r + n : r;
}

// ---------------------------------------------------------------------------
// k2_moments: per node, raw sums over the Q^2 velocities.  Conserved sums
// (S0, S1, S2xx, S2yy, G0) are formed from the row and column sums of the
// velocity grid.  For an FP32 state each 16-term row or column sum is a
// compensated FP32 sum kept as an unevaluated pair (TwoSum, Knuth), and the
// rows and columns are combined in float-float arithmetic (TwoSum and the
// FMA TwoProduct against the velocity powers split into float pairs,
// Ogita-Rump-Oishi): about 2^-44 of the sum of magnitudes, FP64 quality on
// the FP32 pipe (the FP64 pipe of this GPU runs at 1/64 of the FP32 rate).
// The heat-flux sums are plain R sums.  Outputs: the FP64 raw sums (when
// `mom` is given) and, for an FP32 state, the node primitives n, u, T, q in
// FP32 (when `prf` is given: what the stage's field kernel reads).
// ---------------------------------------------------------------------------
enum { P2_N = 0, P2_UX, P2_UY, P2_T, P2_QX, P2_QY, kNumPrf2 };

// velocity powers of the velocity set, passed by value (kernel parameter
// space, read as constant operands once the loops are unrolled)
template <typename R>
struct Pow2 {
    R v[16], v2[16], v3[16];            // xi, xi^2, xi^3 in R
    float h[16], l[16], h2[16], l2[16];  // xi and xi^2 (FP64) as float pairs
};

template <typename R>
struct CompSum {                       // R = double: plain accumulation
    double s = 0.0;
    __device__ __forceinline__ void add(R x) { s += (double)x; }
};
template <>
struct CompSum<float> {                // TwoSum: s + c carries the exact sum to O(n u^2)
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) {
        const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z)));
        s = t;
    }
};

// float-float accumulator (hi, lo)
struct FF {
    float h = 0.0f, l = 0.0f;
    // += (a + b), a pair
    __device__ __forceinline__ void add(float a, float b) {
        const float t = __fadd_rn(h, a), z = __fsub_rn(t, h);
        const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, z)), __fsub_rn(a, z));
        l = __fadd_rn(l, __fadd_rn(e, b));
        h = t;
    }
    // += (xh + xl)(a + b); the xl b term is below the pair's precision
    __device__ __forceinline__ void fma2(float xh, float xl, float a, float b) {
        const float p = __fmul_rn(xh, a), pe = fmaf(xh, a, -p);
        const float t = __fadd_rn(h, p), z = __fsub_rn(t, h);
        const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, z)), __fsub_rn(p, z));
        l = __fadd_rn(l, __fadd_rn(e, pe));
        l = fmaf(xh, b, l);
        l = fmaf(xl, a, l);
        h = t;
    }
    __device__ __forceinline__ float value() const { return h + l; }
    __device__ __forceinline__ double value64() const { return (double)h + (double)l; }
};

// Partial raw sums of one node over half of the y velocities (ky = K0 ..
// K0 + Q/2 - 1) and all x velocities.  Conserved sums: float-float pairs for
// an FP32 state (`a*`, `b*`), plain FP64 for an FP64 state (`d*`); heat-flux
// sums in R.  Every sum is linear in the state, so the two halves add.
template <typename R>
struct MomPart {
    FF a0, a1, a2, a3, b1, b2;               // S0, S1x, S2xx, G0, S1y, S2yy (FP32 state)
    double d0 = 0, d1x = 0, d2xx = 0, dg0 = 0, d1y = 0, d2yy = 0;   // (FP64 state)
    R s2xy = 0, s3x = 0, s3y = 0, g1x = 0, g1y = 0;
};
constexpr int kMomX = 17;                    // values exchanged between the halves

template <typename R, int Q, int K0>
__device__ __forceinline__ void moments_half(const Pair<R>* __restrict__ f, long long N, const Pow2<R>& pw,
                                             const R (*sv)[Q], const float (*sh)[Q], MomPart<R>& P) {
    constexpr bool F32 = std::is_same<R, float>::value;
    constexpr int QH = Q / 2;
    CompSum<R> col[QH];
    // the next row's loads are in flight while a row is summed
    Pair<R> hn[QH];
#pragma unroll
    for (int j = 0; j < QH; ++j) hn[j] = f[(long long)(K0 + j) * N];
    for (int kx = 0; kx < Q; ++kx) {
        CompSum<R> rowF, rowG;
        R p1 = 0, p2 = 0, p3 = 0, pg = 0;          // sum y f, y^2 f, y^3 f, y g over the half row
        Pair<R> hc[QH];
#pragma unroll
        for (int j = 0; j < QH; ++j) hc[j] = hn[j];
        if (kx + 1 < Q) {
            const Pair<R>* q = f + (long long)((kx + 1) * Q + K0) * N;
#pragma unroll
            for (int j = 0; j < QH; ++j) hn[j] = q[j * N];
        }
#pragma unroll
        for (int j = 0; j < QH; ++j) {
            const R fv = hc[j].x, gv = hc[j].y;
            rowF.add(fv);
            rowG.add(gv);
            col[j].add(fv);
            p1 = fma(pw.v[K0 + j], fv, p1);
            p2 = fma(pw.v2[K0 + j], fv, p2);
            p3 = fma(pw.v3[K0 + j], fv, p3);
            pg = fma(pw.v[K0 + j], gv, pg);
        }
        const R xr = sv[0][kx], x2r = sv[1][kx];
        R rfr, rgr;                                 // half-row sums in R
        if constexpr (F32) {
            P.a0.add(rowF.s, rowF.c);
            P.a1.fma2(sh[0][kx], sh[1][kx], rowF.s, rowF.c);
            P.a2.fma2(sh[2][kx], sh[3][kx], rowF.s, rowF.c);
            P.a3.add(rowG.s, rowG.c);
            rfr = rowF.s + rowF.c;
            rgr = rowG.s + rowG.c;
        } else {
            P.d0 += rowF.s;
            P.d1x = fma((double)xr, rowF.s, P.d1x);
            P.d2xx = fma((double)x2r, rowF.s, P.d2xx);
            P.dg0 += rowG.s;
            rfr = (R)rowF.s;
            rgr = (R)rowG.s;
        }
        // sum (x^2 + y^2) f = x^2 rowF + p2;  sum y (x^2 + y^2) f = x^2 p1 + p3
        P.s2xy = fma(xr, p1, P.s2xy);
        P.s3x = fma(xr, fma(x2r, rfr, p2), P.s3x);
        P.s3y += fma(x2r, p1, p3);
        P.g1x = fma(xr, rgr, P.g1x);
        P.g1y += pg;
    }
#pragma unroll
    for (int j = 0; j < QH; ++j) {
        if constexpr (F32) {
            P.b1.fma2(pw.h[K0 + j], pw.l[K0 + j], col[j].s, col[j].c);
            P.b2.fma2(pw.h2[K0 + j], pw.l2[K0 + j], col[j].s, col[j].c);
        } else {
            P.d1y = fma((double)pw.v[K0 + j], col[j].s, P.d1y);
            P.d2yy = fma((double)pw.v2[K0 + j], col[j].s, P.d2yy);
        }
    }
}

// FP32: three CTAs per SM, with the registers of two rows of loads; the FP64
// build (parity checks) keeps its registers
template <typename R>
constexpr int moments_min_blocks() { return std::is_same<R, float>::value ? 3 : 1; }

// Per CTA pass 128 nodes: warp pair (2p, 2p+1) takes nodes 32p .. 32p+31,
// the even warp the y velocities of the first half, the odd warp the second
// half (each load instruction reads 32 consecutive nodes of one plane); the
// odd warp hands its partial sums to the even one through shared memory.
template <typename R, int Q>
__global__ void __launch_bounds__(256, moments_min_blocks<R>())
k2_moments(Slab2 s, const Pow2<R> pw, const Pair<R>* __restrict__ st, double* __restrict__ mom, float* __restrict__ prf,
           unsigned* err) {
    constexpr bool F32 = std::is_same<R, float>::value;
    constexpr int kNodes = 128;
    static_assert(Q % 2 == 0, "the y velocities split in two halves");
    const long long N = s.N;
    // the row loop indexes the powers at run time: from shared memory
    __shared__ R sv[2][Q];
    __shared__ float sh[4][Q];
    __shared__ R xch[kMomX][kNodes];
    if (threadIdx.x < Q) {
        const int k = threadIdx.x;
        sv[0][k] = pw.v[k];
        sv[1][k] = pw.v2[k];
        sh[0][k] = pw.h[k];
        sh[1][k] = pw.l[k];
        sh[2][k] = pw.h2[k];
        sh[3][k] = pw.l2[k];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = warp & 1;
    const int slot = (warp >> 1) * 32 + lane;
    for (long long b0 = (long long)blockIdx.x * kNodes; b0 < N; b0 += (long long)gridDim.x * kNodes) {
        const long long i = b0 + slot;
        MomPart<R> P;
        if (i < N) {
            if (half == 0) moments_half<R, Q, 0>(st + i, N, pw, sv, sh, P);
            else moments_half<R, Q, Q / 2>(st + i, N, pw, sv, sh, P);
        }
        if (half == 1) {
            R v[kMomX];
            if constexpr (F32) {
                const float w[12] = {P.a0.h, P.a0.l, P.a1.h, P.a1.l, P.a2.h, P.a2.l,
                                     P.a3.h, P.a3.l, P.b1.h, P.b1.l, P.b2.h, P.b2.l};
#pragma unroll
                for (int q = 0; q < 12; ++q) v[q] = w[q];
            } else {
                const double w[12] = {P.d0, P.d1x, P.d2xx, P.dg0, P.d1y, P.d2yy, 0, 0, 0, 0, 0, 0};
#pragma unroll
                for (int q = 0; q < 12; ++q) v[q] = w[q];
            }
            v[12] = P.s2xy;
            v[13] = P.s3x;
            v[14] = P.s3y;
            v[15] = P.g1x;
            v[16] = P.g1y;
#pragma unroll
            for (int q = 0; q < kMomX; ++q) xch[q][slot] = v[q];
        }
        __syncthreads();
        if (half == 0 && i < N) {
            const R s2xy = P.s2xy + xch[12][slot], s3x = P.s3x + xch[13][slot], s3y = P.s3y + xch[14][slot];
            const R g1x = P.g1x + xch[15][slot], g1y = P.g1y + xch[16][slot];
            double S0, S1x, S1y, S2xx, S2yy, G0;
            float n32 = 0, S1x32 = 0, S1y32 = 0, S2xx32 = 0, S2yy32 = 0, G032 = 0;
            if constexpr (F32) {
                P.a0.add(xch[0][slot], xch[1][slot]);
                P.a1.add(xch[2][slot], xch[3][slot]);
                P.a2.add(xch[4][slot], xch[5][slot]);
                P.a3.add(xch[6][slot], xch[7][slot]);
                P.b1.add(xch[8][slot], xch[9][slot]);
                P.b2.add(xch[10][slot], xch[11][slot]);
                n32 = P.a0.value(); S1x32 = P.a1.value(); S1y32 = P.b1.value();
                S2xx32 = P.a2.value(); S2yy32 = P.b2.value(); G032 = P.a3.value();
                if (!isfinite(n32) || !isfinite(S2xx32 + S2yy32 + G032)) atomicOr(err, ERR_NONFINITE);
                S0 = P.a0.value64(); S1x = P.a1.value64(); S1y = P.b1.value64();
                S2xx = P.a2.value64(); S2yy = P.b2.value64(); G0 = P.a3.value64();
            } else {
                S0 = P.d0 + xch[0][slot]; S1x = P.d1x + xch[1][slot]; S2xx = P.d2xx + xch[2][slot];
                G0 = P.dg0 + xch[3][slot]; S1y = P.d1y + xch[4][slot]; S2yy = P.d2yy + xch[5][slot];
                if (!isfinite(S0) || !isfinite(S2xx + S2yy + G0)) atomicOr(err, ERR_NONFINITE);
            }
            if (mom) {
                mom[M2_S0 * N + i] = S0;
                mom[M2_S1X * N + i] = S1x;
                mom[M2_S1Y * N + i] = S1y;
                mom[M2_S2XX * N + i] = S2xx;
                mom[M2_S2YY * N + i] = S2yy;
                mom[M2_G0 * N + i] = G0;
                mom[M2_S2XY * N + i] = (double)s2xy;
                mom[M2_S3X * N + i] = (double)s3x;
                mom[M2_S3Y * N + i] = (double)s3y;
                mom[M2_G1X * N + i] = (double)g1x;
                mom[M2_G1Y * N + i] = (double)g1y;
            }
            if constexpr (F32) {
                if (prf) {
                    // primitives in FP32: u = S1/n, (3/2) n T = (S2xx + S2yy)/2 + G0 - n u^2/2,
                    // q_i = sum c_i (c^2/2 F + G) expanded in the raw sums
                    const float n = n32, ux = S1x32 / n, uy = S1y32 / n;
                    const float u2 = ux * ux + uy * uy, S2 = S2xx32 + S2yy32;
                    const float T = (2.0f / 3.0f) * ((0.5f * S2 + G032) / n - 0.5f * u2);
                    const float uS1 = ux * S1x32 + uy * S1y32;
                    const float qx = 0.5f * (s3x - 2.0f * (ux * S2xx32 + uy * s2xy) + u2 * S1x32 - ux * S2 +
                                             2.0f * ux * uS1 - ux * u2 * n) + g1x - ux * G032;
                    const float qy = 0.5f * (s3y - 2.0f * (ux * s2xy + uy * S2yy32) + u2 * S1y32 - uy * S2 +
                                             2.0f * uy * uS1 - uy * u2 * n) + g1y - uy * G032;
                    prf[P2_N * N + i] = n;
                    prf[P2_UX * N + i] = ux;
                    prf[P2_UY * N + i] = uy;
                    prf[P2_T * N + i] = T;
                    prf[P2_QX * N + i] = qx;
                    prf[P2_QY * N + i] = qy;
                }
            }
        }
        __syncthreads();                               // xch is reused by the next pass
    }
}

// n, u, T of one node from its raw sums
__device__ __forceinline__ void prim2(const double* __restrict__ mom, long long N, long long i, double& n, double& ux,
                                      double& uy, double& T) {
    n = mom[M2_S0 * N + i];
    ux = mom[M2_S1X * N + i] / n;
    uy = mom[M2_S1Y * N + i] / n;
    // (3/2) n T = (S2xx + S2yy)/2 + G0 - n u^2 / 2
    T = (2.0 / 3.0) * ((0.5 * (mom[M2_S2XX * N + i] + mom[M2_S2YY * N + i]) + mom[M2_G0 * N + i]) / n -
                       0.5 * (ux * ux + uy * uy));
}

// ---------------------------------------------------------------------------
// k2_fields: node fields of a 16x16 tile, computed in the state precision R
// (the FP32 build reads the FP32 primitives of k2_moments; the FP64 build
// derives them from the FP64 raw sums).
//
// Force disc (rectangle rule over the grid offsets inside r_cut; the taps
// carry dx^2 g2): g2 is radial, so g2x(-a, b) = -g2x(a, b) and
// g2y(-a, b) = g2y(a, b) exactly, and one pass over the offset column pair
// (a, -a) adds g2x (n_+ - n_-) and g2y (n_+ + n_-) (column a = 0 with halved
// g2y).  Each warp takes a host-balanced list of column pairs over the whole
// tile: lane = (column, block of 8 rows); the pass walks the rows of the
// column once and keeps the last 8 weight pairs in a register ring, so each
// staged density pair feeds 16 FMAs (8 rows x 2 components).  The per-warp
// partial forces are summed in warp order (deterministic).
// ---------------------------------------------------------------------------
constexpr int kFRows = 8;            // rows of a force register block (= ring length)
constexpr int kFMaxWarps = 24;       // most warps of a CTA
constexpr int kFPlanHead = 28;       // plan header: a prefix offset per warp and the end, padded to 16 bytes
static_assert(kTile2 == 16 && 2 * kFRows == kTile2 && kFPlanHead > kFMaxWarps && kFPlanHead % 4 == 0,
              "force mapping: 16 x 2 lanes x 8 rows");

// pitch of the staged density row: >= W and = 2 (mod 4), so that rows 8
// apart (the two row blocks of a warp) fall 16 banks apart
__host__ __device__ inline int fields_pitch(int W) { return W + ((6 - W % 4) % 4); }

// nfm: the Fischer-Methfessel taps staged beside the densities (0: none)
template <typename R>
__host__ __device__ inline size_t fields_smem_bytes(int Mf, int mfm, int nfm, int warps) {
    const int H = Mf > mfm + 2 ? Mf : mfm + 2, W = kTile2 + 2 * H, E = kTile2 + 4, Wr = fields_pitch(W);
    const size_t nr = (size_t)(W + kFRows) * Wr, pf = 2 * (size_t)warps * kTile2 * kTile2;
    return sizeof(R) * ((nr > pf ? nr : pf) + 5 * (size_t)E * E + nfm) + sizeof(int) * (size_t)nfm;
}
constexpr size_t kFSmemLimit = 227 * 1024;

template <typename R, int NW>
__global__ void __launch_bounds__(32 * NW)
k2_fields(Slab2 s, const Par2<R> pr, const double* __restrict__ mom, const float* __restrict__ prf, const R* __restrict__ ftw,
          const int* __restrict__ fplan, const int* __restrict__ fm_off, const R* __restrict__ fm_w,
          R* __restrict__ fld, unsigned* err) {
    constexpr bool F32 = std::is_same<R, float>::value;
    using R2 = typename std::conditional<F32, float2, double2>::type;
    extern __shared__ __align__(16) unsigned char sm2raw[];
    R* sm2 = reinterpret_cast<R*>(sm2raw);
    const int H = max(s.Mf, s.mfm + 2), W = kTile2 + 2 * H, E = kTile2 + 4, Wr = fields_pitch(W);
    R* Nr = sm2;                      // n on the tile + H halo, [W + 8][Wr]; rows W.. are zero
    R* U = sm2 + max((W + kFRows) * Wr, 2 * NW * kTile2 * kTile2);
    R* V = U + E * E;                 // ux, uy, T, X, chi on the tile + 2, [E][E] each
    R* Tt = V + E * E;
    R* Xt = Tt + E * E;
    R* Ct = Xt + E * E;
    const int nx = s.nx, ny = s.ny;
    const long long N = s.N;
    const int x0 = blockIdx.x * kTile2, y0 = blockIdx.y * kTile2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a warp per row; one wrap is enough wherever the halo is narrower than the grid
    auto wrap1 = [](int i, int n) {
        i = i < 0 ? i + n : (i >= n ? i - n : i);
        return (unsigned)i < (unsigned)n ? i : wrapi(i, n);
    };
    for (int cy = warp; cy < W + kFRows; cy += NW) {
        const long long row = (long long)wrap1(y0 - H + cy, ny) * nx;
        for (int cx = lane; cx < W; cx += 32) {
            R n = R(0);
            if (cy < W) {
                const long long i = row + wrap1(x0 - H + cx, nx);
                if constexpr (F32) n = prf[P2_N * N + i];
                else n = mom[M2_S0 * N + i];
            }
            Nr[cy * Wr + cx] = n;
        }
    }
    // Fischer-Methfessel taps as offsets in the staged density, where there is
    // room for them: the disc of sigma = 43 dx has 5800 taps (47 KB in FP32), and with
    // r_cut = 2.5 sigma the densities alone take 221 KB.  Else they are read from global
    // memory below.
    R* fw = Ct + E * E;
    int* fo = reinterpret_cast<int*>(fw + s.nfm);
    for (int t = threadIdx.x; s.fm_staged && t < s.nfm; t += 32 * NW) {
        fw[t] = fm_w[t];
        fo[t] = fm_off[2 * t + 1] * Wr + fm_off[2 * t];
    }
    for (int e = threadIdx.x; e < E * E; e += blockDim.x) {
        const int cy = e / E, cx = e % E;
        const long long i = (long long)wrap1(y0 - 2 + cy, ny) * nx + wrap1(x0 - 2 + cx, nx);
        if constexpr (F32) {
            U[e] = prf[P2_UX * N + i];
            V[e] = prf[P2_UY * N + i];
            Tt[e] = prf[P2_T * N + i];
        } else {
            double n, ux, uy, T;
            prim2(mom, N, i, n, ux, uy, T);
            U[e] = ux;
            V[e] = uy;
            Tt[e] = T;
        }
    }
    __syncthreads();
    // Fischer-Methfessel average, chi (Eq. (carnstar)) and X = n^2 chi T on the tile + 2
    for (int e = threadIdx.x; e < E * E; e += blockDim.x) {
        const int cy = e / E, cx = e % E;
        const int hy = cy - 2 + H, hx = cx - 2 + H;   // position in the halo array
        R nb = R(0);
        const R* c = Nr + hy * Wr + hx;
        if (s.fm_staged) {
#pragma unroll 4
            for (int t = 0; t < s.nfm; ++t) nb = fma(fw[t], c[fo[t]], nb);
        } else {
            for (int t = 0; t < s.nfm; ++t)
                nb = fma(__ldg(fm_w + t), c[__ldg(fm_off + 2 * t + 1) * Wr + __ldg(fm_off + 2 * t)], nb);
        }
        const R eta = pr.eta_coef * nb, om = R(1) - eta;
        const R chi = (R(2) - eta) / (R(2) * om * om * om);
        const R n = Nr[hy * Wr + hx];
        Ct[e] = chi;
        Xt[e] = n * n * chi * Tt[e];
    }
    // force over the disc
    const int fxl = lane & 15, yb = lane >> 4;
    R ax[kFRows], ay[kFRows];
#pragma unroll
    for (int k = 0; k < kFRows; ++k) ax[k] = ay[k] = R(0);
    {
        const int4* ent = reinterpret_cast<const int4*>(fplan + kFPlanHead);
        const int e1 = fplan[warp + 1];
        for (int e = fplan[warp]; e < e1; ++e) {
            const int4 en = ent[e];          // column a, weight offset, steps (multiple of 8), half height w
            const int a = en.x, steps = en.z, w = en.w;
            const R* pp = Nr + (yb * kFRows - w + H) * Wr + fxl + H + a;   // n(x + a, row of step 0)
            const R* pm = pp - 2 * a;                                       // n(x - a, ...)
            const R2* g = reinterpret_cast<const R2*>(ftw) + en.y;
            // ring: slot (j & 7) holds the weights of step j, i.e. of offset b = j - w
            R gx[kFRows], gy[kFRows];
#pragma unroll
            for (int k = 0; k < kFRows; ++k) gx[k] = gy[k] = R(0);
            for (int j0 = 0; j0 < steps; j0 += kFRows) {
#pragma unroll
                for (int P = 0; P < kFRows; ++P) {
                    const R vp = pp[(j0 + P) * Wr], vm = pm[(j0 + P) * Wr];
                    const R2 gg = __ldg(g + j0 + P);
                    gx[P] = gg.x;
                    gy[P] = gg.y;
                    const R dd = vp - vm, ss = vp + vm;
                    // row k of the block takes offset b = (j - k) - w: the weights of step j - k
#pragma unroll
                    for (int k = 0; k < kFRows; ++k) {
                        ax[k] = fma(gx[(P - k) & (kFRows - 1)], dd, ax[k]);
                        ay[k] = fma(gy[(P - k) & (kFRows - 1)], ss, ay[k]);
                    }
                }
            }
        }
    }
    constexpr int NN = kTile2 * kTile2;
    const int node = threadIdx.x % NN, tx = node % kTile2, ty = node / kTile2;
    const R n = Nr[(ty + H) * Wr + tx + H];
    __syncthreads();                  // density reads done: its space takes the partial forces
    R* Pf = sm2;                      // [NW][2][NN]
#pragma unroll
    for (int k = 0; k < kFRows; ++k) {
        const int o = (yb * kFRows + k) * kTile2 + fxl;
        Pf[(2 * warp) * NN + o] = ax[k];
        Pf[(2 * warp + 1) * NN + o] = ay[k];
    }
    __syncthreads();
    R fx = R(0), fy = R(0);
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        fx += Pf[(2 * w) * NN + node];
        fy += Pf[(2 * w + 1) * NN + node];
    }
    const int x = x0 + tx, y = y0 + ty;
    if (threadIdx.x >= NN || x >= nx || y >= ny) return;
    const long long i = (long long)y * nx + x;
    const int c = (ty + 2) * E + (tx + 2);
    const R k12 = pr.k12;
    auto d4x = [&](const R* f) { return (f[c - 2] - R(8) * f[c - 1] + R(8) * f[c + 1] - f[c + 2]) * k12; };
    auto d4y = [&](const R* f) { return (f[c - 2 * E] - R(8) * f[c - E] + R(8) * f[c + E] - f[c + 2 * E]) * k12; };
    const R ux = U[c], uy = V[c], T = Tt[c], X = Xt[c], chi = Ct[c];
    const R Ax = d4x(Xt) / X, Ay = d4y(Xt) / X, Bx = d4x(Tt) / T, By = d4y(Tt) / T;
    const R Dxx = d4x(U), Dxy = d4x(V), Dyx = d4y(U), Dyy = d4y(V);
    // heat flux q_i = sum c_i (c^2/2 F + G)
    R qx, qy;
    if constexpr (F32) {
        qx = prf[P2_QX * N + i];
        qy = prf[P2_QY * N + i];
    } else {
        const double S0 = mom[M2_S0 * N + i], S1x = mom[M2_S1X * N + i], S1y = mom[M2_S1Y * N + i];
        const double S2xx = mom[M2_S2XX * N + i], S2yy = mom[M2_S2YY * N + i], S2xy = mom[M2_S2XY * N + i];
        const double S3x = mom[M2_S3X * N + i], S3y = mom[M2_S3Y * N + i], G0 = mom[M2_G0 * N + i];
        const double G1x = mom[M2_G1X * N + i], G1y = mom[M2_G1Y * N + i];
        const double u2 = ux * ux + uy * uy, S2 = S2xx + S2yy;
        const double uS1 = ux * S1x + uy * S1y;
        qx = 0.5 * (S3x - 2.0 * (ux * S2xx + uy * S2xy) + u2 * S1x - ux * S2 + 2.0 * ux * uS1 - ux * u2 * S0) +
             G1x - ux * G0;
        qy = 0.5 * (S3y - 2.0 * (ux * S2xy + uy * S2yy) + u2 * S1y - uy * S2 + 2.0 * uy * uS1 - uy * u2 * S0) +
             G1y - uy * G0;
    }
    // transport, Eqs. (viscosity), (tau), (prandtl)
    const R c16 = R((4.0 / 25.0) * (1.0 + 12.0 / M_PI)), c9 = R((9.0 / 25.0) * (1.0 + 32.0 / (9.0 * M_PI)));
    const R bn = pr.b * n, xx = bn * chi;
    const R mu = pr.mu0_coef * sqrt(T) * (R(1) / chi + R(0.8) * bn + c16 * bn * bn * chi);
    const R tau = mu / (n * T * (R(1) + R(0.4) * xx));
    const R Pr = R(2.0 / 3.0) * (R(1) + R(0.6) * xx) * (R(1) + R(0.8) * xx + c16 * xx * xx) /
                 ((R(1) + R(0.4) * xx) * (R(1) + R(1.2) * xx + c9 * xx * xx));
    const R nu = (s.relax == EVFDLB_RELAX_INV_TAU) ? R(1) / tau : chi / tau;
    if (!(n > R(0)) || !(T > R(0))) atomicOr(err, (isfinite(n) && isfinite(T)) ? ERR_NEGATIVE : ERR_NONFINITE);
    else if (!isfinite(fx + fy) || !isfinite(nu) || !isfinite(qx + qy) || !isfinite(Ax + Ay))
        atomicOr(err, ERR_NONFINITE);
    // polynomial coefficients of nu F^S + J1_F and nu G^S + J1_G over F_MB
    // (K = b n chi, sq = nu s with s = (1 - Pr)/(n T^2), div u = Dxx + Dyy)
    const R K = xx, sq = nu * (R(1) - Pr) / (n * T * T), dv = Dxx + Dyy, iT = R(1) / T;
    R pf[10], pg[10];
    pf[0] = nu + R(0.8) * K * dv;
    pf[1] = R(-0.8) * sq * qx - K * (Ax - R(1.2) * Bx);
    pf[2] = R(-0.8) * sq * qy - K * (Ay - R(1.2) * By);
    pf[3] = R(-0.4) * K * (Dxx + R(0.5) * dv) * iT;
    pf[4] = R(-0.4) * K * (Dxy + Dyx) * iT;
    pf[5] = R(-0.4) * K * (Dyy + R(0.5) * dv) * iT;
    pf[6] = R(0.2) * sq * qx * iT - R(0.3) * K * Bx * iT;
    pf[7] = R(0.2) * sq * qy * iT - R(0.3) * K * By * iT;
    pf[8] = R(0.2) * sq * qx * iT - R(0.3) * K * Bx * iT;
    pf[9] = R(0.2) * sq * qy * iT - R(0.3) * K * By * iT;
    pg[0] = R(0.5) * nu * T + R(0.2) * T * K * dv;
    pg[1] = R(-0.2) * T * sq * qx - R(0.5) * T * K * (Ax - R(0.6) * Bx);
    pg[2] = R(-0.2) * T * sq * qy - R(0.5) * T * K * (Ay - R(0.6) * By);
    pg[3] = R(-0.2) * K * (Dxx + R(0.5) * dv);
    pg[4] = R(-0.2) * K * (Dxy + Dyx);
    pg[5] = R(-0.2) * K * (Dyy + R(0.5) * dv);
    pg[6] = R(0.1) * sq * qx - R(0.15) * K * Bx;
    pg[7] = R(0.1) * sq * qy - R(0.15) * K * By;
    pg[8] = R(0.1) * sq * qx - R(0.15) * K * Bx;
    pg[9] = R(0.1) * sq * qy - R(0.15) * K * By;
    R* o = fld + i;
    o[F2_N * N] = n;
    o[F2_UX * N] = ux;
    o[F2_UY * N] = uy;
    o[F2_T * N] = T;
    o[F2_NU * N] = nu;
    o[F2_FX * N] = fx;
    o[F2_FY * N] = fy;
#pragma unroll
    for (int j = 0; j < 10; ++j) {
        o[(F2_PF + j) * N] = n * pf[j];
        o[(F2_PG + j) * N] = n * pg[j];
    }
}

// ---------------------------------------------------------------------------
// k2_coll: per group of kNB consecutive nodes, the local (velocity-space)
// part of the right-hand side,
//   RL = -nu h + F_x (D (x) I) h + F_y (I (x) D) h + sum_{a<4} phi^a (x) psi^a.
// D = S diag-shift(sqrt(l)) P is the derivative of the force term on the
// Gauss-Hermite set: the synthesis of its coefficient form F sqrt(l) a_{l-1}
// (S P = I on the set, so the relaxation -nu h needs no transform).  The
// projected Shakhov equilibrium and J1, sum_ab P_ab n mu^a_l(u_x) mu^b_m(u_y)
// in coefficient space (the one-axis Gaussian moments
//   mu^0 = m_l, mu^1 = T sqrt(l) m_{l-1}, mu^2 = T m_l + T^2 sqrt(l(l-1)) m_{l-2},
//   mu^3 = 3T^2 sqrt(l) m_{l-1} + T^3 sqrt(l(l-1)(l-2)) m_{l-3},
// m_l = E[psi_l(u + c)], c ~ N(0, T)), synthesise to the rank-4 sum of
// outer products of phi^a = S mu^a(u_x) and psi^a = sum_b P_ab chi^b,
// chi^b = S mu^b(u_y); a row r of the sum is sum_b pr_b chi^b with
// pr_b = sum_a phi^a_r P_ab.
// The node reflection xi -> -xi maps psi_l to (-1)^l psi_l, so S's rows k and
// Q-1-k differ in the sign of the odd orders, and D anticommutes with it.
// With E_j = h_j + h_{Q-1-j}, O_j = h_j - h_{Q-1-j} (j < Q/2) a line's D h is
//   (D h)_k = (DB E)_k + (DA O)_k,   (D h)_{Q-1-k} = (DA O)_k - (DB E)_k,
// DA_kj = (D_kj - D_{k,Q-1-j})/2, DB_kj = (D_kj + D_{k,Q-1-j})/2: two
// (Q/2)^2 blocks instead of Q^2 products per line, and a synthesis is
// (S c)_k = e_k + o_k, (S c)_{Q-1-k} = e_k - o_k over the even and odd orders.
//
// Work layout: a half-warp owns one line (velocity row, then column) of the
// group's 16 nodes, a lane the (F, G) pairs of its node, and the state sits
// plane-major in shared memory (the 16 nodes of a plane in 128 bytes), so
// shared accesses are conflict-free and global accesses whole lines.  A line
// of Q pairs is loaded, split into E and O and multiplied by DA and DB, whose
// entries are literals of the packed multiply-adds: half the instructions of
// scalar arithmetic, and none to fetch the matrices.
//   pass 1 (rows, D along y):  Y = -nu h + F_y (I (x) D) h + sum_b pr_b chi^b
//   pass 2 (columns, along x): RL = Y + F_x (D (x) I) h, and to global
//   memory the stage's local increment V = alpha (base - h) + cb RL, where the
//   advection adds its part in place (base may be the output itself: every
//   element is read and written by the same thread).
// ---------------------------------------------------------------------------
// The matrices of one Q: DA, DB [(Q/2)^2 each], then S [Q][Q] (S[k][l] = w_k
// psi_l(xi_k)).  FP32: evaluated at compile time, so that their entries are
// literals of the multiply-adds (a line of 16 takes 163 instructions; with
// constant-bank entries 204, in scalar and packed arithmetic alike).  FP64: in the constant bank, at
// coll_coff(Q), from the host's extended precision.
__host__ __device__ constexpr int coll_coff(int Q) {
    int o = 0;
    for (int q = 4; q < Q; q += 2) o += q * q / 2 + q * q;
    return o;
}
constexpr int kCollConst = coll_coff(18);
__constant__ double c_coll_d[kCollConst];

constexpr double ct_sqrt(double x) {
    double r = x > 1.0 ? x : 1.0;
    for (int i = 0; i < 60; ++i) r = 0.5 * (r + x / r);
    return r;
}
template <int Q>
struct CollLit {
    float v[Q * Q / 2 + Q * Q];
    float rec[5 * Q];   // 1/sqrt(l+1), sqrt(l/(l+1)), sqrt(l), sqrt(l(l-1)), sqrt(l(l-1)(l-2))
    constexpr CollLit() : v{}, rec{} {
        // orthonormal Hermite polynomials psi_0 .. psi_Q at x
        struct Psi {
            double p[Q + 1];
            constexpr Psi(double x, const double* r) : p{} {
                p[0] = 1.0;
                p[1] = x;
                for (int l = 1; l < Q; ++l) p[l + 1] = (x * p[l] - r[l] * p[l - 1]) / r[l + 1];
            }
        };
        double r[Q + 1] = {};
        for (int l = 0; l <= Q; ++l) r[l] = l ? ct_sqrt((double)l) : 0.0;
        for (int l = 0; l < Q; ++l) {
            rec[l] = (float)(1.0 / r[l + 1]);
            rec[Q + l] = (float)(r[l] / r[l + 1]);
            rec[2 * Q + l] = (float)r[l];
            rec[3 * Q + l] = l >= 1 ? (float)(r[l] * r[l - 1]) : 0.f;
            rec[4 * Q + l] = l >= 2 ? (float)(r[l] * r[l - 1] * r[l - 2]) : 0.f;
        }
        // the Q/2 positive roots of psi_Q, ascending: sign changes on a grid
        // finer than their spacing, then bisection
        double xi[Q] = {}, w[Q] = {};
        int found = 0;
        double a = 0.0, fa = Psi(0.0, r).p[Q];
        for (int i = 1; found < Q / 2; ++i) {
            const double b = 0.1 * i, fb = Psi(b, r).p[Q];
            if ((fa < 0.0) != (fb < 0.0)) {
                double lo = a, hi = b;
                for (int it = 0; it < 52; ++it) {
                    const double m = 0.5 * (lo + hi);
                    if ((Psi(m, r).p[Q] < 0.0) == (fa < 0.0)) lo = m;
                    else hi = m;
                }
                xi[Q / 2 + found] = 0.5 * (lo + hi);
                xi[Q / 2 - 1 - found] = -0.5 * (lo + hi);
                ++found;
            }
            a = b;
            fa = fb;
        }
        // w_k = 1 / sum_{l<Q} psi_l(xi_k)^2 (Christoffel)
        double ps[Q][Q] = {};
        for (int k = 0; k < Q; ++k) {
            const Psi p(xi[k], r);
            double sum = 0.0;
            for (int l = 0; l < Q; ++l) {
                ps[k][l] = p.p[l];
                sum += p.p[l] * p.p[l];
            }
            w[k] = 1.0 / sum;
        }
        constexpr int QH = Q / 2;
        for (int k = 0; k < QH; ++k)
            for (int j = 0; j < QH; ++j) {
                double d0 = 0.0, d1 = 0.0;
                for (int l = 1; l < Q; ++l) {
                    const double c = w[k] * ps[k][l] * r[l];
                    d0 += c * ps[j][l - 1];
                    d1 += c * ps[Q - 1 - j][l - 1];
                }
                v[k * QH + j] = (float)(0.5 * (d0 - d1));
                v[QH * QH + k * QH + j] = (float)(0.5 * (d0 + d1));
            }
        for (int k = 0; k < Q; ++k)
            for (int l = 0; l < Q; ++l) v[2 * QH * QH + k * Q + l] = (float)(w[k] * ps[k][l]);
    }
};
// entry i of the matrices of order Q (i a constant once the loops are unrolled)
template <typename R, int Q>
__device__ __forceinline__ R ccoll(int i) {
    if constexpr (std::is_same<R, float>::value) {
        static constexpr CollLit<Q> lit{};
        return lit.v[i];
    } else {
        return c_coll_d[coll_coff(Q) + i];
    }
}

template <int Q>
struct Coll2Lay {
    static constexpr int K = Q * Q, QH = Q / 2;
    // in values: state tile [K][kNB] pairs; chi4 [kNB][PS] (chi^b at column k,
    // twice, at k 8 + 2 b: the pair operand of both distributions; PS an odd
    // count of 16-byte units in FP32); phi [4][PH] (phi^a_k of node n at
    // k kNB + n; PH = 8 mod 32); mu [2][Q][kNB][4] (axis, order, node, a);
    // sc [kNumFld2][kNB]; rinv, rr, r1, r2, r3 [Q]
    static constexpr int XN = K * 2 * kNB, PS = 8 * Q + 4, PH = Q * kNB + 8;
    static constexpr int CHI = kNB * PS, PHI = 4 * PH, MU = 2 * Q * kNB * 4, SC = kNumFld2 * kNB;
    static constexpr int ONE = 2 * XN + CHI + PHI + SC + MU + 5 * Q;         // k2_coll
    static constexpr int PIPE = 5 * XN + 2 * (CHI + PHI + SC) + MU;          // k2_coll_pipe: two buffers of
                                                                             // what a group brings with it
};

// two consecutive pairs
__device__ __forceinline__ void ld_pairs(const float* p, float2& a, float2& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = make_float2(v.x, v.y), b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld_pairs(const double* p, double2& a, double2& b) {
    a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}

// D h along one line of Q pairs hv: out[k] = sum_j D_kj hv[j]
template <typename R, int Q>
__device__ __forceinline__ void d_line(const Pair<R> (&hv)[Q], Pair<R> (&out)[Q]) {
    constexpr int QH = Q / 2, O1 = QH * QH;
    Pair<R> E[QH], Od[QH];
#pragma unroll
    for (int j = 0; j < QH; ++j) {
        E[j] = add2(hv[j], hv[Q - 1 - j]);
        Od[j] = sub2(hv[j], hv[Q - 1 - j]);
    }
#pragma unroll
    for (int k = 0; k < QH; ++k) {
        Pair<R> u = mul2(splat(ccoll<R, Q>(k * QH)), Od[0]), v = mul2(splat(ccoll<R, Q>(O1 + k * QH)), E[0]);
#pragma unroll
        for (int j = 1; j < QH; ++j) {
            u = fma2(splat(ccoll<R, Q>(k * QH + j)), Od[j], u);
            v = fma2(splat(ccoll<R, Q>(O1 + k * QH + j)), E[j], v);
        }
        out[k] = add2(v, u);
        out[Q - 1 - k] = sub2(u, v);
    }
}

// S c for one vector of Q orders: out[k] = sum_l S_kl c[l]
template <typename R, int Q>
__device__ __forceinline__ void s_line(const R (&c)[Q], R (&out)[Q]) {
    constexpr int QH = Q / 2, OS = 2 * QH * QH;
#pragma unroll
    for (int k = 0; k < QH; ++k) {
        R e = R(0), o = R(0);
#pragma unroll
        for (int l = 0; l < Q; l += 2) {
            e = fma(ccoll<R, Q>(OS + k * Q + l), c[l], e);
            o = fma(ccoll<R, Q>(OS + k * Q + l + 1), c[l + 1], o);
        }
        out[k] = e + o;
        out[Q - 1 - k] = e - o;
    }
}

// The parts of a group's work, shared by the two kernels below.  sc: the
// group's node fields [kNumFld2][kNB]; lane = 2 n + d.
//
// node fields of nodes i0 .. i0 + nb - 1 (the rest benign), by threads tid, tid + nth, ...
template <typename R>
__device__ __forceinline__ void coll_fields(const R* __restrict__ fld, long long N, long long i0, int nb, R* sc, int tid,
                                            int nth) {
    for (int e = tid; e < kNumFld2 * kNB; e += nth) {
        const int n = e % kNB, f = e / kNB;
        sc[e] = (n < nb) ? fld[f * N + i0 + n] : (f == F2_N || f == F2_T ? R(1) : R(0));
    }
}

// one-axis Gaussian moments mu^a_l, one node and axis per thread (32
// threads); rec (FP64; FP32 has literals): the recurrence constants of CollLit
template <typename R, int Q>
__device__ __forceinline__ void coll_mu(const R* sc, const R* rec, R* mu, int tid) {
    auto c = [&](int which, int l) -> R {
        if constexpr (std::is_same<R, float>::value) {
            static constexpr CollLit<Q> lit{};
            return lit.rec[which * Q + l];
        } else {
            return rec[which * Q + l];
        }
    };
    const int n = tid % kNB, axis = tid / kNB;
    const R u = sc[(axis ? F2_UY : F2_UX) * kNB + n], T = sc[F2_T * kNB + n], Tm1 = T - R(1);
    R* out = mu + (axis * Q * kNB + n) * 4;
    R m1v = 0, m2v = 0, m3v = 0;                            // m_{l-1}, m_{l-2}, m_{l-3}
    R m0 = 1;                                               // m_l
#pragma unroll
    for (int l = 0; l < Q; ++l) {
        R* o = out + l * kNB * 4;
        o[0] = m0;
        o[1] = T * c(2, l) * m1v;
        o[2] = T * m0 + T * T * c(3, l) * m2v;
        o[3] = R(3) * T * T * c(2, l) * m1v + T * T * T * c(4, l) * m3v;
        const R mn = fma(u * c(0, l), m0, Tm1 * c(1, l) * m1v);
        m3v = m2v;
        m2v = m1v;
        m1v = m0;
        m0 = mn;
    }
}

// one-axis syntheses, vector `tid` (axis, node, a) of 128:
// phi^a = S mu^a(u_x) to phi, chi^b = S mu^b(u_y) to chi4
template <typename R, int Q>
__device__ __forceinline__ void coll_synth(const R* mu, R* phi, R* chi4, int tid) {
    using Lay = Coll2Lay<Q>;
    const int a = tid % 4, n = (tid / 4) % kNB, axis = tid / (4 * kNB);
    R c[Q], out[Q];
#pragma unroll
    for (int l = 0; l < Q; ++l) c[l] = mu[((axis * Q + l) * kNB + n) * 4 + a];
    s_line<R, Q>(c, out);
    if (axis == 0) {
#pragma unroll
        for (int k = 0; k < Q; ++k) phi[a * Lay::PH + k * kNB + n] = out[k];
    } else {
#pragma unroll
        for (int k = 0; k < Q; ++k) chi4[n * Lay::PS + k * 8 + 2 * a] = chi4[n * Lay::PS + k * 8 + 2 * a + 1] = out[k];
    }
}

// pass 1 on row r (fixed kx) of node n, D along y: from X to Y
template <typename R, int Q>
__device__ __forceinline__ void coll_row(int r, int n, const Pair<R>* X, Pair<R>* Y, const R* sc, const R* phi,
                                         const R* chi4) {
    using Lay = Coll2Lay<Q>;
    using R2 = Pair<R>;
    const R2* h = X + r * Q * kNB + n;
    R2* y = Y + r * Q * kNB + n;
    R2 hv[Q], dy[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) hv[j] = h[j * kNB];
    d_line<R, Q>(hv, dy);
    const R2 mnu = splat(-sc[F2_NU * kNB + n]), fy = splat(sc[F2_FY * kNB + n]);
    // P_ab (the equilibrium polynomials' coefficients of c_x^a c_y^b, times
    // n) at (a+b)(a+b+1)/2 + b of the order (0,0) (1,0) (0,1) (2,0) (1,1)
    // (0,2) (3,0) (2,1) (1,2) (0,3)
    auto P = [&](int i) {
        R2 p;
        p.x = sc[(F2_PF + i) * kNB + n];
        p.y = sc[(F2_PG + i) * kNB + n];
        return p;
    };
    const R2 p0 = splat(phi[0 * Lay::PH + r * kNB + n]), p1 = splat(phi[1 * Lay::PH + r * kNB + n]);
    const R2 p2 = splat(phi[2 * Lay::PH + r * kNB + n]), p3 = splat(phi[3 * Lay::PH + r * kNB + n]);
    // pr_b = sum_{a <= 3-b} phi^a_r P_ab
    const R2 pr0 = fma2(p3, P(6), fma2(p2, P(3), fma2(p1, P(1), mul2(p0, P(0)))));
    const R2 pr1 = fma2(p2, P(7), fma2(p1, P(4), mul2(p0, P(2))));
    const R2 pr2 = fma2(p1, P(8), mul2(p0, P(5)));
    const R2 pr3 = mul2(p0, P(9));
    const R* ch = chi4 + n * Lay::PS;
#pragma unroll
    for (int c = 0; c < Q; ++c) {
        R2 q0, q1, q2, q3;
        ld_pairs(ch + c * 8, q0, q1);
        ld_pairs(ch + c * 8 + 4, q2, q3);
        R2 eq = mul2(pr0, q0);
        eq = fma2(pr1, q1, eq);
        eq = fma2(pr2, q2, eq);
        eq = fma2(pr3, q3, eq);
        y[c * kNB] = fma2(fy, dy[c], fma2(mnu, hv[c], eq));
    }
}

// pass 2 on column c (fixed ky) of node n, D along x, and the store of V at
// g + k N; bv(k): base at plane k of this node
template <typename R, int Q, typename B>
__device__ __forceinline__ void coll_col(int c, int n, const Pair<R>* X, const Pair<R>* Y, const R* sc, bool wb, R cb,
                                         R al, bool valid, Pair<R>* g, long long N, B bv) {
    using R2 = Pair<R>;
    const R2* h = X + c * kNB + n;
    const R2* y = Y + c * kNB + n;
    R2 hv[Q], dx[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) hv[j] = h[j * Q * kNB];
    d_line<R, Q>(hv, dx);
    const R2 fx = splat(sc[F2_FX * kNB + n]), cb2 = splat(cb), al2 = splat(al);
    R2* p = g + (long long)c * N;
#pragma unroll
    for (int r = 0; r < Q; ++r, p += Q * N) {
        R2 v = mul2(cb2, fma2(fx, dx[r], y[r * Q * kNB]));
        if (wb) v = fma2(al2, sub2(bv(r * Q + c), hv[r]), v);
        if (valid) *p = v;
    }
}

// the group's slice of a state, [K][kNB] pairs, by asynchronous copies: 16
// bytes where they stay aligned in every plane, else one pair at a time
template <typename R, int Q>
__device__ __forceinline__ void coll_issue(Pair<R>* dst, const Pair<R>* st, long long N, long long i0, int nb, int tid,
                                           int nth) {
    constexpr int K = Q * Q, CH = 16 / (int)sizeof(Pair<R>), CPP = kNB / CH;   // pairs per copy, copies per plane
    if (CH == 1 || (N & 1) == 0) {                                             // (FP32: nb is even here)
        const int n = (tid % CPP) * CH;                                        // nth is a multiple of CPP
        const Pair<R>* g = st + i0 + n;
        if (n < nb)
            for (int k = tid / CPP; k < K; k += nth / CPP) cp_async16(dst + k * kNB + n, g + (long long)k * N);
    } else {
        const int n = tid % kNB;
        const Pair<R>* g = st + i0 + n;
        if (n < nb)
            for (int k = tid / kNB; k < K; k += nth / kNB)
                cp_async_elem<double>(reinterpret_cast<double*>(dst + k * kNB + n),
                                      reinterpret_cast<const double*>(g + (long long)k * N));
    }
    cp_async_commit();
}

template <typename R, int Q>
__device__ __forceinline__ void coll_tables(const R* __restrict__ rtab, R* rec, int tid, int nth) {
    TableLayout L(Q);
    for (int e = tid; e < Q; e += nth) {
        rec[e] = rtab[L.rinv + e];
        rec[Q + e] = rtab[L.rr + e];
        rec[2 * Q + e] = rtab[L.r1 + e];
        rec[3 * Q + e] = rtab[L.r2 + e];
        rec[4 * Q + e] = rtab[L.r3 + e];
    }
}

// One group per CTA, its phases in sequence: the FP64 build (whose two state
// buffers and prefetches would not fit).
template <typename R, int Q>
__global__ void __launch_bounds__(256, 1)
k2_coll(Slab2 s, const Par2<R> pr, const R* __restrict__ rtab, const Pair<R>* __restrict__ st,
        const R* __restrict__ fld, const Pair<R>* base, Pair<R>* V) {
    using Lay = Coll2Lay<Q>;
    constexpr int NT = 256;
    extern __shared__ __align__(16) double smc[];
    R* chi4 = reinterpret_cast<R*>(smc) + 2 * Lay::XN;
    Pair<R>* X = reinterpret_cast<Pair<R>*>(smc);
    Pair<R>* Y = X + Lay::XN / 2;
    R* phi = chi4 + Lay::CHI;
    R* sc = phi + Lay::PHI;
    R* mu = sc + Lay::SC;
    R* rec = mu + Lay::MU;
    const long long N = s.N, i0 = (long long)blockIdx.x * kNB;
    const int nb = (int)min((long long)kNB, N - i0), tid = threadIdx.x;
    coll_issue<R, Q>(X, st, N, i0, nb, tid, NT);
    coll_tables<R, Q>(rtab, rec, tid, NT);
    coll_fields<R>(fld, N, i0, nb, sc, tid, NT);
    __syncthreads();
    if (tid < 2 * kNB) coll_mu<R, Q>(sc, rec, mu, tid);
    __syncthreads();
    if (tid < 2 * kNB * 4) coll_synth<R, Q>(mu, phi, chi4, tid);
    cp_async_wait_all();
    __syncthreads();
    const int n = tid % kNB, line = tid / kNB;          // a half-warp per row (column)
    if (line < Q) coll_row<R, Q>(line, n, X, Y, sc, phi, chi4);
    __syncthreads();
    const bool valid = n < nb;
    const Pair<R>* bp = base + i0 + n;
    if (line < Q)
        coll_col<R, Q>(line, n, X, Y, sc, pr.with_base != 0, pr.cb, pr.alpha, valid, V + i0 + n, N,
                       [&](int k) { return valid ? bp[(long long)k * N] : splat(R(0)); });
}

// The FP32 form: a resident CTA walks the groups blockIdx.x, + gridDim.x, ...
// with everything of the next group in preparation while it forms this one:
//  - its state and base slices (32 KB each at Q = 16) by asynchronous copies
//    issued a whole group ahead;
//  - its node fields, Gaussian moments and one-axis syntheses by four extra
//    warps (the serial recurrence of coll_mu would idle a CTA that formed it
//    in sequence; with the field loads in that sequence too the preparation
//    was the longer side: 296 us).
// Q/2 warps take two velocity rows, then two columns, of each group, F and G
// in packed arithmetic.
// Bound by DRAM: 172 us at 384^2, Q 16, 5.3 TB/s with the base (24 bytes per
// pair).  Two CTAs per SM that ran load, moments and passes in sequence, in
// scalar arithmetic on constant-bank matrices, took 210 us without the base
// (and 400 us with it read where it is used).
constexpr int kCollPrep = 128;               // threads of the preparing warps
template <int Q>
constexpr int coll_threads() { return kNB * Q + kCollPrep; }
template <int Q>
__global__ void __launch_bounds__(coll_threads<Q>(), 1)
k2_coll_pipe(Slab2 s, const Par2<float> pr, const float2* __restrict__ st, const float* __restrict__ fld,
             const float2* base, float2* V, int groups) {
    using Lay = Coll2Lay<Q>;
    constexpr int NC = kNB * Q, XP = Lay::XN / 2;          // computing threads, pairs of a slice
    extern __shared__ __align__(16) double smc[];
    float2* X = reinterpret_cast<float2*>(smc);            // [2][XP]
    float2* B = X + 2 * XP;                                // [2][XP]
    float2* Y = B + 2 * XP;
    float* chi4 = reinterpret_cast<float*>(Y + XP);        // [2][CHI]
    float* phi = chi4 + 2 * Lay::CHI;                      // [2][PHI]
    float* sc = phi + 2 * Lay::PHI;                        // [2][SC]
    float* mu = sc + 2 * Lay::SC;
    const long long N = s.N;
    const int tid = threadIdx.x;
    const bool wb = pr.with_base != 0;
    auto nodes_of = [&](int g) { return (int)min((long long)kNB, N - (long long)g * kNB); };
    if (tid < NC) {
        auto issue = [&](int g, int b) {
            const long long i0 = (long long)g * kNB;
            coll_issue<float, Q>(X + b * XP, st, N, i0, nodes_of(g), tid, NC);
            if (wb) coll_issue<float, Q>(B + b * XP, base, N, i0, nodes_of(g), tid, NC);
        };
        issue(blockIdx.x, 0);
        const int n = tid % kNB, line = tid / kNB;
        for (int g = blockIdx.x, b = 0; g < groups; g += gridDim.x, b ^= 1) {
            cp_async_wait_all();
            __syncthreads();                 // group g staged and prepared, group g - 1 done
            if (g + (int)gridDim.x < groups) issue(g + gridDim.x, b ^ 1);
            const float2* x = X + b * XP;
            const float* scb = sc + b * Lay::SC;
            coll_row<float, Q>(line, n, x, Y, scb, phi + b * Lay::PHI, chi4 + b * Lay::CHI);
            asm volatile("bar.sync 1, %0;" ::"n"(NC) : "memory");
            const float2* bb = B + b * XP + n;
            coll_col<float, Q>(line, n, x, Y, scb, wb, pr.cb, pr.alpha, n < nodes_of(g), V + (long long)g * kNB + n, N,
                               [&](int k) { return bb[k * kNB]; });
        }
    } else {
        // the fields of the group after the next are in flight meanwhile
        constexpr int NV = (Lay::SC + kCollPrep - 1) / kCollPrep;
        const int t = tid - NC, n = t % kNB;
        const int step = gridDim.x;
        float v[NV];
        auto load = [&](int g) {
            const bool in = g < groups && n < nodes_of(g);
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                const int f = (t + kCollPrep * j) / kNB;
                v[j] = (f < kNumFld2 && in) ? fld[f * N + (long long)g * kNB + n]
                                            : (f == F2_N || f == F2_T ? 1.f : 0.f);
            }
        };
        auto sync = [] { asm volatile("bar.sync 2, %0;" ::"n"(kCollPrep) : "memory"); };
        auto prepare = [&](int g, int b) {                   // v: the fields of group g
            float* scb = sc + b * Lay::SC;
#pragma unroll
            for (int j = 0; j < NV; ++j)
                if (t + kCollPrep * j < Lay::SC) scb[t + kCollPrep * j] = v[j];
            load(g + step);
            sync();
            if (t < 2 * kNB) coll_mu<float, Q>(scb, nullptr, mu, t);
            sync();
            coll_synth<float, Q>(mu, phi + b * Lay::PHI, chi4 + b * Lay::CHI, t);
        };
        load(blockIdx.x);
        prepare(blockIdx.x, 0);
        for (int g = blockIdx.x, b = 0; g < groups; g += step, b ^= 1) {
            __syncthreads();
            if (g + step < groups) prepare(g + step, b ^ 1);
        }
    }
}

// ---------------------------------------------------------------------------
// k2_adv: WENO-5 faces along x and y and the end of the RK stage,
//   V <- hs h + (V + ca (xi_x df_x + xi_y df_y)),
// hs = 1 for a stage (V the increment that k2_coll left, here completed in
// place), 0 for a right-hand side.
// F and G of one velocity are carried together as a pair (packed FP32
// arithmetic, two lanes per instruction): both share the velocity, hence the
// upwind direction of every face, so the pair runs one stencil walk.
//
// A CTA of four warps owns a 32x32 node tile and a run of velocities.  Per
// velocity the halo tile (38x38 pairs) sits in shared memory; the halos of
// the next two velocities are in flight (cp.async, three buffers).  Each
// thread walks two runs of nine faces and keeps the face differences in
// registers:
//   x: lane = row, warp = 8 columns; the 8 differences go to shared memory;
//   y: lane = column, warp = 8 rows; per face after the first the thread holds
//      h and df_y of one node, adds the node's df_x and V and writes it.
// So a node costs one shared store and two shared loads besides the two
// stencil loads, two CTA barriers per velocity serve 1024 nodes, and V comes
// by plain row loads issued before the x walk.  Any nx and ny take this path
// (copies of single pairs from offsets formed once per CTA).  The odd row
// pitches keep the accesses of both walks conflict-free.
// Bound by the FMA pipe (a packed operation holds it two cycles): at 384^2, Q
// 16, 212 us with the pipe 74 % busy and 4.2 TB/s of DRAM, 110 instructions
// per node and velocity.  The form before (32x16 tiles, runs of four or five
// faces, face values in shared memory, separate F and G planes, 16-byte copies
// on aligned tiles alone) took 345 us and 241 instructions, and 376 us against
// now 128 us on a 333x250 grid, whose rows are not 16-byte aligned.
// ---------------------------------------------------------------------------
// The WENO-5 walk of Weno5Run on pairs.  With g_0 = 5 d_1 - 2 d_0,
// g_1 = 6 (s_1 + d_2), g_2 = 3 (d_2 - s_2) (60 times the candidate
// corrections times their linear weights) the face is
// v2 + (sum a_r g_r) / (6 (a_0 + 6 a_1 + 3 a_2)).  The sum is formed of g_r / 64,
// in as many operations, so that in FP32 it does not overflow before that of the
// weighted corrections would (noise of 4000 in F; without it from 2800 on).  The divisor is at least
// 10 (4 eps)^4: a normal FP32 number for eps >= kFtzMinEps, where FTZ takes
// the flushing reciprocal; below, the quotient that also covers subnormals.
constexpr double kFtzMinEps = 1e-9;
template <typename R, bool FTZ>
struct Weno5Run2 {
    using R2 = Pair<R>;
    R2 v2, v3, v4, d0, d1, d2, d3, u0, u1, u2, eps4;
    __device__ __forceinline__ R2 tterm(R2 t) const { return fma2(mul2(splat(R(13.0 / 3.0)), t), t, eps4); }
    __device__ __forceinline__ void start(R2 w0, R2 w1, R2 w2, R2 w3, R2 w4, R eps) {
        eps4 = splat(R(4) * eps);
        v2 = w2;
        v3 = w3;
        v4 = w4;
        d0 = sub2(w1, w0);
        d1 = sub2(w2, w1);
        d2 = sub2(w3, w2);
        d3 = sub2(w4, w3);
        u0 = tterm(sub2(d1, d0));
        u1 = tterm(sub2(d2, d1));
        u2 = tterm(sub2(d3, d2));
    }
    __device__ __forceinline__ R2 quotient(R2 a, R2 b) const {
        if constexpr (std::is_same<R, double>::value) return make_double2(div_face(a.x, b.x), div_face(a.y, b.y));
        else if constexpr (FTZ) return mul2(a, make_float2(rcp_ftz(b.x), rcp_ftz(b.y)));
        else return make_float2(__fdividef(a.x, b.x), __fdividef(a.y, b.y));
    }
    __device__ __forceinline__ R2 face() const {
        // s_0 and the g_r with their signs turned (no negations), the g_r over 64
        const R2 s0 = fma2(splat(R(-3)), d1, d0), s1 = add2(d1, d2), s2 = fma2(splat(R(-3)), d2, d3);
        const R2 e0 = fma2(s0, s0, u0), e1 = fma2(s1, s1, u1), e2 = fma2(s2, s2, u2);
        const R2 E0 = mul2(e0, e0), E1 = mul2(e1, e1), E2 = mul2(e2, e2);
        const R2 a0 = mul2(E1, E2), a1 = mul2(E0, E2), a2 = mul2(E0, E1);
        const R2 y = mul2(splat(R(-12.0 / 64.0)), d2);
        const R2 g0 = fma2(splat(R(2.0 / 64.0)), d0, mul2(splat(R(-5.0 / 64.0)), d1));
        const R2 g1 = fma2(splat(R(-6.0 / 64.0)), d1, y);
        const R2 g2 = fma2(splat(R(3.0 / 64.0)), d3, y);
        const R2 num = fma2(a0, g0, fma2(a1, g1, mul2(a2, g2)));
        const R2 den = fma2(splat(R(6)), a1, fma2(splat(R(3)), a2, a0));
        return fma2(splat(R(-64.0 / 6.0)), quotient(num, den), v2);
    }
    __device__ __forceinline__ void shift(R2 w5) {
        const R2 d4 = sub2(w5, v4);
        u0 = u1;
        u1 = u2;
        u2 = tterm(sub2(d4, d3));
        d0 = d1;
        d1 = d2;
        d2 = d3;
        d3 = d4;
        v2 = v3;
        v3 = v4;
        v4 = w5;
    }
};

constexpr int kPT = 32;                      // tile edge
constexpr int kPW = kPT + 6;                 // halo edge
constexpr int kPP = kPW + 1, kPD = kPT + 1;  // row pitches of the halo and of df_x
constexpr int kPThreads = 128, kPRun = 8;    // nodes per walk
constexpr int kPBufs = 3;
// CTAs per SM.  FP32: four, with 124 registers a thread (212 us at 384^2, Q 16;
// five with 96 serialise each walk: 261 us; three: 215 us).
template <typename R>
constexpr int adv_ctas() { return std::is_same<R, float>::value ? 4 : 2; }
template <typename R>
constexpr size_t adv_smem() { return sizeof(Pair<R>) * (kPBufs * kPW * kPP + kPT * kPD) + sizeof(int) * 2 * kPW; }
static_assert(kPThreads / 32 * kPRun == kPT, "a warp per 8 rows or columns of the tile");

__device__ __forceinline__ void cp_async_wait_1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

template <typename R, int Q, bool FTZ>
__global__ void __launch_bounds__(kPThreads, adv_ctas<R>())
k2_adv(Slab2 s, const Par2<R> pr, const R* __restrict__ rtab, const Pair<R>* __restrict__ src, Pair<R>* V, int planes) {
    using R2 = Pair<R>;
    constexpr int K = Q * Q, NW = kPThreads / 32;
    constexpr int NR = (kPW + NW - 1) / NW;                          // halo rows per warp
    constexpr int NE = (6 * kPW + kPThreads - 1) / kPThreads;        // right-edge elements per thread
    extern __shared__ __align__(16) double sma[];
    R2* const H0 = reinterpret_cast<R2*>(sma);
    R2* const DX = H0 + kPBufs * kPW * kPP;
    int* const rowoff = reinterpret_cast<int*>(DX + kPT * kPD);
    int* const coloff = rowoff + kPW;
    const int nx = s.nx, ny = s.ny;
    const long long N = s.N;
    const int tilesx = (nx + kPT - 1) / kPT;
    const int x0 = (blockIdx.x % tilesx) * kPT, y0 = (blockIdx.x / tilesx) * kPT;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    TableLayout L(Q);
    if (tid < kPW) rowoff[tid] = wrapi(y0 - 3 + tid, ny) * nx;
    else if (tid >= 64 && tid < 64 + kPW) coloff[tid - 64] = wrapi(x0 - 3 + tid - 64, nx);
    __syncthreads();
    // this thread's halo elements, the same for every velocity: the columns
    // 0 .. 31 of rows warp, warp + 4, ... and its share of the columns 32 .. 37
    unsigned go[NR], ge[NE];
    int se[NE];
#pragma unroll
    for (int j = 0; j < NR; ++j) go[j] = (unsigned)(rowoff[min(warp + NW * j, kPW - 1)] + coloff[lane]);
#pragma unroll
    for (int j = 0; j < NE; ++j) {
        const int e = tid + kPThreads * j;
        const int r = min(e / 6, kPW - 1), c = kPT + e % 6;
        ge[j] = (unsigned)(rowoff[r] + coloff[c]);
        se[j] = e < 6 * kPW ? r * kPP + c : -1;
    }
    auto copy = [](R2* dst, const R2* g) {
        if constexpr (sizeof(R2) == 16) cp_async16(dst, g);
        else cp_async_elem<double>(reinterpret_cast<double*>(dst), reinterpret_cast<const double*>(g));
    };
    auto issue = [&](int k, int b) {
        const R2* p = src + (long long)k * N;
        R2* H = H0 + b * kPW * kPP;
        R2* hr = H + warp * kPP + lane;
#pragma unroll
        for (int j = 0; j < NR; ++j)
            if (warp + NW * j < kPW) copy(hr + NW * j * kPP, p + go[j]);
#pragma unroll
        for (int j = 0; j < NE; ++j)
            if (se[j] >= 0) copy(H + se[j], p + ge[j]);
    };
    const R eps = pr.weno_eps;
    const R2 hscale = splat(pr.hs);
    const int k0 = blockIdx.y * planes, k1 = min(k0 + planes, K);
    issue(k0, 0);
    cp_async_commit();
    if (k0 + 1 < k1) issue(k0 + 1, 1);
    cp_async_commit();
    const int x = x0 + lane, yw = y0 + warp * kPRun;
    const int rows = x < nx ? min(kPRun, ny - yw) : 0;               // nodes of this thread's y walk (may be <= 0)
    const unsigned o0 = (unsigned)yw * (unsigned)nx + (unsigned)x;
    for (int k = k0, b = 0; k < k1; ++k, b = b == kPBufs - 1 ? 0 : b + 1) {
        const R vx = rtab[L.xi + k / Q], vy = rtab[L.xi + k % Q];
        const bool px = vx >= R(0), py = vy >= R(0);
        // V of this thread's nodes, in the order of its y walk (up for
        // xi_y >= 0, else down)
        R2* const p = V + (long long)k * N;
        R2 vv[kPRun];
#pragma unroll
        for (int q = 0; q < kPRun; ++q) {
            const int r = py ? q : kPRun - 1 - q;
            vv[q] = r < rows ? p[o0 + (unsigned)(r * nx)] : splat(R(0));
        }
        cp_async_wait_1();                                           // velocity k's halo
        __syncthreads();
        const R2* H = H0 + b * kPW * kPP;
        Weno5Run2<R, FTZ> w;
        // both walks: face f lies below node f; xi >= 0 takes halo cells f ..
        // f+4 and walks up, xi < 0 takes f+5 .. f+1 and walks down, so that a
        // new face minus the one before is df for xi >= 0 and -df for xi < 0
        // and |xi| carries the sign; after a face the walk's v2 is the node
        // between the two
        {
            const int st = px ? 1 : -1;
            const R2* h = H + (lane + 3) * kPP + warp * kPRun + (px ? 0 : kPRun + 5);
            w.start(h[0], h[st], h[2 * st], h[3 * st], h[4 * st], eps);
            R2 f = w.face();
            R2* dx = DX + lane * kPD + warp * kPRun + (px ? 0 : kPRun - 1);
#pragma unroll
            for (int q = 0; q < kPRun; ++q) {
                w.shift(h[(q + 5) * st]);
                const R2 g = w.face();
                dx[q * st] = sub2(g, f);
                f = g;
            }
        }
        __syncthreads();                                             // df_x written, the buffer of k - 1 consumed
        if (k + 2 < k1) issue(k + 2, b == 0 ? kPBufs - 1 : b - 1);
        cp_async_commit();
        {
            const int dir = py ? 1 : -1, st = dir * kPP;
            const R2* h = H + (warp * kPRun + (py ? 0 : kPRun + 5)) * kPP + lane + 3;
            const R2* dx = DX + (warp * kPRun + (py ? 0 : kPRun - 1)) * kPD + lane;
            const R2 cx = splat(pr.ca * (px ? vx : -vx)), cy = splat(pr.ca * (py ? vy : -vy));
            w.start(h[0], h[st], h[2 * st], h[3 * st], h[4 * st], eps);
            R2 f = w.face();
#pragma unroll
            for (int q = 0; q < kPRun; ++q) {
                w.shift(h[(q + 5) * st]);
                const R2 g = w.face();
                const R2 inc = fma2(cy, sub2(g, f), fma2(cx, dx[q * dir * kPD], vv[q]));
                const int r = py ? q : kPRun - 1 - q;
                if (r < rows) p[o0 + (unsigned)(r * nx)] = fma2(hscale, w.v2, inc);
                f = g;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Initial state, node moments and totals.
// ---------------------------------------------------------------------------
// Projected Maxwellian pair: F_{kx,ky} = n phi_kx(ux) phi_ky(uy) with
// phi_k(u) = sum_l S_kl m_l(u, T) (the 2D Gaussian factorises), G = T/2 F.
template <typename R>
__global__ void k2_init(Slab2 s, const double* __restrict__ tab, const double* __restrict__ n0,
                        const double* __restrict__ u0, const double* __restrict__ T0, Pair<R>* st, unsigned* err) {
    const int Q = s.Q;
    const long long N = s.N;
    TableLayout L(Q);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        double n = n0[i], ux = u0[i], uy = u0[N + i], T = T0[i];
        if (!(n > 0.0) || !(T > 0.0) || !isfinite(ux) || !isfinite(uy))
            atomicOr(err, (isfinite(n) && isfinite(T) && isfinite(ux) && isfinite(uy)) ? ERR_NEGATIVE : ERR_NONFINITE);
        double px[16], py[16];
        for (int axis = 0; axis < 2; ++axis) {
            double u = axis ? uy : ux, m0 = 1.0, m1 = 0.0, ml[16];
            for (int l = 0; l < Q; ++l) {
                ml[l] = m0;
                double mn = fma(u * tab[L.rinv + l], m0, (T - 1.0) * tab[L.rr + l] * m1);
                m1 = m0;
                m0 = mn;
            }
            for (int k = 0; k < Q; ++k) {
                double acc = 0.0;
                for (int l = 0; l < Q; ++l) acc = fma(tab[L.S + k * Q + l], ml[l], acc);
                (axis ? py : px)[k] = acc;
            }
        }
        for (int kx = 0; kx < Q; ++kx)
            for (int ky = 0; ky < Q; ++ky) {
                double f = n * px[kx] * py[ky];
                Pair<R> h;
                h.x = (R)f;
                h.y = (R)(0.5 * T * f);
                st[(long long)(kx * Q + ky) * N + i] = h;
            }
    }
}

__global__ void k2_prims(Slab2 s, const double* __restrict__ mom, double* n, double* u, double* T, double* q) {
    const long long N = s.N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        double nn, ux, uy, TT;
        prim2(mom, N, i, nn, ux, uy, TT);
        if (n) n[i] = nn;
        if (u) {
            u[i] = ux;
            u[N + i] = uy;
        }
        if (T) T[i] = TT;
        if (q) {
            const double S0 = mom[M2_S0 * N + i], S1x = mom[M2_S1X * N + i], S1y = mom[M2_S1Y * N + i];
            const double S2xx = mom[M2_S2XX * N + i], S2yy = mom[M2_S2YY * N + i], S2xy = mom[M2_S2XY * N + i];
            const double u2 = ux * ux + uy * uy, S2 = S2xx + S2yy, uS1 = ux * S1x + uy * S1y;
            q[i] = 0.5 * (mom[M2_S3X * N + i] - 2.0 * (ux * S2xx + uy * S2xy) + u2 * S1x - ux * S2 + 2.0 * ux * uS1 -
                          ux * u2 * S0) + mom[M2_G1X * N + i] - ux * mom[M2_G0 * N + i];
            q[N + i] = 0.5 * (mom[M2_S3Y * N + i] - 2.0 * (ux * S2xy + uy * S2yy) + u2 * S1y - uy * S2 + 2.0 * uy * uS1 -
                              uy * u2 * S0) + mom[M2_G1Y * N + i] - uy * mom[M2_G0 * N + i];
        }
    }
}

// {mass, momentum x, momentum y, kinetic + internal energy} x dx^2; one CTA,
// fixed-order tree (deterministic)
__global__ void __launch_bounds__(256) k2_totals(Slab2 s, const double* __restrict__ mom, double* out) {
    __shared__ double red[4][256];
    const long long N = s.N;
    double a[4] = {0, 0, 0, 0};
    for (long long i = threadIdx.x; i < N; i += blockDim.x) {
        a[0] += mom[M2_S0 * N + i];
        a[1] += mom[M2_S1X * N + i];
        a[2] += mom[M2_S1Y * N + i];
        a[3] += 0.5 * (mom[M2_S2XX * N + i] + mom[M2_S2YY * N + i]) + mom[M2_G0 * N + i];
    }
    for (int c = 0; c < 4; ++c) red[c][threadIdx.x] = a[c];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < 4; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 4) out[threadIdx.x] = red[threadIdx.x][0] * s.dx * s.dx;
}

// The interleaved state to or from two FP64 arrays of n = Q^2 N values each.
template <typename R>
__global__ void k2_split(const Pair<R>* __restrict__ in, double* __restrict__ F, double* __restrict__ G, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const Pair<R> h = in[i];
        F[i] = (double)h.x;
        G[i] = (double)h.y;
    }
}
template <typename R>
__global__ void k2_join(const double* __restrict__ F, const double* __restrict__ G, Pair<R>* __restrict__ out, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        Pair<R> h;
        h.x = (R)F[i];
        h.y = (R)G[i];
        out[i] = h;
    }
}

// ---------------------------------------------------------------------------
// Host side: the 2D context.
// ---------------------------------------------------------------------------
namespace {
const long double kPiL2 = 3.141592653589793238462643383279502884L;

// Gauss-Legendre nodes and weights of order n on [-1, 1] in long double
// (Newton on the Legendre recurrence).
void gauss_legendre_ld(int n, std::vector<long double>& x, std::vector<long double>& w) {
    x.resize(n);
    w.resize(n);
    for (int i = 0; i < n; ++i) {
        long double z = cosl(kPiL2 * (i + 0.75L) / (n + 0.5L)), pp = 0;
        for (int it = 0; it < 100; ++it) {
            long double p1 = 1, p2 = 0;
            for (int j = 1; j <= n; ++j) {
                long double p3 = p2;
                p2 = p1;
                p1 = ((2.0L * j - 1.0L) * z * p2 - (j - 1.0L) * p3) / j;
            }
            pp = n * (z * p1 - p2) / (z * z - 1.0L);
            long double dz = p1 / pp;
            z -= dz;
            if (fabsl(dz) < 1e-19L) break;
        }
        x[i] = z;
        w[i] = 2.0L / ((1.0L - z * z) * pp * pp);
    }
}

// g2 at offset (rx, ry) (components), Eq. (force) integrated over z with
// r = sqrt(rho^2 + z^2) > sigma, gamma = 2(s - 1) even:
//   rho >= sigma: Wallis, int (rho^2 + z^2)^-s dz = rho^(1-2s) pi (2s-3)!!/(2s-2)!!;
//   rho <  sigma: with z = rho cot(psi), 2 rho^(1-2s) int_0^{psi0} sin^(2s-2) psi d psi,
//                 psi0 = atan(rho / z0), by 48-point Gauss-Legendre in long double.
void g2_kernel(const evfdlb_params& p, long double rx, long double ry, long double* gx, long double* gy) {
    long double r = sqrtl(rx * rx + ry * ry), sg = p.sigma;
    *gx = *gy = 0;
    if (r == 0) return;
    int s = (int)llround((p.gamma + 2.0) / 2.0);
    long double J;
    if (r >= sg) {
        long double wallis = kPiL2;
        for (int k = 1; k <= s - 1; ++k) wallis *= (2.0L * k - 1.0L) / (2.0L * k);
        J = wallis * powl(r, 1.0L - 2.0L * s);
    } else {
        static std::vector<long double> gxs, gws;
        if (gxs.empty()) gauss_legendre_ld(48, gxs, gws);
        long double z0 = sqrtl(sg * sg - r * r), psi0 = atanl(r / z0), acc = 0;
        for (int i = 0; i < 48; ++i) {
            long double ps = 0.5L * psi0 * (gxs[i] + 1.0L);
            acc += gws[i] * powl(sinl(ps), 2 * s - 2);
        }
        J = 2.0L * powl(r, 1.0L - 2.0L * s) * 0.5L * psi0 * acc;
    }
    long double c = (long double)p.gamma * p.phi_a * powl(sg, (long double)p.gamma) * J;
    *gx = c * rx;
    *gy = c * ry;
}

struct Taps2 {
    std::vector<int> foff, moff;
    std::vector<double> fg, mw;
    int Mf = 0, mfm = 0;
};

Taps2 taps_2d(const evfdlb_params& p) {
    Taps2 t;
    const double dx = p.dx, rc = p.r_cut, sg = p.sigma;
    t.Mf = (int)floor(rc / dx + 1e-9);
    for (int a = -t.Mf; a <= t.Mf; ++a)
        for (int b = -t.Mf; b <= t.Mf; ++b) {
            double rx = a * dx, ry = b * dx;
            if (rx * rx + ry * ry > rc * rc * (1.0 + 1e-12) || (a == 0 && b == 0)) continue;
            long double gx, gy;
            g2_kernel(p, rx, ry, &gx, &gy);
            t.foff.push_back(a);
            t.foff.push_back(b);
            t.fg.push_back((double)(dx * dx * gx));
            t.fg.push_back((double)(dx * dx * gy));
        }
    t.mfm = (int)ceil(sg / dx);
    long double wsum = 0;
    std::vector<long double> w;
    for (int a = -t.mfm; a <= t.mfm; ++a)
        for (int b = -t.mfm; b <= t.mfm; ++b) {
            long double r2 = (long double)(a * a + b * b) * dx * dx;
            if (r2 >= (long double)sg * sg) continue;
            long double v = 2.0L * sqrtl((long double)sg * sg - r2);
            t.moff.push_back(a);
            t.moff.push_back(b);
            w.push_back(v);
            wsum += v;
        }
    for (long double v : w) t.mw.push_back((double)(v / wsum));
    return t;
}

// Force plan of k2_fields: the disc's offset columns a = 0 .. Mf, each as a
// run of `steps` weight pairs (a multiple of 8: offsets b = -w .. w, then
// zeros), column 0 with halved g2y (its pass adds n(x) twice); the columns
// are dealt to the warps longest first, each to the least loaded warp
// (deterministic).  Layout of `plan`: warps + 1 prefix offsets (padded to
// kFPlanHead ints), then per entry {a, weight offset, steps, w}.
struct ForcePlan {
    std::vector<int> plan;
    std::vector<double> w;     // (g2x, g2y) pairs
    bool ok = true;
};

ForcePlan force_plan(const Taps2& t, int warps) {
    ForcePlan fp;
    const int Mf = t.Mf, D = 2 * Mf + 1;
    std::vector<double> gx((size_t)D * D, 0.0), gy((size_t)D * D, 0.0);
    std::vector<char> in((size_t)D * D, 0);
    for (size_t j = 0; j < t.fg.size() / 2; ++j) {
        const size_t k = (size_t)(t.foff[2 * j] + Mf) * D + (t.foff[2 * j + 1] + Mf);
        gx[k] = t.fg[2 * j];
        gy[k] = t.fg[2 * j + 1];
        in[k] = 1;
    }
    auto at = [&](int a, int b) { return (size_t)(a + Mf) * D + (b + Mf); };
    struct Col { int a, w, steps, off; };
    std::vector<Col> cols;
    for (int a = 0; a <= Mf; ++a) {
        int w = -1;
        for (int b = -Mf; b <= Mf; ++b)
            if (in[at(a, b)] || in[at(-a, b)]) w = std::max(w, std::abs(b));
        if (w < 0) continue;
        for (int b = -w; b <= w; ++b)   // the pairing needs the disc's mirror symmetry, exactly
            if (in[at(a, b)] != in[at(-a, b)] || gx[at(a, b)] != -gx[at(-a, b)] || gy[at(a, b)] != gy[at(-a, b)])
                fp.ok = false;
        const int steps = (2 * w + 8 + 7) & ~7;
        cols.push_back({a, w, steps, (int)(fp.w.size() / 2)});
        for (int j = 0; j < steps; ++j) {
            const int b = j - w;
            double x = 0.0, y = 0.0;
            if (b <= w) {
                x = (a == 0) ? 0.0 : gx[at(a, b)];
                y = (a == 0) ? 0.5 * gy[at(a, b)] : gy[at(a, b)];
            }
            fp.w.push_back(x);
            fp.w.push_back(y);
        }
    }
    std::vector<int> order(cols.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int p, int q) { return cols[p].steps > cols[q].steps; });
    std::vector<std::vector<int>> bins(warps);
    std::vector<long long> load(warps, 0);
    for (int ci : order) {
        int best = 0;
        for (int k = 1; k < warps; ++k)
            if (load[k] < load[best]) best = k;
        bins[best].push_back(ci);
        load[best] += cols[ci].steps;
    }
    fp.plan.assign(kFPlanHead, 0);
    int n = 0;
    for (int k = 0; k < warps; ++k) {
        fp.plan[k] = n;
        n += (int)bins[k].size();
    }
    fp.plan[warps] = n;
    for (int k = 0; k < warps; ++k)
        for (int ci : bins[k]) {
            const Col& c = cols[ci];
            fp.plan.insert(fp.plan.end(), {c.a, c.off, c.steps, c.w});
        }
    return fp;
}

// Parity blocks of the force term's derivative on the velocity set,
// D_kj = sum_{l=1}^{Q-1} w_k psi_l(xi_k) sqrt(l) psi_{l-1}(xi_j) (D = S shift P,
// the synthesis of the coefficient form F sqrt(l) a_{l-1}), in long double:
// DA_kj = (D_kj - D_{k,Q-1-j}) / 2 and DB_kj = (D_kj + D_{k,Q-1-j}) / 2 for
// k, j < Q/2, as [QH][QH] each (DA then DB).
std::vector<double> d_blocks(int Q, const double* xi, const double* w) {
    const int QH = Q / 2;
    std::vector<long double> ps((size_t)Q * (Q + 1));
    for (int k = 0; k < Q; ++k) {
        long double* p = ps.data() + (size_t)k * (Q + 1);
        const long double x = xi[k];
        p[0] = 1;
        p[1] = x;
        for (int l = 1; l < Q; ++l) p[l + 1] = (x * p[l] - sqrtl((long double)l) * p[l - 1]) / sqrtl((long double)(l + 1));
    }
    auto D = [&](int k, int j) {
        long double acc = 0;
        for (int l = 1; l < Q; ++l)
            acc += (long double)w[k] * ps[(size_t)k * (Q + 1) + l] * sqrtl((long double)l) * ps[(size_t)j * (Q + 1) + l - 1];
        return acc;
    };
    std::vector<double> out(2 * (size_t)QH * QH);
    for (int k = 0; k < QH; ++k)
        for (int j = 0; j < QH; ++j) {
            const long double a = D(k, j), b = D(k, Q - 1 - j);
            out[k * QH + j] = (double)(0.5L * (a - b));
            out[QH * QH + k * QH + j] = (double)(0.5L * (a + b));
        }
    return out;
}

template <typename R>
Pow2<R> make_pow2(int Q, const double* xi) {
    Pow2<R> p{};
    for (int k = 0; k < Q && k < 16; ++k) {
        const double x = xi[k], x2 = x * x;
        p.v[k] = (R)x;
        p.v2[k] = (R)x2;
        p.v3[k] = (R)(x2 * x);
        p.h[k] = (float)x;
        p.l[k] = (float)(x - (double)p.h[k]);
        p.h2[k] = (float)x2;
        p.l2[k] = (float)(x2 - (double)p.h2[k]);
    }
    return p;
}
}  // namespace

bool validate_2d(const evfdlb_params& p) {
    if (p.dim != 2 || p.nx < 8 || p.ny < 8 || !(p.dx > 0) || !(p.sigma > 0) || !(p.phi_a >= 0)) return false;
    if ((long long)p.nx * p.ny >= (1LL << 31)) return false;   // node offsets are 32-bit in k2_adv
    if (p.Q < 4 || p.Q > 16 || (p.Q & 1) || p.bc != EVFDLB_BC_PERIODIC) return false;
    if (p.relax_mode != EVFDLB_RELAX_INV_TAU && p.relax_mode != EVFDLB_RELAX_CHI_OVER_TAU) return false;
    if (!(p.weno_eps > 0) || (!(p.dt > 0) && !(p.cfl > 0 && p.cfl <= 1))) return false;
    double g2 = (p.gamma + 2.0) / 2.0;
    if (!(p.gamma > 3) || fabs(g2 - llround(g2)) > 1e-12) return false;   // even integer gamma
    if (!(p.r_cut >= p.sigma + 2 * p.dx)) return false;
    if (p.precision != EVFDLB_FP64 && p.precision != EVFDLB_FP32) return false;
    return true;
}

double resolved_dt_2d(const evfdlb_params& p) {
    if (p.dt > 0) return p.dt;
    double xi[kQMax], w[kQMax];
    velocity_set(p.Q, xi, w);
    // dimension-by-dimension upwind: |xi_x| + |xi_y| <= 2 max|xi| per dx
    return p.cfl * p.dx / (2.0 * fabs(xi[p.Q - 1]));
}

double discrete_a_2d(const evfdlb_params& p) {
    Taps2 t = taps_2d(p);
    long double acc = 0;
    for (size_t j = 0; j < t.fg.size() / 2; ++j) acc += (long double)t.foff[2 * j] * p.dx * t.fg[2 * j];
    return (double)(0.5L * acc);
}

struct Ctx2 {
    evfdlb_params p;
    Slab2 s;
    int prec = EVFDLB_FP32;
    double dt = 0.0;
    int sms = 1;                 // SMs of the context's device
    size_t esize = 4;
    cudaStream_t user = nullptr, cap = nullptr;
    void* state[3] = {nullptr, nullptr, nullptr};
    void* fld = nullptr;
    double* mom = nullptr;
    double* tables = nullptr;
    void* rtab = nullptr;
    int* fplan = nullptr;        // force plan: per-warp column lists (k2_fields)
    void* ftw = nullptr;         // force weight pairs per column step, precision R
    int* fm_off = nullptr;
    void* fm_w = nullptr;        // Fischer-Methfessel weights, precision R
    float* prf = nullptr;        // FP32 build: node primitives [kNumPrf2][N] of the stage input
    Pow2<float> pwf{};
    Pow2<double> pwd{};
    double* scratch = nullptr;   // [2 Q^2 N + 8] doubles
    unsigned* err = nullptr;
    cudaGraphExec_t g_one = nullptr;
    size_t smem_fields = 0, smem_coll = 0;
    int coll_ctas = 1;           // resident CTAs of k2_coll_pipe
    int field_warps = 8;         // warps per CTA of k2_fields
    // the model constants in precision R (the stage weights are the caller's)
    template <typename R>
    Par2<R> par() const {
        Par2<R> q{};
        const double sg = p.sigma, idx = 1.0 / p.dx;
        q.k12 = (R)(idx / 12.0);
        q.weno_eps = (R)p.weno_eps;
        q.b = (R)(2.0 * M_PI * sg * sg * sg / 3.0);
        q.eta_coef = (R)(M_PI * sg * sg * sg / 6.0);
        q.mu0_coef = (R)(5.0 / (16.0 * sg * sg * sqrt(M_PI)));
        return q;
    }
};

namespace {
// The velocity kernels are compiled for each even Q of the 2D model (4 .. 16);
// f receives the order as a compile-time constant.
template <typename F>
auto with_q(int Q, F f) {
    switch (Q) {
        case 4: return f(std::integral_constant<int, 4>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 8: return f(std::integral_constant<int, 8>{});
        case 10: return f(std::integral_constant<int, 10>{});
        case 12: return f(std::integral_constant<int, 12>{});
        case 14: return f(std::integral_constant<int, 14>{});
        default: return f(std::integral_constant<int, 16>{});
    }
}

// Warps per CTA of k2_fields: one CTA of 24 per SM where every tile has an SM to
// itself (the force disc's columns then run side by side: 96x64 26.5 -> 17.4
// us), 16 up to one and a half tiles per SM (200x200: 27.5 -> 24.2 us), else 8,
// whose CTAs overlap each other's loads (384x384: 43.7 us against 46.9 and 57.1).
// The force sum adds the warps' columns in this division's order: a grid's results
// may differ in the last place between devices with other numbers of SMs.
int field_warps(const Ctx2* c) {
    const long long tiles = (long long)((c->s.nx + kTile2 - 1) / kTile2) * ((c->s.ny + kTile2 - 1) / kTile2);
    return tiles <= c->sms ? kFMaxWarps : (2 * tiles <= 3LL * c->sms ? 16 : 8);
}
template <typename R>
auto fields_kernel_of(const Ctx2* c) {
    return c->field_warps == 8 ? k2_fields<R, 8> : (c->field_warps == 16 ? k2_fields<R, 16> : k2_fields<R, kFMaxWarps>);
}

// Velocities per CTA of k2_adv: up to 16 (the copy offsets are formed once per
// CTA), fewer where the grid would otherwise hold less than four waves of
// CTAs, one on grids of a few tiles.
template <typename R>
void launch_adv(const Ctx2* c, cudaStream_t st, const Par2<R>& pr, const R* src, R* V) {
    const Slab2& s = c->s;
    const long long tiles = (long long)((s.nx + kPT - 1) / kPT) * ((s.ny + kPT - 1) / kPT), K = (long long)s.Q * s.Q;
    const int planes =
        (int)std::min<long long>(16, std::max<long long>(1, tiles * K / (4LL * adv_ctas<R>() * c->sms)));
    const dim3 g((unsigned)tiles, (unsigned)((K + planes - 1) / planes));
    constexpr bool F32 = std::is_same<R, float>::value;
    const bool ftz = F32 && c->p.weno_eps >= kFtzMinEps;
    with_q(s.Q, [&](auto q) {
        constexpr int Q = decltype(q)::value;
        const Pair<R>* in = (const Pair<R>*)src;
        if (ftz) k2_adv<R, Q, F32><<<g, kPThreads, adv_smem<R>(), st>>>(s, pr, (const R*)c->rtab, in, (Pair<R>*)V, planes);
        else k2_adv<R, Q, false><<<g, kPThreads, adv_smem<R>(), st>>>(s, pr, (const R*)c->rtab, in, (Pair<R>*)V, planes);
    });
}

template <typename R>
void launch_coll(const Ctx2* c, cudaStream_t st, const Par2<R>& pr, const R* src, const R* base, R* V) {
    const Slab2& s = c->s;
    const int groups = (int)((s.N + kNB - 1) / kNB);
    with_q(s.Q, [&](auto q) {
        constexpr int Q = decltype(q)::value;
        const R* fld = (const R*)c->fld;
        const Pair<R> *in = (const Pair<R>*)src, *b = (const Pair<R>*)base;
        if constexpr (std::is_same<R, float>::value)
            k2_coll_pipe<Q><<<std::min(groups, c->coll_ctas), coll_threads<Q>(), c->smem_coll, st>>>(
                s, pr, in, fld, b, (float2*)V, groups);
        else k2_coll<R, Q><<<groups, 256, c->smem_coll, st>>>(s, pr, (const R*)c->rtab, in, fld, b, (Pair<R>*)V);
    });
}

// Shared memory of the velocity kernels of order Q, and the resident CTAs of
// the FP32 collision kernel.
cudaError_t configure_2d(Ctx2* c) {
    return with_q(c->s.Q, [&](auto q) {
        constexpr int Q = decltype(q)::value;
        cudaError_t e;
        if (c->prec == EVFDLB_FP32) {
            c->smem_coll = sizeof(float) * Coll2Lay<Q>::PIPE;
            e = raise_smem_limit((const void*)k2_coll_pipe<Q>, c->smem_coll);
            int per_sm = 0;
            if (e == cudaSuccess)
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k2_coll_pipe<Q>, coll_threads<Q>(), c->smem_coll);
            c->coll_ctas = c->sms * std::max(1, per_sm);
        } else {
            c->smem_coll = sizeof(double) * Coll2Lay<Q>::ONE;
            e = raise_smem_limit((const void*)k2_coll<double, Q>, c->smem_coll);
            if (e == cudaSuccess) e = raise_smem_limit((const void*)k2_adv<double, Q, false>, adv_smem<double>());
        }
        return e;
    });
}

// k2_moments: 128 nodes per CTA pass (grid-stride beyond 8192 CTAs)
int moments_grid(long long N) { return (int)std::min<long long>((N + 127) / 128, 8192); }

template <typename R>
void launch_moments(int Q, int nb, cudaStream_t st, const Slab2& s, const Pow2<R>& pw, const Pair<R>* src, double* mom,
                    float* prf, unsigned* err) {
    with_q(Q, [&](auto q) { k2_moments<R, decltype(q)::value><<<nb, 256, 0, st>>>(s, pw, src, mom, prf, err); });
}

template <typename R>
void queue_stage_t(Ctx2* c, cudaStream_t st, const void* src, const void* base, void* out, double alpha, double beta,
                   int mode) {
    const Slab2& s = c->s;
    const int Q = s.Q;
    constexpr bool F32 = std::is_same<R, float>::value;
    // FP32: the field kernel reads the FP32 primitives; the FP64 raw sums are
    // only needed by the FP64 build and by the diagnostics
    const int nbm = moments_grid(s.N);
    Par2<R> pr = c->template par<R>();
    const double cb = mode == 1 ? 1.0 : beta * c->dt;
    pr.alpha = (R)alpha;
    pr.cb = (R)cb;
    pr.ca = (R)(-cb / c->p.dx);
    pr.with_base = alpha != 0.0;
    pr.hs = (R)(mode == 1 ? 0.0 : 1.0);
    R* V = (R*)out;
    if constexpr (F32) launch_moments<float>(Q, nbm, st, s, c->pwf, (const float2*)src, nullptr, c->prf, c->err);
    else launch_moments<double>(Q, nbm, st, s, c->pwd, (const double2*)src, c->mom, nullptr, c->err);
    dim3 gf((s.nx + kTile2 - 1) / kTile2, (s.ny + kTile2 - 1) / kTile2);
    fields_kernel_of<R>(c)<<<gf, 32 * c->field_warps, c->smem_fields, st>>>(
        s, pr, c->mom, c->prf, (const R*)c->ftw, c->fplan, c->fm_off, (const R*)c->fm_w, (R*)c->fld, c->err);
    launch_coll<R>(c, st, pr, (const R*)src, (const R*)base, V);
    launch_adv<R>(c, st, pr, (const R*)src, V);
}

// mode 0: out = alpha base + beta (src + dt L(src)); mode 1: out = L(src)
void queue_stage(Ctx2* c, cudaStream_t st, const void* src, const void* base, void* out, double alpha, double beta,
                 int mode) {
    if (c->prec == EVFDLB_FP32) queue_stage_t<float>(c, st, src, base, out, alpha, beta, mode);
    else queue_stage_t<double>(c, st, src, base, out, alpha, beta, mode);
}

void queue_step(Ctx2* c, cudaStream_t st) {
    queue_stage(c, st, c->state[0], nullptr, c->state[1], 0.0, 1.0, 0);
    queue_stage(c, st, c->state[1], c->state[0], c->state[2], 0.75, 0.25, 0);
    queue_stage(c, st, c->state[2], c->state[0], c->state[0], 1.0 / 3.0, 2.0 / 3.0, 0);
}

evfdlb_status st2(cudaError_t e) {
    return e == cudaSuccess ? EVFDLB_OK : (e == cudaErrorMemoryAllocation ? EVFDLB_E_OOM : EVFDLB_E_CUDA);
}
}  // namespace

void destroy_2d(Ctx2* c) {
    if (!c) return;
    if (c->g_one) cudaGraphExecDestroy(c->g_one);
    for (int i = 0; i < 3; ++i) cudaFree(c->state[i]);
    cudaFree(c->fld);
    cudaFree(c->mom);
    cudaFree(c->tables);
    if (c->rtab != c->tables) cudaFree(c->rtab);
    cudaFree(c->fplan);
    cudaFree(c->ftw);
    cudaFree(c->fm_off);
    cudaFree(c->fm_w);
    cudaFree(c->prf);
    cudaFree(c->scratch);
    cudaFree(c->err);
    if (c->cap) cudaStreamDestroy(c->cap);
    delete c;
}

evfdlb_status create_2d(const evfdlb_params& p, void* stream, Ctx2** out) {
    *out = nullptr;
    if (!validate_2d(p)) return EVFDLB_E_INVALID_ARG;
    if (p.force_model != EVFDLB_EV1 || p.T_iso != 0.0) return EVFDLB_E_UNSUPPORTED;
    Ctx2* c = new (std::nothrow) Ctx2();
    if (!c) return EVFDLB_E_OOM;
    c->p = p;
    c->prec = p.precision;
    c->esize = (c->prec == EVFDLB_FP32) ? sizeof(float) : sizeof(double);
    c->user = (cudaStream_t)stream;
    Slab2& s = c->s;
    s.nx = p.nx;
    s.ny = p.ny;
    s.Q = p.Q;
    s.relax = p.relax_mode;
    s.N = (long long)p.nx * p.ny;
    s.dx = p.dx;
    c->dt = resolved_dt_2d(p);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        c->sms < 1)
        c->sms = 1;
    Taps2 t = taps_2d(p);
    s.nft = (int)(t.fg.size() / 2);
    s.nfm = (int)t.mw.size();
    s.Mf = t.Mf;
    s.mfm = t.mfm;
    TableLayout L(p.Q);
    std::vector<double> tab(L.total), xi(p.Q), w(p.Q);
    velocity_set(p.Q, xi.data(), w.data());
    build_tables(p.Q, xi.data(), w.data(), tab.data());
    const long long NF = (long long)p.Q * p.Q * s.N;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void** ptr, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(ptr, bytes);
    };
    for (int i = 0; i < 3; ++i) alloc(&c->state[i], c->esize * 2 * NF);
    alloc(&c->fld, c->esize * kNumFld2 * s.N);
    alloc((void**)&c->mom, sizeof(double) * kNumMom2 * s.N);
    alloc((void**)&c->tables, sizeof(double) * tab.size());
    c->field_warps = field_warps(c);
    const ForcePlan fp = force_plan(t, c->field_warps);
    if (!fp.ok) e = cudaErrorInvalidValue;      // the tap set lost its mirror symmetry
    const bool f32 = (c->prec == EVFDLB_FP32);
    alloc((void**)&c->fplan, sizeof(int) * fp.plan.size());
    alloc(&c->ftw, c->esize * fp.w.size());
    alloc((void**)&c->fm_off, sizeof(int) * t.moff.size());
    alloc(&c->fm_w, c->esize * t.mw.size());
    if (f32) alloc((void**)&c->prf, sizeof(float) * kNumPrf2 * s.N);
    alloc((void**)&c->scratch, sizeof(double) * (2 * NF + 8));
    alloc((void**)&c->err, sizeof(unsigned));
    std::vector<float> tabf(tab.begin(), tab.end()), ftwf(fp.w.begin(), fp.w.end()), mwf(t.mw.begin(), t.mw.end());
    if (f32) alloc(&c->rtab, sizeof(float) * tab.size());
    else c->rtab = c->tables;
    c->pwf = make_pow2<float>(p.Q, xi.data());
    c->pwd = make_pow2<double>(p.Q, xi.data());
    if (e == cudaSuccess) e = cudaMemcpy(c->tables, tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && c->prec == EVFDLB_FP32)
        e = cudaMemcpy(c->rtab, tabf.data(), sizeof(float) * tabf.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(c->fplan, fp.plan.data(), sizeof(int) * fp.plan.size(), cudaMemcpyHostToDevice);
    // FP64: the parity blocks and the synthesis matrix of this Q into k2_coll's
    // constant bank (every context of the same Q writes the same values)
    if (e == cudaSuccess && !f32) {
        std::vector<double> dbl = d_blocks(p.Q, xi.data(), w.data());
        dbl.insert(dbl.end(), tab.begin() + L.S, tab.begin() + L.S + p.Q * p.Q);
        e = cudaMemcpyToSymbol(c_coll_d, dbl.data(), sizeof(double) * dbl.size(), sizeof(double) * coll_coff(p.Q));
    }
    if (e == cudaSuccess)
        e = f32 ? cudaMemcpy(c->ftw, ftwf.data(), sizeof(float) * ftwf.size(), cudaMemcpyHostToDevice)
                : cudaMemcpy(c->ftw, fp.w.data(), sizeof(double) * fp.w.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(c->fm_off, t.moff.data(), sizeof(int) * t.moff.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = f32 ? cudaMemcpy(c->fm_w, mwf.data(), sizeof(float) * mwf.size(), cudaMemcpyHostToDevice)
                : cudaMemcpy(c->fm_w, t.mw.data(), sizeof(double) * t.mw.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(c->err, 0, sizeof(unsigned));
    auto fields_smem = [&](int nfm) {
        return f32 ? fields_smem_bytes<float>(s.Mf, s.mfm, nfm, c->field_warps)
                   : fields_smem_bytes<double>(s.Mf, s.mfm, nfm, c->field_warps);
    };
    s.fm_staged = fields_smem(s.nfm) <= kFSmemLimit;
    c->smem_fields = fields_smem(s.fm_staged ? s.nfm : 0);
    if (c->smem_fields > kFSmemLimit) e = cudaErrorInvalidValue;   // force disc too wide for a tile
    if (e == cudaSuccess)
        e = raise_smem_limit(f32 ? (const void*)fields_kernel_of<float>(c) : (const void*)fields_kernel_of<double>(c),
                             c->smem_fields);
    if (e == cudaSuccess) e = configure_2d(c);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
        cudaGraph_t g = nullptr;
        e = cudaStreamBeginCapture(c->cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            queue_step(c, c->cap);
            e = cudaStreamEndCapture(c->cap, &g);
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&c->g_one, g, 0);
        if (g) cudaGraphDestroy(g);
    }
    if (e != cudaSuccess) {
        evfdlb_status r = (e == cudaErrorInvalidValue) ? EVFDLB_E_INVALID_ARG : st2(e);
        destroy_2d(c);
        return r;
    }
    *out = c;
    return EVFDLB_OK;
}

// Reads and clears the device error word (synchronises the stream).
evfdlb_status check_2d(Ctx2* c) {
    unsigned h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, c->err, sizeof(unsigned), cudaMemcpyDeviceToHost, c->user);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->user);
    if (e != cudaSuccess) return st2(e);
    if (h) {
        cudaMemsetAsync(c->err, 0, sizeof(unsigned), c->user);
        return (h & ERR_NONFINITE) ? EVFDLB_E_NONFINITE : EVFDLB_E_NEGATIVE;
    }
    return EVFDLB_OK;
}

long long nodes_2d(const Ctx2* c) { return c->s.N; }
long long dist_2d(const Ctx2* c) { return (long long)c->s.Q * c->s.Q * c->s.N; }
double dt_2d(const Ctx2* c) { return c->dt; }

evfdlb_status init_2d(Ctx2* c, const double* n0, const double* u0, const double* T0, int on_device) {
    const long long N = c->s.N;
    const double *dn = n0, *du = u0, *dT = T0;
    cudaError_t e = cudaSuccess;
    if (!on_device) {
        double* b = c->scratch;   // [4 N] fits: 2 Q^2 N >= 4 N
        e = cudaMemcpyAsync(b, n0, sizeof(double) * N, cudaMemcpyHostToDevice, c->user);
        if (e == cudaSuccess) e = cudaMemcpyAsync(b + N, u0, sizeof(double) * 2 * N, cudaMemcpyHostToDevice, c->user);
        if (e == cudaSuccess) e = cudaMemcpyAsync(b + 3 * N, T0, sizeof(double) * N, cudaMemcpyHostToDevice, c->user);
        dn = b;
        du = b + N;
        dT = b + 3 * N;
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(c->err, 0, sizeof(unsigned), c->user);
    if (e != cudaSuccess) return st2(e);
    int nb = (int)std::min<long long>((N + 255) / 256, 4096);
    if (c->prec == EVFDLB_FP32) k2_init<float><<<nb, 256, 0, c->user>>>(c->s, c->tables, dn, du, dT, (float2*)c->state[0], c->err);
    else k2_init<double><<<nb, 256, 0, c->user>>>(c->s, c->tables, dn, du, dT, (double2*)c->state[0], c->err);
    if ((e = cudaGetLastError()) != cudaSuccess) return st2(e);
    return check_2d(c);
}

evfdlb_status step_async_2d(Ctx2* c, int64_t nsteps) {
    for (int64_t i = 0; i < nsteps; ++i) {
        cudaError_t e = cudaGraphLaunch(c->g_one, c->user);
        if (e != cudaSuccess) return st2(e);
    }
    return EVFDLB_OK;
}

// The interleaved state `src` as F and G: device arrays are written by the
// splitting kernel itself, host arrays go through the scratch block.
cudaError_t split_2d(Ctx2* c, const void* src, double* F, double* G, int on_device) {
    const long long NF = dist_2d(c);
    double *dF = on_device ? F : c->scratch, *dG = on_device ? G : c->scratch + NF;
    if (c->prec == EVFDLB_FP32) k2_split<float><<<4096, 256, 0, c->user>>>((const float2*)src, dF, dG, NF);
    else k2_split<double><<<4096, 256, 0, c->user>>>((const double2*)src, dF, dG, NF);
    cudaError_t e = cudaGetLastError();
    if (on_device) return e;
    if (e == cudaSuccess) e = cudaMemcpyAsync(F, dF, sizeof(double) * NF, cudaMemcpyDeviceToHost, c->user);
    if (e == cudaSuccess) e = cudaMemcpyAsync(G, dG, sizeof(double) * NF, cudaMemcpyDeviceToHost, c->user);
    return e;
}

evfdlb_status get_state_2d(Ctx2* c, double* F, double* G, int on_device) {
    cudaError_t e = split_2d(c, c->state[0], F, G, on_device);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->user);
    return st2(e);
}

evfdlb_status set_state_2d(Ctx2* c, const double* F, const double* G, int on_device) {
    const long long NF = dist_2d(c);
    cudaError_t e = cudaSuccess;
    const double *dF = F, *dG = G;
    if (!on_device) {
        e = cudaMemcpyAsync(c->scratch, F, sizeof(double) * NF, cudaMemcpyHostToDevice, c->user);
        if (e == cudaSuccess) e = cudaMemcpyAsync(c->scratch + NF, G, sizeof(double) * NF, cudaMemcpyHostToDevice, c->user);
        dF = c->scratch;
        dG = c->scratch + NF;
    }
    if (e == cudaSuccess) {
        if (c->prec == EVFDLB_FP32) k2_join<float><<<4096, 256, 0, c->user>>>(dF, dG, (float2*)c->state[0], NF);
        else k2_join<double><<<4096, 256, 0, c->user>>>(dF, dG, (double2*)c->state[0], NF);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(c->err, 0, sizeof(unsigned), c->user);
    if (e != cudaSuccess) return st2(e);
    return check_2d(c);
}

evfdlb_status rhs_2d(Ctx2* c, double* RF, double* RG, int on_device) {
    // into the first intermediate state, which holds nothing between steps
    queue_stage(c, c->user, c->state[0], nullptr, c->state[1], 0.0, 1.0, 1);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = split_2d(c, c->state[1], RF, RG, on_device);
    if (e != cudaSuccess) return st2(e);
    return check_2d(c);
}

evfdlb_status moments_2d(Ctx2* c, double* n, double* u, double* T, double* q, double* totals, int on_device) {
    const long long N = c->s.N;
    int nb = (int)std::min<long long>((N + 255) / 256, 4096);
    const int nbm = moments_grid(N);
    if (c->prec == EVFDLB_FP32)
        launch_moments<float>(c->s.Q, nbm, c->user, c->s, c->pwf, (const float2*)c->state[0], c->mom, nullptr, c->err);
    else
        launch_moments<double>(c->s.Q, nbm, c->user, c->s, c->pwd, (const double2*)c->state[0], c->mom, nullptr, c->err);
    double* b = c->scratch;   // n [N], u [2N], T [N], q [2N], totals [4]
    double* dn = n ? (on_device ? n : b) : nullptr;
    double* du = u ? (on_device ? u : b + N) : nullptr;
    double* dT = T ? (on_device ? T : b + 3 * N) : nullptr;
    double* dq = q ? (on_device ? q : b + 4 * N) : nullptr;
    k2_prims<<<nb, 256, 0, c->user>>>(c->s, c->mom, dn, du, dT, dq);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && !on_device) {
        if (n) e = cudaMemcpyAsync(n, dn, sizeof(double) * N, cudaMemcpyDeviceToHost, c->user);
        if (e == cudaSuccess && u) e = cudaMemcpyAsync(u, du, sizeof(double) * 2 * N, cudaMemcpyDeviceToHost, c->user);
        if (e == cudaSuccess && T) e = cudaMemcpyAsync(T, dT, sizeof(double) * N, cudaMemcpyDeviceToHost, c->user);
        if (e == cudaSuccess && q) e = cudaMemcpyAsync(q, dq, sizeof(double) * 2 * N, cudaMemcpyDeviceToHost, c->user);
    }
    if (e == cudaSuccess && totals) {
        k2_totals<<<1, 256, 0, c->user>>>(c->s, c->mom, b + 6 * N);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(totals, b + 6 * N, sizeof(double) * 4, cudaMemcpyDeviceToHost, c->user);
    }
    if (e != cudaSuccess) return st2(e);
    return check_2d(c);
}

}  // namespace evfdlb
