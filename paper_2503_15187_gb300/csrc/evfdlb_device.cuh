// evfdlb_device.cuh -- device-side building blocks of the EV1 right-hand side
// shared by the forward kernels (evfdlb_kernels.cu) and the adjoint kernels
// (evfdlb_adjoint.cu): boundary indexing, the shared-memory layout of a node
// tile, staging of node inputs and of the state tile, the node fields
// (Fischer-Methfessel average, chi, gradients, force, transport), the
// recurrence form of the equilibrium coefficients, the Hermite analysis, the
// WENO-5 faces, the force term and the raw moment sums.  Not part of the
// public interface.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <mutex>
#include <type_traits>
#include <utility>

#include "evfdlb_internal.h"

namespace evfdlb {

// Launches a kernel as a programmatic dependent of the kernel before it in
// the stream: its CTAs may be scheduled once every CTA of that kernel has
// reached griddepcontrol.launch_dependents (or exited), and stage what no
// kernel writes; griddepcontrol.wait in the kernel holds back everything
// that reads the previous kernel's results until it has completed.  Only
// for launches whose stream predecessor is a kernel (not an event wait).
// Launch errors are left for cudaGetLastError, as with <<<>>>.
template <typename... P, typename... A>
inline void launch_pdl(void (*k)(P...), int grid, int threads, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, k, std::forward<A>(args)...);
}

// Raises the limit on a kernel's dynamic shared memory on the current device to
// at least `bytes`.  The limit belongs to the kernel, not to the context that
// asks, so it is never lowered: another context's launches may need more.
inline cudaError_t raise_smem_limit(const void* kernel, size_t bytes) {
    static std::mutex m;                               // (looking and setting are two calls)
    std::lock_guard<std::mutex> lock(m);
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess || (size_t)a.maxDynamicSharedSizeBytes >= bytes) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

__device__ __forceinline__ int gidx(int i, int nx, int bc) {
    if (bc == EVFDLB_BC_PERIODIC) {
        int r = i % nx;
        return r < 0 ? r + nx : r;
    }
    return i < 0 ? 0 : (i >= nx ? nx - 1 : i);
}

// ---------------------------------------------------------------------------
// Shared-memory layout of one CTA, sized for (Q, Z, M): an FP64 block of node
// fields followed by an R block of velocity-space data.
// ---------------------------------------------------------------------------
template <typename R>
struct Smem {
    double *N;          // n on nodes [i0 - M, i0 + Z + M)
    double *U, *T;      // u, T on nodes [i0 - 2, i0 + Z + 2)
    double *X, *Chi;    // X = n^2 chi T and chi on the same nodes
    double *Sc;         // per-node scalars [kNumScalars][Z]
    double *Mtap;       // staged Fischer-Methfessel taps (2m+1 <= 2M+1)
    R *P, *S;           // analysis / synthesis tables [Q*Q] each
    R *Nr;              // n halo in R (the force convolution), aliases N for FP64
    R *Scr;             // nu and F1 in R, [2][Z]
    R *C;               // coefficients [2][Q][Z] (block of 4 H Z >= 2 Q Z values)
    R *A;               // analysis [2][Q][Z] (on the tensor cores: then the integer
                        // parts of the synthesis, [2 d][H even, Q - H odd][Z])
    R *F;               // state tile with halo [2][Q][Z+6]
    R *Face;            // WENO face values [2][Q][Z+1]
    R *Cc;              // per-node coefficient constants c0..c3 [2][4][Z]
    R *Ftap;            // staged force taps [2M+1] (padded to an even count)
    R *Mm;              // Hermite moments m_l of N(u, T) per node [Q][Z]
    double *Vp;         // velocity powers of the moment sums: xi, xi^2, xi^3 (FP64) [3Q]
    R *Vr;              //   and xi, xi^3 in R [2Q]
    R *EO;              // parity-split state tile [2][2][H][Z] (d, E/O), H = (Q+1)/2; it is
                        // read only before the coefficients are formed, so it shares
                        // their block
    // set by stage_tables:
    const R *Rec;       // recurrence constants rinv, rr, r1, r2, r3 [5Q]
    const uint4 *Ma, *Ms;   // digit slices of the transforms on the tensor cores
    int *Ti;            //   and their exponents sx [16], rk [16], gl [32]
    double *Mp64;       // FP32 state only: group terms of the FP64 moment sums [4][G][Z]
    R *Mp32;            //   and of the R ones [2][G][Z] (see pair_terms_f32)
};

// Length of the R copy of the density halo, rounded up to an even count so
// that the blocks after it stay 8-byte aligned (init_kernel stores doubles in
// the coefficient block).
__host__ __device__ inline size_t nr_len(int Z, int M) { return ((size_t)(Z + 2 * M) + 1) & ~(size_t)1; }

__host__ __device__ inline size_t ftap_len(int M) { return ((size_t)(2 * M + 1) + 1) & ~(size_t)1; }

// Groups of two velocity pairs in the FP32 moment sums (see moment_sum).
__host__ __device__ inline int pair_groups(int Q) { return ((Q + 1) / 2 + 1) / 2; }

// Q*Q rounded up to an even count, so that the table blocks stay aligned for
// two-wide (R2) loads.
__host__ __device__ inline size_t qq_len(int Q) { return ((size_t)Q * Q + 1) & ~(size_t)1; }

// Whether the transforms of an FP64 state run on the tensor cores (FP64_DF: all).
template <typename R, bool DF = false>
__host__ __device__ inline bool on_tensor_cores(int Q) {
    return std::is_same<R, double>::value && (DF || Q >= kTsMinQ);
}

// Length of the table block (s.P and s.S, up to Q*Q entries each; with the
// transforms on the tensor cores their exponents, the recurrence constants and the
// scratch of tile_moment_sums, as long as the largest other Q's tables, so that
// a batch's largest Q needs the most), even.
template <typename R>
__host__ __device__ inline size_t tab_len(int Q) {
    return 2 * qq_len(on_tensor_cores<R>(Q) ? kTsMinQ - 1 : Q);
}

// Length of the block of the FP64 stage's recurrence constants: none where they fit
// into the per-node scalars that its roles leave free (SC_U, SC_FORCE; the last
// place there holds the pools) or, with the transforms on the tensor cores, into
// the table block (counted all the same, as in tab_len).  FP32 reads them from
// global memory.
template <typename R>
__host__ __device__ inline size_t rec_len(int Q, int Z) {
    const int q = on_tensor_cores<R>(Q) ? kTsMinQ - 1 : Q;
    return std::is_same<R, float>::value || 5 * q < 2 * Z ? 0 : 5 * (size_t)q;
}

template <typename R>
__host__ __device__ inline size_t smem_bytes_t(int Q, int Z, int M) {
    // the FP64 block is padded to an even count (16-byte aligned R2 tables)
    size_t nd = (size_t)(Z + 2 * M) + 4 * (size_t)(Z + 4) + (size_t)kNumScalars * Z + (size_t)(2 * M + 1);
    nd = (nd + 1) & ~(size_t)1;
    size_t nr = tab_len<R>(Q) + (std::is_same<R, double>::value ? 0 : nr_len(Z, M)) + 2 * (size_t)Z +
                4 * (size_t)((Q + 1) / 2) * Z + 2 * (size_t)Q * Z + 2 * (size_t)Q * (Z + 6) +
                2 * (size_t)Q * (Z + 1) + 8 * (size_t)Z + ftap_len(M) + (size_t)Q * Z;
    // + the velocity powers (3Q doubles, 2Q R) and one R of padding before them
    size_t bytes = (nd + 3 * (size_t)Q) * sizeof(double) + (nr + 2 * (size_t)Q + 1) * sizeof(R);
    bytes += rec_len<R>(Q, Z) * sizeof(R);
    // + the pair terms of the moment sums (FP32 state)
    if (std::is_same<R, float>::value) bytes += (size_t)pair_groups(Q) * Z * (4 * sizeof(double) + 2 * sizeof(R));
    return bytes;
}

// The digit slices of transforms on the tensor cores lie behind that.  A launch
// whose shared memory does not hold them (a large tile beside thousands of force
// taps) reads them from global memory instead.
template <typename R, bool DF>
__host__ __device__ inline size_t stage_full_bytes(int Q, int Z, int M) {
    if (!on_tensor_cores<R, DF>(Q)) return smem_bytes_t<R>(Q, Z, M);
    return ((smem_bytes_t<R>(Q, Z, M) + 15) & ~(size_t)15) + 2 * (size_t)kTsDoubles * sizeof(double);
}

template <typename R>
__device__ inline Smem<R> carve(double* base, int Q, int Z, int M) {
    Smem<R> s;
    s.N = base;
    s.U = s.N + (Z + 2 * M);
    s.T = s.U + (Z + 4);
    s.X = s.T + (Z + 4);
    s.Chi = s.X + (Z + 4);
    s.Sc = s.Chi + (Z + 4);
    s.Mtap = s.Sc + kNumScalars * Z;
    // Mtap holds 2m+1 <= 2M+1 taps; the FP64 block ends on an even count
    // (the dynamic shared memory starts 16-byte aligned)
    const size_t nd = ((size_t)(s.Mtap - base) + (2 * M + 1) + 1) & ~(size_t)1;
    R* r = reinterpret_cast<R*>(base + nd);
    s.P = r;
    s.S = s.P + qq_len(Q);
    if constexpr (std::is_same<R, double>::value) {
        s.Nr = s.N;
        s.Scr = s.P + tab_len<R>(Q);
    } else {
        s.Nr = s.P + tab_len<R>(Q);
        s.Scr = s.Nr + nr_len(Z, M);
    }
    s.C = s.Scr + 2 * Z;
    s.EO = s.C;
    s.A = s.C + 4 * ((Q + 1) / 2) * Z;
    s.F = s.A + 2 * Q * Z;
    s.Face = s.F + 2 * Q * (Z + 6);
    s.Cc = s.Face + 2 * Q * (Z + 1);
    s.Ftap = s.Cc + 8 * Z;
    s.Mm = s.Ftap + ftap_len(M);
    // the velocity powers close the layout: FP64 first (the R block ends on
    // an even count of doubles' worth: all its segment lengths are even)
    s.Vp = reinterpret_cast<double*>(s.Mm + (size_t)Q * Z + ((size_t)Q * Z) % 2);
    s.Vr = reinterpret_cast<R*>(s.Vp + 3 * Q);
    // Vr ends 8-byte aligned (2Q R values after an aligned block)
    s.Mp64 = reinterpret_cast<double*>(s.Vr + 2 * Q);
    s.Mp32 = reinterpret_cast<R*>(s.Mp64 + 4 * (size_t)pair_groups(Q) * Z);
    return s;
}

enum { SC_N = 0, SC_U, SC_FORCE, SC_T, SC_NU, SC_KQ, SC_K, SC_A, SC_B, SC_D };

// IEEE tests by the bit pattern: integer operations, not the FP64 pipe
// (whose compares sit on the node chain's critical path).
__device__ __forceinline__ bool finite(double x) {
    return ((unsigned long long)__double_as_longlong(x) & 0x7ff0000000000000ull) != 0x7ff0000000000000ull;
}
// x > 0: false for +-0, negatives and NaN, true for +inf
__device__ __forceinline__ bool positive(double x) {
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7ff0000000000000ll;
}

// x != 0 by the bit pattern (+-0 are zero), off the FP64 pipe
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }
__device__ __forceinline__ bool nonzero(float x) { return x != 0.0f; }

// The slab constants in R (see SlabDesc).
template <typename R>
__device__ __forceinline__ R slab_inv_dx(const SlabDesc& sd) {
    if constexpr (std::is_same<R, float>::value) return sd.inv_dx_f;
    else return sd.inv_dx;
}
template <typename R>
__device__ __forceinline__ R slab_dt(const SlabDesc& sd) {
    if constexpr (std::is_same<R, float>::value) return sd.dt_f;
    else return sd.dt;
}
template <typename R>
__device__ __forceinline__ R slab_weno_eps(const SlabDesc& sd) {
    if constexpr (std::is_same<R, float>::value) return sd.weno_eps_f;
    else return sd.weno_eps;
}

// Global load of data that other CTAs of the same launch may have written
// (CG: cached in L2 only, never a stale L1 line), or an ordinary load.
template <bool CG, typename T>
__device__ __forceinline__ T gload(const T* p) {
    if constexpr (CG) return __ldcg(p);
    else return *p;
}

// ---------------------------------------------------------------------------
// Double-float arithmetic: a value is an unevaluated pair of floats (hi, lo) with
// x = hi + lo to about 48 significant bits.
// ---------------------------------------------------------------------------
// The split is exact bit surgery, no FP64 instruction: hi is x with its
// significand cut to 24 bits (the top 23 stored bits), lo the remaining 29
// bits rounded to a float (x = hi + lo to 2^-48 relative).  |x| < 2^-126
// gives (0, 0) and |x| < 2^-74 drops lo (absolute error below 2^-98); a
// double-to-float conversion instruction costs several FP64-pipe slots on
// this GPU, the integer path none.
__device__ __forceinline__ float2 df_split(double x) {
    const long long b = __double_as_longlong(x);
    const unsigned hw = (unsigned)(b >> 32);
    const int ed = (int)((hw >> 20) & 0x7ffu);          // biased double exponent
    const unsigned sgn = hw & 0x80000000u;
    float h, l;
    if (ed >= 897 && ed <= 1150) {                       // normal float range
        h = __uint_as_float(sgn | ((unsigned)(ed - 896) << 23) | (unsigned)((b >> 29) & 0x7fffff));
    } else {
        h = (ed > 1150) ? __uint_as_float(sgn | 0x7f800000u) : 0.f;   // overflow -> inf, flagged downstream
    }
    if (ed >= 949 && ed <= 1150) {                       // 2^(ed - 1075) is a normal float
        const float m = __uint2float_rn((unsigned)(b & 0x1fffffff));
        l = __uint_as_float(__float_as_uint(m * __uint_as_float((unsigned)(ed - 948) << 23)) | sgn);
    } else {
        l = 0.f;
    }
    return make_float2(h, l);
}
// double -> float by bit surgery (the head of df_split: the significand cut
// to 24 bits, within one float ulp), no conversion instruction
__device__ __forceinline__ float d2f_bits(double x) { return df_split(x).x; }
// float -> double by bit surgery (exponent rebiased, significand shifted:
// exact for normal floats, zero for zero and subnormals, inf / NaN kept)
__device__ __forceinline__ double f2d_bits(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned ex = (b >> 23) & 0xffu;
    const unsigned long long e64 = (ex == 0u) ? 0ull : (ex == 0xffu ? 2047ull : (unsigned long long)(ex + 896u));
    const unsigned long long man = (ex == 0u) ? 0ull : (unsigned long long)(b & 0x7fffffu) << 29;
    return __longlong_as_double((long long)(((unsigned long long)(b & 0x80000000u) << 32) | (e64 << 52) | man));
}
// a / b in FP64 by Newton-Raphson reciprocal refinement with a final
// residual correction (Markstein, IBM J. Res. Dev. 34, 1990): a float
// reciprocal of b (b cut to a float by bit surgery, reciprocal to 2^-23),
// one Newton step r <- r + r (1 - b r) (2^-46), q = a r and q <- q + r (a - b q)
// (within about one ulp for numerators of magnitude >= 2^-920; below that the
// residual leaves the normal range and the error grows to at most 2^8 ulp;
// not correctly rounded; an overflowing quotient or an infinite numerator
// gives NaN, non-finite like the IEEE +-inf).  Divisors outside the float
// exponent range take the IEEE quotient.
__device__ __forceinline__ double div_nr(double a, double b) {
    const int ex = (int)((__double_as_longlong(b) >> 52) & 0x7ff);
    if (ex < 1023 - 120 || ex > 1023 + 120) return a / b;
    double r = f2d_bits(__frcp_rn(d2f_bits(b)));
    r = fma(r, fma(-b, r, 1.0), r);
    const double q = a * r;
    return fma(fma(-b, q, a), r, q);
}

// div_nr as one copy of its code: a warp that runs straight-line code once waits
// for its instructions (9 of 10 stalls on the stage of 256 x 16 with every
// quotient of the node roles inlined: 12.5 -> 11.6 us).
static __device__ __noinline__ double div_call(double a, double b) { return div_nr(a, b); }

// a / b to about 2^-46 relative: the float-seeded reciprocal of div_nr after
// its Newton step, times a, without the residual correction (3 FP64
// operations instead of 5).  For the WENO-5 face quotient: its error enters
// the stage as dt xi/dx times the face difference, some 1e-14 of the state
// per step, far inside the FP64 parity bars.  Divisors outside the float
// exponent range take the IEEE quotient.
__device__ __forceinline__ double div_face(double a, double b) {
    const int ex = (int)((__double_as_longlong(b) >> 52) & 0x7ff);
    if (ex < 1023 - 120 || ex > 1023 + 120) return a / b;
    double r = f2d_bits(__frcp_rn(d2f_bits(b)));
    r = fma(r, fma(-b, r, 1.0), r);
    return a * r;
}

// ---------------------------------------------------------------------------
// Phase 0: stage the tables, the density halo, u/T near the tile and the
// state tile (+-3 nodes for WENO-5) into shared memory.
// ---------------------------------------------------------------------------
// The transform tables of the slab: the digit slices where the transforms run
// on the tensor cores, else the parity-split analysis pairs and synthesis rows;
// and the recurrence constants.
template <typename R, bool DF>
__device__ void stage_tables(const SlabDesc& sd, Smem<R>& s, int Z, double* smem, const R* __restrict__ rtab) {
    const int Q = sd.Q;
    TableLayout L(Q);
    const R* tab = rtab + sd.tab_off;
    const bool ts = on_tensor_cores<R, DF>(Q);
    if constexpr (std::is_same<R, double>::value) {
        double* rec = on_tensor_cores<R>(Q) ? s.P + kTsInts / 2
                                            : (rec_len<R>(Q, Z) == 0 ? s.Sc + SC_U * Z : s.Vr + 2 * Q);
        for (int t = threadIdx.x; t < 5 * Q; t += blockDim.x) rec[t] = tab[L.rinv + t];   // rinv .. r3 in a row
        s.Rec = rec;
        s.Ti = reinterpret_cast<int*>(s.P);
    } else {
        s.Rec = tab + L.rinv;
    }
    if (ts) {
        if (threadIdx.x < kTsInts) s.Ti[threadIdx.x] = reinterpret_cast<const int*>(tab + L.Mi)[threadIdx.x];
        s.Ma = reinterpret_cast<const uint4*>(tab + L.Ma);
        s.Ms = reinterpret_cast<const uint4*>(tab + L.Ms);
        unsigned dyn;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
        if (stage_full_bytes<R, DF>(Q, Z, sd.M) <= dyn) {
            uint4* x = reinterpret_cast<uint4*>(reinterpret_cast<char*>(smem) + ((smem_bytes_t<R>(Q, Z, sd.M) + 15) & ~(size_t)15));
#pragma unroll 4
            for (int t = threadIdx.x; t < kTsDoubles; t += blockDim.x) x[t] = s.Ma[t];   // Ma, Ms in a row
            s.Ma = x;
            s.Ms = x + kTsDoubles / 2;
        }
    }
    if (!ts) {
        const ParitySplit ps(Q);
        const int la = ps.analysis_len(), ls = ps.synthesis_len();
#pragma unroll 4
        for (int t = threadIdx.x; t < la; t += blockDim.x) s.P[t] = tab[L.Pp + t];
#pragma unroll 4
        for (int t = threadIdx.x; t < ls; t += blockDim.x) s.S[t] = tab[L.Sp + t];
    }
}

// The node inputs of the tile.
template <typename R, bool CG = false>
__device__ void load_node_inputs(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z,
                                 const double* __restrict__ mom, long long NN) {
    const int M = sd.M, nx = sd.nx, bc = sd.bc;
    const double* S0 = mom + MOM_S0 * NN + sd.node_off;
#pragma unroll 2
    for (int t = threadIdx.x; t < it.nz + 2 * M; t += blockDim.x) {
        double n = gload<CG>(S0 + gidx(it.i0 - M + t, nx, bc));
        s.N[t] = n;
        if constexpr (!std::is_same<R, double>::value) s.Nr[t] = (R)n;
    }
    const double* S1 = mom + MOM_S1 * NN + sd.node_off;
    const double* S2 = mom + MOM_S2 * NN + sd.node_off;
    const double* S3 = mom + MOM_S3 * NN + sd.node_off;
    const double* G0 = mom + MOM_G0 * NN + sd.node_off;
    const double* G1 = mom + MOM_G1 * NN + sd.node_off;
    // the node loop on the last threads of the CTA, whose share of the
    // staging above is smallest, so that it runs beside the tap and table
    // staging of the first warps
    for (int t = (int)blockDim.x - 1 - (int)threadIdx.x; t >= 0 && t < it.nz + 4; t += blockDim.x) {
        int i = gidx(it.i0 - 2 + t, nx, bc);
        const bool tile = (t >= 2 && t < it.nz + 2);
        double n = gload<CG>(S0 + i), s1 = gload<CG>(S1 + i), s2 = gload<CG>(S2 + i), g0 = gload<CG>(G0 + i);
        double s3 = tile ? gload<CG>(S3 + i) : 0.0, g1 = tile ? gload<CG>(G1 + i) : 0.0;
        double inv_n = div_nr(1.0, n);
        double u = s1 * inv_n;
        // (3/2) n T = sum (xi-u)^2/2 F + sum G = S2/2 + G0 - n u^2/2
        s.U[t] = u;
        s.T[t] = (2.0 / 3.0) * ((0.5 * s2 + g0) * inv_n - 0.5 * u * u);
        // heat flux of the tile's nodes, q = (S3 - 3u S2 + 3u^2 S1 - u^3 S0)/2 + G1 - u G0,
        // formed here (in parallel, off the node warps' serial chain); the node
        // fields read it from the KQ slot, which they then overwrite with (1 - Pr) q
        if (tile)
            s.Sc[SC_KQ * Z + (t - 2)] = 0.5 * (s3 - 3.0 * u * s2 + 3.0 * u * u * s1 - u * u * u * n) + g1 - u * g0;
    }
}

// Asynchronous global-to-shared copy of one element (4 or 8 bytes, cp.async,
// L1-allocating); completion by cp_async_wait_all.
template <typename R>
__device__ __forceinline__ void cp_async_elem(R* smem_dst, const R* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    if constexpr (sizeof(R) == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gsrc) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The state tile (+-3 nodes) into s.F by asynchronous copies, all of them in
// flight at once; the caller waits (cp_async_wait_all) and synchronises
// before reading it.
// CG: L2-coherent loads instead of the (L1-allocating) copies, for data
// written earlier in the same launch by other CTAs.
template <typename R, bool CG = false>
__device__ void issue_state_tile(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z,
                                 const R* __restrict__ src, long long NF) {
    static_assert(kZMax + 6 <= 96, "a lane holds at most three tile columns");
    const int Q = sd.Q, nx = sd.nx, bc = sd.bc, W = Z + 6;
    const int cols = it.nz + 6;
    // lanes on columns (the node index of a column formed once per lane),
    // warps on velocity rows
    const int lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    int gi[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int c = lane + 32 * q;
        gi[q] = c < cols ? gidx(it.i0 - 3 + c, nx, bc) : 0;
    }
    for (int r = threadIdx.x >> 5; r < 2 * Q; r += nwarps) {
        const int d = r >= Q ? 1 : 0, k = r - d * Q;
        const R* g = src + d * NF + sd.f_off + (long long)k * nx;
        R* row = s.F + (size_t)r * W;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int c = lane + 32 * q;
            if (c < cols) {
                if constexpr (CG) row[c] = __ldcg(g + gi[q]);
                else cp_async_elem<R>(row + c, g + gi[q]);
            }
        }
    }
    if constexpr (!CG) cp_async_commit();
}

// The parity-split interior columns EO[((d * 2 + par) * H + j) * Z + t] of
// the state tile in s.F: E_j = h_j + h_{Q-1-j}, O_j = h_j - h_{Q-1-j} (the
// middle node of an odd Q: E = h, O = 0); threads tid, tid + nth, ...
template <typename R>
__device__ void split_state_tile(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z, int tid, int nth) {
    const int Q = sd.Q, W = Z + 6, H = (Q + 1) / 2, nz = it.nz;
    for (int e = tid; e < 2 * H * nz; e += nth) {
        const int t = e % nz, r = e / nz;
        const int j = r % H, d = r / H, jm = Q - 1 - j;
        const R v = s.F[(size_t)(d * Q + j) * W + t + 3];
        R* eo = s.EO + ((size_t)(2 * d) * H + j) * Z + t;
        if (jm != j) {
            const R vm = s.F[(size_t)(d * Q + jm) * W + t + 3];
            eo[0] = v + vm;
            eo[(size_t)H * Z] = v - vm;
        } else {
            eo[0] = v;
            eo[(size_t)H * Z] = R(0);
        }
    }
}

// sum_{|j| <= m} tap[j + m] x[j] in four interleaved partial sums: a quarter
// of the dependent chain (an FP64 operation waits for the whole warp to pass
// the FP64 pipe of its scheduler, tens of cycles on this part).
template <typename R, typename T>
__device__ __forceinline__ R tap_sum(const T* __restrict__ tap, const R* x, int m) {
    R a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    int j = -m;
    for (; j + 3 <= m; j += 4) {
        a0 = fma((R)tap[j + m], x[j], a0);
        a1 = fma((R)tap[j + 1 + m], x[j + 1], a1);
        a2 = fma((R)tap[j + 2 + m], x[j + 2], a2);
        a3 = fma((R)tap[j + 3 + m], x[j + 3], a3);
    }
    for (; j <= m; ++j) a0 = fma((R)tap[j + m], x[j], a0);
    return (a0 + a1) + (a2 + a3);
}

// ---------------------------------------------------------------------------
// Phases 1-2: node fields of the tile.
// ---------------------------------------------------------------------------
// Pass 1 (threads tid, tid + nth, ...): Fischer-Methfessel average, chi and X
// on nodes i0-2 .. i0+nz+1.  Pass 2 reads the +-2 neighbours of pass 1, so
// the caller separates the passes with a barrier of the participating threads.
// mtap: the slab's Fischer-Methfessel taps [2m+1] (global or staged).
template <typename R>
__device__ void node_fields_pass1(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s,
                                  const double* __restrict__ mtap, long long NN, double* fields_out, int tid,
                                  int nth) {
    const int M = sd.M, m = sd.m;
    // Fischer-Methfessel average (Sec. II.A), chi (Eq. (carnstar)) and
    // X = n^2 chi T on nodes i0-2 .. i0+nz+1.  Under the outflow rule a ghost
    // node copies every node field of the nearest interior node, so the
    // average is centred on the clamped node; under the periodic rule the
    // window around the ghost position is the wrapped node's window.
    for (int t = tid; t < it.nz + 4; t += nth) {
        int pos = it.i0 - 2 + t;
        int shift = (sd.bc == EVFDLB_BC_OUTFLOW) ? gidx(pos, sd.nx, sd.bc) - pos : 0;
        const double* nn = s.N + (t - 2 + M + shift);
        const double nb = tap_sum<double>(mtap, nn, m);
        double eta = sd.eta_coef * nb, om = 1.0 - eta;
        double chi = div_nr(2.0 - eta, 2.0 * om * om * om);
        double n = nn[0];
        s.Chi[t] = chi;
        s.X[t] = n * n * chi * s.T[t];
        if (fields_out && t >= 2 && t < it.nz + 2) {
            long long NNf = NN;
            fields_out[4 * NNf + sd.node_off + it.i0 + t - 2] = nb;
        }
    }
}

// Pass 2: per tile node, the gradients, the Eq. (F1) force (in R), the heat
// flux, the transport coefficients and the scalars of Sc and Scr.
// ftap: the slab's force taps [2M+1] (global or staged).
// PREFORCE: the tile's Eq. (F1) force sums are already in s.Scr[Z + t]
// (formed by other warps, tile_force_sums), else they are summed here.
template <typename R, bool PREFORCE = false>
__device__ void node_fields_pass2(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z,
                                  const R* __restrict__ ftap, const double* __restrict__ mom, long long NN,
                                  unsigned* err, double* fields_out, int tid, int nth) {
    const int M = sd.M;
    const double inv12 = sd.inv_dx / 12.0;
    (void)mom;
    for (int t = tid; t < it.nz; t += nth) {
        const int c = t + 2;                         // index in the +-2 arrays
        const int i = it.i0 + t;
        double n = s.N[t + M], u = s.U[c], T = s.T[c];
        // fourth-order central differences (Sec. III)
        double dX = (s.X[c - 2] - 8.0 * s.X[c - 1] + 8.0 * s.X[c + 1] - s.X[c + 2]) * inv12;
        double dT = (s.T[c - 2] - 8.0 * s.T[c - 1] + 8.0 * s.T[c + 1] - s.T[c + 2]) * inv12;
        double dU = (s.U[c - 2] - 8.0 * s.U[c - 1] + 8.0 * s.U[c + 1] - s.U[c + 2]) * inv12;
        double X = s.X[c], chi = s.Chi[c];
        double A, B;
        // self-consistent force, Eq. (F1), Simpson taps over |j| <= M
        const R* nn = s.Nr + (t + M);
        const R f1r = PREFORCE ? s.Scr[Z + t] : tap_sum<R>(ftap, nn, M);
        double f1;
        if constexpr (std::is_same<R, float>::value) f1 = f2d_bits(f1r);
        else f1 = (double)f1r;
        // heat flux, formed with the node inputs (load_node_inputs)
        double q = s.Sc[SC_KQ * Z + t];
        // transport, Eqs. (viscosity), (tau), (prandtl)
        double bn, x, mu, tau, Pr, nu;
        if constexpr (std::is_same<R, float>::value) {
            // the FP32 variant: gradient ratios and transport on the FP32 pipe
            // (chi, the gradients' differences and the heat flux stay FP64);
            // values cross by bit surgery, not conversion instructions
            const float fn = d2f_bits(n), fT = d2f_bits(T), fchi = d2f_bits(chi);
            const float fA = d2f_bits(dX) / d2f_bits(X), fB = d2f_bits(dT) / fT;
            const float fbn = d2f_bits(sd.b) * fn, fx = fbn * fchi;
            const float c16 = (float)((4.0 / 25.0) * (1.0 + 12.0 / M_PI)), c9 = (float)((9.0 / 25.0) * (1.0 + 32.0 / (9.0 * M_PI)));
            const float fmu = d2f_bits(sd.mu0_coef) * sqrtf(fT) * (1.0f / fchi + 0.8f * fbn + c16 * fbn * fbn * fchi);
            const float ftau = fmu / (fn * fT * (1.0f + 0.4f * fx));
            const float fPr = (2.0f / 3.0f) * (1.0f + 0.6f * fx) * (1.0f + 0.8f * fx + c16 * fx * fx) /
                              ((1.0f + 0.4f * fx) * (1.0f + 1.2f * fx + c9 * fx * fx));
            const float fnu = (sd.relax == EVFDLB_RELAX_INV_TAU) ? 1.0f / ftau : fchi / ftau;
            A = f2d_bits(fA);
            B = f2d_bits(fB);
            bn = f2d_bits(fbn);
            x = f2d_bits(fx);
            mu = f2d_bits(fmu);
            tau = f2d_bits(ftau);
            Pr = f2d_bits(fPr);
            nu = f2d_bits(fnu);
        } else {
            A = div_nr(dX, X);
            B = div_nr(dT, T);
            bn = sd.b * n;
            x = bn * chi;
            mu = sd.mu0_coef * sqrt(T) *
                 (div_nr(1.0, chi) + 0.8 * bn + (4.0 / 25.0) * (1.0 + 12.0 / M_PI) * bn * bn * chi);
            tau = div_nr(mu, n * T * (1.0 + 0.4 * x));
            Pr = div_nr((2.0 / 3.0) * (1.0 + 0.6 * x) * (1.0 + 0.8 * x + (4.0 / 25.0) * (1.0 + 12.0 / M_PI) * x * x),
                        (1.0 + 0.4 * x) * (1.0 + 1.2 * x + (9.0 / 25.0) * (1.0 + 32.0 / (9.0 * M_PI)) * x * x));
            nu = div_nr((sd.relax == EVFDLB_RELAX_INV_TAU) ? 1.0 : chi, tau);
        }
        double* sc = s.Sc;
        sc[SC_N * Z + t] = n;
        sc[SC_U * Z + t] = u;
        sc[SC_T * Z + t] = T;
        sc[SC_NU * Z + t] = nu;
        sc[SC_FORCE * Z + t] = f1;
        sc[SC_KQ * Z + t] = (1.0 - Pr) * q;
        sc[SC_K * Z + t] = -x * n;        // -b n^2 chi, the prefactor of J1
        sc[SC_A * Z + t] = A;
        sc[SC_B * Z + t] = B;
        sc[SC_D * Z + t] = dU;
        if constexpr (std::is_same<R, float>::value) s.Scr[t] = d2f_bits(nu);
        else s.Scr[t] = (R)nu;
        s.Scr[Z + t] = f1r;
        if (!positive(n) || !positive(T)) {
            atomicOr(err, (finite(n) && finite(T)) ? ERR_NEGATIVE : ERR_NONFINITE);
        } else if (!finite(f1) || !finite(nu) || !finite(q) || !finite(A) || !finite(B)) {
            atomicOr(err, ERR_NONFINITE);
        }
        if (fields_out) {
            long long o = sd.node_off + i;
            double vals[EVFDLB_NFIELDS] = {n, u, T, q, 0.0, chi, f1, mu, tau, Pr, nu, A, B, dU, X, x};
            for (int f = 0; f < EVFDLB_NFIELDS; ++f)
                if (f != 4) fields_out[f * NN + o] = vals[f];
        }
    }
}

// The Eq. (F1) force sums of the tile's nodes, f1_t = sum_{|j| <= M}
// ftap_j n_{t+j}, by half-warps of threads tid, tid + nth, ... (nth a
// multiple of 32): the 16 lanes of a half-warp split a node's 2M+1 taps and
// reduce their partial sums by shuffles; the results go to s.Scr[Z + t].
template <typename R>
__device__ void tile_force_sums(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z,
                                const R* __restrict__ ftap, int tid, int nth) {
    const int M = sd.M, sub = tid & 15;
    const unsigned half = 0xffffu << (threadIdx.x & 16);
    for (int t = tid >> 4; t < it.nz; t += nth >> 4) {
        const R* nn = s.Nr + t;                      // nn[j + M] = n_{t+j}
        R a0 = 0, a1 = 0;
        int j = sub;
        for (; j + 16 < 2 * M + 1; j += 32) {
            a0 = fma(ftap[j], nn[j], a0);
            a1 = fma(ftap[j + 16], nn[j + 16], a1);
        }
        if (j < 2 * M + 1) a0 = fma(ftap[j], nn[j], a0);
        R a = a0 + a1;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(half, a, o);
        if (sub == 0) s.Scr[Z + t] = a;
    }
}

// Both passes with all threads of the CTA.
template <typename R>
__device__ void node_fields(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z,
                            const double* __restrict__ taps, const R* __restrict__ rtaps,
                            const double* __restrict__ mom, long long NN, unsigned* err, double* fields_out) {
    node_fields_pass1<R>(sd, it, s, taps + sd.tap_off + 2 * sd.M + 1, NN, fields_out, threadIdx.x, blockDim.x);
    __syncthreads();
    node_fields_pass2<R>(sd, it, s, Z, rtaps + sd.tap_off, mom, NN, err, fields_out, threadIdx.x, blockDim.x);
}

// ---------------------------------------------------------------------------
// Hermite coefficients of nu F^S + J1_F and nu G^S + J1_G.
// With m_l = E[psi_l(u + c)], c ~ N(0, T) (m_0 = 1,
// m_{l+1} = u m_l / sqrt(l+1) + (T-1) sqrt(l/(l+1)) m_{l-1}) and Stein's
// identity E[c h(c)] = T E[h'(c)], the projections of the reduced Shakhov
// equilibria and of the reduced J1 of Sec. II.B are
//   c_l = c0 m_l + c1 sqrt(l) m_{l-1} + c2 sqrt(l(l-1)) m_{l-2}
//         + c3 sqrt(l(l-1)(l-2)) m_{l-3}
// with per-node constants (K = -b n^2 chi, kq = (1-Pr) q):
//   F: c0 = nu n,             c1 = K A T,
//      c2 = 3/5 K D T,        c3 = nu kq/5 + 3/10 K B T^2
//   G: c0 = nu n T + 2/5 K T D,  c1 = 2/5 nu kq + K T^2 (A + 3/5 B),
//      c2 = 3/5 K T^2 D,         c3 = nu kq T/5 + 3/10 K T^3 B
// node_coefficients or node_roles form the constants per node, hermite_moments
// the m_l (recurrence in R); coefficients() then forms every c_l in
// parallel and adds the force term F1 sqrt(l) a_{l-1}
// (d/dxi [omega psi_{l-1}] = -sqrt(l) omega psi_l).
// ---------------------------------------------------------------------------
// m_0 = 1, m_{l+1} = u m_l / sqrt(l+1) + (T-1) sqrt(l/(l+1)) m_{l-1}, to
// mm[l stride] (u, T widened or narrowed to R as the node constants are)
template <typename R>
__device__ __forceinline__ void hermite_moments(int Q, const R* rec, double u, double T, R* mm, int stride) {
    R ru, Tm1;
    if constexpr (std::is_same<R, float>::value) {
        ru = d2f_bits(u);
        Tm1 = d2f_bits(T - 1.0);
    } else {
        ru = (R)u;
        Tm1 = (R)(T - 1.0);
    }
    R m0 = 1, m1 = 0;
    for (int l = 0; l < Q; ++l) {
        mm[l * stride] = m0;
        R mn = fma(ru * rec[l], m0, Tm1 * rec[Q + l] * m1);
        m1 = m0;
        m0 = mn;
    }
}

// The FP32 state forms the constants on the FP32 pipe (an FP64 state: node_roles).
__device__ inline void node_coefficients(const SlabDesc& sd, const WorkItem& it, const Smem<float>& s, int Z, int tid,
                                         int nth) {
    for (int t = tid; t < it.nz; t += nth) {
        const double* sc = s.Sc;
        auto f = [&](int which) { return d2f_bits(sc[which * Z + t]); };
        const float fn = f(SC_N), fT = f(SC_T), fnu = f(SC_NU), fkq = f(SC_KQ);
        const float fK = f(SC_K), fA = f(SC_A), fB = f(SC_B), fD = f(SC_D);
        float* cF = s.Cc + t;
        float* cG = s.Cc + 4 * Z + t;
        cF[0] = fnu * fn;
        cF[Z] = fK * fA * fT;
        cF[2 * Z] = 0.6f * fK * fD * fT;
        cF[3 * Z] = 0.2f * fnu * fkq + 0.3f * fK * fB * fT * fT;
        cG[0] = fnu * fn * fT + 0.4f * fK * fT * fD;
        cG[Z] = 0.4f * fnu * fkq + fK * fT * fT * (fA + 0.6f * fB);
        cG[2 * Z] = 0.6f * fK * fT * fT * fD;
        cG[3 * Z] = 0.2f * fnu * fkq * fT + 0.3f * fK * fT * fT * fT * fB;
    }
}

// The Hermite moments m_l = E[psi_l(u + c)], c ~ N(0, T), of the tile's
// nodes (the recurrence of node_coefficients) from the node inputs u, T of
// load_node_inputs, by threads tid, tid + nth, ...
template <typename R>
__device__ void node_hermite_moments(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z, int tid,
                                     int nth) {
    for (int t = tid; t < it.nz; t += nth) hermite_moments<R>(sd.Q, s.Rec, s.U[t + 2], s.T[t + 2], s.Mm + t, Z);
}

// ---------------------------------------------------------------------------
// The node work of an FP64 stage, by the first four warps of the CTA (one per
// scheduler: an FP64 instruction occupies its scheduler's pipe for 64 cycles
// whatever the active lanes, so the chain of one node is as long as its
// instruction count and only other schedulers shorten it):
//   warp 0  Fischer-Methfessel average and chi; X; transport; the
//           coefficient constants c0 .. c3;
//   warp 1  u, T, q from the raw sums; the gradients;
//   warp 2  the Hermite moments of the local Gaussian;
//   warp 3  the force sums.
// The transport is written in x = b n chi throughout, with P = 1 + 4/5 x +
// c16 x^2 the factor that mu chi and Pr share:
//   nu = n sqrt(T) chi (1 + 2/5 x) / (mu0 P)  (times chi for the rate chi/tau),
//   Pr = 2/3 (1 + 3/5 x) P / ((1 + 2/5 x) (1 + 6/5 x + c9 x^2)),
// and q = S3/2 + G1 - u (3/2 S2 + G0 - u S1).  On tiles of a few nodes this
// chain is the stage: about 100 FP64 instructions on its longest warp, where
// one warp with everything took 260 (dx = 0.25, Q = 16) to 400: a stage of
// 256 x 16 takes 12.5 us instead of 18.4, of 2000 x 16 (EV2) 15.9 instead of
// 21.0, of 1024 x 24 16.6 instead of 22.5.
// Every sum has a fixed order, so results do not depend on the tile.
// ---------------------------------------------------------------------------
// Raw sums for the roles: n on the density halo; S1, S2, G0 on +-2 nodes (in
// the U, T and X arrays), S3 and G1 of the tile (in the KQ and A scalars).
template <bool CG>
__device__ void load_raw_sums(const SlabDesc& sd, const WorkItem& it, const Smem<double>& s, int Z,
                              const double* __restrict__ mom, long long NN) {
    const int M = sd.M, nx = sd.nx, bc = sd.bc;
    const double* m = mom + sd.node_off;
#pragma unroll 2
    for (int t = threadIdx.x; t < it.nz + 2 * M; t += blockDim.x)
        s.N[t] = gload<CG>(m + MOM_S0 * NN + gidx(it.i0 - M + t, nx, bc));
    for (int t = (int)blockDim.x - 1 - (int)threadIdx.x; t < it.nz + 4; t += blockDim.x) {
        const int i = gidx(it.i0 - 2 + t, nx, bc);
        const bool tile = (t >= 2 && t < it.nz + 2);
        const double s1 = gload<CG>(m + MOM_S1 * NN + i), s2 = gload<CG>(m + MOM_S2 * NN + i);
        const double g0 = gload<CG>(m + MOM_G0 * NN + i);
        const double s3 = tile ? gload<CG>(m + MOM_S3 * NN + i) : 0.0, g1 = tile ? gload<CG>(m + MOM_G1 * NN + i) : 0.0;
        s.U[t] = s1;
        s.T[t] = s2;
        s.X[t] = g0;
        if (tile) {
            s.Sc[SC_KQ * Z + t - 2] = s3;
            s.Sc[SC_A * Z + t - 2] = g1;
        }
    }
}

// sum_j tap[j] x[j], j < n, in C chains over j mod C joined pairwise, by lp
// neighbouring lanes per sum (lp <= C a power of two; sub = the lane's index
// among them): the same operations and order for every lp.
template <int C, int PER>
__device__ __forceinline__ double chain_sum_t(const double* __restrict__ tap, const double* x, int n, int sub) {
    double a[PER];                                 // chains sub PER .. sub PER + PER - 1
#pragma unroll
    for (int c = 0; c < PER; ++c) a[c] = 0.0;
    int j = sub * PER;
    for (; j + PER <= n; j += C) {
#pragma unroll
        for (int c = 0; c < PER; ++c) a[c] = fma(tap[j + c], x[j + c], a[c]);
    }
#pragma unroll
    for (int c = 0; c < PER; ++c)
        if (j + c < n) a[c] = fma(tap[j + c], x[j + c], a[c]);
#pragma unroll
    for (int w = 1; w < PER; w *= 2)
#pragma unroll
        for (int c = 0; c < PER; c += 2 * w) a[c] += a[c + w];
#pragma unroll
    for (int w = 1; w < C / PER; w *= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], w);
    return a[0];
}
template <int C>
__device__ __forceinline__ double chain_sum(const double* __restrict__ tap, const double* x, int n, int lp, int sub) {
    if (lp == 1) return chain_sum_t<C, C>(tap, x, n, sub);
    if (lp == 2) return chain_sum_t<C, C / 2>(tap, x, n, sub);
    if (C == 4 || lp == 4) return chain_sum_t<C, C / 4>(tap, x, n, sub);
    return chain_sum_t<C, (C >= 8 ? C / 8 : 1)>(tap, x, n, sub);
}
// lanes per sum for n sums on one warp
__device__ __forceinline__ int lanes_per(int n, int most) {
    int lp = 1;
    while (lp < most && 2 * lp * n <= 32) lp *= 2;
    return lp;
}

template <bool FO>
__device__ void node_roles(const SlabDesc& sd, const WorkItem& it, const Smem<double>& s, int Z, long long NN,
                           unsigned* err, double* fields_out) {
    const int M = sd.M, nz = it.nz, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* sc = s.Sc;
    auto join3 = [] { asm volatile("bar.sync 1, 96;" ::: "memory"); };    // warps 0, 1, 2
    auto join2 = [] { asm volatile("bar.sync 4, 64;" ::: "memory"); };    // warps 0, 1
    auto field = [&](int f, int t, double v) {
        if constexpr (FO) fields_out[f * NN + sd.node_off + it.i0 + t] = v;
    };
    auto node_ok = [&](int t) { return positive(s.N[t + M]) && positive(s.T[t + 2]); };
    if (warp == 0) {
        // Under the outflow rule a ghost node copies every field of the
        // nearest interior node: the average is centred on the clamped node.
        const int lp = lanes_per(nz + 4, 4), sub = lane % lp;
        for (int t0 = 0; t0 < nz + 4; t0 += 32 / lp) {
            const int t = min(t0 + lane / lp, nz + 3), pos = it.i0 - 2 + t;
            const int shift = (sd.bc == EVFDLB_BC_OUTFLOW) ? gidx(pos, sd.nx, sd.bc) - pos : 0;
            const double nb = chain_sum<4>(s.Mtap, s.N + (t - 2 + M + shift - sd.m), 2 * sd.m + 1, lp, sub);
            const double eta = sd.eta_coef * nb, om = 1.0 - eta;
            const double chi = div_call(2.0 - eta, 2.0 * om * om * om);
            if (sub == 0) {
                s.Chi[t] = chi;
                if (t >= 2 && t < nz + 2) field(4, t - 2, nb);
            }
        }
        join3();
        for (int t = lane; t < nz + 4; t += 32) {
            const int pos = it.i0 - 2 + t;
            const int shift = (sd.bc == EVFDLB_BC_OUTFLOW) ? gidx(pos, sd.nx, sd.bc) - pos : 0;
            const double n = s.N[t - 2 + M + shift];
            s.X[t] = n * n * s.Chi[t] * s.T[t];
        }
        join2();
        for (int t = lane; t < nz; t += 32) {
            const double n = s.N[t + M], T = s.T[t + 2], chi = s.Chi[t + 2], q = sc[SC_KQ * Z + t];
            const double c16 = (4.0 / 25.0) * (1.0 + 12.0 / M_PI), c9 = (9.0 / 25.0) * (1.0 + 32.0 / (9.0 * M_PI));
            const double x = sd.b * n * chi, a = fma(0.4, x, 1.0), P = fma(fma(c16, x, 0.8), x, 1.0), st = sqrt(T);
            double nu = div_call(n * st * chi * a, sd.mu0_coef * P);
            if (sd.relax != EVFDLB_RELAX_INV_TAU) nu *= chi;
            const double Pr = div_call(fma(0.4, x, 2.0 / 3.0) * P, a * fma(fma(c9, x, 1.2), x, 1.0));
            sc[SC_N * Z + t] = n;
            sc[SC_T * Z + t] = T;
            sc[SC_NU * Z + t] = nu;
            sc[SC_KQ * Z + t] = (1.0 - Pr) * q;
            sc[SC_K * Z + t] = -x * n;               // -b n^2 chi, the prefactor of J1
            s.Scr[t] = nu;
            if (!positive(n) || !positive(T)) atomicOr(err, (finite(n) && finite(T)) ? ERR_NEGATIVE : ERR_NONFINITE);
            else if (!finite(nu) || !finite(q)) atomicOr(err, ERR_NONFINITE);
            if constexpr (FO) {
                const double mu = sd.mu0_coef * st * div_call(P, chi);
                field(0, t, n);
                field(1, t, s.U[t + 2]);
                field(2, t, T);
                field(3, t, q);
                field(5, t, chi);
                field(7, t, mu);
                field(8, t, div_call(mu, n * T * a));
                field(9, t, Pr);
                field(10, t, nu);
                field(14, t, s.X[t + 2]);
                field(15, t, x);
            }
        }
        join2();
        // c0 .. c3 of both distributions (see node_coefficients)
        for (int t = lane; t < nz; t += 32) {
            const double n = sc[SC_N * Z + t], T = sc[SC_T * Z + t], nu = sc[SC_NU * Z + t];
            const double kq = sc[SC_KQ * Z + t], K = sc[SC_K * Z + t];
            const double A = sc[SC_A * Z + t], B = sc[SC_B * Z + t], D = sc[SC_D * Z + t];
            const double KT = K * T, KT2 = KT * T, KTD = KT * D, nk = nu * kq;
            const double f0 = nu * n, f2 = 0.6 * KTD, f3 = fma(0.3 * KT2, B, 0.2 * nk);
            double* cF = s.Cc + t;
            double* cG = s.Cc + 4 * Z + t;
            cF[0] = f0;
            cF[Z] = KT * A;
            cF[2 * Z] = f2;
            cF[3 * Z] = f3;
            cG[0] = fma(f0, T, 0.4 * KTD);
            cG[Z] = fma(KT2, fma(0.6, B, A), 0.4 * nk);
            cG[2 * Z] = f2 * T;
            cG[3 * Z] = f3 * T;
        }
    } else if (warp == 1) {
        for (int t = lane; t < nz + 4; t += 32) {
            const bool tile = (t >= 2 && t < nz + 2);
            const int pos = it.i0 - 2 + t;
            const int shift = (sd.bc == EVFDLB_BC_OUTFLOW) ? gidx(pos, sd.nx, sd.bc) - pos : 0;
            const double n = s.N[t - 2 + M + shift], s1 = s.U[t], s2 = s.T[t], g0 = s.X[t];
            const double inv_n = div_call(1.0, n), u = s1 * inv_n;
            s.U[t] = u;
            // (3/2) n T = sum (xi-u)^2/2 F + sum G = S2/2 + G0 - n u^2/2
            s.T[t] = (2.0 / 3.0) * fma(fma(0.5, s2, g0), inv_n, -0.5 * u * u);
            if (tile) {
                const double s3 = sc[SC_KQ * Z + t - 2], g1 = sc[SC_A * Z + t - 2];
                sc[SC_KQ * Z + t - 2] = fma(-u, fma(-u, s1, fma(1.5, s2, g0)), fma(0.5, s3, g1));
            }
        }
        join3();
        const double inv12 = sd.inv_dx / 12.0;
        // fourth-order central differences (Sec. III)
        auto d4 = [&](const double* f) { return fma(8.0, f[1] - f[-1], f[-2] - f[2]) * inv12; };
        for (int t = lane; t < nz; t += 32) {
            sc[SC_D * Z + t] = d4(s.U + t + 2);
            sc[SC_B * Z + t] = div_call(d4(s.T + t + 2), s.T[t + 2]);
        }
        join2();
        for (int t = lane; t < nz; t += 32) {
            const double A = div_call(d4(s.X + t + 2), s.X[t + 2]), B = sc[SC_B * Z + t];
            sc[SC_A * Z + t] = A;
            if (node_ok(t) && (!finite(A) || !finite(B))) atomicOr(err, ERR_NONFINITE);
            field(11, t, A);
            field(12, t, B);
            field(13, t, sc[SC_D * Z + t]);
        }
        join2();
    } else if (warp == 2) {
        join3();
        for (int t = lane; t < nz; t += 32) hermite_moments<double>(sd.Q, s.Rec, s.U[t + 2], s.T[t + 2], s.Mm + t, Z);
    } else {
        // self-consistent force, Eq. (F1) (or the merged Eq. (F2) stencil)
        const int lp = lanes_per(nz, 8), sub = lane % lp;
        for (int t0 = 0; t0 < nz; t0 += 32 / lp) {
            const int t = min(t0 + lane / lp, nz - 1);
            const double f1 = chain_sum<8>(s.Ftap, s.N + t, 2 * M + 1, lp, sub);
            if (sub == 0) {
                s.Scr[Z + t] = f1;
                if (!finite(f1)) atomicOr(err, ERR_NONFINITE);
                field(6, t, f1);
            }
        }
    }
}

template <typename R>
__device__ void coefficients(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z, int tid,
                             int nth) {
    const int Q = sd.Q, nz = it.nz;
    const R *r1 = s.Rec + 2 * Q, *r2 = s.Rec + 3 * Q, *r3 = s.Rec + 4 * Q;
    // one (l, node) per item, both distributions: the scaled moments
    // sqrt(l(l-1)..) m_{l-j} and the force factor F1 sqrt(l) are shared
    for (int e = tid; e < Q * nz; e += nth) {
        const int t = e % nz, l = e / nz;
        const R* mm = s.Mm + t;
        // the sqrt factors vanish where the moment index would be negative
        const R m0 = mm[l * Z];
        const R M1 = r1[l] * mm[max(l - 1, 0) * Z];
        const R M2 = r2[l] * mm[max(l - 2, 0) * Z];
        const R M3 = r3[l] * mm[max(l - 3, 0) * Z];
        const R f = s.Scr[Z + t] * r1[l];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const R* cc = s.Cc + d * 4 * Z + t;
            R c = cc[0] * m0;
            c = fma(cc[Z], M1, c);
            c = fma(cc[2 * Z], M2, c);
            c = fma(cc[3 * Z], M3, c);
            if (l >= 1) c = fma(f, s.A[((size_t)d * Q + l - 1) * Z + t], c);
            s.C[((size_t)d * Q + l) * Z + t] = c;
        }
    }
}

// Warp-sized groups of e = 0 .. n-1 from a shared counter (zeroed before), for
// warps that arrive at different times: f(e) for every e, by one lane each.
template <typename F>
__device__ __forceinline__ void warp_pool(int* next, int n, F f) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        int g = 0;
        if (lane == 0) g = atomicAdd(next, 1);
        g = __shfl_sync(0xffffffffu, g, 0) * 32;
        if (g >= n) return;
        if (g + lane < n) f(g + lane);
    }
}

// ---------------------------------------------------------------------------
// The Hermite transforms of an FP64 stage on the tensor cores, in fixed point
// (see kTsSlices): one warp forms both parities of one distribution for eight
// nodes.  A lane holds the values of rows 2 (lane % 4) + {0, 1, 8, 9} of node
// lane / 4 (the fragment of mma.m16n8k16's B operand), turns them into
// integers on the node's own exponent, cuts their digits, and 21 products per
// parity of digit slices accumulate exactly; the six accumulators join in
// 64-bit integers, which become doubles by bit operations.  Nothing runs on the
// FP64 pipe, which bounds the stage and spent a third of it on the sums.  The
// result carries about 2^-56 of the largest value times the largest entry, below
// the rounding of an FP64 sum of up to 16 terms (2^-53 each), whatever the state
// (see kTsSlices): against 80-bit arithmetic a right-hand side has 0.8 .. 1.1 of the
// plain sums' error (Q = 17 .. 32; noise and liquid slabs up to 4000 steps on, slabs
// after a density step, nodes at T = 0.15 .. 1.5 and u up to 4).  Only within the rows of the
// outermost velocities, 1e-10 of the largest and less, is it a few times theirs.  Columns
// (nodes) are independent, so results do not depend on the tile.  Stage of
// 4096 x 32: 44.6 -> 33.8 us, of 65536 x 24 (tile 32): 438 -> 328 us.
//
// A warp's work is a chain of integer operations (about 900 instructions a
// parity, mostly the digits and the joins; the products take 180 cycles), so the
// phase is bound by latency: values and results go through it four at a time.
// FP64_DF with Q <= 16 has both parities in one block (even orders in rows and
// columns 0-7, odd in 8-15).
// ---------------------------------------------------------------------------
// sign, exponent field (with `shift` added; 0 for zero and subnormal values)
// and 53-bit significand of x
struct FixIn {
    unsigned hi, lo;
    int e;
};
__device__ __forceinline__ FixIn fix_in(double x, int shift) {
    FixIn f;
    f.hi = (unsigned)__double2hiint(x);
    f.lo = (unsigned)__double2loint(x);
    const int e = (int)((f.hi >> 20) & 0x7ffu);
    f.e = e == 0 ? -100000 : (e == 2047 ? 100000 : e + shift);
    return f;
}
// x 2^(lead + 1075 - emax), rounded (emax >= the exponent of x; zero if none)
__device__ __forceinline__ long long fix_value(const FixIn& f, int emax, int lead) {
    // one bit more than wanted, then rounded by it
    const unsigned sh = (unsigned)min(emax - f.e, 63);
    const unsigned long long m = (((unsigned long long)((f.hi & 0xfffffu) | 0x100000u) << 32) | f.lo) << (lead + 1);
    const long long v = (long long)(((m >> sh) + 1) >> 1);
    return (int)f.hi < 0 ? -v : v;
}
// digit slices of two values |v| < 2^59 as FP16 pairs, most significant first
__device__ __forceinline__ void fix_slices(long long va, long long vb, unsigned (&out)[kTsSlices]) {
    // + 512 in every digit makes them the unsigned 10-bit fields u of the sum
    // (the top one up to 1024); 0x6400 + u is the FP16 number 1024 + u
    constexpr unsigned long long bias = 512ull * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) + (1ull << 40) + (1ull << 50));
    const unsigned long long a = (unsigned long long)va + bias, b = (unsigned long long)vb + bias;
    const __half2 off = __half2half2(__short_as_half((short)0x6600));           // 1536 = 1024 + 512
#pragma unroll
    for (int i = 0; i < kTsSlices; ++i) {
        const int pos = 10 * (kTsSlices - 1 - i);
        unsigned ua = (unsigned)(a >> pos), ub = (unsigned)(b >> pos);
        if (i > 0) ua &= 1023u, ub &= 1023u;
        const unsigned w = 0x64006400u + (ua | (ub << 16));
        const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), off);
        out[i] = *reinterpret_cast<const unsigned*>(&h);
    }
}
// acc[s] += the slice products of weight s: table slices A (global fragment
// order in shared memory) times value slices (b0: rows k, k+1; b1: k+8, k+9)
__device__ __forceinline__ void fix_products(const uint4* A, const unsigned (&b0)[kTsSlices],
                                             const unsigned (&b1)[kTsSlices], float (&acc)[kTsSlices][4]) {
#pragma unroll
    for (int s = 0; s < kTsSlices; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[s][c] = 0.f;
#pragma unroll
    for (int i = 0; i < kTsSlices; ++i) {
        const uint4 a = A[i * 32 + (threadIdx.x & 31)];
#pragma unroll
        for (int k = 0; i + k < kTsSlices; ++k) {
            float(&c)[4] = acc[i + k];
            asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
                : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0[k]), "r"(b1[k]));
        }
    }
}
// the sum of the accumulators of element c, in units of 2^3
__device__ __forceinline__ long long fix_join(const float (&acc)[kTsSlices][4], int c) {
    auto g = [&](int s) {
        return ((long long)__float2int_rn(acc[s][c]) << 20) + ((long long)__float2int_rn(acc[s + 1][c]) << 10) +
               __float2int_rn(acc[s + 2][c]);
    };
    return (g(0) << 18) + ((g(3) + 2048) >> 12);
}
// Four values of a lane's node through one 16 x 16 block of the table: results
// for rows lane / 4 (+ 8) of nodes 2 (lane % 4) (+ 1) in the order of the
// accumulator fragment.  One copy of the code serves every task: straight-line
// code that a CTA runs once waits for its instructions (half of all stalls of
// the stage of 4096 x 32 with the tasks inlined, 9 of 10 on 256 x 16).
struct Fix4 {
    long long v[4];
};
static __device__ __noinline__ Fix4 fix_transform(const uint4* A, Fix4 x) {
    unsigned b0[kTsSlices], b1[kTsSlices];
    fix_slices(x.v[0], x.v[1], b0);
    fix_slices(x.v[2], x.v[3], b1);
    float acc[kTsSlices][4];
    fix_products(A, b0, b1, acc);
    Fix4 o;
#pragma unroll
    for (int c = 0; c < 4; ++c) o.v[c] = fix_join(acc, c);
    return o;
}
// v 2^q as a double, rounded to nearest (ties away; zero below the normal
// range), |v| < 2^62; NaN when `bad`
__device__ __forceinline__ double fix_out(long long v, int q, bool bad) {
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int lz = __clzll((long long)a);
    const int e = 62 - lz + q + 1023;                          // exponent field - 1: the leading bit adds one
    // the significand with its leading bit at 52, rounded; a carry out of it
    // goes into the exponent as it should
    unsigned long long r = ((unsigned long long)e << 52) + (((a << (lz - 1)) + 0x200ull) >> 10);
    if (a == 0 || e < 0) r = 0;
    if (e >= 2046) r = 0x7ff0000000000000ull;
    if (v < 0) r |= 0x8000000000000000ull;
    if (bad) r = 0x7ff8000000000000ull;
    return __longlong_as_double((long long)r);
}

// the largest of a value over the four lanes of a node
__device__ __forceinline__ int quad_max(int e) {
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
    return max(e, __shfl_xor_sync(0xffffffffu, e, 2));
}

// Task g of the analysis, a_l = sum_{j<H} psi_l(xi_j) (E_j or O_j), l <= Q-2, E_j
// = h_j + h_{Q-1-j}, O_j = h_j - h_{Q-1-j} (the middle velocity of an odd Q: h, 0),
// formed as integers: distribution g % 2, nodes 8 (g / 2) .. + 7, parities p0 .. p1 - 1.
template <bool DF>
__device__ __forceinline__ void analysis_task(const SlabDesc& sd, const WorkItem& it, const Smem<double>& s, int Z,
                                              int g, int p0, int p1) {
    const int Q = sd.Q, H = (Q + 1) / 2, W = Z + 6, nz = it.nz, lane = threadIdx.x & 31;
    const int d = g & 1, t0 = (g >> 1) * 8, t = min(t0 + lane / 4, nz - 1), k0 = 2 * (lane % 4);
    const double* h = s.F + (size_t)d * Q * W + t + 3;
    FixIn x[4], y[4];
    int emax = -100000;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int j = k0 + (c & 1) + 8 * (c >> 1), jm = Q - 1 - j;
        const bool in = j < H;
        const int sx = in ? s.Ti[j] : 0;
        x[c] = fix_in(in ? h[j * W] : 0.0, -sx);
        y[c] = fix_in(in && jm != j ? h[jm * W] : 0.0, -sx);
        emax = max(emax, max(x[c].e, y[c].e));
    }
    emax = quad_max(emax);
    const bool bad = emax > 50000;
    long long E[4], O[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int j = k0 + (c & 1) + 8 * (c >> 1);
        const long long a = bad ? 0 : fix_value(x[c], emax, 5);
        const long long b = bad ? 0 : fix_value(y[c], emax, 5);
        E[c] = a + b;
        O[c] = 2 * j == Q - 1 ? 0 : a - b;
    }
    const int q = emax - 1077;
    const bool folded = DF && Q <= 16;
    double* A = s.A + (size_t)d * Q * Z;
    for (int par = p0; par < p1; ++par) {
        Fix4 v;
#pragma unroll
        for (int c = 0; c < 4; ++c) v.v[c] = par == 0 ? E[c] : O[c];
        if (folded) v.v[2] = O[0], v.v[3] = O[1];
        const Fix4 o = fix_transform(s.Ma + par * kTsSlices * 32, v);
        // element c: row lane / 4 (+ 8), node t0 + 2 (lane % 4) (+ 1), whose
        // exponent the lanes of that node hold
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int col = k0 + (c & 1), src = col * 4;
            const int qc = __shfl_sync(0xffffffffu, q, src), fl = __shfl_sync(0xffffffffu, (int)bad, src);
            const int l = folded ? 2 * (lane / 4) + (c >> 1) : 2 * (lane / 4 + 8 * (c >> 1)) + par;
            if (l <= Q - 2 && t0 + col < nz) A[l * Z + t0 + col] = fix_out(o.v[c], qc, fl != 0);
        }
    }
}

// Task g of the synthesis: the sum of S_kl c_l over the orders of parity g % 2
// for k < H, distribution (g / 2) % 2, nodes 8 (g / 4) .. + 7, as integers of the
// unit 2^(qn - 1078 + rk_k), qn the exponent of the node's largest coefficient
// (of both parities, so that the two sums share a unit; kTsBad marks a
// non-finite one); E + O is the synthesis at k, E - O at Q-1-k.
constexpr int kTsBad = 1 << 20;
template <bool DF>
__device__ __forceinline__ void synthesis_task(const SlabDesc& sd, const WorkItem& it, const Smem<double>& s, int Z,
                                               long long* part, int* qn, int g) {
    const int Q = sd.Q, H = (Q + 1) / 2, nz = it.nz, lane = threadIdx.x & 31;
    const bool folded = DF && Q <= 16;
    const int par = folded ? 0 : g & 1;
    if (!folded) g >>= 1;
    const int d = g & 1, t0 = (g >> 1) * 8, t = min(t0 + lane / 4, nz - 1), k0 = 2 * (lane % 4);
    const int* gl = s.Ti + 32;
    const double* c0 = s.C + (size_t)d * Q * Z + t;
    FixIn x[4];
    int emax = -100000;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int m = k0 + (c & 1);
        const int l = folded ? 2 * m + (c >> 1) : 2 * (m + 8 * (c >> 1)) + par, lo = folded ? l : l ^ 1;
        x[c] = fix_in(l < Q ? c0[l * Z] : 0.0, l < Q ? gl[l] : 0);
        emax = max(emax, max(x[c].e, fix_in(lo < Q ? c0[lo * Z] : 0.0, lo < Q ? gl[lo] : 0).e));
    }
    emax = quad_max(emax);
    const bool bad = emax > 50000;
    Fix4 v;
#pragma unroll
    for (int c = 0; c < 4; ++c) v.v[c] = bad ? 0 : fix_value(x[c], emax, 6);
    const Fix4 r = fix_transform(s.Ms + par * kTsSlices * 32, v);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int tt = t0 + k0 + (c & 1), k = folded ? lane / 4 : lane / 4 + 8 * (c >> 1);
        const int po = folded ? c >> 1 : par;
        // (the odd part of an odd Q's middle velocity is zero)
        if (k < (po ? Q - H : H) && tt < nz) part[((size_t)d * Q + po * H + k) * Z + tt] = r.v[c];
    }
    if (par == 0 && (lane & 3) == 0 && t0 + lane / 4 < nz) qn[d * Z + t] = bad ? kTsBad : emax;
}
__host__ __device__ inline int transform_tasks(int nz) { return 2 * ((nz + 7) / 8); }

// Parity-split analysis: a_l = sum_{j<H} psi_l(xi_j) (E_j or O_j), l <= Q-2,
// two orders of one parity (l, l+2) per thread sharing each E/O value loaded
// (Pp holds the two table values side by side: one two-wide load).
// Threads tid, tid + nth, ... (next null), or whole warps from the pool `next`.
template <typename R>
__device__ void analysis_eo(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z, int tid, int nth,
                            int* next = nullptr) {
    using R2 = typename std::conditional<std::is_same<R, float>::value, float2, double2>::type;
    const int Q = sd.Q, nz = it.nz;
    const ParitySplit ps(Q);
    const int H = ps.H, G = ps.GE + ps.GO;
    const R2* Pp = reinterpret_cast<const R2*>(s.P);
    auto task = [&](int e) {
        const int t = e % nz, r = e / nz;
        const int g = r % G, d = r / G;
        const int par = g < ps.GE ? 0 : 1;
        const int l0 = par ? 4 * (g - ps.GE) + 1 : 4 * g;
        const R* x = s.EO + ((size_t)(2 * d + par) * H) * Z + t;
        const R2* pp = Pp + (size_t)g * H;
        R a0 = 0, a1 = 0;
        for (int j = 0; j < H; ++j) {
            const R v = x[j * Z];
            const R2 p = pp[j];
            a0 = fma(p.x, v, a0);
            a1 = fma(p.y, v, a1);
        }
        s.A[((size_t)d * Q + l0) * Z + t] = a0;
        if (l0 + 2 <= Q - 2) s.A[((size_t)d * Q + l0 + 2) * Z + t] = a1;
    };
    if (next) warp_pool(next, 2 * G * nz, task);
    else
        for (int e = tid; e < 2 * G * nz; e += nth) task(e);
}

// WENO-5 (Jiang & Shu) faces in difference form, along a run of faces.
// With the upwind stencil v0..v4 (face between v2 and v3) and first
// differences d_i = v_{i+1} - v_i:
//   q0 - v2 = (5 d1 - 2 d0)/6,  q1 - v2 = (d1 + 2 d2)/6,  q2 - v2 = (4 d2 - d3)/6,
//   4 beta_r = 13/3 t_r^2 + s_r^2 with second differences t_0 = d1 - d0,
//   t_1 = d2 - d1, t_2 = d3 - d2 and s_0 = 3 d1 - d0, s_1 = -(d1 + d2),
//   s_2 = d3 - 3 d2,
// and the face value v2 + sum_r w_r (q_r - v2), w_r = a_r / sum a with
// a_r = d_r prod_{s != r} e_s^2, e_s = 4 (eps + beta_s) (the common factor 4
// cancels; one division per face).  Along a run the differences and the
// t-terms of each cell are formed once and shared by the faces that use
// them.  For xi_k < 0 the stencil is mirrored and the run is walked from its
// last face down, so that the new value always enters at v4.
template <typename R>
struct Weno5Run {
    R v2, v3, v4, d0, d1, d2, d3, u0, u1, u2;   // u_r = 13/3 t_r^2 + 4 eps
    R eps4;
    __device__ __forceinline__ R tterm(R t) const { return fma(R(13.0 / 3.0) * t, t, eps4); }
    __device__ __forceinline__ void start(R w0, R w1, R w2, R w3, R w4, R eps) {
        eps4 = R(4) * eps;
        v2 = w2;
        v3 = w3;
        v4 = w4;
        d0 = w1 - w0;
        d1 = w2 - w1;
        d2 = w3 - w2;
        d3 = w4 - w3;
        u0 = tterm(d1 - d0);
        u1 = tterm(d2 - d1);
        u2 = tterm(d3 - d2);
    }
    __device__ __forceinline__ R face() const {
        const R s0 = fma(R(3), d1, -d0), s1 = d1 + d2, s2 = fma(R(-3), d2, d3);
        const R e0 = fma(s0, s0, u0), e1 = fma(s1, s1, u1), e2 = fma(s2, s2, u2);
        const R E0 = e0 * e0, E1 = e1 * e1, E2 = e2 * e2;
        const R a0 = E1 * E2, a1 = E0 * E2, a2 = E0 * E1;
        // linear weights 0.1, 0.6, 0.3 folded into the candidate corrections
        // (0.2 d2 shared by c1 and c2)
        const R c0 = fma(R(5.0 / 60.0), d1, R(-2.0 / 60.0) * d0);
        const R p2 = R(0.2) * d2;
        const R c1 = fma(R(0.1), d1, p2);
        const R c2 = fma(R(-0.05), d3, p2);
        const R num = fma(a0, c0, fma(a1, c1, a2 * c2));
        const R den = fma(R(0.1), a0, fma(R(0.6), a1, R(0.3) * a2));
        R q;
        // FP32: the fast reciprocal-based quotient (2 ulp) is far inside the
        // FP32 variant's error budget; FP64: the Newton-refined reciprocal of
        // div_face (2^-46), cheaper on this part's FP64 pipe than the IEEE
        // division
        if constexpr (std::is_same<R, float>::value) q = __fdividef(num, den);
        else q = div_face(num, den);
        return v2 + q;
    }
    __device__ __forceinline__ void shift(R w5) {
        const R d4 = w5 - v4;
        u0 = u1;
        u1 = u2;
        u2 = tterm(d4 - d3);
        d0 = d1;
        d1 = d2;
        d2 = d3;
        d3 = d4;
        v2 = v3;
        v3 = v4;
        v4 = w5;
    }
};

// Phase 3c: face values h_{i-1/2} for faces f = 0..nz (face f lies between
// tile nodes f-1 and f), upwind by the sign of xi_k; runs of kRun faces per
// thread, consecutive threads on consecutive velocity rows (the row stride
// Z + 6 keeps their shared-memory reads apart), the walk direction chosen by
// index arithmetic so that threads of both signs run the same instructions.
// At xi_k = 0 the face values are formed as for xi_k > 0 and then multiplied
// by xi_k = 0 in the flux difference.
constexpr int kRun = 4;
template <typename R>
__device__ void faces(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z, int tid, int nth) {
    const int Q = sd.Q, W = Z + 6, nf = it.nz + 1, rows = 2 * Q;
    const int nruns = (nf + kRun - 1) / kRun;
    const R* xi = s.Vr;
    const R eps = slab_weno_eps<R>(sd);
    for (int e = tid; e < rows * nruns; e += nth) {
        const int r = e % rows, run = e / rows;
        const int k = r % Q;
        const int fa = run * kRun, n = min(kRun, nf - fa), fl = fa + n - 1;
        const bool pos = xi[k] >= R(0);
        const int dir = pos ? 1 : -1, f0 = pos ? fa : fl;
        // x > 0: face f uses h[f .. f+4], walked up; x < 0: h[f+5 .. f+1], walked down
        const R* hb = s.F + (size_t)r * W + (pos ? fa : fl + 5);
        R* out = s.Face + (size_t)r * (Z + 1);
        Weno5Run<R> w;
        w.start(hb[0], hb[dir], hb[2 * dir], hb[3 * dir], hb[4 * dir], eps);
#pragma unroll
        for (int q = 0; q < kRun; ++q) {
            if (q >= n) break;
            out[f0 + dir * q] = w.face();
            if (q + 1 < n) w.shift(hb[dir * (q + 5)]);
        }
    }
}

// ---------------------------------------------------------------------------
// WENO-5 faces of an FP64 state, split between the pipes.  The FP64 pipe of
// this part takes a warp instruction per scheduler every 64 cycles, the FP32
// pipe one per cycle.  With p = a_0 - a_1, q = a_2 - a_1 and the differences
// dd_0 = t_1 - t_0, dd_1 = t_2 - t_1 (third differences of h) the face of
// Weno5Run is
//   v2 + (-2 d0 + 11 d1 + 24 d2 - 3 d3) / 60                 (linear weights)
//      + (p (dd_1 - 6 dd_0) + q (2 dd_0 - 7 dd_1)) / (20 (a_0 + 6 a_1 + 3 a_2)),
// an identity.  The first line and the e_r are FP64; the rest of the second,
// which vanishes with the third differences, is double-float arithmetic on
// the FP32 pipe (pairs hi + lo from the e_r and t_r; normalised products and
// sums, about 2^-47 each).  17 FP64 operations a face, with its share of a
// cell's, instead of 31.
// The error of a right-hand side against 80-bit arithmetic, by that of the FP64
// form: 0.87 .. 0.93 on smooth profiles (the FP64 quotient is good to 2^-46 of the
// whole difference), 0.97 at grid-scale noise of 1 % of every value, 1.0 at 3 %,
// 1.2 .. 1.3 at 30 %, 1.2 .. 1.8 on slabs of density jumps (there the FP64 form adds
// next to nothing to v2, this one the difference of two parts of the jump's size); a step's
// error, 1.2e-16, is the same in all of these.  Stage of 4096 x 32: 50.6 -> 46.2
// us, of 65536 x 24 (tile 32): 520 -> 439 us.
//
// The e_r are scaled by a power of two to max(e_r) in [1, 2), so that the a_r
// do not overflow whatever the size of the state or of eps.  The divisor is of
// the square of the second largest e_r: beside a jump two of them may stay at
// 4 eps, and where they are small against the third their products leave the
// range in which a pair holds both its halves (from 2^-36 of the largest on the
// quotient loses digits, from 2^-75 on it is 0/0).  The pairs are cut before they
// are scaled, and a value below 2^-74 keeps its upper half alone: with eps and
// differences that small the weights would have 24 bits (faces of grid-scale noise
// of 1e-12 with eps = 1e-32: 6e-8 of it instead of 2e-14).  So a face takes the
// FP64 form unless its second largest e_r is above kSplitRatio of the largest and
// above kSplitLeast (a third one below 2^-74 then weighs less than 2^-14 of
// that, squared), and the largest is in the float range; at the default eps =
// 1e-6 that begins at differences of about 20 between neighbouring nodes, which
// a slab of sigma = 1 does not hold.
// ---------------------------------------------------------------------------
struct dfl {
    float h, l;
};
__device__ __forceinline__ dfl dfl_of(double x) {
    const float2 p = df_split(x);
    return {p.x, p.y};
}
__device__ __forceinline__ dfl dfl_norm(float h, float l) {
    const float s = __fadd_rn(h, l);
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
// sums (Knuth's TwoSum, low parts folded in), not normalised
__device__ __forceinline__ dfl dfl_add(dfl a, dfl b) {
    const float s = __fadd_rn(a.h, b.h), bb = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
    return {s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ dfl dfl_sub(dfl a, dfl b) {
    const float s = __fsub_rn(a.h, b.h), bb = __fsub_rn(s, a.h);
    const float e = __fsub_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fadd_rn(b.h, bb));
    return {s, __fadd_rn(e, __fsub_rn(a.l, b.l))};
}
__device__ __forceinline__ dfl dfl_norm(dfl a) { return dfl_norm(a.h, a.l); }
// products (the FMA's TwoProduct and all cross terms), normalised
__device__ __forceinline__ dfl dfl_mul(dfl a, dfl b) {
    const float p = __fmul_rn(a.h, b.h);
    return dfl_norm(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.l, __fmaf_rn(a.h, b.h, -p)))));
}
__device__ __forceinline__ dfl dfl_sqr(dfl a) {
    const float p = __fmul_rn(a.h, a.h);
    return dfl_norm(p, __fmaf_rn(__fadd_rn(a.h, a.h), a.l, __fmaf_rn(a.l, a.l, __fmaf_rn(a.h, a.h, -p))));
}
// times a small integer, not normalised; times a power of two
__device__ __forceinline__ dfl dfl_muli(dfl a, float b) {
    const float p = __fmul_rn(a.h, b);
    return {p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p))};
}
__device__ __forceinline__ dfl dfl_scale(dfl a, float b) { return {__fmul_rn(a.h, b), __fmul_rn(a.l, b)}; }
__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

constexpr float kSplitRatio = 2.33e-10f;   // 2^-32
constexpr float kSplitLeast = 1e-18f;

// The face of Weno5Run from its differences, in FP64 (the range fallback).
static __device__ __noinline__ double weno5_face_f64(double v2, double d0, double d1, double d2, double d3, double eps) {
    Weno5Run<double> w;
    w.v2 = v2;
    w.eps4 = 4.0 * eps;
    w.d0 = d0;
    w.d1 = d1;
    w.d2 = d2;
    w.d3 = d3;
    w.u0 = w.tterm(d1 - d0);
    w.u1 = w.tterm(d2 - d1);
    w.u2 = w.tterm(d3 - d2);
    return w.face();
}

// The run of Weno5Run on the split form.
struct Weno5Split {
    double v2, v3, v4, d0, d1, d2, d3, u0, u1, u2, eps4;   // u_r = 13/3 t_r^2 + 4 eps
    dfl T2, dd0, dd1;                                      // T2: t_2 as a pair
    __device__ __forceinline__ double tterm(double t) const { return fma((13.0 / 3.0) * t, t, eps4); }
    __device__ __forceinline__ void start(double w0, double w1, double w2, double w3, double w4, double eps) {
        eps4 = 4.0 * eps;
        v2 = w2;
        v3 = w3;
        v4 = w4;
        d0 = w1 - w0;
        d1 = w2 - w1;
        d2 = w3 - w2;
        d3 = w4 - w3;
        const double t0 = d1 - d0, t1 = d2 - d1, t2 = d3 - d2;
        u0 = tterm(t0);
        u1 = tterm(t1);
        u2 = tterm(t2);
        const dfl T0 = dfl_of(t0), T1 = dfl_of(t1);
        T2 = dfl_of(t2);
        dd0 = dfl_sub(T1, T0);
        dd1 = dfl_sub(T2, T1);
    }
    __device__ __forceinline__ double face(double eps) const {
        const double s0 = fma(3.0, d1, -d0), s1 = d1 + d2, s2 = fma(-3.0, d2, d3);
        dfl e0 = dfl_of(fma(s0, s0, u0)), e1 = dfl_of(fma(s1, s1, u1)), e2 = dfl_of(fma(s2, s2, u2));
        const float m = fmaxf(e0.h, fmaxf(e1.h, e2.h));
        const float mid = fmaxf(fminf(e0.h, e1.h), fminf(fmaxf(e0.h, e1.h), e2.h));
        if (!(m < 1e37f && mid > kSplitRatio * m && mid > kSplitLeast)) return weno5_face_f64(v2, d0, d1, d2, d3, eps);
        const float sc = __int_as_float(0x7f000000 - (__float_as_int(m) & 0x7f800000));   // 2^-exponent(m)
        e0 = dfl_scale(e0, sc);
        e1 = dfl_scale(e1, sc);
        e2 = dfl_scale(e2, sc);
        const dfl E0 = dfl_sqr(e0), E1 = dfl_sqr(e1), E2 = dfl_sqr(e2);
        const dfl a0 = dfl_mul(E1, E2), a1 = dfl_mul(E0, E2), a2 = dfl_mul(E0, E1);
        const dfl p = dfl_norm(dfl_sub(a0, a1)), q = dfl_norm(dfl_sub(a2, a1));
        const dfl A = dfl_norm(dfl_sub(dd1, dfl_muli(dd0, 6.f)));
        const dfl B = dfl_norm(dfl_sub(dfl_scale(dd0, 2.f), dfl_muli(dd1, 7.f)));
        const dfl num = dfl_norm(dfl_add(dfl_mul(p, A), dfl_mul(q, B)));
        const dfl den = dfl_norm(dfl_add(a0, dfl_add(dfl_muli(a1, 6.f), dfl_muli(a2, 3.f))));
        const float r = rcp_ftz(den.h);
        const float q1 = __fmul_rn(num.h, r);
        const float q2 = __fmul_rn(__fmaf_rn(-q1, den.l, __fadd_rn(__fmaf_rn(-q1, den.h, num.h), num.l)), r);
        const double lin = fma(24.0 / 60.0, d2, fma(11.0 / 60.0, d1, fma(-3.0 / 60.0, d3, (-2.0 / 60.0) * d0)));
        return v2 + fma(0.05, f2d_bits(q1) + f2d_bits(q2), lin);
    }
    __device__ __forceinline__ void shift(double w5) {
        const double d4 = w5 - v4, t = d4 - d3;
        d0 = d1;
        d1 = d2;
        d2 = d3;
        d3 = d4;
        u0 = u1;
        u1 = u2;
        u2 = tterm(t);
        const dfl T = dfl_of(t);
        dd0 = dd1;
        dd1 = dfl_sub(T, T2);
        T2 = T;
        v2 = v3;
        v3 = v4;
        v4 = w5;
    }
};

// faces() of an FP64 state: the same runs and walk, the split form, taken by
// whole warps from the pool `next`.
__device__ inline void faces_split(const SlabDesc& sd, const WorkItem& it, const Smem<double>& s, int Z, int* next) {
    const int Q = sd.Q, W = Z + 6, nf = it.nz + 1, rows = 2 * Q;
    const int nruns = (nf + kRun - 1) / kRun;
    const double* xi = s.Vp;
    warp_pool(next, rows * nruns, [&](int e) {
        const int r = e % rows, run = e / rows;
        const int k = r % Q;
        const int fa = run * kRun, n = min(kRun, nf - fa), fl = fa + n - 1;
        const bool pos = __double_as_longlong(xi[k]) >= 0 || !nonzero(xi[k]);
        const int dir = pos ? 1 : -1, f0 = pos ? fa : fl;
        const double* hb = s.F + (size_t)r * W + (pos ? fa : fl + 5);
        double* out = s.Face + (size_t)r * (Z + 1);
        Weno5Split w;
        w.start(hb[0], hb[dir], hb[2 * dir], hb[3 * dir], hb[4 * dir], sd.weno_eps);
#pragma unroll 1
        for (int q = 0;; ++q) {
            out[f0 + dir * q] = w.face(sd.weno_eps);
            if (q + 1 >= n) break;
            w.shift(hb[dir * (q + 5)]);
        }
    });
}

// ---------------------------------------------------------------------------
// Double-float arithmetic of the FP64_DF faces (every operation normalised): a
// value is an unevaluated pair hi + lo of floats (about 48 significant bits).  Addition is Knuth's
// TwoSum with the low parts folded in and one renormalisation (Dekker's
// FastTwoSum); multiplication is the FMA TwoProduct with the cross terms;
// the quotient takes the float reciprocal of the divisor's head and two
// remainder corrections (each adds ~24 bits).  __fadd_rn / __fmul_rn keep
// the compiler from contracting the error-free transformations.
// ---------------------------------------------------------------------------
__device__ __forceinline__ dfl dfn_of(double x) {
    const float2 p = df_split(x);
    return {p.x, p.y};
}
__device__ __forceinline__ dfl dfn_add(dfl a, dfl b) {
    const float s = __fadd_rn(a.h, b.h), bb = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
    const float t = __fadd_rn(e, __fadd_rn(a.l, b.l));
    const float h = __fadd_rn(s, t);
    return {h, __fsub_rn(t, __fsub_rn(h, s))};
}
__device__ __forceinline__ dfl dfn_sub(dfl a, dfl b) { return dfn_add(a, {-b.h, -b.l}); }
__device__ __forceinline__ dfl dfn_mul(dfl a, dfl b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    const float h = __fadd_rn(p, e);
    return {h, __fsub_rn(e, __fsub_rn(h, p))};
}
// times a float (exact small integers such as 3)
__device__ __forceinline__ dfl dfn_mulf(dfl a, float b) {
    const float p = __fmul_rn(a.h, b);
    float e = fmaf(a.h, b, -p);
    e = fmaf(a.l, b, e);
    const float h = __fadd_rn(p, e);
    return {h, __fsub_rn(e, __fsub_rn(h, p))};
}
__device__ __forceinline__ dfl dfn_div(dfl a, dfl b) {
    const float r = __frcp_rn(b.h);
    const float q1 = __fmul_rn(a.h, r);
    const dfl r1 = dfn_sub(a, dfn_mulf(b, q1));
    const float q2 = __fmul_rn(r1.h, r);
    const dfl r2 = dfn_sub(r1, dfn_mulf(b, q2));
    const float q3 = __fmul_rn(r2.h, r);
    const float s = __fadd_rn(q1, q2), bb = __fsub_rn(s, q1);
    const float e = __fadd_rn(__fsub_rn(q1, __fsub_rn(s, bb)), __fsub_rn(q2, bb));
    return dfn_add({s, e}, {q3, 0.0f});
}
// the constants of the difference-form WENO-5 face as pairs
__device__ __forceinline__ dfl dfn_const(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}

// The difference-form WENO-5 run of Weno5Run in double-float arithmetic.
struct Weno5RunDF {
    dfl v2, v3, v4, d0, d1, d2, d3, u0, u1, u2;
    dfl eps4, k133;
    __device__ __forceinline__ dfl tterm(dfl t) const { return dfn_add(dfn_mul(dfn_mul(k133, t), t), eps4); }
    // eps4 = 4 eps as a pair (formed once per thread by the caller)
    __device__ __forceinline__ void start(double w0, double w1, double w2, double w3, double w4, dfl e4) {
        eps4 = e4;
        k133 = dfn_const(13.0 / 3.0);
        const dfl a0 = dfn_of(w0), a1 = dfn_of(w1);
        v2 = dfn_of(w2);
        v3 = dfn_of(w3);
        v4 = dfn_of(w4);
        d0 = dfn_sub(a1, a0);
        d1 = dfn_sub(v2, a1);
        d2 = dfn_sub(v3, v2);
        d3 = dfn_sub(v4, v3);
        u0 = tterm(dfn_sub(d1, d0));
        u1 = tterm(dfn_sub(d2, d1));
        u2 = tterm(dfn_sub(d3, d2));
    }
    __device__ __forceinline__ double face() const {
        const dfl s0 = dfn_sub(dfn_mulf(d1, 3.0f), d0), s1 = dfn_add(d1, d2), s2 = dfn_sub(d3, dfn_mulf(d2, 3.0f));
        const dfl e0 = dfn_add(dfn_mul(s0, s0), u0), e1 = dfn_add(dfn_mul(s1, s1), u1), e2 = dfn_add(dfn_mul(s2, s2), u2);
        const dfl E0 = dfn_mul(e0, e0), E1 = dfn_mul(e1, e1), E2 = dfn_mul(e2, e2);
        const dfl a0 = dfn_mul(E1, E2), a1 = dfn_mul(E0, E2), a2 = dfn_mul(E0, E1);
        const dfl c0 = dfn_sub(dfn_mul(dfn_const(5.0 / 60.0), d1), dfn_mul(dfn_const(2.0 / 60.0), d0));
        const dfl c1 = dfn_add(dfn_mul(dfn_const(0.2), d2), dfn_mul(dfn_const(0.1), d1));
        const dfl c2 = dfn_sub(dfn_mul(dfn_const(0.2), d2), dfn_mul(dfn_const(0.05), d3));
        const dfl num = dfn_add(dfn_add(dfn_mul(a0, c0), dfn_mul(a1, c1)), dfn_mul(a2, c2));
        const dfl den = dfn_add(dfn_add(dfn_mul(dfn_const(0.1), a0), dfn_mul(dfn_const(0.6), a1)),
                                dfn_mul(dfn_const(0.3), a2));
        const dfl f = dfn_add(v2, dfn_div(num, den));
        return f2d_bits(f.h) + f2d_bits(f.l);
    }
    __device__ __forceinline__ void shift(double w5) {
        const dfl v5 = dfn_of(w5);
        const dfl d4 = dfn_sub(v5, v4);
        u0 = u1;
        u1 = u2;
        u2 = tterm(dfn_sub(d4, d3));
        d0 = d1;
        d1 = d2;
        d2 = d3;
        d3 = d4;
        v2 = v3;
        v3 = v4;
        v4 = v5;
    }
};

// faces() of the FP64_DF kernel: the same runs and walk, the face values in
// double-float arithmetic on the FP32 pipe, stored as FP64.
__device__ inline void faces_df(const SlabDesc& sd, const WorkItem& it, const Smem<double>& s, int Z, int* next) {
    const int Q = sd.Q, W = Z + 6, nf = it.nz + 1, rows = 2 * Q;
    const int nruns = (nf + kRun - 1) / kRun;
    const double* xi = s.Vp;
    const dfl eps4 = dfn_const(4.0 * sd.weno_eps);
    warp_pool(next, rows * nruns, [&](int e) {
        const int r = e % rows, run = e / rows;
        const int k = r % Q;
        const int fa = run * kRun, n = min(kRun, nf - fa), fl = fa + n - 1;
        const bool pos = xi[k] >= 0.0;
        const int dir = pos ? 1 : -1, f0 = pos ? fa : fl;
        const double* hb = s.F + (size_t)r * W + (pos ? fa : fl + 5);
        double* out = s.Face + (size_t)r * (Z + 1);
        Weno5RunDF w;
        w.start(hb[0], hb[dir], hb[2 * dir], hb[3 * dir], hb[4 * dir], eps4);
#pragma unroll 1
        for (int q = 0;; ++q) {
            out[f0 + dir * q] = w.face();
            if (q + 1 >= n) break;
            w.shift(hb[dir * (q + 5)]);
        }
    });
}

// Raw moment sums of one node from a column h[k * stride] (k < Q).  The
// conserved moments (S0, S1, S2 of F and G0) are summed in FP64; S3 and G1
// (heat flux) in R.  The velocity powers come from xp = [xi, xi^2, xi^3]
// (FP64) and xr = [xi, xi^3] (R).
//
// FP64 state: four interleaved chains over k, joined as ((a0 + a1) + (a2 + a3)).
//
// FP32 state: the pair form.  Velocity j < H = (Q+1)/2 and its mirror Q-1-j
// (xi_{Q-1-j} = -xi_j) give one term per pair, with a = h_j, b = h_{Q-1-j}
// (b = 0 for the middle velocity of an odd Q):
//   S0, G0: a + b;   S1: xi_j (a - b);   S2: xi_j^2 (a + b);
//   S3: xi_j^3 (a - b);   G1: xi_j (a - b),
// the FP64 terms from floats widened exactly by bit surgery.  The pairs 2g
// and 2g+1 form group g < G = (H+1)/2 (term(2g) + term(2g+1); a last lone
// pair alone), and the G group terms are summed in four chains over g mod
// 4, joined as ((c0 + c1) + (c2 + c3)).  Every operation is an explicitly
// rounded one, so the stage kernel, which forms the group terms where it
// writes the new state (pair_terms_f32) and sums them afterwards
// (sum_pair_terms), gets the same bits as a sum formed here in one pass.
__device__ __forceinline__ bool moment_is_f64(int which) {
    return which == MOM_S0 || which == MOM_S1 || which == MOM_S2 || which == MOM_G0;
}

__device__ __forceinline__ double pair_term_f64(int which, int j, int Q, double a, double b,
                                                const double* __restrict__ xp) {
    if (which == MOM_S0 || which == MOM_G0) return __dadd_rn(a, b);
    if (which == MOM_S1) return __dmul_rn(xp[j], __dsub_rn(a, b));
    return __dmul_rn(xp[Q + j], __dadd_rn(a, b));                    // S2
}

__device__ __forceinline__ float pair_term_f32(int which, int j, int Q, float a, float b,
                                               const float* __restrict__ xr) {
    return __fmul_rn(which == MOM_S3 ? xr[Q + j] : xr[j], __fsub_rn(a, b));   // S3, G1
}

template <typename T>
__device__ __forceinline__ T add_rn(T a, T b) {
    if constexpr (std::is_same<T, float>::value) return __fadd_rn(a, b);
    else return __dadd_rn(a, b);
}

// Sum of the n terms term(j) in four chains over j mod 4.
template <typename T, typename F>
__device__ __forceinline__ T sum_chains4(int n, F term) {
    T c0 = 0, c1 = 0, c2 = 0, c3 = 0;
    int j = 0;
    for (; j + 3 < n; j += 4) {
        c0 = add_rn(c0, term(j));
        c1 = add_rn(c1, term(j + 1));
        c2 = add_rn(c2, term(j + 2));
        c3 = add_rn(c3, term(j + 3));
    }
    if (j < n) c0 = add_rn(c0, term(j));
    if (j + 1 < n) c1 = add_rn(c1, term(j + 1));
    if (j + 2 < n) c2 = add_rn(c2, term(j + 2));
    return add_rn(add_rn(c0, c1), add_rn(c2, c3));
}

// Sum of n stored terms v[j * stride], in the order of sum_chains4.
template <typename T>
__device__ __forceinline__ T sum_pair_terms(const T* v, int n, long long stride) {
    return sum_chains4<T>(n, [&](int j) { return v[j * stride]; });
}

template <typename R>
__device__ __forceinline__ double moment_sum(int which, int Q, const R* h, long long stride,
                                             const double* __restrict__ xp, const R* __restrict__ xr) {
    const int p = (which >= MOM_G0) ? which - MOM_G0 : which;   // power of xi
    if constexpr (std::is_same<R, double>::value) {
        const double* w = xp + (p > 0 ? p - 1 : 0) * Q;
        auto acc = [&](double a, int k) { return p == 0 ? a + h[k * stride] : fma(w[k], h[k * stride], a); };
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int k = 0;
        for (; k + 3 < Q; k += 4) {
            a0 = acc(a0, k);
            a1 = acc(a1, k + 1);
            a2 = acc(a2, k + 2);
            a3 = acc(a3, k + 3);
        }
        for (; k < Q; ++k) a0 = acc(a0, k);
        return (a0 + a1) + (a2 + a3);
    } else {
        const int H = (Q + 1) / 2, G = (H + 1) / 2;
        auto ha = [&](int j) { return h[j * stride]; };
        auto hb = [&](int j) { return (Q - 1 - j != j) ? h[(Q - 1 - j) * stride] : 0.f; };
        if (moment_is_f64(which)) {
            auto term = [&](int j) { return pair_term_f64(which, j, Q, f2d_bits(ha(j)), f2d_bits(hb(j)), xp); };
            return sum_chains4<double>(
                G, [&](int g) { return 2 * g + 1 < H ? __dadd_rn(term(2 * g), term(2 * g + 1)) : term(2 * g); });
        }
        auto term = [&](int j) { return pair_term_f32(which, j, Q, ha(j), hb(j), xr); };
        return f2d_bits(sum_chains4<float>(
            G, [&](int g) { return 2 * g + 1 < H ? __fadd_rn(term(2 * g), term(2 * g + 1)) : term(2 * g); }));
    }
}

// The group terms of the four FP64 and two R moment sums for group g of
// one node t and distribution d: pairs j0 = 2g and j1 = 2g+1 (two: j1 < H),
// from the new state's values a0, b0 (velocity j0 and its mirror) and a1, b1;
// b is 0 for a middle velocity.  Into t64[slot][g * Z + t] (S0, S1, S2, G0)
// and t32[slot][g * Z + t] (S3, G1), slot blocks of G Z values.
__device__ __forceinline__ void pair_terms_f32(int d, int g, bool two, int t, int Q, int Z, float a0, float b0,
                                               float a1, float b1, const double* __restrict__ xp,
                                               const float* __restrict__ xr, double* t64, float* t32) {
    const int j0 = 2 * g, j1 = 2 * g + 1;
    const size_t o = (size_t)g * Z + t, blk = (size_t)pair_groups(Q) * Z;
    const double wa0 = f2d_bits(a0), wb0 = f2d_bits(b0), wa1 = f2d_bits(a1), wb1 = f2d_bits(b1);
    auto t8 = [&](int which) {
        const double x = pair_term_f64(which, j0, Q, wa0, wb0, xp);
        return two ? __dadd_rn(x, pair_term_f64(which, j1, Q, wa1, wb1, xp)) : x;
    };
    auto t4 = [&](int which) {
        const float x = pair_term_f32(which, j0, Q, a0, b0, xr);
        return two ? __fadd_rn(x, pair_term_f32(which, j1, Q, a1, b1, xr)) : x;
    };
    if (d == 0) {
        t64[o] = t8(MOM_S0);
        t64[blk + o] = t8(MOM_S1);
        t64[2 * blk + o] = t8(MOM_S2);
        t32[o] = t4(MOM_S3);
    } else {
        t64[3 * blk + o] = t8(MOM_G0);
        t32[blk + o] = t4(MOM_G1);
    }
}

// Velocity powers of moment_sum from the tables xi (FP64) and rxi (R).
template <typename R>
__device__ __forceinline__ void velocity_powers(int Q, const double* __restrict__ xi, const R* __restrict__ rxi,
                                                double* xp, R* xr, int tid, int nth) {
    for (int k = tid; k < Q; k += nth) {
        const double x = xi[k];
        xp[k] = x;
        xp[Q + k] = x * x;
        xp[2 * Q + k] = x * x * x;
        const R y = rxi[k];
        xr[k] = y;
        xr[Q + k] = y * y * y;
    }
}

// Raw moment sums of the tile held in s.F (columns 3 .. nz+2), from velocity
// powers staged in shared memory (xp = [xi, xi^2, xi^3] FP64, xr = [xi, xi^3]
// in R).  Called by all threads once the tile's velocity work is done: one
// sum per warp, lanes on nodes, where the tile allows.
template <typename R>
__device__ void tile_moment_sums_staged(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z,
                                        const double* xp, const R* xr, double* __restrict__ mom_out, long long NN) {
    const int Q = sd.Q, W = Z + 6, nz = it.nz;
    if constexpr (std::is_same<R, double>::value) {
        // small tiles: the four chains of a sum (moment_sum) on four lanes,
        // joined by shuffles in the same order
        if (nz <= 8 && blockDim.x >= 32 * kNumMoments) {
            const int which = threadIdx.x >> 5, t = (threadIdx.x & 31) >> 2, c = threadIdx.x & 3;
            if (which < kNumMoments) {
                const int d = which >= MOM_G0 ? 1 : 0, p = (which >= MOM_G0) ? which - MOM_G0 : which;
                const double* h = s.F + (size_t)d * Q * W + min(t, nz - 1) + 3;
                const double* w = xp + (p > 0 ? p - 1 : 0) * Q;
                double a = 0.0;
                auto acc = [&](int k) { a = p == 0 ? a + h[k * W] : fma(w[k], h[k * W], a); };
                const int Q4 = Q & ~3;
                for (int k = c; k < Q4; k += 4) acc(k);
                if (c == 0)
                    for (int k = Q4; k < Q; ++k) acc(k);
                a += __shfl_xor_sync(0xffffffffu, a, 1);
                a += __shfl_xor_sync(0xffffffffu, a, 2);
                if (c == 0 && t < nz) mom_out[which * NN + sd.node_off + it.i0 + t] = a;
            }
            return;
        }
    }
    if (nz <= 32 && blockDim.x >= 32 * kNumMoments) {
        const int which = threadIdx.x >> 5, t = threadIdx.x & 31;
        if (which < kNumMoments && t < nz) {
            const int d = which >= MOM_G0 ? 1 : 0;
            const R* h = s.F + (size_t)d * Q * W + t + 3;
            mom_out[which * NN + sd.node_off + it.i0 + t] = moment_sum<R>(which, Q, h, W, xp, xr);
        }
        return;
    }
    for (int e = threadIdx.x; e < kNumMoments * nz; e += blockDim.x) {
        int t = e % nz, which = e / nz;
        int d = which >= MOM_G0 ? 1 : 0;
        const R* h = s.F + (size_t)d * Q * W + t + 3;
        mom_out[which * NN + sd.node_off + it.i0 + t] = moment_sum<R>(which, Q, h, W, xp, xr);
    }
}

// The same with the velocity powers formed here first, in the (then free)
// table block s.P / s.S (5 Q values).
template <typename R>
__device__ void tile_moment_sums(const SlabDesc& sd, const WorkItem& it, const Smem<R>& s, int Z,
                                 const double* __restrict__ xi, const R* __restrict__ rxi,
                                 double* __restrict__ mom_out, long long NN) {
    const int Q = sd.Q;
    double* xp = reinterpret_cast<double*>(s.P);
    R* xr = reinterpret_cast<R*>(xp + 3 * Q);
    velocity_powers<R>(Q, xi, rxi, xp, xr, threadIdx.x, blockDim.x);
    __syncthreads();
    tile_moment_sums_staged<R>(sd, it, s, Z, xp, xr, mom_out, NN);
}

}  // namespace evfdlb
