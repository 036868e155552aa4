// Per-voxel constitutive routines shared by the forward Newton and the adjoint kernels
// (Sec. 2.1 Eqs. HookeLaw / PlasticRate with the power-law flow rule, and with the Ma-Roters flow rule of
// Sec. 2.2 Eq. FlowRule).
#pragma once
#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "powtab.cuh"

namespace evp {

template <typename T> __device__ __forceinline__ T dsqrt(T x) { return sqrt(x); }
__device__ __forceinline__ double dsqrt(double x) { return __dsqrt_rn(x); }
template <typename T> __device__ __forceinline__ T drcp(T x) { return (T)1 / x; }
__device__ __forceinline__ double drcp(double x) { return __drcp_rn(x); }

// |x|^(n-1) for the power law; fast path for small integer n (exponentiation by squaring).
template <typename T> __device__ __forceinline__ T pow_nm1(T ax, const MatConst &mc) {
    if (mc.n_int == 10) {
        // the workloads' exponent: |x|^9 = |x| ((|x|^2)^2)^2, the very products the bit loop below forms for
        // e = 9 (its first factor 1 * |x| is exact), in 4 multiplications instead of 18 operations
        const T b2 = ax * ax, b4 = b2 * b2, b8 = b4 * b4;
        return ax * b8;
    }
    if (mc.n_int > 0) {
        // branch-free: the same products in the same order as the bit loop, over all six bits of
        // e <= 63 (selects instead of branches, so independent slip systems can be interleaved)
        const int e = mc.n_int - 1;
        T r = (T)1, b = ax;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            r = ((e >> k) & 1) ? r * b : r;
            b = b * b;
        }
        return r;
    }
    // FP32 kernels keep CUDA's pow. The branch is part of each of them, whichever exponent a run has, and its registers
    // cost the integer exponents: the 128^3 local solve takes 94.0 us an iteration at n = 10 with pow here and 97.8 us
    // with the table-driven power. Where the branch is taken pow is the slower one: at n = 10.37 an iteration's local
    // solve takes 4.80 ms with pow and 2.16 ms with the table.
    if constexpr (sizeof(T) == 4) return ax > (T)0 ? (T)pow((double)ax, mc.n - 1.0) : (T)0;
    else return ax > (T)0 ? (T)pow_tab((double)ax, mc.n - 1.0) : (T)0;
}

// Flow-rule constants in the arithmetic precision.
template <typename TA> __device__ __forceinline__ void flow_consts(const MatConst &mc, TA &dt, TA &g0, TA &nn) {
    if constexpr (sizeof(TA) == 4) { dt = mc.dt_f; g0 = mc.gdot0_f; nn = mc.n_f; }
    else { dt = mc.dt; g0 = mc.gdot0; nn = mc.n; }
}

// Packed lower-triangular index of (i, j), j <= i.
__host__ __device__ constexpr int pk(int i, int j) { return i * (i + 1) / 2 + j; }

// Per-grain tables: compliance rows (36 words) and Schmid vectors (12 x 6 words) per grain, each grain
// starting on a 16-byte boundary (144 g / 288 g bytes), for the FP32 local problems. They are read with
// 16-byte vector loads; the load instructions, not the bytes (the tables sit in L1), are what a
// per-voxel kernel issuing one load per word runs short of.
__device__ __forceinline__ void load_compliance(const float *__restrict__ S, float Sp[21]) {
    float full[36];
    const float4 *S4 = reinterpret_cast<const float4 *>(S);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float4 t = __ldg(S4 + k);
        full[4 * k] = t.x; full[4 * k + 1] = t.y; full[4 * k + 2] = t.z; full[4 * k + 3] = t.w;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) Sp[i * (i + 1) / 2 + j] = full[6 * i + j];
}
// Schmid vectors of slip systems 2p and 2p+1 (12 consecutive words, 16-byte aligned).
__device__ __forceinline__ void load_slip_pair(const float *__restrict__ M, int p, float m[12]) {
    const float4 *M4 = reinterpret_cast<const float4 *>(M + 12 * p);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float4 t = __ldg(M4 + k);
        m[4 * k] = t.x; m[4 * k + 1] = t.y; m[4 * k + 2] = t.z; m[4 * k + 3] = t.w;
    }
}

// ---- the crystal frame ----
// The FP64 local problems are solved in the axes of their crystal: the FP64 pipe (2 multiply-adds per clock and SM)
// bounds them, and there an evaluation takes about half the FP64 operations. The cubic compliance has three
// constants (Cubic) and a Schmid vector of the {111}<110> systems has four entries, +-1/sqrt6 on two normal
// components and +-1/sqrt12 on two shears (Mandel), so the 12 resolved stresses take 21 additions, the plastic strain
// another 28 and the tangent 24 before its scaling, where the sample-frame Schmid vectors take 72, 72 and 252
// multiply-adds. A solve adds three rotations of a symmetric tensor (51 operations each): trial strain and stress in,
// stress out. k_newton_df at 64^3: 373 us per fixed-point iteration, 512 with the sample-frame vectors.
// The FP32 problems stay in the sample frame: rotating the stress in FP32 adds a rounding of the stress itself, and
// the equilibrium residual of the converged FP32 field rose from 5.0e-7 to 7.5e-7 of its tolerance's 1e-6.
// The grain table holds kFrameWords words per grain: R (crystal -> sample, row-major) and a word of padding, which keeps
// each grain's words on a 16-byte boundary.
static_assert(kFrameWords % 2 == 0 && kFrameWords >= 9, "frames are read in 16-byte pairs");
__device__ __forceinline__ void load_frame(const double *__restrict__ R, double r[9]) {
    const double2 *R2 = reinterpret_cast<const double2 *>(R);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double2 t = __ldg(R2 + k);
        r[2 * k] = t.x; r[2 * k + 1] = t.y;
    }
    r[8] = __ldg(R + 8);
}
// out = Mandel(A^T X A) with X the symmetric tensor of Mandel vector x and A given by its entries a(i, j).
template <typename T, typename F> __device__ __forceinline__ void rotate_mandel(const T x[6], F a, T out[6]) {
    const T h = (T)0.70710678118654752440, q2 = (T)1.41421356237309504880;
    const T x23 = h * x[3], x13 = h * x[4], x12 = h * x[5];
    T b[3][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        b[0][j] = x[0] * a(0, j) + x12 * a(1, j) + x13 * a(2, j);
        b[1][j] = x12 * a(0, j) + x[1] * a(1, j) + x23 * a(2, j);
        b[2][j] = x13 * a(0, j) + x23 * a(1, j) + x[2] * a(2, j);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) out[i] = a(0, i) * b[0][i] + a(1, i) * b[1][i] + a(2, i) * b[2][i];
    out[3] = q2 * (a(0, 1) * b[0][2] + a(1, 1) * b[1][2] + a(2, 1) * b[2][2]);
    out[4] = q2 * (a(0, 0) * b[0][2] + a(1, 0) * b[1][2] + a(2, 0) * b[2][2]);
    out[5] = q2 * (a(0, 0) * b[0][1] + a(1, 0) * b[1][1] + a(2, 0) * b[2][1]);
}
template <typename T> __device__ __forceinline__ void to_crystal(const T r[9], const T x[6], T out[6]) {
    rotate_mandel(x, [&](int i, int j) { return r[3 * i + j]; }, out);
}
template <typename T> __device__ __forceinline__ void to_sample(const T r[9], const T x[6], T out[6]) {
    rotate_mandel(x, [&](int i, int j) { return r[3 * j + i]; }, out);
}

// One voxel's local problem: what evaluate needs of the crystal besides the flow rule. enter() takes the trial strain
// and the stress from the sample frame into the frame the problem is solved in, leave() takes the stress back.
template <typename TA> struct Problem;
template <> struct Problem<float> {   // sample frame: compliance (packed lower) and the grain's Schmid vectors
    float Sp[21];
    const float *M;
    __device__ __forceinline__ void init(const LocalTab<float> &t, int g) {
        load_compliance(t.S + 36 * (long)g, Sp);
        M = t.M + 72 * (long)g;
    }
    __device__ __forceinline__ void enter(float *, float *) const {}
    __device__ __forceinline__ void leave(float *) const {}
};
template <> struct Problem<double> {   // crystal frame
    Cubic<double> cu;
    const double *R;
    __device__ __forceinline__ void init(const LocalTab<double> &t, int g) {
        cu = t.cub;
        R = t.R + kFrameWords * (long)g;
    }
    __device__ __forceinline__ void enter(double etr[6], double sg[6]) const {
        double r[9], e[6], s[6];
        load_frame(R, r);
        to_crystal(r, etr, e);
        to_crystal(r, sg, s);
#pragma unroll
        for (int i = 0; i < 6; ++i) { etr[i] = e[i]; sg[i] = s[i]; }
    }
    __device__ __forceinline__ void leave(double sg[6]) const {
        double r[9], s[6];
        load_frame(R, r);
        to_sample(r, sg, s);
#pragma unroll
        for (int i = 0; i < 6; ++i) sg[i] = s[i];
    }
};

// Stored tangent factors (21 words per voxel): 16-byte vector planes, then one scalar plane for the last word.
// FP32: planes 0-4 are float4 (words 4k..4k+3), plane 5 is float (word 20); FP64: planes 0-9 are double2 (words
// 2k, 2k+1), plane 10 is double (word 20). Each plane holds N3 voxels, so a voxel's factors come in 5 (10)
// coalesced vector loads and one scalar load, with no padding words.
template <typename TS> __host__ __device__ constexpr int factor_words() { return 21; }
template <typename TS> __device__ __forceinline__ void load_factors(const TS *__restrict__ fac, long N3, long v, TS F[21]) {
    if constexpr (sizeof(TS) == 4) {
        const float4 *f4 = reinterpret_cast<const float4 *>(fac);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const float4 t = f4[k * N3 + v];
            F[4 * k] = t.x; F[4 * k + 1] = t.y; F[4 * k + 2] = t.z; F[4 * k + 3] = t.w;
        }
        F[20] = fac[20 * N3 + v];
    } else {
        const double2 *f2 = reinterpret_cast<const double2 *>(fac);
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            const double2 t = f2[k * N3 + v];
            F[2 * k] = t.x; F[2 * k + 1] = t.y;
        }
        F[20] = fac[20 * N3 + v];
    }
}
template <typename TS> __device__ __forceinline__ void store_factors(TS *__restrict__ fac, long N3, long v, const TS F[21]) {
    if constexpr (sizeof(TS) == 4) {
        float4 *f4 = reinterpret_cast<float4 *>(fac);
#pragma unroll
        for (int k = 0; k < 5; ++k) f4[k * N3 + v] = make_float4(F[4 * k], F[4 * k + 1], F[4 * k + 2], F[4 * k + 3]);
    } else {
        double2 *f2 = reinterpret_cast<double2 *>(fac);
#pragma unroll
        for (int k = 0; k < 10; ++k) f2[k * N3 + v] = make_double2(F[2 * k], F[2 * k + 1]);
    }
    fac[20 * N3 + v] = F[20];
}

// The same factors staged through shared memory: prefetch_factors starts asynchronous copies of this thread's 21
// words into its own slots (plane-major, blockDim.x threads per plane: the vector planes, then the scalar plane),
// prefetched_factors waits for this thread's copies and reads them. Only the issuing thread reads its slots, so no
// barrier is needed.
template <typename TS> __device__ __forceinline__ void prefetch_factors(const TS *__restrict__ fac, long N3, long v, TS *sh) {
    const int t = threadIdx.x, nt = blockDim.x;
    constexpr int W = sizeof(TS) == 4 ? 4 : 2, P = 20 / W;   // words per vector, vector planes
#pragma unroll
    for (int k = 0; k < P; ++k) {
        const unsigned sa = (unsigned)__cvta_generic_to_shared(sh + (k * nt + t) * W);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(fac + (k * N3 + v) * W) : "memory");
    }
    const unsigned sa = (unsigned)__cvta_generic_to_shared(sh + P * nt * W + t);
    if constexpr (sizeof(TS) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(fac + 20 * N3 + v) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(fac + 20 * N3 + v) : "memory");
}
template <typename TS> __device__ __forceinline__ void prefetched_factors(const TS *sh, TS F[21]) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    const int t = threadIdx.x, nt = blockDim.x;
    constexpr int W = sizeof(TS) == 4 ? 4 : 2, P = 20 / W;
    if constexpr (sizeof(TS) == 4) {
        const float4 *s4 = reinterpret_cast<const float4 *>(sh);
#pragma unroll
        for (int k = 0; k < P; ++k) {
            const float4 q = s4[k * nt + t];
            F[4 * k] = q.x; F[4 * k + 1] = q.y; F[4 * k + 2] = q.z; F[4 * k + 3] = q.w;
        }
    } else {
        const double2 *s2 = reinterpret_cast<const double2 *>(sh);
#pragma unroll
        for (int k = 0; k < P; ++k) {
            const double2 q = s2[k * nt + t];
            F[2 * k] = q.x; F[2 * k + 1] = q.y;
        }
    }
    F[20] = sh[P * nt * W + t];
}

// Residual r, tangent K (packed lower, in TK) and potential phi of a local problem at a stress.
template <typename TA, typename TK = TA> struct Eval {
    TA r[6];
    TK K[21];
    TA phi;
};

__device__ __forceinline__ void evaluate(const float Sp[21], const float *__restrict__ M, const float etr[6], float tauc,
                                         float inv_tc, const float sg[6], const MatConst &mc, Eval<float> &e) {
    float dt, g0, nn;
    flow_consts(mc, dt, g0, nn);
    float phi = 0.f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < 6; ++j) acc += Sp[i >= j ? pk(i, j) : pk(j, i)] * sg[j];
        e.r[i] = acc - etr[i];
        phi += sg[i] * (0.5f * acc - etr[i]);
    }
#pragma unroll
    for (int q = 0; q < 21; ++q) e.K[q] = Sp[q];
    const float cphi = dt * g0 * tauc / (nn + 1.f);
    const float cslope = dt * nn * g0 * inv_tc;
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
      float mm[12];
      load_slip_pair(M, p, mm);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float *m = mm + 6 * h;
        float tau = 0.f;
#pragma unroll
        for (int i = 0; i < 6; ++i) tau += m[i] * sg[i];
        const float x = tau * inv_tc;
        const float ax = fabs(x);
        const float p9 = pow_nm1(ax, mc);       // |x|^(n-1)
        const float p10 = p9 * ax;              // |x|^n
        const float gd = x < 0.f ? -g0 * p10 : g0 * p10;
        const float slope = cslope * p9;
        float sm[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            e.r[i] += dt * gd * m[i];
            sm[i] = slope * m[i];
        }
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) e.K[pk(i, j)] += sm[i] * m[j];
        phi += cphi * p10 * ax;
      }
    }
    e.phi = phi;
}


// ---- Ma-Roters flow rule (Sec. 2.2, Eq. FlowRule) ----
// gdot = A sinh((|tau| - tau_pass) / tau_cut) sign(tau) above the passing stress, A = ga tau_pass; its
// derivative A cosh(.) / tau_cut and the convex potential A tau_cut (cosh(.) - 1) (zero below). With
// u = expm1(x) and w = 1/(1+u) = exp(-x): sinh x = u (1+w)/2 and cosh x - 1 = u (1-w)/2, free of
// cancellation for small x; an overflowing x gives infinities that the line search rejects.
template <typename TA> struct FlowMR {
    const TA *__restrict__ tpi;   // (tau_pass, 1 / tau_cut) pairs, 12 x N3 (layout of MRPtr)
    long N3, v;
    TA tref;                      // stopping scale: min_a tau_pass^a
};
template <typename TA> __device__ __forceinline__ TA flow_ref(TA tauc) { return tauc; }
template <typename TA> __device__ __forceinline__ TA flow_ref(const FlowMR<TA> &f) { return f.tref; }
__device__ __forceinline__ float dexpm1(float x) { return expm1f(x); }
// 1/x rounded to nearest (FP32 reciprocal instruction with its IEEE fix-up) / FP64 division
__device__ __forceinline__ float rcp_fast(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_fast(double x) { return 1.0 / x; }
__device__ __forceinline__ double dexpm1(double x) { return expm1(x); }
template <typename TA> __device__ __forceinline__ TA mr_ga(const MatConst &mc) {
    if constexpr (sizeof(TA) == 4) return mc.mr_ga_f;
    else return mc.mr_ga;
}
template <typename TA>
__device__ __forceinline__ void mr_flow(TA tau, TA tp, TA itc, TA ga, TA &gd, TA &slope, TA &psi) {
    const TA x = (fabs(tau) - tp) * itc;
    if (x > (TA)0) {
        const TA u = dexpm1(x), w = rcp_fast(u + (TA)1), A = ga * tp;
        const TA sh = (TA)0.5 * u * ((TA)1 + w), chm1 = (TA)0.5 * u * ((TA)1 - w);
        gd = tau < (TA)0 ? -A * sh : A * sh;
        slope = A * ((TA)1 + chm1) * itc;
        psi = A * chm1 * rcp_fast(itc);   // the potential only steers the line search
    } else {
        gd = (TA)0; slope = (TA)0; psi = (TA)0;
    }
}
template <typename TA> __device__ __forceinline__ void mr_sys(const FlowMR<TA> &f, int a, TA &tp, TA &itc) {
    if constexpr (sizeof(TA) == 4) {
        const float2 t = __ldg(reinterpret_cast<const float2 *>(f.tpi) + (long)a * f.N3 + f.v);
        tp = t.x; itc = t.y;
    } else {
        const double2 t = __ldg(reinterpret_cast<const double2 *>(f.tpi) + (long)a * f.N3 + f.v);
        tp = t.x; itc = t.y;
    }
}

__device__ __forceinline__ void evaluate(const float Sp[21], const float *__restrict__ M, const float etr[6],
                                         const FlowMR<float> &f, float, const float sg[6], const MatConst &mc, Eval<float> &e) {
    float dt, g0, nn;
    flow_consts(mc, dt, g0, nn);
    const float ga = mr_ga<float>(mc);
    float phi = 0.f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < 6; ++j) acc += Sp[i >= j ? pk(i, j) : pk(j, i)] * sg[j];
        e.r[i] = acc - etr[i];
        phi += sg[i] * (0.5f * acc - etr[i]);
    }
#pragma unroll
    for (int q = 0; q < 21; ++q) e.K[q] = Sp[q];
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
      float mm[12];
      load_slip_pair(M, p, mm);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float *m = mm + 6 * h;
        float tau = 0.f;
#pragma unroll
        for (int i = 0; i < 6; ++i) tau += m[i] * sg[i];
        float tp, itc, gd, slope, psi;
        mr_sys(f, 2 * p + h, tp, itc);
        mr_flow(tau, tp, itc, ga, gd, slope, psi);
        float sm[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            e.r[i] += dt * gd * m[i];
            sm[i] = dt * slope * m[i];
        }
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) e.K[pk(i, j)] += sm[i] * m[j];
        phi += dt * psi;
      }
    }
    e.phi = phi;
}

// Reciprocal: FP32 division for float; for double an FP32 seed refined by two Newton steps
// r <- r (2 - x r) (each doubles the correct bits: 24 -> 48 -> full precision).
__device__ __forceinline__ float rcp_s(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp_s(double x) {
    double r = (double)(1.0f / (float)x);
    double e = fma(-x, r, 1.0);
    r = fma(r, e, r);
    e = fma(-x, r, 1.0);
    return fma(r, e, r);
}

// LDL^T solve of K d = r (K packed lower, SPD; no square roots). L is unit lower, D diagonal.
// Returns false if a pivot is not positive.
template <typename TS, typename TA> __device__ __forceinline__ bool ldl_solve(const TA Kin[21], const TA rin[6], TA dout[6]) {
    TS L[21], invD[6], w[6];
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        TS dj = (TS)Kin[pk(j, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) {
            w[k] = L[pk(j, k)] * L[pk(k, k)];   // L_jk D_k (L[kk] holds D_k)
            dj -= w[k] * L[pk(j, k)];
        }
        ok = ok && (dj > (TS)0);
        dj = dj > (TS)0 ? dj : (TS)1;
        L[pk(j, j)] = dj;
        invD[j] = rcp_s(dj);
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            TS t = (TS)Kin[pk(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= L[pk(i, k)] * w[k];
            L[pk(i, j)] = t * invD[j];
        }
    }
    TS y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        TS t = (TS)rin[i];
#pragma unroll
        for (int k = 0; k < i; ++k) t -= L[pk(i, k)] * y[k];
        y[i] = t;
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        TS t = y[i] * invD[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) t -= L[pk(k, i)] * y[k];
        y[i] = t;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) dout[i] = (TA)y[i];
    return ok;
}


// Residual and potential only (no tangent): the cost of a chord step.
template <typename TA> struct EvalR {
    TA r[6];
    TA phi;
};
// UNROLL: slip-system pairs unrolled per loop trip (6 = fully, letting the table loads run ahead of
// the arithmetic where registers allow).
template <int UNROLL = 1>
__device__ __forceinline__ void evaluate_r(const float Sp[21], const float *__restrict__ M, const float etr[6], float tauc,
                                           float inv_tc, const float sg[6], const MatConst &mc, EvalR<float> &e) {
    float dt, g0, nn;
    flow_consts(mc, dt, g0, nn);
    float phi = 0.f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < 6; ++j) acc += Sp[i >= j ? pk(i, j) : pk(j, i)] * sg[j];
        e.r[i] = acc - etr[i];
        phi += sg[i] * (0.5f * acc - etr[i]);
    }
    const float cphi = dt * g0 * tauc / (nn + 1.f);
#pragma unroll UNROLL
    for (int p = 0; p < 6; ++p) {
        float mm[12];
        load_slip_pair(M, p, mm);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float *m = mm + 6 * h;
            float tau = 0.f;
#pragma unroll
            for (int i = 0; i < 6; ++i) tau += m[i] * sg[i];
            const float x = tau * inv_tc, ax = fabs(x);
            const float p10 = pow_nm1(ax, mc) * ax;
            const float gd = x < 0.f ? -g0 * p10 : g0 * p10;
            const float dg = dt * gd;
#pragma unroll
            for (int i = 0; i < 6; ++i) e.r[i] += dg * m[i];
            phi += cphi * p10 * ax;
        }
    }
    e.phi = phi;
}


template <int UNROLL = 1>
__device__ __forceinline__ void evaluate_r(const float Sp[21], const float *__restrict__ M, const float etr[6],
                                           const FlowMR<float> &f, float, const float sg[6], const MatConst &mc, EvalR<float> &e) {
    float dt, g0, nn;
    flow_consts(mc, dt, g0, nn);
    const float ga = mr_ga<float>(mc);
    float phi = 0.f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < 6; ++j) acc += Sp[i >= j ? pk(i, j) : pk(j, i)] * sg[j];
        e.r[i] = acc - etr[i];
        phi += sg[i] * (0.5f * acc - etr[i]);
    }
#pragma unroll UNROLL
    for (int p = 0; p < 6; ++p) {
        float mm[12];
        load_slip_pair(M, p, mm);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float *m = mm + 6 * h;
            float tau = 0.f;
#pragma unroll
            for (int i = 0; i < 6; ++i) tau += m[i] * sg[i];
            float tp, itc, gd, slope, psi;
            mr_sys(f, 2 * p + h, tp, itc);
            mr_flow(tau, tp, itc, ga, gd, slope, psi);
            const float dg = dt * gd;
#pragma unroll
            for (int i = 0; i < 6; ++i) e.r[i] += dg * m[i];
            phi += dt * psi;
        }
    }
    e.phi = phi;
}

// ---- residual, tangent and potential of one local problem, in the crystal frame ----
// The 12 systems in three families of four, by the pair of axes (i, j) of their slip directions e_i -+ e_j: with
// D = s_ii - s_jj and the family's two shears A, B, the systems' n.sigma.d are D + u, D - u, D + w and D - w
// (u = A - B, w = A + B) up to a sign, which neither flow rule depends on. kFamSys gives their numbers in the
// order of the density fields.
__host__ __device__ constexpr int fam_sys(int f, int q) {
    return f == 0 ? (q == 0 ? 0 : q == 1 ? 3 : q == 2 ? 9 : 6)
         : f == 1 ? (q == 0 ? 1 : q == 1 ? 7 : q == 2 ? 10 : 4)
                  : (q == 0 ? 2 : q == 1 ? 11 : q == 2 ? 8 : 5);
}
// The family's resolved stresses from h = (11, 22, 33, 23, 13, 12), normals scaled by 1/sqrt6, Mandel shears by
// 1/sqrt12: families (2, 3) with A = 12, B = 13; (1, 3) with A = 12, B = 23; (1, 2) with A = 13, B = 23.
template <typename T> __device__ __forceinline__ void fam_stress(int f, const T h[6], T t[4]) {
    const T D = f == 0 ? h[1] - h[2] : f == 1 ? h[0] - h[2] : h[0] - h[1];
    const T A = f == 2 ? h[4] : h[5], B = f == 0 ? h[4] : h[3];
    const T u = A - B, w = A + B;
    t[0] = D + u; t[1] = D - u; t[2] = D + w; t[3] = D - w;
}

// Rates of one family. Power law: t = tau / tau_c, gam = |t|^n sign(t), slope = |t|^(n-1), pot += |t|^(n+1), to be
// scaled by the caller. Ma-Roters: t = tau, gam, slope and pot as in Eq. FlowRule. WK: slopes wanted, in TK, each
// rounded once from TA: as ninth powers of FP32 stress differences they put the FP32 tangent of the FP64 residual off by up
// to 26 units of 2^-24 instead of 5.
template <bool WK, bool WP, typename TK, typename TA>
__device__ __forceinline__ void fam_rates(TA, int, const TA t[4], const MatConst &mc, TA gam[4], TK slope[4], TA &pot) {
    if (mc.n_int == 10) {
        // the workloads' exponent: |t|^9 = |t| ((t^2)^2)^2, the very products pow_nm1's bit loop forms
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const TA b2 = t[q] * t[q], b4 = b2 * b2, b8 = b4 * b4;
            if constexpr (WK) {
                const TA p9 = fabs(t[q]) * b8;
                slope[q] = (TK)p9;
                gam[q] = p9 * t[q];
            } else {
                gam[q] = copysign(b8 * b2, t[q]);
            }
            if constexpr (WP) pot += gam[q] * t[q];
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const TA p = pow_nm1(fabs(t[q]), mc);
            if constexpr (WK) slope[q] = (TK)p;
            gam[q] = p * t[q];
            if constexpr (WP) pot += gam[q] * t[q];
        }
    }
}
template <bool WK, bool WP, typename TK, typename TA>
__device__ __forceinline__ void fam_rates(const FlowMR<TA> &hf, int f, const TA t[4], const MatConst &mc, TA gam[4],
                                          TK slope[4], TA &pot) {
    const TA ga = mr_ga<TA>(mc);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        TA tp, itc, sl, psi;
        mr_sys(hf, fam_sys(f, q), tp, itc);
        mr_flow(t[q], tp, itc, ga, gam[q], sl, psi);
        if constexpr (WK) slope[q] = (TK)sl;
        if constexpr (WP) pot += psi;
    }
}
// Scales of the sums above: stress -> t (a), rates -> strain over the step (g), slopes -> tangent (k), pot (p).
template <typename TA>
__device__ __forceinline__ void flow_scales(TA tauc, TA inv_tc, const MatConst &mc, TA &a, TA &g, TA &k, TA &p) {
    TA dt, g0, nn;
    flow_consts(mc, dt, g0, nn);
    a = inv_tc;
    g = dt * g0;
    k = g * nn * inv_tc;
    p = g * tauc / (nn + (TA)1);
}
template <typename TA>
__device__ __forceinline__ void flow_scales(const FlowMR<TA> &, TA, const MatConst &mc, TA &a, TA &g, TA &k, TA &p) {
    TA dt, g0, nn;
    flow_consts(mc, dt, g0, nn);
    a = (TA)1;
    g = k = p = dt;
}

// r = S sigma + dt sum m gdot(sigma) - eps_tr, with its tangent K (packed lower, in TK; WK) and the potential phi of
// which it is the gradient (WP). All Mandel vectors in the crystal frame.
template <bool WK, bool WP, typename TK, typename TA, typename H>
__device__ __forceinline__ void evaluate_crystal(const Cubic<TA> &cu, const TA etr[6], const H &hf, TA inv_tc,
                                                 const TA sg[6], const MatConst &mc, TA r[6], TK K[21], TA &phi) {
    const TA q6 = (TA)0.40824829046386301637, q12 = (TA)0.28867513459481288225;   // 1/sqrt6, 1/sqrt12
    TA sa, gs, ks, ps;
    flow_scales(hf, inv_tc, mc, sa, gs, ks, ps);
    const TA an = sa * q6, as = sa * q12;
    TA h[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) h[i] = (i < 3 ? an : as) * sg[i];
    TA gD[3], gA[3], gB[3], pot = (TA)0;
    TK W[3], kA[3], kB[3], kX[3];
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        TA t[4], g[4];
        TK w[4];
        fam_stress(f, h, t);
        fam_rates<WK, WP, TK>(hf, f, t, mc, g, w, pot);
        const TA gu = g[0] - g[1], gw = g[2] - g[3];
        gD[f] = (g[0] + g[1]) + (g[2] + g[3]);
        gA[f] = gu + gw;
        gB[f] = gw - gu;
        if constexpr (WK) {   // sum of w t t^T on (D, A, B): DD = AA = BB = W, DA, DB, AB
            const TK p = w[0] + w[1], q = w[2] + w[3], m = w[0] - w[1], n = w[2] - w[3];
            W[f] = p + q;
            kA[f] = m + n;
            kB[f] = n - m;
            kX[f] = q - p;
        }
    }
    const TA fn = gs * q6, fs = gs * q12, st = cu.s12 * (sg[0] + sg[1] + sg[2]);
    const TA ep[6] = {gD[1] + gD[2], gD[0] - gD[2], -(gD[0] + gD[1]), gB[1] + gB[2], gB[0] + gA[2], gA[0] + gA[1]};
    TA el = (TA)0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const TA u = (i < 3 ? cu.d : cu.s44) * sg[i] + (i < 3 ? st - etr[i] : -etr[i]);   // S sigma - eps_tr
        r[i] = (i < 3 ? fn : fs) * ep[i] + u;
        if constexpr (WP) el += sg[i] * (u - etr[i]);
    }
    if constexpr (WP) phi = (TA)0.5 * el + ps * pot;
    if constexpr (WK) {
        const TK ksk = (TK)ks, kn = ksk * (TK)(1.0 / 6.0), kx = ksk * (TK)0.11785113019775792073, kt = ksk * (TK)(1.0 / 12.0);
        const Cubic<TK> ck = cu.template as<TK>();
        const TK s11 = ck.d + ck.s12;
        K[pk(0, 0)] = s11 + kn * (W[1] + W[2]);
        K[pk(1, 0)] = ck.s12 - kn * W[2];
        K[pk(1, 1)] = s11 + kn * (W[0] + W[2]);
        K[pk(2, 0)] = ck.s12 - kn * W[1];
        K[pk(2, 1)] = ck.s12 - kn * W[0];
        K[pk(2, 2)] = s11 + kn * (W[0] + W[1]);
        K[pk(3, 0)] = kx * (kB[1] + kB[2]);
        K[pk(3, 1)] = -kx * kB[2];
        K[pk(3, 2)] = -kx * kB[1];
        K[pk(3, 3)] = ck.s44 + kt * (W[1] + W[2]);
        K[pk(4, 0)] = kx * kA[2];
        K[pk(4, 1)] = kx * (kB[0] - kA[2]);
        K[pk(4, 2)] = -kx * kB[0];
        K[pk(4, 3)] = kt * kX[2];
        K[pk(4, 4)] = ck.s44 + kt * (W[0] + W[2]);
        K[pk(5, 0)] = kx * kA[1];
        K[pk(5, 1)] = kx * kA[0];
        K[pk(5, 2)] = -kx * (kA[0] + kA[1]);
        K[pk(5, 3)] = kt * kX[1];
        K[pk(5, 4)] = kt * kX[0];
        K[pk(5, 5)] = ck.s44 + kt * (W[0] + W[1]);
    }
}

// LDL^T factorisation kept for reuse: F[0..14] = strict lower L (row-major by packed index, diagonal
// slots skipped), F[15..20] = 1/D. Returns false if a pivot is not positive.
template <typename TS, typename TA> __device__ __forceinline__ bool ldl_factor(const TA Kin[21], TS F[21]) {
    TS L[21], invD[6], w[6];
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        TS dj = (TS)Kin[pk(j, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) {
            w[k] = L[pk(j, k)] * L[pk(k, k)];
            dj -= w[k] * L[pk(j, k)];
        }
        ok = ok && (dj > (TS)0);
        dj = dj > (TS)0 ? dj : (TS)1;
        L[pk(j, j)] = dj;
        invD[j] = rcp_s(dj);
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            TS t = (TS)Kin[pk(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= L[pk(i, k)] * w[k];
            L[pk(i, j)] = t * invD[j];
        }
    }
    int q = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) F[q++] = L[pk(i, j)];
#pragma unroll
    for (int j = 0; j < 6; ++j) F[15 + j] = invD[j];
    return ok;
}

template <typename TS, typename TA> __device__ __forceinline__ void ldl_apply(const TS F[21], const TA rin[6], TA dout[6]) {
    // strict-lower index of (i, j), j < i: i(i-1)/2 + j
    TS y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        TS t = (TS)rin[i];
#pragma unroll
        for (int k = 0; k < i; ++k) t -= F[i * (i - 1) / 2 + k] * y[k];
        y[i] = t;
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        TS t = y[i] * F[15 + i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) t -= F[k * (k - 1) / 2 + i] * y[k];
        y[i] = t;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) dout[i] = (TA)y[i];
}

// The forms the solvers call: with the tangent (FP64 residuals may take it in FP32), or without it (the cost of a
// chord step); UNROLL as in evaluate_r.
template <typename TK, typename H>
__device__ __forceinline__ void evaluate(const Problem<double> &p, const double etr[6], const H &hf, double inv_tc,
                                         const double sg[6], const MatConst &mc, Eval<double, TK> &e) {
    evaluate_crystal<true, true, TK>(p.cu, etr, hf, inv_tc, sg, mc, e.r, e.K, e.phi);
}
template <typename H>
__device__ __forceinline__ void evaluate(const Problem<float> &p, const float etr[6], const H &hf, float inv_tc,
                                         const float sg[6], const MatConst &mc, Eval<float> &e) {
    evaluate(p.Sp, p.M, etr, hf, inv_tc, sg, mc, e);
}
template <int UNROLL = 1, typename H>
__device__ __forceinline__ void evaluate_r(const Problem<double> &p, const double etr[6], const H &hf, double inv_tc,
                                           const double sg[6], const MatConst &mc, EvalR<double> &e) {
    evaluate_crystal<false, true, double>(p.cu, etr, hf, inv_tc, sg, mc, e.r, nullptr, e.phi);
}
template <int UNROLL = 1, typename H>
__device__ __forceinline__ void evaluate_r(const Problem<float> &p, const float etr[6], const H &hf, float inv_tc,
                                           const float sg[6], const MatConst &mc, EvalR<float> &e) {
    evaluate_r<UNROLL>(p.Sp, p.M, etr, hf, inv_tc, sg, mc, e);
}

}  // namespace evp
