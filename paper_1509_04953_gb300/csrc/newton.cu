// Per-voxel crystal-plasticity kernels (Sec. 2.1 Eqs. HookeLaw / PlasticRate, Sec. 2.2 flow rule
// and density evolution read as a power law with Kocks-Mecking hardening).
//
// Local problem: find sigma with r(sigma) = S:sigma + dt sum_a m^a gdot^a(sigma) - eps_tr = 0,
// gdot^a = gdot0 |tau^a/tau_c|^n sign(tau^a), tau^a = m^a:sigma. This is the implicit Euler
// stress update of Eq. HookeLaw multiplied by the compliance S = C^-1; its Jacobian
// K = S + dt sum_a (n gdot0 |x^a|^(n-1)/tau_c) m^a (x) m^a is symmetric positive definite, so the
// 6x6 Newton system is solved by an LDL^T factorisation, and r is the gradient of a convex potential Phi used
// for Armijo backtracking. eps_tr = eps^{t+dt} - eps_p^t is carried directly (the "trial" elastic
// strain), which keeps FP32 fields accurate when the total strain is large.
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "local.cuh"
#include "fpctl.cuh"

namespace evp {

namespace {

constexpr int kThreads = 128;

// Local-solve statistics, summed over the block before they touch the shared counters (the same-address
// atomics of every warp of a two-million-voxel launch serialise in L2): flags[0] += failed voxels,
// flags[1] = max(local iterations); 64-bit flags[4..5] += iterations (6x6 solves), [6..7] += residual
// evaluations, [8..9] += tangent refreshes. Every thread of the block calls it once.
__device__ __forceinline__ void block_solve_stats(int fail, int maxit, int it, int ev, int rf, int *flags) {
    __shared__ int sh[kThreads / 32][5];
    int f = fail, mx = maxit, sit = it, sev = ev, srf = rf;
    for (int o = 16; o > 0; o >>= 1) {
        f += __shfl_xor_sync(0xffffffffu, f, o);
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        sit += __shfl_xor_sync(0xffffffffu, sit, o);
        sev += __shfl_xor_sync(0xffffffffu, sev, o);
        srf += __shfl_xor_sync(0xffffffffu, srf, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        sh[w][0] = f; sh[w][1] = mx; sh[w][2] = sit; sh[w][3] = sev; sh[w][4] = srf;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int tf = 0, tm = 0;
        unsigned long long ti = 0, te = 0, tr = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            tf += sh[k][0]; tm = max(tm, sh[k][1]);
            ti += (unsigned)sh[k][2]; te += (unsigned)sh[k][3]; tr += (unsigned)sh[k][4];
        }
        if (tf) atomicAdd(flags, tf);
        if (tm) atomicMax(flags + 1, tm);
        if (ti) atomicAdd(reinterpret_cast<unsigned long long *>(flags + 4), ti);
        if (te) atomicAdd(reinterpret_cast<unsigned long long *>(flags + 6), te);
        if (tr) atomicAdd(reinterpret_cast<unsigned long long *>(flags + 8), tr);
    }
}

// Damped Newton on one voxel. Returns the iteration count (> 0) or minus it on failure.
// H: the power law's tau_c (TA) or the Ma-Roters flow data (FlowMR<TA>, Sec. 2.2).
template <typename TA, typename TS, typename H>
__device__ int newton_voxel(const Problem<TA> &pb, const TA etr[6], const H &hf, TA sg[6],
                            const MatConst &mc, TA tol, int maxit, TA ls_free, int &nevals) {
    const TA tauc = flow_ref(hf);
    const TA inv_tc = drcp(tauc);
    Eval<TA> e;
    evaluate(pb, etr, hf, inv_tc, sg, mc, e);
    nevals = 1;
    for (int it = 1; it <= maxit; ++it) {
        TA d[6];
        if (!ldl_solve<TS, TA>(e.K, e.r, d)) return -it;
        TA rd = (TA)0, dn = (TA)0, sn = (TA)0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            rd += e.r[i] * d[i];
            dn += d[i] * d[i];
            sn += sg[i] * sg[i];
        }
        dn = dsqrt(dn);
        const TA scale = dsqrt(sn) + tauc;
        if (dn <= tol * scale) {
            // The full step is below the stopping tolerance (and far below the line-search
            // threshold), so it is taken and the iteration ends without evaluating the new point.
#pragma unroll
            for (int i = 0; i < 6; ++i) sg[i] -= d[i];
            return it;
        }
        const TA phi0 = e.phi;
        TA s = (TA)1, st[6];
        bool ok = false;
        for (int h = 0; h < 60; ++h) {
#pragma unroll
            for (int i = 0; i < 6; ++i) st[i] = sg[i] - s * d[i];
            evaluate(pb, etr, hf, inv_tc, st, mc, e);
            ++nevals;
            if (e.phi <= phi0 - (TA)1e-4 * s * rd || s * dn <= ls_free * scale) {
                ok = true;
                break;
            }
            s *= (TA)0.5;
        }
        if (!ok) return -it;
#pragma unroll
        for (int i = 0; i < 6; ++i) sg[i] = st[i];
        if (s * dn <= tol * scale) return it;
    }
    return -maxit;
}

template <typename TA, typename TS, bool MR = false>
__global__ void __launch_bounds__(kThreads) k_newton(long N3, const TA *__restrict__ epst, const TA *__restrict__ tauc,
                                                    const int32_t *__restrict__ g0, TA *__restrict__ sig,
                                                    LocalTab<TA> tab, MatConst mc,
                                                    TA tol, int maxit, TA ls_free, int *__restrict__ flags, const int *__restrict__ skip,
    const TA *__restrict__ tol_dev, MRPtr<TA> mrp) {
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    if (tol_dev != nullptr) tol = *tol_dev;   // local tolerance set on the device for this iteration
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = v < N3;
    int r = 1, nev = 0;
    if (valid) {
        Problem<TA> pb;
        pb.init(tab, g0[v]);
        TA etr[6], sg[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            etr[c] = epst[c * N3 + v];
            sg[c] = sig[c * N3 + v];
        }
        pb.enter(etr, sg);
        if constexpr (MR)
            r = newton_voxel<TA, TS>(pb, etr, FlowMR<TA>{mrp.tpi, N3, v, tauc[v]}, sg, mc,
                                     tol, maxit, ls_free, nev);
        else
            r = newton_voxel<TA, TS>(pb, etr, tauc[v], sg, mc, tol, maxit, ls_free, nev);
        pb.leave(sg);
#pragma unroll
        for (int c = 0; c < 6; ++c) sig[c * N3 + v] = sg[c];
    }
    const int its = valid ? (r < 0 ? -r : r) : 0;
    block_solve_stats(valid && r < 0, its, its, nev, 0, flags);
}

// FP64 path: Newton on the FP64 residual with an FP32 tangent and FP32 6x6 solve. Each step is a
// slightly inexact Newton step (tangent rounded to FP32: a few 1e-7 relative), so the iteration contracts at least
// ~1e-6 per step near the solution and stops on the same step-size test; Armijo backtracking on
// the FP64 potential keeps it globally convergent.
__device__ int newton_voxel_df(const Problem<double> &pb, const double etr[6], double tauc, double sg[6],
                               const MatConst &mc, double tol, int maxit, double ls_free, int &nevals) {
    const double inv_tc = drcp(tauc);
    Eval<double, float> e;
    evaluate(pb, etr, tauc, inv_tc, sg, mc, e);
    nevals = 1;
    for (int it = 1; it <= maxit; ++it) {
        float rf[6], df[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) rf[i] = (float)e.r[i];
        if (!ldl_solve<float, float>(e.K, rf, df)) return -it;
        double d[6], rd = 0.0, dn = 0.0, sn = 0.0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            d[i] = (double)df[i];
            rd += e.r[i] * d[i];
            dn += d[i] * d[i];
            sn += sg[i] * sg[i];
        }
        dn = dsqrt(dn);
        const double scale = dsqrt(sn) + tauc;
        if (dn <= tol * scale && rd >= 0.0) {
#pragma unroll
            for (int i = 0; i < 6; ++i) sg[i] -= d[i];
            return it;
        }
        const double phi0 = e.phi;
        double s = 1.0, st[6];
        bool ok = false;
        for (int h = 0; h < 60; ++h) {
#pragma unroll
            for (int i = 0; i < 6; ++i) st[i] = sg[i] - s * d[i];
            evaluate(pb, etr, tauc, inv_tc, st, mc, e);
            ++nevals;
            if (e.phi <= phi0 - 1e-4 * s * rd || s * dn <= ls_free * scale) {
                ok = true;
                break;
            }
            s *= 0.5;
        }
        if (!ok) return -it;
#pragma unroll
        for (int i = 0; i < 6; ++i) sg[i] = st[i];
        if (s * dn <= tol * scale) return it;
    }
    return -maxit;
}

__global__ void __launch_bounds__(kThreads) k_newton_df(long N3, const double *__restrict__ epst,
                                                       const double *__restrict__ tauc, const int32_t *__restrict__ g0,
                                                       double *__restrict__ sig, LocalTab<double> tab,
                                                       MatConst mc, double tol,
                                                       int maxit, int *__restrict__ flags, const int *__restrict__ skip,
    const double *__restrict__ tol_dev) {
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    if (tol_dev != nullptr) tol = *tol_dev;   // local tolerance set on the device for this iteration
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = v < N3;
    int r = 1, nev = 0;
    if (valid) {
        Problem<double> pb;
        pb.init(tab, g0[v]);
        double etr[6], sg[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            etr[c] = epst[c * N3 + v];
            sg[c] = sig[c * N3 + v];
        }
        pb.enter(etr, sg);
        r = newton_voxel_df(pb, etr, tauc[v], sg, mc, tol, maxit, 1e-6, nev);
        pb.leave(sg);
#pragma unroll
        for (int c = 0; c < 6; ++c) sig[c * N3 + v] = sg[c];
    }
    const int its = valid ? (r < 0 ? -r : r) : 0;
    block_solve_stats(valid && r < 0, its, its, nev, 0, flags);
}

// Local solve with Jacobian reuse (chord Newton): the LDL^T factors of the tangent are stored per
// voxel and reused across fixed-point iterations; a step costs one residual evaluation and two
// triangular solves. The factors are refreshed (full tangent + factorisation at the current point)
// on request (first fixed-point iteration of an increment), when a step contracts by less than
// 4x, or after a backtracking line search. The local problem is still solved to the same
// tolerance, so the result matches the exact-Newton one to that tolerance.
//
// The factorisation runs in TF and the factors are stored and applied in TS. On the FP32-field path
// TF = double and TS = float: an FP32 factorisation of this tangent loses the small (elastic) pivots
// to cancellation once a few slip systems are far into the power law, while FP64 factors rounded to
// FP32 afterwards are a componentwise perturbation and keep the Newton direction within about 1e-4
// relative even there, so the reused step runs on the FP32 pipe and reads half the bytes.
template <typename TA, typename TS, typename TF, typename H>
__device__ int chord_voxel(const Problem<TA> &pb, const TA etr[6], const H &hf, TA sg[6],
                           const MatConst &mc, TA tol, int maxit, TA ls_free, TS F[21], bool refresh, int &nevals,
                           int &nref) {
    const TA tauc = flow_ref(hf);
    const TA inv_tc = drcp(tauc);
    EvalR<TA> e;
    evaluate_r(pb, etr, hf, inv_tc, sg, mc, e);
    nevals = 1;
    nref = 0;
    TA prev_step = (TA)-1;
    bool fresh = false;
    for (int it = 1; it <= maxit; ++it) {
        if (refresh) {
            Eval<TA> full;
            evaluate(pb, etr, hf, inv_tc, sg, mc, full);
            ++nevals;
            TF Ff[21];
            if (!ldl_factor<TF, TA>(full.K, Ff)) return -it;
#pragma unroll
            for (int q = 0; q < 21; ++q) F[q] = (TS)Ff[q];
            ++nref;
            refresh = false;
            fresh = true;
        }
        TA d[6];
        ldl_apply<TS, TA>(F, e.r, d);
        TA rd = (TA)0, dn = (TA)0, sn = (TA)0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            rd += e.r[i] * d[i];
            dn += d[i] * d[i];
            sn += sg[i] * sg[i];
        }
        dn = dsqrt(dn);
        const TA scale = dsqrt(sn) + tauc;
        if (dn <= tol * scale && rd >= (TA)0) {
#pragma unroll
            for (int i = 0; i < 6; ++i) sg[i] -= d[i];
            return it;
        }
        if (!fresh && (rd <= (TA)0 || (prev_step > (TA)0 && dn > (TA)0.25 * prev_step))) {
            refresh = true;   // stale tangent: refactor at this point and redo the step
            continue;
        }
        const TA phi0 = e.phi;
        TA s = (TA)1, st[6];
        bool ok = false;
        for (int h = 0; h < 60; ++h) {
#pragma unroll
            for (int i = 0; i < 6; ++i) st[i] = sg[i] - s * d[i];
            evaluate_r(pb, etr, hf, inv_tc, st, mc, e);
            ++nevals;
            if (e.phi <= phi0 - (TA)1e-4 * s * rd || s * dn <= ls_free * scale) {
                ok = true;
                break;
            }
            s *= (TA)0.5;
        }
        if (!ok) return -it;
#pragma unroll
        for (int i = 0; i < 6; ++i) sg[i] = st[i];
        if (s * dn <= tol * scale) return it;
        if (s < (TA)1) refresh = true;
        prev_step = s * dn;
        fresh = false;
    }
    return -maxit;
}

template <typename TA, typename TS, typename TF, bool MR = false>
__global__ void __launch_bounds__(kThreads, sizeof(TA) == 4 ? 3 : 2) k_newton_chord(long N3, const TA *__restrict__ epst, const TA *__restrict__ tauc,
                                                          const int32_t *__restrict__ g0, TA *__restrict__ sig,
                                                          LocalTab<TA> tab,
                                                          TS *__restrict__ fac, MatConst mc, TA tol, int maxit,
                                                          TA ls_free, int force_refresh, int *__restrict__ flags, const int *__restrict__ skip,
    const TA *__restrict__ tol_dev, MRPtr<TA> mrp) {
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    if (tol_dev != nullptr) tol = *tol_dev;   // local tolerance set on the device for this iteration
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = v < N3;
    int r = 1, nev = 0, nref = 0;
    if (valid) {
        Problem<TA> pb;
        pb.init(tab, g0[v]);
        TA etr[6], sg[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            etr[c] = epst[c * N3 + v];
            sg[c] = sig[c * N3 + v];
        }
        pb.enter(etr, sg);
        TS F[21];
        if (!force_refresh) {
            load_factors(fac, N3, v, F);
        }
        if constexpr (MR)
            r = chord_voxel<TA, TS, TF>(pb, etr, FlowMR<TA>{mrp.tpi, N3, v, tauc[v]}, sg,
                                        mc, tol, maxit, ls_free, F, force_refresh != 0, nev, nref);
        else
            r = chord_voxel<TA, TS, TF>(pb, etr, tauc[v], sg, mc, tol, maxit, ls_free, F,
                                        force_refresh != 0, nev, nref);
        pb.leave(sg);
#pragma unroll
        for (int c = 0; c < 6; ++c) sig[c * N3 + v] = sg[c];
        if (nref) {
            store_factors(fac, N3, v, F);
        }
    }
    const int its = valid ? (r < 0 ? -r : r) : 0;
    block_solve_stats(valid && r < 0, its, its, nev, nref, flags);
}

// Tangent reuse in two passes. Most voxels accept the first chord step once the fixed point has
// settled, while a few need line searches or a refreshed tangent; in one kernel the warps holding
// those few run their long loops with most lanes idle. Pass 1 takes the first step for every voxel
// and stores it where it is accepted; the others are appended to a work list (warp-aggregated,
// order immaterial: each voxel's computation is independent and deterministic). Pass 2 runs the
// full chord iteration on the listed voxels only, from their unchanged state, so every result is
// bitwise the one the single-kernel iteration gives.
// TWO: also the chord iteration's next two moves (below); its registers cost one CTA per SM on the FP32 path.
template <typename TA, typename TS, bool MR = false, bool TWO = true>
__global__ void __launch_bounds__(kThreads, sizeof(TA) == 4 ? (TWO ? 7 : 8) : 1) k_chord_first(long N3, const TA *__restrict__ epst,
                                                         const TA *__restrict__ tauc, const int32_t *__restrict__ g0,
                                                         TA *__restrict__ sig, LocalTab<TA> tab,
                                                         const TS *__restrict__ fac,
                                                         MatConst mc, TA tol, TA ls_free, int *__restrict__ flags,
                                                         int32_t *__restrict__ wl, const int *__restrict__ skip,
    const TA *__restrict__ tol_dev, MRPtr<TA> mrp) {
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    if (tol_dev != nullptr) tol = *tol_dev;   // local tolerance set on the device for this iteration
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = v < N3;
    bool done = false, two = false;
    // the stored factors are needed only after the residual: their copies start first, into this thread's slots
    // of shared memory, and run under the other loads and the evaluation
    __shared__ __align__(16) TS fsh[factor_words<TS>() * kThreads];
    if (valid) prefetch_factors(fac, N3, v, fsh);
    if (valid) {
        const int g = g0[v];
        Problem<TA> pb;
        pb.init(tab, g);
        TA etr[6], sg[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            etr[c] = epst[c * N3 + v];
            sg[c] = sig[c * N3 + v];
        }
        const TA tc = tauc[v];
        pb.enter(etr, sg);
        EvalR<TA> e;
        if constexpr (MR)
            evaluate_r<6>(pb, etr, FlowMR<TA>{mrp.tpi, N3, v, tc}, (TA)0, sg, mc, e);
        else
            evaluate_r<6>(pb, etr, tc, drcp(tc), sg, mc, e);
        TS F[21];
        prefetched_factors(fsh, F);
        TA d[6];
        ldl_apply<TS, TA>(F, e.r, d);
        TA rd = (TA)0, dn = (TA)0, sn = (TA)0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            rd += e.r[i] * d[i];
            dn += d[i] * d[i];
            sn += sg[i] * sg[i];
        }
        dn = dsqrt(dn);
        const TA scale = dsqrt(sn) + tc;
        if (dn <= tol * scale && rd >= (TA)0) {   // the acceptance test of chord_voxel
            TA sn6[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) sn6[c] = sg[c] - d[c];
            pb.leave(sn6);
#pragma unroll
            for (int c = 0; c < 6; ++c) sig[c * N3 + v] = sn6[c];
            done = true;
        } else if (TWO && rd > (TA)0) {
            // chord_voxel's next moves while they stay on its common path, with its operations in its order: the
            // full step of the line search (s = 1) passes the sufficient-decrease test, and the chord step from
            // there passes the acceptance test. Anything else goes to pass 2, which starts over from the
            // unchanged state, so every voxel still ends bitwise where the single-kernel iteration puts it.
            // The grain's compliance and the factors are fetched again (from L1 and shared memory) rather than held
            // in registers through the first step.
            const TA s1 = (TA)1, phi0 = e.phi;
            TA st[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) st[i] = sg[i] - s1 * d[i];
            asm volatile("" ::: "memory");
            Problem<TA> pb2;
            pb2.init(tab, g);
            if constexpr (MR)
                evaluate_r(pb2, etr, FlowMR<TA>{mrp.tpi, N3, v, tc}, (TA)0, st, mc, e);
            else
                evaluate_r(pb2, etr, tc, drcp(tc), st, mc, e);
            if (e.phi <= phi0 - (TA)1e-4 * s1 * rd || s1 * dn <= ls_free * scale) {
                prefetched_factors(fsh, F);
                ldl_apply<TS, TA>(F, e.r, d);
                TA rd2 = (TA)0, dn2 = (TA)0, sn2 = (TA)0;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    rd2 += e.r[i] * d[i];
                    dn2 += d[i] * d[i];
                    sn2 += st[i] * st[i];
                }
                dn2 = dsqrt(dn2);
                if (dn2 <= tol * (dsqrt(sn2) + tc) && rd2 >= (TA)0) {
#pragma unroll
                    for (int c = 0; c < 6; ++c) st[c] -= d[c];
                    pb2.leave(st);
#pragma unroll
                    for (int c = 0; c < 6; ++c) sig[c * N3 + v] = st[c];
                    done = true;
                    two = true;
                }
            }
        }
    }
    const unsigned todo = __ballot_sync(0xffffffffu, valid && !done);
    const unsigned twos = __ballot_sync(0xffffffffu, two);
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == 0 && todo) base = atomicAdd(flags + 10, __popc(todo));
    if (lane == 0 && twos) atomicAdd(flags + 11, __popc(twos));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (valid && !done) wl[base + __popc(todo & ((1u << lane) - 1u))] = (int32_t)v;
    // the accepted voxels are counted by pass 2: N3 - listed with one evaluation and one solve each, plus one more
    // of each for the flags[11] voxels accepted after two steps
}

template <typename TA, typename TS, typename TF, bool MR = false>
__global__ void __launch_bounds__(kThreads, sizeof(TA) == 4 ? 3 : 2) k_chord_rest(
    long N3, const TA *__restrict__ epst, const TA *__restrict__ tauc, const int32_t *__restrict__ g0,
    TA *__restrict__ sig, LocalTab<TA> tab, TS *__restrict__ fac, MatConst mc,
    TA tol, int maxit, TA ls_free, int *__restrict__ flags, const int32_t *__restrict__ wl, const int *__restrict__ skip,
    const TA *__restrict__ tol_dev, MRPtr<TA> mrp) {
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    if (tol_dev != nullptr) tol = *tol_dev;   // local tolerance set on the device for this iteration
    const int count = *(volatile const int *)(flags + 10);
    if (blockIdx.x == 0 && threadIdx.x == 0 && N3 - count > 0) {   // pass 1 accepted the others in one or two steps
        const int twos = *(volatile const int *)(flags + 11);
        atomicMax(flags + 1, twos > 0 ? 2 : 1);
        atomicAdd(reinterpret_cast<unsigned long long *>(flags + 4), (unsigned long long)(N3 - count + twos));
        atomicAdd(reinterpret_cast<unsigned long long *>(flags + 6), (unsigned long long)(N3 - count + twos));
    }
    const long stride = (long)gridDim.x * blockDim.x;
    int t_fail = 0, t_mx = 0, t_it = 0, t_ev = 0, t_rf = 0;
    for (long w0 = (long)blockIdx.x * blockDim.x; w0 < count; w0 += stride) {   // block-uniform trip count
        const long w = w0 + threadIdx.x;
        const bool valid = w < count;
        int r = 1, nev = 0, nref = 0;
        if (valid) {
            const long v = wl[w];
            Problem<TA> pb;
            pb.init(tab, g0[v]);
            TA etr[6], sg[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                etr[c] = epst[c * N3 + v];
                sg[c] = sig[c * N3 + v];
            }
            pb.enter(etr, sg);
            TS F[21];
            load_factors(fac, N3, v, F);
            if constexpr (MR)
                r = chord_voxel<TA, TS, TF>(pb, etr, FlowMR<TA>{mrp.tpi, N3, v, tauc[v]},
                                            sg, mc, tol, maxit, ls_free, F, false, nev, nref);
            else
                r = chord_voxel<TA, TS, TF>(pb, etr, tauc[v], sg, mc, tol, maxit, ls_free, F, false,
                                            nev, nref);
            pb.leave(sg);
#pragma unroll
            for (int c = 0; c < 6; ++c) sig[c * N3 + v] = sg[c];
            if (nref) {
                store_factors(fac, N3, v, F);
            }
        }
        if (valid) {
            const int it = r < 0 ? -r : r;
            t_fail += r < 0;
            t_mx = max(t_mx, it);
            t_it += it;
            t_ev += nev;
            t_rf += nref;
        }
    }
    block_solve_stats(t_fail, t_mx, t_it, t_ev, t_rf, flags);
}

// Augmented-Lagrangian local step (the solver the paper names, Sec. 2.1, after Michel et al.):
// with C0 the reference stiffness and S0 = C0^-1, per voxel
//   eps_tr' = S0 lam + eps_tr              (trial strain of the local problem)
//   solve (S + S0) sigma + dt sum m gdot(sigma) = eps_tr'     -> sigma   (Sal = S + S0 per grain)
//   e_tr = eps_tr' - S0 sigma              (local strain, minus eps_p^t)
//   lam  = lam + C0 (eps_tr - e_tr)
//   p    = lam - C0 (e_tr - eps_e^t)       (minus the polarisation; the z pass returns -Gamma0 p)
// init = 1 is the start of an increment: sigma from the plain implicit update at eps_tr (S instead of
// Sal, no lam term), then lam = sigma and e_tr = eps_tr. Partial sums per block: |eps_tr - e_tr|^2,
// |C0 (eps_tr - e_tr)|^2, the six components of lam and the six of sigma.
// The error-free product beside two_sum_f: p + e equals a b exactly.
__device__ __forceinline__ void two_prod_f(float a, float b, float &p, float &e) {
    p = __fmul_rn(a, b);
    e = fmaf(a, b, -p);
}

// C0 x for the isotropic reference stiffness (Lame constants l0, m0), component i of Mandel x.
template <typename T> __device__ __forceinline__ T iso_apply_c0(T l0, T m0, const T x[6], int i) {
    const T tr = x[0] + x[1] + x[2];
    return (T)2 * m0 * x[i] + (i < 3 ? l0 * tr : (T)0);
}

// Adds the warp's sums of 14 per-thread values to acc: lane l gets value l / 2 (lanes 28 .. 31 nothing). Pairwise trees in
// the value type, the values split over the lanes as the tree descends (16 exchanges instead of 14 x 5), then one
// FP64 addition per lane: with the sums in one lane it took 28 FP64-pipe instructions per warp of voxels, 97 us of
// the FP64 pipe in a 128^3 step.
template <typename T> __device__ __forceinline__ void warp_accumulate14(const T (&v)[14], double &acc) {
    const int lane = threadIdx.x & 31;
    T x[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) x[q] = q < 14 ? v[q < 14 ? q : 0] : (T)0;
#pragma unroll
    for (int o = 16; o > 1; o >>= 1) {
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < o / 2) {   // this lane keeps o / 2 of its o values
                const T send = hi ? x[i] : x[i + o / 2], keep = hi ? x[i + o / 2] : x[i];
                x[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
    acc += (double)x[0];
}

// What follows a voxel's local solve: sigma stored, the local strain, the multiplier update, the next transform's input
// and the voxel's terms of the 14 sums. etr is the trial strain eps_tr' of the local problem.
template <typename TA>
__device__ __forceinline__ void al_update(long N3, long v, const TA et[6], const TA lm[6], const TA ee[6], const TA etr[6],
                                          const TA sg[6], TA *__restrict__ sig, TA *__restrict__ lam,
                                          TA *__restrict__ pout, TA l0, TA m0, TA sa, TA sb, TA sa_lo, TA sb_lo,
                                          double sad, double sbd, int init, TA (&sums)[14]) {
    // local strain e_tr = eps_tr' - S0 sigma and the gap d = eps_tr - e_tr to about twice the field
    // precision: near convergence eps_tr and e_tr agree to many digits, and forming them in plain FP32
    // leaves rounding noise in d (hence in the multiplier update) that keeps the iteration from
    // settling. FP64 does it on the FP64 path; the FP32 path uses error-free transformations on the
    // FP32 pipe (the FP64 pipe issues 1/64 as fast).
    TA el[6], d[6], de[6];
    if constexpr (sizeof(TA) == 4) {
        float t1, e1, th, e2;
        two_sum_f(sg[0], sg[1], t1, e1);
        two_sum_f(t1, sg[2], th, e2);
        const float tl = __fadd_rn(e1, e2);   // tr(sigma) = th + tl
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            sig[c * N3 + v] = sg[c];
            if (init) {
                el[c] = et[c];
                d[c] = 0.f;
            } else {
                float p, pe;
                two_prod_f(sa, sg[c], p, pe);
                pe = fmaf(sa_lo, sg[c], pe);   // S0 sigma (shear part) = p + pe
                float sh = p, sl = pe;
                if (c < 3) {
                    float q, qe, se;
                    two_prod_f(sb, th, q, qe);
                    qe = fmaf(sb, tl, fmaf(sb_lo, th, qe));   // sb tr = q + qe
                    two_sum_f(p, -q, sh, se);
                    sl = __fadd_rn(se, __fsub_rn(pe, qe));
                }
                float u, ue, w, we;
                two_sum_f(etr[c], -sh, u, ue);            // e_tr = u + ul
                const float ul = __fsub_rn(ue, sl);
                two_sum_f(et[c], -u, w, we);              // d = eps_tr - e_tr
                d[c] = __fadd_rn(w, __fsub_rn(we, ul));
                el[c] = __fadd_rn(u, ul);
            }
            de[c] = el[c] - ee[c];
        }
    } else {
        double s6[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) s6[c] = (double)sg[c];
        const double str = s6[0] + s6[1] + s6[2];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            sig[c * N3 + v] = sg[c];
            const double eld = init ? (double)et[c] : (double)etr[c] - (sad * s6[c] - (c < 3 ? sbd * str : 0.0));
            d[c] = (TA)((double)et[c] - eld);
            el[c] = (TA)eld;
            de[c] = el[c] - ee[c];
        }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const TA dl = iso_apply_c0(l0, m0, d, c);
        const TA nl = init ? sg[c] : lm[c] + dl;
        lam[c * N3 + v] = nl;
        pout[c * N3 + v] = nl - iso_apply_c0(l0, m0, de, c);
        sums[0] += d[c] * d[c];
        sums[1] += dl * dl;
        sums[2 + c] = nl;
        sums[8 + c] = sg[c];
    }
}

// The block's 14 sums from its lanes' (warp_accumulate14), one column per block in part. rows: 14 doubles per warp.
__device__ __forceinline__ void al_store_sums(double acc, double *rows, double *__restrict__ part) {
    const int lane = threadIdx.x & 31;
    if ((lane & 1) == 0 && lane < 28) rows[(threadIdx.x >> 5) * 14 + (lane >> 1)] = acc;
    __syncthreads();
    if (threadIdx.x < 14) {
        double t = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += rows[k * 14 + threadIdx.x];
        part[(long)threadIdx.x * gridDim.x + blockIdx.x] = t;
    }
}

template <typename TA, typename TS, typename TF, bool MR = false>
__global__ void __launch_bounds__(kThreads, sizeof(TA) == 4 ? 3 : 2) k_al_local(long N3, const TA *__restrict__ epst, const TA *__restrict__ epse,
                                                      const TA *__restrict__ tauc, const int32_t *__restrict__ g0,
                                                      TA *__restrict__ sig, TA *__restrict__ lam, TA *__restrict__ pout,
                                                      LocalTab<TA> tab, MatConst mc, TA l0, TA m0, TA sa,
                                                      TA sb, TA sa_lo, TA sb_lo, double sad, double sbd, TA tol,
                                                      int maxit, TA ls_free, int init,
                                                      int *__restrict__ flags, double *__restrict__ part,
                                                      TS *__restrict__ fac, int refresh, MRPtr<TA> mrp,
                                                      const int *__restrict__ skip, const TA *__restrict__ tol_dev) {
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the increment's iteration has ended
    if (tol_dev != nullptr) tol = *tol_dev;
    constexpr int NV = 14;
    // grid-stride over tiles of blockDim voxels (block-uniform trip count): the block's warps run their tiles
    // without waiting for one another, each adding its tile's sums to its lanes' FP64 accumulators
    __shared__ double rows[(kThreads / 32) * NV];
    double acc = 0.0;
    int t_fail = 0, t_mx = 0, t_it = 0, t_ev = 0;
    const long stride = (long)gridDim.x * blockDim.x;
    for (long v0 = (long)blockIdx.x * blockDim.x; v0 < N3; v0 += stride) {
    const long v = v0 + threadIdx.x;
    const bool valid = v < N3;
    int r = 1, nev = 0;
    TA sums[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) sums[q] = (TA)0;
    if (valid) {
        Problem<TA> pb;
        pb.init(tab, g0[v]);
        // isotropic S0 = C0^-1 = sa I - sb J (Mandel), sa = 1/(2 m0), sb = l0 / (2 m0 (3 l0 + 2 m0))
        TA et[6], lm[6], ee[6], etr[6], sg[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            et[c] = epst[c * N3 + v];
            lm[c] = init ? (TA)0 : lam[c * N3 + v];
            ee[c] = epse[c * N3 + v];
            sg[c] = sig[c * N3 + v];
        }
        const TA ltr = lm[0] + lm[1] + lm[2];
#pragma unroll
        for (int c = 0; c < 6; ++c) etr[c] = et[c] + sa * lm[c] - (c < 3 ? sb * ltr : (TA)0);
        TA el6[6];   // the trial strain in the frame the problem is solved in
#pragma unroll
        for (int c = 0; c < 6; ++c) el6[c] = etr[c];
        pb.enter(el6, sg);
        if (fac) {   // tangent reuse: factors refreshed on request or when a step stalls
            TS F[21];
            if (!refresh) {
                load_factors(fac, N3, v, F);
            }
            int nref = 0;
            if constexpr (MR)
                r = chord_voxel<TA, TS, TF>(pb, el6, FlowMR<TA>{mrp.tpi, N3, v, tauc[v]},
                                            sg, mc, tol, maxit, ls_free, F, refresh != 0, nev, nref);
            else
                r = chord_voxel<TA, TS, TF>(pb, el6, tauc[v], sg, mc, tol, maxit, ls_free, F,
                                            refresh != 0, nev, nref);
            if (nref) {
                store_factors(fac, N3, v, F);
            }
        } else {
            if constexpr (MR)
                r = newton_voxel<TA, TF>(pb, el6, FlowMR<TA>{mrp.tpi, N3, v, tauc[v]}, sg,
                                         mc, tol, maxit, ls_free, nev);
            else
                r = newton_voxel<TA, TF>(pb, el6, tauc[v], sg, mc, tol, maxit, ls_free, nev);
        }
        pb.leave(sg);
        al_update<TA>(N3, v, et, lm, ee, etr, sg, sig, lam, pout, l0, m0, sa, sb, sa_lo, sb_lo, sad, sbd, init, sums);
    }
    if (valid) {
        const int its = r < 0 ? -r : r;
        t_fail += r < 0;
        t_mx = max(t_mx, its);
        t_it += its;
        t_ev += nev;
    }
    warp_accumulate14(sums, acc);
    }
    // flags as in k_newton
    block_solve_stats(t_fail, t_mx, t_it, t_ev, 0, flags);
    al_store_sums(acc, rows, part);
}

// The augmented-Lagrangian step of the FP32 path with stored factors. A full solver in the loop takes 168 registers, so
// 12 warps per SM: its loads (47 words a voxel, 71 with the Ma-Roters law) wait mostly uncovered. Here the loop holds
// the chord iteration's common path only (full steps with the stored factors, as many as it takes, with
// chord_voxel's operations in its order); a voxel that leaves it (a refresh or a backtracking step) is solved from
// the start by al_solve_rest, out of line. Crystal tables and factors are read again at each step, from L1 and shared
// memory, and the operands of the update after the solve, so 72 registers carry 28 warps per SM (local step per
// increment at 4 / 5 / 6 / 7 / 8 CTAs of 128 threads: 7.25 / 6.7 / 6.43 / 6.38 / 6.48 ms at 128^3, and 3.79 / 3.49 / 3.53 /
// 3.35 / 3.36 ms with the Ma-Roters law at 64^3). Per step after the first, averaged over
// an increment's iterations (first three, last quarter): 128^3 148 us (182, 128), 545 MB at 3.7 TB/s, where the full
// solver took 251 (270, 228; 97 of them on the FP64 pipe for the sums, see warp_accumulate14); with Ma-Roters at 64^3
// 59 us (83, 40), 73 (83, 65) before.
constexpr int kAlCtas = 7;
struct AlArgs {
    long N3;
    const float *epst, *epse, *tauc;
    const int32_t *g0;
    float *sig, *lam, *p;
    LocalTab<float> tab;
    MatConst mc;
    float l0, m0, sa, sb, sa_lo, sb_lo, tol, ls_free;
    double sad, sbd;
    int maxit;
    float *fac;
    MRPtr<float> mrp;
};
__device__ __forceinline__ float ld_again(const float *p) {   // a load that is not merged with an earlier one
    float x;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(p));
    return x;
}
template <bool MR, typename F> __device__ __forceinline__ auto with_law(const AlArgs &a, long v, float tc, F f) {
    if constexpr (MR) return f(FlowMR<float>{a.mrp.tpi, a.N3, v, tc});
    else return f(tc);
}
template <typename TF, bool MR>
__device__ __noinline__ int al_solve_rest(const AlArgs &a, float tol, long v, const float etr[6], float sg[6], int &nev) {
    Problem<float> pb;
    pb.init(a.tab, a.g0[v]);
    float F[21];
    load_factors((const float *)a.fac, a.N3, v, F);
    for (int c = 0; c < 6; ++c) sg[c] = a.sig[c * a.N3 + v];
    int nref = 0;
    const int r = with_law<MR>(a, v, a.tauc[v], [&](const auto &hf) {
        return chord_voxel<float, float, TF>(pb, etr, hf, sg, a.mc, tol, a.maxit, a.ls_free, F, false, nev, nref);
    });
    if (nref) store_factors(a.fac, a.N3, v, F);
    return r;
}

template <typename TF, bool MR>
__global__ void __launch_bounds__(kThreads, kAlCtas) k_al_chord(const __grid_constant__ AlArgs a, int *__restrict__ flags,
                                                          double *__restrict__ part, const int *__restrict__ skip,
                                                          const float *__restrict__ tol_dev) {
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the increment's iteration has ended
    const float tol = tol_dev != nullptr ? *tol_dev : a.tol;
    constexpr int NV = 14;
    __shared__ double rows[(kThreads / 32) * NV];
    __shared__ __align__(16) float fsh[21 * kThreads];
    double acc = 0.0;
    const long N3 = a.N3, stride = (long)gridDim.x * blockDim.x;
    int t_fail = 0, t_mx = 0, t_it = 0, t_ev = 0;
    for (long v0 = (long)blockIdx.x * blockDim.x; v0 < N3; v0 += stride) {
        const long v = v0 + threadIdx.x;
        const bool valid = v < N3;
        float sums[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) sums[q] = 0.f;
        if (valid) {
            prefetch_factors((const float *)a.fac, N3, v, fsh);
            int g = a.g0[v];
            const float tc = a.tauc[v];
            float etr[6], sg[6];
            auto trial = [&](const float et[6], const float lm[6]) {
                const float ltr = lm[0] + lm[1] + lm[2];
#pragma unroll
                for (int c = 0; c < 6; ++c) etr[c] = et[c] + a.sa * lm[c] - (c < 3 ? a.sb * ltr : 0.f);
            };
            {
                float et[6], lm[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    et[c] = a.epst[c * N3 + v];
                    lm[c] = a.lam[c * N3 + v];
                    sg[c] = a.sig[c * N3 + v];
                }
                trial(et, lm);
            }
            EvalR<float> e;
            auto residual = [&](const float s[6]) {
                asm volatile("" : "+r"(g));   // the tables are read again: nothing of them is held between steps
                Problem<float> pb;
                pb.init(a.tab, g);
                with_law<MR>(a, v, tc, [&](const auto &hf) { evaluate_r(pb, etr, hf, drcp(tc), s, a.mc, e); });
            };
            residual(sg);
            int r = 0, nev = 1;
            float prev = -1.f;
            for (int it = 1; r == 0; ++it) {
                float d[6];
                {
                    float F[21];
                    prefetched_factors(fsh, F);
                    ldl_apply<float, float>(F, e.r, d);
                }
                float rd = 0.f, dn = 0.f, sn = 0.f;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    rd += e.r[i] * d[i];
                    dn += d[i] * d[i];
                    sn += sg[i] * sg[i];
                }
                dn = dsqrt(dn);
                const float scale = dsqrt(sn) + tc;
                if (dn <= tol * scale && rd >= 0.f) {
#pragma unroll
                    for (int i = 0; i < 6; ++i) sg[i] -= d[i];
                    r = it;
                    break;
                }
                if (it >= a.maxit || rd <= 0.f || (prev > 0.f && dn > 0.25f * prev)) break;
                const float phi0 = e.phi;
#pragma unroll
                for (int i = 0; i < 6; ++i) sg[i] -= d[i];
                residual(sg);
                ++nev;
                if (!(e.phi <= phi0 - 1e-4f * rd || dn <= a.ls_free * scale)) break;
                if (dn <= tol * scale) r = it;
                prev = dn;
            }
            if (r == 0) {   // off the common path
                float s6[6], t6[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) t6[c] = etr[c];
                r = al_solve_rest<TF, MR>(a, tol, v, t6, s6, nev);
#pragma unroll
                for (int c = 0; c < 6; ++c) sg[c] = s6[c];
            }
            {
                float et[6], lm[6], ee[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    et[c] = ld_again(a.epst + c * N3 + v);
                    lm[c] = ld_again(a.lam + c * N3 + v);
                    ee[c] = a.epse[c * N3 + v];
                }
                trial(et, lm);
                al_update<float>(N3, v, et, lm, ee, etr, sg, a.sig, a.lam, a.p, a.l0, a.m0, a.sa, a.sb, a.sa_lo, a.sb_lo,
                                 a.sad, a.sbd, 0, sums);
            }
            const int its = r < 0 ? -r : r;
            t_fail += r < 0;
            t_mx = max(t_mx, its);
            t_it += its;
            t_ev += nev;
        }
        warp_accumulate14(sums, acc);
    }
    block_solve_stats(t_fail, t_mx, t_it, t_ev, 0, flags);
    al_store_sums(acc, rows, part);
}

// Control of the augmented-Lagrangian iteration after each local step: block q adds up sum q of the step's blocks, in a
// fixed order, and the last block to finish runs the stopping tests and, where the iteration goes on, forms the
// macroscopic strain correction on the stress-controlled components from <lam> and the next local tolerance. The host
// queues iterations in batches and reads the control block once per batch (a read after every iteration cost about 25 us
// of a 145 us iteration at 64^3). One block per sum: 1000 partial sums of each are 900 FP64-pipe cycles of an SM.
__global__ void __launch_bounds__(256) k_al_control(AlCtl *c, const double *__restrict__ part, int nparts,
                                                    const int32_t *__restrict__ flags, AlCtlParams p, int first) {
    pdl_wait();
    __shared__ double red[32];
    const int lane = threadIdx.x & 31;
    // every operand is fetched at once: the partial sums, and by warp 0 the control block
    const bool ended = c->done != 0;
    double dEl = 0.0, tol_loc = 0.0;
    int it = 0, nmax = 0, nfail = 0, mx = 0;
    if (threadIdx.x < 32) {
        dEl = lane < 6 ? c->dE[lane] : 0.0;
        tol_loc = c->tol_loc;
        it = c->it + (first ? 0 : 1);
        nmax = c->nmax;
        nfail = flags[0];
        mx = flags[1];
    }
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 1024) {
        double x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = i + 256 * q < nparts ? part[(long)blockIdx.x * nparts + i + 256 * q] : 0.0;
        s += (x[0] + x[1]) + (x[2] + x[3]);
    }
    if (ended) return;
    s = block_sum(s, red);
    if (threadIdx.x >= 32) return;
    unsigned ticket = 0;
    if (lane == 0) {
        c->sum[blockIdx.x] = s;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;\n" : "=r"(ticket) : "l"(&c->ticket) : "memory");
    }
    if (__shfl_sync(0xffffffffu, ticket, 0) != gridDim.x - 1) return;
    __syncwarp();   // lane 0's acquire orders the other lanes' reads of the sums (a shuffle orders no memory)
    const double hl = lane < 14 ? __ldcg(c->sum + lane) * p.inv_n3 : 0.0;   // the means
    const unsigned all = 0xffffffffu;
    // lanes 0-5: component i of |E|^2, |<lam>|^2 and its stress-controlled part, summed over lanes 0-7
    const double mi = __shfl_sync(all, hl, 2 + (lane & 7)), sig = __shfl_sync(all, hl, 8 + (lane & 7));
    const double Ei = lane < 6 ? p.E[lane] + dEl : 0.0, ml = lane < 6 ? mi : 0.0;
    double En = Ei * Ei, mn = ml * ml, mu_n = lane == 2 ? 0.0 : mn;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        En += __shfl_xor_sync(all, En, o);
        mn += __shfl_xor_sync(all, mn, o);
        mu_n += __shfl_xor_sync(all, mu_n, o);
    }
    // lane 0: |<lam>|, 1: |E|, 2 and 3: the RMS gaps, 4: the stress-controlled |<lam>|; then lanes 0-2 their quotients
    const double g0 = __shfl_sync(all, hl, 0), g1 = __shfl_sync(all, hl, 1);
    const double root = sqrt(lane == 0 ? mn : lane == 1 ? En : lane == 2 ? g0 : lane == 3 ? g1 : mu_n);
    const double den = fmax(__shfl_sync(all, root, 0), p.tau0), nE = fmax(__shfl_sync(all, root, 1), 1e-6);
    const double q = __shfl_sync(all, root, 2 + (lane < 3 ? lane : 2)) / (lane == 0 ? nE : den);
    const double ecmp = __shfl_sync(all, q, 0), elam = __shfl_sync(all, q, 1), ebc = __shfl_sync(all, q, 2);
    const double m0 = __shfl_sync(all, mi, 0), m1 = __shfl_sync(all, mi, 1);
    int status = 0, done = 0, conv = 0;
    if (nfail != 0) {
        status = EVP_ERR_NEWTON;
        done = 1;
    } else if (!first) {
        if (!isfinite(ecmp) || !isfinite(elam)) {
            status = EVP_ERR_NONFINITE;
            done = 1;
        } else if (ecmp <= p.tol && elam <= p.tol && ebc <= p.tol && tol_loc <= p.ntol) {
            conv = 1;
            done = 1;
        } else if (it >= p.max_iter) {
            done = 1;
        }
    }
    if (lane < 6) {
        c->mean[lane] = sig;
        const double d = lane == 0 ? p.cb * m1 - p.ca * m0 : lane == 1 ? p.cb * m0 - p.ca * m1 : lane == 2 ? 0.0 : -p.cs * mi;
        if (!done) c->dE[lane] = dEl + d;
    }
    if (lane == 0) {
        c->it = it;
        c->nmax = max(nmax, mx);
        c->nfail = nfail;
        c->status = status;
        c->conv = conv;
        if (!first && nfail == 0) {   // of the last iteration whose local problems were all solved
            c->ecmp = ecmp;
            c->elam = elam;
            c->ebc = ebc;
        }
        if (!done && !first && p.eta > 0.0) {
            c->tol_loc = fmax(p.ntol, p.eta * fmax(ecmp, elam));
            c->tol_loc_f = (float)c->tol_loc;
        }
        c->ticket = 0u;
        c->done = done;
    }
}

// Start of an increment: tau_c from the densities at t (frozen over the increment) and the
// predictor eps_tr = eps_e^t + (r * deps_prev  |  dE).
template <typename TA>
__global__ void __launch_bounds__(256) k_predictor(long N3, const TA *__restrict__ epse, const TA *__restrict__ deps,
                                                  const TA *__restrict__ rho, TA *__restrict__ epst, TA *__restrict__ tauc,
                                                  MatConst mc, TA r, int use_field, TA d0, TA d1, TA d2, TA d3, TA d4,
                                                  TA d5) {
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N3) return;
    // all loads first; arithmetic in the field precision (the FP32 path keeps the FP64 pipe out)
    TA rr[12], ee[6], dd[6];
#pragma unroll
    for (int a = 0; a < 12; ++a) rr[a] = rho[a * N3 + v];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        ee[c] = epse[c * N3 + v];
        dd[c] = use_field ? deps[c * N3 + v] : (TA)0;
    }
    TA rf = (TA)0;
#pragma unroll
    for (int a = 0; a < 12; ++a) rf += rr[a];
    tauc[v] = (TA)mc.tau0 + (TA)mc.alpha_mu_b * sqrt(rf);
    const TA dE[6] = {d0, d1, d2, d3, d4, d5};
#pragma unroll
    for (int c = 0; c < 6; ++c) epst[c * N3 + v] = ee[c] + (use_field ? r * dd[c] : dE[c]);
}

// k = sum of the 12 densities as a double. FP64 fields: summed in FP64. FP32 fields: summed as an unevaluated
// float pair (two-sum per term, the rounding errors added in float) and converted once: the result is within a few
// units of 2^-48 of the exact sum of the FP32 densities (the FP64 running sum is exact for them too, or nearly),
// with 2 FP64-pipe operations instead of 24 on a pipe that runs at 1/64 of the FP32 rate.
__device__ __forceinline__ double density_total(const double r[12]) {
    double kk = 0.0;
#pragma unroll
    for (int a = 0; a < 12; ++a) kk += r[a];
    return kk;
}
__device__ __forceinline__ double density_total(const float r[12]) {
    float hi = r[0], lo = 0.f;
#pragma unroll
    for (int a = 1; a < 12; ++a) {
        float s, e;
        two_sum_f(hi, r[a], s, e);
        hi = s;
        lo = __fadd_rn(lo, e);
    }
    return (double)hi + (double)lo;
}

// After convergence (a7): advance eps_p, eps_e, the strain increment and the densities with
// the converged shear rates; k = rho_tot as a double.
template <typename TA>
__global__ void __launch_bounds__(kThreads) k_state_update(long N3, const TA *__restrict__ sig, const TA *__restrict__ tauc,
                                                          const int32_t *__restrict__ g0, const TA *__restrict__ Mtab,
                                                          const TA *__restrict__ epst, TA *__restrict__ epse,
                                                          TA *__restrict__ epsp, TA *__restrict__ deps, TA *__restrict__ rho,
                                                          double *__restrict__ kf, MatConst mc) {
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N3) return;
    // every operand is loaded before any arithmetic, so a thread has all its requests in flight at once
    const int g = g0[v];
    TA sg[6], tr[6], eo[6], po[6], r[12];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        sg[c] = sig[c * N3 + v];
        tr[c] = epst[c * N3 + v];
        eo[c] = epse[c * N3 + v];
        po[c] = epsp[c * N3 + v];
    }
#pragma unroll
    for (int a = 0; a < 12; ++a) r[a] = rho[a * N3 + v];
    const TA tcv = tauc[v];
    const TA *M = Mtab + 72 * (long)g;
    const TA inv_tc = (TA)1 / tcv;
    const TA g0r = (TA)mc.gdot0, dt = (TA)mc.dt;
    TA ep[6] = {0, 0, 0, 0, 0, 0};
    TA agd[12];
#pragma unroll
    for (int a = 0; a < 12; ++a) {
        TA m[6], tau = (TA)0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            m[i] = __ldg(M + 6 * a + i);
            tau += m[i] * sg[i];
        }
        const TA x = tau * inv_tc, ax = fabs(x);
        const TA p10 = pow_nm1(ax, mc) * ax;
        const TA gd = x < (TA)0 ? -g0r * p10 : g0r * p10;
        agd[a] = fabs(gd);
#pragma unroll
        for (int i = 0; i < 6; ++i) ep[i] += m[i] * gd;
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        epsp[c * N3 + v] = po[c] + dt * ep[c];
        deps[c * N3 + v] = tr[c] - eo[c];
        epse[c * N3 + v] = tr[c] - dt * ep[c];
    }
    // Kocks-Mecking update in the field precision
    TA rf = (TA)0;
#pragma unroll
    for (int a = 0; a < 12; ++a) rf += r[a];
    const TA srf = sqrt(rf), k1 = (TA)mc.k1, k2 = (TA)mc.k2;
    TA nr[12];
#pragma unroll
    for (int a = 0; a < 12; ++a) {
        nr[a] = r[a] + dt * (k1 * srf - k2 * r[a]) * agd[a];
        rho[a * N3 + v] = nr[a];
    }
    kf[v] = density_total(nr);
}

template <typename TA>
__global__ void k_total_strain(long N3, const TA *__restrict__ epse, const TA *__restrict__ epsp, TA *__restrict__ eps) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 6 * N3) eps[i] = epse[i] + epsp[i];
}

template <typename TA> TA ls_free_of() { return sizeof(TA) == 4 ? (TA)1e-3 : (TA)1e-6; }

}  // namespace

// Each launcher runs the power-law kernels, or their Ma-Roters instantiations when mrp.tpi is set.
template <typename TA, typename F> cudaError_t by_law(MRPtr<TA> mrp, F &&go) {
    if (mrp.tpi) go(std::true_type{});
    else go(std::false_type{});
    return cudaGetLastError();
}

template <typename TA>
cudaError_t newton_field(long N3, const TA *epst, const TA *tauc, const int32_t *g0, TA *sig, LocalTab<TA> tab,
                         MatConst mc, double tol, int maxit, int solve_fp64, int *flags,
                         cudaStream_t s, const int *skip, const TA *tol_dev, MRPtr<TA> mrp) {
    const int blocks = (int)((N3 + kThreads - 1) / kThreads);
    return by_law(mrp, [&](auto law) {
        constexpr bool MR = decltype(law)::value;
        if (solve_fp64)
            k_newton<TA, double, MR><<<blocks, kThreads, 0, s>>>(N3, epst, tauc, g0, sig, tab, mc, (TA)tol,
                                                                 maxit, ls_free_of<TA>(), flags, skip, tol_dev, mrp);
        else
            k_newton<TA, TA, MR><<<blocks, kThreads, 0, s>>>(N3, epst, tauc, g0, sig, tab, mc, (TA)tol, maxit,
                                                             ls_free_of<TA>(), flags, skip, tol_dev, mrp);
    });
}

template <typename TA>
cudaError_t newton_chord_field(long N3, const TA *epst, const TA *tauc, const int32_t *g0, TA *sig, LocalTab<TA> tab,
                               void *fac, MatConst mc, double tol, int maxit, int solve_fp64,
                               int force_refresh, int *flags, int32_t *wl, int nsm, cudaStream_t s, const int *skip,
                               const TA *tol_dev, MRPtr<TA> mrp, int two_step) {
    const int blocks = (int)((N3 + kThreads - 1) / kThreads);
    if (!force_refresh && wl) {
        // flags[10] counts the listed voxels; pass 2 reads it on the device (no host round trip). Inside the
        // fixed-point loop (skip set) the kernels run as one programmatic-launch chain: the count starts at zero
        // from the increment's flag reset and is reset by each iteration's control block (fpctl.cuh), so no
        // memset breaks the chain; outside it the count is reset here.
        const bool pdl = skip != nullptr;
        if (!pdl) {
            cudaError_t e = cudaMemsetAsync(flags + 10, 0, 2 * sizeof(int), s);
            if (e != cudaSuccess) return e;
        }
        const int rb = std::min(blocks, nsm * (sizeof(TA) == 4 ? 3 : 2));
        cudaError_t err = cudaSuccess;
        by_law(mrp, [&](auto law) {
            constexpr bool MR = decltype(law)::value;
            if (two_step)
                err = launch_k(pdl, k_chord_first<TA, TA, MR, true>, dim3(blocks), dim3(kThreads), 0, s, N3, epst, tauc,
                               g0, sig, tab, (const TA *)fac, mc, (TA)tol, ls_free_of<TA>(), flags, wl, skip,
                               tol_dev, mrp);
            else
                err = launch_k(pdl, k_chord_first<TA, TA, MR, false>, dim3(blocks), dim3(kThreads), 0, s, N3, epst,
                               tauc, g0, sig, tab, (const TA *)fac, mc, (TA)tol, ls_free_of<TA>(), flags, wl,
                               skip, tol_dev, mrp);
            if (err != cudaSuccess) return;
            if (solve_fp64)
                err = launch_k(pdl, k_chord_rest<TA, TA, double, MR>, dim3(rb), dim3(kThreads), 0, s, N3, epst, tauc,
                               g0, sig, tab, (TA *)fac, mc, (TA)tol, maxit, ls_free_of<TA>(), flags,
                               (const int32_t *)wl, skip, tol_dev, mrp);
            else
                err = launch_k(pdl, k_chord_rest<TA, TA, TA, MR>, dim3(rb), dim3(kThreads), 0, s, N3, epst, tauc, g0,
                               sig, tab, (TA *)fac, mc, (TA)tol, maxit, ls_free_of<TA>(), flags,
                               (const int32_t *)wl, skip, tol_dev, mrp);
        });
        return err != cudaSuccess ? err : cudaGetLastError();
    }
    // factors stored in the field precision; factorised in FP64 unless the FP32 solve is asked for
    return by_law(mrp, [&](auto law) {
        constexpr bool MR = decltype(law)::value;
        if (solve_fp64)
            k_newton_chord<TA, TA, double, MR><<<blocks, kThreads, 0, s>>>(N3, epst, tauc, g0, sig, tab,
                                                                           (TA *)fac, mc, (TA)tol, maxit,
                                                                           ls_free_of<TA>(), force_refresh, flags,
                                                                           skip, tol_dev, mrp);
        else
            k_newton_chord<TA, TA, TA, MR><<<blocks, kThreads, 0, s>>>(N3, epst, tauc, g0, sig, tab, (TA *)fac,
                                                                       mc, (TA)tol, maxit, ls_free_of<TA>(),
                                                                       force_refresh, flags, skip, tol_dev, mrp);
    });
}

int al_blocks(long N3) { return (int)((N3 + kThreads - 1) / kThreads); }
int al_grid(long N3, int nsm, int tsize, int chord) {
    return std::min(al_blocks(N3), std::max(nsm, 1) * (chord ? kAlCtas : tsize == 4 ? 3 : 2));
}

cudaError_t newton_field_df(long N3, const double *epst, const double *tauc, const int32_t *g0, double *sig,
                            LocalTab<double> tab, MatConst mc, double tol, int maxit, int *flags, cudaStream_t s, const int *skip,
                            const double *tol_dev) {
    const int blocks = (int)((N3 + kThreads - 1) / kThreads);
    k_newton_df<<<blocks, kThreads, 0, s>>>(N3, epst, tauc, g0, sig, tab, mc, tol, maxit, flags,
                                            skip, tol_dev);
    return cudaGetLastError();
}

int al_chord(size_t tsize, const void *fac, int refresh) { return tsize == 4 && fac != nullptr && !refresh; }

cudaError_t al_control(AlCtl *ctl, const double *part, int nparts, const int32_t *flags, const AlCtlParams &p, int first,
                       cudaStream_t s) {
    return launch_k(true, k_al_control, dim3(14), dim3(256), 0, s, ctl, part, nparts, flags, p, first);
}

template <typename TA>
cudaError_t al_local(long N3, const TA *epst, const TA *epse, const TA *tauc, const int32_t *g0, TA *sig, TA *lam, TA *p,
                     LocalTab<TA> tab, MatConst mc, double lam0, double mu0, double tol,
                     int maxit, int solve_fp64, int init, int *flags, double *part, void *fac, int refresh,
                     cudaStream_t s, int nsm, MRPtr<TA> mrp, const int *skip, const TA *tol_dev, int *nparts) {
    const int chord = al_chord(sizeof(TA), fac, refresh);
    const int blocks = *nparts = al_grid(N3, nsm, (int)sizeof(TA), chord);
    const double sad = 1.0 / (2.0 * mu0), sbd = lam0 / (2.0 * mu0 * (3.0 * lam0 + 2.0 * mu0));
    const TA sa = (TA)sad, sb = (TA)sbd;
    const TA sa_lo = (TA)(sad - (double)sa), sb_lo = (TA)(sbd - (double)sb);   // S0 = (sa + sa_lo) I - (sb + sb_lo) J
    cudaError_t err = cudaSuccess;
    by_law(mrp, [&](auto law) {
        constexpr bool MR = decltype(law)::value;
        if constexpr (sizeof(TA) == 4) {
            if (chord) {
                const AlArgs a{N3, epst, epse, tauc, g0, sig, lam, p, tab, mc, (TA)lam0, (TA)mu0, sa, sb, sa_lo, sb_lo,
                               (TA)tol, ls_free_of<TA>(), sad, sbd, maxit, (TA *)fac, mrp};
                err = solve_fp64 ? launch_k(true, k_al_chord<double, MR>, dim3(blocks), dim3(kThreads), 0, s, a, flags,
                                            part, skip, tol_dev)
                                 : launch_k(true, k_al_chord<float, MR>, dim3(blocks), dim3(kThreads), 0, s, a, flags,
                                            part, skip, tol_dev);
                return;
            }
        }
        auto go = [&](auto kernel) {
            err = launch_k(true, kernel, dim3(blocks), dim3(kThreads), 0, s, N3, epst, epse, tauc, g0, sig, lam, p, tab,
                           mc, (TA)lam0, (TA)mu0, sa, sb, sa_lo, sb_lo, sad, sbd, (TA)tol, maxit, ls_free_of<TA>(), init,
                           flags, part, (TA *)fac, refresh, mrp, skip, tol_dev);
        };
        if (solve_fp64) go(k_al_local<TA, TA, double, MR>);
        else go(k_al_local<TA, TA, TA, MR>);
    });
    return err != cudaSuccess ? err : cudaGetLastError();
}

template <typename TA>
cudaError_t predictor(long N3, const TA *epse, const TA *deps, const TA *rho, TA *epst, TA *tauc, MatConst mc,
                      double r, const double *dE6, int use_field, cudaStream_t s) {
    const int blocks = (int)((N3 + 255) / 256);
    // the extrapolation ratio and the uniform guess rounded to the field precision once, here
    k_predictor<TA><<<blocks, 256, 0, s>>>(N3, epse, deps, rho, epst, tauc, mc, (TA)r, use_field, (TA)dE6[0],
                                           (TA)dE6[1], (TA)dE6[2], (TA)dE6[3], (TA)dE6[4], (TA)dE6[5]);
    return cudaGetLastError();
}

template <typename TA>
cudaError_t state_update(long N3, const TA *sig, const TA *tauc, const int32_t *g0, const TA *Mtab, TA *epst,
                         TA *epse, TA *epsp, TA *deps, TA *rho, double *k, MatConst mc, cudaStream_t s) {
    const int blocks = (int)((N3 + kThreads - 1) / kThreads);
    k_state_update<TA><<<blocks, kThreads, 0, s>>>(N3, sig, tauc, g0, Mtab, epst, epse, epsp, deps, rho, k, mc);
    return cudaGetLastError();
}

template <typename TA> cudaError_t total_strain(long N3, const TA *epse, const TA *epsp, TA *eps, cudaStream_t s) {
    const long n = 6 * N3;
    k_total_strain<TA><<<(int)((n + 255) / 256), 256, 0, s>>>(N3, epse, epsp, eps);
    return cudaGetLastError();
}

#define EVP_INST(TA)                                                                                              \
    template cudaError_t newton_field<TA>(long, const TA *, const TA *, const int32_t *, TA *, LocalTab<TA>,      \
                                          MatConst, double, int, int, int *, cudaStream_t,           \
                                          const int *, const TA *, MRPtr<TA>);                                   \
    template cudaError_t newton_chord_field<TA>(long, const TA *, const TA *, const int32_t *, TA *, LocalTab<TA>, \
                                                void *, MatConst, double, int, int, int, int *,       \
                                                int32_t *, int, cudaStream_t, const int *, const TA *, MRPtr<TA>, int); \
    template cudaError_t al_local<TA>(long, const TA *, const TA *, const TA *, const int32_t *, TA *, TA *, TA *, \
                                      LocalTab<TA>, MatConst, double, double, double, int, int, \
                                      int, int *, double *, void *, int, cudaStream_t, int, MRPtr<TA>, const int *, \
                                      const TA *, int *);                                                        \
    template cudaError_t predictor<TA>(long, const TA *, const TA *, const TA *, TA *, TA *, MatConst, double,    \
                                       const double *, int, cudaStream_t);                                        \
    template cudaError_t state_update<TA>(long, const TA *, const TA *, const int32_t *, const TA *, TA *, TA *,  \
                                          TA *, TA *, TA *, double *, MatConst, cudaStream_t);                    \
    template cudaError_t total_strain<TA>(long, const TA *, const TA *, TA *, cudaStream_t);
EVP_INST(float)
EVP_INST(double)
#undef EVP_INST

}  // namespace evp
