// Fixed-point control of the basic scheme, on the device (Sec. 2.1 iteration with the mixed boundary
// conditions). After an iteration's z pass has written its partial sums, one warp sums them (in a fixed
// order) into sum |xi.sigma_hat|^2, tests that and the mean stress against the tolerance and computes the
// correction dE_k of the macroscopic strain on the stress-controlled components. The inverse transform adds it to
// the zero-frequency term of the Green-operator output, which the z pass leaves at zero: after the z pass's own inverse
// transform that is the (ky, kx) = (0, 0) entry of every z plane. The host queues iterations in batches and reads this block once per
// batch; once `done` is set, the kernels of the iterations still queued return at once.
//
// The control runs alone at the end of the z pass, so it is a chain of latencies that every iteration waits for. It
// therefore tests squares (no square root, no division: an FP64 one is a chain of some twenty dependent operations on
// this GPU), lets one lane per component do the component's work, and the ticket that selects its block is taken
// before the inverse transform; the next local tolerance, which does need the residuals themselves, is one extra
// block of the inverse transform (fp_next_tolerance). At 32^3 the control took 8.4 us of a 15 us z pass as one thread's
// chain after every block's last store, with the correction written into the spectrum.
#pragma once
#include <cstdint>

#include "../../include/evp.h"
#include "common.cuh"

namespace evp {

struct FpCtl {
    int done, it, conv, status, nmax, nfail;
    unsigned ticket;    // z-pass blocks past their partial sum in this iteration (the last one runs the control)
    int pad;
    double dE[6];       // macroscopic strain increment so far
    double corr[6];     // its correction in this iteration
    double tol_loc;     // local-solve tolerance of the next iteration (see evp_config.newton_adapt)
    float tol_loc_f;
};

// tol2, tau02: the squares of the tolerance and of the floor of |<sigma>|; n6 = N^6; ca, cb, cs: the mixed-BC
// correction's a/det, b/det and 1/(2 mu0).
struct FpCtlParams {
    double n6, tau02, tol2, ca, cb, cs;
    int max_iter;
};

// What the z pass needs to run the control in its last block (ctl == nullptr: no control).
struct ZCtl {
    FpCtl *ctl;
    int32_t *flags;         // flags[0] failed local solves, flags[1] max local iterations, flags[10] the local
                            // solve's work-list count, flags[11] its pass 1's two-step count (both reset here for
                            // the next iteration)
    double *scal;           // scal[0..5] mean stress (written by the z pass), scal[6] residual sum
    FpCtlParams p;
};

// A z-pass block's ticket, taken by the thread that wrote its partial sum. The release orders that sum (and, after the
// block's barrier, the mean stress) before the ticket, the acquire orders the last block's reads after it; a full
// fence (__threadfence) would order every outstanding store.
__device__ __forceinline__ unsigned fp_take_ticket(const ZCtl &z) {
    unsigned t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;\n" : "=r"(t) : "l"(&z.ctl->ticket) : "memory");
    return t;
}

// The 32 lanes of one warp call this with the iteration's nparts partial sums. Between fp_take_ticket and this call lies
// a barrier of the block (those of the inverse transform) or of the warp, which passes the acquire on to the other lanes.
__device__ __forceinline__ void fp_control_warp(const ZCtl &z, const double *__restrict__ part, int nparts) {
    FpCtl *c = z.ctl;
    const FpCtlParams &p = z.p;
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // every operand is fetched at once: the mean by lanes 0-5, the counters by lanes 8-11
    const double m = lane < 6 ? __ldcg(z.scal + lane) : 0.0;
    const int *ip = lane == 8 ? &c->it : lane == 9 ? &c->nmax : lane == 10 ? z.flags : z.flags + 1;
    const int iv = lane >= 8 && lane < 12 ? __ldcg(ip) : 0;
    const double dE = lane < 6 ? __ldcg(c->dE + lane) : 0.0;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = lane; i < nparts; i += 128)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i + 32 * q < nparts) a[q] += __ldcg(part + i + 32 * q);
    double s = (a[0] + a[1]) + (a[2] + a[3]);
    double mn = m * m, mu_n = lane == 2 ? 0.0 : mn;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(all, s, o);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        mn += __shfl_xor_sync(all, mn, o);
        mu_n += __shfl_xor_sync(all, mu_n, o);
    }
    mn = __shfl_sync(all, mn, 0);       // lanes 0-7 hold |<sigma>|^2 and its stress-controlled part
    mu_n = __shfl_sync(all, mu_n, 0);
    const int it = __shfl_sync(all, iv, 8) + 1, nfail = __shfl_sync(all, iv, 10);
    const int nmax = max(__shfl_sync(all, iv, 9), __shfl_sync(all, iv, 11));
    const double m0 = __shfl_sync(all, m, 0), m1 = __shfl_sync(all, m, 1);
    const double den2 = fmax(mn, p.tau02);
    int status = 0, done = 0, conv = 0;
    if (nfail != 0) {
        status = EVP_ERR_NEWTON;
        done = 1;
    } else if (!isfinite(s) || !isfinite(mn)) {
        status = EVP_ERR_NONFINITE;
        done = 1;
    } else if (s <= p.tol2 * den2 * p.n6 && mu_n <= p.tol2 * den2) {   // err_eq <= tol and err_bc <= tol
        conv = 1;
        done = 1;
    } else if (it >= p.max_iter) {
        done = 1;
    }
    if (!done && lane < 6) {
        const double d = lane == 0 ? p.cb * m1 - p.ca * m0 : lane == 1 ? p.cb * m0 - p.ca * m1 : lane == 2 ? 0.0 : -p.cs * m;
        c->dE[lane] = dE + d;
        c->corr[lane] = d;
    }
    if (lane == 0) {
        z.scal[6] = s;
        z.flags[10] = 0;   // the next iteration's first local-solve pass counts its work list from zero,
        z.flags[11] = 0;   // and its voxels accepted after two steps
        c->it = it;
        c->nmax = nmax;
        c->nfail = nfail;
        c->status = status;
        c->conv = conv;
        c->ticket = 0u;
        c->done = done;
    }
}

// Control block of the augmented-Lagrangian iteration (k_al_control) and its constants: the stopping tolerance, the
// macroscopic strain at the start of the increment, ca, cb, cs as in FpCtlParams for its reference medium.
struct AlCtl {
    int done, it, conv, status, nmax, nfail;
    double dE[6];           // macroscopic strain increment: of the last iteration that ran, or for the next
    double mean[6];         // mean stress
    double ecmp, elam, ebc; // residuals
    double sum[14];         // the local step's sums (see k_al_local)
    unsigned ticket;        // blocks of the control that have stored theirs
    double tol_loc;         // local-solve tolerance of the next iteration
    float tol_loc_f;
};
struct AlCtlParams {
    double inv_n3, tau0, tol, ntol, eta, ca, cb, cs, E[6];
    int max_iter;
};

// What the inverse transform of an iteration takes from the control: with ctl (basic scheme) the correction of the
// zero-frequency term, n3 = N^3 times FpCtl.corr (the transforms are unnormalised); with dadd (augmented Lagrangian) the six
// offsets of its last pass in device memory.
struct InvCtl {
    FpCtl *ctl;
    const double *scal;     // as ZCtl.scal
    double n3, tau0, ntol, eta;
    const double *dadd;
};

// Local-solve tolerance of the next iteration: eta times the larger residual, at least ntol.
__device__ __forceinline__ void fp_next_tolerance(const InvCtl &v) {
    if (!(v.eta > 0.0)) return;
    double mn = 0.0, mu_n = 0.0;
    for (int i = 0; i < 6; ++i) {
        const double m = v.scal[i];
        mn += m * m;
        if (i != 2) mu_n += m * m;
    }
    const double den = fmax(sqrt(mn), v.tau0);
    const double err_eq = sqrt(v.scal[6]) / (v.n3 * den), err_bc = sqrt(fmax(mu_n, 0.0)) / den;
    const double tl = fmax(v.ntol, v.eta * fmax(err_eq, err_bc));
    v.ctl->tol_loc = tl;
    v.ctl->tol_loc_f = (float)tl;
}

}  // namespace evp
