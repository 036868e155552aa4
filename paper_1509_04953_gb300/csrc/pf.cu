// Active-set multi-grain Allen-Cahn step (Sec. 2.4, Eqs. TotalFreeEnergy, GBEnergyDensity,
// StoredEnergyDensity, PFGoverning; sparse storage after the cited Gruber / Vedantam technique).
//
// Grid-nondimensional form (lengths dx, energies omega_gb/dx, time dx^2/(M omega_gb)):
//   m = 6/l, kappa = 3l/4, gamma = 3/2,  E' = zeta mu b^2 rho_tot dx / omega_gb
//   eta_i <- eta_i - L dt [ m (eta_i^3 - eta_i + 2 gamma eta_i (S2 - eta_i^2)) - kappa lap(eta_i)
//                            + (i deformed: 2E' eta_i R/S^2 | i recrystallised: -2E' eta_i D/S^2) ]
// with S2 = D + R the local sum of eta^2 over deformed (D, ids < G) and recrystallised (R)
// grains and a periodic 7-point Laplacian. Each voxel stores up to K (id, eta) pairs sorted by
// id (-1 = empty). Candidates at a voxel are the ids present there or at its six neighbours;
// values below `drop` are discarded, the K largest kept (ties to the smaller id) and the grain
// id is the argmax. This file is compiled without FMA contraction so that, in FP64, each value
// is rounded exactly as the plain formula above prescribes.
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace evp {

namespace {

constexpr int KM = 8;   // compile-time capacity of the active set (runtime K <= KM)
constexpr int kPF = 128;

struct Nbr {
    long q[7];   // self, x-, x+, y-, y+, z-, z+
};

// n is a power of two (checked at init): coordinates and periodic wraps by masks and shifts
__device__ __forceinline__ Nbr neighbours(int n, long v) {
    const int lg = __ffs(n) - 1;
    const long msk = n - 1;
    const int x = (int)(v & msk), y = (int)((v >> lg) & msk), z = (int)(v >> (2 * lg));
    const long nn = (long)n * n;
    Nbr b;
    b.q[0] = v;
    b.q[1] = v - x + ((x - 1) & msk);
    b.q[2] = v - x + ((x + 1) & msk);
    b.q[3] = v + (long)(((y - 1) & msk) - y) * n;
    b.q[4] = v + (long)(((y + 1) & msk) - y) * n;
    b.q[5] = v + (long)(((z - 1) & msk) - z) * nn;
    b.q[6] = v + (long)(((z + 1) & msk) - z) * nn;
    return b;
}

constexpr int kEmpty = 0x7fffffff;

// Asynchronous global -> shared copy of B bytes (cp.async; completion by commit / wait groups).
template <int B> __device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (B == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}


// x == 0 (FP64: on the integer pipe)
__device__ __forceinline__ bool pf_zero(float x) { return x == 0.f; }
__device__ __forceinline__ bool pf_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }

// What the update of a point's candidates needs of the point: the driving force Ep, the sums over its own list, and
// whether they are all finite.
template <typename T> struct PFLocal {
    T Ep, S2, D, R, Ssum;
    bool finite;
    __device__ __forceinline__ void close() {
        Ssum = D + R;
        finite = Ep - Ep == (T)0 && S2 - S2 == (T)0;   // S2 bounds D and R
    }
};

// New value of a candidate from its value e0 here and the sum nb of its neighbours' values. Every shortcut gives the
// value of the plain formula: with e0 = 0 (a candidate of the neighbours only; most candidates) all terms but
// the Laplacian's are zero, and a driving force whose numerator is zero (no recrystallised, or no deformed, material at
// the point) needs no quotient. An FP64 quotient is some thirty operations of a pipe that bounds the FP64 step.
template <typename T>
__device__ __forceinline__ T pf_value(bool deformed, T e0, T nb, const PFLocal<T> &pl, T m, T kap, T gam, T Ldt) {
    if (pf_zero(e0) && pl.finite) return Ldt * (kap * nb);
    const T lap = nb - (T)6 * e0;
    const T df0 = m * (e0 * e0 * e0 - e0 + (T)2 * gam * e0 * (pl.S2 - e0 * e0));
    T ddef = (T)0;
    const T other = deformed ? pl.R : pl.D;
    if (pl.Ssum > (T)1e-12 && !(pf_zero(other) && pl.finite)) {
        ddef = (deformed ? (T)2 : -(T)2) * pl.Ep * e0 * other;
        if (!pf_zero(ddef)) ddef = ddef / (pl.Ssum * pl.Ssum);
    }
    return e0 - Ldt * (df0 - kap * lap + ddef);
}

template <typename T>
__global__ void __launch_bounds__(kPF) k_pf(int n, const int32_t *__restrict__ ids, const T *__restrict__ eta,
                                           int32_t *__restrict__ ids2, T *__restrict__ eta2, int32_t *__restrict__ gout,
                                           const double *__restrict__ kf, PFConst pc, int32_t *__restrict__ overflow) {
    const long N3 = (long)n * n * n;
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N3) return;
    const int K = pc.K, G = pc.G;
    const Nbr nb = neighbours(n, v);
    T m, kap, gam, Ldt, drop;   // in the field precision (no FP64 conversions on the FP32 path)
    if constexpr (sizeof(T) == 4) { m = pc.m_f; kap = pc.kappa_f; gam = pc.gam_f; Ldt = pc.L_dt_f; drop = pc.drop_f; }
    else { m = pc.m; kap = pc.kappa; gam = pc.gam; Ldt = pc.L_dt; drop = pc.drop; }
    // local sums over the voxel's own list, ascending id
    PFLocal<T> pl{(T)(pc.Escale * kf[v]), (T)0, (T)0, (T)0};
    for (int j = 0; j < K; ++j) {
        const int id = ids[j * N3 + v];
        if (id < 0) break;
        const T e = eta[j * N3 + v];
        pl.S2 += e * e;
        if (id < G) pl.D += e * e;
        else pl.R += e * e;
    }
    pl.close();
    // merge the seven sorted lists
    int head[7], pos[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) {
        pos[q] = 0;
        const int id = ids[nb.q[q]];
        head[q] = id < 0 ? kEmpty : id;
    }
    // Kept entries in ascending id order (the merge yields candidates in that order): append; past K,
    // drop the worst (smallest value, the larger id among equal values), which leaves the top K by
    // (value desc, id asc) -- the same set a full sort would keep -- still in id order.
    int kid[KM + 1];
    T ke[KM + 1];
#pragma unroll
    for (int j = 0; j <= KM; ++j) {
        kid[j] = kEmpty;
        ke[j] = (T)0;
    }
    int cnt = 0;
    int best_id = kEmpty, kbest_id = kEmpty;
    T best = (T)-INFINITY, kbest = (T)-INFINITY;
    bool ovf = false;
    for (int guard = 0; guard < 7 * KM; ++guard) {
        int c = head[0];
#pragma unroll
        for (int q = 1; q < 7; ++q) c = min(c, head[q]);
        if (c == kEmpty) break;
        T e[7];
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            e[q] = (T)0;
            if (head[q] == c) {
                e[q] = eta[pos[q] * N3 + nb.q[q]];
                ++pos[q];
                int nx = kEmpty;
                if (pos[q] < K) {
                    const int id = ids[pos[q] * N3 + nb.q[q]];
                    nx = id < 0 ? kEmpty : id;
                }
                head[q] = nx;
            }
        }
        const T en = pf_value(c < G, e[0], e[1] + e[2] + e[3] + e[4] + e[5] + e[6], pl, m, kap, gam, Ldt);
        if (en > best) { best = en; best_id = c; }
        if (en >= drop) {
            if (en > kbest) { kbest = en; kbest_id = c; }   // ascending ids: a tie keeps the smaller id
#pragma unroll
            for (int j = 0; j <= KM; ++j)
                if (j == cnt) { kid[j] = c; ke[j] = en; }
            ++cnt;
            if (cnt > K) {   // over capacity: remove the worst entry
                ovf = true;
                int wj = 0, wid = kid[0];
                T wv = ke[0];
#pragma unroll
                for (int j = 1; j <= KM; ++j)
                    if (j < cnt && (ke[j] < wv || (ke[j] == wv && kid[j] > wid))) { wj = j; wv = ke[j]; wid = kid[j]; }
#pragma unroll
                for (int j = 0; j < KM; ++j)
                    if (j >= wj) { kid[j] = kid[j + 1]; ke[j] = ke[j + 1]; }
                kid[KM] = kEmpty;
                ke[KM] = (T)0;
                cnt = K;
            }
        }
    }
    if (cnt == 0 && best_id != kEmpty) {   // nothing above the drop threshold: keep the largest
        kid[0] = best_id;
        ke[0] = best;
        cnt = 1;
        kbest_id = best_id;
    }
    gout[v] = kbest_id;
    // Write the kept entries; then clear the slots the destination still holds from its previous use
    // (every buffer keeps -1 / 0 beyond its entries, so those are the only stale ones).
#pragma unroll
    for (int j = 0; j < KM; ++j)
        if (j < cnt) {
            ids2[j * N3 + v] = kid[j];
            eta2[j * N3 + v] = ke[j];
        }
    for (int j = cnt; j < K; ++j) {
        if (ids2[j * N3 + v] < 0) break;
        ids2[j * N3 + v] = -1;
        eta2[j * N3 + v] = (T)0;
    }
    if (ovf) atomicAdd(overflow, 1);
}

// ---- tiled PF step (grids of 32 points per edge and more) ----
// The same update as k_pf, voxel by voxel and in the same arithmetic order (so FP64 results are bitwise the
// same), organised for the SM. A CTA owns a 32 x 8 column tile and marches through kZC planes of z. The active
// sets of the planes z-1, z, z+1 (interior) and the x/y halo of plane z are staged in shared memory by cp.async,
// as (id, eta) entries with a -1 id after each list's last staged slot: as an unsigned head a negative id lies above every
// grain id, so the seven-list merge reads one entry per step and needs no slot-count checks and no test for an ended list. Which slots to stage comes from a per-row bound: rmax[s] >= the number of
// entries of every point of the 32-point row segment s = (z n + y) (n / 32) + x / 32, so every staged load is
// independent of the others. Each step writes the exact bound of the rows it produced and clears, in the
// destination, the slots between a point's new count and the destination's previous bound, which keeps every
// list -1 / 0 terminated over all K slots (the layout every other reader of the active sets assumes).
// Three plane buffers and one halo buffer keep the FP32 tile at 61 KB (FP64: 92 KB), so three (two) CTAs share an SM
// and cover each other's staging waits.
constexpr int kTX = 32, kTY = 8, kZC = 16;
constexpr int kPlane = kTX * kTY;             // interior points of one plane tile
constexpr int kHalo = 2 * kTX + 2 * kTY;      // rows y0-1, y0+8 and columns x0-1, x0+32 of the centre plane
constexpr int kTileThreads = kTX * kTY;
constexpr int kSlots = KM + 1;                // KM slots and the terminating -1

// Staged (id, eta) entries, element index space: 3 interior plane buffers [buf][slot][point], then the halo
// [slot][halo point]. FP32: 8-byte pairs, one load per entry. FP64: ids and values apart (12 bytes an entry; pairs
// padded to 16 would leave room for one CTA per SM instead of two).
constexpr int kEntries = 3 * kSlots * kPlane + kSlots * kHalo;
template <typename T> struct PFEntries;
template <> struct PFEntries<float> {
    struct alignas(8) Pair { int32_t id; float e; } pr[kEntries];
    __device__ __forceinline__ int32_t *id_ptr(int i) { return &pr[i].id; }
    __device__ __forceinline__ float *e_ptr(int i) { return &pr[i].e; }
    __device__ __forceinline__ void get(int i, uint32_t &id, float &e) const {
        const Pair q = pr[i];
        id = (uint32_t)q.id;
        e = q.e;
    }
};
template <> struct PFEntries<double> {
    double ev[kEntries];
    int32_t idv[kEntries];
    __device__ __forceinline__ int32_t *id_ptr(int i) { return &idv[i]; }
    __device__ __forceinline__ double *e_ptr(int i) { return &ev[i]; }
    __device__ __forceinline__ void get(int i, uint32_t &id, double &e) const {
        id = (uint32_t)idv[i];
        e = ev[i];
    }
};

template <typename T>
struct PFTile {
    PFEntries<T> en;
    uint8_t rin[(kZC + 2) * (kTY + 2)];   // bounds of the current buffer: planes z0-1..z0+kZC, rows y0-1..y0+8
    uint8_t rxl[kZC * kTY], rxr[kZC * kTY];   // bounds of the left / right neighbour segments, planes z0.., rows y0..
    uint8_t rdst[kZC * kTY];              // previous bounds of the destination rows
};

__device__ __forceinline__ int tile_int_index(int buf, int j, int p) { return (buf * kSlots + j) * kPlane + p; }
__device__ __forceinline__ int tile_halo_index(int j, int hp) { return 3 * kSlots * kPlane + j * kHalo + hp; }

// Issue the asynchronous copies of one point's slots [0, R) into the tile (element index base, slot stride) and
// write the terminating -1 at slot R (R <= K <= KM: global memory also holds -1 there when R < K).
template <typename T>
__device__ __forceinline__ void stage_point(PFTile<T> &tb, int base, int stride, int R, int K,
                                            const int32_t *__restrict__ ids, const T *__restrict__ eta, long N3,
                                            long v) {
    R = min(R, K);   // a bound never exceeds K; the clamp keeps every access inside the K slot planes regardless
#pragma unroll
    for (int j = 0; j < KM; ++j)
        if (j < R) {
            cp_async<4>(tb.en.id_ptr(base + j * stride), ids + j * N3 + v);
            cp_async<sizeof(T)>(tb.en.e_ptr(base + j * stride), eta + j * N3 + v);
        }
    *tb.en.id_ptr(base + R * stride) = -1;
}

// a > b and a >= b for order parameters. FP64: on the integer pipe (sign-magnitude order of the bits), since the FP64 pipe
// bounds the step; values that are not finite, which may be NaN, compare as doubles.
__device__ __forceinline__ bool pf_gt(float a, float b) { return a > b; }
__device__ __forceinline__ bool pf_ge(float a, float b) { return a >= b; }
__device__ __forceinline__ long long pf_key(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool pf_nonfinite(double x) { return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000; }
__device__ __forceinline__ bool pf_gt(double a, double b) {
    if (pf_nonfinite(a)) return a > b;
    return pf_key(a) > pf_key(b) && !(pf_zero(a) && pf_zero(b));
}
__device__ __forceinline__ bool pf_ge(double a, double b) {
    if (pf_nonfinite(a)) return a >= b;
    return pf_key(a) >= pf_key(b) || (pf_zero(a) && pf_zero(b));
}

template <typename T>
__global__ void __launch_bounds__(kTileThreads, sizeof(T) == 4 ? 3 : 2)
k_pf_tile(int n, const int32_t *__restrict__ ids, const T *__restrict__ eta, int32_t *__restrict__ ids2,
          T *__restrict__ eta2, int32_t *__restrict__ gout, const double *__restrict__ kf, PFConst pc,
          int32_t *__restrict__ overflow, const uint8_t *__restrict__ rcur, uint8_t *__restrict__ rdst) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PFTile<T> &tb = *reinterpret_cast<PFTile<T> *>(smem_raw);
    const long N3 = (long)n * n * n;
    const int msk = n - 1, nseg = n / kTX;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int xs = blockIdx.x, x0 = xs * kTX, y0 = blockIdx.y * kTY, z0 = blockIdx.z * kZC;
    const int K = pc.K, G = pc.G;
    auto seg = [&](int z, int y, int s) { return ((long)z * n + y) * nseg + s; };
    // row bounds of the chunk
    for (int t = threadIdx.x; t < (kZC + 2) * (kTY + 2); t += kTileThreads) {
        const int pz = t / (kTY + 2), ry = t % (kTY + 2);
        tb.rin[t] = rcur[seg((z0 - 1 + pz) & msk, (y0 - 1 + ry) & msk, xs)];
    }
    for (int t = threadIdx.x; t < kZC * kTY; t += kTileThreads) {
        const int pz = t / kTY, ry = t % kTY;
        tb.rxl[t] = rcur[seg(z0 + pz, y0 + ry, (xs + nseg - 1) % nseg)];
        tb.rxr[t] = rcur[seg(z0 + pz, y0 + ry, (xs + 1) % nseg)];
        tb.rdst[t] = rdst[seg(z0 + pz, y0 + ry, xs)];
    }
    __syncthreads();
    const int p = ty * kTX + tx;
    // plane index pp = 0 .. kZC+1 holds z = z0 - 1 + pp in interior buffer pp % 3
    auto stage_plane = [&](int pp) {
        const int z = (z0 - 1 + pp) & msk;
        const long v = ((long)z * n + (y0 + ty)) * n + x0 + tx;
        stage_point(tb, tile_int_index(pp % 3, 0, p), kPlane, tb.rin[pp * (kTY + 2) + ty + 1], K, ids, eta, N3, v);
    };
    // halo of centre plane i (z = z0 + i)
    auto stage_halo = [&](int i) {
        const int t = threadIdx.x;
        if (t >= kHalo) return;
        const int z = z0 + i;
        int x, y, R;
        if (t < kTX) { x = x0 + t; y = (y0 - 1) & msk; R = tb.rin[(i + 1) * (kTY + 2)]; }
        else if (t < 2 * kTX) { x = x0 + t - kTX; y = (y0 + kTY) & msk; R = tb.rin[(i + 1) * (kTY + 2) + kTY + 1]; }
        else if (t < 2 * kTX + kTY) { x = (x0 - 1) & msk; y = y0 + t - 2 * kTX; R = tb.rxl[i * kTY + t - 2 * kTX]; }
        else { x = (x0 + kTX) & msk; y = y0 + t - 2 * kTX - kTY; R = tb.rxr[i * kTY + t - 2 * kTX - kTY]; }
        const long v = ((long)z * n + y) * n + x;
        stage_point(tb, tile_halo_index(0, t), kHalo, R, K, ids, eta, N3, v);
    };
    stage_plane(0);
    stage_plane(1);
    stage_plane(2);
    stage_halo(0);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();

    T m, kap, gam, Ldt, drop;   // in the field precision (no FP64 conversions on the FP32 path)
    if constexpr (sizeof(T) == 4) { m = pc.m_f; kap = pc.kappa_f; gam = pc.gam_f; Ldt = pc.L_dt_f; drop = pc.drop_f; }
    else { m = pc.m; kap = pc.kappa; gam = pc.gam; Ldt = pc.L_dt; drop = pc.drop; }

    for (int i = 0; i < kZC; ++i) {
        const int z = z0 + i;
        const long v = ((long)z * n + (y0 + ty)) * n + x0 + tx;
        const double kv = kf[v];
        // the seven lists: self, x-, x+, y-, y+, z-, z+ -- element index of the current slot, slot stride
        // (kPlane, or kHalo where a neighbour lies in the halo)
        const int c = (i + 1) % 3;
        int at[7], st[7];
        at[0] = tile_int_index(c, 0, p);
#pragma unroll
        for (int q = 0; q < 7; ++q) st[q] = kPlane;
        if (tx > 0) at[1] = at[0] - 1; else { at[1] = tile_halo_index(0, 2 * kTX + ty); st[1] = kHalo; }
        if (tx < kTX - 1) at[2] = at[0] + 1; else { at[2] = tile_halo_index(0, 2 * kTX + kTY + ty); st[2] = kHalo; }
        if (ty > 0) at[3] = at[0] - kTX; else { at[3] = tile_halo_index(0, tx); st[3] = kHalo; }
        if (ty < kTY - 1) at[4] = at[0] + kTX; else { at[4] = tile_halo_index(0, kTX + tx); st[4] = kHalo; }
        at[5] = tile_int_index(i % 3, 0, p);
        at[6] = tile_int_index((i + 2) % 3, 0, p);

        // local sums over the voxel's own list, ascending id (the list ends at a -1)
        PFLocal<T> pl{(T)(pc.Escale * kv), (T)0, (T)0, (T)0};
        for (int j = 0; j < kSlots; ++j) {
            uint32_t id;
            T e;
            tb.en.get(at[0] + j * kPlane, id, e);
            if ((int32_t)id < 0) break;
            pl.S2 += e * e;
            if ((int32_t)id < G) pl.D += e * e;
            else pl.R += e * e;
        }
        pl.close();
        uint32_t head[7];   // a list's current id; an ended list's negative one is above every id
        T cur[7];
#pragma unroll
        for (int q = 0; q < 7; ++q) tb.en.get(at[q], head[q], cur[q]);
        int kid[KM + 1];
        T ke[KM + 1];
#pragma unroll
        for (int j = 0; j <= KM; ++j) {
            kid[j] = kEmpty;
            ke[j] = (T)0;
        }
        int cnt = 0;
        int best_id = kEmpty;
        T best = (T)-INFINITY;   // the largest value: a kept one if any is (ascending ids: a tie keeps the smaller id)
        bool ovf = false;
        for (int guard = 0; guard < 7 * KM; ++guard) {
            uint32_t uid = head[0];
#pragma unroll
            for (int q = 1; q < 7; ++q) uid = min(uid, head[q]);
            const int cid = (int)uid;
            if (cid < 0) break;   // any negative id ends a list, and as unsigned heads they lie above every id
            T e0 = (T)0, nb = (T)0;
#pragma unroll
            for (int q = 0; q < 7; ++q)
                if (head[q] == uid) {   // take list q's value and advance it
                    if (q == 0) e0 = cur[0];
                    else nb += cur[q];
                    at[q] += st[q];
                    tb.en.get(at[q], head[q], cur[q]);
                }
            const T en = pf_value(cid < G, e0, nb, pl, m, kap, gam, Ldt);
            if (pf_gt(en, best)) { best = en; best_id = cid; }
            if (pf_ge(en, drop)) {
#pragma unroll
                for (int j = 0; j <= KM; ++j)
                    if (j == cnt) { kid[j] = cid; ke[j] = en; }
                ++cnt;
                if (cnt > K) {   // over capacity: remove the worst entry (smallest value, larger id among equals)
                    ovf = true;
                    int wj = 0, wid = kid[0];
                    T wv = ke[0];
#pragma unroll
                    for (int j = 1; j <= KM; ++j)
                        if (j < cnt && (ke[j] < wv || (ke[j] == wv && kid[j] > wid))) { wj = j; wv = ke[j]; wid = kid[j]; }
#pragma unroll
                    for (int j = 0; j < KM; ++j)
                        if (j >= wj) { kid[j] = kid[j + 1]; ke[j] = ke[j + 1]; }
                    kid[KM] = kEmpty;
                    ke[KM] = (T)0;
                    cnt = K;
                }
            }
        }
        if (cnt == 0 && best_id != kEmpty) {   // nothing above the drop threshold: keep the largest
            kid[0] = best_id;
            ke[0] = best;
            cnt = 1;
        }
        gout[v] = best_id;
        // kept entries, then the slots up to the destination's previous bound cleared (beyond it they are empty)
        const int rd = min((int)tb.rdst[i * kTY + ty], K);
#pragma unroll
        for (int j = 0; j < KM; ++j) {
            if (j < cnt) {
                ids2[j * N3 + v] = kid[j];
                eta2[j * N3 + v] = ke[j];
            } else if (j < rd) {
                ids2[j * N3 + v] = -1;
                eta2[j * N3 + v] = (T)0;
            }
        }
        const int rowmax = __reduce_max_sync(0xffffffffu, (unsigned)cnt);
        if (tx == 0) rdst[seg(z, y0 + ty, xs)] = (uint8_t)rowmax;
        const unsigned ob = __ballot_sync(0xffffffffu, ovf);
        if (tx == 0 && ob) atomicAdd(overflow, __popc(ob));
        __syncthreads();   // every thread is done with plane z - 1 and with this halo
        if (i + 1 < kZC) {
            stage_plane(i + 3);   // into the buffer plane z - 1 held
            stage_halo(i + 1);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            __syncthreads();
        }
    }
}

template <typename T>
__global__ void k_pf_soften(long N3, const int32_t *__restrict__ gprev, const int32_t *__restrict__ g, T *__restrict__ rho,
                            double *__restrict__ kf, int G, double s) {
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N3) return;
    if (!(gprev[v] < G && g[v] >= G)) return;
    double kk = 0.0;
    for (int a = 0; a < 12; ++a) {
        const T r = (T)(s * (double)rho[a * N3 + v]);
        rho[a * N3 + v] = r;
        kk += (double)r;
    }
    kf[v] = kk;
}

// Per-voxel discrete free energy (bulk + forward-difference gradient + stored energy) and
// recrystallised count, summed per block in FP64; distinct grain ids marked in a bitmap.
template <typename T>
__global__ void __launch_bounds__(256) k_pf_stats(int n, const int32_t *__restrict__ ids, const T *__restrict__ eta,
                                                 const int32_t *__restrict__ g, const double *__restrict__ kf, PFConst pc,
                                                 uint32_t *__restrict__ bitmap, int bitmap_words, double *__restrict__ part) {
    __shared__ double red[32];
    const long N3 = (long)n * n * n;
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    double F = 0.0, rex = 0.0;
    if (v < N3) {
        const int K = pc.K, G = pc.G;
        const int gi = g[v];
        if (gi >= G) rex = 1.0;
        // one atomic per distinct id of the warp, and none once the bit is set: neighbouring voxels share
        // their ids, and same-address atomics from every voxel serialise
        const bool ok = gi >= 0 && (gi >> 5) < bitmap_words;
        const unsigned peers = __match_any_sync(__activemask(), ok ? gi : -1);
        if (ok && (threadIdx.x & 31) == __ffs(peers) - 1) {
            uint32_t *word = bitmap + (gi >> 5);
            const uint32_t bit = 1u << (gi & 31);
            if (!(*(volatile uint32_t *)word & bit)) atomicOr(word, bit);
        }
        // per-voxel terms in the field precision (the FP32 path keeps the FP64 pipe out), sums in FP64
        using A = T;
        const A gam = sizeof(T) == 4 ? (A)pc.gam_f : (A)pc.gam;
        A f0 = (A)0.25, S2 = (A)0, D = (A)0;
        for (int j = 0; j < K; ++j) {
            const int id = ids[j * N3 + v];
            if (id < 0) break;
            const A e = eta[j * N3 + v];
            f0 += e * e * e * e / (A)4 - e * e / (A)2;
            S2 += e * e;
            if (id < G) D += e * e;
            for (int i2 = j + 1; i2 < K; ++i2) {
                if (ids[i2 * N3 + v] < 0) break;
                const A e2 = eta[i2 * N3 + v];
                f0 += gam * e * e * e2 * e2;
            }
        }
        const A fdef = S2 > (A)1e-12 ? (A)(pc.Escale * kf[v]) * D / S2 : (A)0;
        const Nbr nb = neighbours(n, v);
        A grad = (A)0;
        for (int d = 2; d <= 6; d += 2) {   // x+, y+, z+
            const long w = nb.q[d];
            int pa = 0, pb = 0;
            for (int guard = 0; guard < 2 * KM; ++guard) {
                const int ia = pa < K ? ids[pa * N3 + v] : -1;
                const int ib = pb < K ? ids[pb * N3 + w] : -1;
                const int ca = ia < 0 ? kEmpty : ia, cb = ib < 0 ? kEmpty : ib;
                if (ca == kEmpty && cb == kEmpty) break;
                A ea = (A)0, eb = (A)0;
                if (ca <= cb) { ea = eta[pa * N3 + v]; ++pa; }
                if (cb <= ca) { eb = eta[pb * N3 + w]; ++pb; }
                grad += (eb - ea) * (eb - ea);
            }
        }
        F = (double)((sizeof(T) == 4 ? (A)pc.m_f : (A)pc.m) * f0 +
                     (A)0.5 * (sizeof(T) == 4 ? (A)pc.kappa_f : (A)pc.kappa) * grad + fdef);
    }
    const double sF = block_sum(F, red);
    const double sR = block_sum(rex, red);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = sF;
        part[2 * blockIdx.x + 1] = sR;
    }
}

// The same on grids of 32 points per edge and more: a warp takes a 32-point row segment. It copies the segment's lists
// and those of its y+ and z+ neighbours into shared memory, with the rows' slot bounds (rcur, see k_pf_tile), so every load
// is independent of the others, coalesced and warp-uniform, and merges pairs of lists there (an ended list's negative id
// lies above every grain id as an unsigned number); the x+ neighbour's list is the next lane's. The pair energy accumulates as
// sum_j e_j^2 (e_0^2 + .. + e_(j-1)^2). A warp walks kStatRows rows before its block adds up (the FP64 block sum is 10
// FP64-pipe instructions a warp). 128^3: 142 us FP32 and 523 us FP64, where one thread per point with dependent global
// loads took 226 and 706, and matching the lists pairwise in registers 249 and 706.
constexpr int kStatRows = 4, kStatWarps = 4;
template <typename T> struct PFRow {   // lists of 32 points and of the next one, each ended by a -1
    T e[KM + 1][33];
    int32_t id[KM + 1][33];
};
template <typename T>
__device__ __forceinline__ void stage_row(PFRow<T> &r, int at, const int32_t *__restrict__ ids, const T *__restrict__ eta,
                                          long N3, long v, int R) {
#pragma unroll
    for (int j = 0; j < KM; ++j)
        if (j < R) {
            r.id[j][at] = ids[j * N3 + v];
            r.e[j][at] = eta[j * N3 + v];
        }
    r.id[R][at] = -1;
}
// sum over the ids of either list of the squared difference of their values
template <typename T> __device__ __forceinline__ T pf_diff2(const PFRow<T> &a, int la, const PFRow<T> &b, int lb) {
    T g = (T)0;
    int pa = 0, pb = 0;
    uint32_t ia = (uint32_t)a.id[0][la], ib = (uint32_t)b.id[0][lb];
    while ((int32_t)(ia & ib) >= 0) {   // until both lists have ended (any negative id)
        T ea = (T)0, eb = (T)0;
        const bool ta = ia <= ib, tb = ib <= ia;
        if (ta) {
            ea = a.e[pa][la];
            ia = (uint32_t)a.id[++pa][la];
        }
        if (tb) {
            eb = b.e[pb][lb];
            ib = (uint32_t)b.id[++pb][lb];
        }
        g += (eb - ea) * (eb - ea);
    }
    return g;
}
template <typename T>
__global__ void __launch_bounds__(32 * kStatWarps) k_pf_stats_rows(int n, int K, const int32_t *__restrict__ ids,
                                                                  const T *__restrict__ eta, const int32_t *__restrict__ g,
                                                                  const double *__restrict__ kf, PFConst pc,
                                                                  uint32_t *__restrict__ bitmap, int bitmap_words,
                                                                  const uint8_t *__restrict__ rcur, double *__restrict__ part) {
    __shared__ double red[32];
    __shared__ PFRow<T> rows[kStatWarps][3];
    const long N3 = (long)n * n * n;
    const int msk = n - 1, nseg = n / 32, lane = threadIdx.x & 31, G = pc.G;
    const long nrows = (long)n * n * nseg;
    const T gam = sizeof(T) == 4 ? (T)pc.gam_f : (T)pc.gam, m = sizeof(T) == 4 ? (T)pc.m_f : (T)pc.m;
    const T kap = sizeof(T) == 4 ? (T)pc.kappa_f : (T)pc.kappa;
    double F = 0.0;
    int rex = 0;
    PFRow<T> &own = rows[threadIdx.x >> 5][0], &py = rows[threadIdx.x >> 5][1], &pz = rows[threadIdx.x >> 5][2];
    const long r0 = ((long)blockIdx.x * kStatWarps + (threadIdx.x >> 5)) * kStatRows;
    for (long row = r0; row < min(r0 + kStatRows, nrows); ++row) {
        const int xs = (int)(row % nseg), y = (int)(row / nseg) & msk, z = (int)(row / ((long)nseg * n));
        auto seg = [&](int zz, int yy, int s) { return ((long)zz * n + yy) * nseg + s; };
        auto point = [&](int zz, int yy, int xx) { return ((long)zz * n + yy) * n + xx; };
        const int yp = (y + 1) & msk, zp = (z + 1) & msk, xsp = (xs + 1) % nseg, x = 32 * xs + lane;
        const int R = min((int)rcur[row], K), Rx = min((int)rcur[seg(z, y, xsp)], K);
        const int Ry = min((int)rcur[seg(z, yp, xs)], K), Rz = min((int)rcur[seg(zp, y, xs)], K);
        const long v = point(z, y, x);
        __syncwarp();   // every lane is done with the previous row
        stage_row(own, lane, ids, eta, N3, v, R);
        stage_row(py, lane, ids, eta, N3, point(z, yp, x), Ry);
        stage_row(pz, lane, ids, eta, N3, point(zp, y, x), Rz);
        if (lane == 31) stage_row(own, 32, ids, eta, N3, point(z, y, 32 * xsp), Rx);
        const int gi = g[v];
        const double kv = kf[v];
        if (gi >= G) ++rex;
        // one atomic per distinct id of the warp, and none once the bit is set
        const bool ok = gi >= 0 && (gi >> 5) < bitmap_words;
        const unsigned peers = __match_any_sync(0xffffffffu, ok ? gi : -1);
        if (ok && lane == __ffs(peers) - 1) {
            uint32_t *word = bitmap + (gi >> 5);
            const uint32_t bit = 1u << (gi & 31);
            if (!(*(volatile uint32_t *)word & bit)) atomicOr(word, bit);
        }
        __syncwarp();
        T f0 = (T)0.25, S2 = (T)0, D = (T)0, pairs = (T)0;
        bool all_def = true;
        for (int j = 0; j < R; ++j) {
            const int id = own.id[j][lane];
            if (id < 0) break;
            const T e2 = own.e[j][lane] * own.e[j][lane];
            f0 += e2 * e2 * (T)0.25 - e2 * (T)0.5;
            pairs += e2 * S2;
            S2 += e2;
            if (id < G) D += e2;
            else all_def = false;
        }
        T grad = pf_diff2(own, lane, own, lane + 1);
        grad += pf_diff2(own, lane, py, lane);
        grad += pf_diff2(own, lane, pz, lane);
        const T driving = (T)(pc.Escale * kv);
        const T fdef = S2 > (T)1e-12 ? (all_def ? driving : driving * D / S2) : (T)0;
        F += (double)(m * (f0 + gam * pairs) + (T)0.5 * kap * grad + fdef);
    }
    const double sF = block_sum(F, red);
    __syncthreads();
    const double sR = block_sum((double)rex, red);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = sF;
        part[2 * blockIdx.x + 1] = sR;
    }
}

__global__ void k_popc(const uint32_t *__restrict__ bitmap, int words, double *__restrict__ out_slot) {
    __shared__ double red[32];
    double c = 0.0;
    for (int i = threadIdx.x; i < words; i += blockDim.x) c += (double)__popc(bitmap[i]);
    const double s = block_sum(c, red);
    if (threadIdx.x == 0) *out_slot = s;
}

// Deterministic sum of partials [nparts][nvals] -> out[nvals]: one block per column, fixed order.
__global__ void k_reduce(const double *__restrict__ part, int nparts, int nvals, double *__restrict__ out,
                         const int *__restrict__ skip) {
    if (skip != nullptr && *skip) return;
    __shared__ double red[32];
    const int c = blockIdx.x;
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) s += part[(long)i * nvals + c];
    s = block_sum(s, red);
    if (threadIdx.x == 0) out[c] = s;
}

// ---- 2:1 phase-field grid (Sec. 2.4) ----
// Both grids are cell-centred and periodic: voxel i spans [i, i+1), PF cell I spans [I/2, (I+1)/2).
// Along each axis a PF centre lies between its parent voxel's centre (weight 3/4) and the neighbour on
// its side (weight 1/4). PF point w = X + 2n (Y + 2n Z).
__device__ __forceinline__ void interp_axis(int I, int n, int (&idx)[2], double (&wt)[2]) {
    const int i = I >> 1;
    if ((I & 1) == 0) { idx[0] = (i + n - 1) % n; idx[1] = i; wt[0] = 0.25; wt[1] = 0.75; }
    else { idx[0] = i; idx[1] = (i + 1) % n; wt[0] = 0.75; wt[1] = 0.25; }
}

// kpf = trilinear interpolation of k (rho_tot); the eight terms in (z, y, x) order, weights (wz wy) wx
__global__ void k_interp_k(int n, const double *__restrict__ k, double *__restrict__ kpf) {
    const int m = 2 * n;
    const long M3 = (long)m * m * m;
    const long w = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= M3) return;
    const int X = (int)(w % m), Y = (int)((w / m) % m), Z = (int)(w / ((long)m * m));
    int ix[2], iy[2], iz[2];
    double wx[2], wy[2], wz[2];
    interp_axis(X, n, ix, wx);
    interp_axis(Y, n, iy, wy);
    interp_axis(Z, n, iz, wz);
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                acc += (wz[a] * wy[b]) * wx[c] * k[ix[c] + (long)n * (iy[b] + (long)n * iz[a])];
    kpf[w] = acc;
}

// A voxel's grain id from its eight PF children c = dx + 2 dy + 4 dz: the id with the largest sum of
// order parameters over the children (summed in c order), ties to the smaller id. The children's
// lists are sorted by id, so the eight are merged in ascending id order.
template <typename T>
__global__ void k_restrict(int n, int K, const int32_t *__restrict__ ids, const T *__restrict__ eta,
                           int32_t *__restrict__ g) {
    const long N3 = (long)n * n * n;
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N3) return;
    const int m = 2 * n;
    const long M3 = (long)m * m * m;
    const int x = (int)(v % n), y = (int)((v / n) % n), z = (int)(v / ((long)n * n));
    long ch[8];
    int pos[8], head[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        ch[c] = (2 * x + (c & 1)) + (long)m * ((2 * y + ((c >> 1) & 1)) + (long)m * (2 * z + (c >> 2)));
        pos[c] = 0;
        const int id = ids[ch[c]];
        head[c] = id < 0 ? kEmpty : id;
    }
    int best = -1;
    double bsum = 0.0;
    for (int guard = 0; guard < 8 * KM; ++guard) {
        int cmin = head[0];
#pragma unroll
        for (int c = 1; c < 8; ++c) cmin = min(cmin, head[c]);
        if (cmin == kEmpty) break;
        double sum = 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            if (head[c] == cmin) {
                sum += (double)eta[pos[c] * M3 + ch[c]];
                ++pos[c];
                int nx = kEmpty;
                if (pos[c] < K) {
                    const int id = ids[pos[c] * M3 + ch[c]];
                    nx = id < 0 ? kEmpty : id;
                }
                head[c] = nx;
            }
        }
        if (best < 0 || sum > bsum) { best = cmin; bsum = sum; }   // ascending ids: a tie keeps the smaller
    }
    g[v] = best;
}

// initial active sets on the PF grid: one order parameter 1 of the parent voxel's grain
__global__ void k_pf_init(int n, int r, int K, const int32_t *__restrict__ g0, int32_t *__restrict__ ids,
                          void *__restrict__ eta, int32_t *__restrict__ ids2, void *__restrict__ eta2, int eta_double,
                          int32_t *__restrict__ gpf) {
    const int m = r * n;
    const long M3 = (long)m * m * m;
    const long w = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= M3) return;
    const int X = (int)(w % m), Y = (int)((w / m) % m), Z = (int)(w / ((long)m * m));
    const int gi = g0[X / r + (long)n * (Y / r + (long)n * (Z / r))];
    for (int j = 0; j < K; ++j) {
        ids[j * M3 + w] = j == 0 ? gi : -1;
        ids2[j * M3 + w] = -1;   // the step's destination: empty (it only rewrites slots in use)
        if (eta_double) {
            static_cast<double *>(eta)[j * M3 + w] = j == 0 ? 1.0 : 0.0;
            static_cast<double *>(eta2)[j * M3 + w] = 0.0;
        } else {
            static_cast<float *>(eta)[j * M3 + w] = j == 0 ? 1.f : 0.f;
            static_cast<float *>(eta2)[j * M3 + w] = 0.f;
        }
    }
    gpf[w] = gi;
}

}  // namespace

long pf_row_bounds_bytes(int n) { return n >= kTX ? (long)n * n * (n / kTX) : 0; }

template <typename T>
cudaError_t pf_one_step(int n, const int32_t *ids, const T *eta, int32_t *ids2, T *eta2, int32_t *g, const double *k,
                        PFConst pc, int32_t *overflow, const uint8_t *rcur, uint8_t *rdst, cudaStream_t s) {
    const long N3 = (long)n * n * n;
    if (pc.K > KM || pc.K < 1) return cudaErrorInvalidValue;
    if (n >= kTX && rcur != nullptr && rdst != nullptr) {
        // set on every launch (a host-side call of about a microsecond): the attribute belongs to the current
        // device, so a process that drives several GPUs needs it on each
        const int sm = (int)sizeof(PFTile<T>);
        const cudaError_t e = cudaFuncSetAttribute(k_pf_tile<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        if (e != cudaSuccess) return e;
        const dim3 grid(n / kTX, n / kTY, n / kZC);
        k_pf_tile<T><<<grid, kTileThreads, sm, s>>>(n, ids, eta, ids2, eta2, g, k, pc, overflow, rcur, rdst);
    } else {
        k_pf<T><<<(int)((N3 + kPF - 1) / kPF), kPF, 0, s>>>(n, ids, eta, ids2, eta2, g, k, pc, overflow);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t pf_soften(long N3, const int32_t *gprev, const int32_t *g, T *rho, double *k, int G, double s_soften,
                      cudaStream_t s) {
    k_pf_soften<T><<<(int)((N3 + 255) / 256), 256, 0, s>>>(N3, gprev, g, rho, k, G, s_soften);
    return cudaGetLastError();
}

int pf_stat_blocks(long N3) { return (int)((N3 + 255) / 256); }

template <typename T>
cudaError_t pf_stats_launch(int n, const int32_t *ids, const T *eta, const int32_t *g, const double *k, PFConst pc,
                     uint32_t *bitmap, int bitmap_words, const uint8_t *rcur, double *partials, double *out2, double *ngrains,
                     cudaStream_t s) {
    const long N3 = (long)n * n * n;
    cudaError_t e = cudaMemsetAsync(bitmap, 0, sizeof(uint32_t) * (size_t)bitmap_words, s);
    if (e != cudaSuccess) return e;
    int nb = pf_stat_blocks(N3);
    if (n >= 32 && rcur != nullptr) {
        nb = (int)((N3 / 32 + kStatRows * kStatWarps - 1) / (kStatRows * kStatWarps));
        k_pf_stats_rows<T><<<nb, 32 * kStatWarps, 0, s>>>(n, pc.K, ids, eta, g, k, pc, bitmap, bitmap_words, rcur, partials);
    } else {
        k_pf_stats<T><<<nb, 256, 0, s>>>(n, ids, eta, g, k, pc, bitmap, bitmap_words, partials);
    }
    k_popc<<<1, 1024, 0, s>>>(bitmap, bitmap_words, ngrains);
    return reduce_partials(partials, nb, 2, out2, s);
}

cudaError_t reduce_partials(const double *partials, int nparts, int nvals, double *out, cudaStream_t s,
                            const int *skip) {
    k_reduce<<<nvals, 1024, 0, s>>>(partials, nparts, nvals, out, skip);
    return cudaGetLastError();
}

cudaError_t pf_interp(int n, const double *k, double *kpf, cudaStream_t s) {
    const long M3 = 8L * n * n * n;
    k_interp_k<<<(int)((M3 + 255) / 256), 256, 0, s>>>(n, k, kpf);
    return cudaGetLastError();
}

template <typename T>
cudaError_t pf_restrict(int n, int K, const int32_t *ids, const T *eta, int32_t *g, cudaStream_t s) {
    if (K > KM || K < 1) return cudaErrorInvalidValue;
    const long N3 = (long)n * n * n;
    k_restrict<T><<<(int)((N3 + 127) / 128), 128, 0, s>>>(n, K, ids, eta, g);
    return cudaGetLastError();
}

cudaError_t pf_init(int n, int r, int K, const int32_t *g0, int32_t *ids, void *eta, int32_t *ids2, void *eta2,
                    int eta_double, int32_t *gpf, cudaStream_t s) {
    const long M3 = (long)r * n * r * n * r * n;
    k_pf_init<<<(int)((M3 + 255) / 256), 256, 0, s>>>(n, r, K, g0, ids, eta, ids2, eta2, eta_double, gpf);
    return cudaGetLastError();
}

template cudaError_t pf_restrict<float>(int, int, const int32_t *, const float *, int32_t *, cudaStream_t);
template cudaError_t pf_restrict<double>(int, int, const int32_t *, const double *, int32_t *, cudaStream_t);
template cudaError_t pf_one_step<float>(int, const int32_t *, const float *, int32_t *, float *, int32_t *,
                                        const double *, PFConst, int32_t *, const uint8_t *, uint8_t *, cudaStream_t);
template cudaError_t pf_one_step<double>(int, const int32_t *, const double *, int32_t *, double *, int32_t *,
                                         const double *, PFConst, int32_t *, const uint8_t *, uint8_t *, cudaStream_t);
template cudaError_t pf_soften<float>(long, const int32_t *, const int32_t *, float *, double *, int, double, cudaStream_t);
template cudaError_t pf_soften<double>(long, const int32_t *, const int32_t *, double *, double *, int, double, cudaStream_t);
template cudaError_t pf_stats_launch<float>(int, const int32_t *, const float *, const int32_t *, const double *, PFConst,
                                            uint32_t *, int, const uint8_t *, double *, double *, double *, cudaStream_t);
template cudaError_t pf_stats_launch<double>(int, const int32_t *, const double *, const int32_t *, const double *, PFConst,
                                             uint32_t *, int, const uint8_t *, double *, double *, double *, cudaStream_t);

}  // namespace evp
