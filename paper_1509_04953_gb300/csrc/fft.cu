// Hand-written 3D FFT passes for the Green-operator fixed point (Sec. 2.1: the spectral solve of
// the implicit stress update). One HBM round trip per axis:
//   x pass : real -> half spectrum, two real rows packed as one complex row
//   y pass : complex, lines along y loaded as [kx tile][y] (coalesced along kx)
//   z pass : complex, the six stress components of a [kx tile] x z slab of one ky; the forward
//            transform, the equilibrium residual, the Green-operator contraction and the inverse
//            transform run on the slab while it sits in shared memory
//   y pass : inverse
//   x pass : half spectrum -> real, fused with the strain update eps += field/N^3 + dE
// Where a (field, z) plane fits in shared memory next to two others, the x and y passes run as one launch
// per direction over whole planes (k_fft_xy_r2c, k_fft_xy_c2r), so an iteration crosses HBM three times; at 256^3 in FP32
// a cluster of CTAs holds the plane (k_fft_xy_r2c_cl, k_fft_xy_c2r_cl).
// Spectra are [field][z|kz][ky][kx] with kx = 0..N/2 (row length N/2+1).
//
// Line transforms: Stockham auto-sort with register butterflies. N = R1 * R2 with R1 = 16 (8 for N <= 32, see Shape)
// and R2 = N / R1 <= 16: a radix-R1 pass (no twiddles) and a radix-R2 pass (twiddles W_N^{r j}),
// natural order in and out. Shared-memory lines are padded (one slot per R1) so that the strided
// pass-1 writes hit distinct banks.
#include <cooperative_groups.h>

#include <cmath>
#include <cstdint>
#include <cstdio>

#include "common.cuh"
#include "fpctl.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace evp {

namespace {

constexpr int kThreads = 256;

// Asynchronous global -> shared copies (cp.async): every thread issues all of its loads before
// waiting, so many requests are in flight per SM while the pass is latency-bound.
template <int B> __device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (B == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
    else if constexpr (B == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
    else asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Radices and padded line stride. N = 16 and 32 take R1 = 8: a plane or a slab of such a grid is small, its transform is
// bound by the latency of each thread's chain and by the threads it occupies, and radix-8 items are twice as many and
// half as long as radix-16 ones (32^3 FP32 plane of 16 packed lines: 64 items instead of 32). Their second pass starts
// with the last stage of the radix-16 network (pass2_tail), so the butterflies are those of the radix-16 split. The line strides keep both ways a warp walks a tile (along lines, across lines) at most
// two-way bank-conflicted. NTW: slots of the twiddle table (load_tw).
template <int N> struct Shape {
    static constexpr int R1 = N < 16 ? N : N <= 32 ? 8 : 16;
    static constexpr int R2 = N / R1;
    static constexpr int LS = N >= 64 ? N + N / 16 + 1 : N == 32 ? 38 : N == 16 ? 22 : N + 1;
    static constexpr int NTW = R1 == 8 && R2 > 1 ? N + 8 : N;
};
template <int N> __host__ __device__ constexpr int padn(int i) { return N < 16 ? i : i + i / Shape<N>::R1; }

template <int L> struct Log2 { static constexpr int v = 1 + Log2<L / 2>::v; };
template <> struct Log2<1> { static constexpr int v = 0; };

// cos(pi m / 8), m = 0..15: exact values of the sixteenth roots of unity.
__host__ __device__ constexpr double cos16(int m) {
    return m == 0 ? 1.0 : m == 1 ? 0.92387953251128675613 : m == 2 ? 0.70710678118654752440
         : m == 3 ? 0.38268343236508977173 : m == 4 ? 0.0 : m == 5 ? -0.38268343236508977173
         : m == 6 ? -0.70710678118654752440 : m == 7 ? -0.92387953251128675613 : m == 8 ? -1.0
         : m == 9 ? -0.92387953251128675613 : m == 10 ? -0.70710678118654752440
         : m == 11 ? -0.38268343236508977173 : m == 12 ? 0.0 : m == 13 ? 0.38268343236508977173
         : m == 14 ? 0.70710678118654752440 : 0.92387953251128675613;
}

template <int M> __host__ __device__ constexpr int brev_c(int i) {
    int r = 0;
    for (int b = 0; b < M; ++b) r |= ((i >> b) & 1) << (M - 1 - b);
    return r;
}

// (a, b) <- (a + w b, a - w b), FP64 only, where the FP64 pipe bounds every pass. Each output comes from the operands
// alone, with no more roundings than a product and a sum have; formed as 2 a - (a + w b), in six operations, the second output
// carried the first one's rounding too (rms error of the 128^3 transform 3.29e-16, 3.13e-16 with product and sums).
// Any w, in eight fused operations:
__device__ __forceinline__ void butterfly_w(double2 &a, double2 &b, double2 w) {
    const double2 p = make_double2(fma(-b.y, w.y, fma(b.x, w.x, a.x)), fma(b.x, w.y, fma(b.y, w.x, a.y)));
    b = make_double2(fma(b.y, w.y, fma(-b.x, w.x, a.x)), fma(-b.x, w.y, fma(-b.y, w.x, a.y)));
    a = p;
}
// A constant w = exp(-2 pi i m / 16), conjugated for inv, m (known to the compiler) neither 0 nor 4, in six: with c the larger
// of its parts and r the ratio of the other to it, w b = c (b + r i b) or c (r b + i b), two operations, and the sums with c
// are fused. 1/sqrt2 rounds up by 0.61 of 2^-53, and a factor |w| above 1 on every such path adds up over the stages (a
// relative error of 2.6e-16 of the whole field after the 128^3 pair): m = 6 takes the next number below, so it cancels.
// Forward, inverse and pair at 128^3, rms: 2.88e-16, 2.89e-16, 4.06e-16; products and sums 3.13e-16, 3.13e-16, 4.76e-16.
__device__ __forceinline__ void butterfly_c(double2 &a, double2 &b, int m, bool inv) {
    const double wc = cos16(m), ws = inv ? cos16((m + 12) & 15) : -cos16((m + 12) & 15);
    const bool re = fabs(wc) >= fabs(ws);
    const double c = (re ? wc : ws) * (m == 6 ? 1.0 - 0x1p-53 : 1.0);
    const double t = m % 4 == 2 ? 1.0 : 0.41421356237309504880, r = (wc < 0) != (ws < 0) ? -t : t;   // tan(pi/4), tan(pi/8)
    const double u = re ? fma(-b.y, r, b.x) : fma(b.x, r, -b.y), v = re ? fma(b.x, r, b.y) : fma(b.y, r, b.x);
    b = make_double2(fma(-c, u, a.x), fma(-c, v, a.y));
    a = make_double2(fma(c, u, a.x), fma(c, v, a.y));
}

// Length-R DFT of x held in registers (radix-2 network with constant twiddles). The forward
// twiddle W_{2h}^p = exp(-2 pi i p / 2h) = (cos(pi m/8), -sin(pi m/8)), m = 16 p / 2h, with
// sin(pi m/8) = cos(pi (m + 12)/8). INV uses the conjugate. The twiddles 1 (m = 0) and -i (m = 4; +i inverse)
// are applied as a copy and a swap with a sign change: without fast-math the compiler keeps the products by
// the zero component, and these are 22 of the 32 twiddles of a 16-point DFT (10 of 12 at 8 points).
template <int R, bool INV, int H0, typename C> __device__ __forceinline__ void dft_stages(C (&x)[R]) {
    using T = decltype(C::x);
#pragma unroll
    for (int h = H0; h < R; h <<= 1) {
#pragma unroll
        for (int g = 0; g < R; g += 2 * h) {
#pragma unroll
            for (int p = 0; p < h; ++p) {
                const int m = p * (16 / (2 * h));
                const C b0 = x[g + p + h];
                if constexpr (sizeof(T) == 8) {
                    if (m != 0 && m != 4) {
                        butterfly_c(x[g + p], x[g + p + h], m, INV);
                        continue;
                    }
                }
                C b;
                if (m == 0) {
                    b = b0;
                } else if (m == 4) {
                    b = INV ? cmk<C>(-b0.y, b0.x) : cmk<C>(b0.y, -b0.x);
                } else {
                    const T wc = (T)cos16(m);
                    const T ws = INV ? (T)cos16((m + 12) & 15) : -(T)cos16((m + 12) & 15);
                    b = cmk<C>(b0.x * wc - b0.y * ws, b0.x * ws + b0.y * wc);
                }
                const C a = x[g + p];
                x[g + p] = cadd(a, b);
                x[g + p + h] = csub(a, b);
            }
        }
    }
}
template <int R, bool INV, typename C> __device__ __forceinline__ void dft_reg(C (&x)[R]) {
    constexpr int LR = Log2<R>::v;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int j = brev_c<LR>(i);
        if (j > i) { const C t = x[i]; x[i] = x[j]; x[j] = t; }
    }
    dft_stages<R, INV, 1>(x);
}

// Length-R DFT of w[r] x[r] (w[0] = 1): the twiddles products first. FP64 (R = 2, 4, 8, 16) takes those of the odd half of
// each first-stage pair into the butterfly: R = 8 in 80 operations instead of 84.
template <int R, bool INV, typename C, typename W> __device__ __forceinline__ void dft_twiddled(C (&x)[R], W w) {
    using T = decltype(C::x);
    if constexpr (sizeof(T) == 4 || R < 2) {
#pragma unroll
        for (int r = 1; r < R; ++r) x[r] = cmul(x[r], w(r));
        dft_reg<R, INV>(x);
    } else {
        // the network of dft_reg: bit-reversed order, then the h = 1 stage pairs elements r and r + R/2
        constexpr int LR = Log2<R>::v;
#pragma unroll
        for (int r = 1; r < R / 2; ++r) x[r] = cmul(x[r], w(r));
#pragma unroll
        for (int r = 0; r < R / 2; ++r) butterfly_w(x[r], x[r + R / 2], w(r + R / 2));
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int j = brev_c<LR>(i);
            if (j > i) { const C t = x[i]; x[i] = x[j]; x[j] = t; }
        }
        dft_stages<R, INV, 2>(x);
    }
}

// Item t of the radix-R1 pass -> (line l, j < M1). With M1 = 8 (N = 128) a half-warp spans two lines of 8 items;
// lines l and l + 1 lie 2 LS = 18 banks apart (mod 32) and share a bank pair, lines l and l + 8 lie 16 apart and
// share none. So within each group of 16 lines the half-warps take lines (l, l + 8); the lines past the last full
// group keep the plain order. Any mapping of items to threads gives the same values.
template <int N> __device__ __forceinline__ void pass1_item(int t, int nlines, int &l, int &j) {
    constexpr int M1 = N / Shape<N>::R1;
    if constexpr (M1 == 8 && Shape<N>::LS % 16 == 9) {
        if (t < (nlines >> 4) * 16 * M1) {
            const int hw = t >> 4, lane = t & 15;
            l = ((hw >> 3) << 4) + (hw & 7) + ((lane >> 3) << 3);
            j = lane & 7;
            return;
        }
    }
    l = t / M1;
    j = t - l * M1;
}

// Element r of a z-pass slab -> (z, column xl < TX) for the column loads, the Green-operator phase and the
// stores. With TX = 8 a half-warp spans 8 columns of two planes; planes z and z + 1 put columns 0 and 7 on one bank
// pair (line stride LS = 9 mod 16), planes z and z + 8 (in one 16-plane block) share none. Global accesses keep
// 8 consecutive columns of a plane per half-warp row.
template <int N, int TX> __device__ __forceinline__ void slab_item(int r, int &z, int &xl) {
    if constexpr (TX == 8 && N % 16 == 0 && Shape<N>::LS % 16 == 9) {
        const int hw = r >> 4, lane = r & 15;
        z = ((hw >> 3) << 4) + (hw & 7) + ((lane >> 3) << 3);
        xl = lane & 7;
    } else {
        z = r / TX;
        xl = r % TX;
    }
}

// The two passes of block_fft (R2 > 1), also called on their own by the z pass.
// pass 1: radix R1, Ns = 1: item (l, j < M1) reads slots j + M1 r and writes j R1 + r, so
// every read completes before any write (held in registers across a barrier). With j < M1 and M1 | R1
// the padded slots are padn(j + M1 r) = j + padn(M1 r) and padn(R1 j + r) = (R1 + 1) j + r (r < R1): one base
// address per item and compile-time offsets. Ends with a barrier.
template <int N, bool INV, int MAXIT, typename C> __device__ void bfft_pass1(C *buf, int nlines) {
    constexpr int R1 = Shape<N>::R1, LS = Shape<N>::LS;
    constexpr int M1 = N / R1;
    static_assert(R1 % M1 == 0, "pass-1 stride");
    const int items = nlines * M1;
    C v[MAXIT][R1];
#pragma unroll
    for (int it = 0; it < MAXIT; ++it) {
        const int t = threadIdx.x + it * blockDim.x;
        if (t < items) {
            int l, j;
            pass1_item<N>(t, nlines, l, j);
            const C *src = buf + l * LS + j;
#pragma unroll
            for (int r = 0; r < R1; ++r) v[it][r] = src[padn<N>(r * M1)];
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < MAXIT; ++it) {
        const int t = threadIdx.x + it * blockDim.x;
        if (t < items) {
            int l, j;
            pass1_item<N>(t, nlines, l, j);
            dft_reg<R1, INV>(v[it]);
            C *dst = buf + l * LS + (R1 + 1) * j;
#pragma unroll
            for (int r = 0; r < R1; ++r) dst[r] = v[it][r];
        }
    }
    __syncthreads();
}

// a * w with the rounding of the FP32 product written out (which product of each sum is fused): FY fuses a.y w.x into the
// imaginary part, else a.x w.y.
template <bool FY> __device__ __forceinline__ float2 cmul_r(float2 a, float2 w) {
    return make_float2(fmaf(a.x, w.x, -__fmul_rn(a.y, w.y)),
                       FY ? fmaf(a.y, w.x, __fmul_rn(a.x, w.y)) : fmaf(a.x, w.y, __fmul_rn(a.y, w.x)));
}
template <bool FY> __device__ __forceinline__ double2 cmul_r(double2 a, double2 w) { return cmul(a, w); }

// The arithmetic of the second pass on the R2 values u[r] of slots j + R1 r, in place. N >= 64: twiddles
// tw[R1 r + j], then a radix-R2 DFT. N <= 32: values r and r + R2/2 are the even and odd halves of a radix-16 DFT, so
// its last stage (W16^j, at tw[N + j]) gives its outputs j and j + 8, which then take the twiddles and the radix-R2/2
// DFT of the 16 x R2/2 split; slot j + 8 q holds its output q.
// FP32: which product of each sum is fused (FY of cmul_r, and the selects below) follows the compiler's choices in the
// radix-16 form, so that a transform of 16 or 32 points rounded as it did before the split (compared bit by bit when
// this form came in). Either choice rounds the same number of times; nothing depends on it.
template <int N, bool INV, bool FY = true, typename C> __device__ __forceinline__ void pass2_tail(C (&u)[Shape<N>::R2], int j, const C *tw) {
    constexpr int R1 = Shape<N>::R1, R2 = Shape<N>::R2;
    auto tw_at = [&](int i) {
        C w = tw[i];
        if (INV) w.y = -w.y;
        return w;
    };
    if constexpr (R1 == 16) {
        dft_twiddled<R2, INV>(u, [&](int r) { return tw_at(16 * r + j); });
    } else {
        constexpr int Q = R2 / 2;
        const C w = tw_at(N + j);
        C a[Q], b[Q];
#pragma unroll
        for (int r = 0; r < Q; ++r) {
            if constexpr (sizeof(C) == 16) {
                a[r] = u[r];
                b[r] = u[r + Q];
                butterfly_w(a[r], b[r], w);
                continue;
            }
            const C y = u[r + Q];
            C z;
            if constexpr (sizeof(C) == 8) {
                // rounded as dft_reg's products by constants are (which product of a sum is fused)
                const bool fx = !(j == 6 && !INV), fy = j == 2;
                const float px = fx ? y.x : -y.y, qx = fx ? w.x : w.y, rx = fx ? -y.y : y.x, tx = fx ? w.y : w.x;
                const float py = fy ? y.x : y.y, qy = fy ? w.y : w.x, ry = fy ? y.y : y.x, ty = fy ? w.x : w.y;
                z.x = fmaf(px, qx, __fmul_rn(rx, tx));
                z.y = fmaf(py, qy, __fmul_rn(ry, ty));
            }
            if (j == 0) z = y;   // as in dft_reg: the twiddles 1 and -i (+i inverse) are not multiplied
            if (j == 4) z = INV ? cmk<C>(-y.y, y.x) : cmk<C>(y.y, -y.x);
            a[r] = cadd(u[r], z);
            b[r] = csub(u[r], z);
        }
        if constexpr (Q > 1 && sizeof(C) == 16) {
            dft_twiddled<Q, INV>(a, [&](int r) { return tw_at(16 * r + j); });
            dft_twiddled<Q, INV>(b, [&](int r) { return tw_at(16 * r + j + 8); });
        } else if constexpr (Q > 1) {
#pragma unroll
            for (int r = 1; r < Q; ++r) {
                a[r] = cmul_r<FY>(a[r], tw_at(16 * r + j));
                b[r] = cmul_r<FY>(b[r], tw_at(16 * r + j + 8));
            }
            dft_reg<Q, INV>(a);
            dft_reg<Q, INV>(b);
        }
#pragma unroll
        for (int r = 0; r < Q; ++r) {
            u[2 * r] = a[r];
            u[2 * r + 1] = b[r];
        }
    }
}

// pass 2: item (l, j < R1) reads and writes slots j + R1 r only, which are padn(j + R1 r) = j + (R1 + 1) r.
// Every CTA has a multiple of R1 threads, so a thread's items share one j = threadIdx.x mod R1; at N >= 64 its
// twiddles tw[R1 r + j] = exp(-2 pi i r j / N) are loaded once, into registers. Ends with a barrier.
template <int N, bool INV, typename C> __device__ void bfft_pass2(C *buf, int nlines, const C *tw) {
    constexpr int R1 = Shape<N>::R1, R2 = Shape<N>::R2, LS = Shape<N>::LS;
    const int jt = threadIdx.x & (R1 - 1);
    if constexpr (R1 == 16) {
        C wr[R2];
#pragma unroll
        for (int r = 1; r < R2; ++r) {
            wr[r] = tw[R1 * r + jt];   // r-major: R1 lanes read R1 in a row
            if (INV) wr[r].y = -wr[r].y;
        }
        for (int t = threadIdx.x; t < nlines * R1; t += blockDim.x) {
            C *line = buf + (t / R1) * LS + jt;
            C u[R2];
#pragma unroll
            for (int r = 0; r < R2; ++r) u[r] = line[(R1 + 1) * r];
            dft_twiddled<R2, INV>(u, [&](int r) { return wr[r]; });
#pragma unroll
            for (int r = 0; r < R2; ++r) line[(R1 + 1) * r] = u[r];
        }
    } else {
        for (int t = threadIdx.x; t < nlines * R1; t += blockDim.x) {
            C *line = buf + (t / R1) * LS + jt;
            C u[R2];
#pragma unroll
            for (int r = 0; r < R2; ++r) u[r] = line[(R1 + 1) * r];
            pass2_tail<N, INV, !(N == 32 && !INV)>(u, jt, tw);
#pragma unroll
            for (int r = 0; r < R2; ++r) line[(R1 + 1) * r] = u[r];
        }
    }
    __syncthreads();
}

// In-place transform of nlines padded lines (line l at buf + l*LS). tw: see load_tw. Starts after and ends with a
// barrier. MAXIT >= ceil(nlines * (N/R1) / blockDim).
template <int N, bool INV, int MAXIT, typename C> __device__ void block_fft(C *buf, int nlines, const C *tw) {
    constexpr int R1 = Shape<N>::R1, R2 = Shape<N>::R2, LS = Shape<N>::LS;
    if constexpr (R2 == 1) {   // a single radix-N pass; every line is owned by one thread
        for (int l = threadIdx.x; l < nlines; l += blockDim.x) {
            C v[R1];
#pragma unroll
            for (int r = 0; r < R1; ++r) v[r] = buf[l * LS + padn<N>(r)];
            dft_reg<R1, INV>(v);
#pragma unroll
            for (int r = 0; r < R1; ++r) buf[l * LS + padn<N>(r)] = v[r];
        }
        __syncthreads();
    } else {
        bfft_pass1<N, INV, MAXIT>(buf, nlines);
        bfft_pass2<N, INV>(buf, nlines, tw);
    }
}

// cos(2 pi k / 256), k = 0 .. 64, rounded to nearest: the FP64 twiddles of every N <= 256 by symmetry. Reading them
// replaces a sincospi per CTA and twiddle: 128 of them were about a tenth of an FP64 z-pass CTA's FP64 operations.
// (The FP32 twiddles stay sincospif's, on the FP32 pipe.)
__device__ const double kCos256[65] = {
    1.0, 0.9996988186962042, 0.9987954562051724, 0.9972904566786902, 0.9951847266721969,
    0.99247953459871, 0.989176509964781, 0.9852776423889412, 0.9807852804032304, 0.9757021300385286,
    0.970031253194544, 0.9637760657954398, 0.9569403357322088, 0.9495281805930367, 0.9415440651830208,
    0.9329927988347388, 0.9238795325112867, 0.9142097557035307, 0.9039892931234433, 0.8932243011955153,
    0.881921264348355, 0.8700869911087115, 0.8577286100002721, 0.8448535652497071, 0.8314696123025452,
    0.8175848131515837, 0.8032075314806449, 0.7883464276266062, 0.773010453362737, 0.7572088465064846,
    0.7409511253549591, 0.7242470829514669, 0.7071067811865476, 0.6895405447370669, 0.6715589548470184,
    0.6531728429537768, 0.6343932841636455, 0.6152315905806268, 0.5956993044924334, 0.5758081914178453,
    0.5555702330196022, 0.5349976198870973, 0.5141027441932218, 0.49289819222978404, 0.47139673682599764,
    0.4496113296546066, 0.4275550934302821, 0.40524131400498986, 0.3826834323650898, 0.35989503653498817,
    0.33688985339222005, 0.31368174039889146, 0.2902846772544624, 0.26671275747489837, 0.2429801799032639,
    0.2191012401568698, 0.19509032201612828, 0.17096188876030122, 0.14673047445536175, 0.1224106751992162,
    0.0980171403295606, 0.07356456359966743, 0.049067674327418015, 0.024541228522912288, 0.0,
};
// exp(-2 pi i k / 256), 0 <= k < 256
__device__ __forceinline__ double2 root256(int k) {
    const int q = k >> 6, m = k & 63;
    const double c = __ldg(kCos256 + m), d = __ldg(kCos256 + 64 - m);   // cos, sin of the angle within its quarter
    return q == 0 ? make_double2(c, -d) : q == 1 ? make_double2(-d, -c) : q == 2 ? make_double2(-c, d) : make_double2(d, c);
}
__device__ __forceinline__ float2 root_of(float2, int k, int N) {   // exp(-2 pi i k / N)
    float sn, cs;
    sincospif(-2.0f * (float)k / (float)N, &sn, &cs);
    return make_float2(cs, sn);
}
__device__ __forceinline__ double2 root_of(double2, int k, int N) { return root256(k * (256 / N)); }
// Twiddles into shared memory, once per CTA: slot 16 r + j holds exp(-2 pi i r j / N) for r < N / 16, j < 16 (r j < N),
// so lanes that differ in j read consecutive slots; with radix-8 first passes slots N .. N + 7 hold W16^0 .. W16^7.
template <int N, typename C> __device__ __forceinline__ void load_tw(C *tw_s) {
    using T = decltype(C::x);
    for (int k = threadIdx.x; k < Shape<N>::NTW; k += blockDim.x) {
        if (k < N) {
            tw_s[k] = root_of(C{}, (k >> 4) * (k & 15), N);
        } else {
            const double2 w = root256(16 * (k - N));
            tw_s[k] = cmk<C>((T)w.x, (T)w.y);
        }
    }
}

template <int N> __host__ __device__ constexpr int rowpairs() { return N >= 64 ? 32 : 4096 / (N * 2); }
// Column tiles of the half spectrum (kx = 0..N/2): N/2 columns split into full tiles of TXe, and the
// Nyquist column kx = N/2 appended to tile 0 as one extra line, so no tile is ragged.
template <int N, typename T> __host__ __device__ constexpr int tx_y() {
    return (sizeof(T) == 4 ? 32 : 16) < N / 2 ? (sizeof(T) == 4 ? 32 : 16) : N / 2;
}
// z-pass tiles: 64-byte column segments; two columns on grids of 16 and 32, where wider tiles would leave most of the
// chip idle (32^3 FP32: 256 CTAs instead of 64).
__host__ __device__ constexpr int tx_z_of(int n, int tsize) {
    return n <= 8 ? n / 2 : n <= 32 ? 2 : 32 / tsize;
}
template <int N, typename T> __host__ __device__ constexpr int tx_z() { return tx_z_of(N, sizeof(T)); }
template <int N> __host__ __device__ constexpr int maxit(int lines, int threads = kThreads) {
    return (lines * (N / Shape<N>::R1) + threads - 1) / threads < 1 ? 1
                                                                   : (lines * (N / Shape<N>::R1) + threads - 1) / threads;
}
// Threads of a column-tile CTA: enough that a tile with its extra Nyquist lines (lines + extra)
// needs no more pass-1 register sets than a full tile would at kThreads (the extra set would raise
// register use, and so cut occupancy, for every tile).
template <int N> __host__ __device__ constexpr int tile_threads(int lines, int extra) {
    return ((((lines + extra) * (N / Shape<N>::R1) + maxit<N>(lines) - 1) / maxit<N>(lines) + 31) / 32) * 32 < kThreads
               ? kThreads
               : ((((lines + extra) * (N / Shape<N>::R1) + maxit<N>(lines) - 1) / maxit<N>(lines) + 31) / 32) * 32;
}
template <int N, typename T> __host__ __device__ constexpr int y_threads() { return tile_threads<N>(tx_y<N, T>(), 1); }
// z pass of 256^3 in FP32: the Nyquist column in CTAs of its own (TX rows ky each) instead of on tile 0. Its six lines
// more are what keeps a second CTA off the SM (118 KB of shared memory instead of 106 KB): 432 us a pass with one CTA of
// 288 threads, 387 us with two of 256 (390 us with 384 threads, 419 us with 512). At 128^3 three CTAs fit either way
// (46.4 us, 44.8 us apart), and the residual's sums, which go tile by tile, keep their order there and in Z_FWD_RESID.
__host__ __device__ constexpr bool z_split_of(int n, int tsize) { return n >= 256 && tsize == 4; }
template <int N, typename T, bool SPLIT> __host__ __device__ constexpr int z_threads() {
    return SPLIT ? kThreads : N == 16 || N == 32 ? 128 : tile_threads<N>(6 * tx_z<N, T>(), 6);
}
template <int N, typename T, bool SPLIT> __host__ __device__ constexpr int z_ctas() {
    return SPLIT ? 2 : sizeof(T) == 4 && N <= 128 ? 3 : 1;
}

// ---------------------------------------------------------------------------------------------
// x pass, real -> half spectrum. CTA = RP pairs of rows (y even, y+1) of one (field, z).
// ---------------------------------------------------------------------------------------------
template <typename T, int N>
__global__ void __launch_bounds__(kThreads, N >= 64 && N <= 128 ? (sizeof(T) == 4 ? 6 : 3) : 1) k_fft_x_r2c(const T *__restrict__ in, typename CT<T>::type *__restrict__ out,
                                                       long npairs, const int *__restrict__ skip) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW;
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    constexpr int RP = rowpairs<N>(), LS = Shape<N>::LS, Hx = N / 2 + 1;
    const long p0 = (long)blockIdx.x * RP;
    const int np = (int)min((long)RP, npairs - p0);
    for (int t = threadIdx.x; t < np * N; t += blockDim.x) {
        const int pl = t / N, j = t - pl * N;
        const long row0 = 2 * (p0 + pl);            // global row index = (field*N + z)*N + y
        T *slot = reinterpret_cast<T *>(buf + pl * LS + padn<N>(j));
        cp_async<sizeof(T)>(slot, in + row0 * N + j);
        cp_async<sizeof(T)>(slot + 1, in + (row0 + 1) * N + j);
    }
    cp_async_wait_all();
    __syncthreads();
    block_fft<N, false, maxit<N>(RP)>(buf, np, tw);
    const T h = (T)0.5;
    for (int t = threadIdx.x; t < np * Hx; t += blockDim.x) {
        const int pl = t / Hx, k = t - pl * Hx;
        const C zk = buf[pl * LS + padn<N>(k & (N - 1))];
        const C zc = cconj(buf[pl * LS + padn<N>((N - k) & (N - 1))]);
        const long row0 = 2 * (p0 + pl);
        out[row0 * Hx + k] = cmk<C>(h * (zk.x + zc.x), h * (zk.y + zc.y));
        out[(row0 + 1) * Hx + k] = cmk<C>(h * (zk.y - zc.y), -h * (zk.x - zc.x));   // (zk - zc) / 2i
    }
}

// ---------------------------------------------------------------------------------------------
// x pass, half spectrum -> real (complex-to-real through the same row-pair packing). The CTA's rows
// are contiguous in both the half spectrum and the strain, so both arrive by 16-byte asynchronous
// copies into shared memory before the transform; every global access is then a wide, coalesced one.
// ---------------------------------------------------------------------------------------------
template <int N> __host__ __device__ constexpr int rowpairs_c2r() { return rowpairs<N>() > 16 ? 16 : rowpairs<N>(); }

template <typename T, int N>
__global__ void __launch_bounds__(kThreads) k_fft_x_c2r(const typename CT<T>::type *__restrict__ spec, T *__restrict__ out,
                                                       long npairs, T scale, int has_add, T a0, T a1, T a2, T a3, T a4,
                                                       T a5, const T *__restrict__ base, const int *__restrict__ skip,
                                                       const double *__restrict__ dadd) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW;                          // RP packed lines
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    constexpr int RP = rowpairs_c2r<N>(), LS = Shape<N>::LS, Hx = N / 2 + 1;
    C *hs = buf + RP * LS;                    // 2 RP half-spectrum rows, row-major
    T *bs = reinterpret_cast<T *>(hs + 2 * RP * Hx);   // 2 RP strain rows (with has_add)
    const long p0 = (long)blockIdx.x * RP;
    const int np = (int)min((long)RP, npairs - p0);
    {   // rows 2 p0 .. 2 (p0 + np) - 1: contiguous, 16-byte aligned (2 Hx sizeof(C) and 2 N sizeof(T) are)
        const uint4 *src = reinterpret_cast<const uint4 *>(spec + 2 * p0 * Hx);
        uint4 *dst = reinterpret_cast<uint4 *>(hs);
        const int nchunk = (int)(2 * np * Hx * sizeof(C) / 16);
        for (int t = threadIdx.x; t < nchunk; t += blockDim.x) cp_async<16>(dst + t, src + t);
        if (has_add) {
            const T *bsrc = base ? base : out;
            const uint4 *src2 = reinterpret_cast<const uint4 *>(bsrc + 2 * p0 * N);
            uint4 *dst2 = reinterpret_cast<uint4 *>(bs);
            const int nchunk2 = (int)(2 * np * N * sizeof(T) / 16);
            for (int t = threadIdx.x; t < nchunk2; t += blockDim.x) cp_async<16>(dst2 + t, src2 + t);
        }
    }
    cp_async_wait_all();
    __syncthreads();
    for (int t = threadIdx.x; t < np * N; t += blockDim.x) {
        const int pl = t / N, k = t - pl * N;
        const C *ra = hs + 2 * pl * Hx, *rb = ra + Hx;
        C A, B;
        if (k <= (N >> 1)) {
            A = ra[k];
            B = rb[k];
        } else {
            A = cconj(ra[N - k]);
            B = cconj(rb[N - k]);
        }
        buf[pl * LS + padn<N>(k)] = cmk<C>(A.x - B.y, A.y + B.x);   // A + iB
    }
    __syncthreads();
    block_fft<N, true, maxit<N>(RP)>(buf, np, tw);
    // the offset of a row's field, formed once where the CTA's rows belong to one field (256^3 FP32: 246 us a pass, 287
    // with the selection in the loop)
    auto add_of = [&](long row) -> T {
        const int f = (int)(row / ((long)N * N));
        return dadd ? (T)dadd[f] : f == 0 ? a0 : f == 1 ? a1 : f == 2 ? a2 : f == 3 ? a3 : f == 4 ? a4 : a5;
    };
    constexpr bool one_field = (N * N) % (2 * RP) == 0;
    const T add_cta = one_field && has_add ? add_of(2 * p0) : (T)0;
    for (int t = threadIdx.x; t < np * N; t += blockDim.x) {
        const int pl = t / N, j = t - pl * N;
        const long row0 = 2 * (p0 + pl);
        const C z = buf[pl * LS + padn<N>(j)];
        if (has_add) {
            const T add = one_field ? add_cta : add_of(row0);
            out[row0 * N + j] = bs[2 * pl * N + j] + (z.x * scale + add);
            out[(row0 + 1) * N + j] = bs[(2 * pl + 1) * N + j] + (z.y * scale + add);
        } else {
            out[row0 * N + j] = z.x;
            out[(row0 + 1) * N + j] = z.y;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// y pass: CTA = (field, z, kx tile of TX columns); lines along y.
// ---------------------------------------------------------------------------------------------
template <typename T, int N, bool INV>
__global__ void __launch_bounds__(y_threads<N, T>(), sizeof(T) == 4 && N >= 64 && N <= 128 ? 5 : 1)
k_fft_y(typename CT<T>::type *__restrict__ spec, const int *__restrict__ skip, InvCtl ic) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW;
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    constexpr int TX = tx_y<N, T>(), LS = Shape<N>::LS, Hx = N / 2 + 1;
    if (INV && ic.ctl != nullptr && blockIdx.x == gridDim.x - 1) {   // as in k_fft_xy_c2r
        if (threadIdx.x == 0) fp_next_tolerance(ic);
        return;
    }
    constexpr int ntiles = (N / 2) / TX;
    const int tile = blockIdx.x % ntiles;
    const long plane = blockIdx.x / ntiles;        // field*N + z
    const bool nyq = tile == 0;                    // tile 0 also carries the column kx = N/2 as line TX
    C *base = spec + plane * (long)N * Hx;
    const int kx0 = tile * TX;
    for (int t = threadIdx.x; t < TX * N; t += blockDim.x) {   // TX, N powers of two: shifts, no division
        const int y = t / TX, xl = t % TX;
        cp_async<sizeof(C)>(buf + xl * LS + padn<N>(y), base + (long)y * Hx + kx0 + xl);
    }
    if (nyq)
        for (int y = threadIdx.x; y < N; y += blockDim.x)
            cp_async<sizeof(C)>(buf + TX * LS + padn<N>(y), base + (long)y * Hx + N / 2);
    cp_async_wait_all();
    // the macroscopic strain correction goes into the zero-frequency term (this thread copied it)
    if (INV && ic.ctl != nullptr && tile == 0 && threadIdx.x == 0) buf[0].x += (T)(ic.ctl->corr[plane / N] * ic.n3);
    __syncthreads();
    block_fft<N, INV, maxit<N>(TX + 1, y_threads<N, T>())>(buf, TX + (nyq ? 1 : 0), tw);
    for (int t = threadIdx.x; t < TX * N; t += blockDim.x) {
        const int y = t / TX, xl = t % TX;
        base[(long)y * Hx + kx0 + xl] = buf[xl * LS + padn<N>(y)];
    }
    if (nyq)
        for (int y = threadIdx.x; y < N; y += blockDim.x) base[(long)y * Hx + N / 2] = buf[TX * LS + padn<N>(y)];
}

// ---------------------------------------------------------------------------------------------
// x and y passes fused: CTA = one (field, z) plane held in shared memory. The x transform runs on
// N/2 packed row pairs (line p = rows 2p, 2p+1, as in the x pass); the half-spectrum rows then replace
// their line in place (row 2p at slots 0..N/2 of line p, row 2p+1 at slots N/2+1..N+1), and the y
// transform runs down the N/2+1 columns of that row-major plane. Every value goes through the same
// operations, in the same order, as in the separate x and y passes, so the spectra are bitwise the same;
// the plane crosses HBM once instead of twice. Used where the plane fits (xy_fused).
// ---------------------------------------------------------------------------------------------
// One thread per pass-1 item of the N/2 row-pair lines (x) and of the N/2 regular columns (y); the Nyquist
// column's few pass-1 items run on lanes of warp 0 (col_pass1).
template <int N> __host__ __device__ constexpr int xy_threads() {
    return N == 16 ? 64 : N == 32 ? 128 : (((N / 2) * (N / Shape<N>::R1) + 31) / 32) * 32;
}
template <typename T, int N> __host__ __device__ constexpr size_t smem_xy() {
    return sizeof(typename CT<T>::type) * (Shape<N>::NTW + (size_t)(N / 2) * Shape<N>::LS);
}
// The plane fits next to two others on one SM (FP32 up to N = 128, FP64 up to N = 64), the row pair of the
// half spectrum fits in a padded line (2 (N/2+1) <= LS), and both passes are two-radix Stockham passes.
template <typename T, int N> __host__ __device__ constexpr bool xy_fused() {
    return N >= 16 && Shape<N>::R2 > 1 && 2 * (N / 2 + 1) <= Shape<N>::LS && smem_xy<T, N>() <= 72 * 1024;
}
template <typename T, int N> __host__ __device__ constexpr int xy_ctas() {
    return sizeof(T) == 4 ? (N >= 128 ? 3 : N == 64 ? 8 : 4) : 1;
}

// Slot of half-spectrum row y, column kx in the row-major plane (rows 2p and 2p+1 share line p).
template <int N> __device__ __forceinline__ int xy_at(int y, int kx) {
    return (y >> 1) * Shape<N>::LS + (y & 1) * (N / 2 + 1) + kx;
}

// The passes of the plane transforms, one pass-1 item per thread (blockDim.x >= items). Each has the items,
// operands and twiddles of block_fft's passes (x: lines of the packed row pairs) or of the y pass (columns,
// addressed through xy_at, kx-fastest so a warp touches consecutive slots); only where the values come from
// or go to differs: the first pass of the forward kernel reads HBM straight into registers, and so do the
// inverse kernel's first pass and the forward kernel's last pass store, so none of them round-trips through
// shared memory.

// x pass 1 (bfft_pass1's items) with element e of line l read through ld(l, e). IN_PLACE: ld reads the lines the
// pass writes, so every read comes before any write (a barrier between); otherwise it reads HBM. Ends with a barrier.
template <int N, bool INV, bool IN_PLACE, typename C, typename Ld> __device__ void x_pass1_ld(C *buf, int nlines, Ld ld) {
    constexpr int R1 = Shape<N>::R1, LS = Shape<N>::LS, M1 = N / R1;
    static_assert(R1 % M1 == 0, "pass-1 stride");
    const int t = threadIdx.x;
    const bool on = t < nlines * M1;
    int l = 0, j = 0;
    if (on) pass1_item<N>(t, nlines, l, j);
    C v[R1];
    if (on) {
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = ld(l, j + M1 * r);
    }
    if constexpr (IN_PLACE) __syncthreads();
    if (on) {
        dft_reg<R1, INV>(v);
        C *dst = buf + l * LS + (R1 + 1) * j;
#pragma unroll
        for (int r = 0; r < R1; ++r) dst[r] = v[r];
    }
    __syncthreads();
}

// y pass 1: item (kx, j < M1) takes rows j + M1 r of column kx through ld(y, kx) and writes rows R1 j + r (line
// R1 j / 2 + r / 2, half r & 1). IN_PLACE: ld reads the buffer the pass writes, so every read comes before any write
// (a barrier between). The regular columns kx < N/2 take one item per thread; the Nyquist column's M1 items then run
// on lanes 0..M1-1 of warp 0 (no other item writes that column), reading its rows through ldn(y), which must not
// read what the regular items write (pre(), run by every thread in the read phase, could copy them aside); a warp
// barrier orders those lanes' reads before their in-place writes. Ends with a barrier.
template <int N, bool INV, bool IN_PLACE, typename C, typename Ld, typename Pre, typename LdN>
__device__ void col_pass1(C *buf, Ld ld, Pre pre, LdN ldn) {
    constexpr int R1 = Shape<N>::R1, M1 = N / R1, Hx = N / 2 + 1, LS = Shape<N>::LS;
    static_assert(M1 % 2 == 0 && R1 % 2 == 0 && M1 <= 32, "row pairs");
    auto transform = [&](int j, int kx, C (&v)[R1]) {
        dft_reg<R1, INV>(v);
        C *dst = buf + (R1 / 2) * j * LS + kx;
#pragma unroll
        for (int r = 0; r < R1; ++r) dst[(r >> 1) * LS + (r & 1) * Hx] = v[r];
    };
    const int t = threadIdx.x;
    const bool on = t < (N / 2) * M1;
    const int j = t / (N / 2), kx = t % (N / 2);
    C v[R1];
    if (on) {
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = ld(j + M1 * r, kx);
    }
    pre();
    if constexpr (IN_PLACE) __syncthreads();
    if (on) transform(j, kx, v);
    if (t < M1) {
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = ldn(t + M1 * r);
        __syncwarp((1u << M1) - 1u);   // ldn may read the column these lanes write
        transform(t, N / 2, v);
    }
    __syncthreads();
}

// y pass 2: item (kx, j < R1) transforms rows j + R1 r (line (j >> 1) + R1 / 2 r, half j & 1) and hands its outputs
// (row j + R1 r in u[r]) to st(j, kx, slot of row j, u). Ends with a barrier.
template <int N, bool INV, typename C, typename St> __device__ void col_pass2(C *buf, const C *tw, St st) {
    constexpr int R1 = Shape<N>::R1, R2 = Shape<N>::R2, Hx = N / 2 + 1, LS = Shape<N>::LS;
    for (int t = threadIdx.x; t < Hx * R1; t += blockDim.x) {
        const int j = t / Hx, kx = t - j * Hx;
        C *line = buf + xy_at<N>(j, kx);
        C u[R2];
#pragma unroll
        for (int r = 0; r < R2; ++r) u[r] = line[r * (R1 / 2) * LS];
        pass2_tail<N, INV>(u, j, tw);
        st(j, kx, line, u);
    }
    __syncthreads();
}

// The two half-spectrum rows of each packed line, in place (row 2p at slots 0..N/2, row 2p+1 at N/2+1..N+1): one line per
// warp, which reads the line's values before it writes.
template <int N, typename C> __device__ __forceinline__ void unpack_rows(C *buf, int nlines) {
    constexpr int LS = Shape<N>::LS, Hx = N / 2 + 1, KU = (Hx + 31) / 32;
    const int lane = threadIdx.x & 31;
    const auto h = (decltype(buf->x))0.5;
    for (int p = threadIdx.x >> 5; p < nlines; p += blockDim.x >> 5) {
        C *line = buf + p * LS;
        C a[KU], b[KU];
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            const int k = lane + 32 * u;
            if (k < Hx) {
                const C zk = line[padn<N>(k & (N - 1))];
                const C zc = cconj(line[padn<N>((N - k) & (N - 1))]);
                a[u] = cmk<C>(h * (zk.x + zc.x), h * (zk.y + zc.y));
                b[u] = cmk<C>(h * (zk.y - zc.y), -h * (zk.x - zc.x));   // (zk - zc) / 2i
            }
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            const int k = lane + 32 * u;
            if (k < Hx) {
                line[k] = a[u];
                line[Hx + k] = b[u];
            }
        }
        __syncwarp();
    }
}

template <typename T, int N>
__global__ void __launch_bounds__(xy_threads<N>(), xy_ctas<T, N>())
k_fft_xy_r2c(const T *__restrict__ in, typename CT<T>::type *__restrict__ out, const int *__restrict__ skip) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW;
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    constexpr int Hx = N / 2 + 1, NP = N / 2, R2 = Shape<N>::R2;
    const T *src = in + (long)blockIdx.x * N * N;   // plane = field * N + z
    C *dst = out + (long)blockIdx.x * N * Hx;
    // x: line p packs rows 2p and 2p+1 as one complex row; pass 1 reads them from HBM
    x_pass1_ld<N, false, false>(buf, NP, [&](int p, int e) { return cmk<C>(src[(2 * p) * N + e], src[(2 * p + 1) * N + e]); });
    bfft_pass2<N, false>(buf, NP, tw);
    unpack_rows<N>(buf, NP);
    __syncthreads();
    // y: down the columns of the row-major plane; pass 2 stores rows j + R1 r to HBM
    col_pass1<N, false, true>(
        buf, [&](int y, int kx) { return buf[xy_at<N>(y, kx)]; }, [] {}, [&](int y) { return buf[xy_at<N>(y, N / 2)]; });
    col_pass2<N, false>(buf, tw, [&](int j, int kx, C *, const C (&u)[R2]) {
#pragma unroll
        for (int r = 0; r < R2; ++r) dst[(j + Shape<N>::R1 * r) * Hx + kx] = u[r];
    });
}

// The inverse: y transform down the columns, the row pairs packed as one complex line (A + iB), the x
// transform, and the strain update of the x pass's epilogue.
template <typename T, int N>
__global__ void __launch_bounds__(xy_threads<N>(), xy_ctas<T, N>())
k_fft_xy_c2r(const typename CT<T>::type *__restrict__ spec, T *__restrict__ out, T scale, int has_add, T a0, T a1, T a2,
             T a3, T a4, T a5, const T *__restrict__ base, const int *__restrict__ skip,
             InvCtl ic) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW;
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    constexpr int LS = Shape<N>::LS, Hx = N / 2 + 1, NP = N / 2, R2 = Shape<N>::R2;
    if (ic.ctl != nullptr && blockIdx.x == gridDim.x - 1) {   // an extra CTA prepares the next iteration's tolerance
        if (threadIdx.x == 0) fp_next_tolerance(ic);
        return;
    }
    const C *src = spec + (long)blockIdx.x * N * Hx;
    const T corr = ic.ctl != nullptr ? (T)(ic.ctl->corr[blockIdx.x / N] * ic.n3) : (T)0;
    // y: pass 1 reads the columns from HBM, with the macroscopic strain correction added to the zero-frequency term
    col_pass1<N, true, false>(
        buf,
        [&](int y, int kx) {
            C v = src[y * Hx + kx];
            if (ic.ctl != nullptr && y == 0 && kx == 0) v.x += corr;
            return v;
        },
        [] {}, [&](int y) { return src[y * Hx + N / 2]; });
    col_pass2<N, true>(buf, tw, [](int, int, C *line, const C (&u)[R2]) {
#pragma unroll
        for (int r = 0; r < R2; ++r) line[r * (Shape<N>::R1 / 2) * LS] = u[r];
    });
    // x: pass 1 packs rows 2p and 2p+1 as it reads them (Z[k] = A[k] + i B[k], with A[N-k] = conj A[k] past N/2)
    // and writes the lines in place
    x_pass1_ld<N, true, true>(buf, NP, [&](int p, int k) {
        const C *line = buf + p * LS;
        C A, B;
        if (k <= (N >> 1)) {
            A = line[k];
            B = line[Hx + k];
        } else {
            A = cconj(line[N - k]);
            B = cconj(line[Hx + N - k]);
        }
        return cmk<C>(A.x - B.y, A.y + B.x);
    });
    bfft_pass2<N, true>(buf, NP, tw);
    const long r0 = (long)blockIdx.x * N;   // first row: (field * N + z) * N
    T add = (T)0;
    if (has_add) {
        const int f = (int)(blockIdx.x / N);
        add = ic.dadd ? (T)ic.dadd[f] : f == 0 ? a0 : f == 1 ? a1 : f == 2 ? a2 : f == 3 ? a3 : f == 4 ? a4 : a5;
    }
    const T *bsrc = base ? base : out;
    for (int t = threadIdx.x; t < NP * N; t += blockDim.x) {
        const int p = t / N, j = t - p * N;
        const C z = buf[p * LS + padn<N>(j)];
        const long o0 = (r0 + 2 * p) * N + j, o1 = o0 + N;
        if (has_add) {
            out[o0] = bsrc[o0] + (z.x * scale + add);
            out[o1] = bsrc[o1] + (z.y * scale + add);
        } else {
            out[o0] = z.x;
            out[o1] = z.y;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// The same for planes larger than one SM holds: a cluster of CL CTAs holds the plane. CTA k has the rows
// [2 LB k, 2 LB (k + 1)) as LB packed lines for the x transform and the columns [LB k, LB (k + 1)) for the y transform
// (the last CTA the Nyquist column too); between the two a thread reads the elements of its next item from the CTAs
// that hold them (distributed shared memory), and writes its own CTA's buffer when the whole cluster has read. The
// items, operands and order of operations are those of the separate passes, so the spectra are the same bit by bit.
// Used at 256^3 in FP32 (a plane is 280 KB), where the separate passes cross HBM four times more per iteration and each
// runs near the memory's rate. Forward: 352 us as two passes, 290 us with clusters of 4 (512 threads, 76 KB, two CTAs
// per SM; 342 us with clusters of 2 and one CTA per SM, 306 us with 8). Inverse: 433 us as two passes, 389 us (an
// L2 prefetch of the strain rows ahead of the transforms made it 440 us). At 128^3 in FP64, which the FP64 pipe
// bounds, the same kernels were slower than the separate passes (transform pair 1640-1690 us, 1605 us).
// ---------------------------------------------------------------------------------------------
template <typename T, int N> constexpr int xy_cluster() { return sizeof(T) == 4 && N == 256 ? 4 : 0; }
template <int N, int CL> struct XyPart {
    static constexpr int LB = N / 2 / CL, RB = 2 * LB, P = LB + 1, M1 = N / Shape<N>::R1, NT = LB * M1;
    static constexpr int slots = LB * Shape<N>::LS > N * P ? LB * Shape<N>::LS : N * P;
    template <typename T> static constexpr size_t smem() {
        return sizeof(typename CT<T>::type) * (Shape<N>::NTW + slots + N);
    }
};

template <typename T, int N, int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(XyPart<N, CL>::NT, 2)
k_fft_xy_r2c_cl(const T *__restrict__ in, typename CT<T>::type *__restrict__ out, const int *__restrict__ skip) {
    using C = typename CT<T>::type;
    using X = XyPart<N, CL>;
    constexpr int R1 = Shape<N>::R1, R2 = Shape<N>::R2, Hx = N / 2 + 1, M1 = X::M1, LB = X::LB, RB = X::RB, P = X::P;
    static_assert(R1 == 16 && RB % M1 == 0 && N % M1 == 0, "pass-1 rows of one CTA");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW, *nyq = buf + X::slots;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = blockIdx.x % CL, t = threadIdx.x;
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    const long plane = blockIdx.x / CL;
    const T *src = in + (plane * N + rank * RB) * N;
    C *dst = out + plane * N * Hx;
    x_pass1_ld<N, false, false>(buf, LB, [&](int p, int e) { return cmk<C>(src[(2 * p) * N + e], src[(2 * p + 1) * N + e]); });
    bfft_pass2<N, false>(buf, LB, tw);
    unpack_rows<N>(buf, LB);
    cl.sync();
    const int kxl = t % LB, j1 = t / LB, kx = rank * LB + kxl;
    const bool last = rank == CL - 1;
    C v[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) v[r] = cl.map_shared_rank(buf, M1 * r / RB)[xy_at<N>(j1 + M1 * r % RB, kx)];
    if (last)
        for (int y = t; y < N; y += X::NT) nyq[y] = cl.map_shared_rank(buf, y / RB)[xy_at<N>(y % RB, N / 2)];
    cl.sync();
    auto pass1 = [&](int j, int c) {
        dft_reg<R1, false>(v);
#pragma unroll
        for (int r = 0; r < R1; ++r) buf[(R1 * j + r) * P + c] = v[r];
    };
    pass1(j1, kxl);
    if (last && t < M1) {
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = nyq[t + M1 * r];
        pass1(t, LB);
    }
    __syncthreads();
    auto pass2 = [&](int j, int c) {
        C u[R2];
#pragma unroll
        for (int r = 0; r < R2; ++r) u[r] = buf[(j + R1 * r) * P + c];
        pass2_tail<N, false>(u, j, tw);
#pragma unroll
        for (int r = 0; r < R2; ++r) dst[(j + R1 * r) * Hx + rank * LB + c] = u[r];
    };
    for (int i = t; i < LB * R1; i += X::NT) pass2(i / LB, i % LB);
    if (last && t < R1) pass2(t, LB);
}

template <typename T, int N, int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(XyPart<N, CL>::NT, 2)
k_fft_xy_c2r_cl(const typename CT<T>::type *__restrict__ spec, T *__restrict__ out, T scale, int has_add, T a0, T a1, T a2,
                T a3, T a4, T a5, const T *__restrict__ base, const int *__restrict__ skip, InvCtl ic) {
    using C = typename CT<T>::type;
    using X = XyPart<N, CL>;
    constexpr int R1 = Shape<N>::R1, R2 = Shape<N>::R2, Hx = N / 2 + 1, M1 = X::M1, LB = X::LB, RB = X::RB, P = X::P;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = blockIdx.x % CL, t = threadIdx.x;
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    if (ic.ctl != nullptr && blockIdx.x >= gridDim.x - CL) {   // an extra cluster prepares the next iteration's tolerance
        if (rank == 0 && t == 0) fp_next_tolerance(ic);
        return;
    }
    const long plane = blockIdx.x / CL;
    const int f = (int)(plane / N);
    const C *src = spec + plane * N * Hx;
    const bool last = rank == CL - 1;
    const T *bsrc = base ? base : out;
    const long r0 = plane * N + rank * RB;
    // y: pass 1 from HBM, the macroscopic strain correction added to the zero-frequency term
    auto pass1 = [&](int j, int c) {
        C v[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = src[(j + M1 * r) * Hx + rank * LB + c];
        if (ic.ctl != nullptr && rank == 0 && j == 0 && c == 0) v[0].x += (T)(ic.ctl->corr[f] * ic.n3);
        dft_reg<R1, true>(v);
#pragma unroll
        for (int r = 0; r < R1; ++r) buf[(R1 * j + r) * P + c] = v[r];
    };
    pass1(t / LB, t % LB);
    if (last && t < M1) pass1(t, LB);
    __syncthreads();
    auto pass2 = [&](int j, int c) {   // in place: item (j, c) reads and writes rows j + R1 r
        C u[R2];
#pragma unroll
        for (int r = 0; r < R2; ++r) u[r] = buf[(j + R1 * r) * P + c];
        pass2_tail<N, true>(u, j, tw);
#pragma unroll
        for (int r = 0; r < R2; ++r) buf[(j + R1 * r) * P + c] = u[r];
    };
    for (int i = t; i < LB * R1; i += X::NT) pass2(i / LB, i % LB);
    if (last && t < R1) pass2(t, LB);
    cl.sync();
    // x: pass 1 packs rows 2p and 2p+1 (Z[k] = A[k] + i B[k], with A[N-k] = conj A[k] past N/2); column k is in CTA
    // k / LB. The partner N - k of item j's element r is element R1 - 1 - r of item M1 - j (element R1 - r of itself for
    // j = 0), so each half-spectrum value is read once and the folded half comes by shuffle: 389 us a pass, 472 us with
    // every folded element read from the CTA that holds it.
    static_assert(M1 == 16 && R1 == 16, "a line's items fill a half-warp");
    const int p = t / M1, j = t % M1, row = (rank * RB + 2 * p) * P, mate = (t & 16) | ((M1 - j) & 15);
    C v[R1], w[R1 / 2];
#pragma unroll
    for (int r = 0; r < R1 / 2; ++r) {
        const C *line = cl.map_shared_rank(buf, M1 * r / LB) + row + j + M1 * r % LB;
        const C A = line[0], B = line[P];
        v[r] = cmk<C>(A.x - B.y, A.y + B.x);
        w[r] = cmk<C>(A.x + B.y, B.x - A.y);
    }
#pragma unroll
    for (int r = R1 / 2; r < R1; ++r) {
        v[r].x = __shfl_sync(0xffffffffu, w[R1 - 1 - r].x, mate);
        v[r].y = __shfl_sync(0xffffffffu, w[R1 - 1 - r].y, mate);
        if (j == 0) {
            if (r > R1 / 2) v[r] = w[(R1 - r) % (R1 / 2)];
            else {
                const C *line = cl.map_shared_rank(buf, CL - 1) + row + LB;
                v[r] = cmk<C>(line[0].x - line[P].y, line[0].y + line[P].x);
            }
        }
    }
    cl.sync();
    dft_reg<R1, true>(v);
    {
        C *d = buf + p * Shape<N>::LS + (R1 + 1) * j;
#pragma unroll
        for (int r = 0; r < R1; ++r) d[r] = v[r];
    }
    __syncthreads();
    bfft_pass2<N, true>(buf, LB, tw);
    T add = (T)0;
    if (has_add)
        add = ic.dadd ? (T)ic.dadd[f] : f == 0 ? a0 : f == 1 ? a1 : f == 2 ? a2 : f == 3 ? a3 : f == 4 ? a4 : a5;
#pragma unroll 4
    for (int i = t; i < LB * N; i += X::NT) {
        const int q = i / N, e = i % N;
        const C z = buf[q * Shape<N>::LS + padn<N>(e)];
        const long o0 = (r0 + 2 * q) * N + e, o1 = o0 + N;
        if (has_add) {
            out[o0] = bsrc[o0] + (z.x * scale + add);
            out[o1] = bsrc[o1] + (z.y * scale + add);
        } else {
            out[o0] = z.x;
            out[o1] = z.y;
        }
    }
}

// Constants of the Green operator of the reference medium, formed on the host: the medium, 1/mu0, 1/(2 mu0) and
// c = (lam0+mu0)/(mu0 (lam0+2 mu0)). (As quotients in the kernel they were 90 FP64 operations of every thread.)
template <typename T> struct GammaC { T lam0, mu0, im, ih, c; };

// 1/x for x > 0 from an FP32 seed with two Newton steps (4 multiply-adds; the seed is good to 24 bits).
__device__ __forceinline__ double rcp_pos(double x) {
    double r = (double)__frcp_rn((float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// -Gamma0:sigma at a regular frequency (f1, f2, f3) (not zero, no Nyquist component) and the residual's |xi.sigma|^2,
// xi = w (f1, f2, f3): eps_kh = (n_h v_k + n_k v_h)/(2 mu0) - c n_k n_h (n.v), v = sigma.n, n = xi/|xi|,
// |xi.sigma|^2 = |xi|^2 |v|^2. t: the tensor components 11, 22, 33, 23, 13, 12; s: the result (Mandel).
// FP64 (the FP64 pipe bounds the pass): in terms of xi and one reciprocal, about 95 multiply-adds per frequency where
// normalising xi takes a square root and a division besides. 64^3 FP64 z pass, with GammaC, the tabulated twiddles and
// the butterflies above: 107 us, 133 without them.
template <typename C>
__device__ __forceinline__ double gamma_regular(const C t[6], C s[6], int f1, int f2, int f3, double w,
                                                const GammaC<double> &gc) {
    const double x1 = w * f1, x2 = w * f2, x3 = w * f3;
    const C v1 = cmk<C>(x1 * t[0].x + x2 * t[5].x + x3 * t[4].x, x1 * t[0].y + x2 * t[5].y + x3 * t[4].y);
    const C v2 = cmk<C>(x1 * t[5].x + x2 * t[1].x + x3 * t[3].x, x1 * t[5].y + x2 * t[1].y + x3 * t[3].y);
    const C v3 = cmk<C>(x1 * t[4].x + x2 * t[3].x + x3 * t[2].x, x1 * t[4].y + x2 * t[3].y + x3 * t[2].y);
    const double q = rcp_pos(x1 * x1 + x2 * x2 + x3 * x3);
    const double w1 = x1 * q, w2 = x2 * q, w3 = x3 * q;
    // with a_k = -v_k/(2 mu0) and b_k = a_k + c w_k (xi.v) the entries are w_k (a_k + b_k) and w_h b_k + w_k a_h
    const C ce = cmk<C>(gc.c * (x1 * v1.x + x2 * v2.x + x3 * v3.x), gc.c * (x1 * v1.y + x2 * v2.y + x3 * v3.y));
    const C a1 = cmk<C>(-gc.ih * v1.x, -gc.ih * v1.y), a2 = cmk<C>(-gc.ih * v2.x, -gc.ih * v2.y),
            a3 = cmk<C>(-gc.ih * v3.x, -gc.ih * v3.y);
    const C b1 = cmk<C>(a1.x + w1 * ce.x, a1.y + w1 * ce.y), b2 = cmk<C>(a2.x + w2 * ce.x, a2.y + w2 * ce.y);
    const C b3 = cmk<C>(a3.x + w3 * ce.x, a3.y + w3 * ce.y);
    const double sq2 = 1.41421356237309504880;
    s[0] = cmk<C>(w1 * (a1.x + b1.x), w1 * (a1.y + b1.y));
    s[1] = cmk<C>(w2 * (a2.x + b2.x), w2 * (a2.y + b2.y));
    s[2] = cmk<C>(w3 * (a3.x + b3.x), w3 * (a3.y + b3.y));
    s[3] = cmk<C>(sq2 * (w3 * b2.x + w2 * a3.x), sq2 * (w3 * b2.y + w2 * a3.y));
    s[4] = cmk<C>(sq2 * (w3 * b1.x + w1 * a3.x), sq2 * (w3 * b1.y + w1 * a3.y));
    s[5] = cmk<C>(sq2 * (w2 * b1.x + w1 * a2.x), sq2 * (w2 * b1.y + w1 * a2.y));
    return v1.x * v1.x + v1.y * v1.y + v2.x * v2.x + v2.y * v2.y + v3.x * v3.x + v3.y * v3.y;
}
template <typename C>
__device__ __forceinline__ float gamma_regular(const C t[6], C s[6], int f1, int f2, int f3, float w,
                                               const GammaC<float> &gc) {
    const float inv = 1.0f / sqrtf((float)(f1 * f1 + f2 * f2 + f3 * f3));
    const float n1 = f1 * inv, n2 = f2 * inv, n3 = f3 * inv;
    const C t11 = t[0], t22 = t[1], t33 = t[2], t23 = t[3], t13 = t[4], t12 = t[5];
    const C v1 = cmk<C>(t11.x * n1 + t12.x * n2 + t13.x * n3, t11.y * n1 + t12.y * n2 + t13.y * n3);
    const C v2 = cmk<C>(t12.x * n1 + t22.x * n2 + t23.x * n3, t12.y * n1 + t22.y * n2 + t23.y * n3);
    const C v3 = cmk<C>(t13.x * n1 + t23.x * n2 + t33.x * n3, t13.y * n1 + t23.y * n2 + t33.y * n3);
    const C nv = cmk<C>(n1 * v1.x + n2 * v2.x + n3 * v3.x, n1 * v1.y + n2 * v2.y + n3 * v3.y);
    const float im = gc.im, ih = gc.ih, c = gc.c, sq2 = (float)1.41421356237309504880;
    auto diag = [&](float nk, C vk) {
        return cmk<C>(im * nk * vk.x - c * nk * nk * nv.x, im * nk * vk.y - c * nk * nk * nv.y);
    };
    auto off = [&](float nk, C vk, float nh, C vh) {
        return cmk<C>(ih * (nh * vk.x + nk * vh.x) - c * nk * nh * nv.x, ih * (nh * vk.y + nk * vh.y) - c * nk * nh * nv.y);
    };
    const C e11 = diag(n1, v1), e22 = diag(n2, v2), e33 = diag(n3, v3);
    const C e23 = off(n2, v2, n3, v3), e13 = off(n1, v1, n3, v3), e12 = off(n1, v1, n2, v2);
    s[0] = cmk<C>(-e11.x, -e11.y);
    s[1] = cmk<C>(-e22.x, -e22.y);
    s[2] = cmk<C>(-e33.x, -e33.y);
    s[3] = cmk<C>(-sq2 * e23.x, -sq2 * e23.y);
    s[4] = cmk<C>(-sq2 * e13.x, -sq2 * e13.y);
    s[5] = cmk<C>(-sq2 * e12.x, -sq2 * e12.y);
    const float f2s = (float)(f1 * f1 + f2 * f2 + f3 * f3);
    return (w * w * f2s) * (v1.x * v1.x + v1.y * v1.y + v2.x * v2.x + v2.y * v2.y + v3.x * v3.x + v3.y * v3.y);
}

// Green operator of the isotropic reference medium applied to one spectral stress (Mandel) of frequency index
// (kx, ky, kz): gamma_regular, except that at frequencies with a Nyquist component the compliance of the reference
// medium replaces it and the zero frequency is left to the macroscopic update. Returns -Gamma:sigma in s (in place) if
// apply, and accumulates the residual |xi.sigma|^2 (xi = 2 pi k/N) of the frequency and, for 0 < kx < N/2, of its Hermitian
// partner -k.
template <typename C, typename T>
__device__ __forceinline__ void gamma_point(C s[6], int kx, int ky, int kz, int N, T w, const GammaC<T> &gc, T &acc,
                                            bool partner, bool apply) {
    const int fx = kx;                                   // 0..N/2
    const int fy = ky <= (N >> 1) ? ky : ky - N;
    const int fz = kz <= (N >> 1) ? kz : kz - N;
    const T r2 = (T)0.70710678118654752440;
    const C t11 = s[0], t22 = s[1], t33 = s[2];
    const C t23 = cmk<C>(s[3].x * r2, s[3].y * r2), t13 = cmk<C>(s[4].x * r2, s[4].y * r2),
            t12 = cmk<C>(s[5].x * r2, s[5].y * r2);
    const int h = N >> 1;
    const bool nyq = kx == h || ky == h || kz == h;
    // Where the Green operator is applied (not on a Nyquist plane, not at zero frequency) the residual comes from
    // its v, the same at the Hermitian partner -k
    const bool fused = apply && !nyq && !(fx == 0 && fy == 0 && fz == 0);
    if (fused) {
        const C t[6] = {t11, t22, t33, t23, t13, t12};
        const T vv = gamma_regular(t, s, fx, fy, fz, w, gc);
        acc += (partner ? (T)2 : (T)1) * vv;
        return;
    }
    // equilibrium residual |xi.sigma_hat|^2 at this frequency and, for 0 < kx < N/2, at its Hermitian partner -k
    // (whose signed frequency differs from -xi on Nyquist ky / kz planes)
    const int nparts = partner ? 2 : 1;
    for (int pt = 0; pt < nparts; ++pt) {
        const int gy = pt == 0 ? fy : ((N - ky) % N <= (N >> 1) ? (N - ky) % N : (N - ky) % N - N);
        const int gz = pt == 0 ? fz : ((N - kz) % N <= (N >> 1) ? (N - kz) % N : (N - kz) % N - N);
        const T x1 = w * (pt == 0 ? fx : -fx), x2 = w * gy, x3 = w * gz;
        const C d1 = cmk<C>(x1 * t11.x + x2 * t12.x + x3 * t13.x, x1 * t11.y + x2 * t12.y + x3 * t13.y);
        const C d2 = cmk<C>(x1 * t12.x + x2 * t22.x + x3 * t23.x, x1 * t12.y + x2 * t22.y + x3 * t23.y);
        const C d3 = cmk<C>(x1 * t13.x + x2 * t23.x + x3 * t33.x, x1 * t13.y + x2 * t23.y + x3 * t33.y);
        acc += d1.x * d1.x + d1.y * d1.y + d2.x * d2.x + d2.y * d2.y + d3.x * d3.x + d3.y * d3.y;
    }
    if (!apply) return;
    if (fx == 0 && fy == 0 && fz == 0) {
        for (int i = 0; i < 6; ++i) s[i] = cmk<C>(0, 0);
        return;
    }
    // Nyquist: -S0:sigma, S0 = (1/2mu0)(I - lam0/(3 lam0 + 2 mu0) J)
    const T a = (T)1 / ((T)2 * gc.mu0), b = gc.lam0 / ((T)2 * gc.mu0 * ((T)3 * gc.lam0 + (T)2 * gc.mu0));
    const C tr = cmk<C>(s[0].x + s[1].x + s[2].x, s[0].y + s[1].y + s[2].y);
    for (int i = 0; i < 3; ++i) s[i] = cmk<C>(-(a * s[i].x - b * tr.x), -(a * s[i].y - b * tr.y));
    for (int i = 3; i < 6; ++i) s[i] = cmk<C>(-a * s[i].x, -a * s[i].y);
}

// ---------------------------------------------------------------------------------------------
// z pass: CTA = (ky, kx tile); nf fields x TX columns x N planes in shared memory. SPLIT: the first N / TX CTAs take the
// Nyquist column instead, TX rows ky each.
// ---------------------------------------------------------------------------------------------
template <typename T, int N, bool SPLIT>
__global__ void __launch_bounds__(z_threads<N, T, SPLIT>(), z_ctas<N, T, SPLIT>())
k_fft_z(typename CT<T>::type *__restrict__ spec, int nf, int mode, GammaC<T> gc, double *__restrict__ partials,
        double *__restrict__ mean6, const int *__restrict__ skip, ZCtl zc) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *tw = reinterpret_cast<C *>(smem_raw);
    C *buf = tw + Shape<N>::NTW;
    load_tw<N>(tw);   // constants: under the preceding kernel's tail
    pdl_wait();
    if (skip != nullptr && *skip) return;   // the fixed point has converged
    constexpr int TX = tx_z<N, T>(), LS = Shape<N>::LS, Hx = N / 2 + 1, NT = z_threads<N, T, SPLIT>(),
                  MI = maxit<N>(6 * (SPLIT ? TX : TX + 1), NT);
    __shared__ double red[32];
    constexpr int ntiles = (N / 2) / TX;
    constexpr int NQ = SPLIT ? N / TX : 0;
    const bool column = SPLIT && (int)blockIdx.x < NQ;   // TX rows ky of the Nyquist column
    const int b = (int)blockIdx.x - NQ;
    const int tile = column ? 0 : b % ntiles;
    const int ky0 = column ? (int)blockIdx.x * TX : b / ntiles;
    // lines: f*TX + xl for the TX columns of field f, then (tile 0 without SPLIT) nf*TX + f for the
    // Nyquist column kx = N/2 of field f
    const bool nyq = !SPLIT && tile == 0;
    const int kx0 = column ? N / 2 : tile * TX;
    const int nlines = nf * TX + (nyq ? nf : 0);
    const long col0 = (long)ky0 * Hx + kx0;     // first column of the tile in a plane, and the step to the next
    const int cstep = column ? Hx : 1;
    const long plane = (long)N * Hx;            // one z plane of one field
    const long fstride = plane * N;
    // The slab walk: element r = t mod (TX N) of field f sits at column xl and plane z = slab_item(r). With
    // NT threads and NT | TX N, a thread keeps its column, and its planes advance by DZ = NT / TX per step
    // (slab_item adds DZ to z when r grows by NT, and padn adds DZ + DZ / R1 when DZ is a multiple of R1), so its
    // shared and global addresses advance by constant strides.
    constexpr int DZ = NT / TX, KZ = TX * N / NT;
    constexpr int PZ = Shape<N>::R1, DP = DZ + DZ / PZ;
    constexpr bool walk = N >= 16 && (TX * N) % NT == 0 && DZ % PZ == 0 &&
                          ((TX == 8 && N % 16 == 0 && LS % 16 == 9) ? NT % 128 == 0 : NT % TX == 0);
    int wz = 0, wxl = 0;
    if constexpr (walk) slab_item<N, TX>((int)threadIdx.x, wz, wxl);
    // Item it of an HBM-side step over the slab's lines with L items per line: regular lines (field f, column
    // xl) take it = (f L + i) TX + xl, xl fastest, so 8 lanes touch 8 consecutive columns of one plane; the Nyquist
    // lines (tile 0) follow. Gives the line, the item's index i < L and the column's first element in HBM.
    auto hbm_item = [&](int it, int L, int &l, int &i) -> C * {
        const int nreg = nf * TX * L;
        if (it < nreg) {
            const int xl = it % TX, f = it / (TX * L);
            i = (it / TX) % L;
            l = f * TX + xl;
            return spec + f * fstride + col0 + xl * cstep;
        }
        const int q = it - nreg, f = q / L;
        i = q - f * L;
        l = nf * TX + f;
        return spec + f * fstride + (long)ky0 * Hx + N / 2;
    };
    if (mode != Z_INV) {
        // the forward transform's pass 1 (the whole transform when R2 = 1) straight from HBM: item (line, j < M1)
        // reads elements j + M1 r and writes slots R1 j + r (slot r when R2 = 1), as bfft_pass1
        constexpr int R1 = Shape<N>::R1, M1 = N / R1;
        const int nit = nlines * M1;
        for (int it = threadIdx.x; it < nit; it += blockDim.x) {
            int l, j;
            const C *g = hbm_item(it, M1, l, j);
            C v[R1];
#pragma unroll
            for (int r = 0; r < R1; ++r) v[r] = g[(long)(j + M1 * r) * plane];
            dft_reg<R1, false>(v);
            C *dst = buf + l * LS + (R1 + 1) * j;
#pragma unroll
            for (int r = 0; r < R1; ++r) dst[r] = v[r];
        }
        __syncthreads();
        if constexpr (Shape<N>::R2 > 1) bfft_pass2<N, false>(buf, nlines, tw);
    } else {
        if constexpr (walk) {
            C *sb = buf + wxl * LS + padn<N>(wz);
            const C *gb = spec + (long)wz * plane + col0 + wxl * cstep;
            for (int f = 0; f < nf; ++f) {
#pragma unroll
                for (int k = 0; k < KZ; ++k)
                    cp_async<sizeof(C)>(sb + f * TX * LS + k * DP, gb + f * fstride + (long)k * DZ * plane);
            }
        } else {
            for (int t = threadIdx.x; t < nf * TX * N; t += blockDim.x) {   // TX, N powers of two: shifts
                const int f = t / (TX * N), r = t % (TX * N);
                int z, xl;
                slab_item<N, TX>(r, z, xl);
                cp_async<sizeof(C)>(buf + (f * TX + xl) * LS + padn<N>(z), spec + f * fstride + z * plane + col0 + xl * cstep);
            }
        }
        if (nyq)
            for (int t = threadIdx.x; t < nf * N; t += blockDim.x) {
                const int f = t / N, z = t % N;
                cp_async<sizeof(C)>(buf + (nf * TX + f) * LS + padn<N>(z), spec + f * fstride + z * plane + (long)ky0 * Hx + N / 2);
            }
        cp_async_wait_all();
        __syncthreads();
    }
    unsigned ticket = 0;
    if (mode == Z_FWD_GAMMA_INV || mode == Z_FWD_RESID) {
        const bool apply = mode == Z_FWD_GAMMA_INV;
        T acc = (T)0;   // per-thread sum in the field precision; block and global sums in FP64
        // one frequency: its six field values at p0 + f * fstep in the slab
        auto point = [&](int kz, int kx, int ky, C *p0, int fstep) {
            C s6[6];
            for (int f = 0; f < 6; ++f) s6[f] = p0[f * fstep];
            if (kx == 0 && ky == 0 && kz == 0 && mean6 != nullptr) {
                const double inv = 1.0 / ((double)N * N * N);
                for (int f = 0; f < 6; ++f) mean6[f] = (double)s6[f].x * inv;
            }
            const bool partner = !(kx == 0 || kx == (N >> 1));
            gamma_point<C, T>(s6, kx, ky, kz, N, (T)(6.283185307179586476925 / N), gc, acc, partner, apply);
            if (apply)
                for (int f = 0; f < 6; ++f) p0[f * fstep] = s6[f];
        };
        if constexpr (walk) {   // the same points per thread, in the same order, as the loop below
            C *pb = buf + wxl * LS + padn<N>(wz);
            const int kxw = column ? N / 2 : kx0 + wxl, kyw = column ? ky0 + wxl : ky0;
#pragma unroll
            for (int k = 0; k < KZ; ++k) point(wz + k * DZ, kxw, kyw, pb + k * DP, TX * LS);
            if (nyq)
                for (int t = threadIdx.x; t < N; t += blockDim.x) point(t, N / 2, ky0, buf + nf * TX * LS + padn<N>(t), LS);
        } else {
            const int npts = (TX + (nyq ? 1 : 0)) * N;
            for (int t = threadIdx.x; t < npts; t += blockDim.x) {
                const bool reg = t < TX * N;
                int zr = 0, xr = 0;
                if (reg) slab_item<N, TX>(t, zr, xr);
                const int kz = reg ? zr : t - TX * N;
                const int kx = reg && !column ? kx0 + xr : N / 2, ky = column ? ky0 + xr : ky0;
                const int l0 = reg ? xr : nf * TX, ls = reg ? TX : 1;   // line of field f: l0 + f*ls
                point(kz, kx, ky, buf + l0 * LS + padn<N>(kz), ls * LS);
            }
        }
        __syncthreads();
        const double tot = block_sum((double)acc, red);
        if (threadIdx.x == 0 && partials != nullptr) {
            partials[blockIdx.x] = tot;
            // the block's ticket: taken here, its latency passes under the inverse transform
            if (zc.ctl != nullptr) ticket = fp_take_ticket(zc);
        }
    }
    const bool inv = mode == Z_INV || mode == Z_FWD_GAMMA_INV;
    if constexpr (Shape<N>::R2 > 1) {
        if (inv) {
            bfft_pass1<N, true, MI>(buf, nlines);
            // the inverse transform's pass 2 stored straight to HBM: item (line, j < R1) transforms slots j + R1 r
            // as bfft_pass2 and stores elements j + R1 r
            constexpr int R1 = Shape<N>::R1, R2 = Shape<N>::R2;
            const int nit = nlines * R1;
            for (int it = threadIdx.x; it < nit; it += blockDim.x) {
                int l, j;
                C *g = hbm_item(it, R1, l, j);
                const C *line = buf + l * LS + j;
                C u[R2];
#pragma unroll
                for (int r = 0; r < R2; ++r) u[r] = line[(R1 + 1) * r];
                pass2_tail<N, true>(u, j, tw);
#pragma unroll
                for (int r = 0; r < R2; ++r) g[(long)(j + R1 * r) * plane] = u[r];
            }
        }
    } else if (inv) {
        block_fft<N, true, MI>(buf, nlines, tw);
    }
    if (!inv || Shape<N>::R2 == 1) {   // the slab from shared memory
        if constexpr (walk) {
            const C *sb = buf + wxl * LS + padn<N>(wz);
            C *gb = spec + (long)wz * plane + col0 + wxl * cstep;
            for (int f = 0; f < nf; ++f) {
#pragma unroll
                for (int k = 0; k < KZ; ++k) gb[f * fstride + (long)k * DZ * plane] = sb[f * TX * LS + k * DP];
            }
        } else {
            for (int t = threadIdx.x; t < nf * TX * N; t += blockDim.x) {
                const int f = t / (TX * N), r = t % (TX * N);
                int z, xl;
                slab_item<N, TX>(r, z, xl);
                spec[f * fstride + z * plane + col0 + xl * cstep] = buf[(f * TX + xl) * LS + padn<N>(z)];
            }
        }
        if (nyq)
            for (int t = threadIdx.x; t < nf * N; t += blockDim.x) {
                const int f = t / N, z = t % N;
                spec[f * fstride + z * plane + (long)ky0 * Hx + N / 2] = buf[(nf * TX + f) * LS + padn<N>(z)];
            }
    }
    if (zc.ctl != nullptr) {   // the block with the last ticket runs the fixed-point control (fpctl.cuh)
        if (threadIdx.x >= 32) return;
        if (__shfl_sync(0xffffffffu, ticket, 0) != gridDim.x - 1) return;
        __syncwarp();   // as in k_al_control; the inverse transform's barriers do the same
        fp_control_warp(zc, partials, gridDim.x);
    }
}

template <typename T, int N> size_t smem_x() { return sizeof(typename CT<T>::type) * (Shape<N>::NTW + (size_t)rowpairs<N>() * Shape<N>::LS); }
template <typename T, int N> size_t smem_y() { return sizeof(typename CT<T>::type) * (Shape<N>::NTW + (size_t)(tx_y<N, T>() + 1) * Shape<N>::LS); }
template <typename T, int N> size_t smem_z(int nf, bool split) {
    return sizeof(typename CT<T>::type) * (Shape<N>::NTW + (size_t)nf * (tx_z<N, T>() + (split ? 0 : 1)) * Shape<N>::LS);
}

template <typename K> cudaError_t allow_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename T, int N> cudaError_t x_r2c_n(const T *in, void *spec, int nfields, cudaStream_t s, const int *skip) {
    using C = typename CT<T>::type;
    const long npairs = (long)nfields * N * N / 2;
    const int blocks = (int)((npairs + rowpairs<N>() - 1) / rowpairs<N>());
    const size_t sm = smem_x<T, N>();
    cudaError_t e = allow_smem(k_fft_x_r2c<T, N>, sm);
    if (e != cudaSuccess) return e;
    return launch_k(skip != nullptr, k_fft_x_r2c<T, N>, dim3(blocks), dim3(kThreads), sm, s, in, (C *)spec, npairs, skip);
}

template <typename T, int N>
cudaError_t x_c2r_n(const void *spec, T *out, int nfields, T scale, const double *add6, cudaStream_t s, const T *base,
                    const int *skip, const InvCtl *ic = nullptr) {
    using C = typename CT<T>::type;
    const long npairs = (long)nfields * N * N / 2;
    constexpr int RP = rowpairs_c2r<N>();
    const int blocks = (int)((npairs + RP - 1) / RP);
    const size_t sm = sizeof(C) * (Shape<N>::NTW + (size_t)RP * Shape<N>::LS + 2 * (size_t)RP * (N / 2 + 1)) +
                      sizeof(T) * 2 * (size_t)RP * N;
    cudaError_t e = allow_smem(k_fft_x_c2r<T, N>, sm);
    if (e != cudaSuccess) return e;
    T a[6] = {0, 0, 0, 0, 0, 0};   // rounded to the field precision here, not once per element on the device
    if (add6)
        for (int i = 0; i < 6; ++i) a[i] = (T)add6[i];
    const int has_add = add6 != nullptr;
    return launch_k(skip != nullptr, k_fft_x_c2r<T, N>, dim3(blocks), dim3(kThreads), sm, s, (const C *)spec, out, npairs,
                    scale, has_add, a[0], a[1], a[2], a[3], a[4], a[5], base, skip, ic != nullptr ? ic->dadd : nullptr);
}

template <typename T, int N>
cudaError_t y_n(void *spec, int nfields, int inverse, cudaStream_t s, const int *skip, const InvCtl *icp = nullptr) {
    using C = typename CT<T>::type;
    constexpr int TX = tx_y<N, T>();
    InvCtl ic{};
    if (icp != nullptr) ic = *icp;
    const int blocks = nfields * N * ((N / 2) / TX) + (ic.ctl != nullptr ? 1 : 0);
    const size_t sm = smem_y<T, N>();
    cudaError_t e = inverse ? allow_smem(k_fft_y<T, N, true>, sm) : allow_smem(k_fft_y<T, N, false>, sm);
    if (e != cudaSuccess) return e;
    if (inverse) return launch_k(skip != nullptr, k_fft_y<T, N, true>, dim3(blocks), dim3(y_threads<N, T>()), sm, s, (C *)spec, skip, ic);
    return launch_k(skip != nullptr, k_fft_y<T, N, false>, dim3(blocks), dim3(y_threads<N, T>()), sm, s, (C *)spec, skip, ic);
}

// x and y passes of the forward transform: one launch where the plane fits one CTA (xy_fused) or a cluster, else two
template <typename T, int N> cudaError_t xy_r2c_n(const T *in, void *spec, int nfields, cudaStream_t s, const int *skip) {
    if constexpr (xy_fused<T, N>()) {
        using C = typename CT<T>::type;
        constexpr size_t sm = smem_xy<T, N>();
        cudaError_t e = allow_smem(k_fft_xy_r2c<T, N>, sm);
        if (e != cudaSuccess) return e;
        return launch_k(skip != nullptr, k_fft_xy_r2c<T, N>, dim3(nfields * N), dim3(xy_threads<N>()), sm, s, in,
                        (C *)spec, skip);
    } else if constexpr (xy_cluster<T, N>() > 0) {
        using C = typename CT<T>::type;
        constexpr int CL = xy_cluster<T, N>();
        using X = XyPart<N, CL>;
        constexpr size_t sm = X::template smem<T>();
        cudaError_t e = allow_smem(k_fft_xy_r2c_cl<T, N, CL>, sm);
        if (e != cudaSuccess) return e;
        return launch_k(skip != nullptr, k_fft_xy_r2c_cl<T, N, CL>, dim3(nfields * N * CL), dim3(X::NT), sm, s, in,
                        (C *)spec, skip);
    } else {
        cudaError_t e = x_r2c_n<T, N>(in, spec, nfields, s, skip);
        if (e != cudaSuccess) return e;
        return y_n<T, N>(spec, nfields, 0, s, skip);
    }
}

template <typename T, int N>
cudaError_t xy_c2r_n(const void *spec, T *out, int nfields, T scale, const double *add6, cudaStream_t s, const T *base,
                     const int *skip, const InvCtl *icp) {
    if constexpr (xy_fused<T, N>() || xy_cluster<T, N>() > 0) {
        using C = typename CT<T>::type;
        T a[6] = {0, 0, 0, 0, 0, 0};   // rounded to the field precision here, as in the x pass
        if (add6)
            for (int i = 0; i < 6; ++i) a[i] = (T)add6[i];
        const int has_add = add6 != nullptr;
        InvCtl ic{};
        if (icp != nullptr) ic = *icp;
        if constexpr (!xy_fused<T, N>()) {
            constexpr int CL = xy_cluster<T, N>();
            using X = XyPart<N, CL>;
            constexpr size_t sm = X::template smem<T>();
            cudaError_t e = allow_smem(k_fft_xy_c2r_cl<T, N, CL>, sm);
            if (e != cudaSuccess) return e;
            return launch_k(skip != nullptr, k_fft_xy_c2r_cl<T, N, CL>, dim3((nfields * N + (ic.ctl != nullptr ? 1 : 0)) * CL),
                            dim3(X::NT), sm, s, (const C *)spec, out, scale, has_add, a[0], a[1], a[2], a[3], a[4], a[5],
                            base, skip, ic);
        } else {
            constexpr size_t sm = smem_xy<T, N>();
            cudaError_t e = allow_smem(k_fft_xy_c2r<T, N>, sm);
            if (e != cudaSuccess) return e;
            return launch_k(skip != nullptr, k_fft_xy_c2r<T, N>, dim3(nfields * N + (ic.ctl != nullptr ? 1 : 0)), dim3(xy_threads<N>()), sm, s,
                            (const C *)spec, out, scale, has_add, a[0], a[1], a[2], a[3], a[4], a[5], base, skip, ic);
        }
    } else {
        cudaError_t e = y_n<T, N>(const_cast<void *>(spec), nfields, 1, s, skip, icp);
        if (e != cudaSuccess) return e;
        return x_c2r_n<T, N>(spec, out, nfields, scale, add6, s, base, skip, icp);
    }
}

template <typename T, int N, bool SPLIT>
cudaError_t z_launch(void *spec, int nfields, int mode, double lam0, double mu0, double *partials, double *mean6,
                cudaStream_t s, const int *skip, const ZCtl *zcp) {
    using C = typename CT<T>::type;
    constexpr int TX = tx_z<N, T>();
    const int blocks = N * ((N / 2) / TX) + (SPLIT ? N / TX : 0);
    const size_t sm = smem_z<T, N>(nfields, SPLIT);
    cudaError_t e = allow_smem(k_fft_z<T, N, SPLIT>, smem_z<T, N>(6, SPLIT));
    if (e != cudaSuccess) return e;
    ZCtl zc{};
    if (zcp != nullptr) zc = *zcp;
    GammaC<T> gc{};
    if (mode == Z_FWD_GAMMA_INV) {   // in the field precision, as the kernel would form them
        const T l = (T)lam0, m = (T)mu0;
        gc = GammaC<T>{l, m, (T)1 / m, (T)0.5 / m, (l + m) / (m * (l + (T)2 * m))};
    }
    return launch_k(skip != nullptr, k_fft_z<T, N, SPLIT>, dim3(blocks), dim3(z_threads<N, T, SPLIT>()), sm, s, (C *)spec, nfields, mode,
                    gc, partials, mean6, skip, zc);
}

template <typename T, int N>
cudaError_t z_n(void *spec, int nfields, int mode, double lam0, double mu0, double *partials, double *mean6,
                cudaStream_t s, const int *skip, const ZCtl *zcp) {
    if constexpr (z_split_of(N, sizeof(T)))
        if (mode != Z_FWD_RESID) return z_launch<T, N, true>(spec, nfields, mode, lam0, mu0, partials, mean6, s, skip, zcp);
    return z_launch<T, N, false>(spec, nfields, mode, lam0, mu0, partials, mean6, s, skip, zcp);
}

#define EVP_DISPATCH(N_, CALL)                             \
    switch (N_) {                                          \
        case 4: { constexpr int NN = 4; return CALL; }     \
        case 8: { constexpr int NN = 8; return CALL; }     \
        case 16: { constexpr int NN = 16; return CALL; }   \
        case 32: { constexpr int NN = 32; return CALL; }   \
        case 64: { constexpr int NN = 64; return CALL; }   \
        case 128: { constexpr int NN = 128; return CALL; } \
        case 256: { constexpr int NN = 256; return CALL; } \
        default: return cudaErrorInvalidValue;             \
    }

}  // namespace

int fft_z_blocks(int n, int is_double, int mode) {
    const int t = is_double ? 8 : 4, tx = tx_z_of(n, t);
    return n * ((n / 2) / tx) + (mode != Z_FWD_RESID && z_split_of(n, t) ? n / tx : 0);
}

int fft_xy_fused(int n, int is_double) {
    if (is_double) {
        EVP_DISPATCH(n, (int)(xy_fused<double, NN>() || xy_cluster<double, NN>() > 0))
    }
    EVP_DISPATCH(n, (int)(xy_fused<float, NN>() || xy_cluster<float, NN>() > 0))
}

template <typename T>
cudaError_t fft_xy_r2c(const T *in, void *spec, int n, int nfields, cudaStream_t s, const int *skip) {
    EVP_DISPATCH(n, (xy_r2c_n<T, NN>(in, spec, nfields, s, skip)))
}

template <typename T>
cudaError_t fft_xy_c2r(const void *spec, T *out, int n, int nfields, T scale, const double *add6, cudaStream_t s,
                       const T *base, const int *skip, const InvCtl *ic) {
    // the same contract as the x pass (whole rows in 16-byte chunks where the passes run separately)
    if (((uintptr_t)spec | (uintptr_t)out | (uintptr_t)base) & 15) return cudaErrorInvalidValue;
    EVP_DISPATCH(n, (xy_c2r_n<T, NN>(spec, out, nfields, scale, add6, s, base, skip, ic)))
}

template <typename T>
cudaError_t fft_x_r2c(const T *in, void *spec, int n, int nfields, cudaStream_t s, const int *skip) {
    EVP_DISPATCH(n, (x_r2c_n<T, NN>(in, spec, nfields, s, skip)))
}

template <typename T>
cudaError_t fft_x_c2r(const void *spec, T *out, int n, int nfields, T scale, const double *add6, cudaStream_t s,
                      const T *base, const int *skip, const InvCtl *ic) {
    // the pass copies whole rows in 16-byte chunks
    if (((uintptr_t)spec | (uintptr_t)out | (uintptr_t)base) & 15) return cudaErrorInvalidValue;
    EVP_DISPATCH(n, (x_c2r_n<T, NN>(spec, out, nfields, scale, add6, s, base, skip, ic)))
}

template <typename T>
cudaError_t fft_y(void *spec, int n, int nfields, int inverse, cudaStream_t s, const int *skip, const InvCtl *ic) {
    EVP_DISPATCH(n, (y_n<T, NN>(spec, nfields, inverse, s, skip, ic)))
}

template <typename T>
cudaError_t fft_z(void *spec, int n, int nfields, int mode, double lam0, double mu0, double *partials, double *mean6,
                  cudaStream_t s, const int *skip, const ZCtl *zc) {
    if ((mode == Z_FWD_GAMMA_INV || mode == Z_FWD_RESID) && nfields != 6) return cudaErrorInvalidValue;
    if (zc != nullptr && (mode != Z_FWD_GAMMA_INV || partials == nullptr)) return cudaErrorInvalidValue;
    EVP_DISPATCH(n, (z_n<T, NN>(spec, nfields, mode, lam0, mu0, partials, mean6, s, skip, zc)))
}

#define EVP_FFT_INST(T)                                                                                            \
    template cudaError_t fft_x_r2c<T>(const T *, void *, int, int, cudaStream_t, const int *);                     \
    template cudaError_t fft_x_c2r<T>(const void *, T *, int, int, T, const double *, cudaStream_t, const T *,     \
                                      const int *, const InvCtl *);                                                                \
    template cudaError_t fft_y<T>(void *, int, int, int, cudaStream_t, const int *, const InvCtl *);               \
    template cudaError_t fft_xy_r2c<T>(const T *, void *, int, int, cudaStream_t, const int *);                    \
    template cudaError_t fft_xy_c2r<T>(const void *, T *, int, int, T, const double *, cudaStream_t, const T *,    \
                                       const int *, const InvCtl *);                                               \
    template cudaError_t fft_z<T>(void *, int, int, int, double, double, double *, double *, cudaStream_t,         \
                                  const int *, const ZCtl *);
EVP_FFT_INST(float)
EVP_FFT_INST(double)
#undef EVP_FFT_INST

}  // namespace evp
