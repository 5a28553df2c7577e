// Eigenvectors of a real Schur form (Section 2, Eq. 5) and their back-
// transformation (Eq. 6), with protection against floating-point overflow
// (the requirement of Section 3.1):
//
//   colmax_kernel   per column c of S: max |S[i, c]| over i < c and i < c - 1
//                   (the bounds the overflow guard multiplies with);
//   evinit_kernel   the start vector of each selected eigenvalue (a 1x1 block,
//                   or a 2x2 block = a conjugate pair, stored as real and
//                   imaginary column), zeros elsewhere;
//   evdiag_kernel   back substitution inside one block of up to 32 rows, one
//                   warp per vector;
//   evupd_kernel    the block's contribution to the rows above, one matrix
//                   product over all vectors;
//   evgemm_kernel   X = Q Y; a column block of Y is nonzero only in its leading
//                   rows, so the inner dimension stops there;
//   evnorm_kernel   max |x_i| = 1 per real vector, max(|re| + |im|) = 1 per
//                   complex one.
//
// Back substitution, 32 rows at a time from the bottom for all vectors that
// reach them: Y's rows above a block hold the right-hand side r (starting at
// zero; the start entries enter with their own block's product), the warp of
// a vector solves y[B] = (S[B,B] - lambda I)^-1 r[B] for each diagonal block B
// of the rows and updates the rows above B within them, and one product
// Y[0:lo, :] -= S[0:lo, lo:hi] Y[lo:hi, :] updates everything above.  A pivot
// below smin = max(eps |lambda|, DBL_MIN / eps) is raised to smin.  rb bounds
// max|r| over the remaining rows (|z| = |re| + |im|); before a diagonal block
// is solved and before its update, the vector is scaled by 2^-512 (exact)
// while the next value or the new bound would exceed 2^900.  The bounds only
// grow, so a warp first solves its rows without the guards and redoes them
// with the guards if the bound at the end, or a value, is over the limit.
//
// What bounds it: the FP64 pipe (products at 64 cycles a warp instruction).
// One CTA per vector with a barrier per diagonal block took 40.4 ms for the
// 21.3 GFLOP of the n = 4000 form (0.53 TFLOP/s: a chain of about 30 FP64
// instructions per block between two barriers); in blocks of 32 rows nearly
// all of the work is a matrix product, 25.0 ms in all (0.85 TFLOP/s).
#include "common.cuh"
#include "host.h"

#include <float.h>

#include <algorithm>
#include <vector>

namespace gbr {

namespace {

constexpr int EV_THREADS = 256;
constexpr double EV_BIG = 0x1p900;
constexpr double EV_SHRINK = 0x1p-512;

struct cd {
    double re, im;
};
__device__ __forceinline__ double cabs1(cd z) { return fabs(z.re) + fabs(z.im); }
__device__ __forceinline__ cd cmul(cd a, cd b) {
    return cd{fma(a.re, b.re, -a.im * b.im), fma(a.re, b.im, a.im * b.re)};
}
__device__ __forceinline__ cd csub(cd a, cd b) { return cd{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cd cdiv(cd a, cd b) {  // Smith's algorithm
    if (fabs(b.re) >= fabs(b.im)) {
        const double t = b.im / b.re, d = fma(b.im, t, b.re);
        return cd{fma(a.im, t, a.re) / d, fma(-a.re, t, a.im) / d};
    }
    const double t = b.re / b.im, d = fma(b.re, t, b.im);
    return cd{fma(a.re, t, a.im) / d, fma(a.im, t, -a.re) / d};
}
__device__ __forceinline__ cd perturb(cd d, double smin) {
    const double m = cabs1(d);
    if (m >= smin) return d;
    if (m == 0.0) return cd{smin, 0.0};
    return cd{d.re * (smin / m), d.im * (smin / m)};
}

__global__ void colmax_kernel(int n, const double* __restrict__ S, int ldS, double* __restrict__ cmA,
                              double* __restrict__ cmB) {
    const int c = blockIdx.x;
    if (c >= n) return;
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < c; i += blockDim.x) {
        const double v = fabs(__ldg(&S[cm(i, c, ldS)]));
        a = fmax(a, v);
        if (i < c - 1) b = fmax(b, v);
    }
    for (int o = 16; o; o >>= 1) {
        a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    __shared__ double sa[32], sb[32];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) { sa[w] = a; sb[w] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) { a = fmax(a, sa[i]); b = fmax(b, sb[i]); }
        cmA[c] = a;
        cmB[c] = b;
    }
}

// Block-wide max of v (EV_THREADS threads).
__device__ __forceinline__ double block_max(double v, double* red) {
    for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double m = red[0];
    for (int i = 1; i < EV_THREADS / 32; ++i) m = fmax(m, red[i]);
    return m;
}

// Inverse of the shifted diagonal block B = [b0, b0 + k), S[B,B] - lambda I,
// with a pivot (the 1x1 denominator or the 2x2 determinant) below smin
// raised to smin: inv[0..3] = row-major 2x2 (inv[0] alone for k = 1).
struct BlkInv {
    int b0, k;
    cd inv[4];
};

__device__ __forceinline__ BlkInv block_inverse(const double* __restrict__ S, int ldS, int b0,
                                                int k, double lr, double li, double smin) {
    BlkInv B;
    B.b0 = b0;
    B.k = k;
    const cd one{1.0, 0.0};
    if (k == 1) {
        const cd d = perturb(cd{__ldg(&S[cm(b0, b0, ldS)]) - lr, -li}, smin);
        B.inv[0] = cdiv(one, d);
        B.inv[1] = B.inv[2] = B.inv[3] = cd{0.0, 0.0};
        return B;
    }
    const cd m00 = cd{__ldg(&S[cm(b0, b0, ldS)]) - lr, -li};
    const cd m01 = cd{__ldg(&S[cm(b0, b0 + 1, ldS)]), 0.0};
    const cd m10 = cd{__ldg(&S[cm(b0 + 1, b0, ldS)]), 0.0};
    const cd m11 = cd{__ldg(&S[cm(b0 + 1, b0 + 1, ldS)]) - lr, -li};
    cd det = csub(cmul(m00, m11), cmul(m01, m10));
    const double mx = fmax(fmax(cabs1(m00), cabs1(m01)), fmax(cabs1(m10), cabs1(m11)));
    det = perturb(det, smin * fmax(mx, smin));
    const cd rd = cdiv(one, det);
    B.inv[0] = cmul(m11, rd);
    B.inv[1] = cmul(cd{-m01.re, -m01.im}, rd);
    B.inv[2] = cmul(cd{-m10.re, -m10.im}, rd);
    B.inv[3] = cmul(m00, rd);
    return B;
}

// x = inv r for one block; real arithmetic for real vectors.
template <bool CPLX>
__device__ __forceinline__ void apply_inv(const BlkInv& B, cd r0, cd r1, double f, cd& x0, cd& x1) {
    r0 = cd{r0.re * f, r0.im * f};
    r1 = cd{r1.re * f, r1.im * f};
    if (!CPLX) {
        x0 = cd{fma(B.inv[1].re, r1.re, B.inv[0].re * r0.re), 0.0};
        x1 = cd{fma(B.inv[3].re, r1.re, B.inv[2].re * r0.re), 0.0};
    } else {
        const cd a = cmul(B.inv[0], r0), b = cmul(B.inv[1], r1);
        const cd c = cmul(B.inv[2], r0), d = cmul(B.inv[3], r1);
        x0 = cd{a.re + b.re, a.im + b.im};
        x1 = cd{c.re + d.re, c.im + d.im};
    }
}

// The overflow guards of one block (one thread): scales by 2^-512 while the
// solution could exceed EV_BIG, then while the bound of the update of r by x
// could; returns the number of scalings, with x scaled and rb updated.
template <bool CPLX>
__device__ __forceinline__ int solve_guarded(const BlkInv& B, cd r0, cd r1, double cmx,
                                             double& rb, cd& x0, cd& x1) {
    int s = 0;
    double f = 1.0;
    apply_inv<CPLX>(B, r0, r1, 1.0, x0, x1);
    while (s < 8 && !(fmax(cabs1(x0), cabs1(x1)) <= EV_BIG)) {
        f *= EV_SHRINK;
        ++s;
        apply_inv<CPLX>(B, r0, r1, f, x0, x1);
    }
    rb *= f;
    if (B.b0 > 0) {
        double xm = fmax(cabs1(x0), cabs1(x1));
        int s2 = 0;
        while (s2 < 8 && rb + B.k * cmx * xm > EV_BIG) {
            x0 = cd{x0.re * EV_SHRINK, x0.im * EV_SHRINK};
            x1 = cd{x1.re * EV_SHRINK, x1.im * EV_SHRINK};
            rb *= EV_SHRINK;
            xm *= EV_SHRINK;
            ++s2;
        }
        rb += B.k * cmx * xm;
        s += s2;
    }
    return s;
}

constexpr int EB = 32;  // rows per block of the back substitution: a lane each

// A real pivot raised to smin where it is smaller.
__device__ __forceinline__ double perturb_real(double d, double smin) {
    return fabs(d) >= smin ? d : copysign(smin, d == 0.0 ? 1.0 : d);
}

// Start vectors: blocks[b] = (j, nb, column of Y, -); Y column-major (ldY),
// every row written.  rb[b] = max |S[0:j, j:j+nb] y[j:j+nb]|, the bound of the
// first right-hand side.
__global__ void __launch_bounds__(EV_THREADS)
evinit_kernel(int n, const double* __restrict__ S, int ldS, const int4* __restrict__ blocks,
              double* __restrict__ Y, int ldY, const double* __restrict__ cmA, double* __restrict__ rb,
              int* __restrict__ nscale) {
    __shared__ double red[EV_THREADS / 32];
    const int4 bk = blocks[blockIdx.x];
    const int j = bk.x, nb = bk.y, col = bk.z, tid = threadIdx.x;
    double* yr = Y + (size_t)col * ldY;
    if (nb == 1) {
        for (int i = tid; i < n; i += EV_THREADS) yr[i] = i == j ? 1.0 : 0.0;
        if (tid == 0) {
            rb[blockIdx.x] = cmA[j];
            nscale[col] = 0;
        }
        return;
    }
    const double b = __ldg(&S[cm(j, j + 1, ldS)]), c = __ldg(&S[cm(j + 1, j, ldS)]);
    const double y1i = sqrt(-b * c) / b;
    double m = 0.0;
    for (int i = tid; i < n; i += EV_THREADS) {
        yr[i] = i == j ? 1.0 : 0.0;
        yr[ldY + (size_t)i] = i == j + 1 ? y1i : 0.0;
        if (i < j) m = fmax(m, fabs(__ldg(&S[cm(i, j, ldS)])) + fabs(__ldg(&S[cm(i, j + 1, ldS)]) * y1i));
    }
    m = block_max(m, red);
    if (tid == 0) {
        rb[blockIdx.x] = m;
        nscale[col] = nscale[col + 1] = 0;
    }
}

// The rows [lo, hi) (at most EB, cutting no 2x2 block) of one vector, by one
// warp; lane = row.  D: the diagonal block S[lo:hi, lo:hi] in shared memory
// (column-major, ld EB + 1); cb: per row that starts a diagonal block, its
// column bound (0 for the top of S).
template <bool CPLX>
__device__ __forceinline__ void diag_vector(const double* __restrict__ S, int ldS, int lo, int hi,
                                            const double* D, const double* cb, int4 bk, double* Y,
                                            int ldY, double* rbp, int* __restrict__ nscale) {
    constexpr int LD = EB + 1;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, rows = hi - lo;
    const int j = bk.x, top = min(j, hi) - lo;  // rows [0, top) of the block are solved
    if (top <= 0) return;
    double* yr = Y + (size_t)bk.z * ldY + lo;
    double* yi = yr + ldY;
    double lr = __ldg(&S[cm(j, j, ldS)]), li = 0.0, y1i = 0.0;
    if (CPLX) {
        const double b = __ldg(&S[cm(j, j + 1, ldS)]), c = __ldg(&S[cm(j + 1, j, ldS)]);
        li = sqrt(-b * c);
        y1i = li / b;
    }
    const double smin = fmax(DBL_EPSILON * (fabs(lr) + fabs(li)), DBL_MIN / DBL_EPSILON);
    const bool act = lane < top;
    // 2x2 blocks: bit i of two = rows i, i + 1 form one
    const unsigned two = __ballot_sync(full, lane + 1 < rows && D[lane * LD + lane + 1] != 0.0);
    const bool second = lane > 0 && ((two >> (lane - 1)) & 1u);
    const int k = (two >> lane) & 1u ? 2 : 1;
    // the right-hand side of this row
    double re0 = 0.0, im0 = 0.0;
    if (act) {
        if (j < hi) {
            re0 = -D[(j - lo) * LD + lane];
            if (CPLX) im0 = -D[(j - lo + 1) * LD + lane] * y1i;
        } else {
            re0 = yr[lane];
            if (CPLX) im0 = yi[lane];
        }
    }
    // x of this row = c0 r[b] + c1 r[b + 1] for its block's rows b, b + 1
    cd c0{0.0, 0.0}, c1{0.0, 0.0};
    BlkInv B;
    if (act && !second) {
        if (CPLX) {
            B = block_inverse(S, ldS, lo + lane, k, lr, li, smin);
        } else {
            const double m00 = D[lane * LD + lane] - lr;
            B.b0 = lo + lane;
            B.k = k;
            B.inv[0] = B.inv[1] = B.inv[2] = B.inv[3] = cd{0.0, 0.0};
            if (k == 1) {
                B.inv[0].re = 1.0 / perturb_real(m00, smin);
            } else {
                const double m01 = D[(lane + 1) * LD + lane], m10 = D[lane * LD + lane + 1];
                const double m11 = D[(lane + 1) * LD + lane + 1] - lr;
                const double mx = fmax(fmax(fabs(m00), fabs(m01)), fmax(fabs(m10), fabs(m11)));
                const double rd = 1.0 / perturb_real(fma(m00, m11, -m01 * m10), smin * fmax(mx, smin));
                B.inv[0].re = m11 * rd;
                B.inv[1].re = -m01 * rd;
                B.inv[2].re = -m10 * rd;
                B.inv[3].re = m00 * rd;
            }
        }
        c0 = B.inv[0];
        c1 = B.inv[1];
    }
    {
        const double a = __shfl_up_sync(full, B.inv[2].re, 1), b = __shfl_up_sync(full, B.inv[3].re, 1);
        if (second) c0.re = a, c1.re = b;
        if (CPLX) {
            const double c = __shfl_up_sync(full, B.inv[2].im, 1), d = __shfl_up_sync(full, B.inv[3].im, 1);
            if (second) c0.im = c, c1.im = d;
        }
    }
    double re = re0, im = im0, xr = 0.0, xi = 0.0;
    for (int e = top; e > 0;) {
        const int kb = e >= 2 && ((two >> (e - 2)) & 1u) ? 2 : 1, b = e - kb;
        double x, z = 0.0;
        if (kb == 1) {
            if (CPLX) {
                const cd v = cmul(c0, cd{re, im});
                x = v.re;
                z = v.im;
            } else {
                x = c0.re * re;
            }
        } else {
            const double r0 = __shfl_sync(full, re, b), r1 = __shfl_sync(full, re, b + 1);
            if (CPLX) {
                const double i0 = __shfl_sync(full, im, b), i1 = __shfl_sync(full, im, b + 1);
                const cd v = cmul(c0, cd{r0, i0}), w = cmul(c1, cd{r1, i1});
                x = v.re + w.re;
                z = v.im + w.im;
            } else {
                x = fma(c1.re, r1, c0.re * r0);
            }
        }
        if (lane >= b && lane < e) {
            xr = x;
            xi = z;
        }
        const double x0 = __shfl_sync(full, x, b), z0 = CPLX ? __shfl_sync(full, z, b) : 0.0;
        if (kb == 2) {
            const double x1 = __shfl_sync(full, x, b + 1), s1 = D[(b + 1) * LD + lane];
            if (lane < b) re = fma(-s1, x1, re);
            if (CPLX) {
                const double z1 = __shfl_sync(full, z, b + 1);
                if (lane < b) im = fma(-s1, z1, im);
            }
        }
        const double s0 = D[b * LD + lane];
        if (lane < b) {
            re = fma(-s0, x0, re);
            if (CPLX) im = fma(-s0, z0, im);
        }
        e = b;
    }
    // would a guard have acted?  (the bound grows with every block)
    double rb = *rbp;
    const double mag = CPLX ? fabs(xr) + fabs(xi) : fabs(xr);
    const double mag1 = __shfl_down_sync(full, mag, 1);
    double inc = act && !second ? (double)k * cb[lane] * (k == 2 ? fmax(mag, mag1) : mag) : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) inc += __shfl_xor_sync(full, inc, o);
    const bool fine = (!act || mag <= EV_BIG) && rb + inc <= EV_BIG;  // (NaN is not)
    if (__all_sync(full, fine)) {
        if (act) {
            yr[lane] = xr;
            if (CPLX) yi[lane] = xi;
        }
        if (lane == 0) *rbp = rb + inc;
        return;
    }
    // guarded: block by block, lane 0 decides the scalings
    re = re0;
    im = im0;
    xr = xi = 0.0;
    int s = 0;
    for (int e = top; e > 0;) {
        const int kb = e >= 2 && ((two >> (e - 2)) & 1u) ? 2 : 1, b = e - kb, b2 = b + kb - 1;
        const cd r0{__shfl_sync(full, re, b), __shfl_sync(full, im, b)};
        cd r1{__shfl_sync(full, re, b2), __shfl_sync(full, im, b2)};
        if (kb == 1) r1 = cd{0.0, 0.0};
        BlkInv Bb;
        Bb.b0 = lo + b;
        Bb.k = kb;
#pragma unroll
        for (int t = 0; t < 4; ++t)
            Bb.inv[t] = cd{__shfl_sync(full, B.inv[t].re, b), __shfl_sync(full, B.inv[t].im, b)};
        cd x0{0.0, 0.0}, x1{0.0, 0.0};
        int sb = 0;
        if (lane == 0) sb = solve_guarded<CPLX>(Bb, r0, r1, cb[b], rb, x0, x1);
        sb = __shfl_sync(full, sb, 0);
        x0 = cd{__shfl_sync(full, x0.re, 0), __shfl_sync(full, x0.im, 0)};
        x1 = cd{__shfl_sync(full, x1.re, 0), __shfl_sync(full, x1.im, 0)};
        for (int t = 0; t < sb; ++t) {
            re *= EV_SHRINK;
            im *= EV_SHRINK;
            xr *= EV_SHRINK;
            xi *= EV_SHRINK;
        }
        s += sb;
        if (lane == b) xr = x0.re, xi = x0.im;
        if (kb == 2 && lane == b + 1) xr = x1.re, xi = x1.im;
        if (lane < b) {
            const double s0 = D[b * LD + lane], s1 = kb == 2 ? D[(b + 1) * LD + lane] : 0.0;
            re = fma(-s1, x1.re, fma(-s0, x0.re, re));
            if (CPLX) im = fma(-s1, x1.im, fma(-s0, x0.im, im));
        }
        e = b;
    }
    if (act) {
        yr[lane] = xr;
        if (CPLX) yi[lane] = xi;
    }
    if (lane == 0) *rbp = rb;
    if (s == 0) return;
    // the vector's other rows move to the new scale: the right-hand side
    // above, the solution below (its support ends with its own block)
    double f = 1.0;
    for (int t = 0; t < s; ++t) f *= EV_SHRINK;
    const int end = j + bk.y - lo;
    for (int i = lane - lo; i < end; i += 32) {
        if (i >= 0 && i < top) continue;
        yr[i] *= f;
        if (CPLX) yi[i] *= f;
    }
    if (lane == 0) {
        nscale[bk.z] += s;
        if (CPLX) nscale[bk.z + 1] += s;
    }
}

constexpr int DIAG_WARPS = 4;

// The vectors blocks[r0, r0 + nr) (real) and blocks[c0, c0 + nc) (complex),
// those whose block lies at or below row lo, one per warp.
__global__ void __launch_bounds__(32 * DIAG_WARPS)
evdiag_kernel(const double* __restrict__ S, int ldS, int lo, int hi, const int4* __restrict__ blocks,
              int r0, int nr, int c0, int nc, double* __restrict__ Y, int ldY,
              const double* __restrict__ cmA, const double* __restrict__ cmB, double* __restrict__ rb,
              int* __restrict__ nscale) {
    __shared__ double D[EB * (EB + 1)], cb[EB];
    const int rows = hi - lo, tid = threadIdx.x;
    for (int i = tid; i < EB * EB; i += 32 * DIAG_WARPS) {
        const int r = i & (EB - 1), c = i / EB;
        D[c * (EB + 1) + r] = r < rows && c < rows && r <= c + 1 ? __ldg(&S[cm(lo + r, lo + c, ldS)]) : 0.0;
    }
    __syncthreads();
    if (tid < EB) {
        const bool two = tid + 1 < rows && D[tid * (EB + 1) + tid + 1] != 0.0;
        cb[tid] = tid >= rows || lo + tid == 0 ? 0.0
                  : two ? fmax(cmA[lo + tid], cmB[lo + tid + 1]) : cmA[lo + tid];
    }
    __syncthreads();
    const int v = blockIdx.x * DIAG_WARPS + (tid >> 5);
    if (v < nr)
        diag_vector<false>(S, ldS, lo, hi, D, cb, blocks[r0 + v], Y, ldY, rb + r0 + v, nscale);
    else if (v < nr + nc)
        diag_vector<true>(S, ldS, lo, hi, D, cb, blocks[c0 + v - nr], Y, ldY, rb + c0 + v - nr, nscale);
}

// C (rows x cols) -= A (rows x K) B (K x cols), column-major, K <= EB; C and B
// are rows of the same columns of Y.  Tiles of 32 x 64, 4 x 4 per thread: the
// FP64 pipe needs 64 cycles for a warp's FMA, so operand traffic is no
// concern and small tiles keep the last wave short (a tile alone on an SM
// takes 16 us).
constexpr int UM = 32, UN = 64, LDU = UN + 2;

__global__ void __launch_bounds__(128)
evupd_kernel(int rows, int cols, int K, const double* __restrict__ A, int ldA, const double* B, int ldB,
             double* C, int ldC) {
    __shared__ __align__(16) double As[EB * UM], Bs[EB * LDU];
    const int r0 = blockIdx.x * UM, c0 = blockIdx.y * UN;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rg = (lane & 7) * 4, cg = (warp * 4 + (lane >> 3)) * 2;  // columns cg, cg + 1, cg + 32, cg + 33
    double acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int c = c0 + cg + (u & 1) + 32 * (u >> 1);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            acc[r][u] = r0 + rg + r < rows && c < cols ? C[cm(r0 + rg + r, c, ldC)] : 0.0;
    }
    for (int i = tid; i < EB * UM; i += 128) {
        const int r = i & (UM - 1), k = i / UM;
        As[k * UM + r] = r0 + r < rows && k < K ? __ldg(&A[cm(r0 + r, k, ldA)]) : 0.0;
    }
    for (int i = tid; i < EB * UN; i += 128) {
        const int k = i & (EB - 1), c = i / EB;
        Bs[k * LDU + c] = k < K && c0 + c < cols ? B[cm(k, c0 + c, ldB)] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < EB; ++k) {
        double a[4], b[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const double2 x = *reinterpret_cast<const double2*>(&As[k * UM + rg + 2 * h]);
            const double2 y = *reinterpret_cast<const double2*>(&Bs[k * LDU + cg + 32 * h]);
            a[2 * h] = x.x;
            a[2 * h + 1] = x.y;
            b[2 * h] = y.x;
            b[2 * h + 1] = y.y;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[r][u] = fma(-a[r], b[u], acc[r][u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int c = c0 + cg + (u & 1) + 32 * (u >> 1);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r0 + rg + r < rows && c < cols) C[cm(r0 + rg + r, c, ldC)] = acc[r][u];
    }
}

// C (rows x cols) = A (rows x K) B (K x cols), column-major, K of column
// block cb limited to kmax[cb] (the vectors' support).  FP64 FMAs in register
// tiles (4 x 8 per thread): both this and the tensor-core form (DMMA) are
// bound by the same FP64 pipe, and the FMAs reach the higher rate (the n = 4000
// form's 66 GFLOP: 56.2 ms, 1.18 TFLOP/s; with DMMA 67.9 ms, 0.97).  The column blocks with the longest
// sums are started first, so that the last wave is short.
constexpr int GM = 64, GN = 128, GK = 32;
constexpr int LDA_S = GM + 2, LDB_S = GN + 2;
constexpr size_t kGemmSmem = sizeof(double) * (size_t)GK * (LDA_S + LDB_S);

__global__ void __launch_bounds__(256)
evgemm_kernel(int rows, int cols, const double* __restrict__ A, int ldA,
              const double* __restrict__ B, int ldB, double* __restrict__ C, int ldC,
              const int* __restrict__ kmax) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* As = reinterpret_cast<double*>(smem_raw);  // GK x LDA_S (rows contiguous)
    double* Bs = As + GK * LDA_S;                       // GK x LDB_S (columns contiguous)
    const int cb = gridDim.y - 1 - blockIdx.y;
    const int r0 = blockIdx.x * GM, c0 = cb * GN;
    const int K = kmax[cb];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rg = ((warp & 1) * 8 + (lane & 7)) * 4;   // rows rg .. rg + 3
    const int cg = ((warp >> 1) * 4 + (lane >> 3)) * 2;  // columns cg + {0, 1} + 32 h, h = 0 .. 3
    double acc[4][8];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[r][u] = 0.0;
    for (int k0 = 0; k0 < K; k0 += GK) {
        __syncthreads();
        for (int i = tid; i < GM * GK; i += 256) {
            const int r = i % GM, k = i / GM;
            As[k * LDA_S + r] = (r0 + r < rows && k0 + k < K) ? __ldg(&A[cm(r0 + r, k0 + k, ldA)]) : 0.0;
        }
        for (int i = tid; i < GK * GN; i += 256) {
            const int k = i % GK, c = i / GK;
            Bs[k * LDB_S + c] = (c0 + c < cols && k0 + k < K) ? __ldg(&B[cm(k0 + k, c0 + c, ldB)]) : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < GK; ++k) {
            double a[4], b[8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const double2 x = *reinterpret_cast<const double2*>(&As[k * LDA_S + rg + 2 * h]);
                a[2 * h] = x.x;
                a[2 * h + 1] = x.y;
            }
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const double2 y = *reinterpret_cast<const double2*>(&Bs[k * LDB_S + cg + 32 * h]);
                b[2 * h] = y.x;
                b[2 * h + 1] = y.y;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int u = 0; u < 8; ++u) acc[r][u] = fma(a[r], b[u], acc[r][u]);
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int c = c0 + cg + (u & 1) + 32 * (u >> 1);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r0 + rg + r < rows && c < cols) C[cm(r0 + rg + r, c, ldC)] = acc[r][u];
    }
}

// Normalizes the vector(s) of block b in place: X columns col (and col + 1).
__global__ void __launch_bounds__(EV_THREADS)
evnorm_kernel(int n, const int4* __restrict__ blocks, double* __restrict__ X, int ldX) {
    __shared__ double red[EV_THREADS / 32];
    const int4 bk = blocks[blockIdx.x];
    const int nb = bk.y, col = bk.z;
    double* xr = X + (size_t)col * ldX;
    double* xi = nb == 2 ? X + (size_t)(col + 1) * ldX : nullptr;
    double m = 0.0;
    for (int i = threadIdx.x; i < n; i += EV_THREADS)
        m = fmax(m, fabs(xr[i]) + (xi ? fabs(xi[i]) : 0.0));
    m = block_max(m, red);
    if (m == 0.0) return;
    for (int i = threadIdx.x; i < n; i += EV_THREADS) {
        xr[i] /= m;
        if (xi) xi[i] /= m;
    }
}

template <typename K>
cudaError_t smem_attr(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

cudaError_t launch_colmax(int n, const double* S, int ldS, double* cmA, double* cmB,
                          cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    colmax_kernel<<<n, 128, 0, st>>>(n, S, ldS, cmA, cmB);
    return cudaGetLastError();
}

cudaError_t launch_eigvec(int n, const double* S, int ldS, const uint8_t* sub,
                          const std::vector<int4>& blocks, int nreal, const int4* d_blocks,
                          double* Y, int ldY, const double* cmA, const double* cmB, double* rb,
                          int* nscale, cudaStream_t st) {
    const int nblk = (int)blocks.size();
    if (n == 0 || nblk == 0) return cudaSuccess;
    evinit_kernel<<<nblk, EV_THREADS, 0, st>>>(n, S, ldS, d_blocks, Y, ldY, cmA, rb, nscale);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the columns of Y end with the last block of either kind
    int m = 0;
    for (int i : {nreal - 1, nblk - 1})
        if (i >= 0) m = std::max(m, blocks[i].z + blocks[i].y);
    for (int hi = n; hi > 0;) {
        int lo = std::max(0, hi - EB);
        if (lo > 0 && sub[lo - 1]) ++lo;  // a 2x2 block starts at lo - 1
        // vectors whose block lies at or below lo, their first column
        const auto at = [&](int f, int l) {
            return (int)(std::lower_bound(blocks.begin() + f, blocks.begin() + l, lo,
                                          [](const int4& b, int x) { return b.x < x; }) -
                         blocks.begin());
        };
        const int r0 = at(0, nreal), c0 = at(nreal, nblk);
        const int nr = nreal - r0, nc = nblk - c0;
        int col = m;
        if (nr > 0) col = std::min(col, blocks[r0].z);
        if (nc > 0) col = std::min(col, blocks[c0].z);
        if (nr + nc > 0) {
            evdiag_kernel<<<(nr + nc + DIAG_WARPS - 1) / DIAG_WARPS, 32 * DIAG_WARPS, 0, st>>>(
                S, ldS, lo, hi, d_blocks, r0, nr, c0, nc, Y, ldY, cmA, cmB, rb, nscale);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if (lo > 0) {
                const dim3 grid((lo + UM - 1) / UM, (m - col + UN - 1) / UN);
                double* Yc = Y + (size_t)col * ldY;
                evupd_kernel<<<grid, 128, 0, st>>>(lo, m - col, hi - lo, S + (size_t)lo * ldS, ldS, Yc + lo,
                                                   ldY, Yc, ldY);
                if ((e = cudaGetLastError()) != cudaSuccess) return e;
            }
        }
        hi = lo;
    }
    return cudaSuccess;
}

cudaError_t launch_evgemm(int rows, int cols, const double* A, int ldA, const double* B, int ldB,
                          double* C, int ldC, const int* d_kmax, cudaStream_t st) {
    if (rows == 0 || cols == 0) return cudaSuccess;
    cudaError_t e = smem_attr(evgemm_kernel, kGemmSmem);
    if (e != cudaSuccess) return e;
    dim3 grid((rows + GM - 1) / GM, (cols + GN - 1) / GN);
    evgemm_kernel<<<grid, 256, kGemmSmem, st>>>(rows, cols, A, ldA, B, ldB, C, ldC, d_kmax);
    return cudaGetLastError();
}

int evgemm_col_block() { return GN; }

cudaError_t launch_evnorm(int n, const int4* d_blocks, int nblk, double* X, int ldX, cudaStream_t st) {
    if (n == 0 || nblk == 0) return cudaSuccess;
    evnorm_kernel<<<nblk, EV_THREADS, 0, st>>>(n, d_blocks, X, ldX);
    return cudaGetLastError();
}

}  // namespace gbr
