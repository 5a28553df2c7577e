// Bulge-chasing sweep of the Schur reduction (Section 3.2, "Bulge Chasing
// and Eigenvalue Reordering"): one pipelined QR iteration on an upper
// Hessenberg matrix H, bulges chased down the diagonal by overlapping 3x3
// Householder reflectors, organised as the same window tasks and
// left / right / Q update tiles as the reordering (Fig. 1b, Fig. 2).
//
// Bulges come in chains of nb (one per pair of shifts).  At chain step tau,
// bulge j of a chain (j = 0 introduced first) sits at k_j = tau - 3 j - 1:
//   k = -1       introduction: the reflector maps the three nonzeros of the
//                first column of (H - sigma1 I)(H - sigma2 I),
//                x = (h00^2 + h01 h10 - s h00 + p, h10 (h00 + h11 - s),
//                h10 h21), onto beta e_0 (s = sigma1 + sigma2,
//                p = sigma1 sigma2), on rows / columns 0..2;
//   0..n-3       chase: the reflector maps H[k+1..k+3, k] (two entries at
//                k = n-3) onto beta e_0, on rows / columns k+1..k+3; the
//                annihilated entries become exact zeros.
// Within a step the reflectors of different bulges read columns no other
// reflector of the step writes, and touch disjoint rows (left) and disjoint
// columns (right), so a step is: all reflectors, then all left products,
// then all right products -- the same result as applying them one by one
// from the lowest bulge up.
//
// A window task owns rows / columns [s, s + w) and runs the chain steps
// [t0, t1) that keep every active bulge's rows k+1..k+4 inside the window
// (the planner's guarantee), accumulating U (w x w): the rows of H to the
// right of the window and above it, and Q, get U through the update tiles.
#pragma once

#include "common.cuh"
#include "seeded.cuh"

#include <float.h>

namespace gbr {
namespace swp {

constexpr int SW = 96;                 // largest sweep window
constexpr int SWEEP_THREADS = 512;
constexpr int MAXB = SW / 3;           // bulges a window can hold

// Shared memory of sweep_body: the dense window of H and U (SW x SW each),
// for two steps per bulge its reflector (v1, v2, tau, beta, first row, length).
constexpr size_t kSweepSmem = sizeof(double) * (2 * (size_t)SW * SW + (size_t)2 * MAXB * 4) +
                              sizeof(int) * 2 * 2 * MAXB;

// Reflector I - tau v v^T, v = (1, v1, v2), mapping x (length len = 2 or 3)
// onto beta e_0; tau = 0 when x is a multiple of e_0.
__device__ __forceinline__ void refl3(int len, double x0, double x1, double x2, double* v1,
                                      double* v2, double* tau, double* beta) {
    if (len < 3) x2 = 0.0;
    const double sigma = fma(x1, x1, x2 * x2);
    if (is_zero(sigma)) {
        *v1 = 0.0;
        *v2 = 0.0;
        *tau = 0.0;
        *beta = x0;
        return;
    }
    const double nn = fma(x0, x0, sigma);
    const unsigned e = (unsigned)__double2hiint(nn) >> 20;
    if (e < 100u || e > 1900u) {  // squares near the ends of the range
        const double nrm = sqrt(nn);
        const double b = x0 >= 0.0 ? -nrm : nrm;
        const double inv = 1.0 / (x0 - b);
        *v1 = x1 * inv;
        *v2 = x2 * inv;
        *tau = (b - x0) / b;
        *beta = b;
        return;
    }
    // 23 FP64 instructions in one chain; tau = 2 / |v|^2 from the rounded v
    const double nrm = sqrt64(nn);
    const bool pos = nonneg(x0);
    const double inv = rcp64(pos ? x0 + nrm : x0 - nrm);
    const double a1 = x1 * inv, a2 = x2 * inv;
    *v1 = a1;
    *v2 = a2;
    // The rounding errors of |v|^2 (exact here: |a1|, |a2| <= 1) and of the
    // reciprocal go into one correction: U's departure from orthogonality is 10
    // to 16% below that of tau = (b - x0) / b by CUDA's root and divisions, and
    // 1% above it without the correction, which takes 11 us of a window task.
    // h is in [1/2, 1], so that it and y are normal and half_of holds; low, a
    // rounding error, may be zero or below the normal range.
    const double p = fma(a2, a2, 1.0), q = fma(a1, a1, p);
    const double low = fma(a2, a2, 1.0 - p) + fma(a1, a1, p - q);
    const double h = half_of(q), y = rcp64(h);
    *tau = fma(y, fma(-half_of(y), low, fma(-y, h, 1.0)), y);
    *beta = pos ? -nrm : nrm;
}

// One window task of a sweep.  H: the whole matrix (n x n, ldH); the
// window is [s0, s0 + w); chain steps [t0, t1); nb bulges whose shift
// parameters (s, p) are sp[2 b], sp[2 b + 1]; U (w x w, column-major, ld w)
// is written to Ug.
__device__ __forceinline__ void sweep_body(int n, double* __restrict__ H, int ldH, int s0, int w,
                                           int t0, int t1, int nb, const double* __restrict__ sp,
                                           double* __restrict__ Ug, DevCounters* __restrict__ ctr,
                                           unsigned char* smem_raw) {
    double* Hs = reinterpret_cast<double*>(smem_raw);   // w x w, ld w
    double* Us = Hs + SW * SW;                          // w x w, ld w
    double* Rb = Us + SW * SW;                          // [2][MAXB * 4]: v1, v2, tau, beta
    int* rkb = reinterpret_cast<int*>(Rb + 2 * MAXB * 4);  // [2][MAXB]: local k (or -1: intro)
    int* rlb = rkb + 2 * MAXB;                          // [2][MAXB]: length, U rows
    __shared__ int nact[2];                             // active bulges of a step
    __shared__ int pre_l2[2][MAXB + 1], pre_r2[2][MAXB + 1];
    __shared__ short urlo[SW], urhi[SW];                // nonzero rows of each column of U
    const int tid = threadIdx.x, nth = blockDim.x;
    unsigned long long wflops = 0;

    for (int i = tid; i < w * w; i += nth) {
        const int r = i % w, c = i / w;
        Hs[i] = (r <= c + 4) ? __ldcg(&H[cm(s0 + r, s0 + c, ldH)]) : 0.0;
        Us[i] = (r == c) ? 1.0 : 0.0;
    }
    for (int i = tid; i < w; i += nth) {
        urlo[i] = (short)i;
        urhi[i] = (short)i;
    }
    __syncthreads();
    // Two warp groups: warp 0 (which owns every bulge, one per lane: at most
    // 32) computes the reflectors of step tau + 1 while the other warps apply
    // those of step tau.  A bulge's next input column depends on its own
    // reflector and on ten entries of the window only, which warp 0 reads
    // before the products start and takes through the two products itself, in
    // the same operations.  A step that introduces a bulge is not looked ahead
    // to (at most nb of a chain's steps).  Lane i keeps bulge i's columns and
    // U rows across the step.
    // Measured (w = 64, eight bulges, the n = 4000 sweep): a window task takes
    // 137 us; with the reflectors computed between the products of two steps,
    // by CUDA's root and divisions, it took 163 us.
    const int lane = tid & 31, warp = tid >> 5;
    // the products run on the three sub-partitions without warp 0, whose chain
    // would share its FP64 pipe with them
    constexpr int PT = SWEEP_THREADS / 4 * 3;
    const int prod = (warp & 3) ? ((warp >> 2) * 3 + (warp & 3) - 1) * 32 + lane : -1;
    int my_c1 = 0, my_len = 0, my_lo = 0, my_cnt = 0;   // warp 0: last step's bulge
    // active bulges of a step: -1 <= k_j <= n - 3, k_j = tau - 3 j - 1 (global)
    auto active = [&](int tau, int* jlo) {
        const int over = tau - 1 - (n - 3);  // 3 j >= over
        const int lo = over > 0 ? (over + 2) / 3 : 0;
        const int hi = min(nb - 1, tau >= 0 ? tau / 3 : -1);
        *jlo = lo;
        return max(0, hi - lo + 1);
    };
    // the reflectors of step tau into the buffers of parity par; x(j, kg, len)
    // gives the input column of bulge j (chase steps)
    auto reflectors = [&](int tau, int par, auto&& input) {
        double* R = Rb + par * MAXB * 4;
        int* rk = rkb + par * MAXB;
        int* rl = rlb + par * MAXB;
        int jlo;
        const int na = active(tau, &jlo);
        double x0 = 0.0, x1 = 0.0, x2 = 0.0;
        const int j = jlo + lane, kg = tau - 3 * j - 1;
        const int len = kg < 0 || kg + 3 <= n - 1 ? 3 : 2, kl = kg < 0 ? -1 : kg - s0;
        if (lane < na) {
            if (kg < 0) {
                // introduction (the window starts at row 0)
                const double h00 = Hs[0], h10 = Hs[1], h01 = Hs[w], h11 = Hs[w + 1];
                const double h21 = Hs[w + 2];
                const double ss = sp[2 * j], pp = sp[2 * j + 1];
                x0 = fma(h00, h00, fma(h01, h10, fma(-ss, h00, pp)));
                x1 = h10 * (h00 + h11 - ss);
                x2 = h10 * h21;
            }
        }
        input(na, jlo, kg, kl, len, x0, x1, x2);
        if (my_len) {
            for (int c = 0; c < my_len; ++c) {
                urlo[my_c1 + c] = (short)my_lo;
                urhi[my_c1 + c] = (short)(my_lo + my_cnt - 1);
            }
            my_len = 0;
        }
        __syncwarp();
        int il = 0, ir = 0;
        if (lane < na) {
            double v1, v2, tu, be;
            refl3(len, x0, x1, x2, &v1, &v2, &tu, &be);
            R[lane * 4 + 0] = v1;
            R[lane * 4 + 1] = v2;
            R[lane * 4 + 2] = tu;
            R[lane * 4 + 3] = be;
            rk[lane] = kl;
            // item counts: left = columns [max(k, 0), w); right = rows
            // [0, min(k + 5, w)) of H plus the rows [lo, hi] of U holding
            // the nonzeros of the reflector's columns
            const int c1 = kl + 1;
            int lo = urlo[c1], hi = urhi[c1];
            for (int c = 1; c < len; ++c) {
                lo = min(lo, (int)urlo[c1 + c]);
                hi = max(hi, (int)urhi[c1 + c]);
            }
            il = w - (kl < 0 ? 0 : kl);
            ir = min(kl + 5, w) + (hi - lo + 1);
            // length, first U row and U row count packed into one word
            rl[lane] = len | (lo << 8) | ((hi - lo + 1) << 20);
            my_c1 = c1;
            my_len = len;
            my_lo = lo;
            my_cnt = hi - lo + 1;
            // 4 len flops per updated vector (dot + axpy): the left
            // columns but the input one, the right rows of H and of U
            const int nl = w - (kl < 0 ? 0 : kl) - (kl < 0 ? 0 : 1);
            wflops += 4ull * len * (unsigned long long)(nl + min(kl + 5, w) + my_cnt);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a2 = __shfl_up_sync(0xffffffffu, il, o);
            const int b2 = __shfl_up_sync(0xffffffffu, ir, o);
            if (lane >= o) { il += a2; ir += b2; }
        }
        if (lane < na) { pre_l2[par][lane + 1] = il; pre_r2[par][lane + 1] = ir; }
        if (lane == 0) {
            pre_l2[par][0] = 0;
            pre_r2[par][0] = 0;
            nact[par] = na;
        }
    };
    // input columns read from the window (all earlier steps applied)
    auto from_window = [&](int na, int, int kg, int kl, int len, double& x0, double& x1, double& x2) {
        if (lane < na && kg >= 0) {
            x0 = Hs[kl * w + kl + 1];
            x1 = Hs[kl * w + kl + 2];
            x2 = (len == 3) ? Hs[kl * w + kl + 3] : 0.0;
        }
    };
    if (warp == 0 && t0 < t1) reflectors(t0, 0, from_window);
    for (int tau = t0; tau < t1; ++tau) {
        const int par = (tau - t0) & 1;
        const double* R = Rb + par * MAXB * 4;
        const int* rk = rkb + par * MAXB;
        const int* rl = rlb + par * MAXB;
        const int* pre_l = pre_l2[par];
        const int* pre_r = pre_r2[par];
        const bool last = tau + 1 >= t1;
        // a bulge is introduced at step tau + 1
        const bool intro = (tau + 1) % 3 == 0 && (tau + 1) / 3 < nb;
        __syncthreads();  // reflectors of this step; the products of the step before
        const int na = nact[par];
        // warp 0: rows k + 1 .. k + 4 of columns k + 1 .. k + 3 of each bulge
        double h[3][4];
        if (warp == 0 && !last && !intro) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int r = 0; r < 4; ++r) h[c][r] = 0.0;
            if (lane < na) {
                const int k1 = rk[lane] + 1, len = rl[lane] & 0xff;
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        if (c < len && k1 + r < w) h[c][r] = Hs[(k1 + c) * w + k1 + r];
                // the bulge below turns entry (k + 4, k + 3) into its beta
                if (lane > 0 && rk[lane - 1] == k1 + 2) h[2][3] = R[(lane - 1) * 4 + 3];
            }
        }
        __syncthreads();
        if (warp == 0) {
            if (!last && !intro) {
                double y0 = 0.0, y1 = 0.0, y2 = 0.0;
                if (lane < na) {
                    const double v1 = R[lane * 4 + 0], v2 = R[lane * 4 + 1], tu = R[lane * 4 + 2];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {  // left
                        const double d = tu * fma(v2, h[c][2], fma(v1, h[c][1], h[c][0]));
                        h[c][1] = fma(-d, v1, h[c][1]);
                        h[c][2] = fma(-d, v2, h[c][2]);
                    }
                    // right: column k + 1 of rows k + 2 .. k + 4 (the product
                    // rounded as in the products, not contracted)
                    y0 = h[0][1] - __dmul_rn(tu, fma(v2, h[2][1], fma(v1, h[1][1], h[0][1])));
                    y1 = h[0][2] - __dmul_rn(tu, fma(v2, h[2][2], fma(v1, h[1][2], h[0][2])));
                    y2 = h[0][3] - __dmul_rn(tu, fma(v2, h[2][3], fma(v1, h[1][3], h[0][3])));
                }
                int jlo0;
                active(tau, &jlo0);
                reflectors(tau + 1, par ^ 1, [&](int, int jlo, int, int, int len, double& x0, double& x1,
                                                 double& x2) {
                    // bulges that have left the matrix shift the lanes
                    const int src = (lane + jlo - jlo0) & 31;
                    x0 = __shfl_sync(0xffffffffu, y0, src);
                    x1 = __shfl_sync(0xffffffffu, y1, src);
                    x2 = __shfl_sync(0xffffffffu, y2, src);
                    if (len < 3) x2 = 0.0;
                });
            }
        } else if (prod >= 0) {
            // left: rows k+1 .. k+len of the window, columns [max(k,0), w); the
            // input column gets beta and exact zeros
            const int totl = na > 0 ? pre_l[na] : 0;
            for (int it = prod; it < totl; it += PT) {
                int lo = 0, hi = na - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (pre_l[mid] <= it) lo = mid; else hi = mid - 1;
                }
                const int kl = rk[lo], len = rl[lo] & 0xff, r0 = kl + 1;
                const int c = (kl < 0 ? 0 : kl) + (it - pre_l[lo]);
                const double v1 = R[lo * 4 + 0], v2 = R[lo * 4 + 1], tu = R[lo * 4 + 2];
                double* col = Hs + c * w + r0;
                if (c == kl) {
                    col[0] = R[lo * 4 + 3];
                    col[1] = 0.0;
                    if (len == 3) col[2] = 0.0;
                    continue;
                }
                const double y0 = col[0], y1 = col[1], y2 = (len == 3) ? col[2] : 0.0;
                const double d = tu * fma(v2, y2, fma(v1, y1, y0));
                col[0] = y0 - d;
                col[1] = fma(-d, v1, y1);
                if (len == 3) col[2] = fma(-d, v2, y2);
            }
            asm volatile("bar.sync 1, %0;" ::"n"(PT) : "memory");
            // right: columns k+1 .. k+len of rows [0, min(k+5, w)) of the window
            // and of rows [lo, hi] of U; two items per thread, whose FP64
            // chains interleave
            const int totr = na > 0 ? pre_r[na] : 0;
            struct RightItem {
                double* p;
                double v1, v2, tu;
                int len;  // 0: none
            };
            auto right_item = [&](int it) {
                RightItem t;
                t.p = Hs;
                t.v1 = t.v2 = t.tu = 0.0;
                t.len = 0;
                if (it >= totr) return t;
                int lo = 0, hi = na - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (pre_r[mid] <= it) lo = mid; else hi = mid - 1;
                }
                const int kl = rk[lo], pk = rl[lo], c1 = kl + 1;
                const int nh = min(kl + 5, w), rr = it - pre_r[lo];
                t.len = pk & 0xff;
                t.v1 = R[lo * 4 + 0];
                t.v2 = R[lo * 4 + 1];
                t.tu = R[lo * 4 + 2];
                t.p = rr < nh ? Hs + c1 * w + rr : Us + c1 * w + ((pk >> 8) & 0xfff) + (rr - nh);
                return t;
            };
            for (int it = prod; it < totr; it += 2 * PT) {
                const RightItem a = right_item(it), b = right_item(it + PT);
                const double a0 = a.p[0], a1 = a.p[w], a2 = a.len == 3 ? a.p[2 * w] : 0.0;
                if (!__any_sync(__activemask(), b.len)) {
                    const double d = a.tu * fma(a.v2, a2, fma(a.v1, a1, a0));
                    a.p[0] = a0 - d;
                    a.p[w] = fma(-d, a.v1, a1);
                    if (a.len == 3) a.p[2 * w] = fma(-d, a.v2, a2);
                    continue;
                }
                const double b0 = b.len ? b.p[0] : 0.0, b1 = b.len ? b.p[w] : 0.0;
                const double b2 = b.len == 3 ? b.p[2 * w] : 0.0;
                const double d = a.tu * fma(a.v2, a2, fma(a.v1, a1, a0));
                const double e = b.tu * fma(b.v2, b2, fma(b.v1, b1, b0));
                const double x0 = a0 - d, x1 = fma(-d, a.v1, a1), x2 = fma(-d, a.v2, a2);
                const double y0 = b0 - e, y1 = fma(-e, b.v1, b1), y2 = fma(-e, b.v2, b2);
                a.p[0] = x0;
                a.p[w] = x1;
                if (a.len == 3) a.p[2 * w] = x2;
                if (b.len) {
                    b.p[0] = y0;
                    b.p[w] = y1;
                    if (b.len == 3) b.p[2 * w] = y2;
                }
            }
        }
        if (!last && intro) {
            __syncthreads();
            if (warp == 0) reflectors(tau + 1, par ^ 1, from_window);
        }
    }
    __syncthreads();
    for (int i = tid; i < w * w; i += nth) {
        const int r = i % w, c = i / w;
        if (r <= c + 4) H[cm(s0 + r, s0 + c, ldH)] = Hs[i];
        Ug[i] = Us[i];
    }
    if (wflops) atomicAdd(&ctr->win_flops, wflops);
}

}  // namespace swp
}  // namespace gbr
