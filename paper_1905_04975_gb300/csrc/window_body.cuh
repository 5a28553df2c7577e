// Window task: reorders the selected blocks inside one diagonal window of
// S and accumulates the window's orthogonal transformation U (Section 3.2,
// Fig. 1b; the "window task" that outputs updated tiles and an accumulator).
//
// One CTA owns one window [s, e) of width w.  For w <= WMAX the window of S
// lives in shared memory in packed upper-Hessenberg column order (column c
// keeps rows 0..c+1), U (w x w, starting at the identity) in dense column
// order.  Wider windows (up to WMAX_WIDE) do not fit there: the same packed
// window sits in a global scratch area of the CTA and U is formed in place
// in global memory, both served by the SM's L1 and L2.
//
// The swaps are organised in parallel steps instead of one at a time: in a
// step, every selected block whose upper neighbour is an unselected block
// swaps with it.  Such swaps touch disjoint index ranges, so their left
// transformations (rows) and right transformations (columns) commute and are
// applied concurrently; the result is the same stable partition as moving
// blocks one by one, reached in about w steps instead of m (w - m) swaps on
// the critical path.  A rejected swap leaves the window unchanged and marks
// the block stuck: it never moves again and later selected blocks stop below
// it.
//
// Included by the per-window launch (window.cu) and by the persistent
// scheduler (sched.cu).  Global loads go through L2 (ld.global.cg): in a
// persistent launch other CTAs write S between this CTA's tasks.
#pragma once

#include "common.cuh"
#include "ozaki.cuh"
#include "seeded.cuh"

#include <float.h>

#include <type_traits>

namespace gbr {
namespace win {

constexpr int WIN_THREADS = 512;
// Warps of a window task that compute the swap transforms while the others
// apply the previous step's products (a multiple of 4: the same number on
// each SM sub-partition).
constexpr int WIN_TWARPS = 4;
constexpr int MAXSW = WMAX / 2;  // at most one swap per two positions

__device__ __forceinline__ int poff(int c) { return (c * (c + 3)) >> 1; }



// Edge rows of a window that belong to a 2x2 block cut by the window
// boundary (possible only after a rejected swap made the plan stale) are
// walls: nothing swaps with them and they do not move.
constexpr uint8_t SEL_WALL = 3;

__device__ __forceinline__ double sel4(int i, double a0, double a1, double a2, double a3) {
    return i == 0 ? a0 : (i == 1 ? a1 : (i == 2 ? a2 : a3));
}

// T11 X - X T22 = T12 for 2x2 blocks of D (ld 4), elimination on the 4x4
// Kronecker system with complete pivoting; registers only.
__device__ __forceinline__ bool sylv22_regs(const double* D, double* X) {
    double K[4][4], b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = r & 1, kk = r >> 1;
        b[r] = D[(2 + kk) * 4 + i];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int l = c & 1, mm = c >> 1;
            double v = (kk == mm) ? D[l * 4 + i] : 0.0;
            if (i == l) v -= D[(2 + kk) * 4 + 2 + mm];
            K[r][c] = v;
        }
    }
    unsigned long long kmx = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            unsigned long long a = abs_bits(K[r][c]);
            kmx = a > kmx ? a : kmx;
        }
    const double smin = fmax(DBL_EPSILON * bits_double(kmx), DBL_MIN);
    int perm = 0x3210;  // perm nibble c = original unknown now in column c
    double rp[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        unsigned long long best = 0;
        int pr = s, pc = s;
#pragma unroll
        for (int r = s; r < 4; ++r)
#pragma unroll
            for (int c = s; c < 4; ++c) {
                unsigned long long a = abs_bits(K[r][c]);
                if (a > best) { best = a; pr = r; pc = c; }
            }
#pragma unroll
        for (int r = s + 1; r < 4; ++r)
            if (pr == r) {
#pragma unroll
                for (int c = 0; c < 4; ++c) { double t = K[s][c]; K[s][c] = K[r][c]; K[r][c] = t; }
                double t = b[s]; b[s] = b[r]; b[r] = t;
            }
#pragma unroll
        for (int c = s + 1; c < 4; ++c)
            if (pc == c) {
#pragma unroll
                for (int r = 0; r < 4; ++r) { double t = K[r][s]; K[r][s] = K[r][c]; K[r][c] = t; }
                int ns = (perm >> (4 * s)) & 15, nc = (perm >> (4 * c)) & 15;
                perm &= ~((15 << (4 * s)) | (15 << (4 * c)));
                perm |= (nc << (4 * s)) | (ns << (4 * c));
            }
        double piv = K[s][s];
        if (abs_bits(piv) < abs_bits(smin)) piv = smin;
        rp[s] = 1.0 / piv;
#pragma unroll
        for (int r = s + 1; r < 4; ++r) {
            const double f = K[r][s] * rp[s];
#pragma unroll
            for (int c = s + 1; c < 4; ++c) K[r][c] = fma(-f, K[s][c], K[r][c]);
            b[r] = fma(-f, b[s], b[r]);
        }
    }
    double y[4];
#pragma unroll
    for (int s = 3; s >= 0; --s) {
        double acc = b[s];
#pragma unroll
        for (int c = s + 1; c < 4; ++c) acc = fma(-K[s][c], y[c], acc);
        y[s] = acc * rp[s];
    }
    unsigned long long ym = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) ym = abs_bits(y[c]) > ym ? abs_bits(y[c]) : ym;
    // nan, or above 2^500: the full transform scales such a solution
    if (!(ym < 0x5f30000000000000ULL)) return false;
    // un-permute: X[perm(c)] = y[c]   (X column-major 2x2, index i + 2k)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        double v = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (((perm >> (4 * c)) & 15) == t) v = y[c];
        X[t] = v;
    }
    return true;
}

// ---------------------------------------------------------------------------
// Building blocks of the swap transforms.  What bounds a transform: on this
// part a warp's FP64 instruction holds its sub-partition's pipe for 64 cycles
// and its result is 64 cycles away, whatever the number of active lanes, while
// FP32 and integer instructions cost a cycle or two.  So the transforms keep
// the number of FP64 instructions down: first approximations come from the
// special function unit or from FP32, and FP64 only corrects them.  Measured
// against transforms in FP64 throughout, with 3x3 and 4x4 products: a window
// task of w = 128, m = 64 took 1.90 ms and takes 1.48 ms (median in the
// n = 4000 schedule), one of w = 32, m = 16 took 268 us and took 193 us (1.31
// ms and 145 us since the control of a step runs beside the critical products
// and a lane of a product warp works on two items at once); the rounding
// errors of whole reorderings (orthogonality, residual, swaps sent to the
// double-double retry) are a little smaller than they were.
// ---------------------------------------------------------------------------
// Reflector I - f w w^T with w = (w0, a1, 1) that maps a = (a0, a1, 1) onto
// -sign(a0) |a| e_0: w0 = a0 + sign(a0) |a|, f = 2 / |w|^2 (taken from the
// rounded w, so that only f's own rounding touches the orthogonality).  The
// last component of w stays 1, so that applying it takes six FP64
// instructions (a 3x3 product takes nine).  The last component makes |w|^2 at
// least 2, and a0, a1 are at most 2^500 (see sylv22_regs; a k = 3 solution
// above 2^510 gives NaN or the identity, within the rounding errors of a
// coupling that large): half_of holds.
__device__ __forceinline__ void refl3(double a0, double a1, double* w0, double* f) {
    const double n1 = fma(a1, a1, 1.0);
    const double d = fabs(a0) + sqrt64(fma(a0, a0, n1));
    *w0 = nonneg(a0) ? d : -d;
    *f = rcp64(half_of(fma(d, d, n1)));
}
__device__ __forceinline__ void apply_refl3(double w0, double w1, double f, double* x0, double* x1,
                                            double* x2) {
    const double s = fma(w0, *x0, fma(w1, *x1, *x2)) * f;
    *x0 = fma(-s, w0, *x0);
    *x1 = fma(-s, w1, *x1);
    *x2 -= s;
}

// What follows a 2|2 swap's Sylvester solution X: reflectors, products and
// tests, with lim for the block that must vanish (dc0..dc3: this lane's column
// of D, tb: the bit pattern of 10 eps max|D|).
__device__ __forceinline__ bool swap22_finish(const double (&X)[4], double dc0, double dc1, double dc2,
                                              double dc3, unsigned long long tb,
                                              unsigned long long lim, int l, unsigned hmask,
                                              int hbase, bool strong, double* z, double* dnrc) {
    const int r = l & 3, c = l >> 2;
    // reflector 1 on column 0 of [-X; I], (-x00, -x10, 1, 0); reflector 2 on
    // rows 1..3 of reflector 1 times column 1, (-x01, -x11, 0, 1)
    const double w1 = -X[1];
    double w0, f1, u0, f2;
    refl3(-X[0], w1, &w0, &f1);
    const double s1 = fma(w0, -X[2], w1 * -X[3]) * f1;
    const double q1 = fma(-s1, w1, -X[3]), u1 = -s1;  // (q1, u1, 1)
    refl3(q1, u1, &u0, &f2);
    // Qs = (I - f1 w w^T)(I - f2 u u^T), w = (w0, w1, 1, 0), u = (0, u0, u1, 1)
    const double wu = fma(w1, u0, u1);
    const double wr = sel4(r, w0, w1, 1.0, 0.0), wc = sel4(c, w0, w1, 1.0, 0.0);
    const double ur = sel4(r, 0.0, u0, u1, 1.0), uc = sel4(c, 0.0, u0, u1, 1.0);
    const double ar = f1 * wr;
    double qs = fma(-ar, wc, (r == c) ? 1.0 : 0.0);
    qs = fma(-(f2 * uc), fma(-ar, wu, ur), qs);
    // T = Qs^T D: T[r][c] = sum_a Qs[a][r] D[a][c]
    double T = __shfl_sync(hmask, qs, hbase + 0 + 4 * r) * dc0;
    T = fma(__shfl_sync(hmask, qs, hbase + 1 + 4 * r), dc1, T);
    T = fma(__shfl_sync(hmask, qs, hbase + 2 + 4 * r), dc2, T);
    T = fma(__shfl_sync(hmask, qs, hbase + 3 + 4 * r), dc3, T);
    // Dt = T Qs: Dt[r][c] = sum_b T[r][b] Qs[b][c]
    double Dt = 0.0;
#pragma unroll
    for (int bb = 0; bb < 4; ++bb)
        Dt = fma(__shfl_sync(hmask, T, hbase + r + 4 * bb),
                 __shfl_sync(hmask, qs, hbase + bb + 4 * c), Dt);
    // weak test on the lower-left 2x2 block
    const bool low = (r >= 2 && c < 2);
    bool pass = !__any_sync(hmask, low && abs_bits(Dt) > lim);
    const double Dt0 = low ? 0.0 : Dt;
    if (strong && pass) {
        // P = Qs Dt0: P[r][b] = sum_a Qs[r][a] Dt0[a][b]
        double P = 0.0;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            P = fma(__shfl_sync(hmask, qs, hbase + r + 4 * a),
                    __shfl_sync(hmask, Dt0, hbase + a + 4 * c), P);
        // E = P Qs^T - D: E[r][c] = sum_b P[r][b] Qs[c][b] - D[r][c]
        double E = 0.0;
#pragma unroll
        for (int bb = 0; bb < 4; ++bb)
            E = fma(__shfl_sync(hmask, P, hbase + r + 4 * bb),
                    __shfl_sync(hmask, qs, hbase + c + 4 * bb), E);
        E -= sel4(r, dc0, dc1, dc2, dc3);
        pass = !__any_sync(hmask, abs_bits(E) > tb);
    }
    if (pass) {
        z[0] = w0;
        z[1] = w1;
        z[2] = f1;
        z[3] = u0;
        z[4] = u1;
        z[5] = f2;
        *dnrc = Dt0;
        return true;
    }
    return false;
}

// The swap by elimination, for the seeded solutions that do not serve (out of
// line: it is rare, and the step loop must fit the instruction caches).
static __device__ __noinline__ bool swap22_elim(const double* __restrict__ Sp, int ja, int l,
                                                unsigned hmask, int hbase, bool strong,
                                                unsigned long long tb, double* z, double* dnrc) {
    double D[16], X[4];
#pragma unroll
    for (int cc = 0; cc < 4; ++cc)
#pragma unroll
        for (int rr = 0; rr < 4; ++rr)
            D[cc * 4 + rr] = (rr <= cc + 1) ? Sp[poff(ja + cc) + ja + rr] : 0.0;
    if (!sylv22_regs(D, X)) return false;
    const int c = l >> 2;
    const double* cc = Sp + poff(ja + c) + ja;
    return swap22_finish(X, cc[0], cc[1], c >= 1 ? cc[2] : 0.0, c >= 2 ? cc[3] : 0.0, tb, tb, l, hmask,
                         hbase, strong, z, dnrc);
}

// 2|2 swap by 16 lanes: lane l of the half-warp owns entry (r, c) =
// (l & 3, l >> 2) of the 4x4 matrices.  No re-standardization (done at the end
// of the window).  Returns false if the full transform must run; otherwise
// *dnrc is this lane's entry of the new block and z holds the two reflectors,
// (w0, w1, f) on rows 0..2 and (u0, u1, f') on rows 1..3.
//
// The Sylvester equation A X - X B = C (T11 = A, T22 = B, T12 = C, both
// diagonal blocks shifted by B's first diagonal entry, which cancels) is
// solved in closed form: M X = A C - C adj(B) with M = A^2 - tr(B) A + det(B) I
// (Cayley-Hamilton on B), evaluated in FP32, then refined with FP64 residuals
// until, after at least two corrections, one is at most 2^-40 of the solution.
// A correction can be small by luck while the next would not be, the more
// easily the closer the blocks' eigenvalues; so a seeded solution has to leave
// at most 2.5 eps max|D| in the block that must vanish, a quarter of what the
// weak test allows.  One that does not, or has not converged in six
// corrections, gives way to the elimination with complete pivoting under the
// weak test itself.
// Error in the block that must vanish, in eps max|D|, mean and largest of
// 200 000 swaps of blocks with the same imaginary part and couplings of the
// size of their separation s (host restatement, exact evaluation):
//     s       elimination   2^-36, no limit   2^-40 and 2.5 eps
//     1       0.49   2.8       0.42   2.8        0.42  2.4
//     1e-2    0.39   2.5       0.39   2.6        0.39  2.4
//     1e-4    0.39   2.5       0.40  12          0.39  2.5
//     1e-5    0.39   2.5       0.40  94          0.39  2.5
//     1e-6    0.39   2.9       0.66  1800        0.39  2.9
// 2.00 corrections on average for s >= 0.1, 2.4 at 1e-2, 3.0 at 1e-3; below
// 1e-5 most solutions are the elimination's.
// FP64 instructions: 3 + 5 per correction, 30 for the reflectors, 22 for the
// products and tests; the elimination in FP64, two square roots and five
// divisions took about 200.
__device__ __forceinline__ bool swap22_halfwarp(const double* __restrict__ Sp, int ja, int l,
                                                unsigned hmask, int hbase, bool strong,
                                                double* z, double* dnrc) {
    const int r = l & 3, c = l >> 2;
    const double* c0 = Sp + poff(ja) + ja;
    const double* c1 = Sp + poff(ja + 1) + ja;
    const double* c2 = Sp + poff(ja + 2) + ja;
    const double* c3 = Sp + poff(ja + 3) + ja;
    const double b00 = c2[2];
    const double a00 = c0[0] - b00, a10 = c0[1], a01 = c1[0], a11 = c1[1] - b00;
    const double b10 = c2[3], b01 = c3[2], b11 = c3[3] - b00;
    // this lane's column of D and the largest entry of D
    const double* cc = Sp + poff(ja + c) + ja;
    const double dc0 = cc[0], dc1 = cc[1], dc2 = c >= 1 ? cc[2] : 0.0, dc3 = c >= 2 ? cc[3] : 0.0;
    unsigned long long mx = abs_bits(dc0), t1 = abs_bits(dc1), t2 = abs_bits(dc2), t3 = abs_bits(dc3);
    mx = t1 > mx ? t1 : mx;
    t2 = t3 > t2 ? t3 : t2;
    mx = t2 > mx ? t2 : mx;
    t1 = __shfl_xor_sync(hmask, mx, 4);
    mx = t1 > mx ? t1 : mx;
    t1 = __shfl_xor_sync(hmask, mx, 8);
    mx = t1 > mx ? t1 : mx;
    const unsigned long long tb = thresh_bits(mx);
    // a quarter of it for a seeded solution (exponent arithmetic)
    const unsigned long long tb4 = tb > (3ULL << 52) ? tb - (2ULL << 52) : tb;
    // FP32 copies, scaled by the power of two of the largest entry of A and B
    int em = 0;
    {
        auto up = [&](double v) {
            const int e = (__double2hiint(v) >> 20) & 0x7ff;
            em = e > em ? e : em;
        };
        up(a00); up(a10); up(a01); up(a11); up(b10); up(b01); up(b11);
    }
    const int eoff = em - 127;
    const float fa00 = to_f32(a00, eoff), fa01 = to_f32(a01, eoff), fa10 = to_f32(a10, eoff);
    const float fa11 = to_f32(a11, eoff), fb01 = to_f32(b01, eoff), fb10 = to_f32(b10, eoff);
    const float tr = to_f32(b11, eoff);
    const float com = fmaf(fa01, fa10, -fb01 * fb10), rest = fa00 + fa11 - tr;
    const float m00 = fmaf(fa00, fa00 - tr, com), m11 = fmaf(fa11, fa11 - tr, com);
    const float m01 = fa01 * rest, m10 = fa10 * rest;
    const float rdet = __fdividef(1.0f, fmaf(m00, m11, -m01 * m10));
    float x[4];  // X column by column
    auto solve = [&](float r00, float r10, float r01, float r11) {
        const float y00 = fmaf(fa00 - tr, r00, fmaf(fa01, r10, fb10 * r01));
        const float y10 = fmaf(fa11 - tr, r10, fmaf(fa10, r00, fb10 * r11));
        const float y01 = fmaf(fa00, r01, fmaf(fa01, r11, fb01 * r00));
        const float y11 = fmaf(fa11, r11, fmaf(fa10, r01, fb01 * r10));
        x[0] = fmaf(m11, y00, -m01 * y10) * rdet;
        x[1] = fmaf(m00, y10, -m10 * y00) * rdet;
        x[2] = fmaf(m11, y01, -m01 * y11) * rdet;
        x[3] = fmaf(m00, y11, -m10 * y01) * rdet;
        unsigned m = 0;  // largest |x|, NaN above all
#pragma unroll
        for (int t = 0; t < 4; ++t) m = max(m, __float_as_uint(x[t]) & 0x7fffffffu);
        return __uint_as_float(m);
    };
    // lane's entry (i, k) of the 2x2 matrices X and of the residual
    const int i = l & 1, k = (l >> 1) & 1;
    const double ai0 = i ? a10 : a00, ai1 = i ? a11 : a01;
    const double bk0 = k ? b01 : 0.0, bk1 = k ? b11 : b10;
    const double cik = Sp[poff(ja + 2 + k) + ja + i];
    double X[4], own = cik;
    float xmax = 0.0f;
    bool good = false;
    auto spread = [&](float v) {  // entries (0,0), (1,0), (0,1), (1,1) of the lanes
        return solve(__shfl_sync(hmask, v, hbase), __shfl_sync(hmask, v, hbase + 1),
                     __shfl_sync(hmask, v, hbase + 2), __shfl_sync(hmask, v, hbase + 3));
    };
    xmax = spread(to_f32(cik, eoff));
    own = from_f32(k ? (i ? x[3] : x[2]) : (i ? x[1] : x[0]));
#pragma unroll 1
    for (int it = 0; it < 6; ++it) {
#pragma unroll
        for (int t = 0; t < 4; ++t) X[t] = __shfl_sync(hmask, own, hbase + t);
        double res = fma(-ai0, k ? X[2] : X[0], cik);
        res = fma(-ai1, k ? X[3] : X[1], res);
        res = fma(i ? X[1] : X[0], bk0, res);
        res = fma(i ? X[3] : X[2], bk1, res);
        const float dmax = spread(to_f32(res, eoff));
        own += from_f32(k ? (i ? x[3] : x[2]) : (i ? x[1] : x[0]));
        if (!(dmax <= 0.25f * xmax)) break;  // also NaN: no convergence
        if (it > 0 && dmax <= 9.094947e-13f * xmax) { good = xmax < 1e30f; break; }  // 2^-40
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) X[t] = __shfl_sync(hmask, own, hbase + t);
    if (good && swap22_finish(X, dc0, dc1, dc2, dc3, tb, tb4, l, hmask, hbase, strong, z, dnrc)) return true;
    return swap22_elim(Sp, ja, l, hmask, hbase, strong, tb, z, dnrc);
}

// k = 3 swap by four lanes (all 32 lanes of the warp call it, eight swaps at a
// time; base is the first lane of the quad, q this lane in it).  2|1:
// D = [[A, c], [0, lam]] with A 2x2; X solves (A - lam I) X = c, and the one
// reflector H with H (-x0, -x1, 1)^T = beta e_0 gives H D H with lam first.
// 1|2 is the same on the flipped block F D^T F (F reverses the indices).
// Lane q < 3 owns column q of the block, and row q after the exchange between
// the two products.  The result: z = (w0, w1, f) of the reflector (in flipped
// index order if flip), dn = row q of the new (flipped) block.  Returns
// false, for all four lanes, when this path cannot decide (tiny pivot) or
// the swap fails the weak or strong test.  52 FP64 instructions; one lane per
// swap, with CUDA's divisions and square root, took about 140.
__device__ __forceinline__ bool swap3_quad(const double* __restrict__ Sp, int ja, bool flip, int q,
                                           int base, bool strong, double* z, double* dn) {
    const unsigned full = 0xffffffffu;
    const double* c0 = Sp + poff(ja) + ja;
    const double* c1 = Sp + poff(ja + 1) + ja;
    const double* c2 = Sp + poff(ja + 2) + ja;
    // flipped entry (r, c) is entry (2 - c, 2 - r)
    const double d00 = flip ? c2[2] : c0[0], d10 = flip ? c1[2] : c0[1];
    const double d01 = flip ? c2[1] : c1[0], d11 = c1[1];
    const double d02 = c2[0], d12 = flip ? c1[0] : c2[1], lam = flip ? c0[0] : c2[2];
    unsigned long long mx = abs_bits(d00);
    auto up = [](unsigned long long& m, double v) {
        const unsigned long long b = abs_bits(v);
        m = b > m ? b : m;
    };
    up(mx, d10); up(mx, d01); up(mx, d11); up(mx, d02); up(mx, d12); up(mx, lam);
    const unsigned long long tb = thresh_bits(mx);
    const double a00 = d00 - lam, a11 = d11 - lam;
    const double det = fma(a00, a11, -(d01 * d10));
    // |det| must not be tiny against the entries
    unsigned long long am = abs_bits(a00);
    up(am, d01); up(am, d10); up(am, a11);
    const double amax = bits_double(am);
    bool ok = abs_bits(det) > abs_bits(1e-4 * amax * amax);
    const double rdet = rcp64(ok ? det : 1.0);
    // lane 1 of the quad computes x1, the others x0
    const double xo = fma(q == 1 ? a00 : a11, q == 1 ? d12 : d02, -((q == 1 ? d10 : d01) * (q == 1 ? d02 : d12))) *
                      rdet;
    const double x0 = __shfl_sync(full, xo, base), w1 = -__shfl_sync(full, xo, base + 1);
    double w0, f;
    refl3(-x0, w1, &w0, &f);
    // column q of H D
    double t0 = q == 0 ? d00 : (q == 1 ? d01 : d02), t1 = q == 0 ? d10 : (q == 1 ? d11 : d12);
    double t2 = q >= 2 ? lam : 0.0;
    const double s0 = t0, s1 = t1, s2 = t2;  // column q of D
    apply_refl3(w0, w1, f, &t0, &t1, &t2);
    // 3x3 transposition within the quad (lane 3 mirrors lane 2)
    auto flip3 = [&](double& v0, double& v1, double& v2) {
        const double a0 = __shfl_sync(full, v0, base), a1 = __shfl_sync(full, v1, base);
        const double a2 = __shfl_sync(full, v2, base), b0 = __shfl_sync(full, v0, base + 1);
        const double b1 = __shfl_sync(full, v1, base + 1), b2 = __shfl_sync(full, v2, base + 1);
        const double e0 = __shfl_sync(full, v0, base + 2), e1 = __shfl_sync(full, v1, base + 2);
        const double e2 = __shfl_sync(full, v2, base + 2);
        v0 = q == 0 ? a0 : (q == 1 ? a1 : a2);
        v1 = q == 0 ? b0 : (q == 1 ? b1 : b2);
        v2 = q == 0 ? e0 : (q == 1 ? e1 : e2);
    };
    flip3(t0, t1, t2);                      // row q of H D
    apply_refl3(w0, w1, f, &t0, &t1, &t2);  // row q of H D H
    // weak test: rows 1 and 2 of column 0 must vanish
    if (q > 0) {
        ok = ok && abs_bits(t0) <= tb;
        t0 = 0.0;
    }
    dn[0] = t0;
    dn[1] = t1;
    dn[2] = t2;
    if (strong) {
        apply_refl3(w0, w1, f, &t0, &t1, &t2);  // row q of Dt0 H
        flip3(t0, t1, t2);                      // column q of it
        apply_refl3(w0, w1, f, &t0, &t1, &t2);
        ok = ok && abs_bits(t0 - s0) <= tb && abs_bits(t1 - s1) <= tb && abs_bits(t2 - s2) <= tb;
    }
    z[0] = w0;
    z[1] = w1;
    z[2] = f;
    const unsigned votes = __ballot_sync(full, ok);
    return ((votes >> base) & 15u) == 15u;
}

// Swap types of a step, each handled by its own warps (FP64 issue costs the
// same for 1 or 32 active lanes, so lanes of a warp must share one code path):
//   T_11: 1x1|1x1 (Givens), T_3: 1x2 or 2x1 (k = 3), T_22: 2x2|2x2 (k = 4).
constexpr int T_11 = 0, T_3 = 1, T_22 = 2;

// Writes U's digit slices for the split-precision updates (ozaki.cuh): the
// balanced base-256 digits of every entry relative to the largest exponent of
// its column, as fp16, in the tensor cores' 128-byte-swizzled K-major layout
// [output half][K half][slice][column n mod 64][128 B] (U(k, n) is entry k of
// column n), then one int exponent per column.  Columns/rows beyond w are
// zero.
__device__ __forceinline__ void write_u_slices(const double* U, int w, unsigned char* out) {
    int* cexp = reinterpret_cast<int*>(out + OZ_UDIG_ELEMS * 2);
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5;
    __shared__ int ce[WMAX];
    for (int n = warp; n < WMAX; n += nth / 32) {
        int em = 0;
        if (n < w)
            for (int k = lane; k < w; k += 32) {
                int e = (int)((((unsigned long long)__double_as_longlong(U[n * w + k])) >> 52) & 0x7ff);
                em = e > em ? e : em;
            }
        for (int o = 16; o; o >>= 1) {
            int v = __shfl_xor_sync(0xffffffffu, em, o);
            em = v > em ? v : em;
        }
        if (lane == 0) { ce[n] = em; cexp[n] = em; }
    }
    __syncthreads();
    // unit (column n, 16-byte chunk c of K half kh): consecutive threads fill
    // the 8 chunks of one 128-byte row, then the next column, so the global
    // writes of a warp are 512 contiguous bytes
    for (int u = tid; u < WMAX * (WMAX / 8); u += nth) {
        const int c = u & 7, n = (u >> 3) & (WMAX - 1), kh = u >> 10;
        long long G[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = 64 * kh + 8 * c + j;
            G[j] = (n < w && k < w) ? oz::oz_balanced(U[n * w + k], ce[n]) : oz::OZ_BIAS;
        }
        unsigned char* dst = out + ((size_t)((n >> 6) * 2 + kh) * OZ_SLICES * 64 + (n & 63)) * 128 +
                             (size_t)((c ^ (n & 7)) << 4);
        unsigned wv[4];
#define GBR_PUT_SLICE(P)                                                                   \
        _Pragma("unroll") for (int t = 0; t < 4; ++t) wv[t] =                                  \
            oz::oz_digits2<P>(G[2 * t], G[2 * t + 1]);                                         \
        *reinterpret_cast<uint4*>(dst + (size_t)((P) - 1) * 64 * 128) =                    \
            make_uint4(wv[0], wv[1], wv[2], wv[3]);
        GBR_PUT_SLICE(1) GBR_PUT_SLICE(2) GBR_PUT_SLICE(3) GBR_PUT_SLICE(4) GBR_PUT_SLICE(5)
        GBR_PUT_SLICE(6) GBR_PUT_SLICE(7)
#undef GBR_PUT_SLICE
    }
}

// Dynamic shared memory needed by window_body: U, the packed window, the
// transforms and swap lists of two steps, selection flags.
constexpr size_t kWindowSmem = sizeof(double) * ((size_t)WMAX * WMAX +
                                                 (size_t)((WMAX * (WMAX + 3)) / 2) +
                                                 (size_t)2 * MAXSW * 16) +
                               sizeof(int) * 2 * MAXSW + WMAX;
// A wide window task keeps only the transforms, swap lists and flags here.
constexpr size_t kWindowSmemWide = sizeof(double) * (size_t)2 * (WMAX_WIDE / 2) * 16 +
                                   sizeof(int) * 2 * (WMAX_WIDE / 2) + WMAX_WIDE;

// A swap of a step: its slot's descriptor holds j (first row), k (rows), the
// size p of the block above (0: a standardization rotation) and whether the
// full transform computed it (Z_MATRIX).  A rejected swap has k = 0.  Slots
// are numbered by size, k = 4 first, then k = 3, then k = 2.
constexpr int Z_MATRIX = 16;
__device__ __forceinline__ int sw_desc(int j, int kk, int p) { return j | (kk << 16) | (p << 24); }
__device__ __forceinline__ int sw_j(int d) { return d & 0xffff; }
__device__ __forceinline__ int sw_kk(int d) { return (d >> 16) & 0xff; }
__device__ __forceinline__ int sw_p(int d) { return d >> 24; }

// The slot's transformation Z (x <- x Z for a row x of K values, Z^T x for a
// column):
//   k = 2: Z = [[c, -s], [s, c]] as (c, s);
//   k = 3: one reflector (w0, w1, f), in reversed index order for 1|2;
//   k = 4: two reflectors (w0, w1, f) on 0..2 and (u0, u1, f') on 1..3;
//   Z_MATRIX: the k x k matrix, column-major with leading dimension 4.
// The reflectors take 6 and 12 FP64 instructions where the matrices take 9
// and 16.
//
// One item of a step's products: K values of the packed window or of U at a,
// a + o1, a + o2, a + o3 and the slot's Z (reversed for a flipped reflector).
struct Item {
    double* a;
    const double* z;
    int o1, o2, o3;
    bool ok, matrix;
};
// st, inc: the second value is st after the first, the step then grows by inc.
template <int K>
__device__ __forceinline__ Item make_item(double* a, int st, int inc, int d, const double* z, bool ok) {
    Item t;
    t.matrix = K > 2 && (sw_kk(d) & Z_MATRIX);
    t.ok = ok && sw_kk(d) != 0;
    t.a = a;
    t.o1 = st;
    t.o2 = 2 * st + inc;
    t.o3 = 3 * (st + inc);
    if (K == 3 && sw_p(d) == 1 && !t.matrix) {
        t.a = a + t.o2;
        t.o1 = -(st + inc);
        t.o2 = -t.o2;
    }
    t.z = z;
    return t;
}
template <int K>
__device__ __forceinline__ void item_load(const Item& t, double* x) {
    x[0] = t.a[0];
    x[1] = t.a[t.o1];
    if constexpr (K > 2) x[2] = t.a[t.o2];
    if constexpr (K > 3) x[3] = t.a[t.o3];
}
template <int K>
__device__ __forceinline__ void item_store(const Item& t, const double* x) {
    t.a[0] = x[0];
    t.a[t.o1] = x[1];
    if constexpr (K > 2) t.a[t.o2] = x[2];
    if constexpr (K > 3) t.a[t.o3] = x[3];
}
template <int K, bool MAT>
__device__ __forceinline__ void item_apply(const Item& t, double* x) {
    const double* Z = t.z;
    if constexpr (K == 2) {
        const double c = Z[0], s = Z[1];
        const double y = fma(s, x[1], c * x[0]);
        x[1] = fma(c, x[1], -(s * x[0]));
        x[0] = y;
    } else {
        if (MAT && t.matrix) {
            double y[K];
#pragma unroll
            for (int c = 0; c < K; ++c) {
                double acc = 0.0;
#pragma unroll
                for (int i = 0; i < K; ++i) acc = fma(x[i], Z[c * 4 + i], acc);
                y[c] = acc;
            }
#pragma unroll
            for (int c = 0; c < K; ++c) x[c] = y[c];
        } else {
            apply_refl3(Z[0], Z[1], Z[2], &x[0], &x[1], &x[2]);
            if constexpr (K == 4) apply_refl3(Z[3], Z[4], Z[5], &x[1], &x[2], &x[3]);
        }
    }
}
// One item per lane, or two whose instructions interleave: an FP64 result is
// 64 cycles away, and three product warps per sub-partition with one chain
// each leave its pipe idle half of the time.  All lanes of the warp call.
template <int K>
__device__ __forceinline__ void item_run(const Item& t) {
    if (!t.ok) return;
    double x[K];
    item_load<K>(t, x);
    item_apply<K, true>(t, x);
    item_store<K>(t, x);
}
template <int K>
__device__ __forceinline__ void item_run2(const Item& t, const Item& v) {
    if (!__any_sync(0xffffffffu, v.ok) ||
        (K > 2 && __any_sync(0xffffffffu, (t.ok && t.matrix) || (v.ok && v.matrix)))) {
        item_run<K>(t);
        item_run<K>(v);
        return;
    }
    double x[K], y[K];
#pragma unroll
    for (int i = 0; i < K; ++i) x[i] = y[i] = 0.0;
    if (t.ok) item_load<K>(t, x);
    if (v.ok) item_load<K>(v, y);
    item_apply<K, false>(t, x);
    item_apply<K, false>(v, y);
    if (t.ok) item_store<K>(t, x);
    if (v.ok) item_store<K>(v, y);
}

// Last i in [lo, hi] with pre[i] <= it (pre is nondecreasing, pre[lo] <= it).
__device__ __forceinline__ int prefix_slot(const int* pre, int lo, int hi, int it) {
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= it) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Named barriers of the window task's two warp groups (barrier 0 is
// __syncthreads): PRODUCTS among the product warps, CRIT from the product
// warps (arrive) to the transform warps (wait).
__device__ __forceinline__ void bar_products(int threads) {
    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}
__device__ __forceinline__ void bar_crit_arrive() {
    asm volatile("bar.arrive 2, %0;" ::"n"(WIN_THREADS) : "memory");
}
__device__ __forceinline__ void bar_crit_wait() {
    asm volatile("bar.sync 2, %0;" ::"n"(WIN_THREADS) : "memory");
}

// Near-diagonal part of a step's products.  The next step's transforms read
// only diagonal blocks (entries with c - r <= 3).  A left item (swap at j,
// column c) is critical if c < j + CRIT_L, a right item of S (swap at j of
// size k, row r) if r >= j + k - CRIT_R.  Every product reaching an entry
// with c - r <= 3 is critical; no other product reaches one; and a left
// item that shares an entry with a critical right item is critical itself
// (c <= j2 + k2 - 1 <= r + 7 <= j1 + 10), so that applying all critical left
// items, then all critical right items, then the other left items and the
// other right items applies every entry's left transformation before its
// right one, as the unsplit phases do.
constexpr int CRIT_L = 11, CRIT_R = 8;

// abort_word (ABORT on rejection, else null): a window task that starts
// after it was set does nothing (U = I, *skip_out = 1); a window task that
// rejects a swap sets it, finishes the step it is in, restores the standard
// form of its 2x2 blocks and stops.  skip_out (nullable) receives 0 or 1.
//
// WM is the largest window of the instance: WMAX keeps S and U in shared
// memory; WMAX_WIDE keeps the packed S window in gsp (this CTA's global
// scratch, WIDE_SP_STRIDE doubles) and forms U in place in Ug (no split-
// precision slices).  The steps are the same; only where the two arrays live
// differs.
//
// The steps run as a two-stage pipeline over two groups of warps (blockDim
// must be WIN_THREADS): while the product warps apply step q's left and
// right transformations (to S and to U), the WIN_TWARPS transform warps,
// the same number on each SM sub-partition, compute the transforms of
// step q + 1.  Those read only the
// diagonal blocks of step q + 1, so the product warps first apply the part
// of step q that reaches near the diagonal (CRIT_L, CRIT_R), signal the
// transform warps, and then the rest; the two groups touch disjoint entries
// from there on.  Every entry receives the same operations in the same order
// as in a step-by-step execution, so the result does not change.  The state
// of a step (swap lists, transforms, prefix sums of the product work) is kept
// for two steps, by the step's parity.
template <int WM>
__device__ __forceinline__ void window_body_t(int n, double* __restrict__ S, int ldS, int s0, int w,
                                              uint8_t* __restrict__ gsel, double* __restrict__ Ug,
                                              int strong, DevCounters* __restrict__ ctr,
                                              unsigned char* smem_raw,
                                              unsigned char* __restrict__ uslices,
                                              int* abort_word, int* skip_out,
                                              double* __restrict__ gsp) {
    static_assert(WM == WMAX || WM == WMAX_WIDE, "window kernel instances");
    constexpr bool WIDE = WM > WMAX;
    constexpr int MSW = WM / 2;  // at most one swap per two positions
    constexpr int NTW = WIN_TWARPS;
    static_assert(NTW % 4 == 0 && NTW < WIN_THREADS / 32, "transform warps per sub-partition");
    double* U = WIDE ? Ug : reinterpret_cast<double*>(smem_raw);        // w*w
    double* Sp = WIDE ? gsp : U + WM * WM;                               // packed window
    double* Zbuf = WIDE ? reinterpret_cast<double*>(smem_raw) : Sp + poff(WM);  // [2][MSW * 16]
    int* swbuf = reinterpret_cast<int*>(Zbuf + 2 * MSW * 16);  // [2][MSW]: descriptors
    uint8_t* sel = reinterpret_cast<uint8_t*>(swbuf + 2 * MSW);
    __shared__ int nsw[2], nrej, nacc;  // swaps of a step, by parity; rejected, accepted
    unsigned long long wflops = 0;   // per thread (phase D), summed at the end
    __shared__ int tcnt2[2][3];         // swaps per type (T_11, T_3, T_22: k = 2, 3, 4)
    // prefix sums over the slots: far left-apply columns, far right-apply
    // rows of S, right-apply rows of U
    __shared__ int kpre_l2[2][MSW + 1], kpre_s2[2][MSW + 1], kpre_u2[2][MSW + 1];
    // Rows [urlo[c], urhi[c]] hold every nonzero of column c of U: U starts as
    // I and a swap on columns [j, j+k) mixes only those columns, so the rows
    // outside the union of their ranges stay exactly zero and are skipped.
    __shared__ short urlo[WM], urhi[WM];
    __shared__ short slo2[2][MSW], shi2[2][MSW];  // per slot: U rows its right transform touches

    const int tid = threadIdx.x;
    const int nth = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31;

    if (abort_word) {
        __shared__ int skip;
        __syncthreads();
        if (tid == 0) skip = *reinterpret_cast<volatile int*>(abort_word) != 0;
        __syncthreads();
        if (skip) {
            // the reordering stopped before this window started: U = I
            for (int i = tid; i < w * w; i += nth) Ug[i] = ((i % w) == (i / w)) ? 1.0 : 0.0;
            if (tid == 0 && skip_out) *skip_out = 1;
            return;
        }
    }
    if (tid == 0 && skip_out) *skip_out = 0;

    // load: packed window of S, selection, U = I
    for (int c = 0; c < w; ++c) {
        int rows = min(c + 2, w);
        for (int r = tid; r < rows; r += nth)
            Sp[poff(c) + r] = __ldcg(&S[cm(s0 + r, s0 + c, ldS)]);
    }
    for (int i = tid; i < w * w; i += nth) U[i] = ((i % w) == (i / w)) ? 1.0 : 0.0;
    for (int i = tid; i < w; i += nth) {
        sel[i] = __ldcg(&gsel[s0 + i]);
        urlo[i] = (short)i;
        urhi[i] = (short)i;
    }
    __shared__ int wall_top, wall_bot;
    if (tid == 0) {
        nrej = 0;
        nacc = 0;
        wall_top = s0 > 0 && __ldcg(&S[cm(s0, s0 - 1, ldS)]) != 0.0;
        wall_bot = s0 + w < n && __ldcg(&S[cm(s0 + w, s0 + w - 1, ldS)]) != 0.0;
    }
    __syncthreads();
    if (tid == 0 && wall_top) sel[0] = SEL_WALL;
    if (tid == 0 && wall_bot) sel[w - 1] = SEL_WALL;

    // --- control of a step boundary, by one transform warp while the product
    // warps start on the critical products (integer work on bit masks of the
    // window's positions; with all warps and block barriers between its parts
    // it took 3.4K cycles of a step's 24K).
    //
    // phase D of the step of parity pp with nsq swaps: move the selection
    // flags with the blocks and widen the U row ranges of the columns each
    // accepted transform mixed.
    auto phase_d = [&](int pp, int nsq) {
        const int* desc = swbuf + pp * MSW;
        for (int sw = lane; sw < nsq; sw += 32) {
            const int d = desc[sw], j = sw_j(d), p = sw_p(d), k = sw_kk(d) & (Z_MATRIX - 1);
            if (k == 0) {
                sel[j + p] = SEL_STUCK;  // the selected block
                continue;
            }
            const int lo = slo2[pp][sw], hi = shi2[pp][sw];
            // in-window flops of this accepted transform: k x k applied to
            // w - j - k columns (left) and j rows of S + its U rows (right)
            wflops += 2ull * k * k * (unsigned long long)((w - j - k) + j + (hi - lo + 1));
            const int q = k - p;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < k) {
                    urlo[j + c] = (short)lo;
                    urhi[j + c] = (short)hi;
                    if (p > 0) sel[j + c] = c < q ? SEL_YES : SEL_NO;  // (0: blocks do not move)
                }
        }
        __syncwarp();
    };
    // phase A1 of the step of parity pi: every selected block whose upper
    // neighbour is an unselected block swaps with it.  In the final pass, the
    // 2x2 blocks whose standard form has to be restored are listed instead
    // (the fast swap paths leave it to this pass).  Returns the number of
    // swaps; bit t & 31 of word t >> 5 stands for position t.
    constexpr int NWORD = WM / 32;
    auto list_swaps = [&](int pi, bool fin) {
        int* desc = swbuf + pi * MSW;
        unsigned bs[NWORD], sw[NWORD];     // block starts, swaps (by the selected block's start)
        unsigned one[NWORD], two[NWORD];   // the block above is 1x1; a 2x2 block from here on
        unsigned yes[NWORD], no[NWORD];    // selected, unselected
        unsigned carry = 0;                // the word before ends in a stuck position
#pragma unroll
        for (int i = 0; i < NWORD; ++i) {
            bs[i] = yes[i] = no[i] = 0u;
            if (32 * i < w) {
                const int t = 32 * i + lane;
                const bool in = t < w;
                const bool start = in && (t == 0 || is_zero(Sp[poff(t - 1) + t]));
                const int f = in ? sel[t] : SEL_WALL;
                bs[i] = __ballot_sync(0xffffffffu, start);
                yes[i] = __ballot_sync(0xffffffffu, f == SEL_YES);
                no[i] = __ballot_sync(0xffffffffu, f == SEL_NO);
                // a stuck 2x2 block is flagged on both of its rows
                const unsigned st = __ballot_sync(0xffffffffu, f == SEL_STUCK);
                const unsigned both = ((st << 1) | carry) & ~bs[i];
                if (both) {
                    if (in && ((both >> lane) & 1u)) sel[t] = SEL_STUCK;
                    yes[i] &= ~both;
                    no[i] &= ~both;
                }
                carry = (st | both) >> 31;
            }
        }
        int n4 = 0, n3 = 0, n2 = 0;
#pragma unroll
        for (int i = 0; i < NWORD; ++i) {
            sw[i] = one[i] = two[i] = 0u;
            if (32 * i < w) {
                const unsigned bp = i ? bs[i > 0 ? i - 1 : 0] : 0u, np = i ? no[i > 0 ? i - 1 : 0] : 0u;
                const unsigned bn = i + 1 < NWORD ? bs[i + 1 < NWORD ? i + 1 : i] : 0u;
                const int left = w - 32 * i;  // positions from this word on
                const unsigned more = left > 32 ? ~0u : (1u << (left - 1)) - 1u;  // t + 1 < w
                one[i] = (bs[i] << 1) | (bp >> 31);
                two[i] = ~((bs[i] >> 1) | (bn << 31)) & more;
                if (!fin) {
                    const unsigned nabove = (one[i] & ((no[i] << 1) | (np >> 31))) |
                                            (~one[i] & ((no[i] << 2) | (np >> 30)));
                    sw[i] = bs[i] & yes[i] & nabove;
                    if (i == 0) sw[i] &= ~1u;
                    n4 += __popc(sw[i] & ~one[i] & two[i]);
                    n3 += __popc(sw[i] & (one[i] ^ ~two[i]));
                    n2 += __popc(sw[i] & one[i] & ~two[i]);
                } else {
                    bool stale = false;
                    const int t = 32 * i + lane;
                    if (((bs[i] & two[i]) >> lane) & 1u) {
                        const double m00 = Sp[poff(t) + t], m10 = Sp[poff(t) + t + 1];
                        const double m01 = Sp[poff(t + 1) + t], m11 = Sp[poff(t + 1) + t + 1];
                        stale = !(m00 == m11 && m01 * m10 < 0.0);
                    }
                    sw[i] = __ballot_sync(0xffffffffu, stale);
                    n2 += __popc(sw[i]);
                }
            }
        }
        int at4 = 0, at3 = n4, at2 = n4 + n3;
        const unsigned below = (1u << lane) - 1u;
#pragma unroll
        for (int i = 0; i < NWORD; ++i) {
            if (32 * i < w) {
                const unsigned m4 = fin ? 0u : sw[i] & ~one[i] & two[i];
                const unsigned m3 = fin ? 0u : sw[i] & (one[i] ^ ~two[i]), m2 = sw[i] & ~(m4 | m3);
                if ((sw[i] >> lane) & 1u) {
                    const int t = 32 * i + lane;
                    const int p = (one[i] >> lane) & 1u ? 1 : 2, q = (two[i] >> lane) & 1u ? 2 : 1;
                    const int slot = (m4 >> lane) & 1u   ? at4 + __popc(m4 & below)
                                     : (m3 >> lane) & 1u ? at3 + __popc(m3 & below)
                                                         : at2 + __popc(m2 & below);
                    desc[slot] = fin ? sw_desc(t, 2, 0) : sw_desc(t - p, p + q, p);
                }
                at4 += __popc(m4);
                at3 += __popc(m3);
                at2 += __popc(m2);
            }
        }
        if (lane < 3) tcnt2[pi][lane] = lane == T_11 ? n2 : (lane == T_3 ? n3 : n4);
        return n4 + n3 + n2;
    };

    // Prefix sums of the product work of the ns swaps of the step of parity
    // pi, by one warp: far left columns, far right rows of S, right rows of U
    // (whose range per swap, from urlo/urhi, it also records).  All listed
    // swaps are counted; a rejected one is skipped when applied.
    auto prefix_sums = [&](int pi, int ns) {
        const int* desc = swbuf + pi * MSW;
        int runl = 0, runr = 0, runu = 0;
        for (int base = 0; base < ns; base += 32) {
            const int i = base + lane;
            int nl = 0, nr = 0, nu = 0;
            if (i < ns) {
                // (a swap rejected by now has k = 0: no items)
                const int d = desc[i], j = sw_j(d), k = sw_kk(d) & (Z_MATRIX - 1);
                if (k > 0) {
                    int lo = urlo[j], hi = urhi[j];
                    for (int c = 1; c < k; ++c) {
                        lo = min(lo, (int)urlo[j + c]);
                        hi = max(hi, (int)urhi[j + c]);
                    }
                    slo2[pi][i] = (short)lo;
                    shi2[pi][i] = (short)hi;
                    nl = max(0, w - j - CRIT_L);
                    nr = max(0, j + k - CRIT_R);
                    nu = hi - lo + 1;
                }
            }
            int il = nl, ir = nr, iu = nu;
            for (int o = 1; o < 32; o <<= 1) {
                int a = __shfl_up_sync(0xffffffffu, il, o);
                int b2 = __shfl_up_sync(0xffffffffu, ir, o);
                int c2 = __shfl_up_sync(0xffffffffu, iu, o);
                if (lane >= o) { il += a; ir += b2; iu += c2; }
            }
            if (i < ns) {
                kpre_l2[pi][i + 1] = runl + il;
                kpre_s2[pi][i + 1] = runr + ir;
                kpre_u2[pi][i + 1] = runu + iu;
            }
            runl += __shfl_sync(0xffffffffu, il, 31);
            runr += __shfl_sync(0xffffffffu, ir, 31);
            runu += __shfl_sync(0xffffffffu, iu, 31);
        }
        if (lane == 0) kpre_l2[pi][0] = kpre_s2[pi][0] = kpre_u2[pi][0] = 0;
    };

    // --- phase A2 of the step of parity pi, by the transform warps (warps
    // 0 .. NTW - 1, NTW / 4 per sub-partition).  An FP64 instruction costs the
    // same for 1 or 32 active lanes, so a warp takes swaps of one type at a
    // time, as many as its lanes hold: two 2|2 swaps, eight k = 3 swaps or 32
    // rotations, dealt out in this order (the longest chains first).
    auto transforms = [&](int pi) {
        double* Zs = Zbuf + pi * MSW * 16;
        int* desc = swbuf + pi * MSW;
        const int* tcnt = tcnt2[pi];
        const int n22 = (tcnt[T_22] + 1) >> 1, n3 = (tcnt[T_3] + 7) >> 3;
        const int nunits = n22 + n3 + ((tcnt[T_11] + 31) >> 5);
        // the full transform of a swap, by one lane
        auto full = [&](int slot) {
            const int ja = sw_j(desc[slot]), p = sw_p(desc[slot]), k = sw_kk(desc[slot]);
            double D[16], Zl[16], Dn[16];
            for (int cc = 0; cc < k; ++cc)
                for (int rr = 0; rr < k; ++rr)
                    D[cc * 4 + rr] = (rr <= cc + 1) ? Sp[poff(ja + cc) + ja + rr] : 0.0;
            if (swap_transform(D, p, k - p, strong != 0, Zl, Dn)) {
                for (int cc = 0; cc < k; ++cc)
                    for (int rr = 0; rr <= min(cc + 1, k - 1); ++rr)
                        Sp[poff(ja + cc) + ja + rr] = Dn[cc * 4 + rr];
                for (int e = 0; e < 16; ++e) Zs[slot * 16 + e] = Zl[e];
                desc[slot] = sw_desc(ja, k | Z_MATRIX, p);
                atomicAdd(&nacc, 1);
            } else {
                desc[slot] = sw_desc(ja, 0, p);
                atomicAdd(&nrej, 1);
            }
        };
        for (int u = warp; u < nunits; u += NTW) {
            if (u < n22) {
                // two 2|2 swaps, one per half-warp
                const int h = lane >> 4, l = lane & 15, slot = 2 * u + h;
                const unsigned hmask = h ? 0xffff0000u : 0x0000ffffu;
                if (slot < tcnt[T_22]) {
                    const int ja = sw_j(desc[slot]);
                    double z[6], dnrc = 0.0;
                    const bool ok = swap22_halfwarp(Sp, ja, l, hmask, h * 16, strong != 0, z, &dnrc);
                    const int r = l & 3, c = l >> 2;
                    if (ok) {
                        if (r <= c + 1) Sp[poff(ja + c) + ja + r] = dnrc;
                        if (l == 0) {
#pragma unroll
                            for (int e = 0; e < 6; ++e) Zs[slot * 16 + e] = z[e];
                            atomicAdd(&nacc, 1);
                        }
                    } else if (l == 0) {
                        full(slot);
                    }
                }
                __syncwarp();
            } else if (u < n22 + n3) {
                // eight k = 3 swaps, one per quad of lanes
                const int q = lane & 3, i = 8 * (u - n22) + (lane >> 2);
                const bool act = i < tcnt[T_3];
                const int slot = tcnt[T_22] + (act ? i : tcnt[T_3] - 1);
                const int ja = sw_j(desc[slot]);
                const bool flip = sw_p(desc[slot]) == 1;
                double z[3], dn[3];
                const bool ok = swap3_quad(Sp, ja, flip, q, lane & ~3, strong != 0, z, dn);
                __syncwarp();
                if (act && ok) {
                    // row q of the flipped block: entry (q, c) is (2 - c, 2 - q)
                    if (q < 3)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const int rr = flip ? 2 - c : q, cc = flip ? 2 - q : c;
                            if (rr <= cc + 1) Sp[poff(ja + cc) + ja + rr] = dn[c];
                        }
                    if (q == 0) {
                        Zs[slot * 16] = z[0];
                        Zs[slot * 16 + 1] = z[1];
                        Zs[slot * 16 + 2] = z[2];
                        atomicAdd(&nacc, 1);
                    }
                } else if (act && q == 0) {
                    full(slot);
                }
                __syncwarp();
            } else {
                // 32 rotations
                const int i = 32 * (u - n22 - n3) + lane;
                if (i < tcnt[T_11]) {
                    const int slot = tcnt[T_22] + tcnt[T_3] + i;
                    const int ja = sw_j(desc[slot]), p = sw_p(desc[slot]);
                    double* Z = &Zs[slot * 16];
                    double* c0 = Sp + poff(ja) + ja;
                    double* c1 = Sp + poff(ja + 1) + ja;
                    if (p == 0) {
                        // restore the standard form of the 2x2 block at ja
                        double m[16];
                        m[0] = c0[0];
                        m[1] = c0[1];
                        m[4] = c1[0];
                        m[5] = c1[1];
                        double cs, sn;
                        standardize2(m, &cs, &sn);
                        c0[0] = m[0];
                        c0[1] = m[1];
                        c1[0] = m[4];
                        c1[1] = m[5];
                        Z[0] = cs;
                        Z[1] = sn;
                    } else {
                        // Givens rotation from (t12, t22 - t11), always
                        // accepted; t12 stays (the norm of the block and of
                        // its diagonal do)
                        const double t11 = c0[0], t12 = c1[0], t22 = c1[1];
                        double c = 1.0, sn = 0.0;
                        if (t11 != t22) givens64(t12, t22 - t11, &c, &sn);
                        Z[0] = c;
                        Z[1] = sn;
                        c0[0] = t22;
                        c0[1] = 0.0;
                        c1[1] = t11;
                        atomicAdd(&nacc, 1);
                    }
                }
                __syncwarp();
            }
        }
    };

    // --- phases B and C of the step of parity pp, by the product warps:
    // critical left items, critical right items of S (then the transform
    // warps may start), far left items, far right items of S and the right
    // items of U.  Within each part the items are grouped by k so that the
    // lanes of a warp run the same k, and whole warps claim 32 items at a
    // time (one claim counter per part): an FP64 instruction holds its
    // sub-partition's pipe for the same time with 1 or 32 lanes, and the
    // transform warps load some sub-partitions' pipes more than others, so
    // the warps of the less loaded sub-partitions take more items.
    // has = the step had swaps; the barriers run either way.
    // A small window is bound by the chains of its transforms (w = 32: 7.1K of
    // a step's 10.3K cycles), and the longest one, on warp 0, would share its
    // sub-partition's FP64 pipe with three product warps: there they stay
    // away.  A large window is bound by the products and uses all of them.
    // Measured, a whole window with and without: w = 32 173 and 176 us, w = 48
    // 245 and 257 us, w = 64 343 and 362 us; at w = 96 it costs 3%.
    constexpr int FEW_W = 64;
    const bool few = w <= FEW_W;
    const int npw = (WIN_THREADS / 32 - NTW) - (few ? WIN_THREADS / 128 - NTW / 4 : 0);  // product warps
    const int pw = few ? ((warp & 3) ? (warp >> 2) * 3 + (warp & 3) - 1 - NTW / 4 * 3 : -1) : warp - NTW;
    __shared__ int pclaim[2][4];  // by the parity of the step applied
    auto products = [&](int pp, bool has) {
        const double* Zs = Zbuf + pp * MSW * 16;
        const int* desc = swbuf + pp * MSW;
        const int m4 = tcnt2[pp][T_22], m3 = tcnt2[pp][T_3], m2 = tcnt2[pp][T_11];
        constexpr int NCL = CRIT_L - 2, NCR = CRIT_R - 2;  // item slots per swap
        // The items of part `ph` (t4, t3, t2 of them per size), by chunks of
        // one size, those with the most work per item first: PER items per
        // lane (one for k = 4).  The first chunk of a warp is its own; the
        // claim of the next one is under way while it works.
        auto part = [&](auto PER, int ph, int t4, int t3, int t2, auto&& item) {
            constexpr int per = decltype(PER)::value;
            const int c4 = (t4 + 31) / 32, c3 = c4 + (t3 + 32 * per - 1) / (32 * per);
            const int n = c3 + (t2 + 32 * per - 1) / (32 * per);
            auto chunk = [&](auto K, int base, int t) {
                constexpr int k = decltype(K)::value;
                const int it = base + lane;
                if constexpr (k == 4 || per == 1)
                    item_run<k>(item(K, min(it, t - 1), it < t));
                else
                    item_run2<k>(item(K, min(it, t - 1), it < t), item(K, min(it + 32, t - 1), it + 32 < t));
            };
            for (int c = pw; c < n;) {
                int nx = 0;
                if (n > npw && lane == 0) nx = atomicAdd(&pclaim[pp][ph], 1);
                if (c < c4)
                    chunk(std::integral_constant<int, 4>{}, 32 * c, t4);
                else if (c < c3)
                    chunk(std::integral_constant<int, 3>{}, 32 * per * (c - c4), t3);
                else
                    chunk(std::integral_constant<int, 2>{}, 32 * per * (c - c3), t2);
                if (n <= npw) break;
                c = npw + __shfl_sync(0xffffffffu, nx, 0);
            }
        };
        // slots of size k: first one and their number
        auto first = [&](int k) { return k == 4 ? 0 : (k == 3 ? m4 : m4 + m3); };
        auto many = [&](int k) { return k == 4 ? m4 : (k == 3 ? m3 : m2); };
        constexpr std::integral_constant<int, 1> PER1{};
        constexpr std::integral_constant<int, 2> PER2{};
        if (has)
            part(PER1, 0, m4 * NCL, m3 * NCL, m2 * NCL, [&](auto K, int it, bool ok) {
                constexpr int k = decltype(K)::value;
                const int slot = first(k) + it / NCL, d = desc[slot], j = sw_j(d), c = j + k + it % NCL;
                return make_item<k>(Sp + poff(c) + j, 1, 0, d, Zs + slot * 16, ok && c < min(w, j + CRIT_L));
            });
        bar_products(32 * npw);
        if (has)
            part(PER1, 1, m4 * NCR, m3 * NCR, m2 * NCR, [&](auto K, int it, bool ok) {
                constexpr int k = decltype(K)::value;
                const int slot = first(k) + it / NCR, d = desc[slot], j = sw_j(d), r = j - 1 - it % NCR;
                return make_item<k>(Sp + poff(j) + r, j + 2, 1, d, Zs + slot * 16,
                                    ok && r >= max(0, j + k - CRIT_R));
            });
        __threadfence_block();
        bar_crit_arrive();
        const int* pl = kpre_l2[pp];
        const int* ps = kpre_s2[pp];
        const int* pu = kpre_u2[pp];
        if (has)
            part(PER2, 2, pl[m4], pl[m4 + m3] - pl[m4], pl[m4 + m3 + m2] - pl[m4 + m3],
                 [&](auto K, int it, bool ok) {
                     constexpr int k = decltype(K)::value;
                     const int f = first(k);
                     it += pl[f];
                     const int slot = prefix_slot(pl, f, f + many(k) - 1, it), d = desc[slot], j = sw_j(d);
                     return make_item<k>(Sp + poff(j + CRIT_L + (it - pl[slot])) + j, 1, 0, d, Zs + slot * 16,
                                         ok);
                 });
        bar_products(32 * npw);
        if (has) {
            // far right rows of S, then the rows of U, of each size
            const int s4 = ps[m4], s3 = ps[m4 + m3] - s4, s2 = ps[m4 + m3 + m2] - ps[m4 + m3];
            part(PER2, 3, s4 + pu[m4], s3 + pu[m4 + m3] - pu[m4], s2 + pu[m4 + m3 + m2] - pu[m4 + m3],
                 [&](auto K, int it, bool ok) {
                     constexpr int k = decltype(K)::value;
                     const int ns = k == 4 ? s4 : (k == 3 ? s3 : s2), f = first(k);
                     const bool u = it >= ns;
                     const int* pre = u ? pu : ps;
                     it += pre[f] - (u ? ns : 0);
                     const int slot = prefix_slot(pre, f, f + many(k) - 1, it), d = desc[slot], j = sw_j(d);
                     it -= pre[slot];
                     double* a = u ? U + j * w + slo2[pp][slot] + it : Sp + poff(j) + it;
                     return make_item<k>(a, u ? w : j + 2, u ? 0 : 1, d, Zs + slot * 16, ok);
                 });
        }
    };

    // Step pipeline.  Iteration i: one warp moves the selection flags of step
    // i - 1 (phase D) and lists step i's swaps (phase A1), then the product
    // warps apply step i - 1 while the transform warps compute step i.  Every
    // accepted swap moves a selected block up and every rejected one retires
    // a block, so the steps end within w * w; the cap only guards against a
    // logic error (reported through the counters).
    bool fin = false;  // the final pass (warp 0)
    int ns_prev = 0;
    if (tid < 8) pclaim[tid >> 2][tid & 3] = 0;
    __syncthreads();
    for (int iter = 0;; ++iter) {
        const int pi = iter & 1, pp = pi ^ 1;
        if (warp < NTW) {
            if (warp == 0) {
                if (ns_prev > 0) phase_d(pp, ns_prev);
                if (abort_word && !fin && nrej > 0) {
                    // ABORT: the first rejection stops the reordering; this
                    // window only restores the standard form of its 2x2 blocks
                    fin = true;
                    if (lane == 0) atomicExch(abort_word, 1);
                }
                int ns = 0;
                if (iter > 4 * WM * WM) {
                    if (lane == 0) atomicAdd(&ctr->step_overflow, 1);
                } else {
                    ns = list_swaps(pi, fin);
                    if (ns == 0 && !fin) {
                        // after the last swap: the pass that restores standard forms
                        fin = true;
                        ns = list_swaps(pi, true);
                    }
                }
                if (lane < 4) pclaim[pi][lane] = 0;
                if (lane == 0) nsw[pi] = ns;
            }
            bar_crit_wait();
            const int ns = nsw[pi];
            if (ns > 0) transforms(pi);
            if (warp == NTW - 1 && ns > 0) prefix_sums(pi, ns);
        } else if (pw >= 0) {
            products(pp, ns_prev > 0);
        } else {
            bar_crit_arrive();
        }
        __syncthreads();
        ns_prev = nsw[pi];
        if (ns_prev == 0) break;
    }
    __shared__ unsigned long long wfl_sum;
    if (tid == 0) wfl_sum = 0;
    __syncthreads();
    for (int o = 16; o; o >>= 1) wflops += __shfl_xor_sync(0xffffffffu, wflops, o);
    if (lane == 0) atomicAdd(&wfl_sum, wflops);
    __syncthreads();
    wflops = wfl_sum;
    // store: window of S, selection, U
    for (int c = 0; c < w; ++c) {
        int rows = min(c + 2, w);
        for (int r = tid; r < rows; r += nth)
            S[cm(s0 + r, s0 + c, ldS)] = Sp[poff(c) + r];
    }
    for (int i = tid; i < w; i += nth)
        if (sel[i] != SEL_WALL) gsel[s0 + i] = sel[i];
    if constexpr (!WIDE) {
        for (int i = tid; i < w * w; i += nth) Ug[i] = U[i];
        if (uslices) write_u_slices(U, w, uslices);
    }
    if (tid == 0) {
        atomicAdd(&ctr->swaps, (unsigned long long)nacc);
        atomicAdd(&ctr->rejected, (unsigned long long)nrej);
        atomicAdd(&ctr->win_flops, wflops);
    }
}


// The shared-memory window task (w <= WMAX).
__device__ __forceinline__ void window_body(int n, double* __restrict__ S, int ldS, int s0, int w,
                                            uint8_t* __restrict__ gsel, double* __restrict__ Ug,
                                            int strong, DevCounters* __restrict__ ctr,
                                            unsigned char* smem_raw,
                                            unsigned char* __restrict__ uslices = nullptr,
                                            int* abort_word = nullptr, int* skip_out = nullptr) {
    window_body_t<WMAX>(n, S, ldS, s0, w, gsel, Ug, strong, ctr, smem_raw, uslices, abort_word,
                        skip_out, nullptr);
}

}  // namespace win
}  // namespace gbr
