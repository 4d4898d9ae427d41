// cg_device.cuh -- device helpers of the finite-difference flow-map gradient and the
// largest eigenvalue of the Cauchy-Green tensor (Eq. 1; Sec. 2 "Cauchy-Green"), shared by
// the regular pass (cg_ftle.cu) and the early evaluation (early_cg.cu).
#pragma once
#include "dfloat_device.cuh"
#include "lcs_internal.cuh"

#include <math.h>

__device__ __forceinline__ long long lattice_nbr(const CgLaunch &L, const long long *idx, int b, int off, int *wrap)
{
    long long c[3] = {idx[0], idx[1], idx[2]};
    long long v = c[b] + off;
    *wrap = 0;
    int nb = L.n[b];
    if (L.periodic[b]) {
        if (v < 0) {
            v += nb;
            *wrap = -1;
        } else if (v >= nb) {
            v -= nb;
            *wrap = 1;
        }
    } else if (v < 0 || v >= nb) {
        return -1;
    }
    c[b] = v;
    return c[0] + (long long)L.n[0] * (c[1] + (long long)L.n[1] * c[2]);
}

// RN(x / d) for a fixed divisor d.  FP64 issue limits this pass, so the divisor's quotient takes two
// operations where launch_cg's exhaustive check of the divisor (fixed_divisor_exact) allows it: with
// y + yl = 1/d to 105 bits, yl <= 0, RN(x y + RN(x yl)) is the correctly rounded quotient unless x/d
// lies within about 2^-104 of a midpoint of two FP64 values (Brisebarre & Muller 2008).  Otherwise
// with y = RN(1 / d) alone: q = RN(x y) is within about one ulp of x / d, one FMA-corrected step
// makes it faithful, so the remainder x - q1 d is exact, and RN(q1 + (x - q1 d) y) is the correctly
// rounded quotient (Markstein 1990, Theorem 8).  No overflow or underflow occurs for lattice
// spacings and flow-map differences.  An infinite x gives NaN either way (yl <= 0).
__device__ __forceinline__ double div_fixed(const CgLaunch &L, int b, double x)
{
    const double y = L.rh2[b];
    if (L.div2) return __fma_rn(x, y, __dmul_rn(x, L.rl2[b]));
    const double d = L.h2[b], q = __dmul_rn(x, y);
    const double q1 = __fma_rn(__fma_rn(-q, d, x), y, q);
    return __fma_rn(__fma_rn(-q1, d, x), y, q1);
}

// (double)x without the FP64 pipe's conversion (which issues at the FP64 rate) for a normal x
__device__ __forceinline__ double widen(float x)
{
    const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
    if (e - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
    return (double)x;
}

// neighbour position with the periodic shift of axis b (a == b only; w in {-1, 0, 1})
__device__ __forceinline__ double nbr_pos(float x, int w, double sh, bool shifted)
{
    double v = widen(x);
    if (shifted && w != 0) v = __dadd_rn(v, w > 0 ? sh : -sh);
    return v;
}

__device__ __forceinline__ double eig_max2(const double *C)
{
    // C = [[a, b], [b, c]]: lambda_max = (a + c)/2 + sqrt(((a - c)/2)^2 + b^2)
    double a = C[0], b = C[1], c = C[2];
    double m = __dmul_rn(0.5, __dadd_rn(a, c));
    double d = __dmul_rn(0.5, __dsub_rn(a, c));
    return __dadd_rn(m, sqrt(__dadd_rn(__dmul_rn(d, d), __dmul_rn(b, b))));
}

// ln(lambda_max) in FP32 from the FP64 eigenvalue, for sigma = ln(sqrt(lambda_max)) / |T|: near
// lambda_max = 1 as log1p of the FP64 difference lambda_max - 1 (which keeps its relative
// accuracy where sigma is near 0), elsewhere as log of the rounded eigenvalue (log1p of a
// rounded lambda_max - 1 close to -1 would lose digits: a contracting map, lambda_max << 1)
__device__ __forceinline__ float log_lambda(double lm)
{
    const double d = lm - 1.0;
    return fabs(d) < 0.5 ? log1pf((float)d) : logf((float)lm);
}

// All eigenpairs of the packed symmetric C by cyclic Jacobi rotations in FP64.  Each
// rotation zeroes a_pq with t = tan(theta) the smaller root of t^2 + 2 tau t - 1 = 0,
// tau = (a_qq - a_pp) / (2 a_pq), updates the diagonal as a_pp - t a_pq and a_qq + t a_pq
// (Rutishauser's form), rotates the other row of the pair and accumulates V <- V J.  A pair
// counts as converged when |a_pq| <= 1e-18 sqrt(|a_pp a_qq|), a relative test that keeps
// the small eigenvalues of a graded C accurate; at most 16 sweeps.  Ascending order, each
// eigenvector with its largest-magnitude component positive.
template <int DIM>
__device__ __forceinline__ void eig_jacobi(const double *Cp, double *ev, double *V)
{
    double A[DIM][DIM];
    int o = 0;
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int j = i; j < DIM; ++j) {
            A[i][j] = Cp[o];
            A[j][i] = Cp[o];
            ++o;
        }
    double W[DIM][DIM];
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int j = 0; j < DIM; ++j) W[i][j] = i == j ? 1.0 : 0.0;
    bool bad = false;
#pragma unroll
    for (int i = 0; i < DIM * (DIM + 1) / 2; ++i) bad |= isnan(Cp[i]);
    for (int sweep = 0; sweep < 16 && !bad; ++sweep) {
        bool rotated = false;
#pragma unroll
        for (int p = 0; p < DIM - 1; ++p)
#pragma unroll
            for (int q = p + 1; q < DIM; ++q) {
                const double apq = A[p][q];
                if (!(fabs(apq) > 1e-18 * sqrt(fabs(A[p][p] * A[q][q])))) continue;
                rotated = true;
                const double tau = (A[q][q] - A[p][p]) / (2.0 * apq);
                const double t = copysign(1.0, tau) / (fabs(tau) + sqrt(fma(tau, tau, 1.0)));
                const double c = rsqrt(fma(t, t, 1.0)), s = t * c;
                A[p][p] = fma(-t, apq, A[p][p]);
                A[q][q] = fma(t, apq, A[q][q]);
                A[p][q] = A[q][p] = 0.0;
#pragma unroll
                for (int r = 0; r < DIM; ++r) {
                    if (r == p || r == q) continue;
                    const double arp = A[r][p], arq = A[r][q];
                    A[r][p] = A[p][r] = c * arp - s * arq;
                    A[r][q] = A[q][r] = s * arp + c * arq;
                }
#pragma unroll
                for (int r = 0; r < DIM; ++r) {
                    const double wp = W[r][p], wq = W[r][q];
                    W[r][p] = c * wp - s * wq;
                    W[r][q] = s * wp + c * wq;
                }
            }
        if (!rotated) break;
    }
    int ord[DIM];
#pragma unroll
    for (int i = 0; i < DIM; ++i) ord[i] = i;
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int j = i + 1; j < DIM; ++j)
            if (A[ord[j]][ord[j]] < A[ord[i]][ord[i]]) {
                const int t = ord[i];
                ord[i] = ord[j];
                ord[j] = t;
            }
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        int m = 0;
#pragma unroll
        for (int r = 1; r < DIM; ++r)
            if (fabs(W[r][ord[k]]) > fabs(W[m][ord[k]])) m = r;
        const double sg = W[m][ord[k]] < 0.0 ? -1.0 : 1.0;
        ev[k] = bad ? nan : A[ord[k]][ord[k]];
#pragma unroll
        for (int r = 0; r < DIM; ++r) V[k * DIM + r] = bad ? nan : sg * W[r][ord[k]];
    }
}

// lambda_max by the Jacobi rotations above: matrices outside the scaled range of eig_max3, and
// those whose two largest eigenvalues (nearly) coincide, where no root of the characteristic
// cubic is accurate in FP64 (see eig_max3).  Out of line: rare, and it keeps eig_max3 small.
static __device__ __noinline__ double eig_max3_jacobi(const double *C)
{
    double ev[3], V[9];
    eig_jacobi<3>(C, ev, V);
    return ev[2];
}

__device__ __forceinline__ double eig_max3(const double *C)
{
    const double dmax = fmax(C[0], fmax(C[3], C[5]));
    const double p1 = C[1] * C[1] + C[2] * C[2] + C[4] * C[4];
    if (p1 == 0.0) return dmax;  // diagonal (or NaN, which fmax passes on only if all are NaN)
    // scale by a power of two s so that the largest diagonal entry lies in [1, 2): exact, and it
    // keeps the FP32 steps below in range.  C is positive semidefinite, so dmax > 0 here.
    const int hi = __double2hiint(dmax);
    const int ex = ((hi >> 20) & 0x7ff) - 1023;
    if (!(dmax > 0.0) || ex < -1000 || ex > 1000) return eig_max3_jacobi(C);
    const double s = __hiloint2double((1023 - ex) << 20, 0), is = __hiloint2double((1023 + ex) << 20, 0);
    const double a00 = C[0] * s, a01 = C[1] * s, a02 = C[2] * s, a11 = C[3] * s, a12 = C[4] * s, a22 = C[5] * s;
    const double q = (a00 + a11 + a22) * (1.0 / 3.0);
    const double b00 = a00 - q, b11 = a11 - q, b22 = a22 - q;
    const double p2 = (b00 * b00 + b11 * b11 + b22 * b22 + 2.0 * (p1 * s * s)) * (1.0 / 6.0);
    // eigenvalues are q + 2 p cos(.), p = sqrt(p2) and q >= 1/3: below 1e-28, lambda_max = q to 1e-13
    if (!(p2 >= 1e-28)) return p2 < 1e-28 ? q * is : eig_max3_jacobi(C);
    // y = 1/sqrt(p2): FP32 estimate, two FP64 Newton steps (relative error 1e-7 -> 1e-14 -> 1e-16)
    double y = (double)rsqrtf((float)p2);
    y = y * (1.5 - 0.5 * p2 * y * y);
    y = y * (1.5 - 0.5 * p2 * y * y);
    const double p = p2 * y;
    // r = det((C - qI) / p) / 2 in [-1, 1]; beta = 2 cos(acos(r) / 3) is the largest root of
    // beta^3 - 3 beta - 2 r = 0
    const double det = b00 * (b11 * b22 - a12 * a12) - a01 * (a01 * b22 - a12 * a02) + a02 * (a01 * a12 - b11 * a02);
    const double r = fmin(fmax(0.5 * det * (y * y * y), -1.0), 1.0);
    // r = -1 is a double largest root (beta = 1, lambda_1 = lambda_2).  Near it, with r = -1 + d,
    // the root sits at 1 + sqrt(2 d / 3) + ..., so an error of one ulp in r or in the cubic's value
    // moves it by about the square root of an ulp (1e-8 relative to lambda_max) whatever the
    // polish.  Below 1 + r = 1e-3 (a gap lambda_1 - lambda_2 under about 5% of p) the Jacobi
    // rotations, which are backward stable, give lambda_max instead; above it two Newton steps
    // from the FP32 root reach ~1e-14 relative (f' = 3 (beta^2 - 1) >= 0.15 there).  NaN
    // entries also end up here (fmax and fmin pass -1), and Jacobi returns NaN for them.
    if (!(r >= -1.0 + 1e-3)) return eig_max3_jacobi(C);
    double beta = (double)(2.0f * cosf(acosf((float)r) * (1.0f / 3.0f)));
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        const double f = fma(beta, fma(beta, beta, -3.0), -2.0 * r);
        const double fp = 3.0 * fma(beta, beta, -1.0);
        beta -= f * (double)__frcp_rn((float)fp);
    }
    return (q + p * beta) * is;
}

// ------------------------------------------------ eigenpairs of 3x3 C, split

// v / 2^ex in double-FP32, from v's bits (no FP64 instructions): zero where below the FP32 range
__device__ __forceinline__ dfl narrow_scaled(double v, int ex)
{
    const int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v);
    const int e = ((hi >> 20) & 0x7ff) - 1023 + 127 - ex;   // biased FP32 exponent
    if (e <= 0 || e >= 255) return {0.0f, 0.0f};
    const unsigned sg = (unsigned)hi & 0x80000000u;
    const float h = __uint_as_float(sg | ((unsigned)e << 23) | (((unsigned)hi & 0xfffffu) << 3) | (lo >> 29));
    const float r = (float)(lo & 0x1fffffffu);              // the bits below: r 2^(e - 127 - 52)
    const float l = e > 52 ? r * __uint_as_float((unsigned)(e - 52) << 23) : 0.0f;
    return {h, sg ? -l : l};
}

__device__ __forceinline__ double widen(dfl a) { return __dadd_rn(widen(a.h), widen(a.l)); }

// 1 / sqrt(a) for a >= 1
__device__ __forceinline__ dfl df_rsqrt(dfl a)
{
    const float y = rsqrtf(a.h);
    const dfl u = df_mul(a, df_two_prod(y, y));
    const float e = __fsub_rn(__fsub_rn(1.0f, u.h), u.l);
    return df_fast_sum(y, __fmul_rn(y, __fmaf_rn(__fmul_rn(0.375f, e), e, __fmul_rn(0.5f, e))));
}

// tangent of the Jacobi rotation that annihilates apq, d = aqq - app: the smaller root of t^2 + 2 tau t = 1
__device__ __forceinline__ float jacobi_tan(float d, float apq)
{
    const float tau = __fdividef(d, 2.0f * apq);
    const float t = __fdividef(1.0f, fabsf(tau) + sqrtf(fmaf(tau, tau, 1.0f)));
    return apq == 0.0f ? 0.0f : (fabsf(tau) < 1e18f ? copysignf(t, tau) : __fdividef(0.5f, tau));
}

// All eigenpairs of the packed 3x3 C by Jacobi rotations whose FP64 work is the part that needs it:
//  1. four sweeps on C / 2^ex in FP32, the rotations multiplied up as a quaternion (so the matrix V it
//     stands for is orthonormal to whatever precision V is formed in), which diagonalise C to about 1e-7;
//  2. V and A = V^T C V in FP64;
//  3. the rotations left, in double-FP32: their product as R' = R - I and the changes of A's diagonal as
//     sums of their own, so that both carry 2^-46 of a small quantity.  With t a rotation's tangent and a'
//     the off-diagonal element it leaves, app' = app - t (apq + a') exactly, whatever the rounding of t;
//  4. eigenvalues A_kk + changes and vectors V + V R' in FP64.
// About 185 FP64 operations against 950 for Jacobi rotations in FP64 throughout (eig_jacobi, which serves
// matrices outside the exponent range here, and 2x2 ones).  Same order and signs as eig_jacobi.
// A graded C (rows and columns of different sizes) has small eigenvalues that FP64 rotations give to 2 to 3 u k,
// k the condition number of C scaled to a unit diagonal and u = 2^-53, and this to 3 to 5 u k while the double-FP32
// values of C / 2^ex keep their low halves: down to diagonals of 2^-86 of the largest; at 2^-93 it is 12 u k, at
// 2^-100 78 u k (200,000 matrices each).  Below 2^-80 the FP64 rotations take C.
__device__ __forceinline__ bool eig3_split(const double *C, double *ev, double *Vout)
{
    const double dmax = fmax(C[0], fmax(C[3], C[5]));
    const int ex = ((__double2hiint(dmax) >> 20) & 0x7ff) - 1023;
    const int least = min(__double2hiint(C[0]), min(__double2hiint(C[3]), __double2hiint(C[5])));
    bool fine = dmax > 0.0 && ex > -900 && ex < 900 && least >= __double2hiint(dmax) - (80 << 20);
#pragma unroll
    for (int i = 0; i < 6; ++i) fine = fine && fabs(C[i]) <= 2.0 * dmax;   // false for NaN
    if (!fine) return false;
    // 1. FP32
    float a[3][3], w = 1.0f, q[3] = {0.0f, 0.0f, 0.0f};
    {
        const int at[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) a[i][j] = narrow_scaled(C[at[i][j]], ex).h;
    }
#pragma unroll 1
    for (int sweep = 0; sweep < 4; ++sweep) {
#pragma unroll
        for (int k = 2; k >= 0; --k) {          // rotation about axis k: planes (0, 1), (0, 2), (1, 2)
            const int p = k == 0 ? 1 : 0, r = k == 2 ? 1 : 2, o = k;
            const float apq = a[p][r], t = jacobi_tan(a[r][r] - a[p][p], apq);
            const float c = rsqrtf(fmaf(t, t, 1.0f)), s = t * c;
            a[p][p] = fmaf(-t, apq, a[p][p]);
            a[r][r] = fmaf(t, apq, a[r][r]);
            a[p][r] = a[r][p] = 0.0f;
            const float x = a[o][p], y = a[o][r];
            a[o][p] = a[p][o] = c * x - s * y;
            a[o][r] = a[r][o] = s * x + c * y;
            // V <- V J: J[p][r] = s is the rotation by -theta about x and z, by +theta about y; its
            // quaternion is (1 + c, -+s e_k) up to scale
            const float jw = 0.5f + 0.5f * c, js = (k == 1 ? 0.5f : -0.5f) * s;
            const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
            const float nw = jw * w - js * q[k], nk = jw * q[k] + js * w;
            const float n1 = jw * q[k1] + js * q[k2], n2 = jw * q[k2] - js * q[k1];
            w = nw;
            q[k] = nk;
            q[k1] = n1;
            q[k2] = n2;
        }
    }
    const float nq = rsqrtf(w * w + q[0] * q[0] + q[1] * q[1] + q[2] * q[2]);
    // 2. V and A in FP64
    double V[3][3], A[3][3];
    {
        const double W = widen(w * nq), X = widen(q[0] * nq), Y = widen(q[1] * nq), Z = widen(q[2] * nq);
        const double xx = X * X, yy = Y * Y, zz = Z * Z;
        const double n1 = (W * W - 1.0) + xx + (yy + zz);                  // |q|^2 - 1, of order 1e-7
        const double s = 2.0 * fma(-n1, fma(-n1, 1.0 - n1, 1.0), 1.0);     // 2 / |q|^2
        const double sX = s * X, sY = s * Y, sZ = s * Z;
        const double xy = sX * Y, xz = sX * Z, yz = sY * Z, wx = sX * W, wy = sY * W, wz = sZ * W;
        V[0][0] = fma(-s, yy + zz, 1.0);
        V[1][1] = fma(-s, xx + zz, 1.0);
        V[2][2] = fma(-s, xx + yy, 1.0);
        V[0][1] = xy - wz;
        V[1][0] = xy + wz;
        V[0][2] = xz + wy;
        V[2][0] = xz - wy;
        V[1][2] = yz - wx;
        V[2][1] = yz + wx;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double w0 = fma(C[0], V[0][j], fma(C[1], V[1][j], C[2] * V[2][j]));
            const double w1 = fma(C[1], V[0][j], fma(C[3], V[1][j], C[4] * V[2][j]));
            const double w2 = fma(C[2], V[0][j], fma(C[4], V[1][j], C[5] * V[2][j]));
#pragma unroll
            for (int i = 0; i <= j; ++i) A[i][j] = fma(V[0][i], w0, fma(V[1][i], w1, V[2][i] * w2));
        }
    }
    // 3. the rotations left
    dfl R[3][3], dg[3], d[3], od[3];      // R', diagonal, its changes, off-diagonal opposite axis k
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dg[i] = narrow_scaled(A[i][i], ex);
        d[i] = {0.0f, 0.0f};
#pragma unroll
        for (int j = 0; j < 3; ++j) R[i][j] = {0.0f, 0.0f};
    }
    od[0] = narrow_scaled(A[1][2], ex);
    od[1] = narrow_scaled(A[0][2], ex);
    od[2] = narrow_scaled(A[0][1], ex);
    float widest = 0.0f, most = 1.0f;
#pragma unroll 1
    for (int sweep = 0; sweep < 8; ++sweep) {
        most = 0.0f;
#pragma unroll
        for (int k = 2; k >= 0; --k) {
            const int p = k == 0 ? 1 : 0, r = k == 2 ? 1 : 2;
            const dfl diff = df_add(df_sub(dg[r], dg[p]), df_sub(d[r], d[p]));
            const float t = jacobi_tan(diff.h, od[k].h);
            most = fmaxf(most, fabsf(t));
            const dfl t2 = df_two_prod(t, t), c = df_rsqrt(df_add(t2, 1.0f)), s = df_mul(c, t);
            const dfl c2 = df_mul(c, c);
            // c - 1 = -t^2 c^2 / (1 + c), of full relative accuracy
            const dfl num = df_mul(t2, c2), den = df_add(c, 1.0f);
            const float q0 = __fdividef(num.h, den.h);
            const dfl rem = df_sub(num, df_mul(den, q0));
            const dfl cm1 = df_neg(df_fast_sum(q0, __fdividef(rem.h, den.h)));
            const dfl left = df_mul(c2, df_sub(df_sub(od[k], df_mul(t2, od[k])), df_mul(diff, t)));
            const dfl g = df_mul(df_add(od[k], left), t);
            d[p] = df_sub(d[p], g);
            d[r] = df_add(d[r], g);
            od[k] = left;
            // a[k][p] is the element opposite axis r, a[k][r] the one opposite p
            const dfl x = od[r], y = od[p];
            od[r] = df_sub(df_mul(c, x), df_mul(s, y));
            od[p] = df_add(df_mul(s, x), df_mul(c, y));
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const dfl u = R[i][p], v = R[i][r];
                dfl nu = df_sub(df_add(u, df_mul(cm1, u)), df_mul(s, v));
                dfl nv = df_add(df_add(v, df_mul(cm1, v)), df_mul(s, u));
                if (i == p) {
                    nu = df_add(nu, cm1);
                    nv = df_add(nv, s);
                }
                if (i == r) {
                    nu = df_sub(nu, s);
                    nv = df_add(nv, cm1);
                }
                R[i][p] = nu;
                R[i][r] = nv;
            }
        }
        widest = fmaxf(widest, most);
        if (most < 0x1p-40f) break;   // what is left is of second order in these
    }
    if (!(most < 0x1p-40f)) return false;   // not settled (six sweeps were the most that any of 2.8M matrices took)
    // 4. FP64, in ascending order
    const double scale = __hiloint2double((1023 + ex) << 20, 0);
    double e[3], U[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        e[k] = fma(widen(d[k]), scale, A[k][k]);
        const double r0 = widen(R[0][k]), r1 = widen(R[1][k]), r2 = widen(R[2][k]);
#pragma unroll
        for (int i = 0; i < 3; ++i) U[k][i] = fma(V[i][0], r0, fma(V[i][1], r1, fma(V[i][2], r2, V[i][k])));
    }
    // eigenvalues so near one another that FP32 did not part them leave wide rotations, whose 2^-46 shows in
    // FP64: one symmetric orthonormalisation, the Rayleigh quotients and the vectors' first-order correction
    if (widest > 0x1p-12f) {
        double S[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                S[i][j] = -0.5 * fma(U[i][0], U[j][0], fma(U[i][1], U[j][1], fma(U[i][2], U[j][2], i == j ? -1.0 : 0.0)));
                S[j][i] = S[i][j];
            }
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const double u0 = U[0][r], u1 = U[1][r], u2 = U[2][r];
#pragma unroll
            for (int i = 0; i < 3; ++i) U[i][r] = fma(S[i][0], u0, fma(S[i][1], u1, fma(S[i][2], u2, U[i][r])));
        }
        double w[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            w[k][0] = fma(C[0], U[k][0], fma(C[1], U[k][1], C[2] * U[k][2]));
            w[k][1] = fma(C[1], U[k][0], fma(C[3], U[k][1], C[4] * U[k][2]));
            w[k][2] = fma(C[2], U[k][0], fma(C[4], U[k][1], C[5] * U[k][2]));
            e[k] = fma(U[k][0], w[k][0], fma(U[k][1], w[k][1], U[k][2] * w[k][2]));
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = i + 1; j < 3; ++j) {
                const double aij = fma(U[i][0], w[j][0], fma(U[i][1], w[j][1], U[i][2] * w[j][2]));
                const float den = narrow_scaled(e[i] - e[j], ex).h, t = __fdividef(narrow_scaled(aij, ex).h, den);
                if (den != 0.0f && fabsf(t) < 0x1p-14f) {
                    const double td = widen(t), cm1 = -0.5 * td * td;   // 1 - cos to t^4
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const double u = U[i][r], v = U[j][r];
                        U[i][r] = u + fma(td, v, cm1 * u);
                        U[j][r] = v + fma(-td, u, cm1 * v);
                    }
                }
            }
    }
    const auto order = [&](int i, int j) {
        if (e[j] < e[i]) {
            double x = e[i];
            e[i] = e[j];
            e[j] = x;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                x = U[i][r];
                U[i][r] = U[j][r];
                U[j][r] = x;
            }
        }
    };
    order(0, 1);
    order(0, 2);
    order(1, 2);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double m = U[k][0];
        if (fabs(U[k][1]) > fabs(m)) m = U[k][1];
        if (fabs(U[k][2]) > fabs(m)) m = U[k][2];
        ev[k] = e[k];
#pragma unroll
        for (int r = 0; r < 3; ++r) Vout[k * 3 + r] = m < 0.0 ? -U[k][r] : U[k][r];
    }
    return true;
}

// matrices that eig3_split does not take: NaN, zero, extreme exponents, strong grading, rotations left unsettled
static __device__ __noinline__ void eig3_jacobi(const double *C, double *ev, double *V) { eig_jacobi<3>(C, ev, V); }

// ------------------------------------------------------- differences and FTLE

// one axis of a seed's differences: mode 1 central (F1 - F2) / 2h, 2 forward (-3 F0 + 4 F1 - F2) / 2h,
// 3 backward (3 F0 - 4 F1 + F2) / 2h, 0 none (NaN); w1, w2: periods crossed by the two other points
struct AxisDiff {
    int mode, w1, w2;
};

// the quotient in FP64: every operation round-to-nearest, none contracted (the plain definition's bits)
__device__ __forceinline__ double axis_grad64(const CgLaunch &L, int b, const AxisDiff &d, bool on, float f0, float f1,
                                              float f2)
{
    if (d.mode == 0) return __longlong_as_double(0x7ff8000000000000LL);
    const double sh = L.period[b], F1 = nbr_pos(f1, d.w1, sh, on), F2 = nbr_pos(f2, d.w2, sh, on);
    double x;
    if (d.mode == 1) {
        x = __dsub_rn(F1, F2);
    } else {
        const double F0 = widen(f0);
        x = d.mode == 2 ? __dsub_rn(__dadd_rn(__dmul_rn(-3.0, F0), __dmul_rn(4.0, F1)), F2)
                        : __dadd_rn(__dsub_rn(__dmul_rn(3.0, F0), __dmul_rn(4.0, F1)), F2);
    }
    return div_fixed(L, b, x);
}

// the same quotient in double-FP32: the differences of FP32 positions are exact there
__device__ __forceinline__ dfl axis_grad32(const CgLaunch &L, int b, const AxisDiff &d, bool on, float f0, float f1,
                                           float f2)
{
    if (d.mode == 0) return {__int_as_float(0x7fc00000), 0.0f};
    dfl x;
    int k = d.w1 - d.w2;
    if (d.mode == 1) {
        x = df_two_sum(f1, -f2);
    } else {
        x = df_add(df_add(df_two_prod(-3.0f, f0), 4.0f * f1), -f2);
        k = 4 * d.w1 - d.w2;
        if (d.mode == 3) {
            x = df_neg(x);
            k = -k;
        }
    }
    if (on && k != 0) x = df_add(x, df_mul(dfl{L.psh[b], L.psl[b]}, (float)k));
    return df_mul(x, dfl{L.rhf[b], L.rlf[b]});
}

// C = grad F^T grad F (Eq. 1) in FP64, packed upper triangle row by row, round-to-nearest products
// and sums in the order of a
template <int DIM>
__device__ __forceinline__ void cauchy_green64(const double (*G)[DIM], double *C)
{
    int o = 0;
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int j = i; j < DIM; ++j) {
            // the sum starts from +0.0, which only matters for an off-diagonal sum of negative zeros
            double s = __dmul_rn(G[0][i], G[0][j]);
            if (i != j) s = __dadd_rn(0.0, s);
#pragma unroll
            for (int a = 1; a < DIM; ++a) s = __dadd_rn(s, __dmul_rn(G[a][i], G[a][j]));
            C[o++] = s;
        }
}

template <int DIM>
static __device__ __noinline__ float ftle_from_c64(const double *C, float half_inv_T)
{
    return log_lambda(DIM == 2 ? eig_max2(C) : eig_max3(C)) * half_inv_T;
}

// sigma = ln(lambda_max(G^T G)) * half_inv_T with G in double-FP32 (its entries' magnitudes between
// 2^-40 and 2^40 at the largest: nothing below then leaves the FP32 range); false where sigma needs FP64
template <int DIM>
__device__ __forceinline__ bool ftle_from_grad32(const dfl (*G)[DIM], float half_inv_T, float *sigma)
{
    constexpr int NP = DIM == 2 ? 3 : 6;
    dfl C[NP];
    int o = 0;
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int j = i; j < DIM; ++j) {
            dfl s = df_mul(G[0][i], G[0][j]);
#pragma unroll
            for (int a = 1; a < DIM; ++a) s = df_add(s, df_mul(G[a][i], G[a][j]));
            C[o++] = s;
        }
    float gap = 1.0f, ln;
    if constexpr (DIM == 2)
        ln = df_log(df_eig_max2(C));
    else
        ln = df_log(df_eig_max3(C, &gap));
    *sigma = ln * half_inv_T;
    return fabsf(ln) * gap >= 0x1p-14f;   // 2^-44 / gap of lambda_max is at most 2^-30 of its logarithm
}

// whether G's largest entry lies where ftle_from_grad32 is safe (false for NaN and infinite entries)
template <int DIM>
__device__ __forceinline__ bool grad32_in_range(const dfl (*G)[DIM])
{
    float m = 0.0f;
    bool nan = false;
#pragma unroll
    for (int a = 0; a < DIM; ++a)
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
            m = fmaxf(m, fabsf(G[a][b].h));
            nan |= isnan(G[a][b].h);
        }
    return !nan && m >= 0x1p-40f && m <= 0x1p40f;
}

// FTLE of a seed from its positions f[b][k][a] (axis b, point k = 0 the seed, 1 and 2 the two others,
// component a) in double-FP32, in FP64 where grad F lies outside the safe range or sigma needs it
template <int DIM>
__device__ __forceinline__ float ftle_from_positions(const CgLaunch &L, const AxisDiff *d, const float *f0,
                                                     const float (*f1)[DIM], const float (*f2)[DIM], float half_inv_T)
{
    dfl G[DIM][DIM];
#pragma unroll
    for (int b = 0; b < DIM; ++b)
#pragma unroll
        for (int a = 0; a < DIM; ++a) G[a][b] = axis_grad32(L, b, d[b], a == b, f0[a], f1[b][a], f2[b][a]);
    bool none = false;   // an axis without differences: NaN whatever the others hold
#pragma unroll
    for (int b = 0; b < DIM; ++b) none |= d[b].mode == 0;
    if (none) return __int_as_float(0x7fc00000);
    float sigma;
    if (L.df_ok && grad32_in_range<DIM>(G) && ftle_from_grad32<DIM>(G, half_inv_T, &sigma)) return sigma;
    double G64[DIM][DIM], C[DIM == 2 ? 3 : 6];
#pragma unroll
    for (int b = 0; b < DIM; ++b)
#pragma unroll
        for (int a = 0; a < DIM; ++a) G64[a][b] = axis_grad64(L, b, d[b], a == b, f0[a], f1[b][a], f2[b][a]);
    cauchy_green64<DIM>(G64, C);
    return ftle_from_c64<DIM>(C, half_inv_T);
}
