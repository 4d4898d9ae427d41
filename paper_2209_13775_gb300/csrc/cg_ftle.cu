// cg_ftle.cu -- flow-map gradient, Cauchy-Green tensor, largest eigenvalue, FTLE.
//
// Paper: Eq. 1, C = grad(F)^T grad(F); Sec. 2 "Cauchy-Green": grad F from
// central differences of the final seed positions over the seed lattice, then
// the eigenvalues of C; Sec. 1: the FTLE is derived from the largest one,
// sigma = ln(sqrt(lambda_max)) / |T|.
//
// One thread per seed.  GB300 has two FP64 lanes per SM against 128 FP32 ones, so FP64 issue bounds
// whatever stays in FP64 (ncu: the FP64 pipe 85% busy, issue 14%, when all of it did):
//  * C, lambda_max and the eigenpairs, where asked for: every difference, product and sum of grad F and
//    C is a round-to-nearest FP64 operation without contraction and the division by 2h is correctly
//    rounded (div_fixed: two operations), so both equal the plain FP64 definition bit for bit.
//    lambda_max: 2x2 from the quadratic formula; 3x3 from the characteristic cubic of the shifted,
//    scaled matrix (Smith 1961), whose trigonometric root is taken in FP32 and polished by two FP64
//    Newton steps, and by Jacobi rotations where the two largest eigenvalues (nearly) coincide.  The
//    eigenpairs of a 3x3 C take FP64 for a fifth of their operations (eig3_split): 160^3 seeds 6.23 ->
//    2.12 ms at three blocks per SM (2.25 ms at two), the FP64 pipe 82% busy;
//  * the FTLE, an FP32 output: the same formulas in double-FP32 (dfloat_device.cuh), about 200 FP32
//    operations per seed in 2D and 700 in 3D in place of 65 and 170 FP64 ones, whether or not C or
//    lambda_max is asked for (one call's FTLE does not depend on its other outputs).  Auxiliary
//    points keep FP64 (their divisor is another one at every seed).
// Measured: 64 windows of 2048 x 1024 seeds, FTLE only, advection and differences 95.3 -> 79.7 ms (the
// differences 17.6 -> 2.0); 256^3 seeds with C written, 6.0 -> 2.8 ms (57 FP64 operations per seed
// left of 170: 1.5 ms of FP64 issue).
#include "lcs_internal.cuh"

#include <math.h>

#include "cg_device.cuh"

// grad F of lattice seed p from its 2 DIM auxiliary points (lcs_seed_aux): per axis b the
// difference of the two points' final positions over that of their FP32 starting points,
// RN operations in FP64; NaN unless every point is OK
template <int DIM>
__device__ __forceinline__ void aux_gradient(const CgLaunch &L, int job, long long p, double (*G)[DIM])
{
    const long long M = L.npts;
    const float *X = L.xyz + (size_t)job * DIM * M;
    const unsigned char *S = L.status + (size_t)job * M;
    bool ok = true;
#pragma unroll
    for (int q = 0; q < 2 * DIM; ++q) ok &= S[p * 2 * DIM + q] == LCS_TRACER_OK;
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
    for (int b = 0; b < DIM; ++b) {
        const long long i0 = (p * DIM + b) * 2, i1 = i0 + 1;
        const double den = __dsub_rn((double)L.x0aux[b * M + i0], (double)L.x0aux[b * M + i1]);
#pragma unroll
        for (int a = 0; a < DIM; ++a)
            G[a][b] = ok ? __ddiv_rn(__dsub_rn((double)X[a * M + i0], (double)X[a * M + i1]), den) : nan;
    }
}

// gradient sources: finite differences over the lattice, over auxiliary points, or the
// variational grad F integrated with the flow map
enum { GM_LATTICE = 0, GM_AUX = 1, GM_VAR = 2 };

// The difference rule of axis b at lattice seed p (coordinate c along it, neighbours `stride` apart) and
// the ids of its two other points: central, else forward, else backward, from seeds with status OK only.
// The points two steps away are looked at only where the central difference does not exist.
__device__ __forceinline__ AxisDiff axis_diff(const CgLaunch &L, const unsigned char *__restrict__ S, long long p, int c,
                                              int b, long long stride, bool valid, long long *q1, long long *q2)
{
    const int n = L.n[b];
    const bool per = L.periodic[b] != 0;
    const long long span = stride * n;
    AxisDiff d = {0, 0, 0};
    *q1 = *q2 = p;
    if (!valid) return d;
    const int wp = per && c + 1 >= n ? 1 : 0, wm = per && c < 1 ? -1 : 0;
    const long long p1 = p + stride - wp * span, m1 = p - stride - wm * span;
    const bool okp = (per || c + 1 < n) && S[p1] == LCS_TRACER_OK, okm = (per || c >= 1) && S[m1] == LCS_TRACER_OK;
    if (okp && okm) {
        d = {1, wp, wm};
        *q1 = p1;
        *q2 = m1;
        return d;
    }
    if (okp) {
        const int w = per && c + 2 >= n ? 1 : 0;
        const long long p2 = p + 2 * stride - w * span;
        if ((per || c + 2 < n) && S[p2] == LCS_TRACER_OK) {
            d = {2, wp, w};
            *q1 = p1;
            *q2 = p2;
        }
    } else if (okm) {
        const int w = per && c < 2 ? -1 : 0;
        const long long m2 = p - 2 * stride - w * span;
        if ((per || c >= 2) && S[m2] == LCS_TRACER_OK) {
            d = {3, wm, w};
            *q1 = m1;
            *q2 = m2;
        }
    }
    return d;
}

// F64: C, lambda_max or eigenpairs wanted (EIG: the latter), so grad F and C are formed in FP64 as well
// The FTLE alone: four blocks per SM (64 registers; the positions stay live for the seeds that need FP64, which
// would take 80 and leave three blocks: DP5(4) on 2.1M seeds with its FTLE, 3.295 -> 3.283 ms).
template <int DIM, bool F64, bool EIG, int GM>
__global__ void __launch_bounds__(256, EIG ? 3 : F64 ? 1 : 4) cg_ftle_kernel(const __grid_constant__ CgLaunch L)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int jr = blockIdx.y;        // job relative to job0
    const int job = L.job0 + jr;
    const long long N = L.N;
    if (p >= N) return;
    constexpr int NP = DIM == 2 ? 3 : 6;
    const size_t out = (size_t)jr * N + p;
    const float half_inv_T = L.ftle ? 0.5f / (float)L.absT[job] : 0.0f;   // sigma = ln(lambda) / (2 |T|)
    double G[DIM][DIM];
    if constexpr (GM == GM_AUX) {
        aux_gradient<DIM>(L, job, p, G);
    } else if constexpr (GM == GM_VAR) {
        const bool ok = L.status[(size_t)job * N + p] == LCS_TRACER_OK;
        const float *Mp = L.grad + ((size_t)job * N + p) * DIM * DIM;
        float M[DIM][DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
            for (int b = 0; b < DIM; ++b) M[a][b] = ok ? Mp[a * DIM + b] : __int_as_float(0x7fc00000);
        if (!EIG && L.ftle) {
            dfl Gf[DIM][DIM];
#pragma unroll
            for (int a = 0; a < DIM; ++a)
#pragma unroll
                for (int b = 0; b < DIM; ++b) Gf[a][b] = {M[a][b], 0.0f};
            float s = __int_as_float(0x7fc00000);
            if (ok && !(grad32_in_range<DIM>(Gf) && ftle_from_grad32<DIM>(Gf, half_inv_T, &s))) {
                double C[NP];
#pragma unroll
                for (int a = 0; a < DIM; ++a)
#pragma unroll
                    for (int b = 0; b < DIM; ++b) G[a][b] = (double)M[a][b];
                cauchy_green64<DIM>(G, C);
                s = ftle_from_c64<DIM>(C, half_inv_T);
            }
            L.ftle[out] = s;
        }
        if constexpr (F64) {
#pragma unroll
            for (int a = 0; a < DIM; ++a)
#pragma unroll
                for (int b = 0; b < DIM; ++b) G[a][b] = (double)M[a][b];
        }
    } else {
        const float *X = L.xyz + (size_t)job * DIM * N;
        const unsigned char *S = L.status + (size_t)job * N;
        // lattice coordinates; 32-bit division where the ids fit (a 64-bit one is a long routine)
        int c[3];
        if (N <= 0x7fffffffLL) {
            const unsigned u = (unsigned)p, r = u / (unsigned)L.n[0];
            c[0] = (int)(u - r * (unsigned)L.n[0]);
            c[2] = DIM == 3 ? (int)(r / (unsigned)L.n[1]) : 0;
            c[1] = DIM == 3 ? (int)(r - (unsigned)c[2] * (unsigned)L.n[1]) : (int)r;
        } else {
            c[0] = (int)(p % L.n[0]);
            c[1] = (int)((p / L.n[0]) % L.n[1]);
            c[2] = DIM == 3 ? (int)(p / ((long long)L.n[0] * L.n[1])) : 0;
        }
        const bool valid = S[p] == LCS_TRACER_OK;
        AxisDiff d[DIM];
        float f0[DIM], f1[DIM][DIM], f2[DIM][DIM];
        long long stride = 1;
        bool sided = false;
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
            long long q1, q2;
            d[b] = axis_diff(L, S, p, c[b], b, stride, valid, &q1, &q2);
            stride *= L.n[b];
            sided |= d[b].mode != 1;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                f1[b][a] = X[(size_t)a * N + q1];
                f2[b][a] = X[(size_t)a * N + q2];
            }
        }
#pragma unroll
        for (int a = 0; a < DIM; ++a) f0[a] = sided ? X[(size_t)a * N + p] : 0.0f;
        if (!EIG && L.ftle) L.ftle[out] = ftle_from_positions<DIM>(L, d, f0, f1, f2, half_inv_T);
        if constexpr (F64) {
#pragma unroll
            for (int b = 0; b < DIM; ++b)
#pragma unroll
                for (int a = 0; a < DIM; ++a) G[a][b] = axis_grad64(L, b, d[b], a == b, f0[a], f1[b][a], f2[b][a]);
        }
    }
    if constexpr (F64) {
        double C[NP];
        cauchy_green64<DIM>(G, C);
        if (L.C) {
            double *o = L.C + out * NP;
            if (DIM == 3 && L.c16) {
#pragma unroll
                for (int q = 0; q < NP; q += 2) *reinterpret_cast<double2 *>(o + q) = make_double2(C[q], C[q + 1]);
            } else {
#pragma unroll
                for (int q = 0; q < NP; ++q) o[q] = C[q];
            }
        }
        if constexpr (EIG) {   // lcs_cg_eigen
            double ev[DIM], V[DIM * DIM];
            if constexpr (DIM == 3) {
                if (!eig3_split(C, ev, V)) eig3_jacobi(C, ev, V);
            } else {
                eig_jacobi<2>(C, ev, V);
            }
            if (L.eigval) {
#pragma unroll
                for (int k = 0; k < DIM; ++k) L.eigval[out * DIM + k] = ev[k];
            }
            if (L.eigvec) {
#pragma unroll
                for (int k = 0; k < DIM * DIM; ++k) L.eigvec[out * DIM * DIM + k] = V[k];
            }
        } else if (L.lam || (GM == GM_AUX && L.ftle)) {
            const double lm = DIM == 2 ? eig_max2(C) : eig_max3(C);
            if (L.lam) L.lam[out] = lm;
            if (GM == GM_AUX && L.ftle) L.ftle[out] = log_lambda(lm) * half_inv_T;
        }
    }
}

// ------------------------------------------------------------------- launch

bool fixed_divisor_exact(double d, double *y, double *yl)
{
    typedef unsigned __int128 u128;
    typedef unsigned long long u64;
    // 1/d = y + yl: yl from the exact remainder 1 - y d; y is the upper neighbour where the
    // remainder is positive, so that yl <= 0
    double yh = 1.0 / d, rem = fma(-yh, d, 1.0);
    if (rem > 0.0) {
        yh = nextafter(yh, INFINITY);
        rem = fma(-yh, d, 1.0);
    }
    *y = yh;
    *yl = rem / d;
    if (rem == 0.0) return true;   // d a power of two
    int e;
    const u64 D = (u64)ldexp(frexp(d, &e), 53);   // significand, 2^52 <= D < 2^53
    // |x y + RN(x yl) - x/d| < 2^-104 |x/d|: a wrong rounding needs a significand X of x with
    // X 2^s - (2k + 1) D = r, |r| <= 16, s = 53 (X >= D) or 54 (X < D).  Every such X is tried.
    int v = 0;
    while (!((D >> v) & 1)) ++v;
    const u64 m = D >> v;              // X is determined modulo the odd part of D
    if (m < (1ULL << 46)) return v > 5;  // v > 5: no r qualifies; else more candidates than are worth trying
    u64 inv = 1, half = (m + 1) / 2;     // 2^-(s - v - 1) mod m, from 1/2 mod m
    for (int q = 0; q < 53 - v - 1; ++q) inv = (u64)((u128)inv * half % m);
    for (int s = 53; s <= 54; ++s) {
        if (s == 54) inv = (u64)((u128)inv * half % m);
        for (int r = -16; r <= 16; ++r) {
            // X 2^s = r + (2k + 1) D needs r = D (mod 2^(v+1)) (s > v): then X = ((r + D) / 2^(v+1)) 2^(v+1-s) mod m
            const long long num = (long long)D + r;
            if (r == 0 || num % (1LL << (v + 1))) continue;
            const u64 x = (u64)((u128)((u64)num >> (v + 1)) * inv % m), lo = 1ULL << 52, hi = 1ULL << 53;
            for (u64 X = x + (lo > x ? (lo - x + m - 1) / m * m : 0); X < hi; X += m) {
                const double xd = (double)X;
                if ((X >= D) == (s == 53) && fma(xd, yh, xd * *yl) != xd / d) return false;
            }
        }
    }
    return true;
}

void cg_prepare(CgLaunch &L)
{
    L.df_ok = 1;
    for (int b = 0; b < 3; ++b) {
        L.h2[b] = 2.0 * L.h[b];  // exact
        if (!L.div2) {
            L.rh2[b] = 1.0 / L.h2[b];
            L.rl2[b] = 0.0;
        }
        const double r = 1.0 / L.h2[b];
        L.rhf[b] = (float)r;
        L.rlf[b] = (float)(r - (double)L.rhf[b]);
        L.psh[b] = (float)L.period[b];
        L.psl[b] = (float)(L.period[b] - (double)L.psh[b]);
        if (b < L.dim && !(r >= 0x1p-60 && r <= 0x1p60 && fabs(L.period[b]) <= 0x1p60)) L.df_ok = 0;
    }
}

cudaError_t launch_cg_ftle(const CgLaunch &L0, cudaStream_t s)
{
    if (L0.N == 0 || L0.njobs == 0) return cudaSuccess;
    CgLaunch L = L0;
    cg_prepare(L);
    L.c16 = (uintptr_t)L.C % 16 == 0;
    const bool eig = L.eigval || L.eigvec;
    const int bt = 256;
    dim3 grid((unsigned)((L.N + bt - 1) / bt), (unsigned)L.njobs);
    const int gm = L.grad ? GM_VAR : (L.x0aux ? GM_AUX : GM_LATTICE);
    const bool f64 = L.C || L.lam || gm == GM_AUX;
#define CG_LAUNCH(D, G)                                                   \
    (eig ? cg_ftle_kernel<D, true, true, G><<<grid, bt, 0, s>>>(L)        \
         : f64 ? cg_ftle_kernel<D, true, false, G><<<grid, bt, 0, s>>>(L) \
               : cg_ftle_kernel<D, G == GM_AUX, false, G><<<grid, bt, 0, s>>>(L))
    if (L.dim == 2) {
        if (gm == GM_VAR) CG_LAUNCH(2, GM_VAR);
        else if (gm == GM_AUX) CG_LAUNCH(2, GM_AUX);
        else CG_LAUNCH(2, GM_LATTICE);
    } else {
        if (gm == GM_VAR) CG_LAUNCH(3, GM_VAR);
        else if (gm == GM_AUX) CG_LAUNCH(3, GM_AUX);
        else CG_LAUNCH(3, GM_LATTICE);
    }
#undef CG_LAUNCH
    return cudaGetLastError();
}
