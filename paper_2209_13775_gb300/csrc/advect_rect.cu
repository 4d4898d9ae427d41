// advect_rect.cu -- fixed-step RK4 advection through rectilinear velocity frames.
//
// Paper: Eq. 2 integrated over (t0, t0 + T) from a structured seed grid with
// the classical 4th-order Runge-Kutta method (Sec. 2 "Flow Map", Sec. 3.1),
// velocity interpolated bilinearly / trilinearly in space and linearly in time
// between two frames (Sec. 2 "Interpolator").
//
// Design (differs from the paper's split kernels, Sec. 3.1): one thread owns one
// tracer for the whole integration, with its state in registers; a step is
// four fused stage evaluations.  All tracers of a launch share the time
// schedule, so the frame bracket (k, alpha) of every stage is computed once
// per (job, step, stage) in FP64 by a small kernel and read as a warp-uniform
// broadcast.  Three families of kernels:
//   * gather: nodes read through L1/L2 (any field size, 2D and 3D; in 3D the last cell's corners kept);
//   * 2D time slices: the field blended once to every stage time;
//   * ring (2D): a block keeps three whole frames in shared memory, staged by
//     bulk asynchronous copies (cp.async.bulk + mbarrier) and prefetched one
//     step ahead, so the stage evaluations read shared memory only.
#include "rect_device.cuh"

#include <math.h>

// ===================================================================== schedule

// Stage time of (step n, stage s): t_n = t0 + n h; s = 0: t_n, 1: t_n + h/2, 2: t_n + h.
// Round-to-nearest FP64 operations, no fused multiply-add.
__device__ __forceinline__ double stage_time(double t0, double h, int n, int s)
{
    double t = __dadd_rn(t0, __dmul_rn((double)n, h));
    if (s == 1) t = __dadd_rn(t, __dmul_rn(0.5, h));
    if (s == 2) t = __dadd_rn(t, h);
    return t;
}

// frame bracket: largest k with t_k <= t (after the periodic wrap), clamped to [0, nf-2];
// alpha = (t - t_k) / (t_{k+1} - t_k), clamped to [0, 1] unless time is periodic
__device__ void frame_bracket(const double *__restrict__ times, int nf, int tp, double period, double t,
                              int *k, double *alpha)
{
    if (nf <= 1) {
        *k = 0;
        *alpha = 0.0;
        return;
    }
    double tt = t;
    if (tp) tt = __dsub_rn(t, __dmul_rn(period, floor(__ddiv_rn(__dsub_rn(t, times[0]), period))));
    int lo = 0, hi = nf - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (times[mid] <= tt)
            lo = mid;
        else
            hi = mid - 1;
    }
    int kk = lo < nf - 2 ? lo : nf - 2;
    double a = __ddiv_rn(__dsub_rn(tt, times[kk]), __dsub_rn(times[kk + 1], times[kk]));
    if (!tp) a = fmin(fmax(a, 0.0), 1.0);
    *k = kk;
    *alpha = a;
}

__global__ void rk4_schedule_kernel(const double *__restrict__ times, int nf, int tp, double period,
                                    const JobTable J, JobDev D, SchedEntry *__restrict__ sched)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int nsm = J.nsteps_max;
    long long total = (long long)J.njobs * nsm * 3;
    if (idx < J.njobs) {
        int j = (int)idx;
        D.nsteps[j] = J.nsteps[j];
        D.h[j] = __double2float_rn(J.h[j]);
        D.t0[j] = __double2float_rn(J.t0[j]);
        D.tend[j] = __double2float_rn(__dadd_rn(J.t0[j], J.T[j]));
        D.absT[j] = fabs(J.T[j]);
        for (int q = 0; q < J.nsnap; ++q)   // snapshot slots: |T| of the horizon they hold
            D.absT[J.njobs + j * J.nsnap + q] = fmin(J.snap_T[q], fabs(J.T[j]));
        if (j == 0 && D.snap_n)
            for (int q = 0; q < J.nsnap; ++q) D.snap_n[q] = J.snap_n[q];
        if (D.snap_te)   // t0 + T of the horizon a snapshot holds, as a run with that horizon computes it
            for (int q = 0; q < J.nsnap; ++q) {
                const double a = fmin(J.snap_T[q], fabs(J.T[j]));
                D.snap_te[j * J.nsnap + q] = __double2float_rn(__dadd_rn(J.t0[j], J.T[j] < 0.0 ? -a : a));
            }
        if (D.order) D.order[j] = J.order[j];
        if (D.t0d) D.t0d[j] = J.t0[j];
        if (D.Td) D.Td[j] = J.T[j];
    }
    if (idx >= total || !sched) return;
    int s = (int)(idx % 3);
    int n = (int)((idx / 3) % nsm);
    int job = (int)(idx / (3LL * nsm));
    SchedEntry e = {0, 0.0f};
    if (n < J.nsteps[job]) {
        int k;
        double a;
        frame_bracket(times, nf, tp, period, stage_time(J.t0[job], J.h[job], n, s), &k, &a);
        e.k = k;
        e.a = __double2float_rn(a);
    }
    sched[idx] = e;
}

cudaError_t launch_rk4_schedule(const double *d_times, int nframes, int time_periodic, double period,
                                const JobTable &J, JobDev D, SchedEntry *d_sched, cudaStream_t s)
{
    long long total = (long long)J.njobs * J.nsteps_max * 3;
    if (total < J.njobs) total = J.njobs;
    if (total == 0) return cudaSuccess;
    int bt = 256;
    unsigned grid = (unsigned)((total + bt - 1) / bt);
    rk4_schedule_kernel<<<grid, bt, 0, s>>>(d_times, nframes, time_periodic, period, J, D, d_sched);
    return cudaGetLastError();
}

// ============================================================ gather kernel

template <int ST>
__global__ void __launch_bounds__(256) rk4_gather2_kernel(RectParams P, const char *__restrict__ frames,
                                                          size_t fstride, Rk4Args A)
{
    constexpr int DIM = 2;
    const long long i = thread_tracer(A);
    int job = blockIdx.y;
    if (i < 0) return;
    float x[DIM], cx[DIM];
    int img[DIM];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        x[d] = A.seeds[d * A.N + i];
        cx[d] = 0.0f;
        img[d] = 0;
    }
    wrap_periodic<DIM>(P, x, cx, img);
    const SchedEntry *sc = A.sched + (size_t)job * A.nsteps_max * 3;
    const int ns = A.job_nsteps[job];
    const float h = A.job_h[job];
    unsigned char st = LCS_TRACER_OK;
    float te = A.job_tend[job];
    int si = 0;   // next snapshot
    for (int n = 0; n < ns; ++n) {
        SchedEntry e0 = load_sched(sc + 3 * n), e1 = load_sched(sc + 3 * n + 1), e2 = load_sched(sc + 3 * n + 2);
        rk4_step<2, ST, SRC_GLOBAL>(P, x, cx, h, frames + (size_t)e0.k * fstride,
                                    frames + (size_t)(e0.k + 1) * fstride, e0.a, frames + (size_t)e1.k * fstride,
                                    frames + (size_t)(e1.k + 1) * fstride, e1.a, frames + (size_t)e2.k * fstride,
                                    frames + (size_t)(e2.k + 1) * fstride, e2.a);
        wrap_periodic<DIM>(P, x, cx, img);
        if (rect_left<DIM>(P, x)) {
            st = LCS_TRACER_LEFT;
            te = fmaf((float)(n + 1), h, A.job_t0[job]);
            break;
        }
        for (; si < A.nsnap && snap_step(A, si, ns) == n + 1; ++si)
            store_tracer<DIM>(P, A, snap_slot(A, job, si), i, x, cx, img, st, snap_exit(A, job, si, st, te));
    }
    for (; si < A.nsnap; ++si)  // snapshots after the tracer stopped (or of a zero-step job)
        store_tracer<DIM>(P, A, snap_slot(A, job, si), i, x, cx, img, st, snap_exit(A, job, si, st, te));
    store_tracer<DIM>(P, A, job, i, x, cx, img, st, te);
}

// ------------------------------------------------------------ 3D gather

// Cell i0 (each axis' lower node) and fraction f of x, as axis_cell gives them.  PM >= 0 (boxes whose axes all
// wrap, or all end, within the reach of floor_index: box3_mask): the floor without the conversion pipe, x and y in
// two-lane FP32 instructions; indices more than a period away, which include every coordinate beyond that
// reach, go back to floorf.
template <int PM>
__device__ __forceinline__ void cell3(const RectParams &P, const float *x, int *i0, float *f)
{
    if constexpr (PM >= 0) {
        const float2 M2 = make_float2(FLOOR_MAGIC, FLOOR_MAGIC), m1 = make_float2(-1.0f, -1.0f);
        float2 q = make_float2(x[0], x[1]);
        float z = x[2];
        if constexpr (PM == 0) {
            q.x = fminf(fmaxf(q.x, P.origin[0]), P.hi_node[0]);
            q.y = fminf(fmaxf(q.y, P.origin[1]), P.hi_node[1]);
            z = fminf(fmaxf(z, P.origin[2]), P.hi_node[2]);
        }
        const float2 s = __fmul2_rn(__fadd2_rn(q, make_float2(-P.origin[0], -P.origin[1])),
                                    make_float2(P.inv_h[0], P.inv_h[1]));
        const float sz = __fmul_rn(z - P.origin[2], P.inv_h[2]);
        float2 t = __fadd2_rd(s, M2);
        float tz = __fadd_rd(sz, FLOOR_MAGIC);
        if constexpr (PM == 0) {
            t.x = fminf(t.x, FLOOR_MAGIC + (float)(P.n[0] - 2));
            t.y = fminf(t.y, FLOOR_MAGIC + (float)(P.n[1] - 2));
            tz = fminf(tz, FLOOR_MAGIC + (float)(P.n[2] - 2));
        }
        const float2 fr = __fadd2_rn(s, __ffma2_rn(t, m1, M2));
        f[0] = fr.x;
        f[1] = fr.y;
        f[2] = __fsub_rn(sz, tz - FLOOR_MAGIC);
        i0[0] = floor_index(t.x);
        i0[1] = floor_index(t.y);
        i0[2] = floor_index(tz);
        if constexpr (PM == 7) {
            const float sd[3] = {s.x, s.y, sz};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int n = P.n[d], i = i0[d];
                int w = i < 0 ? i + n : (i >= n ? i - n : i);
                if ((unsigned)w >= (unsigned)n) {
                    const float fl = floorf(sd[d]);
                    f[d] = sd[d] - fl;
                    w = wrap_index_slow((int)fl, n);
                }
                i0[d] = w;
            }
        }
    } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            int i1;
            axis_cell<PM>(P, d, x[d], i0[d], i1, f[d]);
        }
    }
}

// The corners of a tracer's last cell, blended to the time of its last stage (k, a)
struct BlendCache {
    float u[8][3];
    int v0, k;
    float a;
};

// u(x) at schedule entry e: interp3p's values.  Stage 3 of a step shares the time of stage 2 and stage 1 mostly
// that of the stage 4 before, and their points are mostly in the same cells, so half of the stencils need no
// loads, conversions or blends.
template <int ST, int PM>
__device__ __forceinline__ void interp3_cached(const RectParams &P, const float *x, const char *__restrict__ frames,
                                               size_t fstride, SchedEntry e, BlendCache &cc, float *f, float *u)
{
    int i[3];
    cell3<PM>(P, x, i, f);
    const int sy = (int)P.sy, sz = (int)P.sz, v0 = i[0] + i[1] * sy + i[2] * sz;
    if (v0 != cc.v0 || e.k != cc.k || e.a != cc.a) {
        int dx[3] = {1, sy, sz};   // to the upper node of each axis
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (per_axis<PM>(P, d) && i[d] + 1 == P.n[d]) dx[d] -= P.n[d] * dx[d];
        const char *fp = frames + (size_t)e.k * fstride;
        const float g = 1.0f - e.a;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float va[3], vb[3];
            Pair3<ST>::ld(fp, v0 + (q & 1 ? dx[0] : 0) + (q & 2 ? dx[1] : 0) + (q & 4 ? dx[2] : 0), va, vb);
#pragma unroll
            for (int c = 0; c < 3; ++c) cc.u[q][c] = e.a == 0.0f ? va[c] : tblend(va[c], vb[c], e.a, g);
        }
        cc.v0 = v0;
        cc.k = e.k;
        cc.a = e.a;
    }
    const float gx = 1.0f - f[0], gy = 1.0f - f[1], gz = 1.0f - f[2];
    const float a = gy * gz, b = f[1] * gz, c = gy * f[2], d = f[1] * f[2];
    const float w[8] = {gx * a, f[0] * a, gx * b, f[0] * b, gx * c, f[0] * c, gx * d, f[0] * d};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float acc = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) acc = fmaf(w[q], cc.u[q][k], acc);
        u[k] = acc;
    }
}

// One pass over a job's steps, one thread per tracer.  Its loads go through L1 (a corner is both frames of a node,
// 32 bytes in FP32), so the blended corners kept in registers count most; then the issue slots, of which the cell
// search took a quarter.  100 steps of 103,635 tracers on 64^3 FP16 nodes: 642 us before with the corners loaded at
// every stage and the general cell search, 350 us now; 512,000 on FP32: 3.19 ms before, 1.66 ms.  Three blocks per
// SM (80 registers): with four 1.68 and on 128^3 nodes 2.55 ms for 2.37.
template <int ST, int PM>
__global__ void __launch_bounds__(256, 3) rk4_gather3_kernel(const __grid_constant__ RectParams P,
                                                               const char *__restrict__ frames, size_t fstride,
                                                               const __grid_constant__ Rk4Args A)
{
    const long long i = thread_tracer(A);
    const int job = blockIdx.y;
    if (i < 0) return;
    float x[3] = {A.seeds[i], A.seeds[A.N + i], A.seeds[2 * A.N + i]}, cx[3] = {0.0f, 0.0f, 0.0f};
    int img[3] = {0, 0, 0};
    wrap_periodic<3, PM>(P, x, cx, img);
    const SchedEntry *sc = A.sched + (size_t)job * A.nsteps_max * 3;
    const int ns = A.job_nsteps[job];
    const float h = A.job_h[job], hh = 0.5f * h, h6 = h * (1.0f / 6.0f);
    unsigned char st = LCS_TRACER_OK;
    float te = A.job_tend[job];
    int si = 0;   // next snapshot
    BlendCache cc;
    cc.v0 = -1;
    for (int n = 0; n < ns; ++n) {
        const SchedEntry e0 = load_sched(sc + 3 * n), e1 = load_sched(sc + 3 * n + 1), e2 = load_sched(sc + 3 * n + 2);
        float k1[3], k2[3], k3[3], k4[3], y[3], f[3];
        const auto stage = [&](float c, const float *k) {
            const float2 q = __ffma2_rn(make_float2(c, c), make_float2(k[0], k[1]), make_float2(x[0], x[1]));
            y[0] = q.x;
            y[1] = q.y;
            y[2] = fmaf(c, k[2], x[2]);
        };
        interp3_cached<ST, PM>(P, x, frames, fstride, e0, cc, f, k1);
        stage(hh, k1);
        interp3_cached<ST, PM>(P, y, frames, fstride, e1, cc, f, k2);
        stage(hh, k2);
        interp3_cached<ST, PM>(P, y, frames, fstride, e1, cc, f, k3);
        stage(h, k3);
        interp3_cached<ST, PM>(P, y, frames, fstride, e2, cc, f, k4);
        float2 xy = make_float2(x[0], x[1]), cxy = make_float2(cx[0], cx[1]);
        rk4_advance2(xy, cxy, h6, make_float2(k1[0], k1[1]), make_float2(k2[0], k2[1]), make_float2(k3[0], k3[1]),
                     make_float2(k4[0], k4[1]));
        x[0] = xy.x;
        x[1] = xy.y;
        cx[0] = cxy.x;
        cx[1] = cxy.y;
        rk4_advance(x[2], cx[2], h6, k1[2], k2[2], k3[2], k4[2]);
        wrap_periodic_step<3, PM>(P, x, cx, img);
        if (rect_left<3, PM>(P, x)) {
            st = LCS_TRACER_LEFT;
            te = fmaf((float)(n + 1), h, A.job_t0[job]);
            break;
        }
        for (; si < A.nsnap && snap_step(A, si, ns) == n + 1; ++si)
            store_tracer<3>(P, A, snap_slot(A, job, si), i, x, cx, img, st, snap_exit(A, job, si, st, te));
    }
    for (; si < A.nsnap; ++si)  // snapshots after the tracer stopped (or of a zero-step job)
        store_tracer<3>(P, A, snap_slot(A, job, si), i, x, cx, img, st, snap_exit(A, job, si, st, te));
    store_tracer<3>(P, A, job, i, x, cx, img, st, te);
}

// ============================================================ variational

// 2D: u and its spatial Jacobian J[c][d] at x, linear in time between two frames: u with
// interp's arithmetic (node blends first, then make_stencil's weights in order), J from the
// same blended corner values and the derivatives of the weights inside the cell; a
// non-periodic axis on which x lies outside the box gives a zero column (the clamped query
// does not move with x).
template <int ST>
__device__ __forceinline__ void interp_grad(const RectParams &P, const float *x, const char *fa, const char *fb,
                                            float a, float *u, float (*J)[2])
{
    Stencil<2> S;
    make_stencil<2>(P, x, S);
    float f[2], on[2];
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        int i0, i1;
        axis_cell<-1>(P, d, x[d], i0, i1, f[d]);
        on[d] = (P.periodic[d] || (x[d] >= P.origin[d] && x[d] <= P.hi_node[d])) ? P.inv_h[d] : 0.0f;
    }
    float uq[4][2], va[2], vb[2];
    const float g = 1.0f - a;
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // frame fb is read only when a != 0
        node_load<2, ST, SRC_GLOBAL>(fa, S.v[q], va);
        if (a != 0.0f) node_load<2, ST, SRC_GLOBAL>(fb, S.v[q], vb);
#pragma unroll
        for (int c = 0; c < 2; ++c) uq[q][c] = a == 0.0f ? va[c] : tblend(va[c], vb[c], a, g);
    }
    // corner q has offsets (q & 1, q >> 1); d w_q / d x_d = +-(weight of the other axis) / h_d
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        float acc = 0.0f, jx = 0.0f, jy = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            acc = fmaf(S.w[q], uq[q][c], acc);
            const float wx = q >> 1 ? f[1] : 1.0f - f[1], wy = q & 1 ? f[0] : 1.0f - f[0];
            jx = fmaf(q & 1 ? wx : -wx, uq[q][c], jx);
            jy = fmaf(q >> 1 ? wy : -wy, uq[q][c], jy);
        }
        u[c] = acc;
        J[c][0] = jx * on[0];
        J[c][1] = jy * on[1];
    }
}

// RK4 with the variational equations dM/dt = J M: the position follows rk4_step's arithmetic
// exactly (so x(T) equals the other kernels'), M the same stages in FP32
template <int ST>
__global__ void __launch_bounds__(256) rk4_var2_kernel(RectParams P, const char *__restrict__ frames, size_t fstride,
                                                       Rk4Args A)
{
    constexpr int DIM = 2;
    const long long i = thread_tracer(A);
    const int job = blockIdx.y;
    if (i < 0) return;
    float x[DIM], cx[DIM], M[DIM][DIM];
    int img[DIM];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        x[d] = A.seeds[d * A.N + i];
        cx[d] = 0.0f;
        img[d] = 0;
#pragma unroll
        for (int e = 0; e < DIM; ++e) M[d][e] = d == e ? 1.0f : 0.0f;
    }
    wrap_periodic<DIM>(P, x, cx, img);
    const SchedEntry *sc = A.sched + (size_t)job * A.nsteps_max * 3;
    const int ns = A.job_nsteps[job];
    const float h = A.job_h[job], hh = 0.5f * h, h6 = h * (1.0f / 6.0f);
    unsigned char st = LCS_TRACER_OK;
    float te = A.job_tend[job];
    for (int n = 0; n < ns; ++n) {
        const SchedEntry es[3] = {load_sched(sc + 3 * n), load_sched(sc + 3 * n + 1), load_sched(sc + 3 * n + 2)};
        float k[4][DIM], K[4][DIM][DIM], y[DIM], Y[DIM][DIM], J[DIM][DIM];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const SchedEntry e = es[q == 0 ? 0 : (q == 3 ? 2 : 1)];
            const float c = q == 0 ? 0.0f : (q == 3 ? h : hh);
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                y[a] = q == 0 ? x[a] : fmaf(c, k[q - 1][a], x[a]);
#pragma unroll
                for (int b = 0; b < DIM; ++b) Y[a][b] = q == 0 ? M[a][b] : fmaf(c, K[q - 1][a][b], M[a][b]);
            }
            const char *fa = frames + (size_t)e.k * fstride;
            interp_grad<ST>(P, y, fa, fa + fstride, e.a, k[q], J);
#pragma unroll
            for (int a = 0; a < DIM; ++a)
#pragma unroll
                for (int b = 0; b < DIM; ++b) {
                    float acc = 0.0f;
#pragma unroll
                    for (int cc = 0; cc < DIM; ++cc) acc = fmaf(J[a][cc], Y[cc][b], acc);
                    K[q][a][b] = acc;
                }
        }
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            rk4_advance(x[a], cx[a], h6, k[0][a], k[1][a], k[2][a], k[3][a]);
#pragma unroll
            for (int b = 0; b < DIM; ++b)
                M[a][b] = fmaf(h6, (K[0][a][b] + K[3][a][b]) + 2.0f * (K[1][a][b] + K[2][a][b]), M[a][b]);
        }
        wrap_periodic<DIM>(P, x, cx, img);
        if (rect_left<DIM>(P, x)) {
            st = LCS_TRACER_LEFT;
            te = fmaf((float)(n + 1), h, A.job_t0[job]);
            break;
        }
    }
    store_tracer<DIM>(P, A, job, i, x, cx, img, st, te);
    float *o = A.out_grad + ((size_t)job * A.N + i) * DIM * DIM;
#pragma unroll
    for (int a = 0; a < DIM; ++a)
#pragma unroll
        for (int b = 0; b < DIM; ++b) o[a * DIM + b] = M[a][b];
}

// The same in 3D, through the blended corners of the last cell.  Bound by issue (the Jacobian and its product
// with M take two thirds of the instructions).  Two blocks of registers per SM: 262,144 tracers on 64^3 FP32
// nodes, 100 steps, 1.11 ms; three spill, 1.42 ms.
template <int ST, int PM>
__global__ void __launch_bounds__(256, 2) rk4_var3_kernel(const __grid_constant__ RectParams P,
                                                          const char *__restrict__ frames, size_t fstride,
                                                          const __grid_constant__ Rk4Args A)
{
    const long long i = thread_tracer(A);
    const int job = blockIdx.y;
    if (i < 0) return;
    float x[3] = {A.seeds[i], A.seeds[A.N + i], A.seeds[2 * A.N + i]}, cx[3] = {0.0f, 0.0f, 0.0f}, M[3][3];
    int img[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < 9; ++a) M[a / 3][a % 3] = a % 4 ? 0.0f : 1.0f;
    wrap_periodic<3, PM>(P, x, cx, img);
    const SchedEntry *sc = A.sched + (size_t)job * A.nsteps_max * 3;
    const int ns = A.job_nsteps[job];
    const float h = A.job_h[job], hh = 0.5f * h, h6 = h * (1.0f / 6.0f);
    unsigned char st = LCS_TRACER_OK;
    float te = A.job_tend[job];
    BlendCache cc;
    cc.v0 = -1;
    for (int n = 0; n < ns; ++n) {
        const SchedEntry es[3] = {load_sched(sc + 3 * n), load_sched(sc + 3 * n + 1), load_sched(sc + 3 * n + 2)};
        float k[4][3], S03[3][3], S12[3][3], Kp[3][3];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float c = q == 0 ? 0.0f : (q == 3 ? h : hh);
            float y[3], Y[3][3], f[3], on[3], J[3][3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                y[a] = q == 0 ? x[a] : fmaf(c, k[q - 1][a], x[a]);
                on[a] = per_axis<PM>(P, a) || (y[a] >= P.origin[a] && y[a] <= P.hi_node[a]) ? P.inv_h[a] : 0.0f;
#pragma unroll
                for (int b = 0; b < 3; ++b) Y[a][b] = q == 0 ? M[a][b] : fmaf(c, Kp[a][b], M[a][b]);
            }
            interp3_cached<ST, PM>(P, y, frames, fstride, es[q == 0 ? 0 : (q == 3 ? 2 : 1)], cc, f, k[q]);
            float2 uv[8], Jp[3];
            float z[8], Jz[3];
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                uv[b] = make_float2(cc.u[b][0], cc.u[b][1]);
                z[b] = cc.u[b][2];
            }
            trilinear_grad_nodes(uv, f, on, Jp);
            trilinear_grad_nodes(z, f, on, Jz);
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                J[0][b] = Jp[b].x;
                J[1][b] = Jp[b].y;
                J[2][b] = Jz[b];
            }
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    float acc = 0.0f;
#pragma unroll
                    for (int d = 0; d < 3; ++d) acc = fmaf(J[a][d], Y[d][b], acc);
                    Kp[a][b] = acc;
                    if (q == 0) S03[a][b] = acc;
                    else if (q == 1) S12[a][b] = acc;
                    else if (q == 2) S12[a][b] = S12[a][b] + acc;
                    else S03[a][b] = S03[a][b] + acc;
                }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            rk4_advance(x[a], cx[a], h6, k[0][a], k[1][a], k[2][a], k[3][a]);
#pragma unroll
            for (int b = 0; b < 3; ++b) M[a][b] = fmaf(h6, S03[a][b] + 2.0f * S12[a][b], M[a][b]);
        }
        wrap_periodic_step<3, PM>(P, x, cx, img);
        if (rect_left<3, PM>(P, x)) {
            st = LCS_TRACER_LEFT;
            te = fmaf((float)(n + 1), h, A.job_t0[job]);
            break;
        }
    }
    store_tracer<3>(P, A, job, i, x, cx, img, st, te);
    float *o = A.out_grad + ((size_t)job * A.N + i) * 9;
#pragma unroll
    for (int a = 0; a < 9; ++a) o[a] = M[a / 3][a % 3];
}

// ============================================================== ring kernel

// Three frame slots in shared memory, tagged with the frame they hold.  Thread 0
// makes the frames of step n resident (bulk copies into slots no stage of step n
// needs), prefetches those of step n + 1 into a free slot, and publishes the
// slot of every stage frame; a frame that cannot get a slot is read from global
// memory for that step.
#define RING_SLOTS 3
#define RING_GLOBAL (-2)
#define RING_NONE (-1)

struct RingState {
    uint64_t bar[RING_SLOTS];
    int tag[RING_SLOTS];
    unsigned nload[RING_SLOTS];
    int slot[6];   // per stage (0..2): slot of frame k, slot of frame k + 1 (or NONE / GLOBAL)
    int kf[6];     // frame ids for the GLOBAL case
    int abort;     // a wait timed out: the block stops issuing copies and computing
};

struct RingWork {
    int persistent;        // 0: block (x, y) = tile x of job y; 1: items pulled from *queue
    unsigned *queue;       // persistent: item counter, zero at launch
    long long nitems;      // persistent: tiles_per_job * njobs
    int tiles_per_job;
    const int *jorder;     // persistent: job of rank r, longest first
};

__device__ __forceinline__ int ring_find(const RingState &R, int f)
{
    for (int s = 0; s < RING_SLOTS; ++s)
        if (R.tag[s] == f) return s;
    return -1;
}

// frames a step reads: k of each stage, and k + 1 where alpha != 0
__device__ __forceinline__ int step_frames(const SchedEntry *e, int *F)
{
    int m = 0;
    for (int s = 0; s < 3; ++s) {
        int c[2] = {e[s].k, e[s].a != 0.0f ? e[s].k + 1 : -1};
        for (int q = 0; q < 2; ++q) {
            if (c[q] < 0) continue;
            bool dup = false;
            for (int r = 0; r < m; ++r) dup |= (F[r] == c[q]);
            if (!dup) F[m++] = c[q];
        }
    }
    return m;
}

__device__ __forceinline__ bool in_list(const int *F, int m, int f)
{
    for (int r = 0; r < m; ++r)
        if (F[r] == f) return true;
    return false;
}

// thread 0: load frame f into a slot that holds none of the protected frames
__device__ int ring_load(RingState &R, char *slots, const char *frames, size_t fstride, int f, const int *keep,
                         int nkeep, unsigned *errword, uint64_t wait_ns)
{
    int v = -1;
    for (int s = 0; s < RING_SLOTS && v < 0; ++s)
        if (R.tag[s] < 0) v = s;
    for (int s = 0; s < RING_SLOTS && v < 0; ++s)
        if (!in_list(keep, nkeep, R.tag[s])) v = s;
    if (v < 0) return RING_GLOBAL;
    if (R.nload[v] > 0 && !mbar_wait_limit(&R.bar[v], (R.nload[v] - 1) & 1, wait_ns)) {  // previous copy into v
        atomicOr(errword, LCS_ERRBIT_TIMEOUT);
        R.abort = 1;
        return RING_GLOBAL;
    }
    R.tag[v] = f;
    R.nload[v] += 1;
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(&R.bar[v], (unsigned)fstride);
    bulk_g2s(slots + (size_t)v * fstride, frames + (size_t)f * fstride, (unsigned)fstride, &R.bar[v]);
    return v;
}

// Work of one block: the tracers [tile * TPT * bt, (tile + 1) * TPT * bt) of one job, each
// thread holding TPT tracers (sub-tiles of bt consecutive seeds, so loads stay coalesced).
template <int ST, int TPT>
__device__ __forceinline__ void ring_tile(const RectParams &P, const char *__restrict__ frames, size_t fstride,
                                          const Rk4Args &A, unsigned *errword, char *slots, RingState &R, int job,
                                          long long tile)
{
    const int tid = threadIdx.x, bt = blockDim.x;
    long long idx[TPT];
    bool active[TPT], live[TPT];
    float x[TPT][2], cx[TPT][2];
    int img[TPT][2];
    unsigned char st[TPT];
    float te[TPT];
    const float tend = A.job_tend[job];
#pragma unroll
    for (int t = 0; t < TPT; ++t) {
        idx[t] = (tile * TPT + t) * bt + tid;
        active[t] = idx[t] < A.N;
        live[t] = active[t];
        x[t][0] = active[t] ? A.seeds[idx[t]] : 0.0f;
        x[t][1] = active[t] ? A.seeds[A.N + idx[t]] : 0.0f;
        cx[t][0] = cx[t][1] = 0.0f;
        img[t][0] = img[t][1] = 0;
        wrap_periodic<2>(P, x[t], cx[t], img[t]);
        st[t] = LCS_TRACER_OK;
        te[t] = tend;
    }
    const SchedEntry *sc = A.sched + (size_t)job * A.nsteps_max * 3;
    const int ns = A.job_nsteps[job];
    const float h = A.job_h[job];
    int si = 0;   // next snapshot
    for (int n = 0; n < ns; ++n) {
        __syncthreads();  // every thread is done with the previous step's slots
        if (R.abort) break;
        if (tid == 0) {
            SchedEntry e[3] = {sc[3 * n], sc[3 * n + 1], sc[3 * n + 2]};
            int F[6], Fn[6];
            int m = step_frames(e, F);
            for (int r = 0; r < m; ++r)
                if (ring_find(R, F[r]) < 0) ring_load(R, slots, frames, fstride, F[r], F, m, errword, A.wait_ns);
            for (int s = 0; s < 3; ++s) {
                int fa = e[s].k, fb = e[s].k + 1;
                int sa = ring_find(R, fa);
                R.slot[2 * s] = sa >= 0 ? sa : RING_GLOBAL;
                R.kf[2 * s] = fa;
                if (e[s].a != 0.0f) {
                    int sb = ring_find(R, fb);
                    R.slot[2 * s + 1] = sb >= 0 ? sb : RING_GLOBAL;
                } else {
                    R.slot[2 * s + 1] = RING_NONE;
                }
                R.kf[2 * s + 1] = fb;
            }
            if (n + 1 < ns) {  // prefetch the next step's frames into slots this step leaves alone
                SchedEntry en[3] = {sc[3 * n + 3], sc[3 * n + 4], sc[3 * n + 5]};
                int mn = step_frames(en, Fn);
                int keep[12];
                int nk = 0;
                for (int r = 0; r < m; ++r) keep[nk++] = F[r];
                for (int r = 0; r < mn; ++r) keep[nk++] = Fn[r];
                for (int r = 0; r < mn; ++r)
                    if (ring_find(R, Fn[r]) < 0) ring_load(R, slots, frames, fstride, Fn[r], keep, nk, errword, A.wait_ns);
            }
        }
        __syncthreads();
        // wait for the copies this step reads
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            int s = R.slot[q];
            if (s >= 0 && !R.abort && !mbar_wait_limit(&R.bar[s], (R.nload[s] - 1) & 1, A.wait_ns)) {
                atomicOr(errword, LCS_ERRBIT_TIMEOUT);
                R.abort = 1;
            }
        }
        if (R.abort) continue;
        const char *p[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            int s = R.slot[q];
            if (s >= 0)
                p[q] = slots + (size_t)s * fstride;
            else if (s == RING_NONE)
                p[q] = p[q - 1];  // alpha == 0: frame k + 1 is never read; keep a pointer of the same space
            else
                p[q] = frames + (size_t)R.kf[q] * fstride;
        }
        const SchedEntry e0 = load_sched(sc + 3 * n), e1 = load_sched(sc + 3 * n + 1), e2 = load_sched(sc + 3 * n + 2);
        const bool all_smem = (R.slot[0] != RING_GLOBAL) && (R.slot[1] != RING_GLOBAL) &&
                              (R.slot[2] != RING_GLOBAL) && (R.slot[3] != RING_GLOBAL) &&
                              (R.slot[4] != RING_GLOBAL) && (R.slot[5] != RING_GLOBAL);
#pragma unroll
        for (int t = 0; t < TPT; ++t) {
            if (!live[t]) continue;
            // a step whose frames did not all get a slot (e.g. one straddling the periodic wrap, which
            // reads four frames) mixes shared and global pointers: generic loads serve both
            if (all_smem)
                rk4_step<2, ST, SRC_SHARED>(P, x[t], cx[t], h, p[0], p[1], e0.a, p[2], p[3], e1.a, p[4], p[5],
                                            e2.a);
            else
                rk4_step<2, ST, SRC_GENERIC>(P, x[t], cx[t], h, p[0], p[1], e0.a, p[2], p[3], e1.a, p[4], p[5],
                                             e2.a);
            wrap_periodic<2>(P, x[t], cx[t], img[t]);
            if (rect_left<2>(P, x[t])) {
                st[t] = LCS_TRACER_LEFT;
                te[t] = fmaf((float)(n + 1), h, A.job_t0[job]);
                live[t] = false;
            }
        }
        for (; si < A.nsnap && snap_step(A, si, ns) == n + 1; ++si)
#pragma unroll
            for (int t = 0; t < TPT; ++t)
                if (active[t])
                    store_tracer<2>(P, A, snap_slot(A, job, si), idx[t], x[t], cx[t], img[t], st[t],
                                    snap_exit(A, job, si, st[t], te[t]));
    }
    for (; si < A.nsnap; ++si)  // a zero-step job, or a block that stopped on a copy timeout
#pragma unroll
        for (int t = 0; t < TPT; ++t)
            if (active[t])
                store_tracer<2>(P, A, snap_slot(A, job, si), idx[t], x[t], cx[t], img[t], st[t],
                                snap_exit(A, job, si, st[t], te[t]));
#pragma unroll
    for (int t = 0; t < TPT; ++t)
        if (active[t]) store_tracer<2>(P, A, job, idx[t], x[t], cx[t], img[t], st[t], te[t]);
}

// Ring kernel.  Non-persistent: block (x, y) is tile x of job y.  Persistent: the grid
// fills the GPU once and every block pulls (job, tile) items from an atomic counter in
// the order of W.jorder (longest jobs first), keeping its frame ring across items.
template <int ST, int TPT>
__global__ void __launch_bounds__(512, 1) rk4_ring2d_kernel(RectParams P, const char *__restrict__ frames,
                                                         size_t fstride, Rk4Args A, unsigned *errword, RingWork W)
{
    extern __shared__ __align__(128) char slots[];
    __shared__ RingState R;
    __shared__ long long s_item;
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int s = 0; s < RING_SLOTS; ++s) {
            mbar_init(&R.bar[s], 1);
            R.tag[s] = -1;
            R.nload[s] = 0;
        }
        R.abort = 0;
        mbar_fence_init();
    }
    __syncthreads();
    if (!W.persistent) {
        ring_tile<ST, TPT>(P, frames, fstride, A, errword, slots, R, blockIdx.y, blockIdx.x);
    } else {
        for (;;) {
            if (tid == 0) s_item = (long long)atomicAdd(W.queue, 1u);
            __syncthreads();
            const long long item = s_item;
            __syncthreads();
            if (item >= W.nitems || R.abort) break;
            const int job = W.jorder[item / W.tiles_per_job];
            ring_tile<ST, TPT>(P, frames, fstride, A, errword, slots, R, job, item % W.tiles_per_job);
        }
    }
    // drain copies still in flight (prefetches nobody read, or copies a shortened wait gave up on)
    // before the block exits, with the full bound whatever the call's wait limit
    __syncthreads();
    if (tid == 0)
        for (int s = 0; s < RING_SLOTS; ++s)
            if (R.nload[s] > 0 && !mbar_wait_bounded(&R.bar[s], (R.nload[s] - 1) & 1))
                atomicOr(errword, LCS_ERRBIT_TIMEOUT);
    __syncthreads();
}

// ========================================================== 2D time slices

// Variant 5 (2D): every stage time of every job gets its own time slice, the field blended
// to that time once (interp's node-first arithmetic, FP32), stored per node as two float4
// quads (u(i,j), u(i1,j), u(i,j1), u(i1,j1)) and the same for v, with i1, j1 the next node
// (wrapped on a periodic axis, clamped on a closed one).  A stage evaluation is then the
// cell and weights of make_stencil and two 16-byte loads, with the products of interp in
// interp's order: bit-identical to the other variants.  Slice (job, n, stage) is number
// off[job] + 3 n + stage, each 2 * nodes float4.
struct Slice2dOffsets {
    long long off[LCS_MAX_JOBS];
};

// Whether two schedule entries give the same field: the same bracket and weight, or the end of one bracket
// and the start of the next (frame k + 1 with weight 1 and frame k + 1 with the next frame's weight 0).
__device__ __forceinline__ bool same_slice(SchedEntry a, SchedEntry b)
{
    return (a.k == b.k && a.a == b.a) || (a.k + 1 == b.k && a.a == 1.0f && b.a == 0.0f) ||
           (b.k + 1 == a.k && b.a == 1.0f && a.a == 0.0f);
}

// A thread fills its node in FILL_RUN consecutive slices of a job (blocks: nodes x runs x jobs), so the node's
// corners are found once and the frames they are blended from are loaded once per bracket.  shared[job][n] = 1
// where step n starts at the time its step n - 1 ended: that step has no first slice of its own.
#define FILL_RUN 12
template <int ST>
__global__ void __launch_bounds__(256) slice2d_fill_kernel(RectParams P, const char *__restrict__ frames, size_t fstride,
                                                           const SchedEntry *__restrict__ sched, int nsteps_max,
                                                           const int *__restrict__ job_nsteps,
                                                           const __grid_constant__ Slice2dOffsets O, int nodes,
                                                           unsigned char *__restrict__ shared,
                                                           float4 *__restrict__ slices)
{
    const int job = blockIdx.z, v = blockIdx.x * 256 + threadIdx.x;
    const long long nsl = 3LL * job_nsteps[job];
    if (v >= nodes) return;
    const SchedEntry *sc = sched + (size_t)job * nsteps_max * 3;
    const int j = v / P.n[0], i = v - j * P.n[0];
    const int i1 = P.periodic[0] ? (i + 1 == P.n[0] ? 0 : i + 1) : min(i + 1, P.n[0] - 1);
    const int j1 = P.periodic[1] ? (j + 1 == P.n[1] ? 0 : j + 1) : min(j + 1, P.n[1] - 1);
    const int sy = (int)P.sy, corner[4] = {i + j * sy, i1 + j * sy, i + j1 * sy, i1 + j1 * sy};
    float ua[4][2], ub[4][2];
    int ka = -1, kb = -1;
    // (one run per block unless a job has more runs than a grid has rows)
    for (long long l = (long long)blockIdx.y * FILL_RUN; l < nsl;
         l += (l + 1) % FILL_RUN ? 1 : (gridDim.y - 1) * (long long)FILL_RUN + 1) {
        const SchedEntry e = load_sched(sc + l);   // slice l of the job = schedule entry l (= 3 n + stage)
        if (l % 3 == 0) {
            const bool same = l > 0 && same_slice(load_sched(sc + l - 1), e);
            if (v == 0) shared[(size_t)job * nsteps_max + l / 3] = same;
            if (same) continue;                    // the last slice of the step before serves
        }
        const char *fa = frames + (size_t)e.k * fstride;
        if (e.k != ka) {
#pragma unroll
            for (int q = 0; q < 4; ++q) Node<2, ST>::ld(fa, corner[q], ua[q]);
            ka = e.k;
        }
        if (e.a != 0.0f && e.k != kb) {            // frame k + 1 is not read at weight 0 (it may not exist)
#pragma unroll
            for (int q = 0; q < 4; ++q) Node<2, ST>::ld(fa + fstride, corner[q], ub[q]);
            kb = e.k;
        }
        const float g = 1.0f - e.a;
        float u[2][4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) u[c][q] = e.a == 0.0f ? ua[q][c] : tblend(ua[q][c], ub[q][c], e.a, g);
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(slices + ((O.off[job] + l) * nodes + v) * 2),
                     "f"(u[0][0]), "f"(u[0][1]), "f"(u[0][2]), "f"(u[0][3]), "f"(u[1][0]), "f"(u[1][1]), "f"(u[1][2]),
                     "f"(u[1][3])
                     : "memory");
    }
}

// u(x) from a 2D slice: make_stencil's cell and weights, interp's products and order
template <int PM>
__device__ __forceinline__ void interp2s(const RectParams &P, const float *x, const float4 *__restrict__ sl, float *u)
{
    Stencil<2> S;
    make_stencil<2, PM>(P, x, S);
    const float4 qu = __ldg(sl + 2 * S.v[0]), qv = __ldg(sl + 2 * S.v[0] + 1);
    u[0] = fmaf(S.w[3], qu.w, fmaf(S.w[2], qu.z, fmaf(S.w[1], qu.y, fmaf(S.w[0], qu.x, 0.0f))));
    u[1] = fmaf(S.w[3], qv.w, fmaf(S.w[2], qv.z, fmaf(S.w[1], qv.y, fmaf(S.w[0], qv.x, 0.0f))));
}

// PM: compile-time periodicity (bit d: axis d periodic; -1: read from P)
template <int PM>
__global__ void __launch_bounds__(256) rk4_slice2d_kernel(RectParams P, const float4 *__restrict__ slices,
                                                          long long nodes, Slice2dOffsets O,
                                                          const unsigned char *__restrict__ shared, Rk4Args A)
{
    const long long i = thread_tracer(A);
    const int job = blockIdx.y;
    if (i < 0) return;
    float x[2] = {A.seeds[i], A.seeds[A.N + i]}, cx[2] = {0.0f, 0.0f};
    int img[2] = {0, 0};
    wrap_periodic<2, PM>(P, x, cx, img);
    const int ns = A.job_nsteps[job];
    const float h = A.job_h[job];
    const float4 *sj = slices + O.off[job] * 2 * nodes;
    const unsigned char *sh = shared + (size_t)job * A.nsteps_max;
    const size_t ss = 2 * (size_t)nodes;
    unsigned char st = LCS_TRACER_OK;
    float te = A.job_tend[job];
    int si = 0;   // next snapshot
    for (int n = 0; n < ns; ++n) {
        const float4 *s0 = sj + (size_t)(3 * n) * ss;
        float k1[2], k2[2], k3[2], k4[2], y[2];
        const float hh = 0.5f * h;
        interp2s<PM>(P, x, __ldg(sh + n) ? s0 - ss : s0, k1);
#pragma unroll
        for (int c = 0; c < 2; ++c) y[c] = fmaf(hh, k1[c], x[c]);
        interp2s<PM>(P, y, s0 + ss, k2);
#pragma unroll
        for (int c = 0; c < 2; ++c) y[c] = fmaf(hh, k2[c], x[c]);
        interp2s<PM>(P, y, s0 + ss, k3);
#pragma unroll
        for (int c = 0; c < 2; ++c) y[c] = fmaf(h, k3[c], x[c]);
        interp2s<PM>(P, y, s0 + 2 * ss, k4);
        const float h6 = h * (1.0f / 6.0f);
#pragma unroll
        for (int c = 0; c < 2; ++c) rk4_advance(x[c], cx[c], h6, k1[c], k2[c], k3[c], k4[c]);
        wrap_periodic<2, PM>(P, x, cx, img);
        if (rect_left<2, PM>(P, x)) {
            st = LCS_TRACER_LEFT;
            te = fmaf((float)(n + 1), h, A.job_t0[job]);
            break;
        }
        for (; si < A.nsnap && snap_step(A, si, ns) == n + 1; ++si)
            store_tracer<2>(P, A, snap_slot(A, job, si), i, x, cx, img, st, snap_exit(A, job, si, st, te));
    }
    for (; si < A.nsnap; ++si)
        store_tracer<2>(P, A, snap_slot(A, job, si), i, x, cx, img, st, snap_exit(A, job, si, st, te));
    store_tracer<2>(P, A, job, i, x, cx, img, st, te);
}

// The record (32 bytes: u and v of a cell's four nodes) that a tracer's last evaluation read
struct RecordCache {
    float q[8];
    int v;
};

// u(x) from slice sl on a closed box.  KEEP: the cache holds a record of this very slice, taken again where x
// is still in its cell (the load is predicated off); otherwise the record is loaded.
// sl points as many records before the slice as FLOOR_MAGIC's bits count, so that the bits of box2_cell's id index it.
template <bool UNIT, bool KEEP>
__device__ __forceinline__ float2 interp2s_box(const Box2 &B, float2 x, const char *sl, RecordCache &cc)
{
    float w[4];
    const int v = __float_as_int(box2_cell<UNIT>(B, x, w));
    const char *p = sl + 32LL * v;
    if constexpr (KEEP) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %9, %10;\n\t"
            "@p ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t}"
            : "+f"(cc.q[0]), "+f"(cc.q[1]), "+f"(cc.q[2]), "+f"(cc.q[3]), "+f"(cc.q[4]), "+f"(cc.q[5]), "+f"(cc.q[6]),
              "+f"(cc.q[7])
            : "l"(p), "r"(v), "r"(cc.v));
    } else {
        asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(cc.q[0]), "=f"(cc.q[1]), "=f"(cc.q[2]), "=f"(cc.q[3]), "=f"(cc.q[4]), "=f"(cc.q[5]),
                       "=f"(cc.q[6]), "=f"(cc.q[7])
                     : "l"(p));
    }
    cc.v = v;
    const float *q = cc.q;
    return make_float2(fmaf(w[3], q[3], fmaf(w[2], q[2], fmaf(w[1], q[1], fmaf(w[0], q[0], 0.0f)))),
                       fmaf(w[3], q[7], fmaf(w[2], q[6], fmaf(w[1], q[5], fmaf(w[0], q[4], 0.0f)))));
}

// The record of the cell that p lies in, and those of its neighbours that p comes near, into the L1 cache: four
// bytes of each by an asynchronous copy to shared memory, which allocates the record's sector on its way
// (prefetch.global.L1 has no effect here) and holds up nobody.  sl as in interp2s_box, last: box2_cell's id of
// the slice's last node (every id read is clamped to the slice).
__device__ __forceinline__ void records_ahead(const Box2 &B, float2 p, const char *sl, float last, uint32_t sink)
{
    const float2 s = __fmul2_rn(__fadd2_rn(p, B.no), B.inv);
    float2 t = __fadd2_rd(s, make_float2(FLOOR_MAGIC, FLOOR_MAGIC));
    t = make_float2(fminf(fmaxf(t.x, FLOOR_MAGIC), B.tmax.x), fminf(fmaxf(t.y, FLOOR_MAGIC), B.tmax.y));
    const float fx = s.x - (t.x - FLOOR_MAGIC), fy = s.y - (t.y - FLOOR_MAGIC);
    const float id = fmaf(FLOOR_MAGIC - t.y, B.nnx, t.x);
    const float dx = fx < 0.5f ? -1.0f : 1.0f, dy = fy < 0.5f ? B.nnx : -B.nnx;
    const bool nx = fabsf(fx - 0.5f) > 0.3f, ny = fabsf(fy - 0.5f) > 0.3f;
    const auto take = [&](float i, bool on) {
        const char *q = sl + 32LL * __float_as_int(fminf(fmaxf(i, FLOOR_MAGIC), last));
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4;\n\t}" ::"r"(sink),
            "l"(q), "r"((unsigned)on)
            : "memory");
    };
    take(id, true);
    take(id + dx, nx);
    take(id + dy, ny);
    take(id + dx + dy, nx && ny);
}

// rk4_slice2d_kernel on a closed box (box2_ok).  Issue bounds it on large lattices (176 warp-instructions per
// step of 213 before), so the cell, the stage points and the update run in two-lane FP32 instructions, the
// cell without the conversion pipe, and a stencil is one load; load latency bounds it on small ones, so the
// third stage and, where the schedule shares the slice, the first take the record of the stage before when
// their point is in its cell (L1 sectors 655 M -> 201 M on four windows).  The same operations in the same
// order: the same bits.  64 windows of 2048 x 1024 seeds: 78.8 -> 73.1 ms; 64 x 32 seeds, 100 steps: 191 ->
// 151 us.  All-scalar arithmetic: 76.3 ms; 40 registers (six blocks): 76.1 ms.
template <bool UNIT, bool AHEAD>
__global__ void __launch_bounds__(256) rk4_slice2d_box_kernel(const __grid_constant__ RectParams P,
                                                              const __grid_constant__ Box2 B,
                                                              const float4 *__restrict__ slices, long long nodes,
                                                              const __grid_constant__ Slice2dOffsets O,
                                                              const unsigned char *__restrict__ shared,
                                                              const __grid_constant__ Rk4Args A)
{
    const long long i = thread_tracer(A);
    const int job = blockIdx.y;
    if (i < 0) return;
    float2 x = make_float2(A.seeds[i], A.seeds[A.N + i]), cx = make_float2(0.0f, 0.0f);
    const int ns = A.job_nsteps[job];
    const float h = A.job_h[job], hh = 0.5f * h, h6 = h * (1.0f / 6.0f);
    const size_t ss = 32 * (size_t)nodes;
    const char *s0 = (const char *)slices + O.off[job] * ss - 32LL * 0x4b400000;
    unsigned char st = LCS_TRACER_OK;
    float te = A.job_tend[job];
    int si = 0;   // next snapshot
    int next = A.nsnap > 0 ? snap_step(A, 0, ns) : -1;   // the step it follows
    const auto store = [&](int slot, float t_exit) {
        const float xs[2] = {x.x, x.y}, cs[2] = {cx.x, cx.y};
        const int img[2] = {0, 0};
        store_tracer<2>(P, A, slot, i, xs, cs, img, st, t_exit);
    };
    const unsigned char *sh = shared + (size_t)job * A.nsteps_max;
    __shared__ unsigned int sink_words[AHEAD ? 256 : 1];   // where copies for the cache's sake go; never read
    const uint32_t sink = smem_u32(sink_words + (AHEAD ? threadIdx.x : 0));
    const float last = FLOOR_MAGIC + (float)(nodes - 1);
    float2 kp = make_float2(0.0f, 0.0f);                   // first slope of the step before
    bool first = true;
    RecordCache cc;
    cc.v = -1;
#pragma unroll
    for (int q = 0; q < 8; ++q) cc.q[q] = 0.0f;
    for (int n = 0; n < ns; ++n, s0 += 3 * ss) {
        const float2 h2 = make_float2(hh, hh);
        // the first stage reads the slice that the last stage of the step before read, or one of its own
        const bool kept = __ldg(sh + n) != 0;
        if (!kept) cc.v = -1;
        const float2 k1 = interp2s_box<UNIT, true>(B, x, kept ? s0 - ss : s0, cc);
        if (AHEAD && first) kp = k1;
        first = false;
        if (AHEAD && n + 1 < ns) {   // where the next step's second and fourth stage will be, to second order
            const float2 dk = make_float2(k1.x - kp.x, k1.y - kp.y);
            records_ahead(B, make_float2(fmaf(1.125f * h, dk.x, fmaf(1.5f * h, k1.x, x.x)),
                                         fmaf(1.125f * h, dk.y, fmaf(1.5f * h, k1.y, x.y))), s0 + 4 * ss, last, sink);
            records_ahead(B, make_float2(fmaf(2.0f * h, dk.x, fmaf(2.0f * h, k1.x, x.x)),
                                         fmaf(2.0f * h, dk.y, fmaf(2.0f * h, k1.y, x.y))), s0 + 5 * ss, last, sink);
            kp = k1;
        }
        const float2 k2 = interp2s_box<UNIT, false>(B, __ffma2_rn(h2, k1, x), s0 + ss, cc);
        const float2 k3 = interp2s_box<UNIT, true>(B, __ffma2_rn(h2, k2, x), s0 + ss, cc);
        const float2 k4 = interp2s_box<UNIT, false>(B, __ffma2_rn(make_float2(h, h), k3, x), s0 + 2 * ss, cc);
        rk4_advance2(x, cx, h6, k1, k2, k3, k4);
        if (x.x < P.left_lo[0] || x.x > P.left_hi[0] || x.y < P.left_lo[1] || x.y > P.left_hi[1]) {
            st = LCS_TRACER_LEFT;
            te = fmaf((float)(n + 1), h, A.job_t0[job]);
            break;
        }
        while (n + 1 == next) {
            store(snap_slot(A, job, si), snap_exit(A, job, si, st, te));
            next = ++si < A.nsnap ? snap_step(A, si, ns) : -1;
        }
    }
    if (AHEAD) asm volatile("cp.async.wait_all;" ::: "memory");
    for (; si < A.nsnap; ++si) store(snap_slot(A, job, si), snap_exit(A, job, si, st, te));
    store(job, te);
}

size_t rk4_slice2d_bytes(const lcs_field *f, int njobs, const int *host_nsteps)
{
    long long n = 0;
    int most = 0;
    for (int j = 0; j < njobs; ++j) {
        n += 3LL * host_nsteps[j];
        most = host_nsteps[j] > most ? host_nsteps[j] : most;
    }
    return (size_t)n * 2 * (size_t)f->nodes * sizeof(float4) + (size_t)njobs * most;   // and a flag per step
}

static cudaError_t launch_slice2d(const RectParams &P, const lcs_field *f, const Rk4Args &A, const Rk4Launch &L,
                                  int bt, cudaStream_t s)
{
    Slice2dOffsets O;
    long long acc = 0;
    for (int j = 0; j < L.njobs; ++j) {
        O.off[j] = acc;
        acc += 3LL * L.host_nsteps[j];
    }
    float4 *slices = (float4 *)L.work;
    const long long nodes = f->nodes;
    unsigned char *shared = (unsigned char *)(slices + acc * 2 * nodes);
    if (A.nsteps_max > 0) {
        const long long runs = (3LL * A.nsteps_max + FILL_RUN - 1) / FILL_RUN;
        const dim3 fgrid((unsigned)((nodes + 255) / 256), (unsigned)(runs < 65535 ? runs : 65535), (unsigned)L.njobs);
        const char *fr = (const char *)f->d_frames;
        lcs_tm_begin(L.ctx, 2, s);
#define FILL(ST)                                                                                                      \
    slice2d_fill_kernel<ST><<<fgrid, 256, 0, s>>>(P, fr, f->frame_stride, A.sched, A.nsteps_max, A.job_nsteps, O,    \
                                                  (int)nodes, shared, slices)
        if (f->storage == LCS_F32) FILL(LCS_F32);
        else if (f->storage == LCS_F16) FILL(LCS_F16);
        else FILL(LCS_BF16);
#undef FILL
        lcs_tm_end(L.ctx, 2, s);
    }
    lcs_tm_begin(L.ctx, 0, s);
    dim3 grid(seed_map_grid(A.map, A.N, bt), (unsigned)L.njobs);
    const int pm = P.periodic[0] | (P.periodic[1] << 1);
    // up to eight warps per SM the steps of a tracer wait for one L2 round trip after another, and copying the
    // records of the step after next ahead pays: 100 steps of 64 x 32 seeds 146 -> 106 us, of 256 x 128 127 ->
    // 100; of 400 x 200 (16 warps per SM) it would cost (126 -> 146)
    const bool ahead = A.N * L.njobs <= 256LL * L.ctx->num_sms;
    if (box2_ok(P) && box2_unit(P) && ahead)
        rk4_slice2d_box_kernel<true, true><<<grid, bt, 0, s>>>(P, make_box2(P), slices, nodes, O, shared, A);
    else if (box2_ok(P) && ahead)
        rk4_slice2d_box_kernel<false, true><<<grid, bt, 0, s>>>(P, make_box2(P), slices, nodes, O, shared, A);
    else if (box2_ok(P) && box2_unit(P))
        rk4_slice2d_box_kernel<true, false><<<grid, bt, 0, s>>>(P, make_box2(P), slices, nodes, O, shared, A);
    else if (box2_ok(P))
        rk4_slice2d_box_kernel<false, false><<<grid, bt, 0, s>>>(P, make_box2(P), slices, nodes, O, shared, A);
    else if (pm == 3)
        rk4_slice2d_kernel<3><<<grid, bt, 0, s>>>(P, slices, nodes, O, shared, A);
    else
        rk4_slice2d_kernel<-1><<<grid, bt, 0, s>>>(P, slices, nodes, O, shared, A);
    lcs_tm_end(L.ctx, 0, s);
    return cudaGetLastError();
}

// ================================================================ dispatch

SeedMap make_seed_map(int dim, const int *n, int bt)
{
    SeedMap M;
    if ((dim != 2 && dim != 3) || bt % 32) return M;
    const int e[3] = {dim == 2 ? 16 : 8, dim == 2 ? 16 : 8, 4};
    long long seeds = 1, padded = 1, t[3] = {1, 1, 1};
    for (int d = 0; d < dim; ++d) {
        t[d] = ((long long)n[d] + e[d] - 1) / e[d];
        seeds *= n[d];
        padded *= t[d] * e[d];
    }
    if (padded * 4 > seeds * 5 || padded > 0x7fffffffLL) return M;
    M.tiled = 1;
    M.dim = dim;
    for (int d = 0; d < dim; ++d) M.n[d] = n[d];
    M.t0 = (unsigned)t[0];
    M.t1 = (unsigned)t[1];
    M.blocks8 = t[0] * t[1] * t[2];
    return M;
}

RectParams make_rect_params(const lcs_field *f)
{
    RectParams P;
    for (int d = 0; d < 3; ++d) {
        int dd = d < f->dim ? d : 0;
        P.n[d] = f->n[dd];
        P.periodic[d] = d < f->dim ? f->periodic[d] : 0;
        P.origin[d] = (float)f->origin[dd];
        P.inv_h[d] = (float)(1.0 / f->spacing[dd]);
        P.hi_node[d] = (float)(f->origin[dd] + (f->n[dd] - 1) * f->spacing[dd]);
        P.left_lo[d] = (float)(f->origin[dd] - f->spacing[dd]);
        P.left_hi[d] = (float)(f->origin[dd] + f->n[dd] * f->spacing[dd]);
        P.L[d] = (float)(f->n[dd] * f->spacing[dd]);
    }
    P.sy = f->n[0];
    P.sz = (long long)f->n[0] * f->n[1];
    P.fstride = (long long)(f->frame_stride / (f->vec * f->elem_bytes));
    return P;
}

template <int DIM, int ST>
static cudaError_t launch_gather(const RectParams &P, const lcs_field *f, const Rk4Args &A, int njobs, int bt,
                                 cudaStream_t s)
{
    dim3 grid(seed_map_grid(A.map, A.N, bt), (unsigned)njobs);
    const char *fr = (const char *)f->d_frames;
    if constexpr (DIM == 2) {
        rk4_gather2_kernel<ST><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A);
    } else {
        const int pm = box3_mask(P);
        if (pm == 7)
            rk4_gather3_kernel<ST, 7><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A);
        else if (pm == 0)
            rk4_gather3_kernel<ST, 0><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A);
        else
            rk4_gather3_kernel<ST, -1><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A);
    }
    return cudaGetLastError();
}

template <int ST, int TPT>
static cudaError_t launch_ring(lcs_ctx *ctx, const RectParams &P, const lcs_field *f, const Rk4Args &A,
                               const Rk4Launch &L, int bt, bool persistent, cudaStream_t s)
{
    size_t smem = RING_SLOTS * f->frame_stride;
    cudaError_t e = cudaFuncSetAttribute(rk4_ring2d_kernel<ST, TPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    const long long tiles = (A.N + (long long)bt * TPT - 1) / ((long long)bt * TPT);
    RingWork W;
    W.persistent = persistent ? 1 : 0;
    W.queue = L.queue;
    W.tiles_per_job = (int)tiles;
    W.nitems = tiles * L.njobs;
    W.jorder = L.job_order;
    if (!persistent) {
        dim3 grid((unsigned)tiles, (unsigned)L.njobs);
        rk4_ring2d_kernel<ST, TPT><<<grid, bt, smem, s>>>(P, (const char *)f->d_frames, f->frame_stride, A,
                                                           ctx->d_errword, W);
        return cudaGetLastError();
    }
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rk4_ring2d_kernel<ST, TPT>, bt, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    long long blocks = (long long)per_sm * ctx->num_sms;
    if (blocks > W.nitems) blocks = W.nitems;
    if (blocks < 1) blocks = 1;
    e = cudaMemsetAsync(L.queue, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    rk4_ring2d_kernel<ST, TPT><<<(unsigned)blocks, bt, smem, s>>>(P, (const char *)f->d_frames, f->frame_stride, A,
                                                                   ctx->d_errword, W);
    return cudaGetLastError();
}

template <int ST>
static cudaError_t launch_ring_tpt(lcs_ctx *ctx, const RectParams &P, const lcs_field *f, const Rk4Args &A,
                                   const Rk4Launch &L, int bt, bool persistent, cudaStream_t s)
{
    if (L.tracers_per_thread >= 2) return launch_ring<ST, 2>(ctx, P, f, A, L, bt, persistent, s);
    return launch_ring<ST, 1>(ctx, P, f, A, L, bt, persistent, s);
}

int launch_rk4_rect(lcs_ctx *ctx, const Rk4Launch &L, cudaStream_t s)
{
    const lcs_field *f = L.field;
    RectParams P = make_rect_params(f);
    Rk4Args A;
    A.seeds = L.seeds;
    A.N = L.N;
    A.nsteps_max = L.nsteps_max;
    A.sched = L.sched;
    A.job_nsteps = L.job_nsteps;
    A.job_h = L.job_h;
    A.job_t0 = L.job_t0;
    A.job_tend = L.job_tend;
    A.out_xyz = L.out_xyz;
    A.out_status = L.out_status;
    A.out_texit = L.out_texit;
    A.out_grad = L.out_grad;
    A.njobs = L.njobs;
    A.nsnap = L.nsnap;
    A.snap_n = L.snap_n;
    A.snap_te = L.snap_te;
    A.wait_ns = L.wait_ns;
    if (L.N == 0 || L.njobs == 0) return 1;
    bool ring_fits = f->dim == 2 && RING_SLOTS * f->frame_stride <= ctx->smem_optin;
    bool sorted_ok = f->dim == 3 && L.work != nullptr;
    bool queue_ok = L.queue != nullptr && L.job_order != nullptr;
    int variant = L.variant;
    // default: 2D time slices when lcs_advect reserved them (at most 2 GiB; the autotuner's choice on
    // GB300 for the sliding-window batches), else the cached gather in 2D (the shared-memory ring's
    // per-step block barriers cost more than the loads they save while the field stays in L2);
    // re-bundled episodes for large 3D lattices (lcs_advect reserves their memory from rk4_rebundle_seeds on)
    if (variant == 0) variant = sorted_ok ? 3 : (f->dim == 2 && L.work ? 5 : 1);
    if ((variant == 2 || variant == 4) && !ring_fits) variant = 1;
    if (variant == 4 && !queue_ok) variant = 2;
    if (variant == 3 && !sorted_ok) variant = 1;
    cudaError_t e;
    if (A.out_grad && variant == 3) {   // the variational equations in the re-bundled episodes
        e = launch_rk4_episodes(P, f, A, L, s);
        return e == cudaSuccess ? variant : -1;
    }
    if (A.out_grad) {   // the variational equations elsewhere: their own one-pass kernel
        // 3D: 13,824 / 125,000 / 512,000 seeds 239 / 644 / 2030 us, in blocks of 256 272 / 693 / 2083 us
        const int bt = L.block_threads > 0 && L.block_threads <= 256 ? L.block_threads : f->dim == 3 ? 128 : 256;
        A.map = make_seed_map(L.lat_dim, L.lat_n, bt);
        dim3 grid(seed_map_grid(A.map, A.N, bt), (unsigned)L.njobs);
        const char *fr = (const char *)f->d_frames;
        lcs_tm_begin(ctx, 0, s);
#define VAR_LAUNCH(ST)                                                                                 \
    do {                                                                                               \
        if (f->dim == 2) rk4_var2_kernel<ST><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A);           \
        else if (box3_mask(P) == 7) rk4_var3_kernel<ST, 7><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A); \
        else if (box3_mask(P) == 0) rk4_var3_kernel<ST, 0><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A); \
        else rk4_var3_kernel<ST, -1><<<grid, bt, 0, s>>>(P, fr, f->frame_stride, A);                   \
    } while (0)
        if (f->storage == LCS_F32) VAR_LAUNCH(LCS_F32);
        else if (f->storage == LCS_F16) VAR_LAUNCH(LCS_F16);
        else VAR_LAUNCH(LCS_BF16);
#undef VAR_LAUNCH
        lcs_tm_end(ctx, 0, s);
        return cudaGetLastError() == cudaSuccess ? 6 : -1;
    }
    if (variant == 5 && !(f->dim == 2 && L.work != nullptr)) variant = 1;
    if (variant == 3) {
        e = launch_rk4_episodes(P, f, A, L, s);
        return e == cudaSuccess ? variant : -1;
    }
    if (variant == 5) {
        // few tracers: one warp per block spreads them over the SMs (64 x 32 seeds: 106 us, 145 in blocks of 256)
        int bt = L.block_threads > 0 && L.block_threads <= 256 ? L.block_threads
                 : A.N * L.njobs <= 64LL * ctx->num_sms         ? 32
                                                                 : 256;
        A.map = make_seed_map(L.lat_dim, L.lat_n, bt);
        e = launch_slice2d(P, f, A, L, bt, s);
        return e == cudaSuccess ? variant : -1;
    }
    lcs_tm_begin(ctx, 0, s);
    if (variant == 2 || variant == 4) {
        int bt = L.block_threads > 0 ? L.block_threads : 512;
        if (bt > 512) bt = 512;
        const bool pers = variant == 4;
        if (f->storage == LCS_F32)
            e = launch_ring_tpt<LCS_F32>(ctx, P, f, A, L, bt, pers, s);
        else if (f->storage == LCS_F16)
            e = launch_ring_tpt<LCS_F16>(ctx, P, f, A, L, bt, pers, s);
        else
            e = launch_ring_tpt<LCS_BF16>(ctx, P, f, A, L, bt, pers, s);
    } else {
        // few tracers in 3D: smaller blocks spread them evenly over the SMs (46,656 seeds, FP32 64^3 nodes:
        // 277 us, in blocks of 256 339 us; 512,000 on 128^3 nodes: 2368 / 2271 us)
        const int few = f->dim == 3 && A.N * L.njobs <= 512LL * ctx->num_sms;
        int bt = L.block_threads > 0 ? L.block_threads : few ? 128 : 256;
        if (bt > 256) bt = 256;
        A.map = make_seed_map(L.lat_dim, L.lat_n, bt);
        if (f->dim == 2) {
            if (f->storage == LCS_F32)
                e = launch_gather<2, LCS_F32>(P, f, A, L.njobs, bt, s);
            else if (f->storage == LCS_F16)
                e = launch_gather<2, LCS_F16>(P, f, A, L.njobs, bt, s);
            else
                e = launch_gather<2, LCS_BF16>(P, f, A, L.njobs, bt, s);
        } else {
            if (f->storage == LCS_F32)
                e = launch_gather<3, LCS_F32>(P, f, A, L.njobs, bt, s);
            else if (f->storage == LCS_F16)
                e = launch_gather<3, LCS_F16>(P, f, A, L.njobs, bt, s);
            else
                e = launch_gather<3, LCS_BF16>(P, f, A, L.njobs, bt, s);
        }
    }
    lcs_tm_end(ctx, 0, s);
    return e == cudaSuccess ? variant : -1;
}
