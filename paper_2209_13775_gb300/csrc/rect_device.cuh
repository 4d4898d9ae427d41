// rect_device.cuh -- device building blocks of the rectilinear advection kernels:
// storage loads, cell location, (bi/tri)linear stencils, time blending, one RK4
// step, periodic wrapping and the domain-exit test.  Included by advect_rect.cu
// and advect_episodes.cu.
#pragma once

#include "lcs_internal.cuh"

#include <math.h>

// ================================================================ node loads

// Node v of a frame -> FP32 components.  Storage: 2D = 2 components, 3D = 4
// (the 4th is padding); FP16/BF16 are widened to FP32.
template <int DIM, int ST>
struct Node;

// ld: global memory (read-only path); lds: generic address (shared or global);
// lss: shared memory only (explicit shared-space load)
__device__ __forceinline__ unsigned ld_shared_u32(const char *f, int v)
{
    unsigned r;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(smem_u32(f) + 4u * (unsigned)v));
    return r;
}

template <>
struct Node<2, LCS_F32> {
    static __device__ __forceinline__ void ld(const char *f, int v, float *u)
    {
        float2 t = __ldg(reinterpret_cast<const float2 *>(f) + v);
        u[0] = t.x;
        u[1] = t.y;
    }
    static __device__ __forceinline__ void lds(const char *f, int v, float *u)
    {
        float2 t = reinterpret_cast<const float2 *>(f)[v];
        u[0] = t.x;
        u[1] = t.y;
    }
    static __device__ __forceinline__ void lss(const char *f, int v, float *u)
    {
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(u[0]), "=f"(u[1]) : "r"(smem_u32(f) + 8u * (unsigned)v));
    }
};

__device__ __forceinline__ float2 h2f(unsigned r)
{
    __half2 h = *reinterpret_cast<__half2 *>(&r);
    return __half22float2(h);
}

__device__ __forceinline__ float2 b2f(unsigned r)
{
    __nv_bfloat162 h = *reinterpret_cast<__nv_bfloat162 *>(&r);
    return __bfloat1622float2(h);
}

template <>
struct Node<2, LCS_F16> {
    static __device__ __forceinline__ void ld(const char *f, int v, float *u)
    {
        float2 t = h2f(__ldg(reinterpret_cast<const unsigned *>(f) + v));
        u[0] = t.x;
        u[1] = t.y;
    }
    static __device__ __forceinline__ void lds(const char *f, int v, float *u)
    {
        float2 t = h2f(reinterpret_cast<const unsigned *>(f)[v]);
        u[0] = t.x;
        u[1] = t.y;
    }
    static __device__ __forceinline__ void lss(const char *f, int v, float *u)
    {
        float2 t = h2f(ld_shared_u32(f, v));
        u[0] = t.x;
        u[1] = t.y;
    }
};

template <>
struct Node<2, LCS_BF16> {
    static __device__ __forceinline__ void ld(const char *f, int v, float *u)
    {
        float2 t = b2f(__ldg(reinterpret_cast<const unsigned *>(f) + v));
        u[0] = t.x;
        u[1] = t.y;
    }
    static __device__ __forceinline__ void lds(const char *f, int v, float *u)
    {
        float2 t = b2f(reinterpret_cast<const unsigned *>(f)[v]);
        u[0] = t.x;
        u[1] = t.y;
    }
    static __device__ __forceinline__ void lss(const char *f, int v, float *u)
    {
        float2 t = b2f(ld_shared_u32(f, v));
        u[0] = t.x;
        u[1] = t.y;
    }
};

// 3D nodes are stored as interval pairs: node v of pair k holds (u_k, 0, u_{k+1}, 0),
// so one 32-byte (FP32) or 16-byte (FP16/BF16) load brings both frames of a corner.
template <int ST>
struct Pair3;

template <>
struct Pair3<LCS_F32> {
    static __device__ __forceinline__ void ld(const char *f, int v, float *ua, float *ub)
    {
        float t[8];
        asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=f"(t[0]), "=f"(t[1]), "=f"(t[2]), "=f"(t[3]), "=f"(t[4]), "=f"(t[5]), "=f"(t[6]), "=f"(t[7])
            : "l"(f + 32 * (size_t)v));
        ua[0] = t[0];
        ua[1] = t[1];
        ua[2] = t[2];
        ub[0] = t[4];
        ub[1] = t[5];
        ub[2] = t[6];
    }
};

template <>
struct Pair3<LCS_F16> {
    static __device__ __forceinline__ void ld(const char *f, int v, float *ua, float *ub)
    {
        uint4 r = __ldg(reinterpret_cast<const uint4 *>(f) + v);
        float2 a = h2f(r.x), b = h2f(r.y), c = h2f(r.z), d = h2f(r.w);
        ua[0] = a.x;
        ua[1] = a.y;
        ua[2] = b.x;
        ub[0] = c.x;
        ub[1] = c.y;
        ub[2] = d.x;
    }
};

template <>
struct Pair3<LCS_BF16> {
    static __device__ __forceinline__ void ld(const char *f, int v, float *ua, float *ub)
    {
        uint4 r = __ldg(reinterpret_cast<const uint4 *>(f) + v);
        float2 a = b2f(r.x), b = b2f(r.y), c = b2f(r.z), d = b2f(r.w);
        ua[0] = a.x;
        ua[1] = a.y;
        ua[2] = b.x;
        ub[0] = c.x;
        ub[1] = c.y;
        ub[2] = d.x;
    }
};

// ============================================================ interpolation

// Periodicity of axis d: from the compile-time mask PM when PM >= 0 (bit d set =
// periodic), else from the run-time parameters.
template <int PM>
__device__ __forceinline__ bool per_axis(const RectParams &P, int d)
{
    if constexpr (PM >= 0)
        return (PM >> d) & 1;
    else
        return P.periodic[d] != 0;
}

static __device__ __noinline__ int wrap_index_slow(int i, int n)
{
    i %= n;
    return i < 0 ? i + n : i;
}

// Cell along axis d.  Non-periodic: clamp the query into the box, cell i with
// node_i <= x < node_{i+1}, the last cell closed.  Periodic: wrap the index (one
// period up or down inline; farther only through the slow path).
template <int PM>
__device__ __forceinline__ void axis_cell(const RectParams &P, int d, float x, int &i0, int &i1, float &f)
{
    if (per_axis<PM>(P, d)) {
        float s = (x - P.origin[d]) * P.inv_h[d];
        float fl = floorf(s);
        int i = (int)fl;
        f = s - fl;
        const int n = P.n[d];
        i = i < 0 ? i + n : (i >= n ? i - n : i);
        if ((unsigned)i >= (unsigned)n) i = wrap_index_slow(i, n);
        i0 = i;
        i1 = (i + 1 == n) ? 0 : i + 1;
    } else {
        float xc = fminf(fmaxf(x, P.origin[d]), P.hi_node[d]);
        float s = (xc - P.origin[d]) * P.inv_h[d];
        int i = min((int)s, P.n[d] - 2);
        f = s - (float)i;
        i0 = i;
        i1 = i + 1;
    }
}

// Floor of s as a float and an index without the conversion pipe (float-to-int and int-to-float issue
// at an eighth of the FP32 rate): t = s + 3 * 2^22 rounded down carries floor(s) in its low mantissa
// bits for |s| < 2^22.  floor_index of such a t is floor(s); for any larger |s|, infinities and NaN it
// lies outside [-2^22, 2^22), but it is not floor(s) there (from t = 2^24 on it counts every second cell).
// So a closed axis, whose query is clamped to its nodes first, may have FLOOR_MAX_NODES of them; a periodic
// one only half as many: an index in the next period is taken as it is (less n), and must be below 2^22.
#define FLOOR_MAGIC 12582912.0f
#define FLOOR_MAX_NODES (1 << 22)
#define FLOOR_MAX_PERIODIC (1 << 21)
__device__ __forceinline__ int floor_index(float t) { return __float_as_int(t) - 0x4b400000; }

// periodicity mask of a 3D box whose axes lie within the reach of that floor, or -1
static inline int box3_mask(const RectParams &P)
{
    for (int d = 0; d < 3; ++d)
        if (P.n[d] > (P.periodic[d] ? FLOOR_MAX_PERIODIC : FLOOR_MAX_NODES)) return -1;
    return (P.periodic[0] ? 1 : 0) | (P.periodic[1] ? 2 : 0) | (P.periodic[2] ? 4 : 0);
}

// 2D box: the constants of axis_cell for both axes, packed for the two-lane FP32 instructions
struct Box2 {
    float2 no, inv, smax, tmax;    // -origin, 1 / h, the clamped query's largest s, FLOOR_MAGIC + n - 2
    float nnx;                     // -n[0]
};

// boxes that box2_cell serves: node ids and cell indices exact in its FP32 steps
static inline bool box2_ok(const RectParams &P)
{
    return !P.periodic[0] && !P.periodic[1] && (long long)P.n[0] * P.n[1] <= FLOOR_MAX_NODES;
}

static inline Box2 make_box2(const RectParams &P)
{
    Box2 B;
    B.no = make_float2(-P.origin[0], -P.origin[1]);
    B.inv = make_float2(P.inv_h[0], P.inv_h[1]);
    B.smax = make_float2((P.hi_node[0] - P.origin[0]) * P.inv_h[0], (P.hi_node[1] - P.origin[1]) * P.inv_h[1]);
    B.tmax = make_float2(FLOOR_MAGIC + (float)(P.n[0] - 2), FLOOR_MAGIC + (float)(P.n[1] - 2));
    B.nnx = -(float)P.n[0];
    return B;
}

// the largest fraction of a box's last cells is exactly 1 (its clamped query ends on node n - 1)
static inline bool box2_unit(const RectParams &P)
{
    const Box2 B = make_box2(P);
    return B.smax.x == (float)(P.n[0] - 1) && B.smax.y == (float)(P.n[1] - 1);
}

// make_stencil's node and weights on a closed box (box2_ok), both axes at once: the same values from about
// two thirds of the instructions.  axis_cell clamps x to the box and truncates s = (x - o) / h; rounding is
// monotone, so clamping s to the s of the box's ends gives the same s.  UNIT (box2_unit): the clamp to
// [0, n - 1] of s is then that of its cell to [0, n - 2] and of the fraction to [0, 1], which the
// subtraction's saturation does at no cost.  Returns the node id as FLOOR_MAGIC + id.
template <bool UNIT>
__device__ __forceinline__ float box2_cell(const Box2 &B, float2 x, float *w)
{
    float2 s = __fmul2_rn(__fadd2_rn(x, B.no), B.inv);
    if (!UNIT) s = make_float2(fminf(fmaxf(s.x, 0.0f), B.smax.x), fminf(fmaxf(s.y, 0.0f), B.smax.y));
    float2 t = __fadd2_rd(s, make_float2(FLOOR_MAGIC, FLOOR_MAGIC));
    if (UNIT)
        t = make_float2(fminf(fmaxf(t.x, FLOOR_MAGIC), B.tmax.x), fminf(fmaxf(t.y, FLOOR_MAGIC), B.tmax.y));
    else
        t = make_float2(fminf(t.x, B.tmax.x), fminf(t.y, B.tmax.y));
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 nfl = __ffma2_rn(t, m1, make_float2(FLOOR_MAGIC, FLOOR_MAGIC));   // -floor(s), exact
    const float2 f = UNIT ? make_float2(__saturatef(s.x + nfl.x), __saturatef(s.y + nfl.y)) : __fadd2_rn(s, nfl);
    const float2 g = __ffma2_rn(f, m1, make_float2(1.0f, 1.0f));
    w[0] = g.x * g.y;
    w[1] = f.x * g.y;
    w[2] = g.x * f.y;
    w[3] = f.x * f.y;
    return fmaf(nfl.y, B.nnx, t.x);
}

// rk4_advance of both coordinates
__device__ __forceinline__ void rk4_advance2(float2 &x, float2 &c, float h6, float2 k1, float2 k2, float2 k3, float2 k4)
{
    const float2 m1 = make_float2(-1.0f, -1.0f), two = make_float2(2.0f, 2.0f);
    const float2 k = __ffma2_rn(two, __fadd2_rn(k2, k3), __fadd2_rn(k1, k4));
    const float2 d = __ffma2_rn(make_float2(h6, h6), k, c);
    const float2 s = __fadd2_rn(x, d);
    c = __ffma2_rn(__ffma2_rn(x, m1, s), m1, d);
    x = s;
}

// Spatial corners and weights of x (bilinear: 4, trilinear: 8).
template <int DIM>
struct Stencil {
    int v[1 << DIM];
    float w[1 << DIM];
};

template <int DIM, int PM = -1>
__device__ __forceinline__ void make_stencil(const RectParams &P, const float *x, Stencil<DIM> &S)
{
    int i0, i1, j0, j1;
    float fx, fy;
    axis_cell<PM>(P, 0, x[0], i0, i1, fx);
    axis_cell<PM>(P, 1, x[1], j0, j1, fy);
    float gx = 1.0f - fx, gy = 1.0f - fy;
    int r0 = j0 * (int)P.sy, r1 = j1 * (int)P.sy;
    if constexpr (DIM == 2) {
        S.v[0] = i0 + r0;
        S.v[1] = i1 + r0;
        S.v[2] = i0 + r1;
        S.v[3] = i1 + r1;
        S.w[0] = gx * gy;
        S.w[1] = fx * gy;
        S.w[2] = gx * fy;
        S.w[3] = fx * fy;
    } else {
        int k0, k1;
        float fz;
        axis_cell<PM>(P, 2, x[2], k0, k1, fz);
        float gz = 1.0f - fz;
        int p0 = k0 * (int)P.sz, p1 = k1 * (int)P.sz;
        S.v[0] = i0 + r0 + p0;
        S.v[1] = i1 + r0 + p0;
        S.v[2] = i0 + r1 + p0;
        S.v[3] = i1 + r1 + p0;
        S.v[4] = i0 + r0 + p1;
        S.v[5] = i1 + r0 + p1;
        S.v[6] = i0 + r1 + p1;
        S.v[7] = i1 + r1 + p1;
        float a = gy * gz, b = fy * gz, c = gy * fz, d = fy * fz;
        S.w[0] = gx * a;
        S.w[1] = fx * a;
        S.w[2] = gx * b;
        S.w[3] = fx * b;
        S.w[4] = gx * c;
        S.w[5] = fx * c;
        S.w[6] = gx * d;
        S.w[7] = fx * d;
    }
}

// where stage frames live: global memory, any (generic address), shared memory
enum { SRC_GLOBAL = 0, SRC_GENERIC = 1, SRC_SHARED = 2 };

template <int DIM, int ST, int SRC>
__device__ __forceinline__ void node_load(const char *f, int v, float *u)
{
    if constexpr (SRC == SRC_GLOBAL)
        Node<DIM, ST>::ld(f, v, u);
    else if constexpr (SRC == SRC_GENERIC)
        Node<DIM, ST>::lds(f, v, u);
    else
        Node<DIM, ST>::lss(f, v, u);
}

// Time blend of one node, FP32: u = (1 - a) u_k + a u_{k+1} (exactly u_k when a == 0).
// Every kernel blends at the nodes first, then interpolates in space: both orders are the
// same linear map, and one order everywhere makes the kernels agree bit for bit (and lets
// a whole field be blended to a stage time once, as a time slice, with the same result).
__device__ __forceinline__ float tblend(float ua, float ub, float a, float g)
{
    return fmaf(a, ub, g * ua);
}

// u = I[(1 - a) frame fa + a frame fb](x), node blends first; frame fb is not read when a == 0
template <int DIM, int ST, int SRC>
__device__ __forceinline__ void interp(const Stencil<DIM> &S, const char *fa, const char *fb, float a, float *u)
{
    float acc[DIM], va[DIM], vb[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) acc[c] = 0.0f;
    if (a == 0.0f) {
#pragma unroll
        for (int q = 0; q < (1 << DIM); ++q) {
            node_load<DIM, ST, SRC>(fa, S.v[q], va);
#pragma unroll
            for (int c = 0; c < DIM; ++c) acc[c] = fmaf(S.w[q], va[c], acc[c]);
        }
    } else {
        const float g = 1.0f - a;
#pragma unroll
        for (int q = 0; q < (1 << DIM); ++q) {
            node_load<DIM, ST, SRC>(fa, S.v[q], va);
            node_load<DIM, ST, SRC>(fb, S.v[q], vb);
#pragma unroll
            for (int c = 0; c < DIM; ++c) acc[c] = fmaf(S.w[q], tblend(va[c], vb[c], a, g), acc[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < DIM; ++c) u[c] = acc[c];
}

// 3D: u(x, t) from the interval pair k with weight a of frame k + 1
template <int ST>
__device__ __forceinline__ void interp3p(const Stencil<3> &S, const char *fp, float a, float *u)
{
    float acc[3] = {0.0f, 0.0f, 0.0f}, va[3], vb[3];
    const float g = 1.0f - a;
    if (a == 0.0f) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            Pair3<ST>::ld(fp, S.v[q], va, vb);
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[c] = fmaf(S.w[q], va[c], acc[c]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            Pair3<ST>::ld(fp, S.v[q], va, vb);
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[c] = fmaf(S.w[q], tblend(va[c], vb[c], a, g), acc[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) u[c] = acc[c];
}

// Row of the Jacobian of a trilinear interpolant for one component: a, b its corner values on the two
// z-faces as (u(0,0), u(1,0), u(0,1), u(1,1)), f the fractions, on the per-axis factor (1 / h, or 0 where the
// query is clamped).  Differences along an axis interpolated along the other two, both x-corners in one
// two-lane instruction: 13 of them against 24 multiplications by weight derivatives.
__device__ __forceinline__ void trilinear_grad(const float4 &a, const float4 &b, const float *f, const float *on, float *J)
{
    const float2 m1 = make_float2(-1.0f, -1.0f), fy = make_float2(f[1], f[1]), fz = make_float2(f[2], f[2]);
    const float2 a0 = make_float2(a.x, a.y), b0 = make_float2(b.x, b.y);
    const float2 da = __ffma2_rn(a0, m1, make_float2(a.z, a.w)), db = __ffma2_rn(b0, m1, make_float2(b.z, b.w));
    const float2 ea = __ffma2_rn(fy, da, a0), eb = __ffma2_rn(fy, db, b0);
    const float2 g = __ffma2_rn(ea, m1, eb);
    const float2 v = __ffma2_rn(fz, g, ea), dz = __ffma2_rn(fz, __ffma2_rn(da, m1, db), da);
    J[0] = (v.y - v.x) * on[0];
    J[1] = fmaf(f[0], dz.y - dz.x, dz.x) * on[1];
    J[2] = fmaf(f[0], g.y - g.x, g.x) * on[2];
}

__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 vfma(float a, float2 b, float2 c) { return __ffma2_rn(make_float2(a, a), b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 vmul(float a, float2 b) { return __fmul2_rn(make_float2(a, a), b); }

// trilinear_grad's operations on the eight corner values u[k] (offsets k & 1, (k >> 1) & 1, k >> 2) of one
// component (V = float) or of two (float2): the same bits
template <class V>
__device__ __forceinline__ void trilinear_grad_nodes(const V *u, const float *f, const float *on, V *J)
{
    V v[2], dz[2], g[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {   // the two x-corners
        const V da = vfma(-1.0f, u[i], u[2 + i]), db = vfma(-1.0f, u[4 + i], u[6 + i]);
        const V ea = vfma(f[1], da, u[i]), eb = vfma(f[1], db, u[4 + i]);
        g[i] = vfma(-1.0f, ea, eb);
        v[i] = vfma(f[2], g[i], ea);
        dz[i] = vfma(f[2], vfma(-1.0f, da, db), da);
    }
    J[0] = vmul(on[0], vfma(-1.0f, v[0], v[1]));
    J[1] = vmul(on[1], vfma(f[0], vfma(-1.0f, dz[0], dz[1]), dz[0]));
    J[2] = vmul(on[2], vfma(f[0], vfma(-1.0f, g[0], g[1]), g[0]));
}

struct Rk4Args {
    const float *seeds;
    long long N;
    int nsteps_max;
    const SchedEntry *sched;
    const int *job_nsteps;
    const float *job_h;
    const float *job_t0;
    const float *job_tend;
    float *out_xyz;
    unsigned char *out_status;
    float *out_texit;
    float *out_grad = nullptr;       // variational grad F [njobs][N][dim][dim], or null
    int njobs = 0;                   // jobs of the call: snapshot s of job j goes to slot njobs + j nsnap + s
    int nsnap = 0;
    const int *snap_n = nullptr;     // [nsnap] snapshot step counts (device; capped per job at use)
    const float *snap_te = nullptr;  // [njobs][nsnap] snapshot end times, the exit time of a tracer OK there
    unsigned long long wait_ns = LCS_WAIT_LIMIT_NS;  // ring kernels: bound on a wait for a frame copy
    SeedMap map;                     // thread -> tracer of the one-thread-per-tracer kernels
};

// the calling thread's tracer (Rk4Args::map), or -1
__device__ __forceinline__ long long thread_tracer(const Rk4Args &A)
{
    const SeedMap &M = A.map;
    if (!M.tiled) {
        const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
        return i < A.N ? i : -1;
    }
    const unsigned wid = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const unsigned b8 = wid >> 3, w = wid & 7;
    if (b8 >= M.blocks8) return -1;
    const unsigned r = b8 / M.t0, bx = b8 - r * M.t0;
    if (M.dim == 2) {
        const unsigned x = bx * 16 + (w & 1) * 8 + (lane & 7), y = r * 16 + (w >> 1) * 4 + (lane >> 3);
        return x < (unsigned)M.n[0] && y < (unsigned)M.n[1] ? x + (long long)M.n[0] * y : -1;
    }
    const unsigned bz = r / M.t1, by = r - bz * M.t1;
    const unsigned x = bx * 8 + (w & 1) * 4 + (lane & 3), y = by * 8 + ((w >> 1) & 1) * 4 + ((lane >> 2) & 3),
                   z = bz * 4 + (w >> 2) * 2 + (lane >> 4);
    return x < (unsigned)M.n[0] && y < (unsigned)M.n[1] && z < (unsigned)M.n[2]
               ? x + (long long)M.n[0] * (y + (long long)M.n[1] * z)
               : -1;
}

// Step after which snapshot s of a job with ns steps is taken.
__device__ __forceinline__ int snap_step(const Rk4Args &A, int s, int ns) { return min(__ldg(A.snap_n + s), ns); }

__device__ __forceinline__ int snap_slot(const Rk4Args &A, int job, int s) { return A.njobs + job * A.nsnap + s; }

// exit time recorded in snapshot s of a tracer with status st and exit time te
__device__ __forceinline__ float snap_exit(const Rk4Args &A, int job, int s, unsigned char st, float te)
{
    return st == LCS_TRACER_OK ? __ldg(A.snap_te + job * A.nsnap + s) : te;
}

__device__ __forceinline__ SchedEntry load_sched(const SchedEntry *p)
{
    int2 r = __ldg(reinterpret_cast<const int2 *>(p));
    SchedEntry e;
    e.k = r.x;
    e.a = __int_as_float(r.y);
    return e;
}

// periodic axes: keep x in [origin, origin + L) with an integer count of periods; c is the
// coordinate's carried rounding (rk4_advance), which the shift's own rounding joins
template <int DIM, int PM = -1>
__device__ __forceinline__ void wrap_periodic(const RectParams &P, float *x, float *c, int *img)
{
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        if (!per_axis<PM>(P, d)) continue;
        float hiL = P.origin[d] + P.L[d];
        if (x[d] >= hiL) {
            add_carried(x[d], c[d], -P.L[d]);
            img[d] += 1;
        } else if (x[d] < P.origin[d]) {
            add_carried(x[d], c[d], P.L[d]);
            img[d] -= 1;
        }
        if (!(x[d] >= P.origin[d] && x[d] < hiL) && isfinite(x[d])) {  // far outside: full reduction
            float m = floorf((x[d] - P.origin[d]) / P.L[d]);
            add_carried(x[d], c[d], -m * P.L[d]);
            img[d] += (int)m;
            if (x[d] >= hiL) {
                x[d] = P.origin[d];
                c[d] = 0.0f;
            }
        }
    }
}

// wrap_periodic behind one test that the coordinates lie in the box, as they mostly do after a step
template <int DIM, int PM = -1>
__device__ __forceinline__ void wrap_periodic_step(const RectParams &P, float *x, float *c, int *img)
{
    bool in = true;
#pragma unroll
    for (int d = 0; d < DIM; ++d)
        if (per_axis<PM>(P, d)) in = in && x[d] >= P.origin[d] && x[d] < P.origin[d] + P.L[d];
    if (!in) wrap_periodic<DIM, PM>(P, x, c, img);
}

template <int DIM, int PM = -1>
__device__ __forceinline__ bool rect_left(const RectParams &P, const float *x)
{
    bool out = false;
#pragma unroll
    for (int d = 0; d < DIM; ++d)
        if (!per_axis<PM>(P, d)) out |= (x[d] < P.left_lo[d]) || (x[d] > P.left_hi[d]);
    return out;
}

// the flow-map coordinate of a tracer: x + c rounded once, unwrapped on periodic axes
__device__ __forceinline__ float out_coord(const RectParams &P, int d, float x, float c, int img)
{
    const float v = x + c;
    return P.periodic[d] ? fmaf((float)img, P.L[d], v) : v;
}

template <int DIM>
__device__ __forceinline__ void store_tracer(const RectParams &P, const Rk4Args &A, int job, long long i,
                                             const float *x, const float *c, const int *img, unsigned char st,
                                             float te)
{
    float *o = A.out_xyz + (size_t)job * DIM * A.N;
#pragma unroll
    for (int d = 0; d < DIM; ++d) o[d * A.N + i] = out_coord(P, d, x[d], c[d], img[d]);
    A.out_status[(size_t)job * A.N + i] = st;
    A.out_texit[(size_t)job * A.N + i] = te;
}

// one RK4 step of x (+ its carried rounding c); stage frames given by (fa, fb, a) triples
template <int DIM, int ST, int SRC>
__device__ __forceinline__ void rk4_step(const RectParams &P, float *x, float *cx, float h, const char *fa0,
                                         const char *fb0,
                                         float a0, const char *fa1, const char *fb1, float a1, const char *fa2,
                                         const char *fb2, float a2)
{
    float k1[DIM], k2[DIM], k3[DIM], k4[DIM], y[DIM];
    Stencil<DIM> S;
    const float hh = 0.5f * h;
    make_stencil<DIM>(P, x, S);
    interp<DIM, ST, SRC>(S, fa0, fb0, a0, k1);
#pragma unroll
    for (int c = 0; c < DIM; ++c) y[c] = fmaf(hh, k1[c], x[c]);
    make_stencil<DIM>(P, y, S);
    interp<DIM, ST, SRC>(S, fa1, fb1, a1, k2);
#pragma unroll
    for (int c = 0; c < DIM; ++c) y[c] = fmaf(hh, k2[c], x[c]);
    make_stencil<DIM>(P, y, S);
    interp<DIM, ST, SRC>(S, fa1, fb1, a1, k3);
#pragma unroll
    for (int c = 0; c < DIM; ++c) y[c] = fmaf(h, k3[c], x[c]);
    make_stencil<DIM>(P, y, S);
    interp<DIM, ST, SRC>(S, fa2, fb2, a2, k4);
    const float h6 = h * (1.0f / 6.0f);
#pragma unroll
    for (int c = 0; c < DIM; ++c) rk4_advance(x[c], cx[c], h6, k1[c], k2[c], k3[c], k4[c]);
}

// one RK4 step in 3D; stage s reads interval pair ps with weight as
template <int ST, int PM = -1>
__device__ __forceinline__ void rk4_step3p(const RectParams &P, float *x, float *cx, float h, const char *p0, float a0,
                                           const char *p1, float a1, const char *p2, float a2)
{
    float k1[3], k2[3], k3[3], k4[3], y[3];
    Stencil<3> S;
    const float hh = 0.5f * h;
    make_stencil<3, PM>(P, x, S);
    interp3p<ST>(S, p0, a0, k1);
#pragma unroll
    for (int c = 0; c < 3; ++c) y[c] = fmaf(hh, k1[c], x[c]);
    make_stencil<3, PM>(P, y, S);
    interp3p<ST>(S, p1, a1, k2);
#pragma unroll
    for (int c = 0; c < 3; ++c) y[c] = fmaf(hh, k2[c], x[c]);
    make_stencil<3, PM>(P, y, S);
    interp3p<ST>(S, p1, a1, k3);
#pragma unroll
    for (int c = 0; c < 3; ++c) y[c] = fmaf(h, k3[c], x[c]);
    make_stencil<3, PM>(P, y, S);
    interp3p<ST>(S, p2, a2, k4);
    const float h6 = h * (1.0f / 6.0f);
#pragma unroll
    for (int c = 0; c < 3; ++c) rk4_advance(x[c], cx[c], h6, k1[c], k2[c], k3[c], k4[c]);
}

// 3D RK4 with tracers re-bundled by cell between episodes (advect_episodes.cu)
cudaError_t launch_rk4_episodes(const RectParams &P, const lcs_field *f, const Rk4Args &A, const Rk4Launch &L,
                                cudaStream_t s);
