// mlp_infer.cu -- the surrogate network on the tcgen05 tensor cores, and the gated
// surrogate advection built on it.
//
// Network (7 -> 128 -> 128 -> 128 -> 128 -> 3, SiLU).  The features are the rows of every product, as in
// training: Z_l[out][sample] = W_l H_l, so a thread owns a feature (TMEM lane), its bias is one register
// and it stores its activations 16 bytes along the samples into the tile [feature][sample] that is the
// next product's right operand.  Per tile of NS samples the BF16 features phi(x, y, t) are one small
// operand tile, each layer one MMA chain into an FP32 TMEM accumulator, and its epilogue adds the FP32
// bias, applies SiLU (h + h tanh(h) with h = z/2, in packed BF16 arithmetic) and overwrites the layer's
// input tile.  The weights (104 KB of BF16 operand tiles) stay in shared memory for the whole persistent
// launch.  NG warpgroups work on NG tiles at a time, so a tile's epilogue overlaps the others' MMAs.
// The MUFU bounds it (two slots per tanh of a BF16 pair: 73% of its cycles, 0.23 ms at full rate for
// 2,097,229 evaluations): 0.450 ms with the samples as rows and three tiles of 128 per SM, 0.330 with the
// features as rows and six tiles of 64, 0.322 with weights in tensor memory and points loaded ahead (657
// TFLOP/s).  48 x 8: 0.344; 96 x 4: 0.343; 128 x 3: 0.364; 64 x 5: 0.369.
//
// Gated advection over one surrogate step tau (the audit of each 32-tracer group against
// the integrator of Eq. 2, and the integrator where the audit fails) runs in two SIMT
// kernels after the network: an audit kernel with one thread per group, and an apply
// kernel with one thread per tracer that either takes the proposal or integrates the
// sub-interval with the same RK4 arithmetic as the fixed-step path.
#include "mlp_internal.cuh"
#include "rect_device.cuh"
#include "tc_common.cuh"

#include <math.h>

namespace {

__host__ __device__ constexpr uint32_t w_off(int l) { return l == 0 ? 0u : 4096u + 32768u * (uint32_t)(l - 1); }
constexpr uint32_t OFF_BIAS = 106496;
constexpr uint32_t OFF_WG = 108672;    // per-warpgroup regions: activations [128][NS], then phi [16][NS]
constexpr int NS = 64, NG = 6;         // samples per tile, warpgroups (tiles in flight) per CTA
constexpr int TW = 2;                  // hidden layers whose weights the products take from tensor memory
constexpr uint32_t TM_ACC = 64 * TW;   // TMEM: W1..W_TW (64 columns each), then an accumulator per warpgroup
constexpr uint32_t ACT_BYTES = 128 * NS * 2, WG_BYTES = ACT_BYTES + 16 * NS * 2;
constexpr uint32_t INFER_SMEM = OFF_WG + NG * WG_BYTES;
static_assert(INFER_SMEM <= 226 * 1024 && TM_ACC + NG * NS <= 512 && NS % 16 == 0, "shared and tensor memory");

__device__ __forceinline__ void wg_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}

__device__ __forceinline__ uint32_t tanh_bf16x2(uint32_t h)
{
    uint32_t t;
    asm("tanh.approx.bf16x2 %0, %1;" : "=r"(t) : "r"(h));
    return t;
}

__device__ __forceinline__ uint32_t fma_bf16x2(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// one hidden layer's epilogue for feature f of a tile: h = z/2 = acc/2 + b/2 (hb = b/2) rounded to BF16
// pairs, SiLU(z) = h + h tanh(h) in packed BF16 arithmetic, stored as row f of the next operand tile
__device__ __forceinline__ void hidden_epilogue(uint32_t ta, float hb, unsigned char *tile, int f)
{
    const float2 half = make_float2(0.5f, 0.5f), b2 = make_float2(hb, hb);
#pragma unroll
    for (int c0 = 0; c0 < NS; c0 += 16) {
        float acc[16];
        tmem_ld16(ta + c0, acc);
#pragma unroll
        for (int c = 0; c < 16; c += 8) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 h = __ffma2_rn(make_float2(acc[c + 2 * j], acc[c + 2 * j + 1]), half, b2);
                const uint32_t h2 = pack_bf16(h.x, h.y);
                w[j] = fma_bf16x2(h2, tanh_bf16x2(h2), h2);
            }
            *reinterpret_cast<uint4 *>(tile + ckm_offset(128, f, c0 + c)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

__global__ void __launch_bounds__(NG * 128, 1) mlp_step_kernel(const MlpStepArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t bar_w, bar_g[NG];
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag[NG];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int g = warp >> 2;           // warpgroup
    const int f = tid & 127;           // feature = TMEM lane
    if (tid == 0) {
        mbar_init(&bar_w, 1);
        for (int q = 0; q < NG; ++q) {
            mbar_init(&bar_g[q], 1);
            abort_flag[q] = 0;
        }
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) {
        mbar_arrive_expect_tx(&bar_w, MLP_TILE_BYTES);
        bulk_g2s(smem, A.tiles, MLP_TILE_BYTES, &bar_w);
    }
    const bool have_w = !__syncthreads_or(!tc_wait(&bar_w, 0, A.errword, A.wait_ns));
    const uint32_t tmem = tmem_base + TM_ACC + (uint32_t)(g * NS);
    unsigned char *sAct = smem + OFF_WG + g * WG_BYTES;
    unsigned char *sPhi = sAct + ACT_BYTES;
    float *sOut = reinterpret_cast<float *>(sPhi);     // [3][NS] outputs (phi is done by then)
    const float *bias = reinterpret_cast<const float *>(smem + OFF_BIAS);
    const uint32_t uPhi = smem_u32(sPhi), uAct = smem_u32(sAct), uW = smem_u32(smem);
    // A (weights) with K leading, B (activations, features) with the samples leading: descriptor bit 16
    const uint32_t idesc = tc_idesc_bf16(128, NS) | (1u << 16);
    float hb[4] = {0.0f, 0.0f, 0.0f, 0.0f};            // hidden-layer biases, halved
    if (have_w)
#pragma unroll
        for (int l = 0; l < 4; ++l) hb[l] = 0.5f * bias[l * 128 + f];
    // W1 and W2 into tensor memory, where the products take them from: read from shared memory by every MMA
    // they are 4 KB of its 6 KB (0.328 ms with all of them there, 0.325 with W1 moved, 0.322 with both; a
    // third leaves room for five accumulators only: 0.347)
    if (have_w && g < TW) {
        const uint32_t tw = tmem_base + 64 * g + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll
        for (int c = 0; c < 64; c += 16) {
            uint32_t r[16];
#pragma unroll
            for (int q = 0; q < 16; q += 4)
                *reinterpret_cast<uint4 *>(r + q) =
                    *reinterpret_cast<const uint4 *>(smem + w_off(1 + g) + ckm_offset(128, f, 2 * (c + q)));
            tmem_st16(tw + c, r);
        }
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const long long ntiles = (A.n + NS - 1) / NS;
    unsigned phase = 0;
    // a tile's points are loaded while the tile before it goes through the network
    float px = 0.0f, py = 0.0f, pt = A.t_uniform;
    const auto load = [&](long long tile) {
        const long long i = tile * NS + f;
        if (f < NS && i < A.n) {
            px = A.x[i];
            py = A.x[A.stride + i];
            if (A.t) pt = A.t[i];
        }
    };
    load(blockIdx.x + (long long)gridDim.x * g);
    for (long long tile = blockIdx.x + (long long)gridDim.x * g; have_w && tile < ntiles;
         tile += (long long)NG * gridDim.x) {
        const long long i = tile * NS + f;
        const bool live = f < NS && i < A.n;
        const float x = px, y = py, t = pt;
        if (f < NS) {   // features -> BF16 column f of the phi tile (K = 16, rows 7..15 zero)
            float v[8];
            float cy;
            sincosf(A.omega * t, &v[2], &v[3]);
            sincosf(A.kx * x, &v[4], &v[5]);
            sincosf(A.ky * y, &v[6], &cy);
            v[0] = x - A.cx;
            v[1] = y - A.cy;
            v[7] = 0.0f;
#pragma unroll
            for (int k = 0; k < 16; ++k)
                *reinterpret_cast<__nv_bfloat16 *>(sPhi + ckm_offset(16, k, f)) = __float2bfloat16_rn(k < 7 ? v[k & 7] : 0.0f);
        }
        load(tile + (long long)NG * gridDim.x);
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            fence_async_smem();
            tc_fence_before();
            wg_sync(g);
            if (f == 0) {
                tc_fence_after();
                if (l == 0) {
                    tc_mma(tmem, tc_desc(uW, 2048, 128), tc_desc(uPhi, 128, 256), idesc, false);
                } else {
                    // W4 has 16 rows: the product's rows from 16 on read what follows it and are not used
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        if (l <= TW)
                            tc_mma_ts(tmem, tmem_base + 64 * (l - 1) + 8 * kk, tc_desc(uAct + kk * 256, 128, 2048),
                                      idesc, kk > 0);
                        else
                            tc_mma(tmem, l < 4 ? tc_desc(uW + w_off(l) + kk * 4096, 2048, 128)
                                               : tc_desc(uW + w_off(4) + kk * 512, 256, 128),
                                   tc_desc(uAct + kk * 256, 128, 2048), idesc, kk > 0);
                }
                tc_commit(&bar_g[g]);
            }
            if (!tc_wait(&bar_g[g], phase, A.errword)) abort_flag[g] = 1;
            phase ^= 1;
            wg_sync(g);  // every thread of the warpgroup sees the same abort flag
            if (abort_flag[g]) break;
            tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16);
            if (l < 4) {
                hidden_epilogue(ta, hb[l], sAct, f);
            } else if ((warp & 3) == 0) {
                const float bo = f < 3 ? bias[512 + f] : 0.0f;
#pragma unroll
                for (int c = 0; c < NS; c += 16) {
                    float v[16];
                    tmem_ld16(ta + c, v);
                    if (f < 3)
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            *reinterpret_cast<float4 *>(sOut + f * NS + c + j) =
                                make_float4(v[j] + bo, v[j + 1] + bo, v[j + 2] + bo, v[j + 3] + bo);
                }
            }
        }
        if (abort_flag[g]) break;
        wg_sync(g);
        const float o[3] = {sOut[f % NS], sOut[NS + f % NS], sOut[2 * NS + f % NS]};
        if (live) {
            if (A.mode == 0) {
                A.out0[i] = o[0];
                A.out1[i] = o[1];
                A.out2[i] = o[2];
            } else {
                A.out0[i] = fmaf(A.out_scale, o[0], x);
                A.out1[i] = fmaf(A.out_scale, o[1], y);
                A.out2[i] = o[2];
            }
        }
        wg_sync(g);   // the outputs are read before the next tile's features take their place
    }
    if (!have_w) mbar_wait_bounded(&bar_w, 0);         // a wait gave up: what is in flight ends first
    else if (abort_flag[g]) mbar_wait_bounded(&bar_g[g], phase ^ 1);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem_base, 512);
}

// one thread per 32-tracer group: audit lane's RK4 over the sub-interval vs its proposal,
// and the group's largest predicted error; flag = 1 sends the group to the integrator
template <int ST>
__global__ void __launch_bounds__(256) sur_audit_kernel(SurGateArgs G, RectParams P, const char *__restrict__ frames,
                                                        size_t fstride)
{
    const long long grp = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long ngrp = (G.n + 31) / 32;
    if (grp >= ngrp) return;
    const long long i0 = grp * 32;
    const int m = (int)(G.n - i0 < 32 ? G.n - i0 : 32);
    bool fall = false;
    for (int q = 0; q < m; ++q)
        if (G.rho[i0 + q] > G.log_tol || !(G.rho[i0 + q] == G.rho[i0 + q])) fall = true;
    const long long a = i0 + (long long)(lowbias32(lowbias32((unsigned)G.step) ^ (unsigned)grp) % (unsigned)m);
    if (!fall && G.status[a] == LCS_TRACER_OK && G.tol < INFINITY) {
        float x[2] = {G.xyz[a], G.xyz[G.n + a]}, c[2] = {G.cxy[a], G.cxy[G.n + a]};
        const SchedEntry *sc = G.sched + (size_t)G.step * G.S * 3;
        for (int n = 0; n < G.S; ++n) {
            SchedEntry e0 = load_sched(sc + 3 * n), e1 = load_sched(sc + 3 * n + 1), e2 = load_sched(sc + 3 * n + 2);
            rk4_step<2, ST, SRC_GLOBAL>(P, x, c, G.h, frames + (size_t)e0.k * fstride,
                                        frames + (size_t)(e0.k + 1) * fstride, e0.a, frames + (size_t)e1.k * fstride,
                                        frames + (size_t)(e1.k + 1) * fstride, e1.a, frames + (size_t)e2.k * fstride,
                                        frames + (size_t)(e2.k + 1) * fstride, e2.a);
        }
        const float dx = G.xp[a] - (x[0] + c[0]), dy = G.xp[G.n + a] - (x[1] + c[1]);
        const float res = sqrtf(dx * dx + dy * dy);
        fall = !(res <= G.tol);
    }
    G.flag[grp] = fall ? 1 : 0;
}

// one thread per tracer: take the proposal, or integrate the sub-interval where the group failed
template <int ST>
__global__ void __launch_bounds__(256) sur_apply_kernel(SurGateArgs G, RectParams P, const char *__restrict__ frames,
                                                        size_t fstride)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= G.n || G.status[i] != LCS_TRACER_OK) return;
    float x[2], c[2] = {0.0f, 0.0f};
    const int step = G.step;
    if (G.flag[i >> 5]) {
        x[0] = G.xyz[i];
        x[1] = G.xyz[G.n + i];
        c[0] = G.cxy[i];
        c[1] = G.cxy[G.n + i];
        const SchedEntry *sc = G.sched + (size_t)step * G.S * 3;
        for (int n = 0; n < G.S; ++n) {
            SchedEntry e0 = load_sched(sc + 3 * n), e1 = load_sched(sc + 3 * n + 1), e2 = load_sched(sc + 3 * n + 2);
            rk4_step<2, ST, SRC_GLOBAL>(P, x, c, G.h, frames + (size_t)e0.k * fstride,
                                        frames + (size_t)(e0.k + 1) * fstride, e0.a, frames + (size_t)e1.k * fstride,
                                        frames + (size_t)(e1.k + 1) * fstride, e1.a, frames + (size_t)e2.k * fstride,
                                        frames + (size_t)(e2.k + 1) * fstride, e2.a);
            if (rect_left<2>(P, x)) {
                G.status[i] = LCS_TRACER_LEFT;
                G.texit[i] = fmaf((float)(step * G.S + n + 1), G.h, G.t0);
                break;
            }
        }
        G.counts[i] += 1;
    } else {
        x[0] = G.xp[i];
        x[1] = G.xp[G.n + i];
        if (rect_left<2>(P, x)) {
            G.status[i] = LCS_TRACER_LEFT;
            G.texit[i] = fmaf((float)((step + 1) * G.S), G.h, G.t0);
        }
    }
    G.xyz[i] = x[0];
    G.xyz[G.n + i] = x[1];
    G.cxy[i] = c[0];   // a proposal starts without a carried rounding
    G.cxy[G.n + i] = c[1];
}

__global__ void fill_f32_kernel(float *p, long long n, float v)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

// x + c rounded once: the flow map of the surrogate path, as the fixed-step kernels store it
__global__ void settle_f32_kernel(float *x, const float *c, long long n)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) x[i] = x[i] + c[i];
}

}  // namespace

cudaError_t launch_fill_f32(float *p, long long n, float v, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    fill_f32_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p, n, v);
    return cudaGetLastError();
}

cudaError_t launch_settle_f32(float *x, const float *c, long long n, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    settle_f32_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, c, n);
    return cudaGetLastError();
}

cudaError_t launch_mlp_step(const MlpStepArgs &A, int num_sms, cudaStream_t s)
{
    if (A.n <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(mlp_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)INFER_SMEM);
    if (e != cudaSuccess) return e;
    const long long tiles = (A.n + NS - 1) / NS;
    const int grid = (int)(tiles < num_sms ? tiles : num_sms);
    mlp_step_kernel<<<grid, NG * 128, INFER_SMEM, s>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_sur_gate(const SurGateArgs &G, const lcs_field *f, cudaStream_t s)
{
    if (G.n <= 0) return cudaSuccess;
    const RectParams P = make_rect_params(f);
    const char *fr = (const char *)f->d_frames;
    const long long ngrp = (G.n + 31) / 32;
    const unsigned ga = (unsigned)((ngrp + 255) / 256), gt = (unsigned)((G.n + 255) / 256);
    if (f->storage == LCS_F32) {
        sur_audit_kernel<LCS_F32><<<ga, 256, 0, s>>>(G, P, fr, f->frame_stride);
        sur_apply_kernel<LCS_F32><<<gt, 256, 0, s>>>(G, P, fr, f->frame_stride);
    } else if (f->storage == LCS_F16) {
        sur_audit_kernel<LCS_F16><<<ga, 256, 0, s>>>(G, P, fr, f->frame_stride);
        sur_apply_kernel<LCS_F16><<<gt, 256, 0, s>>>(G, P, fr, f->frame_stride);
    } else {
        sur_audit_kernel<LCS_BF16><<<ga, 256, 0, s>>>(G, P, fr, f->frame_stride);
        sur_apply_kernel<LCS_BF16><<<gt, 256, 0, s>>>(G, P, fr, f->frame_stride);
    }
    return cudaGetLastError();
}
