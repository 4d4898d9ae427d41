// mlp_train.cu -- training of the surrogate network: integrator targets, loss and
// gradients (reverse mode), Adam.
//
// Loss and gradients of a batch are one persistent kernel (one CTA per SM, 256 threads) and a sum of the
// CTAs' partial gradients.  A CTA takes tiles of 96 samples through the whole network and back with every
// operand in shared memory and every accumulator in tensor memory, so a step moves the samples, the
// weights and one set of partial gradients per CTA and no activations.
//
// All products are formed with the features as rows: Z_l[out][sample] = W_l H_l, so that a thread owns a
// feature (TMEM lane) and half the samples.  A bias is then one register, a bias gradient a running sum of
// one thread, and the BF16 activations H and gradients dZ are stored 16 bytes along the samples into
// tiles [feature][sample] that serve both as the right operand of the next layer (samples x features) and
// as the operands of the weight gradients (features x samples): the tensor core takes either of the
// two as leading, so nothing is transposed.
//
//   forward    Z_l = W_l H_l,  H_{l+1} = SiLU(Z_l + b_l) kept in shared memory (l = 0..3),  O = W_4 H_4
//   backward   dH_4 = W_4^T dO;  per layer: dH_{l+1} to registers, Z_l formed again in its place (the same
//              MMAs, so the same bits), dZ_l = dH_{l+1} SiLU'(Z_l) over H_{l+1}'s tile, then
//              dH_l = W_l^T dZ_l and dW_l += dZ_l H_l^T
//
// Tensor memory: 96 columns for the products above, 16 for dW_0 and 128 each for dW_1..3, which stay there
// over all of a CTA's tiles (96 samples a tile: 128 would not leave room for them).  dW_4 (three rows)
// is summed from the FP32 dO by the threads.
// The layer-by-layer trainer before this one (27 launches, FP32 pre-activations, activations and their
// transposes through memory) took 1.07 ms per step of 65,536 samples, loss read and Adam included; this
// one 0.120 ms (165 TFLOP/s of the 3 x 100,864 FLOP per sample).  What bounds it now is the chain of a tile
// (13 products, each waited for before its epilogue, on one tile per SM).
#include "mlp_internal.cuh"
#include "rect_device.cuh"
#include "tc_common.cuh"

#include <math.h>

#include <new>

namespace {

__device__ __forceinline__ float tanh_a(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// SiLU of a pair of pre-activations exactly as the inference kernel computes it: h = z/2 rounded to
// BF16, then h + h tanh(h) in packed BF16 arithmetic
__device__ __forceinline__ __nv_bfloat162 silu_pair(float z0, float z1)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(0.5f * z0, 0.5f * z1);
    uint32_t hu = *reinterpret_cast<uint32_t *>(&h), t, d;
    asm("tanh.approx.bf16x2 %0, %1;" : "=r"(t) : "r"(hu));
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(hu), "r"(t), "r"(hu));
    return *reinterpret_cast<__nv_bfloat162 *>(&d);
}

__device__ __forceinline__ float silu_grad_f(float z)
{
    const float s = fmaf(0.5f, tanh_a(0.5f * z), 0.5f);
    return s * fmaf(z, 1.0f - s, 1.0f);
}

struct TrainArgs {
    const void *tiles;                 // the network's operand tiles and biases (MLP_TILE_BYTES)
    const float *xyt;                  // x, y, t rows `xstride` apart
    const float *disp;                 // displacement rows `dstride` apart
    long long xstride, dstride, B;
    float cx, cy, kx, ky, omega;       // features
    float scale, wr;                   // output scale, weight of the error head
    float *part;                       // [CTAs][PART_STRIDE] partial gradients
    double *part_loss;                 // [CTAs]
    unsigned *errword;
    unsigned long long wait_ns;        // bound on a CTA's wait for the weights
};

constexpr int TN = 96;                 // samples per tile
constexpr int TH = TN / 2;             // samples per thread (two warpgroups)
__host__ __device__ constexpr uint32_t w_off(int l) { return l == 0 ? 0u : 4096u + 32768u * (uint32_t)(l - 1); }
constexpr uint32_t BIAS_OFF = 106496;
constexpr uint32_t H_BYTES = 128 * TN * 2;
constexpr uint32_t H_OFF = 108672;     // H_1..H_4, each [128 features][TN samples]
constexpr uint32_t PHI_OFF = H_OFF + 4 * H_BYTES, DO_OFF = PHI_OFF + 16 * TN * 2, OF_OFF = DO_OFF + 16 * TN * 2;
constexpr uint32_t TRAIN_SMEM = OF_OFF + 3 * TN * 4;
static_assert(H_OFF >= MLP_TILE_BYTES && H_OFF % 128 == 0 && TRAIN_SMEM <= 227 * 1024, "shared-memory plan");
constexpr uint32_t TM_WORK = 0, TM_DW0 = 96, TM_DW = 128;   // TMEM columns; dW_l at TM_DW + 128 (l - 1)

// a CTA's partial gradients: dW_1..3 as [l][column / 4][row][column % 4] (lanes = rows store float4
// side by side), dW_0 (16 columns) alike, then dW_4 [half][3][128], db [half][4][128], db_4
constexpr int P_DW0 = 3 * 16384, P_DW4 = P_DW0 + 2048, P_DB = P_DW4 + 768, P_DB4 = P_DB + 1024;
constexpr int PART_STRIDE = P_DB4 + 32;
constexpr int P_OUT = 3 * 16384 + 2048 + 384 + 512 + 3;     // sums the reduction forms

// instruction descriptor with the leading dimension of A and B: 0 = K (tile rows are M or N), 1 = M or N
__host__ __device__ constexpr uint32_t idesc_of(int N, int a_mn, int b_mn)
{
    return tc_idesc_bf16(128, N) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16);
}

// D (+)= A B over STEPS slices of K = 16; *_step: bytes from slice to slice, *_lbo / *_sbo: see tc_desc (K
// leading: lbo between 8-column blocks of K, sbo between 8-row blocks of M or N; M or N leading: lbo
// between 8-row blocks of K, sbo between 8-column blocks of M or N)
template <int STEPS>
__device__ __forceinline__ void mma_chain(uint32_t d, uint32_t a, uint32_t a_step, uint32_t a_lbo, uint32_t a_sbo,
                                          uint32_t b, uint32_t b_step, uint32_t b_lbo, uint32_t b_sbo, uint32_t idesc,
                                          bool accumulate)
{
#pragma unroll
    for (int k = 0; k < STEPS; ++k)
        tc_mma(d, tc_desc(a + k * a_step, a_lbo, a_sbo), tc_desc(b + k * b_step, b_lbo, b_sbo), idesc,
               accumulate || k > 0);
}

__global__ void __launch_bounds__(256, 1) train_step_kernel(const TrainArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t bar_w, bar, bar_end;
    __shared__ uint32_t tmem_base;
    __shared__ double red_l[4];
    __shared__ float red_g[4][3];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int g = tid >> 7, f = tid & 127;            // half of the samples, feature
    if (tid == 0) {
        mbar_init(&bar_w, 1);
        mbar_init(&bar, 1);
        mbar_init(&bar_end, 1);
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
    for (int q = tid; q < 16 * TN / 8; q += 256) {    // rows 3..15 of dO stay zero
        *reinterpret_cast<uint4 *>(smem + DO_OFF + 16 * q) = make_uint4(0, 0, 0, 0);
    }
    bool ok = !__syncthreads_or(!tc_wait(&bar_w, 0, A.errword, A.wait_ns));
    const uint32_t tm = tmem_base, us = smem_u32(smem);
    const uint32_t tw = tm + TM_WORK + ((uint32_t)((warp & 3) * 32) << 16) + TH * g;   // this thread's lane and columns
    const float *bias = reinterpret_cast<const float *>(smem + BIAS_OFF);
    float *of = reinterpret_cast<float *>(smem + OF_OFF);
    float b[4] = {0, 0, 0, 0};
    if (ok)
#pragma unroll
        for (int l = 0; l < 4; ++l) b[l] = bias[l * 128 + f];
    float db[4] = {0, 0, 0, 0}, dw4[3] = {0, 0, 0}, db4[3] = {0, 0, 0};
    double loss = 0.0;
    unsigned phase = 0;
    bool first = true;
    // wait for the MMAs committed last; false (for every thread) when the bounded wait gave up
    const auto done = [&]() {
        const bool bad = !tc_wait(&bar, phase, A.errword);
        phase ^= 1;
        const bool r = !__syncthreads_or(bad);
        tc_fence_after();
        return r;
    };
    // every thread's shared-memory writes and TMEM reads are behind it: thread 0 may issue
    const auto ready = [&]() {
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    };
    const auto h_tile = [&](int l) { return us + H_OFF + (uint32_t)(l - 1) * H_BYTES; };
    const auto layer = [&](int l) {                   // work = W_l H_l (thread 0)
        if (l == 0)
            mma_chain<1>(tm + TM_WORK, us + w_off(0), 0, 2048, 128, us + PHI_OFF, 0, 128, 256, idesc_of(TN, 0, 1), false);
        else
            mma_chain<8>(tm + TM_WORK, us + w_off(l), 4096, 2048, 128, h_tile(l), 256, 128, 2048, idesc_of(TN, 0, 1),
                         false);
    };
    const long long ntiles = (A.B + TN - 1) / TN;
    for (long long tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        const long long i = tile * TN + tid;
        const bool live = tid < TN && i < A.B;
        if (tid < TN) {                               // features -> phi [16][TN], rows 7..15 zero
            float v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            if (live) {
                const float x = A.xyt[i], y = A.xyt[A.xstride + i], t = A.xyt[2 * A.xstride + i];
                float cy;
                sincosf(A.omega * t, &v[2], &v[3]);
                sincosf(A.kx * x, &v[4], &v[5]);
                sincosf(A.ky * y, &v[6], &cy);
                v[0] = x - A.cx;
                v[1] = y - A.cy;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k)
                *reinterpret_cast<__nv_bfloat16 *>(smem + PHI_OFF + ckm_offset(16, k, tid)) =
                    __float2bfloat16_rn(k < 7 ? v[k & 7] : 0.0f);
        }
        // ---- forward
        for (int l = 0; l < 4 && ok; ++l) {
            ready();
            if (tid == 0) {
                layer(l);
                tc_commit(&bar);
            }
            ok = done();
            if (!ok) break;
            unsigned char *h = smem + H_OFF + (uint32_t)l * H_BYTES;
            const float bl = b[l];
#pragma unroll
            for (int c = 0; c < TH; c += 16) {
                float z[16];
                tmem_ld16(tw + c, z);
#pragma unroll
                for (int q = 0; q < 16; q += 8) {
                    __nv_bfloat162 p[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) p[j] = silu_pair(z[q + 2 * j] + bl, z[q + 2 * j + 1] + bl);
                    *reinterpret_cast<uint4 *>(h + ckm_offset(128, f, TH * g + c + q)) = *reinterpret_cast<uint4 *>(p);
                }
            }
        }
        if (!ok) break;
        // ---- outputs: W_4 has 16 rows; the product's rows from 16 on read what follows it and are not used
        ready();
        if (tid == 0) {
            mma_chain<8>(tm + TM_WORK, us + w_off(4), 512, 256, 128, h_tile(4), 256, 128, 2048, idesc_of(TN, 0, 1), false);
            tc_commit(&bar);
        }
        ok = done();
        if (!ok) break;
        if (warp == 0 || warp == 4) {
#pragma unroll
            for (int c = 0; c < TH; c += 16) {
                float o[16];
                tmem_ld16(tw + c, o);
                if ((tid & 31) < 3)
#pragma unroll
                    for (int j = 0; j < 16; ++j) of[(tid & 31) * TN + TH * g + c + j] = o[j];
            }
        }
        tc_fence_before();
        __syncthreads();
        if (tid < TN) {                               // loss and dL/dO of a sample
            float g0 = 0.0f, g1 = 0.0f, g2 = 0.0f;
            if (live) {
                const float s = A.scale;
                const float o0 = of[tid] + bias[512], o1 = of[TN + tid] + bias[513], o2 = of[2 * TN + tid] + bias[514];
                const float dx = A.disp[i], dy = A.disp[A.dstride + i];
                const float e0 = o0 - dx / s, e1 = o1 - dy / s;
                const float px = fmaf(s, o0, -dx), py = fmaf(s, o1, -dy);
                const float er = o2 - log10f(sqrtf(px * px + py * py) + 1e-7f);
                loss += (double)e0 * e0 + (double)e1 * e1 + (double)A.wr * er * er;
                const float inv = 1.0f / (float)A.B;
                g0 = 2.0f * e0 * inv;
                g1 = 2.0f * e1 * inv;
                g2 = 2.0f * A.wr * er * inv;
                db4[0] += g0;
                db4[1] += g1;
                db4[2] += g2;
            }
            of[tid] = g0;
            of[TN + tid] = g1;
            of[2 * TN + tid] = g2;
            __nv_bfloat16 *d = reinterpret_cast<__nv_bfloat16 *>(smem + DO_OFF);
            d[ckm_offset(16, 0, tid) / 2] = __float2bfloat16_rn(g0);
            d[ckm_offset(16, 1, tid) / 2] = __float2bfloat16_rn(g1);
            d[ckm_offset(16, 2, tid) / 2] = __float2bfloat16_rn(g2);
        }
        // ---- backward: dH_4 = W_4^T dO; meanwhile dW_4 from the FP32 dO and this thread's row of H_4
        ready();
        if (tid == 0) {
            mma_chain<1>(tm + TM_WORK, us + w_off(4), 0, 128, 256, us + DO_OFF, 0, 128, 256, idesc_of(TN, 1, 1), false);
            tc_commit(&bar);
        }
#pragma unroll
        for (int c = 0; c < TH; c += 8) {
            const int n = TH * g + c;
            const uint4 r = *reinterpret_cast<const uint4 *>(smem + H_OFF + 3 * H_BYTES + ckm_offset(128, f, n));
            const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&r);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float4 u = *reinterpret_cast<const float4 *>(of + j * TN + n);
                const float4 v = *reinterpret_cast<const float4 *>(of + j * TN + n + 4);
                const float2 h0 = __bfloat1622float2(h2[0]), h1 = __bfloat1622float2(h2[1]);
                const float2 h4 = __bfloat1622float2(h2[2]), h6 = __bfloat1622float2(h2[3]);
                dw4[j] = fmaf(u.x, h0.x, fmaf(u.y, h0.y, fmaf(u.z, h1.x, fmaf(u.w, h1.y, dw4[j]))));
                dw4[j] = fmaf(v.x, h4.x, fmaf(v.y, h4.y, fmaf(v.z, h6.x, fmaf(v.w, h6.y, dw4[j]))));
            }
        }
#pragma unroll
        for (int l = 3; l >= 0; --l) {
            if (!ok) break;
            ok = done();
            if (!ok) break;
            float dh[TH];
#pragma unroll
            for (int c = 0; c < TH; c += 16) tmem_ld16(tw + c, dh + c);
            ready();                                  // every thread holds its dH: Z_l may take its place
            if (tid == 0) {
                layer(l);
                tc_commit(&bar);
            }
            ok = done();                              // with the MMAs issued before: H_{l+1} is no longer read
            if (!ok) break;
            unsigned char *d = smem + H_OFF + (uint32_t)l * H_BYTES;
#pragma unroll
            for (int c = 0; c < TH; c += 16) {
                float z[16];
                tmem_ld16(tw + c, z);
#pragma unroll
                for (int q = 0; q < 16; q += 8) {
                    __nv_bfloat162 p[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float u0 = dh[c + q + 2 * j] * silu_grad_f(z[q + 2 * j] + b[l]);
                        const float u1 = dh[c + q + 2 * j + 1] * silu_grad_f(z[q + 2 * j + 1] + b[l]);
                        db[l] += u0 + u1;
                        p[j] = __floats2bfloat162_rn(u0, u1);
                    }
                    *reinterpret_cast<uint4 *>(d + ckm_offset(128, f, TH * g + c + q)) = *reinterpret_cast<uint4 *>(p);
                }
            }
            ready();
            if (tid == 0) {
                const uint32_t dz = h_tile(l + 1);
                if (l > 0) {                          // dH_l = W_l^T dZ_l, dW_l += dZ_l H_l^T
                    mma_chain<8>(tm + TM_WORK, us + w_off(l), 256, 128, 2048, dz, 256, 128, 2048, idesc_of(TN, 1, 1),
                                 false);
                    tc_commit(&bar);
                    mma_chain<TN / 16>(tm + TM_DW + 128 * (l - 1), dz, 4096, 2048, 128, h_tile(l), 4096, 2048, 128,
                                       idesc_of(128, 0, 0), !first);
                } else {                              // dW_0 += dZ_0 phi^T
                    mma_chain<TN / 16>(tm + TM_DW0, dz, 4096, 2048, 128, us + PHI_OFF, 512, 256, 128,
                                       idesc_of(16, 0, 0), !first);
                    tc_commit(&bar);
                }
            }
        }
        if (!ok) break;
        ok = done();                                  // the next tile overwrites phi and H_1
        first = false;
    }
    // ---- partial gradients of this CTA (every CTA has at least one tile)
    if (ok) {
        float *out = A.part + (size_t)blockIdx.x * PART_STRIDE;
        const uint32_t lane = tm + ((uint32_t)((warp & 3) * 32) << 16);
        for (int q = 0; q < 3 * 4; ++q) {             // this half's 64 columns of dW_1..3, 16 at a time
            const int l = q >> 2, c = 64 * g + 16 * (q & 3);
            float v[16];
            tmem_ld16(lane + TM_DW + 128 * l + c, v);
#pragma unroll
            for (int j = 0; j < 16; j += 4)
                *reinterpret_cast<float4 *>(out + l * 16384 + (c + j) * 128 + 4 * f) =
                    make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
        if (g == 0) {
            float v[16];
            tmem_ld16(lane + TM_DW0, v);
#pragma unroll
            for (int j = 0; j < 16; j += 4)
                *reinterpret_cast<float4 *>(out + P_DW0 + j * 128 + 4 * f) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) out[P_DW4 + g * 384 + j * 128 + f] = dw4[j];
#pragma unroll
        for (int l = 0; l < 4; ++l) out[P_DB + g * 512 + l * 128 + f] = db[l];
        for (int o = 16; o > 0; o >>= 1) {
            loss += __shfl_down_sync(0xffffffffu, loss, o);
#pragma unroll
            for (int j = 0; j < 3; ++j) db4[j] += __shfl_down_sync(0xffffffffu, db4[j], o);
        }
        if (tid < 128 && (tid & 31) == 0) {
            red_l[warp] = loss;
#pragma unroll
            for (int j = 0; j < 3; ++j) red_g[warp][j] = db4[j];
        }
        __syncthreads();
        if (tid == 0) {
            A.part_loss[blockIdx.x] = (red_l[0] + red_l[1]) + (red_l[2] + red_l[3]);
#pragma unroll
            for (int j = 0; j < 3; ++j) out[P_DB4 + j] = (red_g[0][j] + red_g[1][j]) + (red_g[2][j] + red_g[3][j]);
        }
    } else {
        mbar_wait_bounded(&bar_w, 0);                 // a wait gave up: what is in flight, the copy and all MMAs issued,
        if (tid == 0) tc_commit(&bar_end);            // ends first
        mbar_wait_bounded(&bar_end, 0);
        // nothing of an earlier batch is summed in this CTA's place, and the loss tells
        float4 *out = reinterpret_cast<float4 *>(A.part + (size_t)blockIdx.x * PART_STRIDE);
        for (int q = tid; q < PART_STRIDE / 4; q += 256) out[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (tid == 0) A.part_loss[blockIdx.x] = __longlong_as_double(0x7ff8000000000000LL);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tm, 512);
}

// grad = sum over the CTAs' partials (and over the halves of dW_4 and db), in a fixed order; four threads
// share a sum, each taking every fourth CTA.  Block 0 also sums the loss.
__global__ void __launch_bounds__(256) train_reduce_kernel(const float *__restrict__ part,
                                                           const double *__restrict__ part_loss, int nc,
                                                           float *__restrict__ grad, double *__restrict__ loss)
{
    __shared__ float s[4][64];
    const int q = threadIdx.x >> 6, o = blockIdx.x * 64 + (threadIdx.x & 63);
    int src = o, src2 = -1, dst = -1;
    if (o < P_DW0) {
        const int l = o >> 14, r = o & 16383;
        dst = MLP_OFF_W1 + l * MLP_LAYER_STRIDE + ((r >> 2) & 127) * 128 + (r >> 9) * 4 + (r & 3);
    } else if (o < P_DW4) {
        const int r = o - P_DW0, c = (r >> 9) * 4 + (r & 3);
        if (c < 7) dst = MLP_OFF_W0 + ((r >> 2) & 127) * 7 + c;
    } else if (o < P_DW4 + 384) {
        src2 = o + 384;
        dst = MLP_OFF_W4 + (o - P_DW4);
    } else if (o < P_DW4 + 384 + 512) {
        const int r = o - P_DW4 - 384;
        src = P_DB + r;
        src2 = src + 512;
        dst = MLP_OFF_B0 + (r >> 7) * MLP_LAYER_STRIDE + (r & 127);
    } else if (o < P_OUT) {
        const int r = o - P_DW4 - 384 - 512;
        src = P_DB4 + r;
        dst = MLP_OFF_B4 + r;
    }
    float a = 0.0f;
    if (dst >= 0) {
#pragma unroll 4
        for (int c = q; c < nc; c += 4) {
            const float *p = part + (size_t)c * PART_STRIDE;
            a += src2 < 0 ? p[src] : p[src] + p[src2];
        }
    }
    s[q][threadIdx.x & 63] = a;
    __syncthreads();
    if (q == 0 && dst >= 0) grad[dst] = (s[0][threadIdx.x] + s[1][threadIdx.x]) + (s[2][threadIdx.x] + s[3][threadIdx.x]);
    if (blockIdx.x == 0 && threadIdx.x == 0 && loss) {
        double t = 0.0;
        for (int c = 0; c < nc; ++c) t += part_loss[c];
        *loss = t;
    }
}

// Adam on the FP32 parameters; each new value also goes, rounded to BF16, into the operand tiles
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int n, float lr, float b1, float b2, float eps, float bc1, float bc2,
                            unsigned char *__restrict__ tiles)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = fmaf(b1, m[i], (1.0f - b1) * gi);
    const float vi = fmaf(b2, v[i], (1.0f - b2) * gi * gi);
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    p[i] = pi;
    mlp_store_param(tiles, i, pi);
}

// RK4 displacement over tau of each sample (x0, y0, t0), steps of dt; frame times FP32 in smem
template <int ST>
__global__ void __launch_bounds__(256) tr_targets_kernel(RectParams P, const char *__restrict__ frames, size_t fstride,
                                                         const double *__restrict__ times, int nf, int tp, float period,
                                                         const float *__restrict__ xyt, long long n, int S, float h,
                                                         float *__restrict__ disp)
{
    extern __shared__ float s_t[];
    for (int q = threadIdx.x; q < nf; q += blockDim.x) s_t[q] = (float)times[q];
    __syncthreads();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    float x[2] = {xyt[i], xyt[n + i]}, cx[2] = {0.0f, 0.0f};
    const float t0 = xyt[2 * n + i];
    auto bracket = [&](float t, int &k, float &a) {
        if (nf <= 1) {
            k = 0;
            a = 0.0f;
            return;
        }
        float tt = t;
        if (tp) tt = t - period * floorf((t - s_t[0]) / period);
        int lo = 0, hi = nf - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_t[mid] <= tt)
                lo = mid;
            else
                hi = mid - 1;
        }
        k = lo < nf - 2 ? lo : nf - 2;
        a = (tt - s_t[k]) / (s_t[k + 1] - s_t[k]);
        if (!tp) a = fminf(fmaxf(a, 0.0f), 1.0f);
    };
    for (int s = 0; s < S; ++s) {
        const float ts = fmaf((float)s, h, t0);
        int k0, k1, k2;
        float a0, a1, a2;
        bracket(ts, k0, a0);
        bracket(ts + 0.5f * h, k1, a1);
        bracket(ts + h, k2, a2);
        rk4_step<2, ST, SRC_GLOBAL>(P, x, cx, h, frames + (size_t)k0 * fstride, frames + (size_t)(k0 + 1) * fstride,
                                    a0, frames + (size_t)k1 * fstride, frames + (size_t)(k1 + 1) * fstride, a1,
                                    frames + (size_t)k2 * fstride, frames + (size_t)(k2 + 1) * fstride, a2);
    }
    disp[i] = (x[0] - xyt[i]) + cx[0];
    disp[n + i] = (x[1] - xyt[n + i]) + cx[1];
}

// partial gradients, their losses and the batch's loss
size_t work_bytes(int num_sms) { return (size_t)num_sms * (PART_STRIDE * sizeof(float) + sizeof(double)); }

}  // namespace

cudaError_t mlp_reserve(lcs_mlp *m, int num_sms)
{
    if (m->d_work) return cudaSuccess;
    return cudaMalloc(&m->d_work, work_bytes(num_sms));
}

// gradient of the mean loss over B samples (B a multiple of 128) into m->d_grad; summed loss into *d_loss
cudaError_t mlp_loss_grad(lcs_mlp *m, const float *xyt, long long xstride, const float *disp, long long dstride,
                          long long B, float rho_weight, int num_sms, unsigned *errword, double *d_loss, cudaStream_t s)
{
    cudaError_t e = mlp_reserve(m, num_sms);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(train_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TRAIN_SMEM);
    if (e != cudaSuccess) return e;
    TrainArgs A;
    A.tiles = m->d_tiles;
    A.xyt = xyt;
    A.xstride = xstride;
    A.disp = disp;
    A.dstride = dstride;
    A.B = B;
    A.cx = (float)m->d.center[0];
    A.cy = (float)m->d.center[1];
    A.kx = (float)m->d.kx;
    A.ky = (float)m->d.ky;
    A.omega = (float)m->d.omega;
    A.scale = (float)m->d.out_scale;
    A.wr = rho_weight;
    A.part_loss = (double *)m->d_work;
    A.part = (float *)(A.part_loss + num_sms);
    A.errword = errword;
    A.wait_ns = m->wait_ns;
    const long long tiles = (B + TN - 1) / TN;
    const int grid = (int)(tiles < num_sms ? tiles : num_sms);
    train_step_kernel<<<grid, 256, TRAIN_SMEM, s>>>(A);
    train_reduce_kernel<<<(P_OUT + 63) / 64, 256, 0, s>>>(A.part, A.part_loss, grid, m->d_grad, d_loss);
    return cudaGetLastError();
}

cudaError_t mlp_adam(lcs_mlp *m, const float *grad, double lr, double b1, double b2, double eps, cudaStream_t s)
{
    m->adam_steps += 1;
    const double bc1 = 1.0 - pow(b1, (double)m->adam_steps), bc2 = 1.0 - pow(b2, (double)m->adam_steps);
    adam_kernel<<<(MLP_NPARAMS + 255) / 256, 256, 0, s>>>(m->d_params, grad, m->d_m, m->d_v, MLP_NPARAMS, (float)lr,
                                                         (float)b1, (float)b2, (float)eps, (float)bc1, (float)bc2,
                                                         m->d_tiles);
    return cudaGetLastError();
}

cudaError_t mlp_targets(const lcs_field *f, const float *xyt, long long n, int S, double dt, float *disp, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const RectParams P = make_rect_params(f);
    const size_t smem = sizeof(float) * (size_t)(f->nframes > 0 ? f->nframes : 1);
    const unsigned grid = (unsigned)((n + 255) / 256);
    const float h = (float)dt, per = (float)f->period;
    const char *fr = (const char *)f->d_frames;
    if (f->storage == LCS_F32)
        tr_targets_kernel<LCS_F32><<<grid, 256, smem, s>>>(P, fr, f->frame_stride, f->d_times, f->nframes,
                                                          f->time_periodic, per, xyt, n, S, h, disp);
    else if (f->storage == LCS_F16)
        tr_targets_kernel<LCS_F16><<<grid, 256, smem, s>>>(P, fr, f->frame_stride, f->d_times, f->nframes,
                                                          f->time_periodic, per, xyt, n, S, h, disp);
    else
        tr_targets_kernel<LCS_BF16><<<grid, 256, smem, s>>>(P, fr, f->frame_stride, f->d_times, f->nframes,
                                                           f->time_periodic, per, xyt, n, S, h, disp);
    return cudaGetLastError();
}
