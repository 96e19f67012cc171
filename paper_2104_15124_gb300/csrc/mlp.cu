// Learned radius (step a7): a small MLP in -> 64 -> 64 -> 1 with GELU (erf form)
// that predicts log r_k, the log distance from a point to its k-th neighbour,
// from the point's coordinates.  The kNN search uses exp(prediction) as a
// per-point radius guess; the search stays exact whatever the guess.
//
// Forward passes read BF16 weights (a round-to-nearest copy of the FP32
// master) and compute in FP32.  Training: eight threads per sample for the
// forward and the per-sample backward vectors; the weight gradients, sums of
// per-sample outer products, are formed block-wide from shared-memory copies of
// those vectors, written as per-block partials and reduced in a fixed order, so
// a training run is bitwise reproducible.  The reduction applies Adam to the FP32
// master and refreshes the BF16 copy.
#include "vb_internal.cuh"
#include "tc.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

namespace vb {

constexpr int H = VB_MLP_HIDDEN;

__host__ __device__ inline int param_count(int in) { return H * in + H + H * H + H + H + 1; }

struct MlpK {
    int in;
    const __nv_bfloat16* wb;
    float mean[VB_MLP_MAX_IN], scale[VB_MLP_MAX_IN];
    float out_mean, out_scale;
};

static MlpK mk(const vb_mlp* m)
{
    MlpK k;
    k.in = m->in_dim;
    k.wb = (const __nv_bfloat16*)m->weights;
    for (int r = 0; r < VB_MLP_MAX_IN; ++r) {
        k.mean[r] = r < m->in_dim ? m->in_mean[r] : 0.f;
        k.scale[r] = r < m->in_dim && m->in_scale[r] != 0.f ? m->in_scale[r] : 1.f;
    }
    k.out_mean = m->out_mean;
    k.out_scale = m->out_scale != 0.f ? m->out_scale : 1.f;
    return k;
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float z)
{
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// parameter offsets
struct Off {
    int w1, b1, w2, b2, w3, b3;
    __host__ __device__ explicit Off(int in)
    {
        w1 = 0;
        b1 = H * in;
        w2 = b1 + H;
        b2 = w2 + H * H;
        w3 = b2 + H;
        b3 = w3 + H;
    }
};

// Loads the BF16 weights into shared memory as FP32.
__device__ __forceinline__ void load_weights(const MlpK& k, float* W)
{
    const int P = param_count(k.in);
    for (int e = threadIdx.x; e < P; e += blockDim.x) W[e] = __bfloat162float(k.wb[e]);
}

__device__ __forceinline__ void standardise(const MlpK& k, const float* x, int ld, int64_t row, float* xin)
{
    for (int r = 0; r < k.in; ++r) xin[r] = (x[row * ld + r] - k.mean[r]) / k.scale[r];
}

// Forward pass for inference: the hidden layer stays in registers and the second layer is
// folded into the output as it is formed (no per-sample arrays in local memory).
__device__ __forceinline__ float forward_infer(const MlpK& k, const float* W, const float* xin)
{
    const Off o(k.in);
    float h1[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
        float s = W[o.b1 + j];
        for (int r = 0; r < k.in; ++r) s = fmaf(W[o.w1 + j * k.in + r], xin[r], s);
        h1[j] = gelu(s);
    }
    float out = W[o.b3];
    for (int j = 0; j < H; ++j) {
        float s = W[o.b2 + j];
#pragma unroll
        for (int i = 0; i < H; ++i) s = fmaf(W[o.w2 + j * H + i], h1[i], s);
        out = fmaf(W[o.w3 + j], gelu(s), out);
    }
    return out;
}

// ------------------------------------------------------------------ inference
__global__ void __launch_bounds__(128) mlp_predict_kernel(MlpK k, const float* __restrict__ x, int ld, int64_t n,
                                                          float* y, int mode, float shift, float inflate,
                                                          const float* __restrict__ cloud_shift, Clouds cl)
{
    extern __shared__ float W[];
    load_weights(k, W);
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float xin[VB_MLP_MAX_IN];
        standardise(k, x, ld, i, xin);
        const float logr = k.out_mean + k.out_scale * forward_infer(k, W, xin);
        if (mode == 0) {
            y[i] = logr;
        } else {   // squared radius bound for the radius-first kNN search
            const float sh = cloud_shift ? shift + cloud_shift[cloud_of(cl.ptr, cl.B, i)] : shift;
            const float r = expf(logr + sh) * inflate;
            y[i] = __fmul_ru(r, r);
        }
    }
}

// ------------------------------------------------------------------ training
// Per-block partial gradients over rows [r0, r1) of (x, y): part[blockIdx][P], then the loss.
// scale_g multiplies the gradient of sum_i (net(x_i) - y_std_i)^2 (1/batch for a mean).
//
// A block takes GS = 32 samples at a time, eight threads each (a quarter warp: the layers of a sample
// need no block barrier), so a minibatch of 4,096 is 128 blocks of eight warps; with one thread per
// sample it was 32 blocks of four, each with its activations in local memory.  Thread g of a sample forms
// the hidden units g, g + 8, ... (rows of W2 68 floats apart: eight 16-byte reads in one pass over the
// banks); going back it forms units 8 g .. 8 g + 7 from 16-byte pieces of W2's rows.  The weight gradients
// are outer products summed over the 32 samples, a 4 x 4 patch of W2 per thread.  Bound by
// shared-memory reads.  An epoch of 25 minibatches of 4,096 samples in R^4, with Adam in the reduction:
// 4.16 -> 0.67 ms.
constexpr int GS = 32, GT = 256, GLD = H + 4;   // samples, threads, padded row length
constexpr int GRAD_SMEM_FLOATS = H * VB_MLP_MAX_IN + H * GLD + 3 * H + GS * VB_MLP_MAX_IN + 4 * GS * GLD;

__global__ void __launch_bounds__(GT) mlp_grad_kernel(MlpK k, const float* __restrict__ x, int ld,
                                                      const float* __restrict__ y, int64_t r0, int64_t r1,
                                                      float scale_g, float* part)
{
    extern __shared__ __align__(16) float sm[];
    float* W1 = sm;                              // [H][in]
    float* W2 = W1 + H * VB_MLP_MAX_IN;          // [H][GLD]
    float* b1 = W2 + H * GLD;
    float* b2 = b1 + H;
    float* w3 = b2 + H;
    float* sx = w3 + H;                          // [GS][16]
    float* sh1 = sx + GS * VB_MLP_MAX_IN;        // [GS][GLD] first hidden layer
    float* sd1 = sh1 + GS * GLD;                 // its derivative, then d loss / d z1
    float* sd2 = sd1 + GS * GLD;                 // d loss / d z2
    float* sh2 = sd2 + GS * GLD;                 // second hidden layer
    __shared__ float sdo[GS], slo[GS];
    const Off o(k.in);
    const int t = threadIdx.x, in = k.in, P = param_count(in);
    for (int e = t; e < H * in; e += GT) W1[e] = __bfloat162float(k.wb[o.w1 + e]);
    for (int e = t; e < H * H; e += GT) W2[(e / H) * GLD + e % H] = __bfloat162float(k.wb[o.w2 + e]);
    if (t < H) {
        b1[t] = __bfloat162float(k.wb[o.b1 + t]);
        b2[t] = __bfloat162float(k.wb[o.b2 + t]);
        w3[t] = __bfloat162float(k.wb[o.w3 + t]);
    }
    const float b3 = __bfloat162float(k.wb[o.b3]);
    const int s = t / 8, g = t % 8;              // sample and thread of it
    const int j0 = (t / 16) * 4, i0 = (t % 16) * 4;   // the patch of W2's gradient
    // sums of the last 128 samples, and of those before: a block takes 6,600 samples of a million, and one running
    // FP32 sum over them would round as often
    float a2[4][4] = {}, a1[4] = {}, av = 0.f, lsum = 0.f, t2[4][4] = {}, t1[4] = {}, tv = 0.f, tl = 0.f;
    int held = 0;
    auto fold = [&]() {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                t2[a][b] += a2[a][b];
                a2[a][b] = 0.f;
            }
            t1[a] += a1[a];
            a1[a] = 0.f;
        }
        tv += av;
        tl += lsum;
        av = lsum = 0.f;
        held = 0;
    };
    for (int64_t base = r0 + (int64_t)blockIdx.x * GS; base < r1; base += (int64_t)gridDim.x * GS) {
        const int64_t row = base + s;
        const bool ok = row < r1;
        __syncthreads();   // the weights are loaded; the previous samples' sums are done
        for (int r = g; r < in; r += 8) sx[s * VB_MLP_MAX_IN + r] = ok ? (x[row * ld + r] - k.mean[r]) / k.scale[r] : 0.f;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = g + 8 * u;
            float z = b1[j];
            for (int r = 0; r < in; ++r) z = fmaf(W1[j * in + r], sx[s * VB_MLP_MAX_IN + r], z);
            sh1[s * GLD + j] = gelu(z);
            sd1[s * GLD + j] = gelu_d(z);
        }
        __syncwarp();
        float z2[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) z2[u] = b2[g + 8 * u];
#pragma unroll 4
        for (int i = 0; i < H; i += 4) {
            const float4 h = *(const float4*)(sh1 + s * GLD + i);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float4 w = *(const float4*)(W2 + (g + 8 * u) * GLD + i);
                z2[u] = fmaf(w.x, h.x, z2[u]);
                z2[u] = fmaf(w.y, h.y, z2[u]);
                z2[u] = fmaf(w.z, h.z, z2[u]);
                z2[u] = fmaf(w.w, h.w, z2[u]);
            }
        }
        float out = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float h2 = gelu(z2[u]);
            out = fmaf(w3[g + 8 * u], h2, out);
            sh2[s * GLD + g + 8 * u] = ok ? h2 : 0.f;
        }
#pragma unroll
        for (int q = 4; q > 0; q >>= 1) out += __shfl_xor_sync(0xffffffffu, out, q);
        out += b3;
        const float e = ok ? out - (y[row] - k.out_mean) / k.out_scale : 0.f;
        const float dout = 2.f * e * scale_g;
        if (g == 0) {
            sdo[s] = dout;
            lsum += e * e;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) sd2[s * GLD + g + 8 * u] = dout * w3[g + 8 * u] * gelu_d(z2[u]);
        __syncwarp();
        float d1[8] = {};
#pragma unroll 4
        for (int j = 0; j < H; ++j) {
            const float d = sd2[s * GLD + j];
            const float4 w0 = *(const float4*)(W2 + j * GLD + 8 * g), w1 = *(const float4*)(W2 + j * GLD + 8 * g + 4);
            d1[0] = fmaf(w0.x, d, d1[0]);
            d1[1] = fmaf(w0.y, d, d1[1]);
            d1[2] = fmaf(w0.z, d, d1[2]);
            d1[3] = fmaf(w0.w, d, d1[3]);
            d1[4] = fmaf(w1.x, d, d1[4]);
            d1[5] = fmaf(w1.y, d, d1[5]);
            d1[6] = fmaf(w1.z, d, d1[6]);
            d1[7] = fmaf(w1.w, d, d1[7]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) sd1[s * GLD + 8 * g + u] *= d1[u];
        __syncthreads();
        // weight gradients over the 32 samples
#pragma unroll 4
        for (int q = 0; q < GS; ++q) {
            const float4 d = *(const float4*)(sd2 + q * GLD + j0), h = *(const float4*)(sh1 + q * GLD + i0);
            const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) a2[a][b] = fmaf(dv[a], hv[b], a2[a][b]);
        }
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {   // W1: at most 4 of the H in entries per thread
            const int e1 = t + q4 * GT;
            if (e1 < H * in) {
                const int j = e1 / in, r = e1 - j * in;
                for (int q = 0; q < GS; ++q) a1[q4] = fmaf(sd1[q * GLD + j], sx[q * VB_MLP_MAX_IN + r], a1[q4]);
            }
        }
        const int j = t & (H - 1);   // b1, b2, w3: 64 threads each, then b3
        if (t < H)
            for (int q = 0; q < GS; ++q) av += sd1[q * GLD + j];
        else if (t < 2 * H)
            for (int q = 0; q < GS; ++q) av += sd2[q * GLD + j];
        else if (t < 3 * H)
            for (int q = 0; q < GS; ++q) av = fmaf(sdo[q], sh2[q * GLD + j], av);
        else if (t == 3 * H)
            for (int q = 0; q < GS; ++q) av += sdo[q];
        if (++held == 128 / GS) fold();
    }
    fold();
    float* pb = part + (int64_t)blockIdx.x * (P + 1);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) pb[o.w2 + (j0 + a) * H + i0 + b] = t2[a][b];
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4)
        if (t + q4 * GT < H * in) pb[o.w1 + t + q4 * GT] = t1[q4];
    if (t < H) pb[o.b1 + t] = tv;
    else if (t < 2 * H) pb[o.b2 + t - H] = tv;
    else if (t < 3 * H) pb[o.w3 + t - 2 * H] = tv;
    else if (t == 3 * H) pb[o.b3] = tv;
    if (g == 0) slo[s] = tl;
    __syncthreads();
    if (t == 0) {
        float l = 0.f;
        for (int q = 0; q < GS; ++q) l += slo[q];
        pb[P] = l;
    }
}

struct AdamK {
    float* master;   // null: no update
    __nv_bfloat16* wb;
    float *m1, *m2;
    float lr, bc1, bc2;
};

// grad[e] = sum over blocks (FP64, in a fixed order: RED_P threads per parameter, then their sums), loss =
// sum / count, and in a training step Adam's update of the parameter with it.
constexpr int RED_E = 32, RED_P = 8;
__global__ void __launch_bounds__(RED_E * RED_P) mlp_reduce_kernel(const float* __restrict__ part, int nblk, int P,
                                                                   float* grad, float* loss, float inv_count, AdamK ad)
{
    __shared__ double sh[RED_P][RED_E];
    const int c = threadIdx.x % RED_E, p = threadIdx.x / RED_E;
    const int e = blockIdx.x * RED_E + c;
    double s = 0.0;
    if (e <= P)
        for (int b = p; b < nblk; b += RED_P) s += (double)part[(int64_t)b * (P + 1) + e];
    sh[p][c] = s;
    __syncthreads();
    if (p > 0 || e > P) return;
    s = 0.0;
    for (int q = 0; q < RED_P; ++q) s += sh[q][c];
    if (e == P) {
        if (loss) *loss = (float)(s * inv_count);
        return;
    }
    const float ge = (float)s;
    grad[e] = ge;
    if (!ad.master) return;
    const float a = 0.9f * ad.m1[e] + 0.1f * ge;
    const float b = 0.999f * ad.m2[e] + 0.001f * ge * ge;
    ad.m1[e] = a;
    ad.m2[e] = b;
    const float w = ad.master[e] - ad.lr * (a / ad.bc1) / (sqrtf(b / ad.bc2) + 1e-8f);
    ad.master[e] = w;
    ad.wb[e] = __float2bfloat16_rn(w);
}

__global__ void mlp_init_kernel(float* master, __nv_bfloat16* wb, float* m1, float* m2, int in, uint64_t seed)
{
    const int P = param_count(in);
    const Off o(in);
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P) return;
    float sd = 0.f;
    if (e < o.b1) sd = sqrtf(2.f / (float)in);
    else if (e >= o.w2 && e < o.b2) sd = sqrtf(2.f / (float)H);
    else if (e >= o.w3 && e < o.b3) sd = sqrtf(1.f / (float)H);
    // Box-Muller on two counter-based uniforms (splitmix64)
    auto u01 = [&](uint64_t c) {
        uint64_t x = seed + 0x9E3779B97F4A7C15ull * (c + 1);
        x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
        x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
        x ^= x >> 31;
        return ((double)(x >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    };
    const double u1 = u01(2 * (uint64_t)e), u2 = u01(2 * (uint64_t)e + 1);
    const float z = (float)(sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2));
    const float w = sd * z;
    master[e] = w;
    wb[e] = __float2bfloat16_rn(w);
    m1[e] = 0.f;
    m2[e] = 0.f;
}

// ------------------------------------------------------------------ host wrappers
constexpr size_t GRAD_SMEM = sizeof(float) * GRAD_SMEM_FLOATS;
static size_t pred_smem(int in) { return sizeof(float) * (size_t)param_count(in); }
constexpr int GRAD_BLOCKS = 152;

static vb_status set_attrs(int dev)
{
    static bool done[16] = {};
    if (done[dev & 15]) return VB_OK;
    if (cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)GRAD_SMEM) != cudaSuccess)
        return VB_ERR_CUDA;
    done[dev & 15] = true;
    return VB_OK;
}

size_t mlp_ws_bytes(int in, int64_t)
{
    Carve c(nullptr);
    c.take<float>((size_t)GRAD_BLOCKS * (param_count(in) + 1));
    c.take<float>(param_count(in));
    return c.off;
}

static vb_status grad_run(Ctx* ctx, const vb_mlp* m, const float* x, int ld, const float* y, int64_t r0, int64_t r1,
                          float* grad, float* loss, void* ws, size_t ws_bytes, const AdamK& ad)
{
    Carve c(ws);
    float* part = c.take<float>((size_t)GRAD_BLOCKS * (param_count(m->in_dim) + 1));
    if (!ws || ws_bytes < c.off) return VB_ERR_WORKSPACE;
    vb_status st = set_attrs(ctx->device);
    if (st != VB_OK) return st;
    const int P = param_count(m->in_dim);
    const float inv = 1.f / (float)(r1 - r0);
    const int nblk = (int)std::min<int64_t>(GRAD_BLOCKS, (r1 - r0 + GS - 1) / GS);
    mlp_grad_kernel<<<nblk, GT, GRAD_SMEM, ctx->stream>>>(mk(m), x, ld, y, r0, r1, inv, part);
    mlp_reduce_kernel<<<(P + RED_E) / RED_E, RED_E * RED_P, 0, ctx->stream>>>(part, nblk, P, grad, loss, inv, ad);
    ctx->launches += 2;
    return last_launch();
}

// ------------------------------------------------------------------ inference on the tensor cores
// The radius guesses of the kNN search: 128 samples per step, one thread and one tensor-memory
// lane per sample.  Layer 1 is one tcgen05.mma (M = 128 samples, N = 64 hidden units, K = 16:
// the standardised inputs, zero-padded) and layer 2 four (K = 64), both BF16 x BF16 with FP32
// accumulation in tensor memory; biases, GELU and the output layer run in FP32 on the values
// read back with tcgen05.ld.  Weights (BF16) stay in shared memory as the B operands.  The
// activations are rounded to BF16 where the FP32 forward keeps them in FP32, a relative change
// of about 2^-9 that only moves a radius guess (the search stays exact for any guess).
constexpr int MI = 128;   // samples per step
constexpr uint32_t MLP_TMEM_COLS = 128;   // D1 in columns [0, 64), D2 in [64, 128)
constexpr size_t MI_A1 = MI * 16 * 2, MI_B1 = H * 16 * 2, MI_A2 = MI * H * 2, MI_B2 = H * H * 2;
constexpr size_t MI_SMEM = MI_A1 + MI_B1 + MI_A2 + MI_B2 + 3 * H * sizeof(float) + 16;

__global__ void __launch_bounds__(MI) mlp_radius_tc_kernel(MlpK k, const float* __restrict__ xs, int ld, int64_t n,
                                                           float* r2, int mode, float shift, float inflate,
                                                           const float* __restrict__ cloud_shift, Clouds cl,
                                                           DevReport* rep)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __nv_bfloat16* a1 = (__nv_bfloat16*)smem;
    __nv_bfloat16* b1w = (__nv_bfloat16*)(smem + MI_A1);
    __nv_bfloat16* a2 = (__nv_bfloat16*)(smem + MI_A1 + MI_B1);
    __nv_bfloat16* b2w = (__nv_bfloat16*)(smem + MI_A1 + MI_B1 + MI_A2);
    float* bias1 = (float*)(smem + MI_A1 + MI_B1 + MI_A2 + MI_B2);
    float* bias2 = bias1 + H;
    float* w3 = bias2 + H;
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_abort;
    const int t = threadIdx.x, warp = t >> 5;
    const Off o(k.in);
    // B operands: row j (hidden unit) holds its input weights along K
    for (int e = t; e < H * 16; e += MI) {
        const int j = e / 16, r = e % 16;
        const __nv_bfloat16 v = r < k.in ? k.wb[o.w1 + j * k.in + r] : __float2bfloat16_rn(0.f);
        *(__nv_bfloat16*)((char*)b1w + tc::operand_offset(j, r, 16)) = v;
    }
    for (int e = t; e < H * H; e += MI) {
        const int j = e / H, i = e % H;
        *(__nv_bfloat16*)((char*)b2w + tc::operand_offset(j, i, H)) = k.wb[o.w2 + j * H + i];
    }
    for (int j = t; j < H; j += MI) {
        bias1[j] = __bfloat162float(k.wb[o.b1 + j]);
        bias2[j] = __bfloat162float(k.wb[o.b2 + j]);
        w3[j] = __bfloat162float(k.wb[o.w3 + j]);
    }
    const float b3 = __bfloat162float(k.wb[o.b3]);
    if (warp == 0) tc::tmem_alloc(&tmem_base, MLP_TMEM_COLS);
    if (t == 0) { tc::mbar_init(&bar, 1); s_abort = 0; }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tb = tmem_base;
    const uint32_t lane_addr = tb + ((uint32_t)(warp * 32) << 16);
    constexpr uint32_t idesc = tc::idesc_bf16(MI, H);
    uint32_t phase = 0;
    for (int64_t base = (int64_t)blockIdx.x * MI; base < n; base += (int64_t)gridDim.x * MI) {
        const int64_t i = base + t;
        const bool valid = i < n;
        // layer-1 operand: the standardised inputs of this thread's sample, K padded to 16
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint16_t v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int r = 8 * c + e;
                const float xv = valid && r < k.in ? (xs[i * ld + r] - k.mean[r]) / k.scale[r] : 0.f;
                v[e] = __bfloat16_as_ushort(__float2bfloat16_rn(xv));
            }
            *(uint4*)((char*)a1 + tc::operand_offset(t, 8 * c, 16)) = tc::pack8(v);
        }
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (t == 0) {
            tc::mma_bf16(tb, tc::smem_desc(tc::smem_addr(a1), 128, 256), tc::smem_desc(tc::smem_addr(b1w), 128, 256),
                         idesc, 0u);
            tc::mma_commit(&bar);
        }
        bool done = tc::mbar_wait(&bar, phase);
        phase ^= 1u;
        tc::fence_after_sync();
        if (__syncthreads_or(!done)) {
            if (t == 0) { report_error(rep, VB_ERR_TIMEOUT); s_abort = 1; }
            break;
        }
        {
            float z[H];
            tc::tmem_ld64(lane_addr, z);
#pragma unroll
            for (int c = 0; c < H / 8; ++c) {
                uint16_t v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    v[e] = __bfloat16_as_ushort(__float2bfloat16_rn(gelu(z[8 * c + e] + bias1[8 * c + e])));
                *(uint4*)((char*)a2 + tc::operand_offset(t, 8 * c, H)) = tc::pack8(v);
            }
        }
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (t == 0) {
#pragma unroll
            for (int sk = 0; sk < H / 16; ++sk)
                tc::mma_bf16(tb + 64, tc::smem_desc(tc::smem_addr(a2) + sk * 256, 128, (H / 8) * 128),
                             tc::smem_desc(tc::smem_addr(b2w) + sk * 256, 128, (H / 8) * 128), idesc, sk > 0 ? 1u : 0u);
            tc::mma_commit(&bar);
        }
        done = tc::mbar_wait(&bar, phase);
        phase ^= 1u;
        tc::fence_after_sync();
        if (__syncthreads_or(!done)) {
            if (t == 0) { report_error(rep, VB_ERR_TIMEOUT); s_abort = 1; }
            break;
        }
        float z[H];
        tc::tmem_ld64(lane_addr + 64, z);
        float out = b3;
#pragma unroll
        for (int j = 0; j < H; ++j) out = fmaf(w3[j], gelu(z[j] + bias2[j]), out);
        if (valid) {
            const float logr = k.out_mean + k.out_scale * out;
            if (mode == 0) {
                r2[i] = logr;
            } else {   // squared radius bound for the radius-first kNN search
                const float sh = cloud_shift ? shift + cloud_shift[cloud_of(cl.ptr, cl.B, i)] : shift;
                const float r = expf(logr + sh) * inflate;
                r2[i] = __fmul_ru(r, r);
            }
        }
        tc::fence_before_sync();
        __syncthreads();   // the operands of the next step overwrite these only after every read
    }
    if (s_abort) {   // a bounded wait ran out: no further step was issued; the tensor memory goes back
        tc::fence_before_sync();
    }
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tb, MLP_TMEM_COLS);
}

static vb_status mlp_tc_launch(cudaStream_t s, const vb_mlp* mlp, const float* xs, int ld, int64_t n, float* out,
                               int mode, float shift, float inflate, const float* cloud_shift, Clouds cl,
                               DevReport* rep)
{
    static bool attr[16] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (!attr[dev & 15]) {
        if (cudaFuncSetAttribute(mlp_radius_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MI_SMEM + 1024) !=
            cudaSuccess)
            return VB_ERR_CUDA;
        attr[dev & 15] = true;
    }
    // 4 CTAs per SM (128 tensor-memory columns each), persistent over the sample tiles
    const int64_t tiles = (n + MI - 1) / MI;
    const unsigned grid = (unsigned)std::min<int64_t>(tiles, 152 * 4);
    mlp_radius_tc_kernel<<<grid, MI, MI_SMEM + 1024, s>>>(mk(mlp), xs, ld, n, out, mode, shift, inflate, cloud_shift,
                                                          cl, rep);
    return last_launch();
}

vb_status mlp_radius_r2(cudaStream_t s, const vb_mlp* mlp, const float* xs, int64_t n, int m, int mp, float shift,
                        float inflate, float* r2, const float* cloud_shift, Clouds cl, DevReport* rep)
{
    if (!mlp || mlp->in_dim < 1 || mlp->in_dim > VB_MLP_MAX_IN || mlp->in_dim > m || !mlp->weights) return VB_ERR_ARG;
    return mlp_tc_launch(s, mlp, xs, mp, n, r2, 1, shift, inflate, cloud_shift, cl, rep);
}

}  // namespace vb

using namespace vb;

namespace vb {

// Column c of the inputs (c < in) or the targets (c == in): mean and sample standard deviation
// (n - 1), FP64 partials per thread over a fixed stride, then a fixed tree; one block per column.
constexpr int STD_T = 1024;
__global__ void __launch_bounds__(STD_T) mlp_moments_kernel(const float* __restrict__ x, int ld, const float* __restrict__ y,
                                                            int64_t n, int in, double* out)
{
    __shared__ double s1[STD_T], s2[STD_T];
    const int c = blockIdx.x, t = threadIdx.x;
    // shifted by the first value, so that a column far from zero keeps its variance
    const double ref = c < in ? (double)x[c] : (double)y[0];
    double a = 0.0, b = 0.0;
    for (int64_t i = t; i < n; i += STD_T) {
        const double v = (c < in ? (double)x[i * ld + c] : (double)y[i]) - ref;
        a += v;
        b += v * v;
    }
    s1[t] = a;
    s2[t] = b;
    __syncthreads();
    for (int w = STD_T / 2; w > 0; w >>= 1) {
        if (t < w) {
            s1[t] += s1[t + w];
            s2[t] += s2[t + w];
        }
        __syncthreads();
    }
    if (t == 0) {
        const double mean_s = s1[0] / (double)n;
        const double var = n > 1 ? (s2[0] - s1[0] * mean_s) / (double)(n - 1) : 0.0;
        out[2 * c] = ref + mean_s;
        out[2 * c + 1] = sqrt(fmax(var, 0.0));
    }
}

}  // namespace vb

extern "C" {

int64_t vb_mlp_param_count(int32_t in_dim) { return param_count(in_dim); }

vb_status vb_mlp_standardise(vb_ctx* ctx, vb_mlp* m, const float* x, int32_t ld, const float* y, int64_t n, void* ws,
                             size_t ws_bytes)
{
    if (!ctx || !m || !x || !y || n < 1 || ld < m->in_dim || m->in_dim < 1 || m->in_dim > VB_MLP_MAX_IN)
        return VB_ERR_ARG;
    const int in = m->in_dim;
    if (!ws || ws_bytes < sizeof(double) * 2 * (VB_MLP_MAX_IN + 1)) return VB_ERR_WORKSPACE;
    Ctx* c = reinterpret_cast<Ctx*>(ctx);
    double* out = (double*)ws;
    mlp_moments_kernel<<<in + 1, STD_T, 0, c->stream>>>(x, ld, y, n, in, out);
    c->launches += 1;
    vb_status st = last_launch();
    if (st != VB_OK) return st;
    double h[2 * (VB_MLP_MAX_IN + 1)];
    if (cudaMemcpyAsync(h, out, sizeof(double) * 2 * (in + 1), cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
        cudaStreamSynchronize(c->stream) != cudaSuccess)
        return VB_ERR_CUDA;
    for (int r = 0; r < in; ++r) {
        m->in_mean[r] = (float)h[2 * r];
        m->in_scale[r] = (float)std::max(h[2 * r + 1], 1e-12);
    }
    m->out_mean = (float)h[2 * in];
    m->out_scale = (float)std::max(h[2 * in + 1], 1e-12);
    return VB_OK;
}

size_t vb_mlp_workspace(int32_t in_dim, int64_t batch) { return mlp_ws_bytes(in_dim, batch); }

vb_status vb_mlp_init(vb_ctx* ctx, vb_mlp* m, uint64_t seed)
{
    if (!ctx || !m || m->in_dim < 1 || m->in_dim > VB_MLP_MAX_IN || !m->master || !m->weights || !m->adam_m ||
        !m->adam_v)
        return VB_ERR_ARG;
    Ctx* c = reinterpret_cast<Ctx*>(ctx);
    const int P = param_count(m->in_dim);
    mlp_init_kernel<<<(P + 255) / 256, 256, 0, c->stream>>>(m->master, (__nv_bfloat16*)m->weights, m->adam_m,
                                                            m->adam_v, m->in_dim, seed);
    m->step = 0;
    c->launches += 1;
    return last_launch();
}

vb_status vb_mlp_gradient(vb_ctx* ctx, const vb_mlp* m, const float* x, int32_t ld, const float* y, int64_t n,
                          float* grad, float* loss_dev, void* ws, size_t ws_bytes)
{
    if (!ctx || !m || !x || !y || !grad || n < 1 || ld < m->in_dim || m->in_dim < 1 || m->in_dim > VB_MLP_MAX_IN)
        return VB_ERR_ARG;
    return grad_run(reinterpret_cast<Ctx*>(ctx), m, x, ld, y, 0, n, grad, loss_dev, ws, ws_bytes, AdamK{});
}

vb_status vb_mlp_train_epoch(vb_ctx* ctx, vb_mlp* m, const float* x, int32_t ld, const float* y, int64_t n,
                             int32_t batch, float lr, uint64_t seed, float* loss_dev, void* ws, size_t ws_bytes)
{
    if (!ctx || !m || !x || !y || n < 1 || batch < 1 || ld < m->in_dim || m->in_dim < 1 ||
        m->in_dim > VB_MLP_MAX_IN || !(lr > 0.f))
        return VB_ERR_ARG;
    Ctx* c = reinterpret_cast<Ctx*>(ctx);
    Carve cv(ws);
    cv.take<float>((size_t)GRAD_BLOCKS * (param_count(m->in_dim) + 1));
    float* grad = cv.take<float>(param_count(m->in_dim));
    if (!ws || ws_bytes < cv.off) return VB_ERR_WORKSPACE;
    const int64_t nb = (n + batch - 1) / batch;
    const int64_t first = (int64_t)(seed % (uint64_t)nb);
    if (loss_dev && cudaMemsetAsync(loss_dev, 0, sizeof(float), c->stream) != cudaSuccess) return VB_ERR_CUDA;
    for (int64_t b = 0; b < nb; ++b) {
        const int64_t r0 = ((first + b) % nb) * batch;
        const int64_t r1 = std::min<int64_t>(r0 + batch, n);
        const double step = (double)(m->step + 1);
        const AdamK ad{m->master, (__nv_bfloat16*)m->weights, m->adam_m, m->adam_v, lr, 1.f - (float)std::pow(0.9, step),
                       1.f - (float)std::pow(0.999, step)};
        vb_status st = grad_run(c, m, x, ld, y, r0, r1, grad, b == nb - 1 ? loss_dev : nullptr, ws, ws_bytes, ad);
        if (st != VB_OK) return st;
        m->step += 1;
    }
    return VB_OK;
}

vb_status vb_mlp_predict_tc(vb_ctx* ctx, const vb_mlp* m, const float* x, int32_t ld, int64_t n, float* y)
{
    if (!ctx || !m || !x || !y || n < 1 || ld < m->in_dim || m->in_dim < 1 || m->in_dim > VB_MLP_MAX_IN)
        return VB_ERR_ARG;
    Ctx* c = reinterpret_cast<Ctx*>(ctx);
    c->launches += 1;
    return mlp_tc_launch(c->stream, m, x, ld, n, y, 0, 0.f, 1.f, nullptr, Clouds(), c->rep);
}

vb_status vb_mlp_predict(vb_ctx* ctx, const vb_mlp* m, const float* x, int32_t ld, int64_t n, float* y)
{
    if (!ctx || !m || !x || !y || n < 1 || ld < m->in_dim || m->in_dim < 1 || m->in_dim > VB_MLP_MAX_IN)
        return VB_ERR_ARG;
    Ctx* c = reinterpret_cast<Ctx*>(ctx);
    mlp_predict_kernel<<<152 * 4, 128, pred_smem(m->in_dim), c->stream>>>(mk(m), x, ld, n, y, 0, 0.f, 1.f,
                                                                               nullptr, Clouds());
    c->launches += 1;
    return last_launch();
}

}  // extern "C"
