// mlp.cu -- the surrogate gate's per-spin MLP (6 -> 64 -> 64 -> 2), trained and
// evaluated by hand-written kernels.  This learned gate is an addition to
// the method: the paper has none.
//
//   forward : z = W3 relu(W2 relu(W1 x + b1) + b2) + b3, one thread per sample;
//             each hidden value goes at once into the 64 sums of the next layer,
//             held in registers as 32 pairs (packed FMAs), so one 16-byte weight
//             broadcast feeds four multiply-adds (one load per FMA bounded the
//             first form)
//   grad    : mean binary cross-entropy of the two sigmoid outputs; a block
//             takes 128 samples per tile, one thread per sample forward and
//             backward.  Two shared arrays hold the hidden rows, in turn h1, h2,
//             then d1, d2 in their place, so that two blocks share an SM; rows
//             of 68 floats keep 16-byte accesses aligned and spread over the
//             banks.  The weight gradients are outer products over the tile's
//             samples, dW2 in 4 x 8 register tiles (three 16-byte loads for 16
//             packed FMAs)
//   reduce  : sum of the per-block partials
// 128,000 samples in FP32: forward 138 -> 62 us, gradient 352 -> 150 us.  Both are
// bounded by shared-memory wavefronts (about 2.4 per weight broadcast): 50 % and
// 68 % of the pipe, FMA pipe 30 and 34 %.
//   adamw   : Adam with decoupled weight decay on the FP32 master weights
// Precision: FP32, or BF16 (weights, inputs and hidden activations rounded to
// BF16, FP32 accumulation; gradients are taken w.r.t. the rounded forward).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>

#include "hqa_internal.cuh"

namespace {

constexpr int IN = 6, H = 64, OUT = 2;
constexpr int oW1 = 0, ob1 = oW1 + H * IN, oW2 = ob1 + H, ob2 = oW2 + H * H, oW3 = ob2 + H,
              ob3 = oW3 + OUT * H, P = ob3 + OUT;
constexpr int TS = 128;                   // samples per tile = threads per block
constexpr int RS = H + 4;                 // padded shared row

__device__ __forceinline__ float rnd(float x, bool bf)
{
    return bf ? __bfloat162float(__float2bfloat16_rn(x)) : x;
}

__device__ __forceinline__ float sigm(float z) { return 1.f / (1.f + __expf(-z)); }

__device__ __forceinline__ float softplus(float z)
{
    return z > 0.f ? z + log1pf(__expf(-z)) : log1pf(__expf(z));
}

// Pairs of FP32 values, each rounded as the scalar operation (one issue slot).
__device__ __forceinline__ uint64_t pk2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo2(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Weights in shared memory: the parameter vector (W1, b1, W2, b2, W3, b3; every
// array starts on a 16-byte boundary), and W2 transposed, [k][j], for the
// forward pass.
constexpr int kSw = (P + 3) & ~3;

__device__ __forceinline__ void stage_weights(float* sw, float* w2t, const float* __restrict__ w, int bf)
{
    for (int i = threadIdx.x; i < P; i += blockDim.x) sw[i] = rnd(w[i], bf);
    for (int i = threadIdx.x; i < H * H; i += blockDim.x)
        w2t[i] = rnd(w[oW2 + (i % H) * H + i / H], bf);
}

// Both hidden layers of one sample: h1 row by row (sums in the order bias,
// inputs 0 .. 5), each value at once into the 64 sums of the second layer (32
// pairs, in the order bias, k = 0 .. 63), so that h1 is never held: store(k, h1
// of rows k .. k + 3).
template <class Store>
__device__ __forceinline__ void hidden(const float* sw, const float* w2t, const float (&xi)[IN],
                                       uint64_t (&a2)[H / 2], int bf, Store store)
{
#pragma unroll
    for (int j = 0; j < H; j += 4) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(sw + ob2 + j);
        a2[j / 2] = q.x;
        a2[j / 2 + 1] = q.y;
    }
#pragma unroll 1
    for (int k4 = 0; k4 < H; k4 += 4) {
        float h1[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2* wr = reinterpret_cast<const float2*>(sw + oW1 + (k4 + e) * IN);
            float a = sw[ob1 + k4 + e];
#pragma unroll
            for (int i = 0; i < IN / 2; ++i) {
                const float2 u = wr[i];
                a = fmaf(u.x, xi[2 * i], a);
                a = fmaf(u.y, xi[2 * i + 1], a);
            }
            h1[e] = rnd(fmaxf(a, 0.f), bf);
        }
        store(k4, make_float4(h1[0], h1[1], h1[2], h1[3]));
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint64_t hh = pk2(h1[e], h1[e]);
            const ulonglong2* wt = reinterpret_cast<const ulonglong2*>(w2t + (k4 + e) * H);
#pragma unroll
            for (int j = 0; j < H / 4; ++j) {
                const ulonglong2 q = wt[j];
                a2[2 * j] = fma2(q.x, hh, a2[2 * j]);
                a2[2 * j + 1] = fma2(q.y, hh, a2[2 * j + 1]);
            }
        }
    }
}

__global__ void __launch_bounds__(TS) k_mlp_forward(int64_t n, const float* __restrict__ x,
                                                    float* __restrict__ z,
                                                    const float* __restrict__ w, int bf)
{
    __shared__ __align__(16) float sw[kSw], w2t[H * H];
    stage_weights(sw, w2t, w, bf);
    __syncthreads();
    for (int64_t s = blockIdx.x * (int64_t)TS + threadIdx.x; s < n; s += (int64_t)gridDim.x * TS) {
        float xi[IN];
#pragma unroll
        for (int i = 0; i < IN; ++i) xi[i] = rnd(x[s * IN + i], bf);
        uint64_t a2[H / 2];
        hidden(sw, w2t, xi, a2, bf, [](int, float4) {});
        float z0 = sw[ob3], z1 = sw[ob3 + 1];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const float h2 = rnd(fmaxf((j & 1) ? hi2(a2[j / 2]) : lo2(a2[j / 2]), 0.f), bf);
            z0 = fmaf(sw[oW3 + j], h2, z0);
            z1 = fmaf(sw[oW3 + H + j], h2, z1);
        }
        z[s * OUT] = z0;
        z[s * OUT + 1] = z1;
    }
}

// Shared layout (floats): weights | W2 transposed | x [TS][IN] | h1, then d1
// [TS][RS] | h2, then d2 [TS][RS] | dz [TS][OUT].
__global__ void __launch_bounds__(TS, 2) k_mlp_grad(int64_t n, const float* __restrict__ x,
                                                    const float* __restrict__ y,
                                                    const float* __restrict__ w,
                                                    float* __restrict__ part, int bf, float inv_n)
{
    extern __shared__ __align__(16) float sm[];
    float* sw = sm;
    float* w2t = sw + kSw;
    float* xs = w2t + H * H;
    float* as = xs + TS * IN;
    float* bs = as + TS * RS;
    float* dzs = bs + TS * RS;
    const int t = threadIdx.x;
    float* a_row = as + t * RS;
    float* b_row = bs + t * RS;
    stage_weights(sw, w2t, w, bf);
    // this thread's gradients: dW2 rows 4 ty .. +3, columns 8 tx .. +7; dW3 entry
    // (t / 64, t % 64); b1 (t < 64) or b2 entry t % 64; W1 entries t, t + 128, t + 256
    const int ty = t / 8, tx = t % 8, k64 = t % H;
    float g2[4][8], g3 = 0.f, gb = 0.f, g1[3] = {0.f, 0.f, 0.f}, gb3 = 0.f, lsum = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) g2[i][j] = 0.f;
    __syncthreads();
    for (int64_t tile = blockIdx.x; tile * TS < n; tile += gridDim.x) {
        const int64_t s = tile * TS + t;
        const bool valid = s < n;
        // ---- forward; rows past the end stay zero ----
        float xi[IN];
#pragma unroll
        for (int i = 0; i < IN; ++i) {
            xi[i] = valid ? rnd(x[s * IN + i], bf) : 0.f;
            xs[t * IN + i] = xi[i];
        }
        float z0 = sw[ob3], z1 = sw[ob3 + 1];
        {
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            uint64_t a2[H / 2];
            hidden(sw, w2t, xi, a2, bf,
                   [&](int k, float4 v) { *reinterpret_cast<float4*>(a_row + k) = valid ? v : zero; });
#pragma unroll
            for (int j = 0; j < H; j += 4) {
                float h2[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    h2[e] = rnd(fmaxf((e & 1) ? hi2(a2[(j + e) / 2]) : lo2(a2[(j + e) / 2]), 0.f), bf);
                    z0 = fmaf(sw[oW3 + j + e], h2[e], z0);
                    z1 = fmaf(sw[oW3 + H + j + e], h2[e], z1);
                }
                *reinterpret_cast<float4*>(b_row + j) =
                    valid ? make_float4(h2[0], h2[1], h2[2], h2[3]) : zero;
            }
        }
        // ---- loss and d loss / d z ----
        float dz0 = 0.f, dz1 = 0.f;
        if (valid) {
            const float y0 = y[s * OUT], y1 = y[s * OUT + 1];
            lsum += softplus(z0) - y0 * z0 + softplus(z1) - y1 * z1;
            dz0 = (sigm(z0) - y0) * inv_n;
            dz1 = (sigm(z1) - y1) * inv_n;
        }
        dzs[t * OUT] = dz0;
        dzs[t * OUT + 1] = dz1;
        __syncthreads();
        // ---- layer 3 gradients ----
        {
            float g = 0.f;
            const int o = t / H;
#pragma unroll 8
            for (int u = 0; u < TS; ++u) g = fmaf(dzs[u * OUT + o], bs[u * RS + k64], g);
            g3 += g;
            if (t < OUT) {
                float b = 0.f;
                for (int u = 0; u < TS; ++u) b += dzs[u * OUT + t];
                gb3 += b;
            }
        }
        __syncthreads();
        // ---- backward through layer 3 and the second ReLU (d2 replaces h2), and
        //      through layer 2 ----
        uint64_t dh1[H / 2];
#pragma unroll
        for (int k = 0; k < H / 2; ++k) dh1[k] = 0ull;
#pragma unroll 1
        for (int j = 0; j < H; j += 4) {
            const float4 hv = *reinterpret_cast<const float4*>(b_row + j);
            const float hh[4] = {hv.x, hv.y, hv.z, hv.w};
            float d[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float g = fmaf(sw[oW3 + j + e], dz0, sw[oW3 + H + j + e] * dz1);
                d[e] = hh[e] > 0.f ? g : 0.f;
            }
            *reinterpret_cast<float4*>(b_row + j) = make_float4(d[0], d[1], d[2], d[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint64_t dd = pk2(d[e], d[e]);
                const ulonglong2* wr = reinterpret_cast<const ulonglong2*>(sw + oW2 + (j + e) * H);
#pragma unroll
                for (int k = 0; k < H / 4; ++k) {
                    const ulonglong2 q = wr[k];
                    dh1[2 * k] = fma2(q.x, dd, dh1[2 * k]);
                    dh1[2 * k + 1] = fma2(q.y, dd, dh1[2 * k + 1]);
                }
            }
        }
        __syncthreads();
        // ---- dW2 = sum over samples of d2 h1^T ----
        uint64_t acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll 2
        for (int u = 0; u < TS; ++u) {
            const float4 d = *reinterpret_cast<const float4*>(bs + u * RS + 4 * ty);
            const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(as + u * RS + 8 * tx);
            const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(as + u * RS + 8 * tx + 4);
            const uint64_t dv[4] = {pk2(d.x, d.x), pk2(d.y, d.y), pk2(d.z, d.z), pk2(d.w, d.w)};
            const uint64_t hv[4] = {p.x, p.y, q.x, q.y};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(dv[i], hv[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                g2[i][2 * j] += lo2(acc[i][j]);
                g2[i][2 * j + 1] += hi2(acc[i][j]);
            }
        if (t >= H) {
            float b = 0.f;
#pragma unroll 8
            for (int u = 0; u < TS; ++u) b += bs[u * RS + k64];
            gb += b;
        }
        __syncthreads();
        // ---- first ReLU (d1 replaces h1), layer 1 gradients ----
#pragma unroll
        for (int k = 0; k < H; k += 4) {
            const float4 hv = *reinterpret_cast<const float4*>(a_row + k);
            *reinterpret_cast<float4*>(a_row + k) =
                make_float4(hv.x > 0.f ? lo2(dh1[k / 2]) : 0.f, hv.y > 0.f ? hi2(dh1[k / 2]) : 0.f,
                            hv.z > 0.f ? lo2(dh1[k / 2 + 1]) : 0.f,
                            hv.w > 0.f ? hi2(dh1[k / 2 + 1]) : 0.f);
        }
        __syncthreads();
        if (t < H) {
            float b = 0.f;
#pragma unroll 8
            for (int u = 0; u < TS; ++u) b += as[u * RS + k64];
            gb += b;
        }
        // entry k 6 + i of dW1; threads t .. t + 31 read k close together
        float c1[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
        for (int u = 0; u < TS; ++u)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int e = t + TS * q;
                c1[q] = fmaf(as[u * RS + e / IN], xs[u * IN + e % IN], c1[q]);
            }
#pragma unroll
        for (int q = 0; q < 3; ++q) g1[q] += c1[q];
        __syncthreads();
    }
    float* out = part + (size_t)blockIdx.x * (P + 1);
#pragma unroll
    for (int q = 0; q < 3; ++q) out[oW1 + t + TS * q] = g1[q];
    out[(t < H ? ob1 : ob2) + k64] = gb;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) out[oW2 + (4 * ty + i) * H + 8 * tx + j] = g2[i][j];
    out[oW3 + t] = g3;
    if (t < OUT) out[ob3 + t] = gb3;
    // loss: block sum
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    __shared__ float sl[TS / 32];
    if ((t & 31) == 0) sl[t >> 5] = lsum;
    __syncthreads();
    if (t == 0) {
        float v = 0.f;
        for (int k = 0; k < TS / 32; ++k) v += sl[k];
        out[P] = v * inv_n;
    }
}
static_assert(TS == OUT * H && TS * 3 == H * IN && P == oW2 + H * H + H + OUT * H + OUT,
              "one thread's share of the gradients");

// A warp per 32 parameters and eighth of the blocks' partials, in a fixed order.
constexpr int kRedWarps = 8;

__global__ void __launch_bounds__(32 * kRedWarps) k_mlp_reduce(int nparts,
                                                               const float* __restrict__ part,
                                                               float* __restrict__ grad,
                                                               float* __restrict__ loss)
{
    __shared__ float sh[kRedWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (p <= P)
#pragma unroll 4
        for (int b = warp; b < nparts; b += kRedWarps) s += part[(size_t)b * (P + 1) + p];
    sh[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && p <= P) {
        float v = 0.f;
        for (int k = 0; k < kRedWarps; ++k) v += sh[k][lane];
        if (p < P) grad[p] = v;
        else if (loss) *loss = v;
    }
}

__global__ void k_mlp_adamw(float* __restrict__ w, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, float lr, float b1,
                            float b2, float eps, float wd, float c1, float c2)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x) {
        const float gp = g[p];
        const float mp = b1 * m[p] + (1.f - b1) * gp;
        const float vp = b2 * v[p] + (1.f - b2) * gp * gp;
        m[p] = mp;
        v[p] = vp;
        const float mh = mp / c1, vh = vp / c2;
        w[p] -= lr * (mh / (sqrtf(vh) + eps) + wd * w[p]);
    }
}

size_t grad_smem()
{
    return sizeof(float) * (kSw + H * H + TS * IN + 2 * TS * RS + TS * OUT);
}

}  // namespace

struct hqa_mlp {
    int device = 0;
    int sm_count = 0;
    float* d_w = nullptr;
    float* d_m = nullptr;
    float* d_v = nullptr;
    float* d_part = nullptr;
    size_t part_cap = 0;
    int64_t step = 0;
};

extern "C" {

hqa_status hqa_mlp_create(const float* params, hqa_mlp** out)
{
    if (!out || !params) return HQA_ERR_INVALID_ARG;
    *out = nullptr;
    for (int p = 0; p < P; ++p)
        if (!std::isfinite(params[p])) return HQA_ERR_NONFINITE_INPUT;
    hqa_mlp* m = new (std::nothrow) hqa_mlp();
    if (!m) return HQA_ERR_OOM;
    auto fail = [&](hqa_status s) {
        cudaFree(m->d_w);
        cudaFree(m->d_m);
        cudaFree(m->d_v);
        delete m;
        return s;
    };
    if (cudaGetDevice(&m->device) != cudaSuccess) return fail(HQA_ERR_CUDA);
    cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, m->device);
    if (cudaMalloc(&m->d_w, P * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&m->d_m, P * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&m->d_v, P * sizeof(float)) != cudaSuccess)
        return fail(HQA_ERR_OOM);
    if (cudaMemcpy(m->d_w, params, P * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->d_m, 0, P * sizeof(float)) != cudaSuccess ||
        cudaMemset(m->d_v, 0, P * sizeof(float)) != cudaSuccess)
        return fail(HQA_ERR_CUDA);
    *out = m;
    return HQA_OK;
}

hqa_status hqa_mlp_params(const hqa_mlp* m, float* params)
{
    if (!m || !params) return HQA_ERR_INVALID_ARG;
    HQA_CUDA_TRY(cudaDeviceSynchronize());
    HQA_CUDA_TRY(cudaMemcpy(params, m->d_w, P * sizeof(float), cudaMemcpyDeviceToHost));
    return HQA_OK;
}

hqa_status hqa_mlp_forward(hqa_mlp* m, int64_t n, const float* x, float* logits, int32_t precision,
                           void* stream)
{
    if (!m || n < 0 || (n > 0 && (!x || !logits))) return HQA_ERR_INVALID_ARG;
    if (precision != HQA_PREC_FP32 && precision != HQA_PREC_BF16) return HQA_ERR_INVALID_ARG;
    if (n == 0) return HQA_OK;
    const int64_t blocks = std::min<int64_t>((n + TS - 1) / TS, (int64_t)m->sm_count * 5);
    k_mlp_forward<<<(int)blocks, TS, 0, static_cast<cudaStream_t>(stream)>>>(
        n, x, logits, m->d_w, precision == HQA_PREC_BF16);
    return cudaGetLastError() == cudaSuccess ? HQA_OK : HQA_ERR_CUDA;
}

hqa_status hqa_mlp_grad(hqa_mlp* m, int64_t n, const float* x, const float* y, float* grad,
                        float* loss, int32_t precision, void* stream)
{
    if (!m || n < 1 || !x || !y || !grad) return HQA_ERR_INVALID_ARG;
    if (precision != HQA_PREC_FP32 && precision != HQA_PREC_BF16) return HQA_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t tiles = (n + TS - 1) / TS;
    const int blocks = (int)std::min<int64_t>(tiles, (int64_t)m->sm_count * 2);
    const size_t need = (size_t)blocks * (P + 1) * sizeof(float);
    if (need > m->part_cap) {
        cudaFree(m->d_part);
        m->d_part = nullptr;
        m->part_cap = 0;
        HQA_CUDA_TRY(cudaMalloc(&m->d_part, need));
        m->part_cap = need;
    }
    const size_t smem = grad_smem();
    HQA_CUDA_TRY(cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_mlp_grad<<<blocks, TS, smem, st>>>(n, x, y, m->d_w, m->d_part, precision == HQA_PREC_BF16,
                                         1.f / (float)n);
    k_mlp_reduce<<<(P + 1 + 31) / 32, 32 * kRedWarps, 0, st>>>(blocks, m->d_part, grad, loss);
    return cudaGetLastError() == cudaSuccess ? HQA_OK : HQA_ERR_CUDA;
}

hqa_status hqa_mlp_adamw(hqa_mlp* m, const float* grad, float lr, float beta1, float beta2,
                         float eps, float weight_decay, void* stream)
{
    if (!m || !grad || !(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f))
        return HQA_ERR_INVALID_ARG;
    ++m->step;
    const float c1 = 1.f - powf(beta1, (float)m->step), c2 = 1.f - powf(beta2, (float)m->step);
    k_mlp_adamw<<<(P + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(
        m->d_w, grad, m->d_m, m->d_v, lr, beta1, beta2, eps, weight_decay, c1, c2);
    return cudaGetLastError() == cudaSuccess ? HQA_OK : HQA_ERR_CUDA;
}

void hqa_mlp_destroy(hqa_mlp* m)
{
    if (!m) return;
    cudaDeviceSynchronize();
    cudaFree(m->d_w);
    cudaFree(m->d_m);
    cudaFree(m->d_v);
    cudaFree(m->d_part);
    delete m;
}

}  // extern "C"
