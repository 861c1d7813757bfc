// sparse_complete.cu -- few replicas of a small complete graph (the SK instances a
// user starts with), one replica per CTA: a step is a chain of latencies.
//
// Same method as sparse_md.cu.  All couplings of a row are held as factors (-1, 0
// on the diagonal, +1), so the field needs no lists: eight lanes share a row, each
// reads every eighth group of four fluxes by one 16-byte load, and the eight sums
// meet in shuffles.  A step has one barrier and one exchange through shared memory;
// the list form (k_sparse_md_split) has two barriers and scattered 4-byte gathers,
// whose wavefronts fill half of its time.  150 steps of one replica, whole call,
// list form before and this form: N = 100 132 -> 41 us, N = 20 28 us (its launch and
// set-up take about 10), N = 200 404 (the form before the list split) -> 199 us.
#include <cuda_bf16.h>

#include <algorithm>

#include "hqa_internal.cuh"

namespace {

constexpr int kRowLanes = 8;
constexpr int kCThreads = 1024;
constexpr int kCRows = kCThreads / kRowLanes;   // rows of one pass
constexpr int kCMaxN = 2 * kCRows;

struct CompleteArgs {
    const int32_t* col;    // row i: entries i (N - 1) to (i + 1) (N - 1) - 1
    const int8_t* val;
    const StepCoef* sched;
    const float* h;        // [N] or null
    const float* phi0;     // HQA_INIT_GIVEN
    const float* p0;
    float* phi_out;
    float* p_out;
    float* phibar_out;
    uint32_t* status;
    uint64_t seed;
    int64_t S;
    int32_t W, N, M, init;
};

__device__ __forceinline__ uint64_t c_splitmix(uint64_t seed, uint64_t counter)
{
    // SplitMix64 (Steele, Lea, Flood 2014): output number counter+1 of the stream.
    uint64_t z = seed + (counter + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t c_pack(float x, float y)
{
    return (uint64_t)__float_as_uint(x) | ((uint64_t)__float_as_uint(y) << 32);
}

__device__ __forceinline__ uint64_t c_fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ float c_operand(float x, bool bf16)
{
    return bf16 ? __bfloat162float(__float2bfloat16_rn(x)) : x;
}

__device__ __forceinline__ void c_initial(const CompleteArgs& a, int rep, int row, float& phi, float& p)
{
    const uint64_t c = ((uint64_t)rep << 32) | (uint64_t)row;
    if (a.init == HQA_INIT_GIVEN) {
        phi = a.phi0[(size_t)rep * a.N + row];
        p = a.p0[(size_t)rep * a.N + row];
    } else {
        p = (c_splitmix(a.seed, c) >> 63) ? -1.f : 1.f;
        if (a.init == HQA_INIT_RANDOM_FLUX) {
            const uint64_t z = c_splitmix(a.seed, c | (1ull << 62));
            phi = (float)((int64_t)(z >> 40) - (1 << 23)) * 0x1p-26f;
        }
    }
}

// The couplings into J[row][col] (bytes, zeroed before), four entries a load.
template <class Put>
__device__ __forceinline__ void c_scatter(const CompleteArgs& a, int8_t* J, int stride, Put put)
{
    const int per = a.N - 1, nnz = a.N * per;
#pragma unroll 4
    for (int e = 4 * threadIdx.x; e < nnz; e += 4 * blockDim.x) {
        int c[4], v[4];
        if (e + 4 <= nnz) {
            const int4 cc = __ldg(reinterpret_cast<const int4*>(a.col + e));
            const char4 vv = __ldg(reinterpret_cast<const char4*>(a.val + e));
            c[0] = cc.x; c[1] = cc.y; c[2] = cc.z; c[3] = cc.w;
            v[0] = vv.x; v[1] = vv.y; v[2] = vv.z; v[3] = vv.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                c[k] = e + k < nnz ? __ldg(a.col + e + k) : 0;
                v[k] = e + k < nnz ? __ldg(a.val + e + k) : 0;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (e + k < nnz) J[(e + k) / per * stride + c[k]] = put(v[k]);
    }
}

// N <= 32 NQ <= 128.  Eight lanes carry four rows, 16 NQ factors in registers, so
// that a 16-byte load of fluxes feeds sixteen products; a warp covers 16 rows.  The
// sums meet in two, one and one shuffles that hand each row to one pair of lanes,
// which keeps its state.  One row per lane group (four times the loads of the same
// fluxes) took 70 us at N = 100 against 41: a 16-byte load of 32 lanes is four
// wavefronts, also where four rows read the same 128 bytes.
template <int NQ, bool BF16>
__global__ void __launch_bounds__(256, 1) k_md_complete(const CompleteArgs a)
{
    constexpr int COLS = NQ * 32;
    extern __shared__ __align__(16) unsigned char smem[];
    float* const op = reinterpret_cast<float*>(smem);                       // [2][COLS]
    int8_t* const J = reinterpret_cast<int8_t*>(smem + 2 * COLS * 4);       // [N][COLS], set-up
    const int N = a.N, rep = blockIdx.x, t = threadIdx.x;
    const int l = t & (kRowLanes - 1), first = t / kRowLanes * 4, row = first + (l >> 1);
    for (int o = t; o < 2 * COLS; o += blockDim.x) op[o] = 0.f;
    for (int o = t; o < N * COLS / 4; o += blockDim.x) reinterpret_cast<uint32_t*>(J)[o] = 0u;
    float phi = 0.f, p = 0.f, w = 0.f, h2 = 0.f;
    const bool ok = row < N;
    if (ok) {
        c_initial(a, rep, row, phi, p);
        if (a.h) h2 = 2.f * __ldg(a.h + row);
    }
    __syncthreads();
    c_scatter(a, J, COLS, [](int v) { return (int8_t)v; });
    if (ok) op[row] = c_operand(phi, BF16);   // both lanes of a pair, the same value
    __syncthreads();
    uint64_t f[4][NQ][2];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            char4 x = make_char4(0, 0, 0, 0);
            if (first + s < N)
                x = *reinterpret_cast<const char4*>(J + (first + s) * COLS + (q * kRowLanes + l) * 4);
            f[s][q][0] = c_pack((float)x.x, (float)x.y);
            f[s][q][1] = c_pack((float)x.z, (float)x.w);
        }
    const int64_t win0 = a.S - (int64_t)a.W;
    const int mhalf = (a.M - 2) / 2;
    const bool up = l & 4, mid = l & 2;
    const float4* src = reinterpret_cast<const float4*>(op) + l;
    float* dst = op + COLS + row;
    int flip = COLS;               // dst of the next step lies -flip, +flip, ...
    for (int64_t j = 0; j < a.S; ++j) {
        const float4 cf = __ldg(reinterpret_cast<const float4*>(a.sched) + j);
        uint64_t s01[4] = {}, s23[4] = {};
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 x = src[q * kRowLanes];
            const uint64_t x01 = c_pack(x.x, x.y), x23 = c_pack(x.z, x.w);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                s01[s] = c_fma2(f[s][q][0], x01, s01[s]);
                s23[s] = c_fma2(f[s][q][1], x23, s23[s]);
            }
        }
        float v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s)
            v[s] = (__uint_as_float((uint32_t)s01[s]) + __uint_as_float((uint32_t)(s01[s] >> 32))) +
                   (__uint_as_float((uint32_t)s23[s]) + __uint_as_float((uint32_t)(s23[s] >> 32)));
        const float g0 = __shfl_xor_sync(0xffffffffu, up ? v[0] : v[2], 4);
        const float g1 = __shfl_xor_sync(0xffffffffu, up ? v[1] : v[3], 4);
        const float u0 = (up ? v[2] : v[0]) + g0, u1 = (up ? v[3] : v[1]) + g1;
        float L = (mid ? u1 : u0) + __shfl_xor_sync(0xffffffffu, mid ? u0 : u1, 2);
        L += __shfl_xor_sync(0xffffffffu, L, 1);
        L += h2 * fabsf(phi);
        const float phi2 = phi * phi;
        const float pw = pot_pow(phi, phi2, mhalf);
        p = p - fmaf(cf.x, pw, cf.y * L);
        phi = fmaf(cf.z, p, phi);
        if (ok && !(l & 1)) *dst = c_operand(phi, BF16);
        if (j >= win0) w += phi;
        src += flip / 4;
        dst -= flip;
        flip = -flip;
        __syncthreads();
    }
    bool bad = false;
    if (ok && !(l & 1)) {
        const size_t o = (size_t)rep * N + row;
        if (a.phi_out) a.phi_out[o] = phi;
        if (a.p_out) a.p_out[o] = p;
        if (a.phibar_out) a.phibar_out[o] = w * (1.0f / (float)(a.S < a.W ? a.S : (int64_t)a.W));
        bad = !(isfinite(phi) && isfinite(p));
    }
    if (__syncthreads_or(bad) && t == 0) atomicOr(a.status, HQA_DEV_NONFINITE);
}

// 128 < N <= 32 NQ <= 256: two rows per eight lanes.  The factors are bytes in
// shared memory, the top bytes of +-1/2 (a word expands to four floats by byte
// permutes; 64 registers a thread don't hold them), with 32 bytes between rows that
// keep a warp's four rows apart.
template <int NQ, bool BF16>
__global__ void __launch_bounds__(kCThreads, 1) k_md_complete_wide(const CompleteArgs a)
{
    constexpr int COLS = NQ * 32, JROW = COLS + 32, PASS = 2;
    extern __shared__ __align__(16) unsigned char smem[];
    float* const op = reinterpret_cast<float*>(smem);                       // [2][COLS]
    int8_t* const J = reinterpret_cast<int8_t*>(smem + 2 * COLS * 4);       // [N][JROW]
    const int N = a.N, rep = blockIdx.x, t = threadIdx.x;
    const int l = t & (kRowLanes - 1), row0 = t / kRowLanes;

    for (int o = t; o < 2 * COLS; o += blockDim.x) op[o] = 0.f;
    for (int o = t; o < N * JROW / 4; o += blockDim.x) reinterpret_cast<uint32_t*>(J)[o] = 0u;
    float phi[PASS], p[PASS], w[PASS], h2[PASS];
    bool ok[PASS];
    const uint32_t* fb[PASS];
#pragma unroll
    for (int s = 0; s < PASS; ++s) {
        const int row = row0 + s * kCRows;
        ok[s] = row < N;
        phi[s] = p[s] = w[s] = h2[s] = 0.f;
        // rows past the end read row 0's factors, and their sums go nowhere
        fb[s] = reinterpret_cast<const uint32_t*>(J + (ok[s] ? row : 0) * JROW) + l;
        if (!ok[s]) continue;
        c_initial(a, rep, row, phi[s], p[s]);
        if (a.h) h2[s] = 2.f * __ldg(a.h + row);
    }
    __syncthreads();
    c_scatter(a, J, JROW, [](int v) { return (int8_t)(v > 0 ? 0x3f : 0xbf); });
#pragma unroll
    for (int s = 0; s < PASS; ++s)
        if (ok[s] && l == 0) op[row0 + s * kCRows] = c_operand(phi[s], BF16);
    __syncthreads();
    const int64_t win0 = a.S - (int64_t)a.W;
    const int mhalf = (a.M - 2) / 2;
    const float4* src = reinterpret_cast<const float4*>(op) + l;
    float* dst = op + COLS + row0;
    int flip = COLS;               // dst of the next step lies -flip, +flip, ...
    for (int64_t j = 0; j < a.S; ++j) {
        const float4 cf = __ldg(reinterpret_cast<const float4*>(a.sched) + j);
        uint64_t s01[PASS], s23[PASS];
#pragma unroll
        for (int s = 0; s < PASS; ++s) s01[s] = s23[s] = 0ull;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 x = src[q * kRowLanes];
            const uint64_t x01 = c_pack(x.x, x.y), x23 = c_pack(x.z, x.w);
#pragma unroll
            for (int s = 0; s < PASS; ++s) {
                const uint32_t u = fb[s][q * kRowLanes];
                const auto f2 = [u](uint32_t lo, uint32_t hi) {
                    return (uint64_t)__byte_perm(u, 0u, lo) | ((uint64_t)__byte_perm(u, 0u, hi) << 32);
                };
                s01[s] = c_fma2(f2(0x0444u, 0x1444u), x01, s01[s]);
                s23[s] = c_fma2(f2(0x2444u, 0x3444u), x23, s23[s]);
            }
        }
#pragma unroll
        for (int s = 0; s < PASS; ++s) {
            float L = (__uint_as_float((uint32_t)s01[s]) + __uint_as_float((uint32_t)(s01[s] >> 32))) +
                      (__uint_as_float((uint32_t)s23[s]) + __uint_as_float((uint32_t)(s23[s] >> 32)));
#pragma unroll
            for (int k = 1; k < kRowLanes; k *= 2) L += __shfl_xor_sync(0xffffffffu, L, k);
            L *= 2.f;
            L += h2[s] * fabsf(phi[s]);
            const float phi2 = phi[s] * phi[s];
            const float pw = pot_pow(phi[s], phi2, mhalf);
            p[s] = p[s] - fmaf(cf.x, pw, cf.y * L);
            phi[s] = fmaf(cf.z, p[s], phi[s]);
            if (l == 0 && ok[s]) dst[s * kCRows] = c_operand(phi[s], BF16);
            if (j >= win0) w[s] += phi[s];
        }
        src += flip / 4;
        dst -= flip;
        flip = -flip;
        __syncthreads();
    }
    bool bad = false;
#pragma unroll
    for (int s = 0; s < PASS; ++s) {
        if (!ok[s] || l != 0) continue;
        const size_t o = (size_t)rep * N + row0 + s * kCRows;
        if (a.phi_out) a.phi_out[o] = phi[s];
        if (a.p_out) a.p_out[o] = p[s];
        if (a.phibar_out) a.phibar_out[o] = w[s] * (1.0f / (float)(a.S < a.W ? a.S : (int64_t)a.W));
        bad |= !(isfinite(phi[s]) && isfinite(p[s]));
    }
    if (__syncthreads_or(bad) && t == 0) atomicOr(a.status, HQA_DEV_NONFINITE);
}

template <int NQ, bool BF16>
cudaError_t launch_complete(const CompleteArgs& a, int R, cudaStream_t st)
{
    constexpr bool wide = NQ > 4;
    const void* fn;
    if constexpr (wide) fn = (const void*)k_md_complete_wide<NQ, BF16>;
    else fn = (const void*)k_md_complete<NQ, BF16>;
    const size_t smem = 2 * NQ * 32 * 4 + (size_t)a.N * (NQ * 32 + (wide ? 32 : 0));
    const cudaError_t e = hqa_smem_attr(fn, smem);
    if (e != cudaSuccess) return e;
    const int threads = wide ? kCThreads : 32 * ((a.N + 15) / 16);
    void* args[] = {const_cast<CompleteArgs*>(&a)};
    return cudaLaunchKernel(fn, dim3(R), dim3(threads), args, smem, st);
}

template <bool BF16>
cudaError_t dispatch_complete(const CompleteArgs& a, int R, cudaStream_t st)
{
    if (a.N <= 32) return launch_complete<1, BF16>(a, R, st);
    if (a.N <= 64) return launch_complete<2, BF16>(a, R, st);
    if (a.N <= 96) return launch_complete<3, BF16>(a, R, st);
    if (a.N <= 128) return launch_complete<4, BF16>(a, R, st);
    return a.N <= 192 ? launch_complete<6, BF16>(a, R, st) : launch_complete<8, BF16>(a, R, st);
}

}  // namespace

// A complete graph with +-1 couplings of at most 256 spins, one replica per CTA
// and at most one CTA per SM.  Only complete graphs: their rows have no zero
// factors but the diagonal's, so no lane multiplies for nothing, and a flux that
// diverges reaches every row either way.
bool hqa_complete_possible(const hqa_ctx* ctx, int32_t R)
{
    return !ctx->is_batch && ctx->unit && ctx->d_val_i8 && ctx->N >= 2 && ctx->N <= kCMaxN &&
           ctx->nnz == (int64_t)ctx->N * (ctx->N - 1) && R <= ctx->sm_count;
}

hqa_status hqa_complete_launch_md(hqa_ctx* ctx, int prec, const StepCoef* d_sched, int64_t S,
                                  int32_t W, int32_t R, uint64_t seed, int init, const float* phi0,
                                  const float* p0, int M, float* phi_out, float* p_out,
                                  float* phibar_out, cudaStream_t st)
{
    CompleteArgs a{};
    a.col = ctx->d_col;
    a.val = ctx->d_val_i8;
    a.sched = d_sched;
    a.h = ctx->has_h ? ctx->d_h : nullptr;
    a.phi0 = phi0;
    a.p0 = p0;
    a.phi_out = phi_out;
    a.p_out = p_out;
    a.phibar_out = phibar_out;
    a.status = ctx->d_status;
    a.seed = seed;
    a.S = S;
    a.W = W;
    a.N = ctx->N;
    a.M = M;
    a.init = init;
    const cudaError_t e = prec == HQA_PREC_BF16 ? dispatch_complete<true>(a, R, st)
                                                : dispatch_complete<false>(a, R, st);
    return e == cudaSuccess ? HQA_OK : HQA_ERR_CUDA;
}
