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
// set-up take about 10), and in place of the vector form (sparse_md_vec.cu)
// N = 100 x 152 replicas 205 -> 41 us, N = 256 x 152 518 -> 164 us.
#include <cuda_bf16.h>

#include <algorithm>

#include "hqa_internal.cuh"

namespace {

constexpr int kRowLanes = 8;
constexpr int kCMaxN = 256;

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

__device__ __forceinline__ uint64_t c_bits(uint32_t x, uint32_t y)
{
    return (uint64_t)x | ((uint64_t)y << 32);
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

// N <= 32 NQ <= 256.  Eight lanes carry four rows, 16 NQ factors in registers, so
// that a 16-byte load of fluxes feeds sixteen products; a warp covers 16 rows.  The
// sums meet in two, one and one shuffles that hand each row to one pair of lanes,
// which keeps its state.  One row per lane group (four times the loads of the same
// fluxes) took 70 us at N = 100 against 41: a 16-byte load of 32 lanes is four
// wavefronts, also where four rows read the same 128 bytes.
// Up to N = 128 the factors are pairs of floats.  Beyond, they are bytes, the top
// ones of +-1/2, and a byte permute expands each; its zero bytes come from shared
// memory, or else the expansion would be moved in front of the loop, where the
// registers end.  (Two rows per eight lanes with the bytes read from shared memory
// at every step: N = 200 199 us, against 164 at N = 256.)
template <int NQ, bool BF16>
__global__ void __launch_bounds__(NQ > 4 ? 512 : 256, 1) k_md_complete(const CompleteArgs a)
{
    constexpr int COLS = NQ * 32;
    constexpr bool BYTES = NQ > 4;
    extern __shared__ __align__(16) unsigned char smem[];
    float* const op = reinterpret_cast<float*>(smem);                       // [2][COLS]
    const volatile uint32_t* const zero = reinterpret_cast<uint32_t*>(smem + 2 * COLS * 4);
    int8_t* const J = reinterpret_cast<int8_t*>(smem + 2 * COLS * 4 + 16);  // [N][COLS], set-up
    const int N = a.N, rep = blockIdx.x, t = threadIdx.x;
    const int l = t & (kRowLanes - 1), first = t / kRowLanes * 4, row = first + (l >> 1);
    for (int o = t; o < 2 * COLS + 4; o += blockDim.x) op[o] = 0.f;
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
    uint64_t f[BYTES ? 1 : 4][BYTES ? 1 : NQ][2];
    uint32_t b[BYTES ? 4 : 1][BYTES ? NQ : 1];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            char4 x = make_char4(0, 0, 0, 0);
            if (first + s < N)
                x = *reinterpret_cast<const char4*>(J + (first + s) * COLS + (q * kRowLanes + l) * 4);
            if constexpr (BYTES) {
                const auto top = [](int v) { return __float_as_uint(0.5f * (float)v) >> 24; };
                b[s][q] = top(x.x) | (top(x.y) << 8) | (top(x.z) << 16) | (top(x.w) << 24);
            } else {
                f[s][q][0] = c_pack((float)x.x, (float)x.y);
                f[s][q][1] = c_pack((float)x.z, (float)x.w);
            }
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
        uint32_t z = 0u;
        if constexpr (BYTES) z = *zero;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 x = src[q * kRowLanes];
            const uint64_t x01 = c_pack(x.x, x.y), x23 = c_pack(x.z, x.w);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if constexpr (BYTES) {
                    const uint32_t u = b[s][q];
                    s01[s] = c_fma2(c_bits(__byte_perm(u, z, 0x0444u), __byte_perm(u, z, 0x1444u)), x01, s01[s]);
                    s23[s] = c_fma2(c_bits(__byte_perm(u, z, 0x2444u), __byte_perm(u, z, 0x3444u)), x23, s23[s]);
                } else {
                    s01[s] = c_fma2(f[s][q][0], x01, s01[s]);
                    s23[s] = c_fma2(f[s][q][1], x23, s23[s]);
                }
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
        if constexpr (BYTES) L *= 2.f;
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

int c_threads(int N) { return 32 * ((N + 15) / 16); }
size_t c_smem(int N) { return 16 + (size_t)(8 + N) * ((N + 31) / 32 * 32); }

template <int NQ, bool BF16>
cudaError_t launch_complete(const CompleteArgs& a, int R, cudaStream_t st)
{
    const void* fn = (const void*)k_md_complete<NQ, BF16>;
    const size_t smem = c_smem(a.N);
    const cudaError_t e = hqa_smem_attr(fn, smem);
    if (e != cudaSuccess) return e;
    void* args[] = {const_cast<CompleteArgs*>(&a)};
    return cudaLaunchKernel(fn, dim3(R), dim3(c_threads(a.N)), args, smem, st);
}

template <bool BF16>
cudaError_t dispatch_complete(const CompleteArgs& a, int R, cudaStream_t st)
{
    switch ((a.N + 31) / 32) {
    case 1: return launch_complete<1, BF16>(a, R, st);
    case 2: return launch_complete<2, BF16>(a, R, st);
    case 3: return launch_complete<3, BF16>(a, R, st);
    case 4: return launch_complete<4, BF16>(a, R, st);
    case 5: return launch_complete<5, BF16>(a, R, st);
    case 6: return launch_complete<6, BF16>(a, R, st);
    case 7: return launch_complete<7, BF16>(a, R, st);
    default: return launch_complete<8, BF16>(a, R, st);
    }
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

void hqa_complete_shape(const hqa_ctx* ctx, int32_t* threads, int64_t* smem_bytes)
{
    *threads = c_threads(ctx->N);
    *smem_bytes = (int64_t)c_smem(ctx->N);
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
