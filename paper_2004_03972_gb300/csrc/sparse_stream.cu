// sparse_stream.cu -- streaming sparse MD kernel for instances whose flux
// operand does not fit in one SM's shared memory (large N, many replicas).
//
// The operand lives in global memory, spin-major and replica-contiguous:
//   op[2]  [N][Rpad] flux operand (FP32, or BF16 with an FP32 master copy),
//          double-buffered across steps; L2-resident at the sizes it serves
//          (N = 20000, 256 replicas: 10 MB in BF16)
//   phi    [N][Rpad] FP32 master (BF16 operand only)
//   p, w   [N][Rpad] FP32 momenta and window sums
// A "cell" is one spin i and one 16-byte vector of V replicas (V = 8 in BF16,
// 4 in FP32).  Each CTA of a persistent cooperative grid, one per SM, owns a
// contiguous range of cells in row-major order, its threads every 768th, so a
// warp's lanes cover consecutive vectors of a row: the gather of neighbour j's
// vectors is one coalesced read of row j (512 bytes for 256 replicas in BF16),
// and the lanes of a row share its neighbour list (broadcast loads of the CSR
// column and sign).  Each step (Methods, "Leapfrog algorithm"):
//   L = sum_k J_ik op[cur][col_k][v] + 2 h_i |phi_i|,
//   p <- p - (kA phi^(M-1) + kB L),  phi <- phi + dA p,
// writes op[nxt], and ends with a grid-wide barrier: an arrival counter
// (release by __threadfence, acquire by ld.acquire) whose wait gives up after
// 2 s, latches HQA_ERR_TIMEOUT and makes every CTA leave.  Operand reads of
// other SMs' writes bypass L1 (ld.global.cg).
//
// The state a cell's owner alone uses (p, and the FP32 master) stays in shared
// memory for the whole run, as many cells as fit (3500 BF16 or 14000 FP32 cells
// per SM); the rest stay in global memory.  That takes 68 of the 174 MB that a
// step moved through L2 at N = 20000 x 256 in BF16, and one CTA per SM makes a
// barrier 152 arrivals instead of one per 256 threads.  Per step there: BF16
// 20.9 -> 14.7 us, FP32 20.6 -> 19.4 us, and with the ranges cut at whole warps
// (first_cell) 12.4 and 17.2; N = 8000 x 40 FP32 5.3 -> 3.9 us, mostly the barrier
// and two rounds of gathers.  Beyond L2 (operand buffers, sums and the state that is
// not resident above about 100 MB) this form and the one before it are within 7 %.
#include <cuda_bf16.h>

#include <algorithm>

#include "hqa_internal.cuh"

namespace {

constexpr int kThreads = 256;     // field, set-up and output kernels
// 768 threads (80 registers) with six gathers in flight each.  N = 20000 x 256,
// us per step, BF16 / FP32: 1024 threads and four gathers 15.3 / 19.1 (but 5.0
// against 4.0 at N = 8000 x 40), eight gathers 17.8 / 21.7, 512 threads 21 / 27.
constexpr int kMDThreads = 768;
constexpr int kGatherBatch = 6;   // neighbour gathers issued together
constexpr uint64_t kWaitNs = 2000000000ull;   // 2 s bound on the grid barrier

struct StreamArgs {
    const int32_t* row_ptr;
    const int32_t* col;
    const int8_t* val;
    const float* h;        // [N] or null
    const StepCoef* sched;
    void* op0;             // [N][Rpad] operand buffers (FP32 or BF16)
    void* op1;
    float* phi;            // [N][Rpad] FP32 master (BF16 operand only)
    float* p;
    float* w;
    unsigned int* bar;     // grid barrier arrival counter; [1] not 0: a tiny state
    uint32_t* status;
    int64_t S;
    int W, N, Rpad, M;
    int nres;              // cells per CTA whose state stays in shared memory
    int wred;              // window sums by reductions
};

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p)
{
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier on a monotonic counter: every CTA arrives once per step;
// returns false (on every thread of the CTA) when the wait timed out here or
// another CTA latched a timeout.
__device__ bool grid_sync(unsigned int* bar, unsigned int target, uint32_t* status)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        __threadfence();
        atomicAdd(bar, 1u);
        const uint64_t t0 = globaltimer();
        uint32_t spins = 0;
        while (ld_acquire(bar) < target) {
            if ((++spins & 63u) == 0) {
                if (*(volatile uint32_t*)status & HQA_DEV_TIMEOUT) { ok = 0; break; }
                if (globaltimer() - t0 > kWaitNs) {
                    atomicOr(status, HQA_DEV_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <bool BF16>
struct Vec;
template <>
struct Vec<false> {   // 4 FP32 replicas
    static constexpr int V = 4;
    __device__ static void load(const void* base, size_t e, float (&x)[4])
    {
        const float4 q = __ldcg(reinterpret_cast<const float4*>(static_cast<const float*>(base) + e));
        x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
    }
    __device__ static void store(void* base, size_t e, const float (&x)[4])
    {
        *reinterpret_cast<float4*>(static_cast<float*>(base) + e) = make_float4(x[0], x[1], x[2], x[3]);
    }
};
template <>
struct Vec<true> {    // 8 BF16 replicas
    static constexpr int V = 8;
    __device__ static void load(const void* base, size_t e, float (&x)[8])
    {
        const uint4 q = __ldcg(reinterpret_cast<const uint4*>(
            static_cast<const __nv_bfloat16*>(base) + e));
        const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            x[2 * k] = __uint_as_float(u[k] << 16);
            x[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u);
        }
    }
    __device__ static void store(void* base, size_t e, const float (&x)[8])
    {
        uint32_t u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * k]));
            const uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * k + 1]));
            u[k] = lo | (hi << 16);
        }
        *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(base) + e) =
            make_uint4(u[0], u[1], u[2], u[3]);
    }
};

// L += the cell's four or eight values of one neighbour, with its sign.
template <bool BF16>
struct Gather;
template <>
struct Gather<false> {
    float4 x;
    __device__ void load(const void* op, size_t e)
    {
        x = __ldcg(reinterpret_cast<const float4*>(static_cast<const float*>(op) + e));
    }
    __device__ void add(float (&L)[4], bool neg) const
    {
        const float s = neg ? -1.f : 1.f;
        L[0] = fmaf(s, x.x, L[0]); L[1] = fmaf(s, x.y, L[1]);
        L[2] = fmaf(s, x.z, L[2]); L[3] = fmaf(s, x.w, L[3]);
    }
};
template <>
struct Gather<true> {
    uint4 x;
    __device__ void load(const void* op, size_t e)
    {
        x = __ldcg(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(op) + e));
    }
    // the mixed add widens the BF16 value itself; the sign goes on before
    __device__ void add(float (&L)[8], bool neg) const
    {
        const uint32_t u[4] = {x.x, x.y, x.z, x.w};
        const uint32_t m = neg ? 0x80008000u : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\t"
                "add.rn.f32.bf16 %0, l, %0;\n\tadd.rn.f32.bf16 %1, h, %1;\n\t}"
                : "+f"(L[2 * k]), "+f"(L[2 * k + 1]) : "r"(u[k] ^ m));
    }
};

// Sum over neighbours k0 .. k1 - 1 in their order; ent(k): column, bit 31 set
// for J = -1.  kGatherBatch gathers are in flight at once.
template <bool BF16, class Ent>
__device__ __forceinline__ void row_sum(const void* op, int rpad, int c, int k0, int k1, Ent ent,
                                        float (&L)[Vec<BF16>::V])
{
#pragma unroll
    for (int e = 0; e < Vec<BF16>::V; ++e) L[e] = 0.f;
    if constexpr (!BF16) {
        // one loop, its last pass predicated (fewer rounds for short rows)
        for (int k = k0; k < k1; k += kGatherBatch) {
            uint32_t j[kGatherBatch];
            Gather<BF16> x[kGatherBatch];
#pragma unroll
            for (int u = 0; u < kGatherBatch; ++u)
                if (k + u < k1) {
                    j[u] = ent(k + u);
                    x[u].load(op, (size_t)(j[u] & 0x7fffffffu) * rpad + c);
                }
#pragma unroll
            for (int u = 0; u < kGatherBatch; ++u)
                if (k + u < k1) x[u].add(L, j[u] >> 31);
        }
        return;
    }
    // BF16: whole batches, then pairs (the predicated form spills: 14.7 -> 19.3 us)
    int k = k0;
    for (; k + kGatherBatch <= k1; k += kGatherBatch) {
        uint32_t j[kGatherBatch];
        Gather<BF16> x[kGatherBatch];
#pragma unroll
        for (int u = 0; u < kGatherBatch; ++u) j[u] = ent(k + u);
#pragma unroll
        for (int u = 0; u < kGatherBatch; ++u)
            x[u].load(op, (size_t)(j[u] & 0x7fffffffu) * rpad + c);
#pragma unroll
        for (int u = 0; u < kGatherBatch; ++u) x[u].add(L, j[u] >> 31);
    }
    for (; k + 2 <= k1; k += 2) {
        const uint32_t j0 = ent(k), j1 = ent(k + 1);
        Gather<BF16> x0, x1;
        x0.load(op, (size_t)(j0 & 0x7fffffffu) * rpad + c);
        x1.load(op, (size_t)(j1 & 0x7fffffffu) * rpad + c);
        x0.add(L, j0 >> 31);
        x1.add(L, j1 >> 31);
    }
    if (k < k1) {
        const uint32_t j = ent(k);
        Gather<BF16> x;
        x.load(op, (size_t)(j & 0x7fffffffu) * rpad + c);
        x.add(L, j >> 31);
    }
}

// Field of one cell (row i, replica vector starting at column c) from operand `op`.
template <bool BF16>
__device__ __forceinline__ void cell_field(const StreamArgs& a, const void* op, int i, int c,
                                           float (&L)[Vec<BF16>::V])
{
    row_sum<BF16>(op, a.Rpad, c, __ldg(a.row_ptr + i), __ldg(a.row_ptr + i + 1),
                  [&](int k) { return (uint32_t)__ldg(a.col + k) | (__ldg(a.val + k) < 0 ? 0x80000000u : 0u); },
                  L);
}

__device__ __forceinline__ void put4(float4* dst, const float* x)
{
    *dst = make_float4(x[0], x[1], x[2], x[3]);
}

__device__ __forceinline__ void get4(float* x, const float4* src)
{
    const float4 q = *src;
    x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
}

// First cell of CTA b of g, in units of 32 where rows are a multiple of 32 vectors:
// a warp then stays within one row (one list length, four full lines per gather).
// N = 20000 x 256 BF16, 100 steps, 1888 -> 1637 us, FP32, 60 steps, 1454 -> 1250 us;
// other row lengths, where a warp spans rows all the same, lost up to 9 % (measured
// before the lanes of a warp met after their sums).
__host__ __device__ inline int64_t cell_unit(int nv) { return nv % 32 == 0 ? 32 : 1; }
__host__ __device__ inline int64_t first_cell(int64_t cells, int nv, int64_t b, int64_t g)
{
    return cells / cell_unit(nv) * b / g * cell_unit(nv);
}

// Whether the lanes of a warp meet after their sums.  Where they lie in two rows or
// more the sums end at different passes, and the lanes then stay apart up to the
// barrier: FP32, N = 40000 x 100 21.9 -> 16.1 us a step, 20000 x 200 16.2 -> 15.2.
// Rows of whole warps (N = 8000 x 128 6.0 / 6.4), rows of a few vectors (5000 x 8 3.4 /
// 3.7, so many rows that some lane is always late) and BF16 (3 %) lose by it.
inline bool lanes_meet(int nv, bool bf16) { return !bf16 && nv % 32 != 0 && nv >= 8; }

// 16-byte state vectors of a cell: p, and in BF16 the FP32 master before it.
template <bool BF16>
constexpr int kPlanes = BF16 ? 4 : 1;

// MEET: the lanes of a warp come together after their sums (lanes_meet).
template <bool BF16, bool STAGED, bool MEET>
__global__ void __launch_bounds__(kMDThreads, 1) k_sparse_stream(const StreamArgs a)
{
    constexpr int V = Vec<BF16>::V, NP = kPlanes<BF16>;
    extern __shared__ float4 st[];   // [NP][nres], then (STAGED) the lists
    const int nv = a.Rpad / V;
    const int64_t cells = (int64_t)a.N * nv;
    const int64_t c0 = first_cell(cells, nv, blockIdx.x, gridDim.x), c1 = first_cell(cells, nv, blockIdx.x + 1, gridDim.x);
    const int mine = (int)(c1 - c0), nres = min(mine, a.nres);
    const int64_t first = c0 + threadIdx.x;
    const int i0 = (int)(first / nv), v0 = (int)(first % nv);
    const int di = kMDThreads / nv, dv = kMDThreads % nv;
    const int64_t win0 = a.S - (int64_t)a.W;
    __shared__ uint32_t s_tiny;   // marked by the set-up; in shared memory, as a register costs 1 %
    if (threadIdx.x == 0) s_tiny = __ldcg(a.bar + 1);
    const int mhalf = (a.M - 2) / 2;
    // global address of plane q of the cell at offset o
    const auto gplane = [&](int q, size_t o) {
        return reinterpret_cast<float4*>((BF16 && q < 2 ? a.phi : a.p) + o + 4 * (BF16 ? q & 1 : 0));
    };
    for (int l = threadIdx.x; l < nres; l += kMDThreads) {
        const int64_t cell = c0 + l;
        const size_t o = (size_t)(cell / nv) * a.Rpad + (size_t)(cell % nv) * V;
#pragma unroll
        for (int q = 0; q < NP; ++q) st[q * a.nres + l] = *gplane(q, o);
    }
    // STAGED: the rows' entry offsets and their entries
    const int rowA = (int)(c0 / nv), rows = mine > 0 ? (int)((c1 - 1) / nv) - rowA + 1 : 0;
    int* s_off = reinterpret_cast<int*>(st + (size_t)NP * a.nres);
    uint32_t* s_ent = reinterpret_cast<uint32_t*>(s_off + rows + 1);
    if constexpr (STAGED) {
        const int kA = rows ? a.row_ptr[rowA] : 0, kB = rows ? a.row_ptr[rowA + rows] : 0;
        for (int k = threadIdx.x; k <= rows; k += kMDThreads)
            s_off[k] = (rows ? a.row_ptr[rowA + k] : 0) - kA;
        for (int k = kA + (int)threadIdx.x; k < kB; k += kMDThreads)
            s_ent[k - kA] = (uint32_t)a.col[k] | (a.val[k] < 0 ? 0x80000000u : 0u);
    }
    __syncthreads();
    for (int64_t m = 0; m < a.S; ++m) {
        const float4 cf = __ldg(reinterpret_cast<const float4*>(a.sched) + m);
        const void* cur = (m & 1) ? a.op1 : a.op0;
        void* nxt = (m & 1) ? a.op0 : a.op1;
        const bool in_win = m >= win0;
        int i = i0, v = v0;
        // MEET: all lanes of a warp take part in each of its rounds
        for (int l = threadIdx.x; (MEET ? l & ~31 : l) < mine; l += kMDThreads) {
            const bool on = !MEET || l < mine;
            if (!on) {
                i = rowA;
                v = 0;
            }
            const int c = v * V;
            const size_t o = (size_t)i * a.Rpad + c;
            float own[V];   // FP32: the cell's own flux, on its way with the gathers
            if constexpr (!BF16) Vec<false>::load(cur, o, own);
            float L[V];
            if constexpr (STAGED)
                row_sum<BF16>(cur, a.Rpad, c, s_off[i - rowA], s_off[i - rowA + 1],
                              [&](int k) { return s_ent[k]; }, L);
            else
                cell_field<BF16>(a, cur, i, c, L);
            if constexpr (MEET) __syncwarp();
            if (!on) break;
            const float hr = a.h ? 2.f * __ldg(a.h + i) : 0.f;
            const bool res = l < nres;
            float sv[4 * NP], fn[V];
#pragma unroll
            for (int q = 0; q < NP; ++q) get4(sv + 4 * q, res ? st + q * a.nres + l : gplane(q, o));
            float* ph = sv;
            float* pp = sv + (BF16 ? 8 : 0);
            if constexpr (!BF16) ph = own;
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const float Le = hr != 0.f ? L[e] + hr * fabsf(ph[e]) : L[e];
                const float phi2 = ph[e] * ph[e];
                const float pw = pot_pow(ph[e], phi2, mhalf);
                pp[e] = pp[e] - fmaf(cf.x, pw, cf.y * Le);
                fn[e] = fmaf(cf.z, pp[e], ph[e]);
                ph[e] = fn[e];
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) put4(res ? st + q * a.nres + l : gplane(q, o), sv + 4 * q);
            // one owner per window sum: the reduction gives the load, add and
            // store's result without waiting for the load (bitwise outside the
            // states that hqa_tiny_state marks)
            if (in_win) {
                const bool red = a.wred && s_tiny == 0u;
#pragma unroll
                for (int e = 0; e < V; e += 4) {
                    float4* w = reinterpret_cast<float4*>(a.w + o + e);
                    if (red) {
                        atomicAdd(w, make_float4(fn[e], fn[e + 1], fn[e + 2], fn[e + 3]));
                    } else {
                        float4 q = *w;
                        q.x += fn[e]; q.y += fn[e + 1]; q.z += fn[e + 2]; q.w += fn[e + 3];
                        *w = q;
                    }
                }
            }
            Vec<BF16>::store(nxt, o, fn);
            i += di;
            v += dv;
            if (v >= nv) {
                v -= nv;
                ++i;
            }
        }
        if (!grid_sync(a.bar, (unsigned int)(gridDim.x * (m + 1)), a.status)) return;
    }
    for (int l = threadIdx.x; l < nres; l += kMDThreads) {
        const int64_t cell = c0 + l;
        const size_t o = (size_t)(cell / nv) * a.Rpad + (size_t)(cell % nv) * V;
#pragma unroll
        for (int q = 0; q < NP; ++q) *gplane(q, o) = st[q * a.nres + l];
    }
}

// Field only: L[r][i] = sum_k J_ik phi[r][col_k] + 2 h_i |phi[r][i]| from an
// operand already in the streaming layout.
template <bool BF16>
__global__ void __launch_bounds__(kThreads) k_sparse_stream_field(const StreamArgs a, int R,
                                                                  const float* phi_in, float* L_out)
{
    constexpr int V = Vec<BF16>::V;
    const int nv = a.Rpad / V;
    const int64_t cells = (int64_t)a.N * nv;
    for (int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; cell < cells;
         cell += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(cell / nv), c = (int)(cell % nv) * V;
        float L[V];
        cell_field<BF16>(a, a.op0, i, c, L);
        const float hr = a.h ? 2.f * __ldg(a.h + i) : 0.f;
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const int r = c + e;
            if (r >= R) continue;
            float v = L[e];
            if (hr != 0.f) v += hr * fabsf(phi_in[(size_t)r * a.N + i]);
            L_out[(size_t)r * a.N + i] = v;
        }
    }
}

// phi(0), p(0) (SplitMix64 or the caller's [R][N] arrays) into the streaming
// layout; window sums and padding replicas zero.  A block moves tiles of 32
// spins x 32 replicas through shared memory: both layouts read and write whole
// lines (one thread per element in the streaming order read a line per element:
// N = 20000 x 256, 49 + 63 us for set-up and output, now 35 together).
constexpr int kTile = 32, kTileRows = 8;   // blocks of 32 x 8 threads

template <bool BF16>
__global__ void __launch_bounds__(kTile * kTileRows)
k_stream_init(StreamArgs a, int R, uint64_t seed, int init, const float* phi0, const float* p0)
{
    __shared__ float tf[kTile][kTile + 1], tq[kTile][kTile + 1];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int ni = (a.N + kTile - 1) / kTile, nr = (a.Rpad + kTile - 1) / kTile;
    for (int64_t t = blockIdx.x; t < (int64_t)ni * nr; t += gridDim.x) {
        const int ib = (int)(t % ni) * kTile, rb = (int)(t / ni) * kTile;
        for (int k = ty; k < kTile; k += kTileRows) {
            const int r = rb + k, i = ib + tx;
            float f = 0.f, q = 0.f;
            if (r < R && i < a.N) {
                const uint64_t c = ((uint64_t)r << 32) | (uint64_t)i;
                if (init == HQA_INIT_GIVEN) {
                    f = phi0[(size_t)r * a.N + i];
                    q = p0[(size_t)r * a.N + i];
                    if (hqa_tiny_state(f, q)) a.bar[1] = 1u;
                } else {
                    uint64_t z = seed + (c + 1ull) * 0x9E3779B97F4A7C15ull;  // SplitMix64
                    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
                    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
                    z ^= z >> 31;
                    q = (z >> 63) ? -1.f : 1.f;
                    if (init == HQA_INIT_RANDOM_FLUX) {
                        uint64_t y = seed + ((c | (1ull << 62)) + 1ull) * 0x9E3779B97F4A7C15ull;
                        y = (y ^ (y >> 30)) * 0xBF58476D1CE4E5B9ull;
                        y = (y ^ (y >> 27)) * 0x94D049BB133111EBull;
                        y ^= y >> 31;
                        f = (float)((int64_t)(y >> 40) - (1 << 23)) * 0x1p-26f;
                    }
                }
            }
            tf[k][tx] = f;
            tq[k][tx] = q;
        }
        __syncthreads();
        for (int k = ty; k < kTile; k += kTileRows) {
            const int i = ib + k, r = rb + tx;
            if (i >= a.N || r >= a.Rpad) continue;
            const size_t idx = (size_t)i * a.Rpad + r;
            const float f = tf[tx][k];
            if constexpr (BF16) {
                static_cast<__nv_bfloat16*>(a.op0)[idx] = __float2bfloat16_rn(f);
                a.phi[idx] = f;
            } else {
                static_cast<float*>(a.op0)[idx] = f;
            }
            a.p[idx] = tq[tx][k];
            a.w[idx] = 0.f;
        }
        __syncthreads();
    }
}

// [R][N] operand from the caller's phi (field only).
template <bool BF16>
__global__ void k_stream_load(StreamArgs a, int R, const float* phi)
{
    const size_t total = (size_t)a.N * a.Rpad;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(idx / a.Rpad), r = (int)(idx % a.Rpad);
        const float f = r < R ? phi[(size_t)r * a.N + i] : 0.f;
        if constexpr (BF16) static_cast<__nv_bfloat16*>(a.op0)[idx] = __float2bfloat16_rn(f);
        else static_cast<float*>(a.op0)[idx] = f;
    }
}

template <bool BF16>
__global__ void __launch_bounds__(kTile * kTileRows)
k_stream_out(StreamArgs a, int R, const void* fin, float inv_w, float* phi_out, float* p_out,
             float* phibar_out)
{
    __shared__ float tf[kTile][kTile + 1], tq[kTile][kTile + 1], tw[kTile][kTile + 1];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int ni = (a.N + kTile - 1) / kTile, nr = (R + kTile - 1) / kTile;
    bool bad = false;
    for (int64_t t = blockIdx.x; t < (int64_t)ni * nr; t += gridDim.x) {
        const int ib = (int)(t % ni) * kTile, rb = (int)(t / ni) * kTile;
        for (int k = ty; k < kTile; k += kTileRows) {
            const int i = ib + k, r = rb + tx;
            if (i >= a.N || r >= R) continue;
            const size_t o = (size_t)i * a.Rpad + r;
            const float f = BF16 ? a.phi[o] : static_cast<const float*>(fin)[o];
            const float q = a.p[o];
            tf[k][tx] = f;
            tq[k][tx] = q;
            if (phibar_out) tw[k][tx] = a.w[o] * inv_w;
            bad |= !(isfinite(f) && isfinite(q));
        }
        __syncthreads();
        for (int k = ty; k < kTile; k += kTileRows) {
            const int r = rb + k, i = ib + tx;
            if (i >= a.N || r >= R) continue;
            const size_t idx = (size_t)r * a.N + i;
            if (phi_out) phi_out[idx] = tf[tx][k];
            if (p_out) p_out[idx] = tq[tx][k];
            if (phibar_out) phibar_out[idx] = tw[tx][k];
        }
        __syncthreads();
    }
    if (__syncthreads_or(bad) && tx == 0 && ty == 0) atomicOr(a.status, HQA_DEV_NONFINITE);
}

int grid_1d(size_t n) { return (int)std::min<size_t>(8192, (n + 255) / 256); }

// Workspace: operand buffers, FP32 master (BF16), p, w, barrier counter.
hqa_status stream_args(hqa_ctx* ctx, int32_t R, bool bf16, StreamArgs* a)
{
    const int V = bf16 ? 8 : 4;
    const int Rpad = (R + V - 1) / V * V;
    const size_t n = (size_t)ctx->N * Rpad;
    const size_t es = bf16 ? 2 : 4;
    const auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t off_op1 = up(n * es), off_phi = off_op1 + up(n * es);
    const size_t off_p = off_phi + (bf16 ? up(n * 4) : 0), off_w = off_p + up(n * 4);
    const size_t off_bar = off_w + up(n * 4), need = off_bar + 256;
    hqa_status s = hqa_reserve(ctx, &ctx->d_state, &ctx->state_cap, need);
    if (s != HQA_OK) return s;
    char* b = static_cast<char*>(ctx->d_state);
    *a = StreamArgs{};
    a->row_ptr = ctx->d_row_ptr;
    a->col = ctx->d_col;
    a->val = ctx->d_val_i8;
    a->h = ctx->has_h ? ctx->d_h : nullptr;
    a->op0 = b;
    a->op1 = b + off_op1;
    a->phi = bf16 ? reinterpret_cast<float*>(b + off_phi) : nullptr;
    a->p = reinterpret_cast<float*>(b + off_p);
    a->w = reinterpret_cast<float*>(b + off_w);
    a->bar = reinterpret_cast<unsigned int*>(b + off_bar);
    a->status = ctx->d_status;
    a->N = ctx->N;
    a->Rpad = Rpad;
    return HQA_OK;
}

}  // namespace

bool hqa_stream_supported(const hqa_ctx* ctx, int prec)
{
    return !ctx->is_batch && ctx->unit && ctx->integer && ctx->d_val_i8 &&
           (prec == HQA_PREC_FP32 || prec == HQA_PREC_BF16);
}

hqa_status hqa_stream_launch_md(hqa_ctx* ctx, int prec, const StepCoef* d_sched, int64_t S,
                                int32_t W, int32_t R, uint64_t seed, int init, const float* phi0,
                                const float* p0, int M, float* phi_out, float* p_out,
                                float* phibar_out, cudaStream_t st)
{
    if (!hqa_stream_supported(ctx, prec)) return HQA_ERR_UNSUPPORTED;
    const bool bf16 = prec == HQA_PREC_BF16;
    StreamArgs a;
    hqa_status s = stream_args(ctx, R, bf16, &a);
    if (s != HQA_OK) return s;
    a.sched = d_sched;
    a.S = S;
    a.W = W;
    a.M = M;
    const dim3 tile(kTile, kTileRows);
    const auto tiles = [&](int reps) {
        return (unsigned)std::min<int64_t>(
            65536, (int64_t)((ctx->N + kTile - 1) / kTile) * ((reps + kTile - 1) / kTile));
    };
    if (cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned int), st) != cudaSuccess) return HQA_ERR_CUDA;
    if (bf16) k_stream_init<true><<<tiles(a.Rpad), tile, 0, st>>>(a, R, seed, init, phi0, p0);
    else k_stream_init<false><<<tiles(a.Rpad), tile, 0, st>>>(a, R, seed, init, phi0, p0);
    // persistent grid: every CTA co-resident (the per-step barrier waits on all of
    // them), one per SM; small problems take fewer, at least a quarter full
    const int64_t cells = (int64_t)ctx->N * (a.Rpad / (bf16 ? 8 : 4));
    const int grid = (int)std::max<int64_t>(
        1, std::min<int64_t>(ctx->sm_count, (cells + kMDThreads / 4 - 1) / (kMDThreads / 4)));
    const size_t cell_bytes = sizeof(float4) * (bf16 ? kPlanes<true> : kPlanes<false>);
    // the CTAs' neighbour lists go first where the largest takes at most 32 KB
    const int nv = a.Rpad / (bf16 ? 8 : 4);
    size_t lists = 0;
    for (int b = 0; b < grid; ++b) {
        const int64_t i0 = first_cell(cells, nv, b, grid) / nv;
        const int64_t i1 = (first_cell(cells, nv, b + 1, grid) - 1) / nv;
        lists = std::max(lists, (size_t)(i1 - i0 + 2 + ctx->row_ptr[i1 + 1] - ctx->row_ptr[i0]) * 4);
    }
    const bool staged = lists <= 32 * 1024;
    if (!staged) lists = 0;
    const int64_t most = (cells / cell_unit(nv) + grid - 1) / grid * cell_unit(nv);   // of a CTA
    a.nres = (int)std::min<int64_t>(most,
                                    (int64_t)((ctx->smem_optin - 1024 - lists) / cell_bytes));
    const size_t n = (size_t)ctx->N * a.Rpad;
    // bytes of operand buffers and state in global memory, with nres cells a CTA resident
    const auto touched = [&](int nres) {
        const double spilled = std::max(0.0, 1.0 - (double)nres * grid / (double)cells);
        return (double)n * (2 * (bf16 ? 2 : 4) + spilled * (bf16 ? 8 : 4));
    };
    // Beyond L2 gathers wait for DRAM, and what holds them meanwhile is L1, which
    // shares its memory with the resident state: rows that spread over more lines
    // (no whole warps) then gain more from L1.  us per step, all that fits resident /
    // this many: FP32 N = 60000 x 300 109 / 91, 60000 x 240 76 / 68; BF16 60000 x 400
    // 122 / 103, 40000 x 400 70 / 65; nearer to L2 BF16 40000 x 300 (0.86 of L2) 45.8 /
    // 47.7; rows of whole warps lost 5 %.
    if (nv % 32 != 0 && touched(a.nres) > 0.9 * (double)ctx->l2_bytes)
        a.nres = std::min(a.nres, bf16 ? 1024 : 6144);
    const size_t smem = a.nres * cell_bytes + lists;
    // window sums by reductions while what a step touches in global memory (both
    // operand buffers, the sums, the state that is not resident) stays in L2;
    // beyond, a reduction waits for its line from DRAM in L2 and holds up the
    // gathers (N = 40000 x 256 BF16, 100 steps: 5.5 ms without, 5.9 with)
    a.wred = touched(a.nres) + 4.0 * (double)n < 0.7 * (double)ctx->l2_bytes;
    const bool meet = lanes_meet(nv, bf16);
    const void* fn = bf16 ? (staged ? (const void*)k_sparse_stream<true, true, false>
                                    : (const void*)k_sparse_stream<true, false, false>)
                   : meet ? (staged ? (const void*)k_sparse_stream<false, true, true>
                                    : (const void*)k_sparse_stream<false, false, true>)
                          : (staged ? (const void*)k_sparse_stream<false, true, false>
                                    : (const void*)k_sparse_stream<false, false, false>);
    if (hqa_smem_attr(fn, smem) != cudaSuccess) return HQA_ERR_CUDA;
    void* args[] = {&a};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kMDThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return hqa_capture_note(hqa_capturing() ? HQA_ERR_UNSUPPORTED : HQA_ERR_CUDA);
    }
    const int64_t nwin = S < W ? S : W;
    const void* fin = (S & 1) ? a.op1 : a.op0;
    if (bf16)
        k_stream_out<true><<<tiles(R), tile, 0, st>>>(
            a, R, fin, 1.0f / (float)nwin, phi_out, p_out, phibar_out);
    else
        k_stream_out<false><<<tiles(R), tile, 0, st>>>(
            a, R, fin, 1.0f / (float)nwin, phi_out, p_out, phibar_out);
    return cudaGetLastError() == cudaSuccess ? HQA_OK : HQA_ERR_CUDA;
}

hqa_status hqa_stream_field(hqa_ctx* ctx, int prec, int32_t R, const float* phi, float* L,
                            cudaStream_t st)
{
    if (!hqa_stream_supported(ctx, prec)) return HQA_ERR_UNSUPPORTED;
    const bool bf16 = prec == HQA_PREC_BF16;
    StreamArgs a;
    hqa_status s = stream_args(ctx, R, bf16, &a);
    if (s != HQA_OK) return s;
    const size_t n = (size_t)ctx->N * a.Rpad;
    const int64_t cells = (int64_t)ctx->N * (a.Rpad / (bf16 ? 8 : 4));
    const int g = (int)std::min<int64_t>(8192, (cells + kThreads - 1) / kThreads);
    if (bf16) {
        k_stream_load<true><<<grid_1d(n), 256, 0, st>>>(a, R, phi);
        k_sparse_stream_field<true><<<g, kThreads, 0, st>>>(a, R, phi, L);
    } else {
        k_stream_load<false><<<grid_1d(n), 256, 0, st>>>(a, R, phi);
        k_sparse_stream_field<false><<<g, kThreads, 0, st>>>(a, R, phi, L);
    }
    return cudaGetLastError() == cudaSuccess ? HQA_OK : HQA_ERR_CUDA;
}
