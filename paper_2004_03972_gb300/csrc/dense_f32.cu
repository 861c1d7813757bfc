// dense_f32.cu -- the FP32 dense MD on the tcgen05 tensor cores.
//
// The field L = J Phi of an FP32 run (Methods, "Leapfrog algorithm") is a
// contraction that the CUDA cores bound at 80 TFLOP/s.  Here it runs on the
// BF16 tensor cores from slices of phi, at an error against FP64 that is below
// the FP32 sum's in all but the states named below:
//
//   phi = b0 + b1 + b2,  b0 = phi rounded to a multiple of u, then to BF16,
//                        b1 = the rest rounded to BF16,
//                        b2 = what that leaves, rounded to BF16,
//
// 24 significant bits of phi in three BF16 numbers.  u is a power of two, 2^-k of
// the largest |phi| of the 32 spins that a warp holds of that replica: with
// 2^k <= 2^23 / (largest row sum of |J|) every product with a +-1 coupling is a
// whole number of units, a row's sum stays below 2^24 of them, and the FP32
// accumulator adds b0's products without any rounding.  (The tensor core truncates
// what does not fit its FP32 accumulator, which is what limits an ordinary hi + lo
// split: the FP16X2 operand errs 12 times the FP32 sum on K2000.)  b1 and b2 are
// 2^-8 and 2^-16 of b0, so truncation there costs next to nothing; each slice has
// its own accumulator, and the epilogue adds the three, smallest first.  Fluxes
// below u / 2 have no b0 and keep 17 bits, 2^-25 of the group's largest.
//
// The unit follows from the fluxes of one replica at one step and from nothing
// else: a replica's bits do not depend on the others of the launch, a resumed run
// has the bits of an unbroken one, and the accuracy is the same at every scale of
// phi.  One unit for 16 to 64 replicas, taken from the largest |phi| two steps
// before, cost a replica 1000 times smaller than its neighbours two digits.
//
// Error of the field against FP64 (2-norm over a replica's spins, the largest of
// 40), these slices / the FP32 sum on the CUDA cores: uniform, normal and
// log-uniform fluxes at any scale 2.6e-8 to 7e-8 / 1.9e-7 at N = 64, 2.6e-8
// (+-1) and 1.5e-7 (real) / 8.5e-7 at 2000, 3e-7 / 2.0e-6 at 12000.  Where the
// 32-spin groups of ONE replica differ in scale by 2^6 (real J, large N) to 2^10
// (+-1), the small groups' b0 is truncated against the sum of the large ones, up
// to half a last place per 16 spins: every other 64 spins 1e-5 of the rest
// 1.4e-6 / 8.6e-7 at N = 2000 and 7.4e-6 / 2.0e-6 at 12000, one flux 2^20 times
// all others 4.5e-6 / 1.3e-6 and 2.5e-5 / 3e-6.  A unit for the whole replica would
// mend that and take bits from small groups that couple among themselves only.
//
// Couplings: +-1 (any integer up to 127) is one exact BF16 slice.  Real
// couplings are cut the same way (a_0 + a_1 + a_2; a_0 a multiple of 2^-7 of a
// power of two per row), and the products a_i b_j with i + j <= 2 are kept,
// accumulator i + j: six MMA columns per replica instead of three.
//
// The three slices of a k-tile lie one after another in shared memory, so one
// MMA of N = 3 NC columns runs all of them against one coupling tile, and the
// real case's a_1 and a_2 are MMAs of 2 NC and NC columns into the shifted
// accumulator.  Roles, ring and synchronisation are those of the 16-bit kernel
// (dense_md_kernel.cuh): a TMA producer warp, an MMA warp, epilogue warps,
// phi in TMEM, p in global memory, a column-group arrival counter per half;
// pairs of row tiles share cta_group::2 MMAs where the row tiles pair up and
// J is one slice.  While the producer waits for the column group it already
// loads coupling tiles into free stages, since only phi depends on the other
// CTAs (real N = 500 x 200: 7.3 -> 6.9 us per step, measured with that unit, as
// is the next; filling the ring before looking at the counter cost K2000 x 1024
// 17.5 -> 18.5 us).
//
// What bounds it: the SM's intake from L2, 28 KB per k-tile of a pair's CTA at
// about 100 GB/s of the 128 that an SM can take (64 B/clk); the MMAs would need
// two thirds of the step.  Real couplings of N = 1000 x 512 the same: 60 KB per
// k-tile (three coupling slices), 960 KB a step at 90 GB/s.  Measured against the
// CUDA-core form (dense_simt.cu), per step: K2000 +-1 x 1024 replicas 210 -> 16.5
// us, real N = 1000 x 512 115 -> 10.7 us; error against FP64 after 40 steps (2-norm,
// p) 6.9e-7 -> 3.7e-7 and 7.6e-7 -> 4.7e-7.  (A unit from the largest |phi| of the
// replicas that share a tile, passed between the CTAs each step, took 17.5 and
// 12.0 us.)
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "dense_md_kernel.cuh"

namespace {

using hqa_dense::BK;
using hqa_dense::BM;
using hqa_dense::kWaitNs;

// 8 epilogue warps: a half of 64 replicas is four 16-column chunks, two per
// warp of a lane quarter.  12 leave one group a second chunk and the others
// idle, and spill (K2000 x 1024: 18.6 us per step against 18.4)
constexpr int kEpiWarps = 8;
constexpr int kGroups = kEpiWarps / 4;        // chunk stride: warps per lane quarter
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr uint32_t kStg = 16 * 128 * 2;       // staging tile: 16 replicas x 128 spins
constexpr uint32_t A_BYTES = BM * BK * 2;

struct F32Args {
    float* phi;              // [Rpad][Npad]
    float* p;
    float* w;
    uint16_t* phib;          // [2][Rpad][3 Npad] BF16 slices
    const StepCoef* sched;
    const float* h;          // [N] or null
    const float* rscale;     // [Npad] power of two per coupling row, or null (all 1)
    unsigned int* gbar;      // [groups] arrival counters
    uint32_t* tiny;          // not 0: window sums without reductions (hqa_tiny_state)
    uint32_t* status;
    int64_t S;
    int W, N, Npad, Rpad, R, KT, Mt, M;
    int rep0;
    uint32_t ushift;         // 23 - k in the exponent field
};

// 1.5 * 2^23 units for a warp's 32 fluxes of one replica (f: this lane's):
// adding and subtracting it rounds to a multiple of the unit.
__device__ __forceinline__ float round_const(uint32_t f, uint32_t ushift)
{
    const uint32_t e = __reduce_max_sync(0xffffffffu, f & 0x7f800000u) + ushift;
    return __uint_as_float(min(e, 0x7f000000u) | 0x00400000u);
}

__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi)   // lo -> bits 0-15
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ uint64_t widen_bf16x2(uint32_t v)
{
    return hqa_dense::pk2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}

// The three slices of a pair of values.
__device__ __forceinline__ void slices2(uint64_t f, uint64_t c0, uint32_t (&b)[3])
{
    using namespace hqa_dense;
    const uint64_t t0 = sub2(add2(f, c0), c0);
    b[0] = cvt_bf16x2(lo2(t0), hi2(t0));
    const uint64_t r1 = sub2(f, widen_bf16x2(b[0]));
    b[1] = cvt_bf16x2(lo2(r1), hi2(r1));
    const uint64_t r2 = sub2(r1, widen_bf16x2(b[1]));
    b[2] = cvt_bf16x2(lo2(r2), hi2(r2));
}

// NC replicas per half, NJ coupling slices, HV halves per CTA, KSUB k-tiles per
// ring stage: their coupling tiles, then their slice tiles.
template <int NC, int NJ, int HV, int STAGES, int KSUB, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
k_dense_f32(const __grid_constant__ CUtensorMap tmJ, const __grid_constant__ CUtensorMap tmB,
            const __grid_constant__ CUtensorMap tmS, const F32Args a)
{
    constexpr int NBR = PAIR ? 3 * NC / 2 : 3 * NC;      // phi rows staged by this CTA
    constexpr uint32_t B_BYTES = NBR * BK * 2;
    constexpr uint32_t STAGE = KSUB * (NJ * A_BYTES + B_BYTES);
    constexpr uint32_t B_OFF = KSUB * NJ * A_BYTES;
    constexpr uint32_t COLS = HV * 4 * NC;               // accumulators, then phi
    constexpr uint32_t TMEM_COLS = COLS <= 64 ? 64 : COLS <= 128 ? 128 : COLS <= 256 ? 256 : 512;
    constexpr uint32_t PHI0 = HV * 3 * NC;               // first phi column
    static_assert(NC % 16 == 0 && COLS <= 512 && STAGE % 1024 == 0, "tile shape");
    static_assert(!PAIR || (NJ == 1 && (3 * NC) % 32 == 0 && (NC / 2) % 8 == 0), "pair shape");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bar = base + STAGES * STAGE;
    const uint32_t full0 = bar, empty0 = bar + 8 * STAGES, pfull0 = bar + 16 * STAGES;
    const uint32_t accf0 = bar + 24 * STAGES, acce0 = accf0 + 16, tmem_slot = accf0 + 32,
                   done_bar = accf0 + 40;
    static_assert(24 * STAGES + 48 <= 1024, "barrier block");
    __shared__ int s_abort;
    __shared__ uint32_t s_tiny;   // *a.tiny: here, as a register held through the steps costs up to 3 %
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mt = blockIdx.x % a.Mt, nc = blockIdx.x / a.Mt;
    const uint32_t crank = PAIR ? tc::cluster_rank() : 0u;
    const int m0 = mt * BM, n0 = nc * HV * NC;

    if (threadIdx.x == 0) {
        s_abort = 0;
        s_tiny = __ldcg(a.tiny);
        for (int s = 0; s < STAGES; ++s) {
            tc::mbar_init(full0 + 8 * s, 1);
            tc::mbar_init(empty0 + 8 * s, 1);
            tc::mbar_init(pfull0 + 8 * s, 1);
        }
        for (int hh = 0; hh < 2; ++hh) {
            tc::mbar_init(accf0 + 8 * hh, 1);
            tc::mbar_init(acce0 + 8 * hh, PAIR ? 2 * kEpiWarps : kEpiWarps);
        }
        tc::mbar_init(done_bar, 1);
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tmJ);
        tc::prefetch_tmap(&tmB);
        tc::prefetch_tmap(&tmS);
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            tc::tmem_alloc2(tmem_slot, TMEM_COLS);
            tc::tmem_relinquish2();
        } else {
            tc::tmem_alloc(tmem_slot, TMEM_COLS);
            tc::tmem_relinquish();
        }
    }
    tc::tc_fence_before();
    if constexpr (PAIR) tc::cluster_sync();
    else __syncthreads();
    tc::tc_fence_after();
    uint32_t tmem;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem) : "r"(tmem_slot));
    volatile int* abort = &s_abort;
    volatile uint32_t* gstatus = a.status;

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer ----
            uint32_t it = 0;
            auto is_free = [&](uint32_t q) {   // the stage of iteration q, without blocking
                return q < STAGES ||
                       tc::mbar_test<PAIR>(empty0 + 8 * (q % STAGES), ((q / STAGES) - 1) & 1);
            };
            auto wait_free = [&](uint32_t q) {
                if (q < STAGES) return true;
                const uint32_t e = empty0 + 8 * (q % STAGES), ph = ((q / STAGES) - 1) & 1;
                return PAIR ? tc::mbar_wait_cl(e, ph, abort, kWaitNs) : tc::mbar_wait(e, ph, abort, kWaitNs);
            };
            auto load_j = [&](uint32_t q, int kt) {
                const int s = q % STAGES;
                tc::mbar_expect_tx(full0 + 8 * s, STAGE);
#pragma unroll
                for (int k = 0; k < KSUB; ++k)
#pragma unroll
                    for (int j = 0; j < NJ; ++j)
                        tc::tma_load_2d(base + s * STAGE + (k * NJ + j) * A_BYTES, &tmJ,
                                        j * a.Npad + (kt * KSUB + k) * BK, m0, full0 + 8 * s);
            };
            auto load_b = [&](uint32_t q, int kt, int brow) {
                const int s = q % STAGES;
#pragma unroll
                for (int k = 0; k < KSUB; ++k) {
                    const uint32_t sb = base + s * STAGE + B_OFF + k * B_BYTES;
                    const int x = (kt * KSUB + k) * BK;
                    if constexpr (PAIR) {
                        // rows [3 NC / 2 rank, + 3 NC / 2) of the stacked slices, in half tiles
#pragma unroll
                        for (int u = 0; u < 3; ++u) {
                            const int q2 = 3 * (int)crank + u;
                            tc::tma_load_2d(sb + u * (NC / 2) * BK * 2, &tmB, (q2 >> 1) * a.Npad + x,
                                            brow + (q2 & 1) * (NC / 2), full0 + 8 * s);
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < 3; ++u)
                            tc::tma_load_2d(sb + u * NC * BK * 2, &tmB, u * a.Npad + x, brow,
                                            full0 + 8 * s);
                    }
                }
            };
            const int KT = a.KT / KSUB;
            for (int64_t m = 0; m < a.S && !*abort; ++m)
                for (int hh = 0; hh < HV && !*abort; ++hh) {
                    // until the column group has finished the last step, coupling
                    // tiles go into whatever stages are free
                    int pre = 0;
                    if (m > 0) {
                        const unsigned int* g = a.gbar + HV * nc + hh;
                        const unsigned int target = (unsigned int)(a.Mt * m);
                        const uint64_t t0 = tc::globaltimer();
                        uint32_t spins = 0;
                        while (hqa_dense::ld_acquire(g) < target) {
                            if (pre < STAGES && pre < KT && is_free(it + pre)) {
                                load_j(it + pre, pre);
                                ++pre;
                            }
                            if ((++spins & 63u) == 0) {
                                if (*abort || (*gstatus & HQA_DEV_TIMEOUT)) { *abort = 1; break; }
                                if (tc::globaltimer() - t0 > kWaitNs) { *abort = 1; break; }
                            }
                        }
                        if (*abort) { it += pre; break; }
                        tc::fence_proxy_async_global();
                    }
                    const int brow = (int)(m & 1) * a.Rpad + n0 + hh * NC;
                    for (int kt = 0; kt < KT; ++kt, ++it) {
                        if (kt >= pre) {
                            if (!wait_free(it)) break;
                            load_j(it, kt);
                        }
                        load_b(it, kt, brow);
                    }
                }
            // drain: every issued copy must land before the CTA can exit
            if (*abort)
                for (uint32_t k = (it > STAGES ? it - STAGES : 0); k < it; ++k) {
                    volatile int no_abort = 0;
                    tc::mbar_wait(full0 + 8 * (k % STAGES), (k / STAGES) & 1, &no_abort, 20000000ull);
                }
        }
    } else if (warp == 1) {
        if (lane == 0 && PAIR && crank != 0) {
            // ---- odd CTA of a pair: relay each landed stage to the MMA issuer ----
            uint32_t it = 0;
            const uint32_t peer = tc::mapa(pfull0, 0);
            const int KT = a.KT / KSUB;
            for (int64_t m = 0; m < a.S && !*abort; ++m)
                for (int hh = 0; hh < HV && !*abort; ++hh)
                    for (int kt = 0; kt < KT; ++kt, ++it) {
                        const int s = it % STAGES;
                        if (!tc::mbar_wait(full0 + 8 * s, (it / STAGES) & 1, abort, kWaitNs)) break;
                        tc::mbar_arrive_remote(peer + 8 * s);
                    }
        } else if (lane == 0) {
            // ---- MMA issuer ----
            uint32_t it = 0;
            const int KT = a.KT / KSUB;
            for (int64_t m = 0; m < a.S && !*abort; ++m)
                for (int hh = 0; hh < HV && !*abort; ++hh) {
                    if (m > 0) {
                        const uint32_t ph = (uint32_t)((m - 1) & 1);
                        if (!(PAIR ? tc::mbar_wait_cl(acce0 + 8 * hh, ph, abort, kWaitNs)
                                   : tc::mbar_wait(acce0 + 8 * hh, ph, abort, kWaitNs)))
                            break;
                    }
                    tc::tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(hh * 3 * NC);
                    for (int kt = 0; kt < KT; ++kt, ++it) {
                        const int s = it % STAGES;
                        if (!tc::mbar_wait(full0 + 8 * s, (it / STAGES) & 1, abort, kWaitNs)) break;
                        if (PAIR && !tc::mbar_wait_cl(pfull0 + 8 * s, (it / STAGES) & 1, abort, kWaitNs))
                            break;
                        tc::tc_fence_after();
                        const uint32_t sa = base + s * STAGE;
#pragma unroll
                        for (int k = 0; k < KSUB; ++k) {
                            const uint64_t bd = tc::sdesc_k128(sa + B_OFF + k * B_BYTES);
#pragma unroll
                            for (int j = 0; j < NJ; ++j) {
                                // slice j of J against the first 3 - j of phi, accumulators j .. 2
                                const uint64_t ad = tc::sdesc_k128(sa + (k * NJ + j) * A_BYTES);
#pragma unroll
                                for (int kk = 0; kk < BK / 16; ++kk) {
                                    const uint32_t add = j > 0 || (kt | k | kk) != 0;
                                    if constexpr (PAIR)
                                        tc::mma2_f16(d, ad + 2 * kk, bd + 2 * kk,
                                                     tc::idesc_bf16(2 * BM, 3 * NC), add);
                                    else
                                        tc::mma_bf16(d + (uint32_t)(j * NC), ad + 2 * kk, bd + 2 * kk,
                                                     tc::idesc_bf16(BM, (3 - j) * NC), add);
                                }
                            }
                        }
                        if constexpr (PAIR) tc::mma_commit2(empty0 + 8 * s, 3);
                        else tc::mma_commit(empty0 + 8 * s);
                    }
                    if constexpr (PAIR) tc::mma_commit2(accf0 + 8 * hh, 3);
                    else tc::mma_commit(accf0 + 8 * hh);
                }
            if constexpr (PAIR) {
                volatile int no_abort = 0;
                tc::mma_commit2(done_bar, 1);
                tc::mbar_wait_cl(done_bar, 0, &no_abort, kWaitNs);
            }
        }
    } else {
        // ---- epilogue warps: kick, drift, operand slices, window ----
        using namespace hqa_dense;
        const int ew = warp - 2;
        const int quarter = warp & 3;         // TMEM lanes 32 quarter .. +31
        const int csel = ew >> 2;             // first chunk of this warp
        const int row = m0 + 32 * quarter + lane;
        const bool row_ok = row < a.N;
        const float hr = (a.h && row_ok) ? 2.f * a.h[row] : 0.f;
        const float rs = a.rscale ? a.rscale[row] : 1.f;
        const int mhalf = (a.M - 2) / 2;
        const int64_t win0 = a.S - (int64_t)a.W;
        const uint32_t tl = tmem + ((uint32_t)(32 * quarter) << 16);
        const uint32_t rloc = (uint32_t)(32 * quarter + lane);
        const uint32_t acce_to = (PAIR && crank != 0) ? tc::mapa(acce0, 0) : acce0;
        // the four warps of one csel: named barrier 2 + csel, staging tiles at stg
        const uint32_t stg = bar + 1024 + (uint32_t)(csel * 3) * kStg;
        const bool gleader = (ew & 3) == 0 && lane == 0;
        for (int hh = 0; hh < HV; ++hh)
            for (int c = csel; c < NC / 16; c += kGroups) {
                uint32_t v[16];
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    v[j] = __float_as_uint(a.phi[(size_t)(n0 + hh * NC + c * 16 + j) * a.Npad + row]);
                tc::tmem_st16(tl + PHI0 + (uint32_t)(hh * NC + c * 16), v);
            }
        tc::tmem_wait_st();
        bool stop = false;
        for (int64_t m = 0; m < a.S && !stop; ++m) {
            const float4 cf = __ldg(reinterpret_cast<const float4*>(a.sched) + m);
            const bool in_win = m >= win0 && *(volatile uint32_t*)&s_tiny == 0u;
            for (int hh = 0; hh < HV && !stop; ++hh) {
                float pp[16];
                if (row_ok && csel < NC / 16) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        pp[j] = a.p[(size_t)(n0 + hh * NC + csel * 16 + j) * a.Npad + row];
                }
                bool ok = __all_sync(0xffffffffu,
                                     PAIR ? tc::mbar_wait_cl(accf0 + 8 * hh, (uint32_t)(m & 1), abort, kWaitNs)
                                          : tc::mbar_wait(accf0 + 8 * hh, (uint32_t)(m & 1), abort, kWaitNs));
                tc::tc_fence_after();
                ok = tc::named_bar_and(2 + csel, 128, ok);
                if (ok) {
                    const uint64_t hr2 = pk2(hr, hr), rs2 = pk2(rs, rs);
                    const uint64_t cx2 = pk2(cf.x, cf.x), cy2 = pk2(cf.y, cf.y), cz2 = pk2(cf.z, cf.z);
#pragma unroll 1
                    for (int c = csel; c < NC / 16; c += kGroups) {
                        const int col = hh * NC + c * 16;
                        const uint32_t dcol = tl + (uint32_t)(hh * 3 * NC + c * 16);
                        uint32_t v0[16], v1[16], v2[16], fv[16];
                        tc::tmem_ld16(dcol, v0);
                        tc::tmem_ld16(dcol + NC, v1);
                        tc::tmem_ld16(dcol + 2 * NC, v2);
                        tc::tmem_ld16(tl + PHI0 + (uint32_t)col, fv);
                        float npp[16];
                        const bool more = row_ok && c + kGroups < NC / 16;
                        if (more) {
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                npp[j] = a.p[(size_t)(n0 + col + 16 * kGroups + j) * a.Npad + row];
                        }
                        // the staging tiles are free once the last chunk's stores have read them
                        if (gleader) tc::bulk_wait_read0();
                        tc::named_bar(2 + csel, 128);
                        tc::tmem_wait_ld();
                        if (row_ok) {
#pragma unroll
                            for (int j = 0; j < 16; j += 2) {
                                const size_t o0 = (size_t)(n0 + col + j) * a.Npad + row;
                                const size_t o1 = o0 + a.Npad;
                                auto pr = [&](const uint32_t (&x)[16]) {
                                    return pk2(__uint_as_float(x[j]), __uint_as_float(x[j + 1]));
                                };
                                const uint64_t f2 = pr(fv);
                                const uint64_t s2 = add2(add2(pr(v2), pr(v1)), pr(v0));
                                const uint64_t L2 =
                                    fma2(hr2, f2 & 0x7fffffff7fffffffull, mul2(s2, rs2));
                                const uint64_t sq2 = mul2(f2, f2);
                                uint64_t pw2 = f2;
#pragma unroll
                                for (int q = 0; q < kMaxMHalf; ++q)
                                    if (q < mhalf) pw2 = mul2(pw2, sq2);
                                const uint64_t pn2 = sub2(pk2(pp[j], pp[j + 1]), fma2(cx2, pw2, mul2(cy2, L2)));
                                const uint64_t fn2 = fma2(cz2, pn2, f2);
                                a.p[o0] = lo2(pn2);
                                a.p[o1] = hi2(pn2);
                                const float fl = lo2(fn2), fh = hi2(fn2);
                                fv[j] = __float_as_uint(fl);
                                fv[j + 1] = __float_as_uint(fh);
                                if (in_win) {
                                    win_add(a.w + o0, fl);
                                    win_add(a.w + o1, fh);
                                }
                            }
                        }
                        // the operand; spin rows beyond N keep a zero one
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            uint32_t b[3];
                            slices2(pk2(__uint_as_float(fv[j]), __uint_as_float(fv[j + 1])),
                                    pk2(round_const(fv[j], a.ushift), round_const(fv[j + 1], a.ushift)), b);
                            const uint32_t sb = stg + (uint32_t)(j * 128) * 2u + rloc * 2u;
#pragma unroll
                            for (int u = 0; u < 3; ++u) {
                                sts_u16(sb + u * kStg, (uint16_t)b[u]);
                                sts_u16(sb + u * kStg + 256u, (uint16_t)(b[u] >> 16));
                            }
                        }
                        // .sync.aligned: every lane of the warp, outside the row_ok branch
                        tc::tmem_st16(tl + PHI0 + (uint32_t)col, fv);
                        tc::tmem_wait_st();
                        tc::fence_proxy_async_smem();
                        tc::named_bar(2 + csel, 128);
                        if (gleader) {
                            const int y = (int)((m + 1) & 1) * a.Rpad + n0 + col;
#pragma unroll
                            for (int u = 0; u < 3; ++u)
                                tc::tma_store_2d(&tmS, u * a.Npad + m0, y, stg + u * kStg);
                            tc::bulk_commit();
                        }
                        if (more) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) pp[j] = npp[j];
                        }
                    }
                    tc::tc_fence_before();
                    if (lane == 0) {
                        if (PAIR && crank != 0) tc::mbar_arrive_remote(acce_to + 8 * hh);
                        else tc::mbar_arrive(acce0 + 8 * hh);
                    }
                }
                // this half's operand stores complete in global memory
                if (gleader) tc::bulk_wait0();
                tc::fence_proxy_async_global();
                // all epilogue warps meet here every half-step; the barrier also
                // ORs the abort flags so every warp leaves at the same point
                uint32_t any;
                asm volatile(
                    "{\n\t.reg .pred q, r;\n\tsetp.ne.u32 q, %1, 0;\n\t"
                    "barrier.red.or.pred r, 1, %2, q;\n\tselp.u32 %0, 1, 0, r;\n\t}"
                    : "=r"(any) : "r"((uint32_t)(!ok || *abort)), "n"(32 * kEpiWarps) : "memory");
                if (any) {
                    *abort = 1;
                    stop = true;
                } else if (ew == 0 && lane == 0) {
                    __threadfence();
                    atomicAdd(a.gbar + HV * nc + hh, 1u);
                }
            }
            // a marked state: the step's window sums, from the fluxes in TMEM
            if (m >= win0 && !in_win && !stop)
                for (int hh = 0; hh < HV; ++hh)
                    for (int c = csel; c < NC / 16; c += kGroups) {
                        const int col = hh * NC + c * 16;
                        win_plain_tmem(a.w + (size_t)(n0 + col) * a.Npad + row, a.Npad,
                                       tl + PHI0 + (uint32_t)col, row_ok);
                    }
        }
        // final phi for the output kernel (p is already in global memory)
        for (int hh = 0; hh < HV; ++hh)
            for (int c = csel; c < NC / 16; c += kGroups) {
                uint32_t v[16];
                tc::tmem_ld16(tl + PHI0 + (uint32_t)(hh * NC + c * 16), v);
                tc::tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    a.phi[(size_t)(n0 + hh * NC + c * 16 + j) * a.Npad + row] = __uint_as_float(v[j]);
            }
    }
    tc::tc_fence_before();
    __syncwarp();
    if constexpr (PAIR) tc::cluster_sync();
    else __syncthreads();
    if (*abort && threadIdx.x == 0) atomicOr(a.status, HQA_DEV_TIMEOUT);
    if (warp == 1) {
        tc::tc_fence_after();
        if constexpr (PAIR) tc::tmem_dealloc2(tmem, TMEM_COLS);
        else tc::tmem_dealloc(tmem, TMEM_COLS);
    }
}

// State set-up: phi(0), p(0) (SplitMix64 or caller-given), window sums 0,
// padding zero, and the slices of phi(0) in operand buffer 0 (step 0 writes all
// of buffer 1).
__global__ void k_f32_init(F32Args a, uint64_t seed, int init, const float* phi0, const float* p0)
{
    const size_t total = (size_t)a.Rpad * a.Npad;       // Npad is a multiple of 32: a warp
                                                        // holds the 32 spins of one unit
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(idx / a.Npad), i = (int)(idx % a.Npad);
        float phi = 0.f, p = 0.f;
        if (r < a.R && i < a.N) {
            const uint64_t c = ((uint64_t)(a.rep0 + r) << 32) | (uint64_t)i;
            if (init == HQA_INIT_GIVEN) {
                phi = phi0[(size_t)r * a.N + i];
                p = p0[(size_t)r * a.N + i];
            } else {
                uint64_t z = seed + (c + 1ull) * 0x9E3779B97F4A7C15ull;  // SplitMix64
                z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
                z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
                z ^= z >> 31;
                p = (z >> 63) ? -1.f : 1.f;
                if (init == HQA_INIT_RANDOM_FLUX) {
                    uint64_t y = seed + ((c | (1ull << 62)) + 1ull) * 0x9E3779B97F4A7C15ull;
                    y = (y ^ (y >> 30)) * 0xBF58476D1CE4E5B9ull;
                    y = (y ^ (y >> 27)) * 0x94D049BB133111EBull;
                    y ^= y >> 31;
                    phi = (float)((int64_t)(y >> 40) - (1 << 23)) * 0x1p-26f;
                }
            }
        }
        if (init == HQA_INIT_GIVEN && r < a.R && i < a.N && hqa_tiny_state(phi, p)) *a.tiny = 1u;
        a.phi[idx] = phi;
        a.p[idx] = p;
        a.w[idx] = 0.f;
        uint32_t b[3];
        slices2(hqa_dense::pk2(phi, 0.f), hqa_dense::pk2(round_const(__float_as_uint(phi), a.ushift), 1.f), b);
        uint16_t* o = a.phib + (size_t)r * 3 * a.Npad + i;
#pragma unroll
        for (int u = 0; u < 3; ++u) o[(size_t)u * a.Npad] = (uint16_t)b[u];
    }
}

// The power of two that bounds a row whose largest |J| has these bits: below 2^e,
// with e kept where the scale and the slices stay normal numbers.
__host__ __device__ inline int row_exponent(uint32_t bits)
{
    const int e = (int)(bits >> 23) - 126;
    return e < -100 ? -100 : e > 127 ? 127 : e;
}

// Row i of J as a_0 + a_1 + a_2 times a power of two (scale[i]): multiples of
// 2^-7 and two BF16 rests, for |J_ij| 2^-e <= 1.  One block per row of the
// [Mpad][3 Mpad] operand (zeroed before).  seen[0]: bit 0 some a_1, bit 1 some
// a_2 is not zero; seen[1]: the largest row sum of |a_0| in units of 2^-7.
__global__ void __launch_bounds__(256) k_f32_coupling_slices(
    const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
    const float* __restrict__ val, int N, int Mpad, uint16_t* __restrict__ out,
    float* __restrict__ scale, uint32_t* seen)
{
    __shared__ uint32_t s_big, s_sum;
    const int i = blockIdx.x;
    if (threadIdx.x == 0) s_big = s_sum = 0;
    __syncthreads();
    const int k0 = i < N ? row_ptr[i] : 0, k1 = i < N ? row_ptr[i + 1] : 0;
    uint32_t big = 0;
    for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x)
        big = max(big, __float_as_uint(fabsf(val[k])));
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_big, big);
    __syncthreads();
    const int e = row_exponent(s_big);
    if (threadIdx.x == 0) scale[i] = ldexpf(1.f, e);
    uint16_t* o = out + (size_t)i * 3 * Mpad;
    uint32_t some = 0, sum = 0;
    for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x) {
        const float x = ldexpf(val[k], -e);   // exact, like every difference below
        const auto b = [](float v) { return __float2bfloat16_rn(v); };
        const __nv_bfloat16 b0 = b(rintf(x * 0x1p7f) * 0x1p-7f);
        const float r1 = x - __bfloat162float(b0);
        const __nv_bfloat16 b1 = b(r1);
        const __nv_bfloat16 b2 = b(r1 - __bfloat162float(b1));
        o[col[k]] = __bfloat16_as_ushort(b0);
        o[Mpad + col[k]] = __bfloat16_as_ushort(b1);
        o[2 * Mpad + col[k]] = __bfloat16_as_ushort(b2);
        sum += (uint32_t)fabsf(__bfloat162float(b0) * 0x1p7f);
        some |= (__bfloat162float(b1) != 0.f ? 1u : 0u) | (__bfloat162float(b2) != 0.f ? 2u : 0u);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, sum);
    if (some) atomicOr(seen, some);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(seen + 1, s_sum);
}

struct Shape {
    int NC, HV;       // replicas per half, halves per CTA
    bool pair;
};

// Shared memory: alignment slack, ring, barrier block, staging tiles.
constexpr size_t f32_smem(int nc, int nj, bool pair, int ksub, int stages)
{
    return 1024 + (size_t)stages * ksub * (nj * A_BYTES + (pair ? 3 * nc / 2 : 3 * nc) * BK * 2) +
           1024 + kGroups * 3 * kStg;
}

constexpr int f32_stages(int nc, int nj, bool pair, int ksub)
{
    int s = 8;
    while (s > 0 && f32_smem(nc, nj, pair, ksub, s) > 227 * 1024 - 64) --s;
    return s;
}

// Two k-tiles per stage wherever two such stages fit (Npad is a multiple of
// 128, so the k-tiles pair up): the MMA thread pays for every stage it waits
// for (K2000 x 1024: 22.0 -> 18.4 us per step).
constexpr int f32_ksub(int nc, int nj, bool pair) { return f32_stages(nc, nj, pair, 2) >= 2 ? 2 : 1; }

template <int NC, int NJ, int HV, bool PAIR>
hqa_status launch_t(hqa_ctx* ctx, const F32Args& a, int grid, cudaStream_t st, const CUtensorMap& tmJ,
                    const CUtensorMap& tmB, const CUtensorMap& tmS)
{
    constexpr int KSUB = f32_ksub(NC, NJ, PAIR);
    constexpr int STAGES = f32_stages(NC, NJ, PAIR, KSUB);
    constexpr size_t smem = f32_smem(NC, NJ, PAIR, KSUB, STAGES);
    static_assert(STAGES >= 2, "ring depth");
    if (smem > ctx->smem_optin) return HQA_ERR_TOO_LARGE;
    const void* fn = (const void*)k_dense_f32<NC, NJ, HV, STAGES, KSUB, PAIR>;
    if (hqa_smem_attr(fn, smem) != cudaSuccess) return HQA_ERR_CUDA;
    void* args[] = {const_cast<CUtensorMap*>(&tmJ), const_cast<CUtensorMap*>(&tmB),
                    const_cast<CUtensorMap*>(&tmS), const_cast<F32Args*>(&a)};
    // every CTA co-resident (the column-group counters are waited on across
    // CTAs): a cooperative launch, or for pairs a cluster launch after an
    // occupancy check, as in dense_md_kernel.cuh
    cudaLaunchAttribute attr[1];
    if constexpr (PAIR) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if constexpr (PAIR) {
        int ncl = 0;
        if (cudaOccupancyMaxActiveClusters(&ncl, fn, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            return HQA_ERR_CUDA;
        }
        if (ncl < grid / 2) return HQA_ERR_TOO_LARGE;
    }
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        (void)cudaGetLastError();
        return HQA_ERR_TOO_LARGE;
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return hqa_capture_note(hqa_capturing() ? HQA_ERR_UNSUPPORTED : HQA_ERR_CUDA);
    }
    return HQA_OK;
}

template <int NC, int HV>
hqa_status launch_nj(hqa_ctx* ctx, const F32Args& a, int nj, bool pair, int grid, cudaStream_t st,
                     const CUtensorMap& tmJ, const CUtensorMap& tmB, const CUtensorMap& tmS)
{
    if constexpr (NC == 64) {
        if (pair) return launch_t<NC, 1, HV, true>(ctx, a, grid, st, tmJ, tmB, tmS);
    }
    return nj == 1 ? launch_t<NC, 1, HV, false>(ctx, a, grid, st, tmJ, tmB, tmS)
         : nj == 2 ? launch_t<NC, 2, HV, false>(ctx, a, grid, st, tmJ, tmB, tmS)
                   : launch_t<NC, 3, HV, false>(ctx, a, grid, st, tmJ, tmB, tmS);
}

hqa_status launch(hqa_ctx* ctx, const F32Args& a, const Shape& s, int nj, int grid, cudaStream_t st,
                  const CUtensorMap& tmJ, const CUtensorMap& tmB, const CUtensorMap& tmS)
{
    if (s.NC == 64 && s.HV == 2) return launch_nj<64, 2>(ctx, a, nj, s.pair, grid, st, tmJ, tmB, tmS);
    if (s.NC == 64) return launch_nj<64, 1>(ctx, a, nj, s.pair, grid, st, tmJ, tmB, tmS);
    if (s.NC == 32) return launch_nj<32, 1>(ctx, a, nj, s.pair, grid, st, tmJ, tmB, tmS);
    return launch_nj<16, 1>(ctx, a, nj, s.pair, grid, st, tmJ, tmB, tmS);
}

// Whether J is one BF16 slice, as k_f32_coupling_slices will find it, without
// building anything: a plan query needs to know, also during a capture.  The first
// coupling that is not a multiple of 2^-7 of its row's power of two ends the look.
bool one_slice(hqa_ctx* ctx)
{
    if (ctx->f32_nj) return ctx->f32_nj == 1;
    if (ctx->f32_one < 0) {
        ctx->f32_one = 1;
        for (int i = 0; i < ctx->N && ctx->f32_one && !ctx->j_whole; ++i) {
            float big = 0.f;
            for (int64_t k = ctx->row_ptr[i]; k < ctx->row_ptr[i + 1]; ++k)
                big = std::max(big, std::fabs(ctx->val[k]));
            uint32_t bits;
            std::memcpy(&bits, &big, 4);
            for (int64_t k = ctx->row_ptr[i]; k < ctx->row_ptr[i + 1]; ++k) {
                const float x = std::ldexp(ctx->val[k], 7 - row_exponent(bits));
                if (x != std::rint(x)) {
                    ctx->f32_one = 0;
                    break;
                }
            }
        }
    }
    return ctx->f32_one == 1;
}

// Replicas one launch takes: as many column groups as fit next to the row
// tiles with one CTA per SM.
int chunk_replicas(const hqa_ctx* ctx, const Shape& s)
{
    return (ctx->sm_count / (ctx->Mpad / BM)) * s.HV * s.NC;
}

// The narrowest tile that runs all replicas in one launch (a narrow tile
// spreads few replicas over more SMs), else the widest.
Shape pick_shape(hqa_ctx* ctx, int R)
{
    const bool pairs = one_slice(ctx) && (ctx->Mpad / BM) % 2 == 0;
    const Shape c[4] = {{16, 1, false}, {32, 1, false}, {64, 1, pairs}, {64, 2, pairs}};
    for (int k = 0; k < 3; ++k)
        if (R <= chunk_replicas(ctx, c[k])) return c[k];
    return c[3];
}

}  // namespace

bool hqa_f32tc_possible(const hqa_ctx* ctx)
{
    return !ctx->is_batch && ctx->dense_input && ctx->dense_tc && ctx->Mpad / BM <= ctx->sm_count;
}

// k of the slice unit: units fine enough for 2^k steps up to the group's largest
// power of two, coarse enough that a row's sum of `lsb` coupling units stays
// exact.  Beyond k = 7 (whole couplings) b0 holds no more bits; real ones gain
// up to 10, where the products a_1 b_2 and a_2 b_1 that are left out are smaller.
// Below 5 the rests would miss bits: there only sums of one sign can be truncated.
static int unit_steps(double sum, bool whole)
{
    const int k = 23 - (int)std::ceil(std::log2(std::max(sum, 1.0)));
    return std::max(5, std::min(k, whole ? 7 : 10));
}

// Coupling slices, built on first use: the BF16 copy of J when J is whole
// numbers up to 127, else up to three slices per row.
hqa_status hqa_f32tc_prepare(hqa_ctx* ctx)
{
    if (ctx->f32_nj) return HQA_OK;
    if (!hqa_f32tc_possible(ctx)) return HQA_ERR_UNSUPPORTED;
    if (ctx->j_whole) {
        int64_t most = 0;
        for (int i = 0; i < ctx->N; ++i) most = std::max(most, ctx->row_ptr[i + 1] - ctx->row_ptr[i]);
        ctx->f32_k = unit_steps((double)most * ctx->j_max, true);
        ctx->f32_nj = 1;
        return HQA_OK;
    }
    if (hqa_capturing()) return hqa_capture_note(HQA_ERR_UNSUPPORTED);
    const size_t Mp = (size_t)ctx->Mpad, bytes = 3 * Mp * Mp * sizeof(uint16_t);
    // kept by the context also when a later call here fails: the next one goes on with them
    if (!ctx->d_Jsl) HQA_CUDA_TRY(cudaMalloc(&ctx->d_Jsl, bytes));
    if (!ctx->d_Jscale) HQA_CUDA_TRY(cudaMalloc(&ctx->d_Jscale, (Mp + 2) * sizeof(float)));
    HQA_CUDA_TRY(cudaMemset(ctx->d_Jsl, 0, bytes));
    HQA_CUDA_TRY(cudaMemset(ctx->d_Jscale, 0, (Mp + 2) * sizeof(float)));
    uint32_t* d_seen = reinterpret_cast<uint32_t*>(ctx->d_Jscale + Mp);
    k_f32_coupling_slices<<<ctx->Mpad, 256>>>(ctx->d_row_ptr, ctx->d_col, ctx->d_val, ctx->N,
                                              ctx->Mpad, static_cast<uint16_t*>(ctx->d_Jsl),
                                              ctx->d_Jscale, d_seen);
    HQA_CUDA_TRY(cudaGetLastError());
    uint32_t seen[2] = {0, 0};
    HQA_CUDA_TRY(cudaMemcpy(seen, d_seen, sizeof(seen), cudaMemcpyDeviceToHost));
    if (!hqa_dense_tmap16(&ctx->tmJsl, ctx->d_Jsl, Mp, 3 * Mp, BK, BM, true, false)) return HQA_ERR_CUDA;
    ++ctx->generation;
    ctx->f32_k = unit_steps(seen[1], false);
    ctx->f32_nj = (seen[0] & 2u) ? 3 : (seen[0] & 1u) ? 2 : 1;
    return HQA_OK;
}

void hqa_f32tc_plan(hqa_ctx* ctx, int32_t R, int* rb, int* grid, int* chunks)
{
    const Shape sh = pick_shape(ctx, R);
    const int Rc = chunk_replicas(ctx, sh);
    *chunks = (R + Rc - 1) / Rc;
    const int per = (R + *chunks - 1) / *chunks;
    *rb = sh.HV * sh.NC;
    *grid = ctx->Mpad / BM * ((per + *rb - 1) / *rb);
}

static hqa_status f32_chunk(hqa_ctx* ctx, const Shape& sh, const StepCoef* d_sched, int64_t S,
                            int32_t W, int32_t R, int32_t rep0, uint64_t seed, int init,
                            const float* phi0, const float* p0, int M, float* phi_out, float* p_out,
                            float* phibar_out, cudaStream_t st)
{
    const int Mt = ctx->Mpad / BM, cols = sh.HV * sh.NC;
    const int Nc = (R + cols - 1) / cols, Rpad = Nc * cols, groups = Nc * sh.HV;
    const size_t n = (size_t)Rpad * ctx->Mpad;
    // state: phi, p, w (FP32), two operand buffers of three slices, group counters,
    // the mark of a tiny state
    const size_t off_b = 3 * n * 4, off_g = off_b + 2 * 3 * n * 2;
    const size_t need = off_g + ((size_t)groups + 1) * 4;
    hqa_status s = hqa_reserve(ctx, &ctx->d_state, &ctx->state_cap, need);
    if (s != HQA_OK) return s;
    char* b = static_cast<char*>(ctx->d_state);
    F32Args a{};
    a.phi = reinterpret_cast<float*>(b);
    a.p = a.phi + n;
    a.w = a.p + n;
    a.phib = reinterpret_cast<uint16_t*>(b + off_b);
    a.gbar = reinterpret_cast<unsigned int*>(b + off_g);
    a.tiny = a.gbar + groups;
    a.sched = d_sched;
    a.h = ctx->has_h ? ctx->d_h : nullptr;
    a.rscale = ctx->d_Jscale;
    a.status = ctx->d_status;
    a.S = S;
    a.W = W;
    a.N = ctx->N;
    a.Npad = ctx->Mpad;
    a.Rpad = Rpad;
    a.R = R;
    a.KT = ctx->Mpad / BK;
    a.Mt = Mt;
    a.M = M;
    a.rep0 = rep0;
    a.ushift = (uint32_t)(23 - ctx->f32_k) << 23;
    CUtensorMap tmB, tmS;
    if (!hqa_dense_tmap16(&tmB, a.phib, (uint64_t)2 * Rpad, (uint64_t)3 * ctx->Mpad, BK,
                          sh.pair ? sh.NC / 2 : sh.NC, true, false) ||
        !hqa_dense_tmap16(&tmS, a.phib, (uint64_t)2 * Rpad, (uint64_t)3 * ctx->Mpad, 128, 16, false, false))
        return HQA_ERR_CUDA;
    if (cudaMemsetAsync(a.gbar, 0, ((size_t)groups + 1) * 4, st) != cudaSuccess) return HQA_ERR_CUDA;
    const int g = (int)std::min<size_t>(8192, (n + 255) / 256);
    k_f32_init<<<g, 256, 0, st>>>(a, seed, init, phi0, p0);
    s = launch(ctx, a, sh, ctx->f32_nj, Mt * Nc, st, ctx->d_Jsl ? ctx->tmJsl : ctx->tmJ, tmB, tmS);
    if (s != HQA_OK) return s;
    hqa_dense::DenseMDArgs o{};
    o.phi = a.phi;
    o.p = a.p;
    o.w = a.w;
    o.status = a.status;
    o.N = a.N;
    o.Npad = a.Npad;
    o.R = R;
    hqa_dense::k_dense_out<<<(int)std::min<size_t>(8192, ((size_t)R * ctx->N + 255) / 256), 256, 0, st>>>(
        o, 1.0f / (float)(S < W ? S : W), phi_out, p_out, phibar_out);
    return cudaGetLastError() == cudaSuccess ? HQA_OK : HQA_ERR_CUDA;
}

hqa_status hqa_f32tc_launch_md(hqa_ctx* ctx, const StepCoef* d_sched, int64_t S, int32_t W,
                               int32_t R, uint64_t seed, int init, const float* phi0,
                               const float* p0, int M, float* phi_out, float* p_out,
                               float* phibar_out, cudaStream_t st)
{
    hqa_status s = hqa_f32tc_prepare(ctx);
    if (s != HQA_OK) return s;
    const Shape sh = pick_shape(ctx, R);
    const int most = chunk_replicas(ctx, sh);
    const int C = (R + most - 1) / most, Rc = (R + C - 1) / C;
    for (int r0 = 0; r0 < R; r0 += Rc) {
        const size_t o = (size_t)r0 * ctx->N;
        s = f32_chunk(ctx, sh, d_sched, S, W, std::min(Rc, R - r0), r0, seed, init,
                      phi0 ? phi0 + o : nullptr, p0 ? p0 + o : nullptr, M,
                      phi_out ? phi_out + o : nullptr, p_out ? p_out + o : nullptr,
                      phibar_out ? phibar_out + o : nullptr, st);
        if (s != HQA_OK) return s;
    }
    return HQA_OK;
}
