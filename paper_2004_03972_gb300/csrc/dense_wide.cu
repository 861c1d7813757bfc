// dense_wide.cu -- the 16-bit dense MD of large instances: 256 x 256 tiles dealt
// to CTA pairs across steps.
//
// The persistent kernel of dense_md_kernel.cuh gives every CTA one row tile for
// the whole run.  From N about 4900 on its grid cannot hold two or three column
// groups (N = 10000: 79 row tiles on 152 SMs, 1024 replicas in two runs one after
// another), its column tiles no longer fit on chip, and an SM takes in 48 KB per
// k-tile for 128 x 256 outputs, all that its 64 B/clk from L2 allow.
//
// Here the work of a step is cut into units of 256 spins x 256 replicas, one
// cta_group::2 MMA tile (M = 256, N = 256), which takes in 32 KB per k-tile and
// CTA.  Units are numbered step by step, within a step by column block and then
// by row tile, and pair p of the grid takes units p, p + P, p + 2 P, ...: a step's
// uneven rest flows into the next step.  A unit of step m needs all row tiles of
// its column block at step m - 1 and nothing else; those come about one step's
// worth of units earlier, so the wait is short, and since every pair takes its
// units in order and a unit depends on smaller numbers only, some pair can always
// go on.  State (phi, p, FP32) lives in global memory and passes between SMs with
// the operand; reads of it bypass L1.
//
// Per pair: a TMA producer warp, an MMA warp (issued by the even CTA, the odd one
// relays landed stages), 8 epilogue warps, two accumulators of 256 columns, so that
// a unit's epilogue runs under the next unit's MMAs.  Products accumulate in the
// order of the kernel above (K runs over [hi | hi | lo] segments, or hi and lo per
// k-tile for an exact J), so results are bit for bit the same.
//
// N = 10000 x 1024 replicas, BF16x2 (three passes), per step: 714 -> 486 us, 1.26
// PFLOP/s issued.  What bounds it: an SM takes in 66 GB/s, all of them together 10
// TB/s from L2, half of that from DRAM through it (J's 607 MB pass about twice a
// step, 2.6 TB/s), at a clock that the power limit lowers.
#include <algorithm>

#include "dense_md_kernel.cuh"

namespace {

using hqa_dense::BK;
using hqa_dense::BM;
using hqa_dense::kWaitNs;

constexpr int kEpiWarps = 8;
constexpr int kCS = kEpiWarps / 4;            // chunk stride: warps per lane quarter
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kNU = 256;                      // replicas per unit
constexpr int kKSub = 2;                      // k-tiles per ring stage
constexpr uint32_t A_BYTES = BM * BK * 2;
constexpr uint32_t B_BYTES = kNU / 2 * BK * 2;   // this CTA's half of a phi tile

struct WideArgs {
    hqa_dense::DenseMDArgs a;
    int RT, CB;            // row tiles of 256, column blocks of 256
};

template <int KSEG>
constexpr uint32_t kStage = kKSub * (A_BYTES + (KSEG == 2 ? 2 : 1) * B_BYTES);
template <int KSEG>
constexpr int kStages = KSEG == 2 ? 2 : 3;

template <int KSEG>
constexpr size_t wide_smem() { return 1024 + (size_t)kStages<KSEG> * kStage<KSEG> + 1024; }

// The window sums of a thread's chunks of a unit without reductions.  Out of line:
// within the unit's code it cost N = 5400 x 1000 BF16 1.2 of 49.6 us a step.
__device__ __noinline__ void win_plain_unit(float* w, const float* phi, int Npad)
{
#pragma unroll 1
    for (int c = 0; c < kNU / 16 / kCS; ++c)
#pragma unroll 1
        for (int j = 0; j < 16; ++j) {
            const size_t o = (size_t)(c * kCS * 16 + j) * Npad;
            hqa_dense::win_plain(w + o, *(const volatile float*)(phi + o));
        }
}

template <int KSEG, bool F16>
__global__ void __launch_bounds__(kThreads, 1)
k_dense_wide(const __grid_constant__ CUtensorMap tmJ, const __grid_constant__ CUtensorMap tmB,
             const WideArgs w)
{
    constexpr uint32_t STAGE = kStage<KSEG>;
    constexpr int STAGES = kStages<KSEG>;
    constexpr uint32_t B_OFF = kKSub * A_BYTES, B2_OFF = B_OFF + kKSub * B_BYTES;
    const hqa_dense::DenseMDArgs& a = w.a;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bar = base + STAGES * STAGE;
    const uint32_t full0 = bar, empty0 = bar + 8 * STAGES, pfull0 = bar + 16 * STAGES;
    const uint32_t accf0 = bar + 24 * STAGES, acce0 = accf0 + 16, tmem_slot = accf0 + 32,
                   done_bar = accf0 + 40;
    __shared__ int s_abort;
    __shared__ uint32_t s_tiny;   // *a.tiny: here, as a register held through the steps costs up to 3 %
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t crank = tc::cluster_rank();
    const int64_t U = (int64_t)w.RT * w.CB, total = U * a.S;
    const int64_t first = blockIdx.x / 2, P = gridDim.x / 2;

    if (threadIdx.x == 0) {
        s_abort = 0;
        s_tiny = __ldcg(a.tiny);
        for (int s = 0; s < STAGES; ++s) {
            tc::mbar_init(full0 + 8 * s, 1);
            tc::mbar_init(empty0 + 8 * s, 1);
            tc::mbar_init(pfull0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(accf0 + 8 * b, 1);
            tc::mbar_init(acce0 + 8 * b, 2 * kEpiWarps);
        }
        tc::mbar_init(done_bar, 1);
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tmJ);
        tc::prefetch_tmap(&tmB);
    }
    if (warp == 1) {
        tc::tmem_alloc2(tmem_slot, 512);
        tc::tmem_relinquish2();
    }
    tc::tc_fence_before();
    tc::cluster_sync();   // the peer's barriers exist before any remote arrive
    tc::tc_fence_after();
    uint32_t tmem;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem) : "r"(tmem_slot));
    volatile int* abort = &s_abort;
    volatile uint32_t* gstatus = a.status;
    const int KTT = (KSEG == 2 ? a.KT : KSEG * a.KT) / kKSub;   // ring stages per unit

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer ----
            uint32_t it = 0;
            for (int64_t g = first; g < total && !*abort; g += P) {
                const int64_t m = g / U;
                const int u = (int)(g % U), cb = u / w.RT, rt = u % w.RT;
                if (a.wait_flag && m == a.wait_step) {
                    const uint64_t t0 = tc::globaltimer();
                    uint32_t spins = 0;
                    while (hqa_dense::ld_acquire(a.wait_flag) == 0u) {
                        if ((++spins & 63u) == 0 && (*abort || tc::globaltimer() - t0 > a.wait_ns)) {
                            *abort = 1;
                            break;
                        }
                    }
                    if (*abort) break;
                }
                if (m > 0) {
                    // both CTAs of all RT pairs of the column block finished step m - 1
                    const unsigned int target = (unsigned int)(2 * w.RT * m);
                    const uint64_t t0 = tc::globaltimer();
                    uint32_t spins = 0;
                    while (hqa_dense::ld_acquire(a.gbar + cb) < target) {
                        if ((++spins & 63u) == 0) {
                            if (*abort || (*gstatus & HQA_DEV_TIMEOUT)) { *abort = 1; break; }
                            if (tc::globaltimer() - t0 > kWaitNs) { *abort = 1; break; }
                        }
                    }
                    if (*abort) break;
                    tc::fence_proxy_async_global();
                }
                const int m0 = rt * 2 * BM + (int)crank * BM;
                const int brow = (int)(m & 1) * a.Rpad + cb * kNU + (int)crank * (kNU / 2);
                for (int kt = 0; kt < KTT; ++kt, ++it) {
                    const int s = it % STAGES;
                    if (it >= STAGES &&
                        !tc::mbar_wait_cl(empty0 + 8 * s, ((it / STAGES) - 1) & 1, abort, kWaitNs))
                        break;
                    const uint32_t sa = base + s * STAGE;
                    tc::mbar_expect_tx(full0 + 8 * s, STAGE);
#pragma unroll
                    for (int k = 0; k < kKSub; ++k) {
                        const int x = (kt * kKSub + k) * BK;
                        tc::tma_load_2d(sa + k * A_BYTES, &tmJ, x, m0, full0 + 8 * s);
                        tc::tma_load_2d(sa + B_OFF + k * B_BYTES, &tmB, x, brow, full0 + 8 * s);
                        if constexpr (KSEG == 2)
                            tc::tma_load_2d(sa + B2_OFF + k * B_BYTES, &tmB, a.Npad + x, brow,
                                            full0 + 8 * s);
                    }
                }
            }
            // drain: every issued stage must land before the CTA can exit
            if (*abort)
                for (uint32_t k = (it > STAGES ? it - STAGES : 0); k < it; ++k) {
                    volatile int no_abort = 0;
                    tc::mbar_wait(full0 + 8 * (k % STAGES), (k / STAGES) & 1, &no_abort, 20000000ull);
                }
        }
    } else if (warp == 1) {
        if (lane == 0 && crank != 0) {
            // ---- odd CTA: relay each landed stage to the MMA issuer ----
            uint32_t it = 0;
            const uint32_t peer = tc::mapa(pfull0, 0);
            for (int64_t g = first; g < total && !*abort; g += P)
                for (int kt = 0; kt < KTT; ++kt, ++it) {
                    const int s = it % STAGES;
                    if (!tc::mbar_wait(full0 + 8 * s, (it / STAGES) & 1, abort, kWaitNs)) break;
                    tc::mbar_arrive_remote(peer + 8 * s);
                }
        } else if (lane == 0) {
            // ---- MMA issuer ----
            constexpr uint32_t idesc = F16 ? tc::idesc_f16(2 * BM, kNU) : tc::idesc_bf16(2 * BM, kNU);
            uint32_t it = 0, i = 0;
            for (int64_t g = first; g < total && !*abort; g += P, ++i) {
                const uint32_t b = i & 1u;
                if (i >= 2 && !tc::mbar_wait_cl(acce0 + 8 * b, ((i >> 1) - 1) & 1, abort, kWaitNs)) break;
                tc::tc_fence_after();
                const uint32_t d = tmem + b * kNU;
                for (int kt = 0; kt < KTT; ++kt, ++it) {
                    const int s = it % STAGES;
                    if (!tc::mbar_wait(full0 + 8 * s, (it / STAGES) & 1, abort, kWaitNs)) break;
                    if (!tc::mbar_wait_cl(pfull0 + 8 * s, (it / STAGES) & 1, abort, kWaitNs)) break;
                    tc::tc_fence_after();
                    const uint32_t sa = base + s * STAGE;
#pragma unroll
                    for (int k = 0; k < kKSub; ++k) {
                        const uint64_t ad = tc::sdesc_k128(sa + k * A_BYTES);
                        const uint64_t bd = tc::sdesc_k128(sa + B_OFF + k * B_BYTES);
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk)
                            tc::mma2_f16(d, ad + 2 * kk, bd + 2 * kk, idesc, (kt | k | kk) != 0);
                        if constexpr (KSEG == 2) {   // J phi_lo into the same accumulator
                            const uint64_t bd1 = tc::sdesc_k128(sa + B2_OFF + k * B_BYTES);
#pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk)
                                tc::mma2_f16(d, ad + 2 * kk, bd1 + 2 * kk, idesc, 1u);
                        }
                    }
                    tc::mma_commit2(empty0 + 8 * s, 3);
                }
                tc::mma_commit2(accf0 + 8 * b, 3);
            }
            // every MMA issued completes before either CTA frees its memory
            volatile int no_abort = 0;
            tc::mma_commit2(done_bar, 1);
            tc::mbar_wait_cl(done_bar, 0, &no_abort, kWaitNs);
        }
    } else {
        // ---- epilogue warps: kick, drift, 16-bit operand, window ----
        using namespace hqa_dense;
        const int ew = warp - 2;
        const int quarter = warp & 3;         // TMEM lanes 32 quarter .. +31
        const int csel = ew >> 2;             // first chunk of this warp
        const uint32_t tl = tmem + ((uint32_t)(32 * quarter) << 16);
        const uint32_t acce_to = crank != 0 ? tc::mapa(acce0, 0) : acce0;
        const int mhalf = (a.M - 2) / 2;
        const int64_t win0 = a.S - (int64_t)a.W;
        const int Kb = KSEG * a.Npad;         // operand row: [hi], [hi | lo] or [hi | hi | lo]
        bool stop = false;
        uint32_t i = 0;
        for (int64_t g = first; g < total && !stop; g += P, ++i) {
            const int64_t m = g / U;
            const int u = (int)(g % U), cb = u / w.RT, rt = u % w.RT;
            const uint32_t b = i & 1u;
            const float4 cf = __ldg(reinterpret_cast<const float4*>(a.sched) + m);
            const bool in_win = m >= win0 && *(volatile uint32_t*)&s_tiny == 0u;
            const int row = rt * 2 * BM + (int)crank * BM + 32 * quarter + lane;
            const bool row_ok = row < a.N;
            const float hr = (a.h && row_ok) ? 2.f * __ldg(a.h + row) : 0.f;
            uint16_t* nb = a.phib + (size_t)((m + 1) & 1) * a.Rpad * Kb;
            const bool ok = __all_sync(
                0xffffffffu, tc::mbar_wait_cl(accf0 + 8 * b, (i >> 1) & 1, abort, kWaitNs));
            tc::tc_fence_after();
            if (ok) {
                // the state was written by other CTAs: their arrivals on the block's
                // counter are acquired here too, and the reads bypass L1
                if (lane == 0 && m > 0) (void)ld_acquire(a.gbar + cb);
                __syncwarp();
                float ph[16], pp[16];
                const auto load = [&](int c, float (&f)[16], float (&q)[16]) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const size_t o = (size_t)(cb * kNU + c * 16 + j) * a.Npad + row;
                        f[j] = __ldcg(a.phi + o);
                        q[j] = __ldcg(a.p + o);
                    }
                };
                if (row_ok) load(csel, ph, pp);
#pragma unroll 1
                for (int c = csel; c < kNU / 16; c += kCS) {
                    uint32_t v[16];
                    tc::tmem_ld16(tl + b * kNU + (uint32_t)(c * 16), v);
                    float nph[16], npp[16];
                    const bool more = row_ok && c + kCS < kNU / 16;
                    if (more) load(c + kCS, nph, npp);
                    tc::tmem_wait_ld();
                    if (row_ok) {
                        const int rbase = cb * kNU + c * 16;
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const size_t o = (size_t)(rbase + j) * a.Npad + row;
                            const float L = __uint_as_float(v[j]) * a.lscale + hr * fabsf(ph[j]);
                            const float phi2 = ph[j] * ph[j];
                            const float pw = pot_pow(ph[j], phi2, mhalf);
                            const float pn = pp[j] - fmaf(cf.x, pw, cf.y * L);
                            const float fn = fmaf(cf.z, pn, ph[j]);
                            __stcg(a.p + o, pn);
                            __stcg(a.phi + o, fn);
                            const size_t ob = (size_t)(rbase + j) * Kb + row;
                            const float fs = fn * a.oscale;
                            const uint16_t hi = cvt16<F16>(fs);
                            nb[ob] = hi;
                            if (KSEG == 2) nb[ob + a.Npad] = cvt16<F16>(fs - from16<F16>(hi));
                            if (KSEG == 3) {
                                nb[ob + a.Npad] = hi;
                                nb[ob + 2 * a.Npad] = cvt16<F16>(fs - from16<F16>(hi));
                            }
                            if (in_win) win_add(a.w + o, fn);
                        }
                    }
                    if (more) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            ph[j] = nph[j];
                            pp[j] = npp[j];
                        }
                    }
                }
                // the accumulator may be overwritten once every epilogue warp has read it
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (crank != 0) tc::mbar_arrive_remote(acce_to + 8 * b);
                    else tc::mbar_arrive(acce0 + 8 * b);
                }
                // a marked state: the unit's window sums, before another pair may have it
                if (m >= win0 && !in_win && row_ok)
                    win_plain_unit(a.w + (size_t)(cb * kNU + csel * 16) * a.Npad + row,
                                   a.phi + (size_t)(cb * kNU + csel * 16) * a.Npad + row, a.Npad);
            }
            // operand and state -> visible to the other CTAs' TMA loads and reads
            tc::fence_proxy_async_global();
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
                atomicAdd(a.gbar + cb, 1u);
            }
        }
    }
    tc::tc_fence_before();
    __syncwarp();
    tc::cluster_sync();
    if (*abort && threadIdx.x == 0) atomicOr(a.status, HQA_DEV_TIMEOUT);
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc2(tmem, 512);
    }
}

template <int KSEG, bool F16>
hqa_status launch_t(hqa_ctx* ctx, const WideArgs& w, cudaStream_t st, const CUtensorMap& tmA,
                    const CUtensorMap& tmB)
{
    constexpr size_t smem = wide_smem<KSEG>();
    if (smem > ctx->smem_optin) return HQA_ERR_TOO_LARGE;
    const void* fn = (const void*)k_dense_wide<KSEG, F16>;
    if (hqa_smem_attr(fn, smem) != cudaSuccess) return HQA_ERR_CUDA;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (ctx->sm_count / 2));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // every pair co-resident (units wait for units of other pairs)
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, fn, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return HQA_ERR_CUDA;
    }
    const int64_t units = (int64_t)w.RT * w.CB;
    const int pairs = (int)std::min<int64_t>(std::min(ncl, ctx->sm_count / 2), units);
    if (pairs < 1) return HQA_ERR_TOO_LARGE;
    cfg.gridDim = dim3(2 * pairs);
    void* args[] = {const_cast<CUtensorMap*>(&tmA), const_cast<CUtensorMap*>(&tmB),
                    const_cast<WideArgs*>(&w)};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return hqa_capture_note(hqa_capturing() ? HQA_ERR_UNSUPPORTED : HQA_ERR_CUDA);
    }
    return HQA_OK;
}

}  // namespace

// Replicas per column block.
int hqa_wide_block() { return kNU; }

hqa_status hqa_wide_launch(hqa_ctx* ctx, const hqa_dense::DenseMDArgs& a, int kseg, bool f16,
                           cudaStream_t st, const CUtensorMap& tmA, const CUtensorMap& tmB)
{
    WideArgs w;
    w.a = a;
    w.RT = (a.Mt + 1) / 2;
    w.CB = a.Rpad / kNU;
    if (a.Rpad % kNU != 0 || a.KT % kKSub != 0) return HQA_ERR_INVALID_ARG;
    if (f16)
        return kseg == 3 ? launch_t<3, true>(ctx, w, st, tmA, tmB)
             : kseg == 2 ? launch_t<2, true>(ctx, w, st, tmA, tmB)
                         : launch_t<1, true>(ctx, w, st, tmA, tmB);
    return kseg == 3 ? launch_t<3, false>(ctx, w, st, tmA, tmB)
         : kseg == 2 ? launch_t<2, false>(ctx, w, st, tmA, tmB)
                     : launch_t<1, false>(ctx, w, st, tmA, tmB);
}
