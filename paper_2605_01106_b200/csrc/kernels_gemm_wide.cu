// Projection for hundreds of activation rows (prompt passes, large batches): the contraction of kernels_gemm_tc.cu -
// D = W x^T, weights as the M operand, activations as bf16 head + bf16 remainder - where the tensor pipe, not the
// weight stream, is the bound.
//  * A pair of CTAs (tcgen05 cta_group::2) works on a tile of 256 weight rows x n activation rows: each CTA stages its own
//    128 weight rows and half of the packed activation rows, so a K block of 64 costs 16 KB + 128 n bytes of L2 reads per SM.
//  * n <= 128: head and remainder are the two halves of the MMA's N = 2 n columns (one CTA stages the heads, the other the
//    remainders).  n > 128: both planes go into the SAME n columns, two MMAs per K step.  Consecutive MMAs on one accumulator
//    follow each other no faster than about 115 cycles, so a narrow tile (n <= 64) takes its K steps in turn through two
//    accumulators and the epilogue adds them (measured at n = 64, both planes into one accumulator: 921 cycles per K
//    block instead of 256).
//  * Two accumulator buffers of 256 columns: the epilogue of a tile runs while the next tile is contracted.
//  * A sum in tensor memory loses about 2^-26 of itself per MMA to truncation, and a spread of 0.6 of that around this mean
//    (gemm_tc_common.cuh).  The mean is put back; against the spread a chain ends after 64 MMAs: longer K ranges (SEG) go
//    through the two buffers in segments that the epilogue warps add up in fp32 registers.  Segments of 16 or 32 MMAs are
//    shorter than the way from the commit through the epilogue to the issuer and back (3B-class prompt of 2048: 58 and 61
//    instead of 53 ms).
//  * One persistent CTA per SM; warp roles: eight epilogue warps (twelve where they hold the sums), one TMA producer, one
//    MMA issuer.
//  * n is a run-time multiple of 16 chosen by the launcher so that the tiles fill the GPU evenly (a residual projection
//    of the 3B-class model at 2048 rows: n = 96 gives 220 tiles for 74 pairs; n = 256 would leave a second round almost
//    empty).
// No K split: at these sizes there are enough tiles, so nothing is exchanged between pairs.  Every wait is bounded.
#include "hs_internal.h"
#include "hs_device.cuh"
#include "gemm_tc_common.cuh"
#include <algorithm>

namespace {
using namespace hsd;

__host__ __device__ constexpr int gw_epi_warps(bool seg) { return seg ? 12 : 8; }
__host__ __device__ constexpr int gw_threads(bool seg) { return (gw_epi_warps(seg) + 2) * 32; }
constexpr int GW_MAXSTAGES = 8;
constexpr int GW_CHAIN = 64;        // MMAs that add up in one accumulator, at most
constexpr int GW_GROUPS = 11;       // groups of eight activation rows a thread of the epilogue holds: a third of n = 256
constexpr uint32_t GW_A_BYTES = TC_BM * TC_BK * 2;
constexpr size_t GW_SMEM_MAX = 220 * 1024;
constexpr size_t GW_MISC_BYTES = (256 + 128 + 4 * 256) * 4;       // rstd[n], next norm weights[128], sums of squares [4][n]

// the leader CTA of a pair has the even rank: its barriers collect the bytes of both
__device__ __forceinline__ uint32_t leader_bar(uint64_t *bar) { return smem_u32(bar) & 0xFEFFFFFFu; }
__device__ __forceinline__ void tma_pair_2d(void *dst_smem, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(smem_u32(dst_smem)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n\t}"
                 :: "r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(0u) : "memory");
}
// arrives on the barrier at this offset in both CTAs of the pair
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 :: "r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
// the eight registers of a tensor-memory load are valid behind this
__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]) :: "memory");
}

// t.bnh: activation rows per tile (n); t.ns: stages; t.rb: accumulators a narrow tile alternates between; t.seg: K blocks
// per segment.  grid = 2 x pairs, clusters of two along x.
template <int EPI, bool SEG>
__global__ void __launch_bounds__(gw_threads(SEG), 1)
gemm_wide_kernel(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
                 const __grid_constant__ CUtensorMap mB, const TcArgs a, const int ntiles, const int mtiles) {
    constexpr int EPI_WARPS = gw_epi_warps(SEG);
    auto epi_sync = [] { asm volatile("bar.sync 1, %0;" :: "n"(EPI_WARPS * 32) : "memory"); };
    extern __shared__ unsigned char smraw[];
    __shared__ __align__(8) uint64_t full_bar[GW_MAXSTAGES], empty_bar[GW_MAXSTAGES], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_s;
    const uint32_t sbase = (smem_u32(smraw) + 1023u) & ~1023u;
    unsigned char *stages = smraw + (sbase - smem_u32(smraw));
    const int n = a.bnh, nk = a.nk0 + a.nk1, NS = a.ns;
    const bool cat = n <= 128;                        // planes side by side
    const uint32_t BB = (uint32_t)n * TC_BK * 2, STAGE = GW_A_BYTES + BB;      // BB: this CTA's share of the activation rows
    float *rstd_s = reinterpret_cast<float *>(stages + a.off_misc);       // [256]
    float *nw_s = rstd_s + 256;                                           // [128]
    float *ssred = nw_s + 128;                                            // [4][256]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)(blockIdx.x & 1), pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1), total = ntiles * mtiles;
    if (tid == 0) {
        for (int s = 0; s < NS; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 2 * EPI_WARPS); }
        mbar_fence_init();
    }
    if (warp == EPI_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&tmem_base_s)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_arrive(); cluster_wait();                 // both CTAs' barriers exist before either signals the other's
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_base_s;
    bool ok = true;
    auto wait = [](uint64_t *bar, uint32_t parity) { return mbar_wait_n(bar, parity, 1 << 20); };

    if (warp == EPI_WARPS) {
        // ---- TMA producer: this CTA's weight rows and its half of the activation rows; bytes counted at the leader
        if (lane == 0) {
            const int first_end = nk < NS ? nk : NS;
            auto load_a = [&](int s, int kb, int m0) {
                if (rank == 0) mbar_expect_tx(&full_bar[s], 2 * STAGE);
                const uint32_t bar = leader_bar(&full_bar[s]);
                if (kb < a.nk0) tma_pair_2d(stages + (size_t)s * STAGE, &mA0, kb * TC_BK, m0, bar);
                else tma_pair_2d(stages + (size_t)s * STAGE, &mA1, (kb - a.nk0) * TC_BK, m0, bar);
            };
            auto load_b = [&](int s, int kb, int n0) {
                unsigned char *bs = stages + (size_t)s * STAGE + GW_A_BYTES;
                const uint32_t bar = leader_bar(&full_bar[s]);
                if (cat) { tma_pair_2d(bs, &mB, kb * TC_BK, rank * a.rpad + n0, bar); return; }
                tma_pair_2d(bs, &mB, kb * TC_BK, n0 + rank * (n / 2), bar);
                tma_pair_2d(bs + BB / 2, &mB, kb * TC_BK, a.rpad + n0 + rank * (n / 2), bar);
            };
            int s = 0; uint32_t ph = 0;
            bool waited = false;
            for (int tile = pair; tile < total && ok; tile += npairs) {
                const int m0 = (tile / ntiles) * 2 * TC_BM + rank * TC_BM, n0 = (tile % ntiles) * n;
                int kb0 = 0;
                if (!waited) {                        // the first stages' weights depend on nothing
                    for (int kb = 0; kb < first_end; ++kb) load_a(kb, kb, m0);
                    pdl_wait();
                    for (int kb = 0; kb < first_end; ++kb) load_b(kb, kb, n0);
                    waited = true;
                    kb0 = first_end;
                    s = first_end; if (s == NS) { s = 0; ph = 1; }
                }
                for (int kb = kb0; kb < nk; ++kb) {
                    // the first pass over the ring finds every stage free: the barrier's phase before any completion
                    if (!wait(&empty_bar[s], ph ^ 1u)) { ok = false; break; }
                    load_a(s, kb, m0);
                    load_b(s, kb, n0);
                    if (++s == NS) { s = 0; ph ^= 1u; }
                }
            }
            if (!waited) pdl_wait();
        }
    } else if (warp == EPI_WARPS + 1) {
        // ---- MMA issuer (leader only): tiles alternate between the two accumulator buffers
        if (lane == 0 && rank == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((cat ? 2 * n : n) >> 3) << 17) | ((uint32_t)(2 * TC_BM >> 4) << 24);
            const int sets = a.rb;
            int s = 0, it = 0; uint32_t ph = 0;               // it: accumulators filled so far (a tile each, or a segment)
            for (int tile = pair; tile < total && ok; tile += npairs) {
                uint32_t d = tmem_d;
                for (int kb = 0, in = 0; kb < nk; ++kb) {     // in: K blocks that the accumulator holds
                    if (in == 0) {
                        if (!wait(&acc_empty[it & 1], ((uint32_t)(it >> 1) & 1u) ^ 1u)) { ok = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        d = tmem_d + (uint32_t)(it & 1) * 256u;
                    }
                    if (!wait(&full_bar[s], ph)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = sbase + (uint32_t)s * STAGE;
                    const uint64_t ad = umma_desc(sa), bh = umma_desc(sa + GW_A_BYTES), bl = umma_desc(sa + GW_A_BYTES + BB / 2);
                    if (cat) {
#pragma unroll
                        for (int k = 0; k < TC_BK / 16; ++k)
                            umma_pair(d + (uint32_t)((k & (sets - 1)) * 2 * n), ad + 2 * k, bh + 2 * k, idesc, (in > 0 || k >= sets) ? 1u : 0u);
                    } else {
#pragma unroll
                        for (int k = 0; k < TC_BK / 16; ++k) {
                            umma_pair(d, ad + 2 * k, bh + 2 * k, idesc, (in > 0 || k > 0) ? 1u : 0u);
                            umma_pair(d, ad + 2 * k, bl + 2 * k, idesc, 1u);
                        }
                    }
                    umma_commit_pair(&empty_bar[s]);
                    if (++s == NS) { s = 0; ph ^= 1u; }
                    ++in;
                    if (kb + 1 == nk || (SEG && in == a.seg)) { umma_commit_pair(&acc_full[it & 1]); ++it; in = 0; }
                }
            }
        }
        __syncwarp();
        pdl_trigger();                                // the last tile is issued: what follows may take the freed SMs
    } else {
        // ---- epilogue: thread = weight row, warps w and w + 4 share a lane quarter and split the activation rows
        pdl_wait();
        const int lrow = (warp & 3) * 32 + lane, part = warp >> 2;
        const bool stats = EPI == EPI_RESID && a.pk_out != nullptr && a.ss_out != nullptr;
        const uint32_t empty0 = dsmem_addr(smem_u32(&acc_empty[0]), 0);
        // the accumulator is free: tell the leader's MMA warp.  (No release at cluster scope: only tensor-memory reads, which
        // are complete, have to come before it.)
        auto release = [&](int buf) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" :: "r"(empty0 + (uint32_t)buf * 8u) : "memory");
        };
        int it = 0;
        for (int tile = pair; tile < total; tile += npairs) {            // (after a failed wait too: the block barriers below)
            const int mt = tile / ntiles, n0 = (tile - mt * ntiles) * n, m0 = mt * 2 * TC_BM + rank * TC_BM;
            const int row = m0 + lrow, nact = a.nrows - n0;
            // 1/rms of the tile's activation rows (times what truncation took), weights folded into the packed output: while the tile is
            // contracted
            epi_sync();                               // the previous tile is done with rstd_s / nw_s / ssred
            if (tid < n) {
                const float r = a.ss_in ? tc_rstd(a, a.ss_in + min(n0 + tid, a.rpad - 1), a.rpad) : 1.f;
                rstd_s[tid] = SEG ? r : r * a.found;
            }
            if (tid < TC_BM) nw_s[tid] = (a.pk_nw && m0 + tid < a.O) ? a.pk_nw[m0 + tid] : 1.f;
            epi_sync();
            const float nw = nw_s[lrow];
            const uint32_t lane_addr = tmem_d + ((uint32_t)((warp & 3) * 32) << 16);
            if constexpr (!SEG) {
                const int buf = it & 1, c_lo = part * (n / 2), c_hi = c_lo + n / 2;
                float res[8], rnext[8];
                if (EPI == EPI_RESID) tc_load_resid(a, res, n0 + c_lo, nact - c_lo, row);
                if (ok && !wait(&acc_full[buf], (uint32_t)(it >> 1) & 1u)) ok = false;
                ok = __all_sync(0xffffffffu, ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t taddr = lane_addr + (uint32_t)buf * 256u;
                for (int c0 = c_lo; c0 < c_hi && ok; c0 += 8) {
                    uint32_t x[8], y[8];
                    tmem_ld8(taddr + (uint32_t)c0, x);
                    if (cat) tmem_ld8(taddr + (uint32_t)(n + c0), y);
                    if (EPI == EPI_RESID && c0 + 8 < c_hi) tc_load_resid(a, rnext, n0 + c0 + 8, nact - (c0 + 8), row);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    float v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = cat ? __uint_as_float(x[j]) + __uint_as_float(y[j]) : __uint_as_float(x[j]);
                    for (int q = 1; q < a.rb; ++q) {
                        tmem_ld8(taddr + (uint32_t)(q * 2 * n + c0), x);
                        tmem_ld8(taddr + (uint32_t)(q * 2 * n + n + c0), y);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int j = 0; j < 8; ++j) v[j] += __uint_as_float(x[j]) + __uint_as_float(y[j]);
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] *= rstd_s[c0 + j];
                    const float sq = tc_finish<EPI, 8>(a, v, res, n0 + c0, nact - c0, row, nw, lane);
                    if (stats && (lane & 3) == 0) ssred[(warp & 3) * 256 + c0 + (lane >> 2)] = sq;
                    if (EPI == EPI_RESID)
#pragma unroll
                        for (int j = 0; j < 8; ++j) res[j] = rnext[j];
                }
                release(buf);
                ++it;
            } else {
                // a third of the tile's groups of eight rows; the sums start from the residual, whose loads hide behind the
                // first segment
                const int g_lo = part * (n / 8) / 3, ng = (part + 1) * (n / 8) / 3 - g_lo, c_lo = 8 * g_lo;
                float acc[GW_GROUPS][8];
#pragma unroll
                for (int g = 0; g < GW_GROUPS; ++g) {
                    if (EPI == EPI_RESID) tc_load_resid(a, acc[g], n0 + c_lo + 8 * g, g < ng ? nact - (c_lo + 8 * g) : 0, row);
                    else
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[g][j] = 0.f;
                }
                for (int kb = 0; kb < nk; kb += a.seg, ++it) {
                    const float gain = 1.f + a.found * (float)min(a.seg, nk - kb);
                    if (ok && !wait(&acc_full[it & 1], (uint32_t)(it >> 1) & 1u)) ok = false;
                    ok = __all_sync(0xffffffffu, ok);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t taddr = lane_addr + (uint32_t)(it & 1) * 256u + (uint32_t)c_lo;
                    for (int plane = 0; plane < (cat ? 2 * a.rb : 1) && ok; ++plane) {
                        const uint32_t tp = taddr + (uint32_t)(plane * n);
#pragma unroll
                        for (int g = 0; g < GW_GROUPS; g += 2) {
                            if (g >= ng) break;
                            const bool two = g + 1 < GW_GROUPS && g + 1 < ng;
                            uint32_t x[8], y[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                            tmem_ld8(tp + (uint32_t)(8 * g), x);
                            if (two) tmem_ld8(tp + (uint32_t)(8 * g + 8), y);
                            tmem_wait8(x); tmem_wait8(y);
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                acc[g][j] = fmaf(__uint_as_float(x[j]), gain, acc[g][j]);
                                if (g + 1 < GW_GROUPS) acc[g + 1 < GW_GROUPS ? g + 1 : g][j] = fmaf(__uint_as_float(y[j]), gain, acc[g + 1 < GW_GROUPS ? g + 1 : g][j]);
                            }
                        }
                    }
                    release(it & 1);
                }
                // three groups at a time, the rest of the sums moved up behind them: unrolled over all groups the epilogue is
                // 30 KB of instructions, which every launch fetches anew
                const float none[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                for (int q = 0; 3 * q < ng && ok; ++q) {
#pragma unroll
                    for (int u = 0; u < 3; ++u) {
                        if (3 * q + u >= ng) break;
                        const int c0 = c_lo + 8 * (3 * q + u);
                        if (EPI != EPI_RESID)
#pragma unroll
                            for (int j = 0; j < 8; ++j) acc[u][j] *= rstd_s[c0 + j];
                        const float sq = tc_finish<EPI, 8>(a, acc[u], none, n0 + c0, nact - c0, row, nw, lane);
                        if (stats && (lane & 3) == 0) ssred[(warp & 3) * 256 + c0 + (lane >> 2)] = sq;
                    }
#pragma unroll
                    for (int g = 0; g + 3 < GW_GROUPS; ++g)
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[g][j] = acc[g + 3][j];
                }
            }
            if (stats) {
                epi_sync();
                if (tid < n && tid < nact)
                    a.ss_out[(size_t)(2 * mt + rank) * a.rpad + n0 + tid] = (ssred[tid] + ssred[256 + tid]) + (ssred[512 + tid] + ssred[768 + tid]);
            }
        }
    }
    if (!ok) atomicCAS(a.status, 0, (int)HS_ERR_TIMEOUT);
    __syncwarp();
    __syncthreads();
    cluster_arrive(); cluster_wait();                 // nobody signals or reads this CTA's shared memory any more
    if (warp == EPI_WARPS) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" :: "r"(tmem_d), "r"(512u) : "memory");
}

int g_pairs = 0;                    // CTA pairs the GPU keeps resident at once

template <int EPI, bool SEG>
cudaError_t configure_one() {
    cudaError_t e = cudaFuncSetAttribute(gemm_wide_kernel<EPI, SEG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GW_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_wide_kernel<EPI, SEG>, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    return e;
}
template <int EPI>
cudaError_t configure_epi() {
    const cudaError_t e = configure_one<EPI, false>();
    return e == cudaSuccess ? configure_one<EPI, true>() : e;
}

}  // namespace

// Enough tiles of 256 x 128 to give most pairs one; below, the K split of gemm_tc_kernel fills the GPU better (residual
// projections of the 0.5B-class model at 512 rows: 26 against 30 us), as long as it splits K into ranges (`range` K blocks per
// CTA) whose MMAs may all add up in one accumulator.  Prompt passes of fewer rows: where the weight rows alone give most pairs
// a tile.
bool gemm_wide_applies(int nrows, int O, int range, bool prompt) {
    const int64_t tiles = (int64_t)((O + 255) / 256) * ((nrows + 127) / 128);
    if (g_pairs == 0) return false;
    return nrows >= 192 ? tiles >= 64 || 4 * range > GW_CHAIN : prompt && nrows >= 64 && tiles >= 48 && 4 * range > GW_CHAIN;
}

cudaError_t configure_gemm_wide() {
    cudaError_t e = configure_epi<EPI_STORE>();
    if (e == cudaSuccess) e = configure_epi<EPI_RESID>();
    if (e == cudaSuccess) e = configure_epi<EPI_SWIGLU>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(148); cfg.blockDim = dim3(gw_threads(true)); cfg.dynamicSmemBytes = GW_SMEM_MAX;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_wide_kernel<EPI_STORE, true>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    g_pairs = n;
    return cudaSuccess;
}

cudaError_t launch_gemm_wide(const GemvArgs &a, int32_t *status, cudaStream_t s, int64_t *launches, int *oparts) {
    if (a.epi == EPI_RESID && a.pk_in && a.ss_in) return cudaErrorInvalidValue;     // (the residual goes in before the 1/rms factor would)
    const int Kt = a.K0 + a.K1, nk = Kt / TC_BK, mtiles = (a.O + 2 * TC_BM - 1) / (2 * TC_BM), rpad = gemm_tc_rows(a.nrows);
    // Activation rows per tile: cycles of the busiest pair.  A K block takes its tensor time - n / 2 cycles per MMA, eight of
    // them on one accumulator (n > 128) or four of N = 2 n, each no less than 115 cycles divided by the accumulators it
    // alternates between - or the time to read its operands from L2 (about 56 bytes a cycle and SM), whichever is longer;
    // nothing hides the last tile's epilogue.
    int n = 256, sets = 1;
    int64_t best = INT64_MAX;
    for (int cand = 256; cand >= 48; cand -= 16) {
        const int r = cand <= 64 ? 2 : 1;
        const int tens = cand > 128 ? 8 * std::max(cand / 2, 115) : 4 * std::max(std::max(cand, 40), 115 / r), l2 = (16384 + 128 * cand) / 56;
        const int64_t tiles = (int64_t)mtiles * ((a.nrows + cand - 1) / cand), rounds = (tiles + g_pairs - 1) / g_pairs;
        const int64_t cost = rounds * nk * std::max(tens, l2) + 24 * cand;
        if (cost < best) { best = cost; n = cand; sets = r; }
    }
    const int ntiles = (a.nrows + n - 1) / n;
    const size_t stage = GW_A_BYTES + (size_t)n * TC_BK * 2;
    int ns = (int)((GW_SMEM_MAX - GW_MISC_BYTES - 1024) / stage);
    if (ns > GW_MAXSTAGES) ns = GW_MAXSTAGES;
    const __nv_bfloat16 *xb = a.pk_in;
    if (!xb) {
        if ((int64_t)rpad > a.xb_rows) return cudaErrorInvalidValue;
        const cudaError_t e = launch_pack(a, rpad, s, launches);
        if (e != cudaSuccess) return e;
        xb = a.xb;
    }
    CUtensorMap mA0, mA1, mB;
    cudaError_t e = hs_make_tile_map(&mA0, a.W0, a.O, a.K0, a.ldw0, TC_BM);
    if (e == cudaSuccess) e = a.K1 ? hs_make_tile_map(&mA1, a.W1, a.O, a.K1, a.ldw1, TC_BM) : hs_make_tile_map(&mA1, a.W0, a.O, a.K0, a.ldw0, TC_BM);
    if (e == cudaSuccess) e = hs_make_tile_map(&mB, xb, (uint64_t)2 * rpad, Kt, Kt, n <= 128 ? n : n / 2);
    if (e != cudaSuccess) return e;
    TcArgs t{};
    t.O = a.O; t.nk0 = a.K0 / TC_BK; t.nk1 = a.K1 / TC_BK; t.nrows = a.nrows; t.rpad = rpad; t.bnh = n; t.ns = ns; t.rb = sets;
    t.out = a.out; t.ldo = a.ldo; t.resid = a.resid; t.rparts = a.rparts; t.rpstride = a.rpstride; t.status = status;
    if (a.pk_in && a.ss_in) { t.ss_in = a.ss_in; t.ss_parts = a.ss_parts; t.inv_k = 1.f / (float)a.K0; t.eps = a.eps; }
    if (a.pk_out && a.epi != EPI_STORE) {
        t.pk_out = a.pk_out; t.pk_ld = a.pk_ld; t.pk_nw = a.pk_nw;
        t.ss_out = a.epi == EPI_RESID ? a.ss_out : nullptr;
    }
    if (a.ss_parts_out && t.ss_out) *a.ss_parts_out = (a.O + TC_BM - 1) / TC_BM;
    t.off_misc = (int)((size_t)ns * stage);
    // segments of equal length, none with more than GW_CHAIN MMAs on an accumulator
    const int most = GW_CHAIN / (n > 128 ? 8 : 4) * sets, nseg = (nk + most - 1) / most;
    t.seg = (nk + nseg - 1) / nseg;
    const float per = (n > 128 ? 8.f : 4.f / (float)sets) * TC_LOST;      // MMAs per accumulator and K block, times what each loses
    t.found = nseg > 1 ? per : 1.f + per * (float)nk;
    if (oparts) *oparts = 1;
    if (launches) ++*launches;
    const int tiles = ntiles * mtiles;
    const dim3 grid(2 * (tiles < g_pairs ? tiles : g_pairs)), block(gw_threads(nseg > 1));
    const size_t smem = GW_SMEM_MAX;          // one CTA per SM: the pair's tensor memory is allocated whole
#define WIDE(epi_) (nseg > 1 ? launch_pdl_cluster(gemm_wide_kernel<epi_, true>, grid, block, smem, s, 2, mA0, mA1, mB, t, ntiles, mtiles) \
                             : launch_pdl_cluster(gemm_wide_kernel<epi_, false>, grid, block, smem, s, 2, mA0, mA1, mB, t, ntiles, mtiles))
    return a.epi == EPI_STORE ? WIDE(EPI_STORE) : a.epi == EPI_RESID ? WIDE(EPI_RESID) : WIDE(EPI_SWIGLU);
#undef WIDE
}
