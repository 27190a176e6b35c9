// Projection for several activation rows (from 4 or 6 on, tc_rows in hs_api.cu): a dense contraction, run on the
// fifth-generation tensor cores.  out[r][o] = sum_j W[o][j] x[r][j] is computed as D = A B^T with
//   A = a tile of 128 rows of the weight matrix (bf16, K-major; 64 rows in residual projections whose tiles would leave
//       half of the GPU idle), streamed by TMA tensor copies into 128-byte swizzled shared-memory stages,
//   B = the activation rows as bf16 head and bf16 remainder planes (x = head + remainder to 2^-17, the RMSNorm weight
//       folded in); a CTA takes BNH rows of each plane as the N = 2 * BNH columns of its tile.  The planes are written by the
//       kernel that produces the rows - the epilogue of the projection before, the mixer of a draft step or a DeltaNet layer -
//       with partial sums of squares beside them, from which 1/rms is applied to the finished sums; or, where nobody does (the
//       embedding, what mixer and attention of a verify pass hand on), by pack_kernel with 1/rms folded in,
//   D = 128 (64) x N fp32 accumulators in tensor memory; the epilogue reads them back with tcgen05.ld, adds the head
//       and remainder columns and applies the store / residual / SwiGLU epilogue.
// One elected thread issues the TMA copies, one issues tcgen05.mma (K = 16 per instruction, four per 64-column
// stage) and releases stages with tcgen05.commit; all eight warps run the epilogue (whole K range: thread = weight row, two
// warps per lane quarter, each half of the columns).  Every wait is bounded.
// Every CTA fetches its own tiles (no copy is shared between CTAs).
// The weights are the large operand, so the grid is filled by splitting K, not N: the CTAs of a thread-block
// cluster (up to 8) take consecutive K ranges of the same tile.  Each finishes an equal share of the tile's activation rows: the
// others store their partial sums of those rows straight into its shared memory, and after one cluster barrier it adds them
// in rank order, four columns of a weight row per thread - every weight byte is fetched once and the result does not depend
// on timing.
#include "hs_internal.h"
#include "hs_device.cuh"
#include "gemm_tc_common.cuh"
#include <cuda.h>
#include <cstdio>
#include <cstdlib>

namespace {
using namespace hsd;

constexpr int TC_THREADS = 256;    // two warps per tensor-memory lane quarter: each takes half of the columns in the epilogue
constexpr int TC_MAXSTAGES = 8;

// ---- tensor maps (driver entry point fetched once; the library does not link libcuda) ----------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;

// 2-D bf16 tensor [rows][cols] with row stride ld (elements), box = TC_BK columns x box_rows rows, 128-byte swizzle
cudaError_t make_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows) {
    if (!g_encode) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)TC_BK, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// ---- pack: fp32 activation rows -> bf16 head plane | bf16 remainder plane, [2][rpad][Kt], norm folded in -----
struct PackArgs {
    const float *x0; int ldx0, K0, xparts; int64_t xpstride; const float *norm_w; float eps;
    const float *x1; int ldx1, K1;
    __nv_bfloat16 *xb; int nrows, rpad;
};

__global__ void __launch_bounds__(256) pack_kernel(const PackArgs a) {
    const int r = blockIdx.x, Kt = a.K0 + a.K1;
    __shared__ float red[8];
    __nv_bfloat16 *hi = a.xb + (size_t)r * Kt, *lo = a.xb + ((size_t)a.rpad + r) * Kt;
    pdl_trigger();
    pdl_wait();
    if (r >= a.nrows) {                        // padding rows are zero in both planes
        for (int c = threadIdx.x * 8; c < Kt; c += blockDim.x * 8) {
            *reinterpret_cast<uint4 *>(hi + c) = make_uint4(0, 0, 0, 0);
            *reinterpret_cast<uint4 *>(lo + c) = make_uint4(0, 0, 0, 0);
        }
        return;
    }
    float rstd = 1.f;
    if (a.norm_w) {
        float ss = 0.f;
        for (int c = threadIdx.x * 4; c < a.K0; c += blockDim.x * 4) {
            float4 v = __ldcg(reinterpret_cast<const float4 *>(a.x0 + (size_t)r * a.ldx0 + c));
            for (int q = 1; q < a.xparts; ++q) {
                const float4 u = __ldcg(reinterpret_cast<const float4 *>(a.x0 + (size_t)q * a.xpstride + (size_t)r * a.ldx0 + c));
                v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
            }
            ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
        ss = warp_sum(ss);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
        __syncthreads();
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += red[w];
        rstd = rsqrtf(t / (float)a.K0 + a.eps);
    }
    for (int c = threadIdx.x * 4; c < Kt; c += blockDim.x * 4) {
        float4 v;
        if (c < a.K0) {
            v = __ldcg(reinterpret_cast<const float4 *>(a.x0 + (size_t)r * a.ldx0 + c));
            for (int q = 1; q < a.xparts; ++q) {
                const float4 u = __ldcg(reinterpret_cast<const float4 *>(a.x0 + (size_t)q * a.xpstride + (size_t)r * a.ldx0 + c));
                v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
            }
            if (a.norm_w) {
                const float4 nw = *reinterpret_cast<const float4 *>(a.norm_w + c);
                v.x *= nw.x * rstd; v.y *= nw.y * rstd; v.z *= nw.z * rstd; v.w *= nw.w * rstd;
            }
        } else {
            v = __ldcg(reinterpret_cast<const float4 *>(a.x1 + (size_t)r * a.ldx1 + (c - a.K0)));
        }
        const float x[4] = {v.x, v.y, v.z, v.w};
        uint32_t hw[2], lw[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const __nv_bfloat16 h0 = __float2bfloat16_rn(x[2 * e]), h1 = __float2bfloat16_rn(x[2 * e + 1]);
            const __nv_bfloat16 l0 = __float2bfloat16_rn(x[2 * e] - __bfloat162float(h0)), l1 = __float2bfloat16_rn(x[2 * e + 1] - __bfloat162float(h1));
            hw[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
            lw[e] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
        }
        *reinterpret_cast<uint2 *>(hi + c) = make_uint2(hw[0], hw[1]);
        *reinterpret_cast<uint2 *>(lo + c) = make_uint2(lw[0], lw[1]);
    }
}

// ---- the contraction ---------------------------------------------------------------------------------------
// BN: N of the MMA = 2 * bnh (head columns, then remainder columns).  BM: weight rows per tile; 64 only with a K split (row r of
// the tile is then lane r % 16 of tensor-memory quarter r / 16).  EPI: the epilogue, fixed at compile time.
template <int BN, int BM, int EPI>
__global__ void __launch_bounds__(TC_THREADS, 2)
gemm_tc_kernel(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
               const __grid_constant__ CUtensorMap mB, const TcArgs a) {
    constexpr uint32_t A_BYTES = BM * TC_BK * 2, B_BYTES = BN * TC_BK * 2, STAGE = A_BYTES + B_BYTES;
    constexpr uint32_t TCOLS = BN < 32 ? 32 : BN;
    constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    constexpr int BNH = BN / 2, RW = BM / 32, CG = 8 / RW;     // finishing a split tile: RW warps side by side, CG groups of four columns at a time
    extern __shared__ unsigned char smraw[];
    __shared__ __align__(8) uint64_t full_bar[TC_MAXSTAGES], empty_bar[TC_MAXSTAGES], done_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ int failed_s;
    const uint32_t sbase = (smem_u32(smraw) + 1023u) & ~1023u;            // swizzled tiles need 1024-byte alignment
    unsigned char *stages = smraw + (sbase - smem_u32(smraw));
    float *rx = reinterpret_cast<float *>(stages + a.off_rx);             // [S][rb / 4][BM][4]: partial tiles sent by the cluster's ranks
    float *rstd_s = reinterpret_cast<float *>(stages + a.off_misc);       // [BNH] 1/rms and what truncation took
    float *nw_s = rstd_s + 128;                                           // [128]
    float *ssred = nw_s + 128;                                            // [4][BNH]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // grid = (K splits = cluster size, weight-row tiles, activation-row tiles)
    const int S = (int)gridDim.x, q = (int)blockIdx.x;
    const int m0 = blockIdx.y * BM, n0h = blockIdx.z * BNH;
    const int nk = a.nk0 + a.nk1, NS = a.ns;
    const int kb0 = (int)((long long)q * nk / S), kb1 = (int)((long long)(q + 1) * nk / S), nkl = kb1 - kb0;
    if (a.early_trigger) pdl_trigger();
    if (tid == 0) {
        for (int s = 0; s < NS; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&done_bar, 1);
        mbar_fence_init();
        failed_s = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&tmem_base_s)), "r"(TCOLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // parameters (nothing a kernel writes): the weights folded into the packed output
    if (tid >= 256 - BM) {
        const int i = tid - (256 - BM);
        nw_s[i] = (a.pk_nw && m0 + i < a.O) ? a.pk_nw[m0 + i] : 1.f;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_base_s;
    // first phase of the cluster barrier: "this CTA runs" - a rank's shared memory may be written once every rank has
    // arrived here; nobody waits for it before the exchange at the end
    if (S > 1) cluster_arrive();

    if (warp == 0 && lane == 0) {
        // ---- TMA producer.  Weight tiles depend on nothing: the first stages are requested before the wait.
        auto load_a = [&](int i) {                      // i: k block relative to kb0
            const int s = i % NS, kb = kb0 + i;
            mbar_expect_tx(&full_bar[s], STAGE);
            if (kb < a.nk0) tma_load_2d_stream(stages + (size_t)s * STAGE, &mA0, kb * TC_BK, m0, &full_bar[s]);
            else tma_load_2d_stream(stages + (size_t)s * STAGE, &mA1, (kb - a.nk0) * TC_BK, m0, &full_bar[s]);
        };
        auto load_b = [&](int i) {
            const int s = i % NS, kb = kb0 + i;
            unsigned char *bs = stages + (size_t)s * STAGE + A_BYTES;
            tma_load_2d(bs, &mB, kb * TC_BK, n0h, &full_bar[s]);
            tma_load_2d(bs + (size_t)BNH * TC_BK * 2, &mB, kb * TC_BK, a.rpad + n0h, &full_bar[s]);
        };
        const int pre = nkl < NS ? nkl : NS;
        for (int i = 0; i < pre; ++i) load_a(i);
        pdl_wait();
        for (int i = 0; i < pre; ++i) load_b(i);
        for (int i = NS; i < nkl; ++i) {
            if (!mbar_wait(&empty_bar[i % NS], (uint32_t)(i / NS - 1) & 1u)) { failed_s = 1; break; }
            load_a(i);
            load_b(i);
        }
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer
        for (int i = 0; i < nkl; ++i) {
            const int s = i % NS;
            if (!mbar_wait(&full_bar[s], (uint32_t)(i / NS) & 1u)) { failed_s = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sa = sbase + (uint32_t)s * STAGE;
            const uint64_t ad = umma_desc(sa), bd = umma_desc(sa + A_BYTES);
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)       // 32 bytes further along K per instruction (descriptor units of 16 bytes)
                umma_bf16(tmem_d, ad + 2 * k, bd + 2 * k, IDESC, (i > 0 || k > 0) ? 1u : 0u);
            umma_commit(&empty_bar[s]);                 // the stage is free once these MMAs have read it
        }
        umma_commit(&done_bar);                         // accumulators complete
    } else if (warp >= 2) {
        // ---- the other warps: pull the next projection's weights into L2, then the 1/rms factors of this tile's rows
        if (a.pf_bytes > 0) {
            const long long ncta = (long long)gridDim.x * gridDim.y * gridDim.z;
            const long long cta = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
            const long long per = ((a.pf_bytes + ncta - 1) / ncta + 15) & ~15ll;
            const long long lo = cta * per, hi = min(lo + per, a.pf_bytes & ~15ll);
#pragma unroll 1
            for (long long o = lo + (long long)(tid - 64) * 4096; o < hi; o += (TC_THREADS - 64) * 4096)
                prefetch_l2(reinterpret_cast<const char *>(a.pf_ptr) + o, (uint32_t)min(4096ll, hi - o));
        }
        pdl_wait();
        if (a.ss_in && a.ss_by_row) {
            // many partial sums (one per block of the mixer): a warp per activation row, three rows at a time
            constexpr int W = TC_THREADS / 32 - 2;
#pragma unroll 1
            for (int i0 = warp - 2; i0 < BNH; i0 += 3 * W) {
                float t[3] = {0.f, 0.f, 0.f};
                for (int p0 = lane; p0 < a.ss_parts; p0 += 128) {
                    float x[3][4];
#pragma unroll
                    for (int r = 0; r < 3; ++r)
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            x[r][u] = n0h + i0 + r * W < a.nrows && p0 + 32 * u < a.ss_parts ? __ldcg(a.ss_in + (size_t)(n0h + i0 + r * W) * a.ss_parts + p0 + 32 * u) : 0.f;
#pragma unroll
                    for (int r = 0; r < 3; ++r) t[r] += (x[r][0] + x[r][1]) + (x[r][2] + x[r][3]);
                }
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const float tot = warp_sum(t[r]);
                    if (lane == 0 && i0 + r * W < BNH) rstd_s[i0 + r * W] = rsqrtf(tot * a.inv_k + a.eps) * a.found;
                }
            }
        } else
#pragma unroll 1
        for (int i = tid - 64; i < BNH; i += TC_THREADS - 64) {
            rstd_s[i] = (a.ss_in ? tc_rstd(a, a.ss_in + n0h + i, a.rpad) : 1.f) * a.found;
        }
    }
    if (warp < 2 && !(warp == 0 && lane == 0)) pdl_wait();          // the epilogue reads the residual stream
    __syncwarp();
    // ---- epilogue.  Whole K range: thread = accumulator lane = weight row, warps w and w + 4 share a lane quarter and split the
    //      columns (activation rows).  K split: rank p finishes the activation rows [p * rb, (p + 1) * rb) of the tile (the last ranks
    //      may find none), four columns of a weight row per thread at a time.
    const int nact = a.nrows - n0h;                     // activation rows of this tile that exist
    const bool stats = EPI == EPI_RESID && a.pk_out != nullptr && a.ss_out != nullptr;
    const int half = warp >> 2, rb = a.rb;
    const int c_lo = S > 1 ? min(q * rb, BNH) : 0, c_n = S > 1 ? min(rb, BNH - c_lo) : BNH;     // the tile's activation rows this CTA finishes
    const int frow = S > 1 ? (warp % RW) * 32 + lane : (warp & 3) * 32 + lane, cg = warp / RW;
    const int row = m0 + frow;
    // the first columns this thread finishes: their residual is requested now, the trip to L2 hides behind the contraction
    float res4[4], res[8];
    if (EPI == EPI_RESID) {
        if (S > 1) tc_load_resid<4>(a, res4, n0h + c_lo + cg * 4, min(c_n - cg * 4, nact - (c_lo + cg * 4)), row);
        else if (BM == TC_BM) tc_load_resid<8>(a, res, n0h + half * (BNH / 2), nact - half * (BNH / 2), row);
    }
    __syncthreads();                                    // rstd_s complete
    const float nw = nw_s[frow];
    const bool ok = mbar_wait(&done_bar, 0) && !failed_s;
    if (!a.early_trigger) pdl_trigger();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = tmem_d + ((uint32_t)((warp & 3) * 32) << 16);
    if (!ok && tid == 0) atomicCAS(a.status, 0, (int)HS_ERR_TIMEOUT);
    if (S == 1) {
        if (BM == TC_BM && ok) {
            for (int c0 = half * (BNH / 2); c0 < (half + 1) * (BNH / 2); c0 += 8) {
                uint32_t h[8], l[8];
                tmem_ld8(taddr + (uint32_t)c0, h);
                tmem_ld8(taddr + (uint32_t)(BNH + c0), l);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                float v[8], rnext[8];
                if (EPI == EPI_RESID && c0 + 8 < (half + 1) * (BNH / 2)) tc_load_resid<8>(a, rnext, n0h + c0 + 8, nact - (c0 + 8), row);
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = (__uint_as_float(h[j]) + __uint_as_float(l[j])) * rstd_s[c0 + j];
                const float sq = tc_finish<EPI, 8>(a, v, res, n0h + c0, nact - c0, row, nw, lane);
                if (stats && (lane & 3) == 0) ssred[(warp & 3) * BNH + c0 + (lane >> 2)] = sq;
                if (EPI == EPI_RESID)
#pragma unroll
                    for (int j = 0; j < 8; ++j) res[j] = rnext[j];
            }
        }
    } else {
        // Every rank sends the matching columns of its partial tile straight into rank p's shared memory
        // ([sender][four columns][weight row]: remote stores of 16 bytes, side by side for the lanes of a warp), ONE cluster
        // barrier, then each rank adds the S partials of its rows in rank order - the result does not depend on timing.
        // (With a weight row's columns side by side the lanes of a store, and of a load, were rb * 4 bytes apart and hit the same
        // banks: 128 rows of the 0.5B-class model, down-projection at 320 activation rows 3.5 us sending and 4.8 us adding.)
        cluster_wait();                                 // every rank runs: its receive area may be written
        const int lrow = BM == TC_BM ? (warp & 3) * 32 + lane : (warp & 3) * 16 + (lane & 15);
        const bool has_row = BM == TC_BM || lane < 16;
        const uint32_t rx_mine = smem_u32(rx) + (uint32_t)((q * (rb >> 2) * BM + lrow) * 16);
        for (int c0 = half * (BNH / 2); c0 < (half + 1) * (BNH / 2); c0 += 8) {
            uint32_t h[8], l[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) h[j] = l[j] = 0u;
            if (ok && nkl > 0) {
                tmem_ld8(taddr + (uint32_t)c0, h);
                tmem_ld8(taddr + (uint32_t)(BNH + c0), l);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            }
#pragma unroll
            for (int e = 0; e < 8; e += 4) {
                const uint32_t p = ((uint32_t)(c0 + e) * (uint32_t)a.rb_inv) >> 16, cl = (uint32_t)(c0 + e) - p * (uint32_t)rb;      // (c0 + e) / rb
                if (has_row)
                    dsmem_st_v4(dsmem_addr(rx_mine + (cl >> 2) * (BM * 16), p), __uint_as_float(h[e]) + __uint_as_float(l[e]), __uint_as_float(h[e + 1]) + __uint_as_float(l[e + 1]),
                                __uint_as_float(h[e + 2]) + __uint_as_float(l[e + 2]), __uint_as_float(h[e + 3]) + __uint_as_float(l[e + 3]));
            }
        }
        cluster_arrive(); cluster_wait();
        for (int cl0 = cg * 4; cl0 < c_n; cl0 += 4 * CG) {
            float v[4], rnext[4];
            if (EPI == EPI_RESID && cl0 + 4 * CG < c_n) tc_load_resid<4>(a, rnext, n0h + c_lo + cl0 + 4 * CG, nact - (c_lo + cl0 + 4 * CG), row);
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = 0.f;
            const float4 *pr = reinterpret_cast<const float4 *>(rx) + (cl0 >> 2) * BM + frow;
#pragma unroll
            for (int p = 0; p < 8; ++p)
                if (p < S) { const float4 x = pr[p * (rb >> 2) * BM]; v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w; }
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] *= rstd_s[c_lo + cl0 + j];
            const float sq = tc_finish<EPI, 4>(a, v, res4, n0h + c_lo + cl0, nact - (c_lo + cl0), row, nw, lane);
            if (stats && (lane & 7) == 0) ssred[(warp % RW) * BNH + c_lo + cl0 + (lane >> 3)] = sq;
            if (EPI == EPI_RESID)
#pragma unroll
                for (int j = 0; j < 4; ++j) res4[j] = rnext[j];
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (stats && ok) {
        // sums of squares of the finished rows over this tile's weight rows, 32 after 32
        for (int i = tid; i < c_n; i += TC_THREADS) {
            const int c = c_lo + i;
            if (c < nact) a.ss_out[(size_t)blockIdx.y * a.rpad + n0h + c] = BM == TC_BM ? (ssred[c] + ssred[BNH + c]) + (ssred[2 * BNH + c] + ssred[3 * BNH + c]) : ssred[c] + ssred[BNH + c];
        }
    }
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_d), "r"(TCOLS) : "memory");
}

constexpr size_t tc_stage_bytes(int bn, int bm) { return (size_t)bm * TC_BK * 2 + (size_t)bn * TC_BK * 2; }
constexpr size_t TC_SMEM_MAX = 200 * 1024;
constexpr size_t TC_SMEM_PAIR = 110 * 1024;   // up to this two CTAs fit on an SM
constexpr size_t TC_MISC_BYTES = (128 + 128 + 4 * 128) * 4;
int g_tc_clusters[2][9];     // clusters of S CTAs that run at once with one CTA per SM ([0]; [1]: the same query at the smaller footprint)

template <int BN, int BM, int EPI>
cudaError_t launch_tc(const CUtensorMap &mA0, const CUtensorMap &mA1, const CUtensorMap &mB, const TcArgs &t, dim3 grid, size_t smem, cudaStream_t s) {
    static bool configured = false;
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<BN, BM, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM_MAX);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_tc_kernel<BN, BM, EPI>, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    return launch_pdl_cluster(gemm_tc_kernel<BN, BM, EPI>, grid, dim3(TC_THREADS), smem, s, (int)grid.x, mA0, mA1, mB, t);
}
template <int BN>
cudaError_t launch_tc_epi(int epi, int bm, const CUtensorMap &mA0, const CUtensorMap &mA1, const CUtensorMap &mB, const TcArgs &t, dim3 grid, size_t smem, cudaStream_t s) {
    if (epi == EPI_STORE) return launch_tc<BN, TC_BM, EPI_STORE>(mA0, mA1, mB, t, grid, smem, s);
    if (epi == EPI_RESID) return bm == 64 ? launch_tc<BN, 64, EPI_RESID>(mA0, mA1, mB, t, grid, smem, s) : launch_tc<BN, TC_BM, EPI_RESID>(mA0, mA1, mB, t, grid, smem, s);
    return launch_tc<BN, TC_BM, EPI_SWIGLU>(mA0, mA1, mB, t, grid, smem, s);
}

}  // namespace

bool g_hs_gemm_tc = true;
bool g_hs_tensor_maps = false;

cudaError_t hs_make_tile_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows) {
    return make_map(map, base, rows, cols, ld, box_rows);
}
cudaError_t hs_make_f32_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_cols, uint32_t box_rows) {
    if (!g_encode) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {ld * 4};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void *>(base), dims, strides, box, estr,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// K or V cache of one layer as a 2-D bf16 tensor [rows][hd]: boxes of 64 columns x 128 rows, 128-byte swizzle
cudaError_t hs_make_kv_tensor_map(CUtensorMap *map, const void *base, uint64_t rows, int hd) {
    if (hd % 64) return cudaErrorInvalidValue;
    return make_map(map, base, rows, (uint64_t)hd, (uint64_t)hd, 128);
}

cudaError_t configure_gemm_tc() {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (e != cudaSuccess) return e;
    if (qres != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    g_hs_tensor_maps = true;
    e = cudaFuncSetAttribute(pack_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(gemm_tc_kernel<32, TC_BM, EPI_STORE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM_MAX);
    if (e != cudaSuccess) return e;
    for (int pair = 0; pair < 2; ++pair)
        for (int S = 1; S <= 8; ++S) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(S, 148 / S); cfg.blockDim = dim3(TC_THREADS); cfg.dynamicSmemBytes = pair ? TC_SMEM_PAIR : TC_SMEM_MAX;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = S; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
            cfg.attrs = at; cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, gemm_tc_kernel<32, TC_BM, EPI_STORE>, &cfg) == cudaSuccess && n > 0) g_tc_clusters[pair][S] = n;
            else { g_tc_clusters[pair][S] = S == 1 ? 148 : 0; cudaGetLastError(); }
            if (getenv("HS_VERBOSE")) fprintf(stderr, "libhs: tcgen05 projection, clusters of %d CTAs (%d per SM) resident at once: %d\n", S, pair + 1, g_tc_clusters[pair][S]);
        }
    return cudaSuccess;
}

// Rows per plane per CTA (a power of two, 16..128) and rows per plane of the packed operand for nrows activation rows.
static int tc_bnh(int nrows) { int b = 16; while (b < 128 && b < nrows) b <<= 1; return b; }
int gemm_tc_rows(int nrows) { const int b = tc_bnh(nrows); return (nrows + b - 1) / b * b; }

cudaError_t launch_pack(const GemvArgs &a, int rpad, cudaStream_t s, int64_t *launches) {
    const PackArgs p{a.x0, a.ldx0, a.K0, a.xparts, a.xpstride, a.norm_w, a.eps, a.x1, a.ldx1, a.K1, a.xb, a.nrows, rpad};
    if (launches) ++*launches;
    return launch_pdl(pack_kernel, dim3(rpad), dim3(256), 0, s, p);
}

cudaError_t launch_gemm_tc(const GemvArgs &a, int32_t *status, cudaStream_t s, int64_t *launches, int *oparts) {
    if ((!a.xb && !a.pk_in) || (a.K0 & 63) || (a.K1 & 63) || a.nrows < 1) return cudaErrorInvalidValue;
    const int Kt = a.K0 + a.K1;
    const int mtiles = (a.O + TC_BM - 1) / TC_BM, nk = Kt / TC_BK;
    // Rows per plane per CTA.  The packed operand is laid out for the largest tile (rpad rows per plane); a small
    // weight matrix is cheap to read again from L2, so its activation rows are cut into more, smaller tiles, which
    // shortens every CTA's epilogue and spares the K split (measured on 1024-wide layers: 64 rows 4 %, 128 rows 6 %,
    // 192 rows 4 % per pass; large matrices and more than 256 rows lose)
    const int rpad = gemm_tc_rows(a.nrows);
    int bnh = tc_bnh(a.nrows);
    if ((int64_t)a.O * Kt * 2 <= ((int64_t)20 << 20)) {
        const int cap = a.nrows <= 64 ? 32 : a.nrows <= 256 ? 64 : 128;
        if (bnh > cap) bnh = cap;
    }
    const int ntiles = (a.nrows + bnh - 1) / bnh;
    // K split (cluster size, 1..8): the weights are the large operand, so the grid is filled by splitting K, as long as
    // all CTAs still run at once, at most one per SM, and every CTA keeps at least two K blocks.  Rank p of a cluster
    // finishes rb activation rows of the tile (a multiple of four).  A residual projection of few weight rows cannot fill half of the
    // GPU that way: it goes out in tiles of 64 weight rows, twice as many.
    // (the CTAs of a cluster share a GPC, so fewer clusters of S CTAs than SMs / S may run at once: g_tc_clusters)
    struct Split { int S, rb; size_t rx_bytes, budget; };
    auto split_for = [&](int bm) {
        const size_t stage = tc_stage_bytes(2 * bnh, bm);
        const int tiles = (a.O + bm - 1) / bm * ntiles;
        Split r{1, 4, 0, TC_SMEM_MAX};
        for (int cand = 1; cand <= 8; ++cand) {
            if (cand > 1 && nk / cand < 2) break;
            const int crb = ((bnh + cand - 1) / cand + 3) / 4 * 4;
            const size_t crx = cand > 1 ? (size_t)cand * crb * bm * 4 : 0;
            // Stages as deep as shared memory allows: a refill costs a trip to L2 on the critical path (measured: deep
            // stages with one CTA per SM beat two co-resident CTAs with two or three stages each).  Few activation rows
            // make the stages small: then two CTAs fit on an SM with four or more stages each, more CTAs than SMs still
            // run at once and the CTAs of the next projection can stream their weights while this one finishes.
            // More tiles than SMs would otherwise run in two rounds, the second nearly empty: there three stages are enough
            // for a pair (measured: 4-6 % per verify pass on the batched workloads; with two stages it loses again).
            const bool pair = TC_SMEM_PAIR >= 4 * stage + crx + TC_MISC_BYTES + 1024 ||
                              (tiles * cand > 148 && TC_SMEM_PAIR >= 3 * stage + crx + TC_MISC_BYTES + 1024);
            // with two CTAs per SM twice as many clusters run at once (the occupancy query is made for one per SM)
            if (cand > 1 && tiles > g_tc_clusters[0][cand] * (pair ? 2 : 1)) continue;
            if (cand > 1 && tiles * cand > (pair ? 2 * 148 : 148)) continue;
            r = Split{cand, crb, crx, pair ? TC_SMEM_PAIR : TC_SMEM_MAX};
        }
        return r;
    };
    Split sp = split_for(TC_BM);
    int bm = TC_BM;
    if (a.epi == EPI_RESID && mtiles * ntiles * sp.S <= 74) {
        const Split half = split_for(64);
        if (half.S > 1) { sp = half; bm = 64; }
    }
    const int S = sp.S, rb = sp.rb;
    const size_t stage = tc_stage_bytes(2 * bnh, bm), rx_bytes = sp.rx_bytes, budget = sp.budget;
    const int nkl = (nk + S - 1) / S;
    if (gemm_wide_applies(a.nrows, a.O, nkl, a.prompt)) return launch_gemm_wide(a, status, s, launches, oparts);
    int ns = (int)((budget - rx_bytes - TC_MISC_BYTES - 1024) / stage);
    if (ns > TC_MAXSTAGES) ns = TC_MAXSTAGES;
    if (ns > nkl) ns = nkl;
    if (ns < 1) return cudaErrorInvalidValue;
    size_t smem = (size_t)ns * stage + rx_bytes + TC_MISC_BYTES + 1024;
    // tensor memory is not oversubscribed: a CTA's share of the SM's shared memory is at least its share of the
    // 512 tensor-memory columns, so an allocation never has to wait for a CTA of another cluster (which could
    // itself be waiting, at its cluster barrier, for a peer queued behind this one)
    const size_t tcols = 2 * bnh < 32 ? 32 : 2 * bnh, share = (size_t)228 * 1024 * tcols / 512 + 1024;
    if (smem < share) smem = share;
    if (smem > TC_SMEM_MAX) return cudaErrorInvalidValue;
    const __nv_bfloat16 *xb = a.pk_in;
    if (!xb) {
        if ((int64_t)rpad > a.xb_rows) return cudaErrorInvalidValue;
        const cudaError_t e = launch_pack(a, rpad, s, launches);
        if (e != cudaSuccess) return e;
        xb = a.xb;
    }
    CUtensorMap mA0, mA1, mB;
    cudaError_t e = make_map(&mA0, a.W0, a.O, a.K0, a.ldw0, bm);
    if (e == cudaSuccess) e = a.K1 ? make_map(&mA1, a.W1, a.O, a.K1, a.ldw1, bm) : make_map(&mA1, a.W0, a.O, a.K0, a.ldw0, bm);
    if (e == cudaSuccess) e = make_map(&mB, xb, (uint64_t)2 * rpad, Kt, Kt, bnh);
    if (e != cudaSuccess) return e;
    TcArgs t{};
    t.O = a.O; t.nk0 = a.K0 / TC_BK; t.nk1 = a.K1 / TC_BK; t.nrows = a.nrows; t.rpad = rpad; t.bnh = bnh; t.ns = ns; t.rb = rb; t.rb_inv = 65536 / rb + 1;
    t.out = a.out; t.ldo = a.ldo; t.resid = a.resid; t.rparts = a.rparts; t.rpstride = a.rpstride; t.status = status;
    if (a.pk_in && a.ss_in) { t.ss_in = a.ss_in; t.ss_parts = a.ss_parts; t.inv_k = 1.f / (float)a.K0; t.eps = a.eps; t.ss_by_row = a.ss_by_row; }
    if (a.pk_out && a.epi != EPI_STORE) {
        t.pk_out = a.pk_out; t.pk_ld = a.pk_ld; t.pk_nw = a.pk_nw;
        t.ss_out = a.epi == EPI_RESID ? a.ss_out : nullptr;
    }
    t.pf_ptr = a.pf_ptr; t.pf_bytes = a.pf_ptr ? (long long)a.pf_bytes : 0;
    t.off_rx = (int)((size_t)ns * stage); t.off_misc = (int)((size_t)ns * stage + rx_bytes);
    t.early_trigger = a.early_trigger; t.found = 1.f + (float)(nk * (TC_BK / 16)) / (float)S * TC_LOST;
    if (oparts) *oparts = 1;
    if (launches) ++*launches;
    if (a.ss_parts_out && t.ss_out) *a.ss_parts_out = (a.O + bm - 1) / bm;
    const dim3 grid(S, (a.O + bm - 1) / bm, ntiles);
    switch (2 * bnh) {
        case 32: return launch_tc_epi<32>(a.epi, bm, mA0, mA1, mB, t, grid, smem, s);
        case 64: return launch_tc_epi<64>(a.epi, bm, mA0, mA1, mB, t, grid, smem, s);
        case 128: return launch_tc_epi<128>(a.epi, bm, mA0, mA1, mB, t, grid, smem, s);
        default: return launch_tc_epi<256>(a.epi, bm, mA0, mA1, mB, t, grid, smem, s);
    }
}
